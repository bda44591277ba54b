"""The fused single-phase step at the edges of its chunks (512 elements per warp, 8192 per tile) and of
its alignments: gradients at every offset from a 16-byte boundary, sizes just below, at and above the
edges, odd sizes, every block size; codes, scales, messages and the decoded error bit for bit."""
import pytest

from paper_2312_08538_b200 import workloads as wl
from tests.test_gpu_parity import run_single_phase

pytestmark = pytest.mark.gpu

# each 1-D tensor moves what follows by one element
EDGES = [(1, 511, 1), (1, 1, 0), (1, 513, 1), (2, 1, 0), (16, 32, 1), (1, 1, 0), (3, 5, 1), (1, 8191, 1), (1, 1, 0), (2, 4096, 1),
         (1, 8193, 1), (1, 2, 1), (129, 127, 1), (1, 1, 0), (33, 1024, 1)]


@pytest.mark.parametrize("qkind", ["randk", "randblock", "identity"])
@pytest.mark.parametrize("c", [dict(kind="int8", block=256), dict(kind="int8", block=32, scale_dtype="fp16"),
                               dict(kind="int8", block=64), dict(kind="int4", block=128, scale_dtype="fp16"),
                               dict(kind="int4", block=64), dict(kind="int8", block=64, iconef=1),
                               dict(kind="int4", block=256, scale_dtype="fp16", iconef=1),
                               dict(kind="stochquant", block=128, levels=20), dict(kind="identity"),
                               dict(kind="identity", beta=0.5)])
def test_edges_bit_exact(qkind, c):
    cfg = wl.config("tiny")
    cfg.update(tensors=EDGES, n_workers=2, q=dict(kind=qkind, k_num=1, k_den=9, seed=31), c=dict(c))
    run_single_phase(cfg, 3, exact_values=True)
