"""The low-rank model update at the edges of its tiles: every rank class, widths with and without
16-byte rows, more than one column tile, row remainders, parameters off a 16-byte boundary."""
import pytest
import torch

from paper_2312_08538_b200 import workloads as wl
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

SHAPES = [(70, 64, 1), (3, 1, 0), (33, 257, 1), (9, 1028, 1), (5, 4, 1), (260, 1027, 1), (2, 600, 1)]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("rank", [1, 2, 3, 4, 8])
def test_update_is_phat_qmean(rank, offset):
    cfg = wl.config("resnet50-mini")
    cfg.update(tensors=SHAPES, n_workers=2, q=dict(kind="lowrank", rank=rank))
    eng = pu.make_gpu(cfg, q_init=wl.q_init(cfg, "cuda"))
    gd, _ = pu.grads_both(cfg, 0)
    total = wl.total_elems(SHAPES)
    x = torch.randn(total + offset, device="cuda")[offset:]
    want = x.double().clone()
    sums = eng.full_step(0, gd)
    eng.apply_update(x, sums)
    off = off1 = 0
    for l, (r, c, k) in enumerate(SHAPES):
        if k and c > 1:
            f = eng.factors(l, 0)
            delta = f["p_hat"].double() @ f["q_prev"].double().T
        else:
            delta = sums[3][off1:off1 + r * c].double() / 2
            off1 += r * c
        want[off:off + r * c] -= delta.reshape(-1)
        off += r * c
    assert torch.allclose(x.double(), want, rtol=0, atol=1e-6 * float(want.abs().max()))
