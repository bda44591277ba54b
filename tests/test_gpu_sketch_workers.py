"""The count-sketch step with the workers' sketches interleaved: one to nine workers, one to seven sketch
rows, several groups of tensors, a tensor too large for a group, against the oracle and against the
generic kernel (sums of bucket entries in another order)."""
import pytest
import torch

from paper_2312_08538_b200 import workloads as wl
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

SMALL = [(37, 53, 1), (19, 1, 0), (1, 7, 1), (1, 1025, 1), (64, 129, 1), (300, 1, 0), (2, 512, 1), (5, 1000, 1)]


def _run(cfg, fast, steps=3):
    eng = pu.make_gpu(cfg, fast=fast)
    outs = []
    for t in range(steps):
        g = [wl.gradient(cfg, i, t, device="cuda") for i in range(cfg["n_workers"])]
        res = eng.full_step(t, g)
        outs += [v.clone() for _, v in sorted(res.items())]
    outs += [eng.decompress_error(i) for i in range(cfg["n_workers"])]
    return outs


@pytest.mark.parametrize("qkind", ["randk", "randblock", "identity"])
@pytest.mark.parametrize("workers,rows,beta", [(1, 5, 0.0), (2, 3, 0.0), (3, 5, 0.5), (4, 7, 0.0), (8, 5, 0.0), (9, 1, 0.25)])
@pytest.mark.parametrize("extra", [[], [(1100, 1000, 1)]])   # below and above the size that interleaves
def test_interleaved_equals_generic(qkind, workers, rows, beta, extra):
    cfg = wl.config("tiny")
    cfg.update(tensors=SMALL + extra, n_workers=workers, q=dict(kind=qkind, k_num=1, k_den=20, seed=5),
               c=dict(kind="countsketch", cs_rows=rows, cs_col_div=10, seed=9, beta=beta))
    for a, b in zip(_run(cfg, True), _run(cfg, False)):
        assert a.shape == b.shape
        if a.numel():
            rms = b.double().square().mean().sqrt().clamp_min(1e-30)
            assert float(((a - b).double().abs() / torch.maximum(b.double().abs(), rms)).max()) < 1e-5


def test_groups_and_a_tensor_beyond_a_group():
    cfg = wl.config("tiny")
    cfg.update(tensors=[(1024, 1024, 1), (7, 3, 1), (1500, 1024, 1), (4000, 2001, 1), (640, 640, 1)], n_workers=8,
               q=dict(kind="randk", k_num=1, k_den=100, seed=5), c=dict(kind="countsketch", cs_rows=3, cs_col_div=5, seed=9))
    for a, b in zip(_run(cfg, True, 2), _run(cfg, False, 2)):
        rms = b.double().square().mean().sqrt().clamp_min(1e-30)
        assert float(((a - b).double().abs() / torch.maximum(b.double().abs(), rms)).max()) < 1e-5
