"""A residual that is not a number leaves the other codes of its quantisation block, and the block's scale, as they are
without it.  The kernels for every codec are the reference."""
import numpy as np
import pytest
import torch

from paper_2312_08538_b200 import workloads as wl
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

ODD = [(70, 33, 1), (3, 1, 0), (9, 31, 1), (130, 257, 1), (1, 700, 1), (300, 5, 1), (17, 2049, 1)]


def _lowrank(tensors, rank, c, last=3):
    """Steps whose Q_i has a NaN in two of its columns' rows: both columns of the residual are NaN throughout."""
    from paper_2312_08538_b200 import binding as b
    cfg = wl.config("resnet50-mini")
    cfg.update(tensors=tensors, n_workers=2, q=dict(kind="lowrank", rank=rank), c=c, grad="normal1e-3")
    q0 = wl.q_init(cfg, "cuda")
    eng, ref = (pu.make_gpu(cfg, q_init=q0, fast=f) for f in (True, False))
    eng.set_fused(last == 4)
    layers = [l for l, t in enumerate(tensors) if t[2]]
    gd, _ = pu.grads_both(cfg, 0)
    for e in (eng, ref):
        e.step(0, gd, 0)
        e.reduce_messages(b.MSG_P)
    for l in layers:
        eng.factors(l, 0)["p_hat"].copy_(ref.factors(l, 0)["p_hat"])
    for e in (eng, ref):
        e.step(0, gd, 2)
    bad = {l: [0, 2 * tensors[l][1] // 3] for l in layers}
    for l in layers:
        for i in range(2):
            q = ref.factors(l, i)["q_i"]
            q[bad[l]] = float("nan")
            eng.factors(l, i)["q_i"].copy_(q)
    eng.step(0, gd, last)
    ref.step(0, gd, 3)
    o = pu.make_oracle(cfg, q_init=q0.cpu().numpy())
    for l in layers:
        keep = np.ones((tensors[l][0], tensors[l][1]), bool)
        keep[:, bad[l]] = False
        for i in range(2):
            (ca, sa), (cb, sb) = (pu.gpu_state_arrays(e, o, i, l) for e in (eng, ref))
            assert np.isfinite(sa).all() and np.array_equal(sa, sb), (l, i)
            assert np.array_equal(ca[keep.ravel()], cb[keep.ravel()]), (l, i)


@pytest.mark.parametrize("rank,c", [(2, dict(kind="int4", block=64, scale_dtype="fp16")), (3, dict(kind="int8", block=32)),
                                    (4, dict(kind="int4", block=256)), (8, dict(kind="int8", block=128, scale_dtype="fp16", beta=0.5))])
@pytest.mark.parametrize("more", [[], [(2000, 1001, 1)]])   # (eight and sixteen elements per lane)
def test_lowrank_passes_for_any_shape(rank, c, more):
    _lowrank(ODD + more, rank, c)


ALIGNED = [(64, 512, 1), (8, 1, 0), (40, 768, 1), (128, 64, 1), (33, 1024, 1)]


@pytest.mark.parametrize("rank,c", [(4, dict(kind="int4", block=128, scale_dtype="fp16")), (4, dict(kind="int8", block=256)),
                                    (8, dict(kind="int4", block=128, scale_dtype="fp16")), (8, dict(kind="int8", block=32, scale_dtype="fp16", beta=0.5))])
@pytest.mark.parametrize("more", [[], [(20000, 1536, 1)]])   # one launch per pass, and one per CTA size
def test_tuned_lowrank_passes(rank, c, more):
    _lowrank(ALIGNED + more, rank, c)


@pytest.mark.parametrize("rank,c", [(4, dict(kind="int4", block=128, scale_dtype="fp16")), (8, dict(kind="int8", block=256))])
def test_fused_lowrank_passes(rank, c):
    """Its residual is formed with the Q_i found in the message buffer (phase 4)."""
    _lowrank([(64, 512, 1), (40, 768, 1), (4099, 1600, 1)], rank, c, last=4)


@pytest.mark.parametrize("c", [dict(kind="int4", block=64, scale_dtype="fp16"), dict(kind="int8", block=256)])
@pytest.mark.parametrize("iconef", [0, 1, 2])
def test_single_phase_steps(c, iconef):
    """A gradient element that is NaN: its residual alone is."""
    cfg = wl.config("tiny")
    cfg.update(tensors=[(64, 512, 1), (8, 1, 0), (33, 1024, 1)], n_workers=2, q=dict(kind="randk", k_num=1, k_den=1000, seed=4), c=dict(c, iconef=iconef))
    eng, ref = (pu.make_gpu(cfg, fast=f) for f in (True, False))
    bad = torch.arange(5, 64 * 512, 1001, device="cuda")
    gd, _ = pu.grads_both(cfg, 0)
    for g in gd:
        g[bad] = float("nan")
    for e in (eng, ref):
        e.full_step(0, gd)
    o = pu.make_oracle(cfg)
    keep = np.ones(64 * 512, bool)
    keep[bad.cpu().numpy()] = False
    for second in ((False, True) if iconef == 1 else (False,)):
        for i in range(2):
            (ca, sa), (cb, sb) = (pu.gpu_state_arrays(e, o, i, 0, second) for e in (eng, ref))
            assert np.isfinite(sa).all() and np.array_equal(sa, sb), (i, second)
            assert np.array_equal(ca[keep], cb[keep]), (i, second)
