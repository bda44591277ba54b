"""The count-sketch step with the workers' sketches interleaved: one to sixteen workers, one to seven sketch
rows, several groups of tensors, a tensor too large for a group, one that holds most of the model (whose
new sketch is built in the place of the old one), against the generic kernel (sums of bucket entries
in another order) and against the oracle."""
import pytest
import torch

from paper_2312_08538_b200 import workloads as wl
from tests import parity_util as pu
from tests.test_gpu_parity import run_single_phase

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
@pytest.mark.parametrize("workers,rows,beta", [(1, 5, 0.0), (2, 3, 0.0), (3, 5, 0.5), (4, 7, 0.0), (7, 3, 0.0), (8, 5, 0.0), (9, 1, 0.25), (16, 3, 0.0)])
@pytest.mark.parametrize("extra", [[], [(1100, 1000, 1)]])   # below and, from two workers on, above the size that interleaves
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


@pytest.mark.parametrize("workers", [2, 3, 4, 9])
def test_a_tensor_beyond_the_l2_that_is_the_model(workers):
    """Half of its records among the states: 5 x 1332371 of them, an odd number."""
    cfg = wl.config("tiny")
    cfg.update(tensors=[(7, 1, 0), (3, 4441238, 1)], n_workers=workers, q=dict(kind="randk", k_num=1, k_den=100, seed=5),
               c=dict(kind="countsketch", cs_rows=5, cs_col_div=10, seed=9, beta=0.5))
    for a, b in zip(_run(cfg, True, 2), _run(cfg, False, 2)):
        rms = b.double().square().mean().sqrt().clamp_min(1e-30)
        assert float(((a - b).double().abs() / torch.maximum(b.double().abs(), rms)).max()) < 1e-5


@pytest.mark.parametrize("qkind", ["randk", "randblock", "identity"])
@pytest.mark.parametrize("workers,rows", [(8, 701), (7, 1021), (3, 1401), (2, 2801)])
def test_reading_and_adding_in_two_walks(qkind, workers, rows):
    """Tensors whose old values fit L2 and whose old and new ones do not, in a model with room for r between the walks."""
    cfg = wl.config("tiny")
    cfg.update(tensors=[(rows, 1001, 1), (7, 1, 0), (rows, 999, 1), (rows + 3, 1000, 1), (rows, 1003, 1)], n_workers=workers,
               q=dict(kind=qkind, k_num=1, k_den=20, seed=5), c=dict(kind="countsketch", cs_rows=5, cs_col_div=2, seed=9, beta=0.5))
    for a, b in zip(_run(cfg, True, 2), _run(cfg, False, 2)):
        rms = b.double().square().mean().sqrt().clamp_min(1e-30)
        assert float(((a - b).double().abs() / torch.maximum(b.double().abs(), rms)).max()) < 1e-5


@pytest.mark.parametrize("qkind", ["randk", "identity"])
@pytest.mark.parametrize("workers,sketch_rows,rows", [(8, 3, 1201), (9, 3, 701), (16, 3, 701), (9, 7, 301), (16, 1, 1701), (9, 5, 421)])
def test_two_walks_over_other_sketches_and_batches_of_workers(qkind, workers, sketch_rows, rows):
    """Three rows, five and the general form, one and two batches of eight workers (the last one not full)."""
    cfg = wl.config("tiny")
    cfg.update(tensors=[(rows, 1001, 1), (rows, 999, 1), (rows + 3, 1000, 1), (rows, 1003, 1), (rows + 1, 1002, 1)], n_workers=workers,
               q=dict(kind=qkind, k_num=1, k_den=20, seed=5),
               c=dict(kind="countsketch", cs_rows=sketch_rows, cs_col_div=2, seed=9, beta=0.5))
    if qkind == "identity":   # interleaving, reading, adding, back: four launches per tensor (three in one walk)
        eng = pu.make_gpu(cfg)
        before = eng.launch_count()
        eng.step(0, [wl.gradient(cfg, i, 0, device="cuda") for i in range(workers)], 0)
        assert eng.launch_count() - before == 4 * len(cfg["tensors"])
    for a, b in zip(_run(cfg, True, 2), _run(cfg, False, 2)):
        rms = b.double().square().mean().sqrt().clamp_min(1e-30)
        assert float(((a - b).double().abs() / torch.maximum(b.double().abs(), rms)).max()) < 1e-5


# three tensors of a similar size, which fit the scratch with their new records, and one that does not
@pytest.mark.parametrize("tensors", [[(600, 1000, 1), (300, 1, 0), (601, 1000, 1), (599, 1001, 1)], [(37, 53, 1), (1100, 1001, 1), (64, 1, 0)]])
@pytest.mark.parametrize("qkind,workers,rows", [("randk", 2, 5), ("randblock", 3, 3), ("randk", 8, 5), ("identity", 9, 7)])
def test_interleaved_equals_the_oracle(tensors, qkind, workers, rows):
    cfg = wl.config("tiny")
    cfg.update(tensors=tensors, n_workers=workers, q=dict(kind=qkind, k_num=1, k_den=20, seed=5),
               c=dict(kind="countsketch", cs_rows=rows, cs_col_div=10, seed=9))
    run_single_phase(cfg, 2, exact_values=False)


def test_kernel_choice_changes_between_steps():
    """The step on interleaved workers leaves its result where the old sketch was, the others in the second buffer."""
    cfg = wl.config("tiny")
    cfg.update(tensors=[(1100, 1000, 1), (37, 53, 1)], n_workers=4, q=dict(kind="randk", k_num=1, k_den=20, seed=5),
               c=dict(kind="countsketch", cs_rows=3, cs_col_div=10, seed=9))
    eng, ref = pu.make_gpu(cfg), pu.make_gpu(cfg, fast=False)
    for t in range(5):
        eng.set_fast_path(t % 3 != 1)
        g = [wl.gradient(cfg, i, t, device="cuda") for i in range(4)]
        eng.full_step(t, g)
        ref.full_step(t, g)
    for i in range(4):
        a, b = eng.decompress_error(i), ref.decompress_error(i)
        assert float((a - b).double().norm() / b.double().norm()) < 1e-5
        for l in range(2):
            # a bucket sums about ten residuals, each with the rounding of the buckets it was estimated from: in five
            # steps 2^-24 sqrt(10)^5
            a, b = (e.state(i, l)[0].view(torch.float32).double() for e in (eng, ref))
            assert float((a - b).norm() / b.norm()) < 2e-5
