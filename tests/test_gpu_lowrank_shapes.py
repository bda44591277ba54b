"""Low-rank passes for any shape: widths around a warp, a chunk and eight chunks, tensors thinner than the
rank, odd offsets, every rank, block size and both scale types, with and without beta.  Factors against
the oracle; stored codes and scales teacher-forced, bit for bit.  The order of
the factors' sums is that of the kernels for every codec: free-running steps give the same bits on both."""
import numpy as np
import pytest
import torch

from paper_2312_08538_b200 import workloads as wl
from tests import parity_util as pu

pytestmark = pytest.mark.gpu

EDGES = [(70, 33, 1), (3, 1, 0), (9, 31, 1), (40, 255, 1), (5, 1, 0), (130, 257, 1), (1, 700, 1), (300, 5, 1), (17, 2049, 1),
         (2, 9000, 1), (64, 127, 1)]


@pytest.mark.parametrize("rank,c", [(1, dict(kind="int8", block=256)), (2, dict(kind="int4", block=128, scale_dtype="fp16")),
                                    (3, dict(kind="int8", block=32, scale_dtype="fp16")), (4, dict(kind="int4", block=64)),
                                    (4, dict(kind="int8", block=128, scale_dtype="fp16", beta=0.3)),
                                    (8, dict(kind="int4", block=256, scale_dtype="fp16", beta=0.9)), (8, dict(kind="int8", block=64))])
def test_passes_on_edges(rank, c):
    from paper_2312_08538_b200 import binding as b
    cfg = wl.config("resnet50-mini")
    cfg.update(tensors=EDGES, n_workers=2, q=dict(kind="lowrank", rank=rank), c=c, grad="normal1e-3")
    q0 = wl.q_init(cfg, "cuda")
    eng, o = pu.make_gpu(cfg, q_init=q0), pu.make_oracle(cfg, q_init=q0.cpu().numpy())
    for t in range(2):
        pu.load_state_from_oracle(eng, o)
        gd, gh = pu.grads_both(cfg, t)
        res = o.step(t, gh)
        eng.step(t, gd, 0)
        for l in o.compressed:
            for i in range(o.N):
                assert pu.frob_err(eng.factors(l, i)["p_i"].cpu().numpy(), res[l].P[i]) <= 1e-5, (t, l, "P_i")
        eng.reduce_messages(b.MSG_P)
        for l in o.compressed:
            eng.factors(l, 0)["p_hat"].copy_(torch.from_numpy(res[l].Phat).cuda())
        eng.step(t, gd, 2)
        for l in o.compressed:
            for i in range(o.N):
                f = eng.factors(l, i)["q_i"]
                assert pu.frob_err(f.cpu().numpy(), res[l].Qi[i]) <= 1e-5, (t, l, "Q_i")
                f.copy_(torch.from_numpy(res[l].Qi[i]).cuda())
        eng.step(t, gd, 3)
        for l in o.compressed:
            for i in range(o.N):
                ga, gs = pu.gpu_state_arrays(eng, o, i, l)
                oa, os_ = pu.oracle_state_arrays(o, i, l)
                assert np.array_equal(ga, oa) and np.array_equal(gs, os_), (t, l, i)
        eng.reduce_messages(b.MSG_Q)


@pytest.mark.parametrize("rank,c", [(1, dict(kind="int8", block=256)), (2, dict(kind="int4", block=128, scale_dtype="fp16")),
                                    (3, dict(kind="int8", block=32, scale_dtype="fp16")), (4, dict(kind="int4", block=64, beta=0.3)),
                                    (8, dict(kind="int8", block=128))])
@pytest.mark.parametrize("many", [False, True])   # one row per warp in pass 1, or four
def test_order_of_sums(rank, c, many):
    from paper_2312_08538_b200 import binding as b
    cfg = wl.config("resnet50-mini")
    shapes = EDGES + [(256, 65, 1), (257, 63, 1), (1030, 129, 1)] + ([(30011, 97, 1)] if many else [])
    cfg.update(tensors=shapes, n_workers=2, q=dict(kind="lowrank", rank=rank), c=c, grad="normal1e-3")
    q0 = wl.q_init(cfg, "cuda")
    both = [pu.make_gpu(cfg, q_init=q0, fast=f) for f in (True, False)]
    layers = [l for l, t in enumerate(shapes) if t[2]]
    for t in range(3):
        gd, _ = pu.grads_both(cfg, t)
        for e, f in zip(both, (True, False)):
            e.step(t, gd, 0)
            e.set_fast_path(True)   # (the same Gram-Schmidt)
            e.reduce_messages(b.MSG_P)
            e.set_fast_path(f)
            e.step(t, gd, 1)
        for l in layers:
            for i in range(2):
                x, y = (e.factors(l, i) for e in both)
                for k in ("p_i", "q_i"):
                    assert torch.equal(x[k], y[k]), (t, l, i, k)
        for e in both:
            e.reduce_messages(b.MSG_Q)


# what tall models take beside it: rows of one word per lane and more, tiles of 32, 64 and 128 columns on and off whole words, chunks
# of pass 3 that hold one, two and many rows, and row counts around a stage and a tile
BIG = [(60011, 97, 1), (3, 1, 0), (1001, 57, 1), (1003, 58, 1), (1005, 25, 1), (257, 26, 1), (255, 121, 1), (256, 122, 1), (273, 128, 1),
       (271, 136, 1), (77, 511, 1), (5, 1, 0), (33, 512, 1), (65, 513, 1), (19, 1023, 1), (15, 2000, 1), (1, 999, 1), (2, 130, 1)]


@pytest.mark.parametrize("rank,c", [(1, dict(kind="int4", block=64)), (2, dict(kind="int8", block=32, scale_dtype="fp16")),
                                    (3, dict(kind="int4", block=128, scale_dtype="fp16")), (4, dict(kind="int8", block=256, beta=0.3)),
                                    (8, dict(kind="int4", block=256, scale_dtype="fp16")), (8, dict(kind="int8", block=128, scale_dtype="fp16", beta=0.9))])
def test_tall_models_give_the_bits_of_the_kernels_for_every_codec(rank, c):
    from paper_2312_08538_b200 import binding as b
    cfg = wl.config("resnet50-mini")
    cfg.update(tensors=BIG, n_workers=2, q=dict(kind="lowrank", rank=rank), c=c, grad="normal1e-3")
    q0 = wl.q_init(cfg, "cuda")
    both = [pu.make_gpu(cfg, q_init=q0, fast=f) for f in (True, False)]
    # the second gradient buffer is off every vector alignment
    room = torch.empty(sum(r * k for r, k, _ in BIG) + 1, device="cuda")
    for t in range(3):
        gd, _ = pu.grads_both(cfg, t)
        room[1:].copy_(gd[1])
        gd = [gd[0], room[1:]]
        for e, f in zip(both, (True, False)):
            e.step(t, gd, 0)
            e.set_fast_path(True)   # (the same Gram-Schmidt)
            e.reduce_messages(b.MSG_P)
            e.set_fast_path(f)
            e.step(t, gd, 1)
        for l in [l for l, x in enumerate(BIG) if x[2]]:
            for i in range(2):
                x, y = (e.factors(l, i) for e in both)
                for k in ("p_i", "q_i"):
                    assert torch.equal(x[k], y[k]), (t, l, i, k)
        for i in range(2):
            x, y = (e.decompress_error(i) for e in both)
            assert torch.equal(x, y), (t, i)
        for e in both:
            e.reduce_messages(b.MSG_Q)


@pytest.mark.parametrize("tensors", [[(1, 97, 1)] + BIG, [(1, 97, 1), (70, 33, 1), (3, 1, 0), (2, 61, 1), (300, 257, 1), (64, 512, 1)]])
@pytest.mark.parametrize("rank,c", [(2, dict(kind="int8", block=256)), (2, dict(kind="int4", block=64, beta=0.5)), (3, dict(kind="int8", block=64, scale_dtype="fp16")),
                                    (4, dict(kind="int4", block=128, scale_dtype="fp16")), (5, dict(kind="int8", block=256)), (6, dict(kind="int4", block=256)),
                                    (7, dict(kind="int8", block=32, beta=0.9)), (8, dict(kind="int4", block=128, scale_dtype="fp16"))])
def test_ranks_without_kernels_of_their_own(monkeypatch, tensors, rank, c):
    """Ranks between those that the kernels are made for, and factors off their vectors' boundaries behind a tensor of one row."""
    monkeypatch.setitem(globals(), "BIG", tensors)
    test_tall_models_give_the_bits_of_the_kernels_for_every_codec(rank, c)


@pytest.mark.parametrize("rank,c", [(4, dict(kind="int8", block=256)), (8, dict(kind="int4", block=128, scale_dtype="fp16")),
                                    (4, dict(kind="int4", block=64, scale_dtype="fp16", beta=0.9)), (8, dict(kind="int8", block=32, scale_dtype="fp16"))])
def test_all_widths_in_one_launch(rank, c):
    """One launch per pass over narrow, middling and wide matrices (tiles that share a CTA, with a remainder), 1-D
    tensors, and shapes that only the passes for any shape take; more tiles of a factor's sum than are added singly."""
    cfg = wl.config("resnet50-mini")
    cfg.update(tensors=[(41, 32, 1), (64, 1, 0), (33, 96, 1), (130, 256, 1), (2065, 320, 1), (21, 576, 1), (11, 1152, 1), (70, 147, 1),
                        (2100, 1, 0), (301, 2048, 1), (3, 4608, 1), (8500, 37, 1)],
               n_workers=2, q=dict(kind="lowrank", rank=rank), c=c, grad="normal1e-3")
    from tests.test_gpu_parity import lowrank_teacher_forced
    lowrank_teacher_forced(cfg, 2, fast=True, scale_with_cond=True)


@pytest.mark.parametrize("c", [dict(kind="int8", block=256), dict(kind="int4", block=64, scale_dtype="fp16", beta=0.9)])
def test_many_elements_of_other_shapes_beside_a_tuned_matrix(c):
    """Up to 18 M elements at rank 8 they share its launches, beyond that each pass has one of their own: three more
    launches, the same bits."""
    from paper_2312_08538_b200 import binding as b
    launches = []
    for rows in (2252, 2254):   # 18 M elements of eight workers between them
        cfg = wl.config("resnet50-mini")
        cfg.update(tensors=[(512, 256, 1), (77, 1, 0), (rows, 999, 1)], n_workers=8, q=dict(kind="lowrank", rank=8), c=c, grad="normal1e-3")
        q0 = wl.q_init(cfg, "cuda")
        both = [pu.make_gpu(cfg, q_init=q0, fast=f) for f in (True, False)]
        for t in range(2):
            gd, _ = pu.grads_both(cfg, t)
            for e, f in zip(both, (True, False)):
                before = e.launch_count()
                e.step(t, gd, 0)
                e.set_fast_path(True)   # (the same Gram-Schmidt)
                e.reduce_messages(b.MSG_P)
                e.set_fast_path(f)
                e.step(t, gd, 2)
                e.step(t, gd, 3)
                if f and t == 1:
                    launches.append(e.launch_count() - before)
            dense = [e.reduce_messages(b.MSG_DENSE1D) for e in both]
            assert torch.equal(*dense)
            for i in range(8):
                x, y = (e.factors(2, i) for e in both)
                for k in ("p_i", "q_i"):
                    assert torch.equal(x[k], y[k]), (rows, t, i, k)
                u, v = (e.decompress_error(i)[512 * 256:] for e in both)
                assert torch.equal(u, v), (rows, t, i)
            for e in both:
                e.reduce_messages(b.MSG_Q)
    assert launches[1] == launches[0] + 3
