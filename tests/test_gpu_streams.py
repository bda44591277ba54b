"""Calls on a stream of their own, behind an event of another stream and in a captured graph: a kernel may come onto the
SMs before the one ahead of it in the stream has ended, but not before what an event holds the stream back for."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(300, 128, 1), (77, 1, 0), (1000, 512, 1), (64, 147, 1), (2, 1, 0), (3000, 256, 1), (40, 1152, 1), (700, 33, 1)]
JOBS = {
    "randk-int8": (dict(kind="randk", k_num=1, k_den=50, seed=3), dict(kind="int8", block=256)),
    "randk-large": (dict(kind="randk", k_num=1, k_den=50, seed=3), dict(kind="int4", block=128, scale_dtype="fp16", iconef=1)),
    "randblock-dense": (dict(kind="randblock", k_num=1, k_den=10, seed=3), dict(kind="identity")),
    "rank4-int4": (dict(kind="lowrank", rank=4), dict(kind="int4", block=128, scale_dtype="fp16")),
    "rank2-int8": (dict(kind="lowrank", rank=2), dict(kind="int8", block=256)),
    "rank4-rowsketch": (dict(kind="lowrank", rank=4), dict(kind="rowsketch", cs_rows=1, cs_col_div=10, beta=0.9, seed=5)),
}


class Job:
    def __init__(self, name, seed=1):
        from paper_2312_08538_b200 import binding as b
        self.b, (q, c) = b, JOBS[name]
        shapes = SHAPES + ([(2100, 1024, 1)] if name == "randk-large" else [])   # (not selected by clusters)
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.total = sum(r * k for r, k, _ in shapes)
        q0 = None
        if q["kind"] == "lowrank":
            q0 = torch.randn(sum(k * min(q["rank"], r, k) for r, k, z in shapes if z and k > 1), generator=self.gen, device="cuda")
        self.eng = b.ConEF(shapes, 2, q, c, 0.1, q_init=q0)
        self.x = torch.randn(self.total, generator=self.gen, device="cuda")
        self.src = [[torch.randn(self.total, generator=self.gen, device="cuda") * 1e-3 for _ in range(2)] for _ in range(4)]
        self.grads = [torch.zeros(self.total, device="cuda") for _ in range(2)]
        which = (b.MSG_P, b.MSG_Q) if q["kind"] == "lowrank" else (b.MSG_VALUES,)
        self.sums = {m: torch.zeros(self.eng.message_elems(m), device="cuda") for m in which + (b.MSG_DENSE1D,)}
        self.err = [torch.zeros(self.eng.error_elems(), device="cuda") for _ in range(2)]

    def load(self, t):
        for g, s in zip(self.grads, self.src[t]):
            g.copy_(s)

    def step(self, t):
        self.eng.full_step(t, self.grads, self.sums)
        self.eng.apply_update(self.x, self.sums)
        for i, e in enumerate(self.err):
            self.eng.decompress_error(i, e)

    def results(self):
        torch.cuda.synchronize()
        return [self.x.clone()] + [s.clone() for s in self.sums.values()] + [e.clone() for e in self.err]


def _synchronised(name, steps):
    job, out = Job(name), []
    for t in range(steps):
        job.load(t)
        torch.cuda.synchronize()
        job.step(t)
        out.append(job.results())
    return out


def _busy(a, n=6):
    for _ in range(n):   # (some milliseconds of work)
        a = a @ a * 1e-4
    return a


@pytest.mark.parametrize("name", sorted(JOBS))
def test_a_step_behind_an_event_of_another_stream(name):
    """The gradients are written late on another stream; the step's own stream has a finished kernel ahead of the wait."""
    want = _synchronised(name, 3)
    job = Job(name)
    ours, other = torch.cuda.Stream(), torch.cuda.Stream()
    a = torch.randn(6144, 6144, device="cuda")
    torch.cuda.synchronize()
    for t in range(3):
        done, ready = torch.cuda.Event(), torch.cuda.Event()
        done.record(ours)
        with torch.cuda.stream(other):
            other.wait_event(done)
            for g in job.grads:
                g.zero_()
            a = _busy(a)
            job.load(t)
            ready.record(other)
        ours.wait_event(ready)
        with torch.cuda.stream(ours):
            job.step(t)
        for x, y in zip(job.results(), want[t]):
            assert torch.equal(x, y), t


@pytest.mark.parametrize("name", sorted(JOBS))
def test_steps_in_a_captured_graph(name):
    """Two steps behind an event in one graph; replayed once they leave what two steps leave."""
    want = _synchronised(name, 3)
    job = Job(name)
    job.load(0)
    job.step(0)   # (what is loaded and set up on a first call is not captured)
    job.results()
    graph, ours, other = torch.cuda.CUDAGraph(), torch.cuda.Stream(), torch.cuda.Stream()
    a = torch.randn(6144, 6144, device="cuda")
    with torch.cuda.stream(other):
        _busy(a, 1)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=ours):
        for t in (1, 2):
            other.wait_stream(ours)
            with torch.cuda.stream(other):
                _busy(a, 2)
                job.load(t)
            ours.wait_stream(other)
            job.step(t)
    graph.replay()
    for x, y in zip(job.results(), want[2]):
        assert torch.equal(x, y)


def test_decode_right_behind_the_side_streams():
    """Passes of matrices of several widths run on side streams; the stored error is expanded next, without a
    reduction in between.  (Long tiles, so that each width has a launch of its own: 99 M elements, eight workers.)"""
    from paper_2312_08538_b200 import binding as b
    shapes = [(20000, 1600, 1), (32768, 1024, 1), (43690, 768, 1)]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    total = sum(r * c for r, c, _ in shapes)
    q0 = torch.randn(sum(c for _, c, _ in shapes) * 4, generator=gen, device="cuda")
    eng = b.ConEF(shapes, 8, dict(kind="lowrank", rank=4), dict(kind="int4", block=64, scale_dtype="fp16"), 0.1, q_init=q0)
    grads = [torch.randn(total, generator=gen, device="cuda") for _ in range(8)]
    out = [torch.empty(total, device="cuda") for _ in range(2)]
    for t in range(2):
        eng.step(t, grads, 0)
        eng.reduce_messages(b.MSG_P)
        eng.step(t, grads, 1)
        for i, o in zip((0, 7), out):
            eng.decompress_error(i, o)
        torch.cuda.synchronize()
        for i, o in zip((0, 7), out):
            assert torch.equal(o, eng.decompress_error(i)), (t, i)
        assert out[0].abs().max() > 0
        eng.reduce_messages(b.MSG_Q)
