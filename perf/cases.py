"""What is timed: the calls a training job makes of this library, over the range of jobs it serves.

A pass of a "step" case is one iteration as a data-parallel job runs it: every worker's gradient is
compressed with error feedback (``full_step``: all phases and reductions) and the mean message is
applied to the parameters (``apply_update``).  "decode" is the stored error of every worker expanded
to fp32 (error norms, checkpoints for another compressor).  "indices" is the receiving side of a
random-k message, which recomputes the shared index sets without a context.

A case names its parameter list either by a configuration of ``workloads`` or as shapes,
"rows x cols" separated by commas (a length alone is a 1-D tensor, which passes through uncompressed).
"""
import math

import torch

from paper_2312_08538_b200 import binding as cb
from paper_2312_08538_b200 import workloads as wl

_STEP = dict(task="step", workers=1, q="randk", rank=0, k_den=100, c="int8", block=256, scale="fp32", beta=0.0,
             iconef=0, cs_rows=0, cs_div=10, grad="normal", lr=0.1)


def _case(**kw):
    return dict(_STEP, **kw)


def listed():
    return [
        # one small layer on two workers: launches and host time are all there is
        _case(name="tiny-randk-int8", tensors="256x512", workers=2),
        # image classification, PowerSGD-style compressor: 54 convolutions of very different sizes
        _case(name="resnet50-rank4-int8", tensors="resnet50", workers=4, q="lowrank", rank=4, grad="layerscaled"),
        # language model of ordinary size at the highest rank, small error state
        _case(name="gpt2-small-rank8-int4", tensors="gpt2-small", workers=4, q="lowrank", rank=8, c="int4", block=128,
              scale="fp16", grad="student", lr=0.05),
        # the largest model: 1.6 billion parameters, two workers' gradients on this GPU
        _case(name="gpt2-xl-rank4-int4", tensors="gpt2-xl", workers=2, q="lowrank", rank=4, c="int4", block=128,
              scale="fp16", grad="student", lr=0.05),
        # translation model with the count sketch as error compressor, eight workers
        _case(name="transformer-big-countsketch", tensors="transformer-big", workers=8, c="countsketch", cs_rows=5),
        # the same model as a distributed job runs it, one worker per GPU, int8 error state
        _case(name="transformer-big-int8-1worker", tensors="transformer-big"),
        # low-rank gradients on a row sketch in binary16 with partial error feedback
        _case(name="gpt2-small-rank4-rowsketch", tensors="gpt2-small", q="lowrank", rank=4, c="rowsketch", scale="fp16",
              beta=0.9, cs_rows=1, grad="student", lr=0.05),
        # layer sizes that are multiples of nothing (a recurrent model with an odd vocabulary): rank 2
        _case(name="ragged-rank2-int4", tensors="33279x650,2600x650,2600,2600x650,2600,2600x650,2600,2601x651,2601,33279",
              workers=2, q="lowrank", rank=2, c="int4", block=128, scale="fp16", grad="student"),
        # classical error feedback: dense fp32 error, one contiguous random block is sent
        _case(name="resnet50-randblock-dense", tensors="resnet50", workers=4, q="randblock", k_den=10, c="identity",
              grad="layerscaled"),
        # the improved error feedback with two int8 states, on layers behind an odd-sized one
        _case(name="iconef1-odd-int8", tensors="33x1021,33,4096x1024,4096,1024x4096,1024,1024x1024,1024,4097x1024",
              workers=4, iconef=1),
        # expanding the stored int4 error of two workers
        _case(name="decode-transformer-big-int4", task="decode", tensors="transformer-big", workers=2, c="int4",
              block=128, scale="fp16"),
        # the receiver of random-k messages of an image model: one index set per convolution
        _case(name="indices-resnet50", task="indices", tensors="resnet50"),
    ]


# ------------------------------------------------------------------ further cases of the same ranges

def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _shapes(rng, total, most):
    n = rng.randint(1, 12)
    aligned = rng.random() < 0.5   # model widths are multiples of 64 in one half of the jobs, anything in the other
    out = []
    for _ in range(n):
        d = min(most, max(64.0, total / n * rng.uniform(0.4, 1.6)))
        cols = max(2, int(math.sqrt(d * _log_uniform(rng, 0.125, 8.0))))
        if aligned:
            cols = max(64, cols // 64 * 64)
        rows = max(1, int(d / cols))
        out.append("%dx%d" % (rows, cols))
        if rng.random() < 0.7:
            out.append("%d" % cols)
    return ",".join(out)


def draw(rng):
    kind = rng.choice(["flat", "flat", "lowrank", "lowrank", "sketch", "rowsketch", "decode", "indices"])
    workers = rng.choice([1, 2, 4, 8])
    steps = _log_uniform(rng, 1 << 15, 1 << 29)   # elements over all workers
    if kind == "indices":
        return _case(task="indices", tensors=_shapes(rng, min(steps, 1 << 27), 1 << 24), k_den=rng.choice([10, 50, 100, 1000]))
    quant = rng.choice([dict(c="int8", block=256, scale="fp32"), dict(c="int4", block=128, scale="fp16"),
                        dict(c="int8", block=128, scale="fp16"), dict(c="int4", block=64, scale="fp32")])
    kw = dict(tensors=_shapes(rng, steps / workers, 1 << 30), workers=workers, grad=rng.choice(["normal", "student"]))
    sparse = dict(q=rng.choice(["randk", "randk", "randblock"]), k_den=rng.choice([10, 50, 100, 1000]))
    if kind == "flat":
        if rng.random() < 0.25:
            return _case(**kw, **sparse, c="identity")
        return _case(**kw, **sparse, **quant, iconef=rng.choice([0, 0, 1]))
    if kind == "lowrank":
        return _case(**kw, **quant, q="lowrank", rank=rng.choice([1, 2, 4, 4, 8]))
    if kind == "sketch":
        return _case(**kw, **sparse, c="countsketch", cs_rows=rng.choice([3, 5]), cs_div=rng.choice([5, 10, 20]))
    if kind == "rowsketch":
        low = dict(q="lowrank", rank=rng.choice([2, 4]))
        return _case(**kw, **rng.choice([low, sparse]), c="rowsketch", scale=rng.choice(["fp16", "fp32"]), beta=0.9,
                     cs_rows=1, cs_div=rng.choice([5, 10]))
    return _case(**kw, **sparse, **quant, task="decode")


# ------------------------------------------------------------------ inputs

def _tensors(case):
    text = case["tensors"]
    if text[0].isalpha():
        return wl.config(text)["tensors"]
    out = []
    for item in text.split(","):
        rows, _, cols = item.partition("x")
        out.append((int(rows), int(cols or 1), 1 if cols else 0))
    return out


def _compressed(tensors):
    return [l for l, (r, c, k) in enumerate(tensors) if k and c > 1]


def _gradient(case, tensors, gen, out):
    """Gradients around 1e-3: normal, heavy-tailed (Student-t, 3 degrees of freedom), or with a scale per tensor."""
    chunk = 1 << 26
    for lo in range(0, out.numel(), chunk):
        part = out[lo:lo + chunk]
        part.normal_(generator=gen)
        if case["grad"] == "student":
            chi = torch.zeros_like(part)
            for _ in range(3):
                chi += torch.empty_like(part).normal_(generator=gen).square_()
            part /= chi.div_(3.0).sqrt_()
        part *= 1e-3
    if case["grad"] == "layerscaled":
        scales = torch.rand(len(tensors), generator=gen, device=out.device).mul_(2.0).sub_(1.0).tolist()
        off = 0
        for (r, c, _), s in zip(tensors, scales):
            out[off:off + r * c] *= 10.0 ** s
            off += r * c


def _stored_error(ctx, worker):
    """The stored error of one worker, all tensors: the bytes of the workspace from its first state to its last."""
    which = _compressed(ctx.tensors)
    first = ctx.state(worker, which[0])[0]
    ends = [v for v in ctx.state(worker, which[-1]) if v is not None]
    if ctx.c["iconef"] == 1:
        ends += [v for v in ctx.state(worker, which[-1], second=True) if v is not None]
    base = ctx.workspace.data_ptr()
    span = ctx.workspace[first.data_ptr() - base:max(v.data_ptr() + v.numel() for v in ends) - base]
    if ctx.c["kind"] in ("identity", "countsketch"):
        return span.view(torch.float32)
    if ctx.c["kind"] == "rowsketch":
        return span.view(torch.float16 if ctx.c["scale_dtype"] == "fp16" else torch.float32)
    return span


def prepare(case, seed):
    tensors = _tensors(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["task"] == "indices":
        sizes = [(l, tensors[l][0] * tensors[l][1]) for l in _compressed(tensors)]
        sets = [(l, d, max(1, d // case["k_den"])) for l, d in sizes]
        return dict(case=case, seed=seed, t=0, sets=sets,
                    out=[torch.empty(k, dtype=torch.int32, device="cuda") for _, _, k in sets])
    q = dict(kind=case["q"], rank=case["rank"], k_num=1, k_den=case["k_den"], seed=seed + 13)
    c = dict(kind=case["c"], block=case["block"], scale_dtype=case["scale"], cs_rows=case["cs_rows"] or 5,
             cs_col_div=case["cs_div"], seed=seed + 17, beta=case["beta"], iconef=case["iconef"])
    q_init = None
    if case["q"] == "lowrank":
        q_init = torch.randn(sum(tensors[l][1] * min(case["rank"], *tensors[l][:2]) for l in _compressed(tensors)),
                             generator=gen, device="cuda")
    ctx = cb.ConEF(tensors, case["workers"], q, c, case["lr"], q_init=q_init)
    total = sum(r * k for r, k, _ in tensors)
    grads = [torch.empty(total, device="cuda") for _ in range(case["workers"])]
    which = (cb.MSG_P, cb.MSG_Q) if case["q"] == "lowrank" else (cb.MSG_VALUES,)
    sums = {m: torch.empty(ctx.message_elems(m), device="cuda") for m in which + (cb.MSG_DENSE1D,)}
    # a job in mid-training: the workers' stored errors are those of an earlier iteration
    for g in grads:
        _gradient(case, tensors, gen, g)
    ctx.full_step(0, grads, sums)
    state = dict(case=case, ctx=ctx, t=1, sums=sums, grads=grads)
    if case["task"] == "decode":
        del state["grads"]
        state["out"] = [torch.empty(ctx.error_elems(), device="cuda") for _ in range(case["workers"])]
        return state
    for g in grads:
        _gradient(case, tensors, gen, g)
    state["x"] = torch.randn(total, generator=gen, device="cuda").mul_(0.02)
    if case["c"] not in ("countsketch", "rowsketch"):   # (a sketch is written to another buffer in every step)
        state["errors"] = [_stored_error(ctx, i) for i in range(case["workers"])]
    return state


def run(state):
    case = state["case"]
    t = state["t"]
    state["t"] = t + 1
    if case["task"] == "indices":
        for (tensor, d, k), out in zip(state["sets"], state["out"]):
            cb.conef_randk_indices_noalloc(state["seed"], tensor, t, d, k, out)
        return state["out"]
    ctx = state["ctx"]
    if case["task"] == "decode":
        for i, out in enumerate(state["out"]):
            ctx.decompress_error(i, out)
        return state["out"]
    sums = ctx.full_step(t, state["grads"], state["sums"])
    ctx.apply_update(state["x"], sums)
    errors = state.get("errors") or [_stored_error(ctx, i) for i in range(case["workers"])]
    return dict(parameters=state["x"], messages=[sums[m] for m in sorted(sums)], errors=errors)


# ------------------------------------------------------------------ what a pass cannot do without

def _state_bytes(case, rows, cols):
    d = rows * cols
    if case["c"] == "identity":
        return 4 * d
    if case["c"] == "countsketch":
        return 4 * case["cs_rows"] * max(1, d // case["cs_div"])
    if case["c"] == "rowsketch":
        return (2 if case["scale"] == "fp16" else 4) * case["cs_rows"] * max(1, rows // case["cs_div"]) * cols
    code = d if case["c"] == "int8" else (d + 1) // 2
    return (code + (2 if case["scale"] == "fp16" else 4) * -(-d // case["block"])) * (2 if case["iconef"] == 1 else 1)


def work(case):
    tensors = _tensors(case)
    n = case["workers"]
    nbytes = flops = 0
    for r, c, k in tensors:
        d = r * c
        if not (k and c > 1):
            if case["task"] == "step":   # gradients in, the sum out, the parameters updated
                nbytes += 4 * n * d + 4 * d + 8 * d
                flops += 2 * n * d
            continue
        kept = max(1, d // case["k_den"])
        if case["task"] == "indices":
            nbytes += 4 * kept
            continue
        state = _state_bytes(case, r, c)
        if case["task"] == "decode":
            nbytes += n * (state + 4 * d)
            flops += n * d
            continue
        nbytes += n * (4 * d + 2 * state)
        flops += 4 * n * d
        if case["q"] == "lowrank":
            rank = min(case["rank"], r, c)
            nbytes += 8 * d + 4 * (r + c) * rank       # dense update of the parameters, the summed factors
            flops += (6 * n + 2) * rank * d            # two products and the residual per worker, the update
        else:
            nbytes += (8 + 4 + 4) * kept               # parameters, sums and indices of the kept coordinates
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    if case["task"] == "indices":
        return "exact"
    if case["c"] == "countsketch":
        # fp32 bucket sums in any order (decode reads the sketch of the step before)
        return dict(rel=1e-5)
    if case["q"] == "lowrank":
        # fp32 sums over up to 50 257 terms in any order; a stored code or a binary16 entry next to a
        # rounding boundary may land on the other side
        return dict(rel=1e-3 if case["c"] == "rowsketch" and case["scale"] == "fp16" else 1e-4, max=5e-3, differ=5e-3)
    # elementwise fp32 operations in a fixed order, integer codes
    return "exact"
