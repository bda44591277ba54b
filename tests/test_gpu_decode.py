"""The stored error expanded to fp32 at the edges of the decode tiles (1024 elements, 4096 in large models; output on and
off 16-byte boundaries), against the codes and scales read back from the state."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(64, 64), (1, 4095), (3, 4097), (128, 100), (5, 7), (64, 128)]


def _expand(ctx, worker, tensor, d, kind, block, scale_dtype, second):
    a, b = (x.cpu().numpy() for x in ctx.state(worker, tensor, second))
    s = b.view(np.float16 if scale_dtype == "fp16" else np.float32).astype(np.float32)
    c = a.view(np.int8).astype(np.float32)
    if kind == "int4":
        nib = np.stack([a & 15, a >> 4], 1).reshape(-1)[:d].astype(np.int32)
        c = ((nib ^ 8) - 8).astype(np.float32)
    return c * np.repeat(s, block)[:d]


@pytest.mark.parametrize("iconef", [0, 1])
@pytest.mark.parametrize("kind,block,scale_dtype", [("int8", 256, "fp32"), ("int8", 32, "fp16"), ("int4", 128, "fp16"),
                                                    ("int4", 64, "fp32")])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("shapes", [SHAPES, SHAPES + [(1, 1024), (1, 1023), (1600, 1600)]])
def test_decode_equals_codes_times_scales(kind, block, scale_dtype, iconef, offset, shapes):
    from paper_2312_08538_b200 import binding as b
    ctx = b.ConEF([(r, c, 1) for r, c in shapes], 2, dict(kind="randk", k_num=1, k_den=10, seed=3),
                  dict(kind=kind, block=block, scale_dtype=scale_dtype, iconef=iconef), 0.1)
    total = sum(r * c for r, c in shapes)
    ctx.step(0, [torch.randn(total, device="cuda") for _ in range(2)], 0)
    out = torch.full((total + offset + 1,), 7.0, device="cuda")
    ctx.decompress_error(1, out[offset:])
    want = [_expand(ctx, 1, l, r * c, kind, block, scale_dtype, False) +
            (_expand(ctx, 1, l, r * c, kind, block, scale_dtype, True) if iconef else 0) for l, (r, c) in enumerate(shapes)]
    got = out.cpu().numpy()
    assert np.array_equal(got[offset:offset + total], np.concatenate(want).astype(np.float32))
    assert got[offset + total] == 7.0
