"""wtconv_launch_count against the kernels that a call really enqueues (counted by the profiler), for every kernel family."""
import pytest
import torch

from paper_2608_10805_b200 import wtconv as wt

pytestmark = pytest.mark.gpu

SHAPES = [
    (2, 8, 56, 56, 5, 3, "f32", 0, "plane"), (3, 10, 40, 36, 5, 3, "f32", 0, "plane"), (12, 32, 7, 7, 5, 1, "f32", 0, "team"),
    (64, 64, 20, 24, 7, 2, "f32", 0, "tiled"), (61, 64, 14, 13, 5, 5, "bf16", 0, "plane"),  # (block-per-plane kernels; several levels on tensor cores)
    (2, 8, 56, 56, 3, 3, "f32", 0, "plane"), (2, 6, 20, 24, 7, 2, "f32", 0, "tiled"), (1, 2, 99, 201, 5, 2, "f32", 0, "window"),
    (1, 2, 225, 225, 5, 5, "f32", 0, "window"), (1, 2, 225, 225, 3, 4, "f32", 0, "window"),
    (24, 40, 31, 30, 5, 1, "bf16", 0, "tensor"), (33, 96, 50, 56, 3, 1, "bf16", 0, "tensor"), (33, 48, 50, 56, 3, 1, "bf16", 0, "plane/tensor"), (128, 768, 7, 7, 5, 1, "bf16", 0, "team/tensor"),
    (3, 16, 136, 200, 5, 3, "f16", 0, "panel"), (3, 16, 136, 200, 5, 3, "f16", wt.FLAG_NO_WINDOW, "tiled"), (2, 24, 161, 138, 5, 1, "f16", 0, "panel"),
]


def kernels(fn):
    fn()
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    return sum(1 for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA and not e.name.lower().startswith("mem"))


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s[:7])))
def test_launch_count(shape):
    B, C, H, W, k, L, dtype, flags, name = shape
    d = wt.make_desc(B, C, H, W, k, L, dtype, flags)
    assert wt.wtconv_plan_name(d) == name
    x = torch.randn(B, C, H, W, device="cuda").to(wt.DTYPE_NAMES[dtype])
    p = [torch.randn(*s, device="cuda") for s in ((C, k, k), (C,), (L, C, 4, k, k), (L, C, 4))]
    out, gx, gp, ws = torch.empty_like(x), torch.empty_like(x), [torch.empty_like(t) for t in p], wt.alloc_workspace(d)
    got = (kernels(lambda: wt.wtconv_forward(d, x, p[0], p[1], None, p[2], p[3], out, ws)),
           kernels(lambda: wt.wtconv_backward(d, x, x, p[0], p[1], None, p[2], p[3], gx, gp[0], gp[1], None, gp[2], gp[3], ws)))
    assert got == wt.wtconv_launch_count(d)
