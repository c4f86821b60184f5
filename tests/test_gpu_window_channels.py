"""Window kernels whose blocks work through several channels: what a channel's gradient flush leaves in shared memory must not
reach the next channel's sums."""
import pytest
import torch

from paper_2608_10805_b200 import wtconv as wt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,C,H,W,L", [("f32", 640, 101, 101, 2), ("f32", 620, 99, 107, 1), ("f16", 640, 77, 106, 2)])
def test_many_channels_per_block(dtype, C, H, W, L):
    gen = torch.Generator(device="cuda").manual_seed(C)
    td = wt.DTYPE_NAMES[dtype]
    x, g = (torch.randn(1, C, H, W, generator=gen, device="cuda").to(td) for _ in range(2))
    w0, wl = (0.1 * torch.randn(*s, generator=gen, device="cuda") for s in ((C, 5, 5), (L, C, 4, 5, 5)))
    s0, sl = (0.5 + torch.rand(*s, generator=gen, device="cuda") for s in ((C,), (L, C, 4)))
    got = {}
    for flags in (wt.FLAG_PREFER_WINDOW, wt.FLAG_TILED_ONLY):
        d = wt.make_desc(1, C, H, W, 5, L, td, flags)
        assert wt.wtconv_plan_name(d) == ("window" if flags == wt.FLAG_PREFER_WINDOW else "tiled")
        out, grads = wt.forward_backward(d, x, g, w0, s0, None, wl, sl)
        got[flags] = [out] + [grads[n] for n in ("dx", "dw0", "ds0", "dwl", "dsl")]
    for a, b in zip(got[wt.FLAG_PREFER_WINDOW], got[wt.FLAG_TILED_ONLY]):
        assert torch.isfinite(a).all() and (a - b).abs().max() <= (1e-4 if a.dtype == torch.float32 else 4e-3) * b.abs().max()
