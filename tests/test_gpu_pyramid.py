"""Whole planes of several levels on the tensor cores (base convolution, level 1) and FMA units (levels >= 2): against the fp64
oracle at the edges of their tiles and units, with infinities and NaNs, and with waits that run out."""
import numpy as np
import pytest
import torch

from helpers import GRAD_NAMES, TOL, rel_err, run_gpu, run_oracle
from helpers import to_dev
from paper_2608_10805_b200 import inputs, wtconv as wt

pytestmark = pytest.mark.gpu

SHAPES = [  # B, C, H, W, k, L
    (32, 148, 28, 28, 5, 2),   # several operand arrays
    (13, 64, 30, 26, 5, 3),    # a unit of five images, rows of pairs
    (24, 149, 29, 31, 5, 4),   # odd rows, a row more than whole blocks of four, several units a block
    (16, 148, 56, 56, 5, 3),   # one operand array, levels >= 2 a unit ahead
    (8, 148, 57, 45, 3, 2),    # 3 x 3, one operand array, odd rows
    (64, 150, 14, 14, 5, 2),   # many units a block
    (8, 148, 61, 64, 5, 2),    # the widest plane
    (13, 74, 40, 64, 5, 3),    # planes in batches that do not divide eight
    (13, 148, 30, 26, 5, 3),   # a last octet of five images, rows of pairs
    (72, 300, 14, 14, 5, 3),   # many units a block
    (5, 139, 77, 4, 3, 8),     # fewer than eight images, the narrowest plane, more than 64 rows, every level
    (16, 148, 100, 31, 5, 3),  # four MMA tiles of one plane
]


def pyramid(B, C, H, W, k, L, dtype, flags=0):
    return "pyramid" in wt.wtconv_plan_describe(wt.make_desc(B, C, H, W, k, L, wt.DTYPE_NAMES[dtype], flags))


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_against_the_oracle(shape, dtype):
    w = inputs.Workload("pyramid", *shape, dtype, 500 + SHAPES.index(shape))
    assert pyramid(*shape, dtype)
    I = inputs.make_inputs(w, bias=SHAPES.index(shape) % 2 == 0)
    out, grads = run_gpu(w, I)
    ref, ref_grads = run_oracle(w, I)
    assert rel_err(out, ref) < TOL[dtype] / 4  # the only extra error is the final rounding: 2^-8 / 2^-11
    for n in GRAD_NAMES:
        if ref_grads.get(n) is not None and ref_grads[n].size:
            # parameter gradients are sums in fp32 of exact products: far inside the storage type's tolerance
            assert rel_err(grads[n], ref_grads[n]) < (TOL[dtype] / 4 if n == "dx" else 1e-5), n


BACKWARD_SHAPES = [  # B, C, H, W, k, L
    (13, 64, 30, 26, 5, 3),    # a unit of five images, copies of pairs
    (61, 96, 29, 31, 5, 4),    # odd rows, a last unit that is not full, a row more than whole blocks of four
    (16, 148, 56, 56, 5, 3),   # one pair of operand arrays, planes in two batches, four-row tiles
    (40, 148, 57, 45, 5, 2),   # odd rows, one pair of arrays
    (64, 150, 14, 14, 3, 2),   # 3 x 3, four octets a unit, several channels a block
    (61, 64, 14, 13, 5, 5),    # levels down to one coefficient, units of four octets
    (8, 148, 61, 64, 5, 2),    # the widest plane
    (13, 74, 40, 64, 5, 3),    # rows of whole 16-byte words
    (61, 296, 14, 14, 3, 3),   # 3 x 3, several octets a unit and channels a block
    (5, 139, 77, 4, 3, 8),     # fewer than eight images, the narrowest plane, more than 64 rows, every level
    (16, 148, 100, 31, 5, 3),
]


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape", BACKWARD_SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_backward_against_the_oracle(shape, dtype):
    w = inputs.Workload("pyramid", *shape, dtype, 600 + BACKWARD_SHAPES.index(shape))
    assert "pyramid gradients" in wt.wtconv_plan_describe(wt.make_desc(*shape, wt.DTYPE_NAMES[dtype]))
    I = inputs.make_inputs(w, bias=BACKWARD_SHAPES.index(shape) % 2 == 0)
    _, grads = run_gpu(w, I)
    _, ref_grads = run_oracle(w, I)
    for n in GRAD_NAMES:
        if ref_grads.get(n) is not None and ref_grads[n].size:
            # as above: grad_x is rounded once, parameter gradients are sums in fp32 of exact products
            assert rel_err(grads[n], ref_grads[n]) < (TOL[dtype] / 4 if n == "dx" else 1e-5), n
            # chains of eight truncated additions, the rest rounded: 1 - 4e-7 measured on these shapes, as on the FMA kernels
            assert n not in ("dw0", "dwl") or rel_err(grads[n], ref_grads[n]) < 1e-6, n


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape", [(8, 592, 48, 48, 5, 3), (28, 608, 16, 16, 5, 4), (8, 444, 56, 56, 5, 3)], ids=lambda s: "x".join(map(str, s)))
def test_every_unit_another_channel(shape, dtype):
    """Levels >= 2 run ahead of the loads: a channel's scale and bias are not its neighbours'."""
    B, C, H, W, k, L = shape
    assert "direct" in wt.wtconv_plan_describe(wt.make_desc(*shape, wt.DTYPE_NAMES[dtype]))
    gen = torch.Generator(device="cuda").manual_seed(4)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    x = rnd(B, C, H, W).to(wt.DTYPE_NAMES[dtype])
    size = 2.0 ** (torch.arange(C, device="cuda") % 9 - 4)
    p = [0.1 * rnd(C, k, k) * size[:, None, None], 0.5 + rnd(C).abs(), rnd(C) * size, 0.1 * rnd(L, C, 4, k, k) * size[:, None, None, None], 0.5 + rnd(L, C, 4).abs()]
    res = []
    for flags in (0, wt.FLAG_NO_WINDOW):
        d = wt.make_desc(*shape, wt.DTYPE_NAMES[dtype], flags)
        out = torch.empty_like(x)
        wt.wtconv_forward(d, x, *p, out, wt.alloc_workspace(d))
        res.append(out.float())
    err, big = (res[0] - res[1]).abs().amax((0, 2, 3)), res[1].abs().amax((0, 2, 3))
    assert (err <= 2.0 ** (-7 if dtype == "bf16" else -10) * big).all()  # the final rounding on either side


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape,buffers,backward", [((60, 162, 5, 5, 5, 8), 4, True), ((15, 735, 5, 6, 5, 8), 4, True), ((72, 300, 14, 14, 5, 3), 4, True),
                                                    ((128, 600, 12, 12, 5, 3), 3, True)], ids=lambda s: str(s).replace(", ", "x"))
def test_the_next_channels_weights_wait_for_units_under_way(shape, buffers, backward, dtype):
    """Three or four operand arrays and few MMAs a unit: several loaded units wait for their MMAs when a channel's weights, scale and
    bias are replaced.  Channels differ by powers of two, each is compared by itself, in calls that follow one another."""
    B, C, H, W, k, L = shape
    plan = wt.wtconv_plan_describe(wt.make_desc(*shape, wt.DTYPE_NAMES[dtype]))
    S, T, n, bufs, units = (int(plan.split("fwd[pyramid")[1].split(q)[1].split()[0].strip(",")) for q in (" S=", " T=", " n=", " buffers=", " units="))
    assert bufs == buffers and T * n <= 6 and units >= 4 * 148 and ("pyramid gradients" in plan) == backward
    gen = torch.Generator(device="cuda").manual_seed(6)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    x, g = (rnd(B, C, H, W).to(wt.DTYPE_NAMES[dtype]) for _ in range(2))
    size = 2.0 ** (5 * torch.arange(C, device="cuda") % 9 - 4)
    p = [0.1 * rnd(C, k, k) * size[:, None, None], 0.5 + rnd(C).abs(), rnd(C) * size, 0.1 * rnd(L, C, 4, k, k) * size[:, None, None, None], 0.5 + rnd(L, C, 4).abs()]
    res = []
    for flags, calls in ((wt.FLAG_NO_WINDOW, 1), (0, 6)):
        d = wt.make_desc(*shape, wt.DTYPE_NAMES[dtype], flags)
        ws = wt.alloc_workspace(d)
        outs = [[torch.empty_like(x), torch.empty_like(x)] + [torch.empty_like(q) for q in p] for _ in range(calls)]
        for o in outs:
            wt.wtconv_forward(d, x, *p, o[0], ws)
            wt.wtconv_backward(d, x, g, *p, *o[1:], ws)
        res += outs
    per_channel = lambda t, dim: t.float().movedim(dim, 0).flatten(1).abs().amax(1)
    for o in res[1:]:
        for i, dim in ((0, 1), (1, 1), (2, 0), (5, 1)):  # out, grad_x, the weights' gradients
            err = per_channel(o[i].float() - res[0][i].float(), dim)
            # activations: the final rounding on either side; weight gradients: sums of thousands of products in fp32
            assert (err <= (2.0 ** (-7 if dtype == "bf16" else -10) if i < 2 else 1e-4) * per_channel(res[0][i], dim)).all(), i


def test_the_range_of_the_coefficients():
    """Values whose plain sums over a coefficient's pixels (and products of such sums) are beyond fp32, while the transform's own
    coefficients, outputs and gradients are not."""
    shape = B, C, H, W, k, L = 128, 64, 16, 16, 5, 5
    plan = wt.wtconv_plan_describe(wt.make_desc(*shape, "bf16"))
    assert "fwd[pyramid" in plan and "pyramid gradients" in plan
    w = inputs.Workload("range", *shape, "bf16", 78)
    data = inputs.make_inputs(w)
    data["s0"][:], data["sl"][:] = 1, 1
    shade = {n: 1 + np.abs(data[n]) / 64 for n in ("x", "g")}  # (at most 1.1)
    for x_exp, g_exp in ((121, -121), (-121, 121), (56, 54)):
        for n, e in (("x", x_exp), ("g", g_exp)):
            data[n] = torch.from_numpy(np.float32(2.0 ** e) * shade[n]).bfloat16().float().numpy()
        out, grads = run_gpu(w, data, guarded=False)
        ref, ref_grads = run_oracle(w, data)
        for got, want, tol in ((out, ref, TOL["bf16"] / 4), *((grads[n], ref_grads[n], TOL["bf16"] / 4 if n == "dx" else 1e-5) for n in GRAD_NAMES if n != "db0")):
            assert np.abs(want).max() < 3e38 and rel_err(got, want) < tol


NON_FINITE_SHAPES = [(64, 96, 28, 28, 5, 2), (13, 148, 30, 26, 3, 3), (61, 96, 29, 31, 5, 4), (16, 148, 56, 56, 5, 3), (61, 192, 14, 13, 5, 4)]


def with_infinities(shape, dtype):
    """Infinities and NaNs at the planes' edges and in the middle, those of x and of grad_out in channels of their own."""
    B, C, H, W, k, L = shape
    w = inputs.Workload("pyramid", *shape, dtype, 930)
    plan = wt.wtconv_plan_describe(wt.make_desc(*shape, wt.DTYPE_NAMES[dtype]))
    assert "fwd[pyramid" in plan and "pyramid gradients" in plan
    data = inputs.make_inputs(w)
    for n, channels in (("x", (0, 1, 2, C - 1)), ("g", (4, 5, 6, C - 2))):
        for c, (b, y, x_, v) in zip(channels, ((0, H // 2, W // 2, np.inf), (1, 0, W - 1, np.nan), (B - 1, H - 1, 0, -np.inf), (2, H - 1, W - 1, np.inf))):
            data[n][b, c, y, x_] = v
    return w, data


def run_unchecked(w, data, flags=0):
    dt = wt.DTYPE_NAMES[w.dtype]
    out, grads = wt.forward_backward(wt.make_desc(w.B, w.C, w.H, w.W, w.k, w.L, dt, flags), to_dev(data["x"], dt), to_dev(data["g"], dt), to_dev(data["w0"]),
                                     to_dev(data["s0"]), None, to_dev(data["wl"]), to_dev(data["sl"]))
    return out.double().cpu().numpy(), {n: v.double().cpu().numpy() for n, v in grads.items() if v is not None}


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape", NON_FINITE_SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_outputs_and_grad_x_are_non_finite_where_the_oracles_are(shape, dtype):
    w, data = with_infinities(shape, dtype)
    out, grads = run_unchecked(w, data)
    ref, ref_grads = run_oracle(w, data)
    for a, want in ((out, ref), (grads["dx"], ref_grads["dx"])):
        fin = np.isfinite(want)
        assert 0 < fin.sum() < fin.size and (np.isfinite(a) == fin).all()
        assert rel_err(a[fin], want[fin]) < TOL[dtype] / 4


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("shape", NON_FINITE_SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_weight_gradients_are_non_finite_where_their_taps_meet_it(shape, dtype):
    """Base convolution and level 1: where the oracle's are (which multiplies grad_out with zeros around x: not further there).  Levels
    >= 2: no further than on the block-per-plane kernels."""
    w, data = with_infinities(shape, dtype)
    grads, family, ref = run_unchecked(w, data)[1], run_unchecked(w, data, wt.FLAG_NO_WINDOW)[1], run_oracle(w, data)[1]
    for a, want in ((grads["dw0"], ref["dw0"]), (grads["dwl"][0], ref["dwl"][0])):
        fin, got = np.isfinite(want), np.isfinite(a)
        assert 0 < fin.sum() < fin.size and got[fin].all() and (got == fin)[:4].all() and (got == fin)[-1].all() and not got[4].any()
        assert rel_err(a[fin], want[fin]) < 1e-5
    assert all(np.isfinite(grads[n][np.isfinite(family[n])]).all() for n in ("dwl", "dsl", "ds0"))


@pytest.mark.parametrize("where", [(0, 0), (27, 27), (13, 8)])
def test_infinities_reach_their_own_stencil_only(where):
    """The same elements are non-finite as on the kernels that compute every product on its own."""
    B, C, H, W, k, L = SHAPES[0]
    assert pyramid(B, C, H, W, k, L, "bf16")
    gen = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    x = rnd(B, C, H, W).to(torch.bfloat16)
    x[1, 5, where[0], where[1]] = float("inf")
    x[9, 7, where[0], where[1]] = float("nan")
    p = [0.1 * rnd(C, k, k), rnd(C), None, 0.1 * rnd(L, C, 4, k, k), rnd(L, C, 4)]
    res = []
    for flags in (0, wt.FLAG_NO_WINDOW):
        d = wt.make_desc(B, C, H, W, k, L, torch.bfloat16, flags)
        out = torch.empty_like(x)
        wt.wtconv_forward(d, x, *p, out, wt.alloc_workspace(d))
        res.append(out)
    assert torch.equal(torch.isfinite(res[0]), torch.isfinite(res[1]))
    ok = torch.isfinite(res[0])
    assert (res[0][ok].float() - res[1][ok].float()).abs().max() <= 2.0 ** -7 * res[1][ok].float().abs().max()
    assert int((~ok).sum()) > 0


def test_waits_that_run_out_are_reported_and_the_next_call_is_clean():
    B, C, H, W, k, L = SHAPES[0]
    assert pyramid(B, C, H, W, k, L, "f16", wt.FLAG_TEST_NO_COPY)
    x = torch.randn(B, C, H, W, device="cuda").half()
    p = [torch.randn(C, k, k, device="cuda"), torch.randn(C, device="cuda"), None, torch.randn(L, C, 4, k, k, device="cuda"), torch.randn(L, C, 4, device="cuda")]
    flag = torch.zeros(2, dtype=torch.int32).pin_memory()
    out = torch.empty_like(x)
    ws = wt.alloc_workspace(wt.make_desc(B, C, H, W, k, L, torch.float16))
    for i, flags in enumerate((wt.FLAG_TEST_NO_COPY, 0)):
        d = wt.make_desc(B, C, H, W, k, L, torch.float16, flags)
        wt.wtconv_forward(d, x, *p, out, ws)
        wt.wtconv_read_status(d, ws, flag[i:i + 1])
    torch.cuda.synchronize()
    assert flag.tolist() == [1, 0]


def test_backward_waits_that_run_out_are_reported_and_the_next_call_is_clean():
    B, C, H, W, k, L = BACKWARD_SHAPES[0]
    assert "pyramid gradients" in wt.wtconv_plan_describe(wt.make_desc(B, C, H, W, k, L, torch.float16, wt.FLAG_TEST_NO_COPY))
    x, g = (torch.randn(B, C, H, W, device="cuda").half() for _ in range(2))
    p = [torch.randn(C, k, k, device="cuda"), torch.randn(C, device="cuda"), None, torch.randn(L, C, 4, k, k, device="cuda"), torch.randn(L, C, 4, device="cuda")]
    flag = torch.zeros(2, dtype=torch.int32).pin_memory()
    grads = [torch.empty_like(x)] + [None if q is None else torch.empty_like(q) for q in p]
    ws = wt.alloc_workspace(wt.make_desc(B, C, H, W, k, L, torch.float16))
    for i, flags in enumerate((wt.FLAG_TEST_NO_COPY, 0)):
        d = wt.make_desc(B, C, H, W, k, L, torch.float16, flags)
        wt.wtconv_backward(d, x, g, *p, *grads, ws)
        wt.wtconv_read_status(d, ws, flag[i:i + 1])
    torch.cuda.synchronize()
    assert flag.tolist() == [1, 0]
