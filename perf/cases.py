"""The WTConv layer's work as its users have it done: what is timed, on which inputs, and how close results must be.

A case names a layer call: the activation shape [B][C][H][W] and storage type, kernel size k, levels L, and how the
layer is reached (`mode`):

  forward        wtconv_forward on buffers the program keeps (inference through the C ABI)
  train          wtconv_forward and wtconv_backward on buffers the program keeps (a training step of the layer)
  module_infer   WTConv2d under torch.no_grad()
  module_train   WTConv2d forward and torch.autograd.grad of everything it has a gradient for
  host           wtconv_step_host: forward and backward from pinned host buffers and back

Activations and upstream gradients are N(0, 1), depthwise weights N(0, 0.1), scales U(0.5, 1.5), biases N(0, 0.1).
"""
import torch

from paper_2608_10805_b200 import io_model
from paper_2608_10805_b200 import wtconv as wt
from paper_2608_10805_b200.autograd import WTConv2d

BYTES = {"f32": 4, "f16": 2, "bf16": 2}


def _case(name, mode, B, C, H, W, k, L, dtype, bias=False):
    return {"name": name, "mode": mode, "B": B, "C": C, "H": H, "W": W, "k": k, "L": L, "dtype": dtype, "bias": bias}


def listed():
    return [
        # one image through the last stage's layer: the smallest call, all latency
        _case("infer_stage4_b1", "module_infer", 1, 768, 7, 7, 5, 1, "bf16", True),
        # fine-tuning with a few images per GPU through the module: launches and host work count
        _case("module_train_stage2_b8", "module_train", 8, 192, 28, 28, 5, 2, "bf16", True),
        # a training step of the four stages' layers of WTConvNeXt-T at 128 images per GPU
        _case("stage1_train_bf16", "train", 128, 96, 56, 56, 5, 3, "bf16"),
        _case("stage2_train_bf16", "train", 128, 192, 28, 28, 5, 2, "bf16"),
        _case("stage3_train_bf16", "train", 128, 384, 14, 14, 5, 1, "bf16"),
        _case("stage4_train_bf16", "train", 128, 768, 7, 7, 5, 1, "bf16"),
        # inference in full precision with all five levels (the deepest point of the level sweep)
        _case("sweep_L5_forward_f32", "forward", 32, 128, 64, 64, 5, 5, "f32"),
        # the kernel-size variants of the stage-1 layer
        _case("stage1_k3_train_f32", "train", 16, 96, 56, 56, 3, 3, "f32"),
        _case("stage1_k7_train_f32", "train", 16, 96, 56, 56, 7, 3, "f32"),
        # dense prediction: planes far beyond one SM's shared memory, with even rows (the largest case) and odd ones
        _case("large_train_f16", "train", 16, 256, 256, 256, 5, 5, "f16"),
        _case("large_odd_forward_f16", "forward", 16, 256, 225, 225, 5, 5, "f16"),
        # a step whose data live on the host, copies included
        _case("host_step_stage2_b32", "host", 32, 192, 28, 28, 5, 2, "bf16"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    largest = next(c for c in listed() if c["name"] == "large_train_f16")
    most = work(largest)
    while True:
        side = _log_uniform(rng, 7, 256)
        H = max(7, min(256, round(side * (0.8 + 0.4 * rng.random()))))
        W = max(7, min(256, round(side * (0.8 + 0.4 * rng.random()))))
        if rng.random() < 0.4:
            H = W = side  # square planes, as most networks have them
        mode = rng.choices(["forward", "train", "module_infer", "module_train", "host"], [30, 40, 10, 15, 5])[0]
        case = {"mode": mode, "B": _log_uniform(rng, 1, 128), "C": _log_uniform(rng, 16, 768), "H": H, "W": W,
                "k": rng.choices([3, 5, 7], [20, 65, 15])[0], "L": rng.choice([1, 2, 3, 4, 5]),
                "dtype": rng.choice(["f32", "f16", "bf16"]), "bias": rng.random() < 0.4}
        if rng.random() < 0.7:
            case["C"] = max(16, case["C"] // 16 * 16)  # channel counts are mostly multiples of 16
        w = work(case)
        n = case["B"] * case["C"] * H * W
        if w["flops"] > most["flops"] / 4 or w["bytes"] > most["bytes"] / 4:
            continue
        if mode == "host" and n * BYTES[case["dtype"]] > (64 << 20):
            continue
        return case


def _parameters(case, gen):
    C, k, L = case["C"], case["k"], case["L"]
    randn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    unif = lambda *s: 0.5 + torch.rand(s, generator=gen, device="cuda")
    return {"w0": 0.1 * randn(C, k, k), "s0": unif(C), "b0": 0.1 * randn(C) if case["bias"] else None,
            "wl": 0.1 * randn(L, C, 4, k, k), "sl": unif(L, C, 4)}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = wt.DTYPE_NAMES[case["dtype"]]
    shape = (case["B"], case["C"], case["H"], case["W"])

    def activation():
        t = torch.empty(shape, dtype=dtype, device="cuda")
        return t.normal_(generator=gen)

    x, p = activation(), _parameters(case, gen)
    mode = case["mode"]
    g = None if mode in ("forward", "module_infer") else activation()
    if mode in ("module_infer", "module_train"):
        layer = WTConv2d(case["C"], case["k"], case["L"], bias=case["bias"])
        with torch.no_grad():
            for n, v in p.items():
                if v is not None:
                    getattr(layer, n).copy_(v)
        leaves = [x] + [q for q in (layer.w0, layer.s0, layer.b0, layer.wl, layer.sl) if q is not None]
        if mode == "module_train":
            x.requires_grad_(True)
        return {"mode": mode, "layer": layer, "x": x, "g": g, "leaves": leaves}
    desc = wt.make_desc(*shape, case["k"], case["L"], dtype)
    s = {"mode": mode, "desc": desc, "x": x, "g": g, "out": torch.empty_like(x), **p}
    if mode != "forward":
        s["gx"] = torch.empty_like(x)
        for n, v in p.items():
            s["g" + n] = None if v is None else torch.empty_like(v)
    if mode == "host":
        s = {n: v.cpu().pin_memory() if isinstance(v, torch.Tensor) else v for n, v in s.items()}
        s["ws"] = torch.empty(wt.wtconv_step_host_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    else:
        s["ws"] = wt.alloc_workspace(desc)
    return s


def run(s):
    mode = s["mode"]
    if mode == "module_infer":
        with torch.no_grad():
            return s["layer"](s["x"])
    if mode == "module_train":
        out = s["layer"](s["x"])
        return [out, *torch.autograd.grad(out, s["leaves"], s["g"])]
    params = (s["w0"], s["s0"], s["b0"], s["wl"], s["sl"])
    if mode == "host":
        wt.wtconv_step_host(s["desc"], s["x"], s["g"], *params, s["out"], s["gx"], s["gw0"], s["gs0"], s["gb0"], s["gwl"],
                            s["gsl"], s["ws"])
    else:
        wt.wtconv_forward(s["desc"], s["x"], *params, s["out"], s["ws"])
        if mode == "forward":
            return s["out"]
        wt.wtconv_backward(s["desc"], s["x"], s["g"], *params, s["gx"], s["gw0"], s["gs0"], s["gb0"], s["gwl"], s["gsl"], s["ws"])
    return [t for t in (s["out"], s["gx"], s["gw0"], s["gs0"], s["gb0"], s["gwl"], s["gsl"]) if t is not None]


def work(case):
    """Forward: x in, out out.  A training step reads x for each of its two calls, which a training program keeps apart by
    the rest of the network.  Parameters once per call, their gradients once.  A host step's bytes are the same traffic
    on the device side; its copies cross the host link."""
    B, C, H, W, k, L = (case[n] for n in ("B", "C", "H", "W", "k", "L"))
    train = case["mode"] in ("train", "module_train", "host")
    act = B * C * H * W * BYTES[case["dtype"]]
    par = 4 * C * ((k * k + 1) * (1 + 4 * L) + (1 if case["bias"] else 0))
    flops = io_model.algorithmic_flops(B, C, H, W, k, L, "fwd+bwd" if train else "fwd")
    return {"bytes": 5 * act + 3 * par if train else 2 * act + par, "flops": flops}


def tolerance(case):
    """All arithmetic is float32.  float32 results differ by the order of the sums; 16-bit results by the final rounding of
    a value that may fall on either side of a rounding boundary: one unit in the last place of a few elements."""
    return {"f32": {"rel": 1e-5}, "f16": {"rel": 2e-4, "max": 2e-3}, "bf16": {"rel": 1.5e-3, "max": 1.6e-2}}[case["dtype"]]
