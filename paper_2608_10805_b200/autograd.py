"""torch.autograd front end of the WTConv library: the layer as an autograd node and as an nn.Module.

Marshalling only: forward calls `wtconv_forward`, backward calls `wtconv_backward` (which recomputes
everything it needs from x, so nothing but x and the parameters is kept between the two calls - the
on-chip recomputation of Sec. 4.1 applied to training memory).  The node lives in the native module
(csrc_torch/wtconv_torch.cpp).  Parameters are float32 in every activation dtype.  The layer is Algorithm 1 of
the paper: base depthwise conv with scale (and optional bias) plus L Haar levels with their own depthwise convs and scales.
"""
import collections

import torch

from . import wtconv as wt


class _StatusWatch:
    """Deferred check of the kernels' bounded waits, without synchronising.

    The layer's calls report a wait that runs out by writing one word of pinned host memory; every later layer call looks
    at it and raises: the outputs of that earlier call were not valid.  For calls made outside the layer, `after_call`
    copies the status word of their workspace (asynchronously, on the same stream) into a pinned host integer and records
    an event; later calls look at the copies whose events have completed.  `drain()` waits for everything outstanding (call
    it before trusting results at the end of a run)."""

    def __init__(self):
        self.pending = collections.deque()
        self.free = []

    def after_call(self, desc, ws):
        flag = self.free.pop() if self.free else torch.zeros(1, dtype=torch.int32).pin_memory()
        wt.wtconv_read_status(desc, ws, flag)
        ev = torch.cuda.Event()
        ev.record()
        self.pending.append((ev, flag))
        self.poll()

    def poll(self, wait=False):
        bad = wt.native().take_alarm()
        while self.pending and (wait or self.pending[0][0].query()):
            ev, flag = self.pending.popleft()
            if wait:
                ev.synchronize()
            bad = int(flag[0]) != 0 or bad
            self.free.append(flag)
        if bad:
            raise wt.WTConvError(11, "a bounded device-side wait ran out in an earlier WTConv call; its outputs are not valid")

    def drain(self):
        if wt.native().used():
            torch.cuda.synchronize()
        self.poll(wait=True)


status_watch = _StatusWatch()


class WTConvFunction:
    """out = WTConv(x; w0, s0, b0, wl, sl).  b0 may be None.  k and L are read from wl's shape."""

    @staticmethod
    def apply(x, w0, s0, b0, wl, sl):
        return (wt._native or wt.native()).layer(x, w0, s0, b0, wl, sl)


class WTConv2d(torch.nn.Module):
    """Depthwise wavelet convolution layer (Algorithm 1): `channels` planes, kernel size k in {3, 5, 7},
    `levels` Haar levels.  Initialisation follows the benchmark's recipe: weights N(0, 0.1), level scales
    0.1, base scale 1 — any other initialisation can be written into the parameters afterwards."""

    def __init__(self, channels, kernel_size=5, levels=1, bias=True, device="cuda"):
        super().__init__()
        k, C, L = kernel_size, channels, levels
        self.channels, self.kernel_size, self.levels = C, k, L
        P = torch.nn.Parameter
        self.w0 = P(0.1 * torch.randn(C, k, k, device=device))
        self.s0 = P(torch.ones(C, device=device))
        self.b0 = P(torch.zeros(C, device=device)) if bias else None
        self.wl = P(0.1 * torch.randn(L, C, 4, k, k, device=device))
        self.sl = P(torch.full((L, C, 4), 0.1, device=device))

    def forward(self, x):
        return WTConvFunction.apply(x, self.w0, self.s0, self.b0, self.wl, self.sl)
