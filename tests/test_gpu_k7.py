"""7 x 7 kernels on the block-per-plane kernels (halo of three rows, four columns), against the fp64 oracle and, over random
shapes, against the per-level kernels they replace."""
import numpy as np
import pytest
import torch

from helpers import TOL, assert_close, run_gpu, run_oracle
from paper_2608_10805_b200 import inputs
from paper_2608_10805_b200 import wtconv as wt
from paper_2608_10805_b200.inputs import Workload

pytestmark = pytest.mark.gpu

# tile edges (4 x 4 and 4 x 8), odd grids at every level, one tile, several planes per unit, no level, the largest plane served
SHAPES = [(3, 5, 7, 7, 3), (2, 16, 14, 14, 1), (2, 8, 28, 28, 2), (3, 4, 33, 29, 3), (2, 3, 56, 56, 3), (1, 2, 64, 64, 5), (5, 7, 9, 12, 2),
          (2, 3, 1, 19, 2), (1, 1, 1, 1, 1), (2, 4, 17, 31, 0), (9, 32, 8, 8, 1), (1, 2, 66, 60, 2)]


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("B,C,H,W,L", SHAPES)
def test_against_the_oracle(B, C, H, W, L, dtype):
    wl = Workload("k7_%dx%d_L%d" % (H, W, L), B, C, H, W, 7, L, dtype, 700 + H + W)
    assert "plane" in wt.wtconv_plan_describe(wt.make_desc(B, C, H, W, 7, L, wt.DTYPE_NAMES[dtype]))
    I = inputs.make_inputs(wl, bias=True)
    assert_close(wl, run_gpu(wl, I), run_oracle(wl, I))


@pytest.mark.parametrize("seed", range(12))
def test_against_the_per_level_kernels(seed):
    rng = np.random.default_rng(seed)
    H, W, L = int(rng.integers(2, 66)), int(rng.integers(2, 66)), int(rng.integers(0, 6))
    wl = Workload("k7_%d" % seed, int(rng.integers(1, 7)), int(rng.integers(1, 40)), H, W, 7, L, ["f32", "f16", "bf16"][seed % 3], 40 + seed)
    I = inputs.make_inputs(wl, bias=seed % 2 == 0)
    a, b = run_gpu(wl, I), run_gpu(wl, I, flags=wt.FLAG_TILED_ONLY)
    assert_close(wl, a, b, tol=2 * TOL[wl.dtype])  # each side is within the tolerance of the exact result


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("B,C,H,W,L", SHAPES)
def test_block_per_plane_kernels_against_the_oracle(B, C, H, W, L, dtype):
    """Few planes take the per-level kernels, unless these are kept away."""
    wl = Workload("k7_%dx%d_L%d" % (H, W, L), B, C, H, W, 7, L, dtype, 700 + H + W)
    assert wt.wtconv_plan_describe(wt.make_desc(B, C, H, W, 7, L, wt.DTYPE_NAMES[dtype], wt.FLAG_NO_TEAM)).startswith("plane")
    I = inputs.make_inputs(wl, bias=True)
    assert_close(wl, run_gpu(wl, I, flags=wt.FLAG_NO_TEAM), run_oracle(wl, I))


@pytest.mark.parametrize("seed", range(12))
def test_block_per_plane_kernels_against_the_per_level_kernels(seed):
    rng = np.random.default_rng(seed)
    H, W, L = int(rng.integers(2, 66)), int(rng.integers(2, 66)), int(rng.integers(0, 6))
    wl = Workload("k7_%d" % seed, int(rng.integers(1, 7)), int(rng.integers(1, 40)), H, W, 7, L, ["f32", "f16", "bf16"][seed % 3], 40 + seed)
    I = inputs.make_inputs(wl, bias=seed % 2 == 0)
    a, b = run_gpu(wl, I, flags=wt.FLAG_NO_TEAM), run_gpu(wl, I, flags=wt.FLAG_TILED_ONLY)
    assert_close(wl, a, b, tol=2 * TOL[wl.dtype])  # each side is within the tolerance of the exact result
