"""GPU parity: the linear kernel that splits K over a cluster (outputs with few tiles) against the fp64 oracle.

Shapes are chosen for the places where the kernel can go wrong: one k-block and a ragged one, clusters of 2, 4 and 8
with uneven shares of the k-blocks, row counts at the edges of the 8-row X tile, of the 32-row warps and of the
128-row tile, ragged last column tiles, rings shorter than the k-loop, one and two CTAs per SM, and residual == out.
Tolerances are those of the 16-bit paths; the exchange of fp32 partial sums adds nothing that shows at 16 bits.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import Guarded, assert_close_bf16, to_device, to_f64

pytestmark = pytest.mark.gpu

# (M, N, K): (columns of a tile, CTAs per tile, two CTAs per SM) on 148 SMs (test_linear_plans.py checks that)
SHAPES = {
    (1, 8, 8): (64, 1, True), (1, 72, 136): (64, 1, True),             # one and three k-blocks, one column tile
    (7, 200, 520): (64, 4, True), (8, 264, 576): (64, 4, True),        # 9 k-blocks: shares of 2 and 3
    (16, 768, 3080): (64, 8, True), (33, 768, 4096): (64, 8, True),    # 49 k-blocks, the last of 8 columns; a second row warp
    (64, 4104, 1024): (64, 4, True), (65, 776, 776): (64, 4, False),   # two CTAs per SM / one
    (127, 2304, 768): (64, 2, False), (128, 768, 3072): (64, 8, False),  # whole row tile
    (40, 17000, 192): (128, 1, True),                                  # 128-column tiles: 133 CTAs
    (40, 38400, 192): (128, 1, True), (100, 38400, 136): (128, 1, True),  # 300 CTAs: more than run at once
    (129, 2048, 1544): (64, 2, False), (184, 1032, 4096): (128, 4, False), (300, 264, 2056): (64, 8, False),  # several row tiles
    (700, 3072, 136): (128, 1, False),                                 # several row tiles, one CTA per tile and per SM
}


def _case(M, N, K, dtype="bf16"):
    x = wl.normal_tensor(wl.seed_for(81, "x"), (M, K), dtype)
    w = wl.normal_tensor(wl.seed_for(81, "w"), (K, N), dtype, std=1.0 / np.sqrt(K))
    b = wl.normal_tensor(wl.seed_for(81, "b"), (N,), dtype, std=0.5)
    r = wl.normal_tensor(wl.seed_for(81, "q"), (M, N), dtype)
    return x, w, b, r


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("w_layout", [binding.W_KN, binding.W_NK])
def test_edges_of_tiles_and_shares(shape, w_layout):
    M, N, K = shape
    x, w, b, r = _case(M, N, K)
    wdev = to_device(w) if w_layout == binding.W_KN else to_device(w).t().contiguous()
    g = Guarded((M, N), torch.bfloat16)
    binding.linear_act(to_device(x), wdev, to_device(b), to_device(r), binding.ACT_GELU_TANH, w_layout, out=g.tensor)
    binding.check_status()
    assert_close_bf16(g.tensor, oracle.linear_act(x.values, w.values, b.values, r.values, oracle.ACT_GELU_TANH, 0))
    g.assert_intact()


@pytest.mark.parametrize("act", [binding.ACT_GELU_ERF, binding.ACT_RELU, binding.ACT_SILU, binding.ACT_NONE])
def test_activations_in_fp16(act):
    M, N, K = 24, 776, 1160
    x, w, b, _ = _case(M, N, K, "f16")
    y = binding.linear_act(to_device(x), to_device(w), to_device(b), None, act)
    assert_close_bf16(y, oracle.linear_act(x.values, w.values, b.values, None, act, 0))


@pytest.mark.parametrize("shape", [(1, 8, 8), (9, 72, 520), (128, 200, 2056), (33, 14336, 128), (64, 1024, 4096)])
@pytest.mark.parametrize("w_layout", [binding.W_KN, binding.W_NK])
def test_swiglu_one_row_tile(shape, w_layout):
    M, N, K = shape
    x, wg, _, _ = _case(M, N, K)
    wu = wl.normal_tensor(wl.seed_for(82, "w"), (K, N), "bf16", std=1.0 / np.sqrt(K))
    g, u = to_device(wg), to_device(wu)
    if w_layout == binding.W_NK:
        g, u = g.t().contiguous(), u.t().contiguous()
    y = binding.linear_swiglu(to_device(x), g, u, w_layout)
    binding.check_status()
    ref = oracle.linear_swiglu(x.values, wg.values, wu.values, 0)
    # as in test_parity_linear_swiglu: the product's own rounding, 2^-8 of the value, on top of the common bound
    assert np.all(np.abs(to_f64(y) - ref) <= 2e-2 + 2.0 ** -8 * np.abs(ref))


def test_runs_are_bitwise_equal_and_residual_may_be_the_output():
    M, N, K = 100, 768, 3072
    x, w, b, r = _case(M, N, K)
    xd, wd, bd, rd = to_device(x), to_device(w), to_device(b), to_device(r)
    want = binding.linear_act(xd, wd, bd, rd, binding.ACT_SILU)
    for _ in range(20):
        y = rd.clone()
        binding.linear_act(xd, wd, bd, y, binding.ACT_SILU, out=y)
        assert torch.equal(y, want)
