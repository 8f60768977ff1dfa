"""GPU parity: the linear on CTA pairs where whole rounds take two column tiles at a time: rows, columns and K that end inside a tile,
an odd number of column tiles, tiles that no round of double tiles is full of, whole and in halves, several rounds; both weight
layouts, bias and residual, fp16, the gated form.  fp64 oracle on sampled rows; tolerances of test_parity_linear and, gated, with
half an ulp of the output on top (test_parity_linear_swiglu)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import BF16_MAX_ABS, BF16_MEAN_ABS, Guarded, assert_close_bf16, to_device, to_f64

pytestmark = pytest.mark.gpu


def _rows(M):  # the first and last rows, and some of every row tile
    return np.unique(np.concatenate([np.arange(0, M, 37), [M - 2, M - 1]]))


@pytest.mark.parametrize("M,N,K,layout,dtype,extras", [
    (2100, 4400, 2056, binding.W_NK, "bf16", True),    # 9 x 18 tiles: one round of double tiles, 14 tiles in halves
    (2560, 3840, 2048, binding.W_KN, "bf16", False),   # 10 x 15: 70 double tiles are no round: all tile by tile
    (2817, 3752, 2048, binding.W_KN, "f16", True),     # 12 x 15: one round, ten double tiles and an odd column left over: 32 tiles in halves
    (5000, 8200, 2112, binding.W_NK, "f16", False),    # 20 x 33: four rounds and an odd column: 68 tiles
])
def test_linear(M, N, K, layout, dtype, extras):
    x = wl.normal_tensor(wl.seed_for(97, "x"), (M, K), dtype)
    w = wl.normal_tensor(wl.seed_for(97, "w"), (K, N), dtype, std=K ** -0.5)
    b, r = wl.normal_tensor(wl.seed_for(97, "b"), (N,), dtype), wl.normal_tensor(wl.seed_for(97, "q"), (M, N), dtype)
    dw = to_device(w) if layout == binding.W_KN else to_device(w).t().contiguous()
    g = Guarded((M, N), dw.dtype)
    act = binding.ACT_GELU_TANH if extras else binding.ACT_NONE
    binding.linear_act(to_device(x), dw, to_device(b) if extras else None, to_device(r) if extras else None, act, layout, out=g.tensor)
    binding.check_status()
    at = _rows(M)
    ref = oracle.linear_act(x.values[at], w.values, b.values if extras else None, r.values[at] if extras else None, act, 0)
    assert_close_bf16(g.tensor[torch.from_numpy(at).cuda()], ref)
    assert torch.isfinite(g.tensor.float()).all()
    g.assert_intact()


@pytest.mark.parametrize("M,N,K,layout", [(1300, 3200, 2056, binding.W_NK), (1100, 4000, 2048, binding.W_KN), (2300, 4240, 2048, binding.W_NK)])
def test_gated(M, N, K, layout):
    """6 x 25, 5 x 32 and 9 x 34 tiles (of 128 outputs): one and two rounds of double tiles, an odd column, halves and whole tiles left."""
    x = wl.normal_tensor(wl.seed_for(98, "x"), (M, K), "bf16")
    wg, wu = (wl.normal_tensor(wl.seed_for(98, t), (K, N), "bf16", std=K ** -0.5) for t in ("w", "b"))
    put = (lambda t: to_device(t)) if layout == binding.W_KN else (lambda t: to_device(t).t().contiguous())
    g = Guarded((M, N), torch.bfloat16)
    binding.linear_swiglu(to_device(x), put(wg), put(wu), layout, out=g.tensor)
    binding.check_status()
    at = _rows(M)
    ref = oracle.linear_swiglu(x.values[at], wg.values, wu.values, 0)
    got = to_f64(g.tensor[torch.from_numpy(at).cuda()])
    err = np.abs(got - ref)
    assert (err - 2.0 ** -8 * np.abs(ref)).max() <= BF16_MAX_ABS and err.mean() <= BF16_MEAN_ABS
    assert torch.isfinite(g.tensor.float()).all()
    g.assert_intact()
