"""GPU parity: fp32 attention at the edges of its tiles (16 and 64 query rows, 64 and 128 keys, 16- and 32-key shares of a
warp) in both forms: few 16-row tiles, and more than 5.5 per SM (64-row tiles).  fp64 oracle, max-abs 1e-4."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import Guarded, assert_close_f32, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,mask,lens", [
    (1, 2, 1, 1, 1, 64, 0, None), (1, 3, 3, 15, 17, 64, 1, None), (2, 2, 2, 16, 128, 128, 0, None),
    (1, 4, 2, 17, 129, 64, 1, None), (1, 2, 2, 130, 100, 64, 1, None),   # rows without a visible key
    (3, 2, 2, 33, 200, 64, 2, (0, 16, 113)), (3, 2, 2, 33, 200, 128, 3, (1, 128, 129)),
    (4, 120, 120, 33, 65, 64, 3, (0, 1, 64, 65)), (4, 120, 60, 65, 63, 128, 1, None),  # 64-row tiles
    (2, 110, 110, 64, 130, 64, 2, (64, 130)),
])
def test_tiles(B, Hq, Hkv, Sq, Skv, D, mask, lens):
    w = wl.attention_workload("t", 61, B, Hq, Hkv, Sq, Skv, D, mask, 1.0 / np.sqrt(D), "f32", lens_range=(1, Skv))
    k, v = to_device(w.k), to_device(w.v)
    dl = None
    if lens is not None:
        w.lens = np.array(lens, dtype=np.int32)
        dl = torch.from_numpy(w.lens).cuda()
    ref = oracle.attn(w.q.values, w.k.values, w.v.values, mask, w.lens if lens is not None else None, w.scale)
    if lens is not None:  # padding may hold anything
        for b, n in enumerate(lens):
            k[b, :, n:] = float("nan")
            v[b, :, n:] = float("nan")
    g = Guarded((B, Hq, Sq, D), torch.float32)
    binding.attn_fused_f32(to_device(w.q), k, v, mask, dl, w.scale, out=g.tensor)
    binding.check_status()
    assert_close_f32(g.tensor, ref)
    g.assert_intact()


@pytest.mark.parametrize("B,H,Sq,Skv,D", [
    (1, 2, 100, 100, 64), (1, 2, 70, 133, 128),          # 16-row CTAs
    (8, 32, 100, 100, 64), (8, 32, 100, 137, 64), (8, 32, 70, 71, 128),  # 64-row CTAs
])
def test_a_later_v_row_reaches_no_earlier_tile_of_16_queries(B, H, Sq, Skv, D):
    """NaN and Inf in V rows that the causal mask hides from every query of a 16-row tile leave that tile as it is, bit for
    bit, wherever the row lies among the keys that a warp takes at once."""
    w = wl.attention_workload("t", 62, B, H, H, Sq, Skv, D, wl.MASK_CAUSAL, 1.0 / np.sqrt(D), "f32")
    q, k, v = to_device(w.q), to_device(w.k), to_device(w.v)
    clean = binding.attn_fused_f32(q, k, v, wl.MASK_CAUSAL, None, w.scale)
    for first_hidden in range(16, Sq, 16):        # the tile of queries first_hidden - 16 .. first_hidden - 1
        dirty = v.clone()
        dirty[:, :, first_hidden + Skv - Sq::2] = float("nan")
        dirty[:, :, first_hidden + Skv - Sq + 1::2] = float("inf")
        out = binding.attn_fused_f32(q, k, dirty, wl.MASK_CAUSAL, None, w.scale)
        assert torch.equal(out[:, :, :first_hidden], clean[:, :, :first_hidden])
    binding.check_status()


@pytest.mark.parametrize("B,H,S,D", [(1, 2, 40, 64), (1, 2, 40, 128), (8, 32, 100, 64), (8, 32, 100, 128)])
@pytest.mark.parametrize("factor,scale", [(1e19, 1.2e-38), (1e25, 0.0)])
def test_products_that_only_the_scale_brings_into_range(B, H, S, D, factor, scale):
    """q . k is beyond what fp32 holds, (scale * q) . k is not: the scale is applied to q, not to the sum."""
    w = wl.attention_workload("t", 63, B, H, H, S, S, D, wl.MASK_CAUSAL, 1.0, "f32")
    q, k, v = to_device(w.q) * factor, to_device(w.k) * factor, to_device(w.v)
    out = binding.attn_fused_f32(q, k, v, wl.MASK_CAUSAL, None, scale)
    binding.check_status()
    eff = scale * factor * factor
    pick = np.array([0, B - 1])
    ref = oracle.attn(w.q.values[pick], w.k.values[pick], w.v.values[pick], wl.MASK_CAUSAL, None, eff)
    assert_close_f32(out[[0, B - 1]], ref)
