"""GPU parity: 16-bit attention with more work items than SMs, where a CTA takes items out of the launch queue, loads the next
item's Q and issues its first scores behind the last products of the current one.  Items of very different cost side by
side: empty sequences, one key, one half-step, several; odd head counts (the second tile of an item is absent), odd
group sizes (two consecutive tiles of a head, the last one beyond Sq), rows that see no key.  fp64 oracle; runs are equal
bit for bit whatever CTA took which item."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import Guarded, assert_close_bf16, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,mask,lens", [
    (40, 8, 8, 130, 200, 64, 2, [0, 1, 63, 64, 65, 128, 129, 200]),     # a CTA per tile, empty ones among full ones
    (24, 15, 15, 100, 70, 64, 3, [70, 1, 0, 64]),                       # all tiles at once; rows without a visible key
    # head sizes up to 64 in many short tiles: pairs of heads with private K/V streams, then grouped heads in pairs of tiles
    (90, 8, 8, 130, 200, 64, 2, [0, 1, 63, 64, 65, 128, 129, 200]),     # empty items among full ones
    (64, 15, 15, 100, 70, 64, 3, [70, 1, 0, 64]),                       # odd head count (no second tile); rows without a visible key
    (100, 9, 9, 20, 129, 40, 1, None),                                  # head size below the kernel's, three half-steps
    (60, 10, 10, 257, 257, 64, 0, None),                                # a last tile of one row
    (50, 32, 8, 61, 200, 64, 3, [200, 0, 1, 64, 65, 129]),              # four heads of 32 rows
    (64, 28, 4, 130, 130, 64, 1, None),                                 # seven heads of 18 rows, two of the 128 out of use
    (64, 28, 4, 195, 195, 56, 1, None),                                 # an odd number of tiles: the last item has one
    (30, 7, 1, 260, 333, 128, 3, [333, 10, 0, 64, 100]),                # odd group: three tiles of a head in two items
    (50, 8, 2, 40, 300, 128, 2, [300, 0, 1, 65, 257]),                  # one tile per head, pairs of heads
    (64, 12, 12, 128, 128, 64, 1, None),                                # two half-steps each
    (20, 10, 2, 300, 300, 96, 1, None),
])
def test_many_uneven_items(B, Hq, Hkv, Sq, Skv, D, mask, lens):
    w = wl.attention_workload("t", 71, B, Hq, Hkv, Sq, Skv, D, mask, 1.0 / np.sqrt(D), "bf16", lens_range=(1, Skv))
    dl = None
    if lens is not None:
        w.lens = np.array((lens * B)[:B], dtype=np.int32)
        dl = torch.from_numpy(w.lens).cuda()
    q, k, v = to_device(w.q), to_device(w.k), to_device(w.v)
    g = Guarded((B, Hq, Sq, D), torch.bfloat16)
    binding.attn_fused(q, k, v, mask, dl, w.scale, out=g.tensor)
    binding.check_status()
    pick = np.unique(np.concatenate([np.arange(min(B, 8)), [B - 1]]))  # the oracle checks a period of the lengths and the last entry
    ref = oracle.attn(w.q.values[pick], w.k.values[pick], w.v.values[pick], mask, w.lens[pick] if lens is not None else None, w.scale)
    assert_close_bf16(g.tensor[torch.from_numpy(pick).cuda()], ref)
    g.assert_intact()
    assert torch.isfinite(g.tensor.float()).all()
    for _ in range(10):
        assert torch.equal(binding.attn_fused(q, k, v, mask, dl, w.scale), g.tensor)
    binding.check_status()


def test_many_items_with_a_bias():
    """The bias of a half-step is read ahead; -inf entries, ragged keys, more items than SMs."""
    B, H, Sq, Skv, D = 12, 16, 200, 201, 64
    w = wl.attention_workload("t", 72, B, H, H, Sq, Skv, D, wl.MASK_CAUSAL, 0.125, "bf16")
    bias = wl.normal_tensor(wl.seed_for(72, "b"), (B, 1, Sq, Skv), "f32").values.copy()
    bias[:, :, ::3, 5:70] = -np.inf
    got = binding.attn_fused_bias(to_device(w.q), to_device(w.k), to_device(w.v), torch.from_numpy(bias.astype(np.float32)).cuda(),
                                  wl.MASK_CAUSAL, None, 0.125)
    binding.check_status()
    ref = oracle.attn_bias(w.q.values[:3], w.k.values[:3], w.v.values[:3], bias[:3].astype(np.float64), wl.MASK_CAUSAL, None, 0.125)
    assert_close_bf16(got[:3], ref)


@pytest.mark.parametrize("B,H,Sq,Skv,D,heads", [
    (24, 15, 100, 200, 64, 1),    # odd head count: the last item of a batch entry has one tile
    (24, 15, 100, 130, 40, 15),   # a bias per head, head size below the kernel's
    (10, 9, 130, 70, 64, 1),      # two row tiles per head
    (11, 16, 90, 261, 56, 16),    # even head count, a ragged last step
])
@pytest.mark.parametrize("mask", [wl.MASK_PADDING, wl.MASK_PADDING | wl.MASK_CAUSAL])
def test_pairs_of_heads_with_a_bias_and_lengths(B, H, Sq, Skv, D, heads, mask):
    """Up to 64 columns, one head per tile and more tiles than SMs: an item is two heads, each with its own K and V copies.  Unequal
    streams, empty items among full ones, NaN in the padded rows."""
    assert B * H * -(-Sq // 128) > 148
    w = wl.attention_workload("t", 73, B, H, H, Sq, Skv, D, mask, D ** -0.5, "bf16", lens_range=(1, Skv))
    w.lens = np.array(([Skv, 0, 1, 64, 65, min(128, Skv), 129] * B)[:B], dtype=np.int32).clip(0, Skv)
    q, k, v = to_device(w.q), to_device(w.k), to_device(w.v)
    for b in range(B):
        k[b, :, int(w.lens[b]):] = float("nan")
        v[b, :, int(w.lens[b]):] = float("nan")
    bias = wl.normal_tensor(wl.seed_for(73, "b"), (B, heads, Sq, Skv), "f32").values.astype(np.float32)
    bias[:, :, ::7, 3:60] = -np.inf
    g = Guarded((B, H, Sq, D), torch.bfloat16)
    binding.attn_fused_bias(q, k, v, torch.from_numpy(bias).cuda(), mask, torch.from_numpy(w.lens).cuda(), w.scale, out=g.tensor)
    binding.check_status()
    pick = np.unique([*range(7), B - 1])
    ref = oracle.attn_bias(w.q.values[pick], w.k.values[pick], w.v.values[pick], bias[pick].astype(np.float64), mask, w.lens[pick], w.scale)
    assert_close_bf16(g.tensor[torch.from_numpy(pick).cuda()], ref)
    assert torch.isfinite(g.tensor.float()).all()
    g.assert_intact()
