"""GPU parity: query heads of one KV group in one tile.  Group sizes that fill the 128 rows (2, 4, 8, 16), that leave some out of
use (3, 5, 6, 7, 12, 15), that are packed in part (32) or not at all (17); query rows that end inside a head's share of the
tile, on its edge and one beyond; causal offsets that are no multiple of a 64-key step; every mask; one tile per item (few
tiles), two, and more items than SMs; strided views, fp16, a bias per head, head sizes above 128.  fp64 oracle; outputs start as
NaN between guard bytes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import Guarded, assert_close_bf16, to_device

pytestmark = pytest.mark.gpu


def _run(B, Hq, Hkv, Sq, Skv, D, mask, dtype="bf16", lens=None, strided=False):
    w = wl.attention_workload("t", 83, B, Hq, Hkv, Sq, Skv, D, mask, 1.0 / np.sqrt(D), dtype, lens_range=(1, Skv))
    dl = None
    if mask & wl.MASK_PADDING:
        w.lens = np.array(((lens or [Skv, 0, 1, 65]) * B)[:B], dtype=np.int32).clip(0, Skv)
        dl = torch.from_numpy(w.lens).cuda()
    q, k, v = to_device(w.q), to_device(w.k), to_device(w.v)
    if strided:  # token-major rows, heads side by side, as a fused projection leaves them
        g = Guarded((B, Sq, Hq, D), q.dtype)
        qv, kv, vv = (t.transpose(1, 2).contiguous().transpose(1, 2) for t in (q, k, v))
        out = g.tensor.transpose(1, 2)
        binding.attn_fused_strided(qv, kv, vv, out, mask, dl, w.scale)
    else:
        g = Guarded((B, Hq, Sq, D), q.dtype)
        out = (binding.attn_fused_f16 if dtype == "f16" else binding.attn_fused)(q, k, v, mask, dl, w.scale, out=g.tensor)
    binding.check_status()
    assert_close_bf16(out, oracle.attn(w.q.values, w.k.values, w.v.values, mask, w.lens if dl is not None else None, w.scale))
    g.assert_intact()


@pytest.mark.parametrize("G,rows", [(2, 64), (3, 42), (4, 32), (5, 25), (6, 21), (7, 18), (8, 16), (12, 10), (15, 8), (16, 8), (17, 128), (32, 8)])
@pytest.mark.parametrize("D", [64, 128])
def test_rows_around_a_heads_share_of_the_tile(G, rows, D):
    for Sq, Skv, mask in ((1, 70, 1), (rows - 1, 200, 3), (rows, rows, 1), (rows + 1, 129, 2), (2 * rows + 3, 2 * rows + 80, 3), (5 * rows + 1, 300, 0)):
        _run(2, 2 * G, 2, Sq, Skv, D, mask)


@pytest.mark.parametrize("G,rows", [(2, 64), (3, 42), (4, 32), (5, 25), (6, 21), (7, 18), (8, 16), (12, 10), (15, 8), (16, 8)])
@pytest.mark.parametrize("D", [64, 128])
def test_rows_around_a_heads_share_with_many_items(G, rows, D):
    """Above 64 columns few items, which all run at once, have one head per tile; these do not run at once."""
    B = 320 // (2 * G) + 1
    for Sq, Skv, mask in ((rows - 1, 200, 3), (rows + 1, 129, 2), (2 * rows + 3, 2 * rows + 80, 3), (5 * rows + 1, 5 * rows + 1, 1)):
        w = wl.attention_workload("t", 86, B, 2 * G, 2, Sq, Skv, D, mask, D ** -0.5, "bf16", lens_range=(1, Skv))
        dl = None
        if mask & wl.MASK_PADDING:
            w.lens = np.array(([Skv, 0, 1, 65] * B)[:B], dtype=np.int32)
            dl = torch.from_numpy(w.lens).cuda()
        g = Guarded((B, 2 * G, Sq, D), torch.bfloat16)
        binding.attn_fused(to_device(w.q), to_device(w.k), to_device(w.v), mask, dl, w.scale, out=g.tensor)
        binding.check_status()
        pick = np.unique([0, 1, 2, 3, B - 1])  # a period of the lengths and the last entry
        ref = oracle.attn(w.q.values[pick], w.k.values[pick], w.v.values[pick], mask, w.lens[pick] if dl is not None else None, w.scale)
        assert_close_bf16(g.tensor[torch.from_numpy(pick).cuda()], ref)
        assert torch.isfinite(g.tensor.float()).all()
        g.assert_intact()


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,mask", [
    (1, 28, 4, 1179, 1179, 128, 1),  # pairs of tiles of one head, as many items as SMs or fewer
    (1, 28, 4, 1355, 1355, 96, 1),   # a few short items wait
    (2, 10, 2, 900, 900, 128, 1),    # a tile per item with grouped heads only
    (1, 28, 4, 100, 333, 80, 3),     # a tile per item, one head each
    (6, 28, 4, 250, 300, 80, 2),     # more items than SMs, as many tiles as with grouped heads
])
def test_one_head_per_tile_or_more(B, Hq, Hkv, Sq, Skv, D, mask):
    _run(B, Hq, Hkv, Sq, Skv, D, mask)


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,mask", [
    (6, 28, 4, 333, 601, 128, 3),   # more items than SMs, 126 rows in use, empty sequences among full ones
    (40, 16, 4, 130, 130, 80, 1),   # more items than SMs, all rows in use, head size below the kernel's
    (9, 24, 2, 95, 70, 64, 3),      # rows that see no key
    (3, 32, 8, 130, 517, 96, 2),
])
@pytest.mark.parametrize("strided", [False, True])
def test_many_packed_items(B, Hq, Hkv, Sq, Skv, D, mask, strided):
    _run(B, Hq, Hkv, Sq, Skv, D, mask, strided=strided, lens=[Skv, 0, 1, 64, 65, Skv // 2])


@pytest.mark.parametrize("G", [3, 4, 7])
@pytest.mark.parametrize("D", [64, 128])
def test_fp16(G, D):
    _run(3, 4 * G, 4, 77, 205, D, 3, "f16")


@pytest.mark.parametrize("G,Sq,Skv,D,mask", [(2, 65, 130, 256, 1), (4, 33, 200, 192, 3), (7, 37, 100, 256, 3), (5, 130, 130, 136, 1), (8, 300, 300, 256, 1), (3, 200, 333, 256, 2)])
def test_head_sizes_above_128(G, Sq, Skv, D, mask):
    _run(4, 4 * G, 4, Sq, Skv, D, mask)
    _run(24, 4 * G, 4, Sq, Skv, D, mask)  # several items per CTA


@pytest.mark.parametrize("G,heads", [(4, 1), (4, 8), (7, 14), (3, 1)])
@pytest.mark.parametrize("D", [64, 128])
def test_bias(G, heads, D):
    Hkv = 2
    Hq, B, Sq, Skv = G * Hkv, 3, 75, 141
    heads = 1 if heads == 1 else Hq
    w = wl.attention_workload("t", 84, B, Hq, Hkv, Sq, Skv, D, wl.MASK_CAUSAL, 0.1, "bf16")
    bias = wl.normal_tensor(wl.seed_for(84, "b"), (B, heads, Sq, Skv), "f32").values.copy()
    bias[:, :, ::5, 3:40] = -np.inf
    got = binding.attn_fused_bias(to_device(w.q), to_device(w.k), to_device(w.v), torch.from_numpy(bias.astype(np.float32)).cuda(),
                                  wl.MASK_CAUSAL, None, 0.1)
    binding.check_status()
    assert_close_bf16(got, oracle.attn_bias(w.q.values, w.k.values, w.v.values, bias.astype(np.float64), wl.MASK_CAUSAL, None, 0.1))


def test_padded_values_do_not_reach_unused_rows_or_results():
    """NaN in the caller's padding; tiles with rows out of use, several items per CTA."""
    B, Hq, Hkv, Sq, Skv = 40, 14, 2, 60, 200
    for D in (64, 128):
        w = wl.attention_workload("t", 85, B, Hq, Hkv, Sq, Skv, D, wl.MASK_PADDING, 0.125, "bf16", lens_range=(1, Skv))
        w.lens = np.array(([150, 1, 64, 200] * B)[:B], dtype=np.int32)
        q, k, v = to_device(w.q), to_device(w.k), to_device(w.v)
        for b in range(B):
            k[b, :, w.lens[b]:] = float("nan")
            v[b, :, w.lens[b]:] = float("nan")
        got = binding.attn_fused(q, k, v, wl.MASK_PADDING, torch.from_numpy(w.lens).cuda(), 0.125)
        binding.check_status()
        assert_close_bf16(got[:8], oracle.attn(w.q.values[:8], w.k.values[:8], w.v.values[:8], wl.MASK_PADDING, w.lens[:8], 0.125))
        assert torch.isfinite(got.float()).all()
