"""GPU parity: decode over sequences cut into more than 32 pieces whose warps merge in shared memory first (33 to 140 pieces,
at most one per worker), at the edges of that rule: 33 pieces, a kv head that starts inside a CTA, one and several sequences
of very different lengths, a sequence with a single piece or none beside a long one, 140 pieces; and just beyond, where they
merge on two levels in the workspace (141 and 256 pieces, more pieces than workers).  fp64 oracle; the workspace's counters
are left at zero, and a second call gives the same bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import assert_close_bf16, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,Smax,D,splits,lens", [
    (1, 8, 2, 16 * 33, 128, 33, [16 * 33]),
    (1, 6, 2, 16 * 35 + 3, 64, 40, [16 * 35 + 3]),           # 36 pieces: the second kv head starts inside a CTA
    (3, 8, 8, 3000, 64, 43, [3000, 5, 0]),                   # one piece and none beside 38 (pieces of five blocks)
    (2, 32, 8, 9000, 128, 64, [9000, 4321]),
    (1, 8, 1, 16 * 140, 128, 140, [16 * 140]),               # 20 CTAs, the most pieces of the rule
    (1, 8, 1, 16 * 141, 128, 141, [16 * 141]),               # one more: two levels
    (1, 21, 7, 16 * 140, 64, 140, [16 * 140 - 9]),           # 980 pieces for 1036 workers: kv heads that share a CTA
    (1, 4, 1, 16 * 256, 128, 256, [16 * 256]),               # two levels, the most pieces of all
    (5, 8, 8, 2000, 96, 125, [2000, 1999, 1500, 17, 2000]),  # two levels: possibly more pieces than workers
    (30, 8, 8, 600, 128, 36, [600] * 30),                    # the same rule, 5 pieces a sequence
])
@pytest.mark.parametrize("f16", [False, True])
def test_grouped(B, Hq, Hkv, Smax, D, splits, lens, f16):
    d = wl.decode_workload("t", 75, B, Hq, Hkv, Smax, D, splits, D ** -0.5, (1, Smax), dtype="f16" if f16 else "bf16")
    d.lens = np.array(lens, dtype=np.int32)
    q, k, v = to_device(d.q), to_device(d.k_cache), to_device(d.v_cache)
    dl = torch.from_numpy(d.lens).cuda()
    ws = torch.empty(binding.attn_decode_workspace_bytes(B, Hq, D, splits), dtype=torch.uint8, device="cuda")
    binding.attn_decode_workspace_init(ws)
    out = binding.attn_decode_splitkv(q, k, v, dl, splits, d.scale, workspace=ws)
    binding.check_status()
    assert_close_bf16(out, oracle.attn_decode(d.q.values, d.k_cache.values, d.v_cache.values, d.lens, d.scale))
    for _ in range(3):
        again = binding.attn_decode_splitkv(q, k, v, dl, splits, d.scale, workspace=ws)
        assert torch.equal(again, out)
    binding.check_status()
    counters = max(1088 << 10, 68 * B * Hq)  # bytes at the start of the workspace
    assert not ws[:counters].any()
