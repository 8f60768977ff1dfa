"""GPU parity: the decode step whose lengths are written by the kernel right before it in the stream.  The step looks at the lengths
before that kernel has completed, to ask for its first blocks; what counts are the lengths afterwards.  A linear with the
identity as weights writes them (16-bit patterns through bf16, exact), over lengths that are different, longer or shorter; many
rounds in a row, with one, few and more than 32 sequences, pieces merged in one level, by CTA and in two levels."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import assert_close_bf16, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,Smax,D,splits", [(1, 8, 2, 3000, 128, 16), (7, 12, 12, 900, 64, 16), (32, 8, 8, 300, 128, 16),
                                                    (40, 8, 2, 300, 64, 16), (2, 8, 2, 6000, 64, 86), (3, 4, 1, 9000, 128, 256)])
def test_lengths_written_by_the_previous_kernel(B, Hq, Hkv, Smax, D, splits):
    w = wl.decode_workload("t", 95, B, Hq, Hkv, Smax, D, splits, D ** -0.5, (128, Smax))
    q, k, v = to_device(w.q), to_device(w.k_cache), to_device(w.v_cache)
    rng = np.random.RandomState(B)
    # lengths as the bits of pairs (low, high) of bf16 numbers: 128 and more are normal numbers, which the product with 1 keeps
    choices = [np.full(B, Smax, np.int32), rng.randint(128, Smax + 1, B).astype(np.int32), np.full(B, 128, np.int32)]
    want = [oracle.attn_decode(w.q.values, w.k_cache.values, w.v_cache.values, c, w.scale) for c in choices]
    x = [torch.zeros((1, 128), dtype=torch.int16, device="cuda") for _ in choices]
    for t, c in zip(x, choices):
        t[0, :2 * B:2] = torch.from_numpy(c.astype(np.int16)).cuda()
    eye = torch.eye(128, device="cuda").bfloat16()
    holder = torch.zeros((1, 128), dtype=torch.bfloat16, device="cuda")
    lens = holder.view(torch.int32)[0, :B]
    ws = torch.empty(binding.attn_decode_workspace_bytes(B, Hq, D, splits), dtype=torch.uint8, device="cuda")
    binding.attn_decode_workspace_init(ws)
    outs = [torch.full_like(q, float("nan")) for _ in range(30)]  # nothing else is launched in between
    for i in range(30):
        binding.linear_act(x[i % 3].view(torch.bfloat16), eye, act=binding.ACT_NONE, w_layout=binding.W_NK, out=holder)
        binding.attn_decode_splitkv(q, k, v, lens, splits, w.scale, out=outs[i], workspace=ws)
    binding.check_status()
    assert torch.equal(lens.cpu(), torch.from_numpy(choices[29 % 3]))
    for i in range(3):
        assert_close_bf16(outs[i], want[i])
    for i in range(3, 30):
        assert torch.equal(outs[i], outs[i - 3])
