"""GPU parity: the int8-weight linear at the edges of its tiles (token shares of 16, features of 128, k-blocks of 64), of the
split of K over clusters and of the persistent schedule, against the fp64 oracle; tolerances as in test_parity_linear_w8."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_16498_b200 import binding, workloads as wl
from util import Guarded, assert_close_bf16, to_device

pytestmark = pytest.mark.gpu


# (M, N, K): (tokens per tile, tiles, CTAs per tile, converter groups, ring stages) on 148 SMs (test_linear_plans.py checks that)
SHAPES = {
    (1, 8, 16): (16, 1, 1, 3, 16), (2, 136, 80): (16, 2, 1, 3, 16),           # one and two k-blocks, ragged features
    (15, 768, 784): (16, 6, 4, 3, 16), (17, 264, 4096): (32, 3, 8, 3, 16),    # a token share just below / above 16
    (191, 128, 1040): (192, 1, 8, 3, 3), (192, 384, 512): (192, 3, 4, 3, 4),  # the largest single tile; no more stages than groups
    (193, 1000, 2064): (112, 16, 8, 3, 6), (385, 128, 4096): (144, 3, 8, 3, 5),  # two and three token tiles over clusters
    (1000, 2056, 192): (176, 102, 1, 3, 6), (1000, 2048, 3088): (176, 96, 1, 3, 6),  # most of one round, short and long k-loop
    (4001, 3080, 208): (176, 575, 1, 3, 6), (4001, 3080, 784): (176, 575, 1, 3, 6),  # four rounds of the persistent schedule
    (4001, 3080, 3088): (176, 575, 1, 4, 6),                                  # the same with four converter groups
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("extras", [True, False])
def test_edges(shape, extras):
    M, N, K = shape
    x = wl.normal_tensor(wl.seed_for(91, "x"), (M, K), "f16")
    wq = wl.uniform_int(wl.seed_for(91, "w"), N * K, -127, 127).reshape(N, K).astype(np.int8)
    scale = ((0.5 + wl.splitmix64(wl.seed_for(91, "lens"), N) % np.uint64(1000) / 1000.0) / (73.6 * np.sqrt(K))).astype(np.float32)
    b = wl.normal_tensor(wl.seed_for(91, "b"), (N,), "f16", std=0.5)
    r = wl.normal_tensor(wl.seed_for(91, "q"), (M, N), "f16")
    act = binding.ACT_GELU_ERF if extras else binding.ACT_RELU
    g = Guarded((M, N), torch.float16)
    binding.linear_act_w8a16(to_device(x), torch.from_numpy(wq).cuda(), torch.from_numpy(scale).cuda(),
                             to_device(b) if extras else None, to_device(r) if extras else None, act, out=g.tensor)
    binding.check_status()
    step = 1 if M <= 200 else 7 if M <= 1000 else 29
    rows = np.unique(np.concatenate([np.arange(0, M, step), [M - 1]]))
    ref = oracle.linear_w8(x.values[rows], wq.astype(np.float64), scale.astype(np.float64), b.values if extras else None,
                           r.values[rows] if extras else None, act)
    assert_close_bf16(g.tensor[torch.from_numpy(rows).cuda()], ref)
    assert torch.isfinite(g.tensor.float()).all()
    g.assert_intact()
