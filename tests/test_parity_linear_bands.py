"""GPU parity: the order of the CTA pairs' tiles.  Several bands of row tiles with a shorter last one, of 16 row tiles and (long K) of
eight; and the last round's tiles in halves, for the gated form in both weight layouts, with the second half of the last column tile
whole, partly or wholly beyond N.  Small K: every element against the fp64 oracle; long K: rows of every band.  Outputs between guard
bytes; the host-side plans say that the shapes take what they are here for."""
import numpy as np
import pytest
import torch

import oracle
import plans
from paper_2604_16498_b200 import binding, workloads as wl
from test_parity_linear_swiglu import assert_close_bf16 as assert_close_gated
from util import Guarded, assert_close_bf16, to_device

# (M, N, K): (row tiles, column tiles, row tiles of a band, halved tiles)
PLAIN = {
    (4252, 4360, 136): (17, 18, 16, 10),   # a last band of one row tile; halves in it; 8 columns in the last column tile
    (8350, 4552, 64): (33, 18, 16, 2),     # two full bands and one row tile; halves, the last one partly beyond N
    (5000, 4200, 72): (20, 17, 16, 0),     # a last band of four
}
GATED = {
    (4252, 2072, 64): (17, 17, 16, 0),     # two bands; 24 outputs in the last column tile
    (1250, 1832, 136): (5, 15, 1, 1),      # one halved tile, its second half wholly beyond N
    (1250, 1896, 136): (5, 15, 1, 1),      # its second half partly beyond N
    (1790, 1920, 64): (7, 15, 1, 31),      # two rows of halved tiles, whole ones
    (1790, 1856, 72): (7, 15, 1, 31),      # the last column tile's second half begins at N
    (900, 2344, 136): (4, 19, 16, 2),      # halves in a band: rows of the last column tile
    (4352, 2336, 64): (17, 19, 16, 27),    # and in the last band
}
LONG_PLAIN = {(2600, 4360, 12288): (11, 18, 8, 0)}  # bands of eight row tiles, three in the last
LONG_GATED = {(2600, 2056, 12288): (11, 17, 8, 0)}


def test_the_shapes_take_the_plans_they_are_here_for():
    for shapes, gated in ((PLAIN, False), (GATED, True), (LONG_PLAIN, False), (LONG_GATED, True)):
        for shape, want in shapes.items():
            got = plans.pair(*shape, gated)
            assert got == want, (shape, got)


def test_a_band_has_eight_row_tiles_or_as_many_as_48_mb_hold_up_to_sixteen():
    for K in (8, 64, 768, 4096, 6144, 6152, 8192, 12288, 12296, 53248):
        rows = plans.pair(100000, 8192, K)[2]
        assert rows == max(8, min(16, (48 << 20) // (512 * K)))
    assert plans.pair(100000, 4096, 64)[2] == 1 and plans.pair(100000, 4097, 64)[2] == 16


def _draw(seed, M, N, K, mats):
    x = wl.normal_tensor(wl.seed_for(seed, "x"), (M, K), "bf16")
    return [x] + [wl.normal_tensor(wl.seed_for(seed, n), (K, N), "bf16", std=K ** -0.5) for n in "wb"[:mats]]


def _weight(w, layout):
    return to_device(w) if layout == binding.W_KN else to_device(w).t().contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [binding.W_KN, binding.W_NK])
@pytest.mark.parametrize("shape", PLAIN)
def test_plain(shape, layout):
    M, N, K = shape
    x, w = _draw(87, M, N, K, 1)
    g = Guarded((M, N), torch.bfloat16)
    binding.linear_act(to_device(x), _weight(w, layout), act=binding.ACT_NONE, w_layout=layout, out=g.tensor)
    binding.check_status()
    assert_close_bf16(g.tensor, x.values @ w.values)
    g.assert_intact()


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [binding.W_KN, binding.W_NK])
@pytest.mark.parametrize("shape", GATED)
def test_gated(shape, layout):
    M, N, K = shape
    x, wg, wu = _draw(88, M, N, K, 2)
    g = Guarded((M, N), torch.bfloat16)
    binding.linear_swiglu(to_device(x), _weight(wg, layout), _weight(wu, layout), layout, out=g.tensor)
    binding.check_status()
    assert_close_gated(g.tensor, oracle.linear_swiglu(x.values, wg.values, wu.values, 0))
    g.assert_intact()


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [binding.W_KN, binding.W_NK])
@pytest.mark.parametrize("gated", [False, True])
def test_long_k(gated, layout):
    """Rows of every band against the same product in 64 bits."""
    (M, N, K), = LONG_GATED if gated else LONG_PLAIN
    gen = torch.Generator(device="cuda").manual_seed(89)
    x, *ws = (torch.randn(s, generator=gen, device="cuda").mul_(std).bfloat16() for s, std in (((M, K), 1.0),) + (((K, N), K ** -0.5),) * (1 + gated))
    rows = torch.tensor([0, 127, 128, 255, 256, 1023, 1791, 2047, 2048, 2049, 2303, 2304, 2559, 2560, M - 1], device="cuda")
    g = Guarded((M, N), torch.bfloat16)
    given = [w if layout == binding.W_KN else w.t().contiguous() for w in ws]
    want = [x[rows].double() @ w.double() for w in ws]
    if gated:
        binding.linear_swiglu(x, *given, layout, out=g.tensor)
        want = [torch.nn.functional.silu(want[0]) * want[1]]
    else:
        binding.linear_act(x, *given, act=binding.ACT_NONE, w_layout=layout, out=g.tensor)
    binding.check_status()
    (assert_close_gated if gated else assert_close_bf16)(g.tensor[rows], want[0].cpu().numpy())
    assert torch.isfinite(g.tensor.float()).all()
    g.assert_intact()
