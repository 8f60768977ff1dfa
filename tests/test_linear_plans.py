"""The host-side plans of the linears over many shapes: what the kernels take for granted about them.  No GPU."""
import random

import plans
from test_parity_linear_split import SHAPES as SPLIT_SHAPES
from test_parity_linear_w8_edges import SHAPES as W8_SHAPES


def test_int8_linear_has_a_ring_stage_for_every_converter_group_and_fits_shared_memory():
    rng = random.Random(5)
    shapes = [(M, N, K) for M in range(1, 400) for N, K in ((128, 1040), (128, 4096), (384, 512), (4096, 14336), (20000, 4096))]
    shapes += [(rng.randint(1, 20000), 8 * rng.randint(1, 4000), 16 * rng.randint(1, 1000)) for _ in range(20000)]
    fewest = 99
    for sms in (148, 132, 16):
        for M, N, K in shapes:
            p = plans.w8(M, N, K, sms)
            assert p is not None
            assert p.stages >= p.groups and p.groups in (3, 4)
            assert 16 <= p.nt <= 192 and p.nt % 16 == 0 and p.nt * p.tiles_t >= M > p.nt * (p.tiles_t - 1)
            assert p.tiles == p.tiles_t * ((N + 127) // 128)
            kblocks = (K + 63) // 64
            assert p.split == 1 or (kblocks >= 2 * p.split and p.tiles * p.split <= sms)
            assert p.split == 1 or p.own4 * p.split * 4 >= p.nt
            # ring, exchange buffer, output staging, barriers, alignment slack
            assert p.stages * (8192 + 128 * p.nt) + p.recv_bytes + 16384 + 376 + 1024 <= 227 * 1024
            fewest = min(fewest, p.stages)
    assert fewest == 3  # 192 tokens and clusters of eight: the case that has just enough


def test_a_plan_exists_only_below_2_31_tiles():
    assert plans.w8((1 << 31) - 200, 64 * 8 * 400, 16) is None


def test_the_shapes_of_the_parity_tests_take_the_paths_they_are_there_for():
    for shape, want in W8_SHAPES.items():
        p = plans.w8(*shape)
        assert (p.nt, p.tiles, p.split, p.groups, p.stages) == want, shape
    for shape, want in SPLIT_SHAPES.items():
        assert plans.split(*shape) == want, shape
