"""The static tile schedule of the single persistent launch, checked on the CPU: every M-block covered once
by every column tile of every phase, no deadlock for any number of CTA pairs and vector workers, counters
end at their thresholds."""
import numpy as np
import pytest

from paper_2605_23764_b200 import binding, build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _expected_items(counts, d, F, is_bwd, n_shared=0):
    mblocks = (counts + 127) // 128
    units = (mblocks + 1) // 2
    # an expert merges its last two units, in every row-space phase, when its M-block count is odd, at least 3, and the last
    # block holds <= 64 rows -- unless it is a shared one
    Ep = len(counts)
    merged = units - ((mblocks % 2 == 1) & (mblocks >= 3) & (counts - (mblocks - 1) * 128 <= 64) & (np.arange(Ep) < Ep - n_shared))
    if not is_bwd:
        return int(merged.sum()) * ((F + 127) // 128 + (d + 255) // 256)
    return (int(merged.sum()) * ((F + 255) // 256) + Ep * ((d + 255) // 256) +
            int(merged.sum()) * ((d + 255) // 256) + Ep * ((2 * F + 255) // 256))


@pytest.mark.parametrize("is_bwd", [0, 1])
@pytest.mark.parametrize("workers", [(1, 1), (3, 2), (74, 592), (74, 2368)])
def test_schedule_is_sound(is_bwd, workers):
    rng = np.random.default_rng(7 + is_bwd)
    cases = [
        rng.integers(0, 700, 24),                      # mixed sizes
        np.array([0, 0, 5, 0, 1300, 0, 129, 0]),       # empty experts, one large
        np.array([3000]),                              # a single expert
        np.zeros(6, int),                              # nothing routed at all
        np.full(64, 128),                              # exactly one M-block each
        np.array([300, 257, 320, 576]),                # every expert ends in a merged item
        np.array([300, 257, 320, 577]),                # and its neighbour, whose last block holds 65 rows
        np.array([384, 321, 640, 385]),                # full last blocks / even counts: nothing merges
    ]
    d, F = 520, 272
    for counts in cases:
        T = max(1, int(counts.sum()) // 2)
        rc, stats = binding.moe_debug_simulate_schedule(counts, T, 2, 0, d, F, is_bwd, *workers)
        assert rc == 0, (counts.tolist(), rc)
        assert stats[0] == _expected_items(counts, d, F, is_bwd)


@pytest.mark.parametrize("is_bwd", [0, 1])
@pytest.mark.parametrize("d", [8, 256, 568, 576, 2040, 2048, 7168])
def test_every_operator_merges_at_every_reduction_length(is_bwd, d):
    counts = np.array([300, 257, 320, 577, 321, 384, 0, 64])
    rc, stats = binding.moe_debug_simulate_schedule(counts, 1111, 2, 0, d, 272, is_bwd, 74, 592)
    assert rc == 0 and stats[0] == _expected_items(counts, d, 272, is_bwd)


def test_balanced_units_cover_every_mblock_once():
    """Token-column tiles: the units of an expert (one or two M-blocks each) partition its M-blocks, and a
    lone M-block never comes last when there are three or more (the simulation checks the coverage)."""
    for n in list(range(0, 1200, 7)) + [128, 256, 257, 384, 385, 512, 640, 641]:
        counts = np.array([n, 1, 300])
        for is_bwd in (0, 1):
            rc, stats = binding.moe_debug_simulate_schedule(counts, 64, 2, 1, 384, 48, is_bwd, 5, 7)
            assert rc == 0, (n, rc)


def test_training_config_schedule():
    """Config-4-like counts (256 experts, ~256 rows each) with the launch's real worker counts."""
    rng = np.random.default_rng(4)
    counts = rng.binomial(65536, 1 / 256, 256)
    for is_bwd in (0, 1):
        rc, stats = binding.moe_debug_simulate_schedule(counts, 8192, 8, 0, 7168, 2048, is_bwd, 74, 1184)
        assert rc == 0


def test_skewed_config_schedule():
    """Config-3-like counts: Zipf popularity, empty experts, one expert with thousands of rows."""
    rng = np.random.default_rng(3)
    q = (np.arange(128) + 1.0) ** -1.2
    counts = rng.multinomial(131072, q / q.sum())
    counts[-4:] = 0
    rc, stats = binding.moe_debug_simulate_schedule(counts, 16384, 8, 0, 4096, 1536, 0, 74, 1184)
    assert rc == 0


def test_layout_takes_the_kernels_where_a_cluster_does_not_fit():
    def blocks(*a, **kw):
        return binding.moe_debug_layout_blocks(*a, **kw)
    assert blocks(123, 8, 64) == 1 and blocks(124, 8, 64) == 8           # 984 and 992 slots
    assert blocks(1024, 8, 64) == 8 and blocks(1025, 8, 64) == 16        # 1024 slots to a block, and one token more
    assert blocks(8192, 8, 256) == 16 and blocks(8193, 8, 256) == 0      # 65536 slots, and one token more
    assert blocks(124, 8, 384) == 8 and blocks(124, 8, 385) == 0
    for T in (124, 1024):
        assert blocks(T, 8, 64, fits16=False) == 8 and blocks(T, 8, 64, fits8=False) == 0
    for T in (1025, 8192):
        assert blocks(T, 8, 64, fits8=False) == 16 and blocks(T, 8, 64, fits16=False) == 0
    assert blocks(123, 8, 64, fits8=False, fits16=False) == 1


@pytest.mark.parametrize("is_bwd", [0, 1])
@pytest.mark.parametrize("T", [257, 300, 320, 321, 576, 1060, 4096, 4100])
def test_shared_experts_do_not_merge(is_bwd, T):
    """A call's operand ring is the same for 4096 and for 4100 tokens: a shared expert's short last block merges with nothing."""
    for n_shared in (1, 2):
        counts = np.array([128, 300, 0, 250] + [T] * n_shared)
        rc, stats = binding.moe_debug_simulate_schedule(counts, T, 2, n_shared, 264, 272, is_bwd, 74, 592)
        assert rc == 0 and stats[0] == _expected_items(counts, 264, 272, is_bwd, n_shared)


def test_operand_ring_by_tokens_and_largest_expert():
    ring = binding.moe_debug_ring
    assert [ring(0, T, T)[0] for T in (32, 128, 129, 160, 161, 192, 193, 224, 225, 256)] == [11, 8, 7, 7, 7, 7, 6, 6, 6, 6]
    assert [ring(1, T, T)[0] for T in (32, 128, 129, 160, 161, 192, 193, 224, 225, 256)] == [11, 8, 8, 8, 7, 7, 6, 6, 6, 6]
    for is_bwd in (0, 1):
        for T in (1, 31, 33, 127, 129, 160, 192, 255, 257, 4096, 16384):
            # ids repeated in a token give an expert more rows than there are tokens
            for largest in {1, 32, 33, T, T + 1, 128, 129, 160, 161, 256, 257, 300, 8 * T}:
                for merged in (False, True) if largest > 256 else (False,):
                    stages, tokens = ring(is_bwd, T, largest, merged)
                    # the widest tile there can be: the largest expert's rows up to 256, or a merged item's 128 + 128 + 64
                    need = 320 if merged else min(256, (largest + 31) // 32 * 32)
                    assert tokens >= need and stages >= 5, (is_bwd, T, largest, merged, stages, tokens)
            assert ring(is_bwd, T, min(T, 128))[0] >= 8   # as deep as the largest expert allows, whatever the call's size


@pytest.mark.parametrize("is_bwd", [0, 1])
@pytest.mark.parametrize("pairs", [1, 2, 5, 74])
@pytest.mark.parametrize("d,F", [(4096, 8), (2048, 64), (256, 520)])   # items of one, one and nine k-blocks of F
def test_schedule_with_batches_of_tickets(is_bwd, pairs, d, F):
    """Many short items: pairs hold up to eight of them whose events are not met yet; long experts and shared ones among them."""
    rng = np.random.default_rng(pairs)
    counts = np.concatenate([rng.integers(0, 90, 96), [1000, 640, 640]])   # the last two: shared experts
    rc, stats = binding.moe_debug_simulate_schedule(counts, 640, 8, 2, d, F, is_bwd, pairs, 3)
    assert rc == 0
