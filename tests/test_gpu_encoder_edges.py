"""The encoder at the sizes where it changes its way of working: gradients whose tiles are all on the GPU at once (up to
two per SM) and beyond, tiles without, with few and with only kept entries.  Streams byte-equal to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import gpu_util as G
from paper_2112_04291_b200 import binding

pytestmark = pytest.mark.gpu

TILE = 16384


def _check(grads, base, tau=128, l=2):
    n = grads[0].size
    pg, po = binding.params(base, tau, l, 14), oracle.params(base, tau, l, 14)
    binding.ensure_workspace(n, pg)
    cap = min(binding.compress_bound(n, pg), (8 * n + 4096 + 255) & ~255)
    bufs = [G.Guarded(cap, fill=0x5C) for _ in grads]
    dev = [G.to_dev(v) for v in grads]
    for rep in range(2):
        assert binding.compress_batch(dev, pg, [b.view for b in bufs]) == 0
        for v, b in zip(grads, bufs):
            rc, want = oracle.compress(v, po)
            total, d, status = binding.stream_info(b.view)
            assert status == rc == 0 and total == want.size and b.intact()
            assert np.array_equal(b.view[:total].cpu().numpy(), want)


def _tiles(n, counts, seed, small=1e-9):
    """A gradient whose tile t has counts[t % len(counts)] entries far above the threshold of base 1.2, the others far below it."""
    rng = np.random.default_rng(seed)
    v = (rng.standard_normal(n) * small).astype(np.float32)
    for t in range(-(-n // TILE)):
        lo, span = t * TILE, min(TILE, n - t * TILE)
        c = min(span, counts[t % len(counts)])
        k = rng.choice(span, c, replace=False)
        v[lo + k] = (rng.uniform(0.5, 2.0, c) * rng.choice([-1.0, 1.0], c)).astype(np.float32)
    return v


# kept entries of a tile around what a lane, a warp, a block takes in one step, and whole tiles; the last tile ragged
@pytest.mark.parametrize("l", [1, 2, 5])
@pytest.mark.parametrize("counts", [(0, 1), (31, 32, 33), (511, 512, 513), (1023, 1024, 1025), (4095, 4096, 4097), (TILE, TILE - 1, 0)])
def test_kept_entries_of_a_tile(counts, l):
    _check([_tiles(7 * TILE - 11, counts, 10 * l + counts[0])], 1.2, l=l)


# tiles of a launch around the number that is resident at once (two per SM of 148), by one gradient and by several
@pytest.mark.parametrize("workers,tiles", [(1, 1), (1, 2), (1, 148), (1, 149), (1, 295), (1, 296), (1, 297), (2, 148), (2, 149), (8, 37), (8, 38)])
def test_tiles_of_a_launch(workers, tiles):
    _check([_tiles(tiles * TILE - 3, (5 * w, 3, 200), 70 + w) for w in range(workers)], 1.2)


def test_tau_below_the_largest_and_no_entry_kept():
    _check([_tiles(5 * TILE + 1, (700, 3), 5)], 1.5, tau=40)
    _check([np.zeros(5 * TILE + 1, np.float32), _tiles(5 * TILE + 1, (0, 0, 1), 6)], 1.2)


def _check_groups(v, base, group_log2, l=2, tau=128):
    n = v.size
    pg, po = binding.params(base, tau, l, group_log2), oracle.params(base, tau, l, group_log2)
    binding.ensure_workspace(n, pg)
    cap = (binding.compress_bound(n, pg) + 255) & ~255
    buf, dev = G.Guarded(cap, fill=0x5C), G.to_dev(v)
    rc, want = oracle.compress(v, po)
    for rep in range(2):
        assert binding.compress(dev, pg, buf.view) == 0
        total, d, status = binding.stream_info(buf.view)
        assert status == rc == 0 and total == want.size and buf.intact()
        assert np.array_equal(buf.view[:total].cpu().numpy(), want)


# other group sizes: a unit of 4096 entries is up to 16 groups, a group up to 256 units; kept entries around what a warp takes (512),
# what the block takes at a time (4096), and more; tiles without, with few and with only kept entries
@pytest.mark.parametrize("group_log2", [8, 11, 12, 13, 16, 20])
@pytest.mark.parametrize("counts", [(0, 1), (127, 129), (511, 513, 0, 2047), (4095, 4097), (TILE, 0, TILE - 1)])
def test_other_group_sizes(group_log2, counts):
    _check_groups(_tiles(11 * TILE - 5, counts, 40 + counts[0]), 1.2, group_log2, l=1 + counts[0] % 5)


def test_other_group_sizes_many_tiles():
    for group_log2 in (10, 15, 18):
        _check_groups(_tiles(400 * TILE + 7, (3, 0, 0, 0, 40, 900, 0, TILE), group_log2), 1.2, group_log2)


# a few entries carry the sum: a wide margin below the estimate
@pytest.mark.parametrize("group_log2", [10, 14, 17])
def test_tiles_read_again(group_log2):
    n = 310 * TILE + 1
    rng = np.random.default_rng(3)
    v = (rng.standard_normal(n) * 1e-3).astype(np.float32)
    v[::4 * 101] += 50.0
    v[1::3001] *= 30.0
    _check_groups(v, 1.05, group_log2)
    _check_groups(v, 1.1, group_log2)


# every entry kept: units without lists, the longest blobs (what has no room in the workspace: test_gpu_workspace.py)
@pytest.mark.parametrize("group_log2", [9, 14, 16])
def test_blobs_without_room(group_log2):
    n = (1 << 26) + 3
    _check_groups(np.where(np.arange(n) % 7, np.float32(1.0), np.float32(-2.0)).astype(np.float32), 1.2, group_log2, l=5)


# blocks that are not given the sum's nodes by the blocks that form them form them for themselves: with a single look before that, no
# launch gives up and no bit changes
@pytest.mark.parametrize("workers,n,group_log2", [(1, 300 * TILE + 5, 14), (3, 310 * TILE - 9, 14), (1, 300 * TILE + 5, 10), (2, 700 * TILE + 1, 17)])
def test_sum_without_help_from_other_blocks(workers, n, group_log2):
    grads = [_tiles(n, (3, 0, 40, 900), 90 + w) for w in range(workers)]
    pg, po = binding.params(1.2, 128, 2, group_log2), oracle.params(1.2, 128, 2, group_log2)
    binding.ensure_workspace(n, pg)
    bufs = [G.Guarded((binding.compress_bound(n, pg) + 255) & ~255) for _ in grads]
    dev = [G.to_dev(v) for v in grads]
    try:
        binding.debug_set_wait_limits(block_polls=1)
        for rep in range(3):
            assert binding.compress_batch(dev, pg, [b.view for b in bufs]) == 0
            for v, b in zip(grads, bufs):
                rc, want = oracle.compress(v, po)
                total, d, status = binding.stream_info(b.view)
                assert status == rc == 0 and total == want.size and b.intact()
                assert np.array_equal(b.view[:total].cpu().numpy(), want)
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(binding.ensure_workspace(n, pg))


# an estimate that is too high: the entries that the sample looks at (four at each of 32 * 768 regular places) are four times the
# others, the kept ones lie elsewhere, in every third unit of 4096.  Exactly the tiles (other group sizes: units) that hold kept
# entries are read again, and none of them where the same values stand in another order
@pytest.mark.parametrize("group_log2", [9, 14, 16])
def test_estimate_above_the_threshold(group_log2):
    n = 310 * TILE + 1
    rng = np.random.default_rng(4)
    v = (0.5 * rng.choice([-1.0, 1.0], n)).astype(np.float32)
    step = (n >> 2) // (32 * 768)
    at = 4 * (np.arange(32 * 768) * step + step // 2)
    for i in range(4):
        v[at + i] = 2.0
    keys = rng.choice(n - 1, 3000, replace=False)
    keys = keys[((keys >> 12) % 3 == 0) & (keys % 7 != 0)]
    keys = keys[~np.isin(keys >> 2, at >> 2)]
    v[keys] = -3.0
    base = float((np.abs(v, dtype=np.float64).sum() / 2.5) ** (1 / 128))
    again = np.unique(keys >> (14 if group_log2 == 14 else 12)).size
    _check_groups(v, base, group_log2)
    assert binding.listed_tiles(1) == [again] and again > 100
    _check_groups(rng.permutation(v), base, group_log2)
    assert binding.listed_tiles(1) == [0]
