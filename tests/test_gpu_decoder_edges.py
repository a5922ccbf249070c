"""The decoder at the key counts where it changes its way of working: groups for one warp or a whole block, the group's
slice of dense_out in shared memory or its entries alone, all streams together or one after the other.  Decoded sums
and the model update (three arrays, and packed) bit-equal to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
import gpu_util as G
from paper_2112_04291_b200 import binding

pytestmark = pytest.mark.gpu

TILE = 16384
HYPER = (1e-3, 0.9, 0.999, 1e-8)


def _streams(n, counts, workers, seed, tau=128, group_log2=14, l=2):
    """One stream per worker with exactly counts[g] kept keys in group g; half of the keys shared with the worker before."""
    rng = np.random.default_rng(seed)
    out, prev = [], None
    po = oracle.params(1.3 if tau == 128 else 1.9, tau, l, group_log2)
    for w in range(workers):
        v = np.zeros(n, np.float32)
        keys = []
        for g, c in enumerate(counts):
            lo, span = g << group_log2, min(1 << group_log2, n - (g << group_log2))
            c = min(c, span)
            if prev is None:
                k = rng.choice(span, c, replace=False)
            else:
                old = rng.choice(prev[g], c // 2, replace=False)
                k = np.concatenate([old, rng.choice(np.setdiff1d(np.arange(span), old), c - c // 2, replace=False)])
            keys.append(k)
            v[lo + k] = (rng.uniform(0.5, 2.0, c) * rng.choice([-1.0, 1.0], c)).astype(np.float32)
        prev = keys
        rc, s = oracle.compress(v, po)
        assert rc == 0 and int(np.frombuffer(s[24:32].tobytes(), np.uint64)[0]) == sum(len(k) for k in keys)
        out.append(s)
    return out, po, binding.params(po.base, tau, l, group_log2)


def _check(n, counts, workers, seed, tau=128, update=True, group_log2=14, l=2):
    streams, po, pg = _streams(n, counts, workers, seed, tau, group_log2, l)
    rng = np.random.default_rng(seed + 1)
    binding.ensure_workspace(n, pg)
    dev = [G.to_dev(np.concatenate([s, np.zeros(-s.size % 16 + 16, np.uint8)])) for s in streams]
    sizes = [s.size for s in streams]
    want = rng.standard_normal(n).astype(np.float32)
    buf = G.Guarded(4 * n)
    dense = buf.view.view(torch.float32)
    dense.copy_(torch.from_numpy(want))
    for s in streams:
        assert oracle.decompress_accumulate(s, n, po, want) == 0
    assert binding.decompress_accumulate_batch(dev, sizes, n, pg, dense) == 0
    assert binding.decode_status() == 0 and buf.intact()
    assert np.array_equal(dense.cpu().numpy(), want)
    if not update:
        return
    theta, m, v = (rng.standard_normal(n).astype(np.float32), (rng.standard_normal(n) * 1e-3).astype(np.float32),
                   (rng.standard_normal(n) ** 2 * 1e-6).astype(np.float32))
    arrays = [torch.from_numpy(x.copy()).to(G.dev()) for x in (theta, m, v)] + [torch.zeros(n, dtype=torch.float32, device=G.dev())]
    packed = torch.stack(arrays, dim=1).reshape(-1)
    assert oracle.sparse_adam_update(streams, n, po, *HYPER, theta, m, v) == 0
    assert binding.sparse_adam_update_batch(dev, sizes, n, pg, binding.Adam(*HYPER), arrays[3], *arrays[:3]) == 0
    if group_log2 <= 14:
        assert binding.sparse_adam_update_packed_batch(dev, sizes, n, pg, binding.Adam(*HYPER), packed) == 0
    assert binding.decode_status() == 0
    packed = packed.reshape(n, 4)
    for i, x in enumerate((theta, m, v, np.zeros(n, np.float32))):
        assert np.array_equal(arrays[i].cpu().numpy(), x), i
        assert group_log2 > 14 or np.array_equal(packed[:, i].cpu().numpy(), x), i


# one stream: warp / block (256), sweep of the update (768, packed 2048), slice of dense_out (1536 on so few entries), words of a blob that fit
# the stage (4096 words at 8 + 2 + up to 8 bits a key), keys that fit the lists (8192); the last group is ragged
@pytest.mark.parametrize("count", [1, 32, 33, 255, 256, 257, 767, 768, 1535, 1536, 2047, 2048, 2049, 4096, 4097, 8184, 8192, 8193, TILE])
def test_one_stream(count):
    _check(3 * TILE - 5, [count, 0, max(1, count - 1)], 1, 100 + count)


# several streams: the same sizes for all streams of a group together (warp / block: 248)
@pytest.mark.parametrize("workers,count", [(2, 1), (2, 124), (2, 125), (3, 83), (4, 62), (4, 63), (8, 31), (8, 32), (4, 192), (4, 383), (4, 384), (4, 512),
                                           (3, 700), (2, 2048), (8, 256), (4, 2048), (4, 2049), (8, 1023), (8, 1025), (5, 2100), (3, 9000), (2, TILE)])
def test_several_streams(workers, count):
    _check(3 * TILE + 1, [count, 2, count + 1, 1], workers, 300 + 10 * workers + count)


# codes are checked against tau only where tau leaves some out
def test_tau_below_the_largest():
    _check(2 * TILE + 3, [900, 40, 1], 1, 7, tau=33)
    _check(2 * TILE + 3, [900, 40, 1], 4, 8, tau=33)


# many groups per block: one warp takes up to 1024 keys of one stream; a few large groups among many small ones are shared
@pytest.mark.parametrize("workers", [1, 3])
def test_many_groups_per_block(workers):
    groups = 2400
    rng = np.random.default_rng(workers)
    counts = rng.integers(0, 4, groups)
    counts[300:330] = [1023, 1024, 1025] * 10
    counts[1000:1012] = 300
    _check(groups * TILE - 9, counts.tolist(), workers, 40 + workers, update=False)


# groups wider than the slice of dense_out: all streams' keys in one list of up to 2^14, stream by stream, and streams beyond a list; blobs
# in the stage (4096 words together, 2048 one at a time) or read where they are
@pytest.mark.parametrize("group_log2", [15, 17, 20])
@pytest.mark.parametrize("workers,count", [(1, 1), (1, 700), (1, 5000), (1, 16384), (1, 16385), (1, 30000), (2, 300), (2, 4000), (3, 5464), (8, 200), (8, 1500), (5, 2048), (8, 2100)])
def test_wide_groups(workers, count, group_log2):
    _check((3 << group_log2) - 5, [count, 0, max(1, count - 1)], workers, 700 + workers + count, group_log2=group_log2)


# streams that fail in one group are left out there as a whole, the others not
@pytest.mark.parametrize("group_log2,count", [(14, 40), (14, 90), (14, 170), (14, 400), (16, 300), (16, 6000)])
def test_failed_streams_are_left_out(group_log2, count):
    n, workers = (3 << group_log2) - 5, 6
    streams, po, pg = _streams(n, [count, count + 1, count], workers, 900 + count, group_log2=group_log2)
    sound = np.random.default_rng(5).standard_normal(n).astype(np.float32)
    dense = torch.from_numpy(sound.copy()).to(G.dev())
    for w in (0, 2, 3, 5):
        assert oracle.decompress_accumulate(streams[w], n, po, sound) == 0
    for w in (1, 4):                                       # the first deltas of group 1 become 0
        s = streams[w] = streams[w].copy()
        cnt, off = (int(x) for x in np.frombuffer(s[72:80].tobytes(), np.uint32))
        cnt &= 0xFFFFFF
        bits = np.unpackbits(s[4 * off:4 * off + 2 * cnt + 16])
        bits[10 * cnt:10 * cnt + 40] = 0
        s[4 * off:4 * off + 2 * cnt + 16] = np.packbits(bits)
    status = [oracle.decompress_accumulate(s, n, po, np.zeros(n, np.float32)) for s in streams]
    assert [bool(x) for x in status] == [False, True, False, False, True, False]
    binding.ensure_workspace(n, pg)
    dev = [G.to_dev(np.concatenate([s, np.zeros(-s.size % 16 + 16, np.uint8)])) for s in streams]
    assert binding.decompress_accumulate_batch(dev, [s.size for s in streams], n, pg, dense) == 0
    assert binding.decode_status() == status[1]
    lo, hi = 1 << group_log2, 2 << group_log2
    assert np.array_equal(dense.cpu().numpy()[lo:hi], sound[lo:hi])


# groups of several streams for teams of one, two and four warps (at most 6 bytes an entry and the blobs in 4, 8 and 16 KiB; by ranks what 24 KiB
# hold; groups as unlike as these 249 keys at most) and beyond, next to each other in one block; many groups to a block, few, and one
@pytest.mark.parametrize("groups,workers,l,group_log2", [(2700, 8, 2, 14), (740, 2, 2, 14), (740, 3, 1, 14), (740, 4, 5, 14), (740, 8, 2, 14),
                                                         (740, 8, 5, 10), (740, 5, 3, 11), (290, 2, 5, 14), (290, 8, 1, 14)])
def test_teams_of_warps(groups, workers, l, group_log2):
    rng = np.random.default_rng(workers + l)
    totals = rng.choice([0, 8, 60, 64, 65, 230, 248, 256, 380, 470, 480, 490, 500, 512, 540, 767, 768, 769, 940, 960, 1000, 1500, 1535, 1536, 1600], groups)
    if groups > 1000:
        totals[rng.random(groups) < 0.7] = 0
    counts = np.minimum(-(-totals // workers), 1 << group_log2)
    _check((groups << group_log2) - 9, counts.tolist(), workers, 500 + workers, group_log2=group_log2, l=l, update=groups == 740)


@pytest.mark.parametrize("workers,count", [(2, 200), (3, 110), (8, 30), (8, 100), (8, 190), (8, 300)])
def test_teams_on_groups_of_two_tiles(workers, count):
    _check((40 << 15) - 9, [count, count + 1] * 20, workers, 600 + count, group_log2=15)


# alike groups of more than 1000 keys over all streams, a few to a block: over the slice of dense_out, those of 2^15 by teams of four warps; keys at the
# edges of 32 and of the groups, streams that fail in one group (ranks: test_gpu_decoder_ranks.py)
@pytest.mark.parametrize("workers,count,group_log2", [(6, 170, 14), (3, 500, 14), (8, 130, 15), (7, 200, 11)])
def test_teams_of_four_warps(workers, count, group_log2):
    groups, size = 620, 1 << group_log2
    n = groups * size - 3
    rng = np.random.default_rng(count)
    po, pg = oracle.params(1.3, 128, 2, group_log2), binding.params(1.3, 128, 2, group_log2)
    edges = np.array([0, 31, 32, 63, 127, 128, size // 2, size - 33, size - 32, size - 4])
    streams = []
    for w in range(workers):
        v = np.zeros(n, np.float32)
        for g in range(groups):
            k = np.unique(np.concatenate([rng.choice(edges, 6, replace=False), rng.integers(0, size - 4, count)]))
            v[g * size + k] = (rng.uniform(0.5, 2.0, k.size) * rng.choice([-1.0, 1.0], k.size)).astype(np.float32)
        rc, s = oracle.compress(v, po)
        assert rc == 0
        streams.append(s)
    bad, group = (1, 2), 300
    lo, hi = group * size, (group + 1) * size
    dense0 = rng.standard_normal(n).astype(np.float32)
    want, sound = dense0.copy(), dense0.copy()
    for w, s in enumerate(streams):
        assert oracle.decompress_accumulate(s, n, po, want) == 0
        assert w in bad or oracle.decompress_accumulate(s, n, po, sound) == 0
    binding.ensure_workspace(n, pg)

    def decode():
        dense = torch.from_numpy(dense0.copy()).to(G.dev())
        dev = [G.to_dev(np.concatenate([s, np.zeros(-s.size % 16 + 16, np.uint8)])) for s in streams]
        assert binding.decompress_accumulate_batch(dev, [s.size for s in streams], n, pg, dense) == 0
        return dense.cpu().numpy(), binding.decode_status()

    got, status = decode()
    assert status == 0 and np.array_equal(got, want)
    for w in bad:                                          # the first deltas of one group become 0
        s = streams[w] = streams[w].copy()
        cnt, off = (int(x) for x in np.frombuffer(s[64 + 8 * group:72 + 8 * group].tobytes(), np.uint32))
        cnt &= 0xFFFFFF
        bits = np.unpackbits(s[4 * off:4 * off + 2 * cnt + 16])
        bits[10 * cnt:10 * cnt + 40] = 0
        s[4 * off:4 * off + 2 * cnt + 16] = np.packbits(bits)
    want[lo:hi] = sound[lo:hi]
    got, status = decode()
    assert status == oracle.decompress_accumulate(streams[bad[0]], n, po, np.zeros(n, np.float32)) != 0
    assert np.array_equal(got, want)
