"""The decoder where it has many groups of several streams with about as many keys: teams of four warps that give every key its rank by a bit
for every index of the group.  Aggregation, the update in one launch and on the packed state, and as a pass of its own (more than eight
streams); sound streams, and streams that fail in one group.  What each case is meant to reach is asked of the library's own rules."""
import numpy as np
import pytest
import torch

import oracle
import gpu_util as G
from paper_2112_04291_b200 import binding

pytestmark = pytest.mark.gpu

HYPER = (1e-3, 0.9, 0.999, 1e-8)
BLOCKS_PER_SM = 2


def _blocks():
    return BLOCKS_PER_SM * torch.cuda.get_device_properties(0).multi_processor_count


def _streams(n, group_log2, workers, count, seed):
    """Every stream with `count` random keys in each group (those drawn twice once) and a few at the edges of 32 and of the group."""
    rng = np.random.default_rng(seed)
    size, groups = 1 << group_log2, -(-n >> group_log2)
    edges = np.array([0, 31, 32, 63, 127, 128, size // 2, size - 33, size - 32, size - 4])
    out, po = [], oracle.params(1.3, 128, 2, group_log2)
    for _ in range(workers):
        k = np.concatenate([rng.integers(0, size, (groups, count)), rng.choice(edges, (groups, 6))], axis=1) + size * np.arange(groups)[:, None]
        k = np.unique(k[k < n])
        v = np.zeros(n, np.float32)
        v[k] = (rng.uniform(0.5, 2.0, k.size) * rng.choice([-1.0, 1.0], k.size)).astype(np.float32)
        rc, s = oracle.compress(v, po)
        assert rc == 0 and int(np.frombuffer(s[24:28].tobytes(), np.uint32)[0]) == k.size
        out.append(s)
    return out, po, binding.params(1.3, 128, 2, group_log2)


def _routes(streams, n, group_log2, mode, bulk=True):
    """Who decodes the groups of one launch."""
    groups, blocks = -(-n >> group_log2), _blocks()
    keys, words, kept = np.zeros(groups, np.int64), np.zeros(groups, np.int64), 0
    for s in streams:
        d = np.frombuffer(s[64:64 + 8 * groups].tobytes(), np.uint32).reshape(groups, 2).astype(np.int64)
        keys += d[:, 0] & 0xFFFFFF
        words += np.diff(np.append(d[:, 1], s.size // 4))
        kept += int(np.frombuffer(s[24:28].tobytes(), np.uint32)[0])
    mean = kept // groups
    alike = mean if np.all((2 * keys >= mean) & (keys <= 2 * mean)) else 0
    owned = {groups // blocks, -(-groups // blocks)}
    return {binding.debug_decoder_route(mode, len(streams), n, group_log2, o, alike if o > 1 else 0, int(k), int(w), bulk)
            for o in owned for k, w in set(zip(keys.tolist(), words.tolist()))}


def _damage(s, group):
    """The first deltas of one group become 0."""
    s = s.copy()
    cnt, off = (int(x) for x in np.frombuffer(s[64 + 8 * group:72 + 8 * group].tobytes(), np.uint32))
    cnt &= 0xFFFFFF
    bits = np.unpackbits(s[4 * off:4 * off + 2 * cnt + 16])
    bits[10 * cnt:10 * cnt + 40] = 0
    s[4 * off:4 * off + 2 * cnt + 16] = np.packbits(bits)
    return s


def _dev(streams):
    return [G.to_dev(np.concatenate([s, np.zeros(-s.size % 16 + 16, np.uint8)])) for s in streams]


def _check_decode(streams, n, po, pg, want, dense0, shift=0):
    dense = torch.zeros(n + 4, dtype=torch.float32, device=G.dev())[shift:shift + n]
    dense.copy_(torch.from_numpy(dense0))
    assert binding.decompress_accumulate_batch(_dev(streams), [s.size for s in streams], n, pg, dense) == 0
    status = binding.decode_status()
    assert np.array_equal(dense.cpu().numpy(), want)
    return status


def _check_update(streams, n, pg, model, want, packed):
    arrays = [torch.from_numpy(x.copy()).to(G.dev()) for x in model] + [torch.zeros(n, dtype=torch.float32, device=G.dev())]
    dev, sizes = _dev(streams), [s.size for s in streams]
    if packed:
        state = torch.stack(arrays, dim=1).reshape(-1)
        assert binding.sparse_adam_update_packed_batch(dev, sizes, n, pg, binding.Adam(*HYPER), state) == 0
        arrays = list(state.reshape(n, 4).unbind(1))
    else:
        assert binding.sparse_adam_update_batch(dev, sizes, n, pg, binding.Adam(*HYPER), arrays[3], *arrays[:3]) == 0
    status = binding.decode_status()
    for i, x in enumerate(want + [np.zeros(n, np.float32)]):
        assert np.array_equal(arrays[i].cpu().numpy(), x), i
    return status


# groups of the grid's blocks, streams, random keys a group of each, group_log2, modes that go by ranks, entries that dense_out is off 16 bytes
@pytest.mark.parametrize("owned,workers,count,group_log2,modes,shift", [
    (5, 6, 130, 14, (0, 2, 3), 0),            # 800 keys a group
    (5, 8, 60, 11, (0, 2, 3), 0),             # 510: lists of 4 keys a thread
    (6, 3, 250, 10, (0, 2, 3), 0),            # 680: streams of more keys than one round takes
    (5, 2, 300, 12, (0, 2, 3), 1),            # 590
    (5, 8, 55, 8, (0, 2, 3), 3),              # 425 of 256 indices: the smallest bit map
    (2, 7, 90, 15, (2,), 0),                  # 660: the largest
    (5, 10, 66, 11, (0, 1), 0),               # ten streams: eight of 560 keys, and two
    (5, 3, 400, 15, (0,), 0),                 # 1200 of 2^15: no slice to go over
    (5, 4, 330, 13, (0,), 2),                 # 1320, where the slice is not aligned
    (6, 8, 22, 11, (2,), 0),                  # 215, the update
    (5, 8, 300, 11, (3,), 0),                 # 2200: as many as the memory holds
])
def test_ranks(owned, workers, count, group_log2, modes, shift):
    groups, size = owned * _blocks() + 7, 1 << group_log2
    n = groups * size - 3
    streams, po, pg = _streams(n, group_log2, workers, count, 1000 + count)
    for mode in modes:
        assert _routes(streams[:8], n, group_log2, mode, mode != 0 or shift == 0) == {"four warps by ranks"}, mode
    bad, group = (1, workers - 1 if workers < 8 else 6), groups // 2 + 1
    lo, hi = group * size, (group + 1) * size
    damaged = [_damage(s, group) if w in bad else s for w, s in enumerate(streams)]
    sound = [s for w, s in enumerate(streams) if w not in bad]
    first = oracle.decompress_accumulate(damaged[bad[0]], n, po, np.zeros(n, np.float32))
    assert first != 0
    rng = np.random.default_rng(count)
    binding.ensure_workspace(n, pg)
    dense0 = rng.standard_normal(n).astype(np.float32)
    want, rest = dense0.copy(), dense0.copy()
    for s in streams:
        assert oracle.decompress_accumulate(s, n, po, want) == 0
    for s in sound:
        assert oracle.decompress_accumulate(s, n, po, rest) == 0
    assert _check_decode(streams, n, po, pg, want, dense0, shift) == 0
    want[lo:hi] = rest[lo:hi]                      # a stream that fails in a group is left out there as a whole
    assert _check_decode(damaged, n, po, pg, want, dense0, shift) == first
    model = [rng.standard_normal(n).astype(np.float32), (rng.standard_normal(n) * 1e-3).astype(np.float32), (rng.standard_normal(n) ** 2 * 1e-6).astype(np.float32)]
    want, rest = [x.copy() for x in model], [x.copy() for x in model]
    assert oracle.sparse_adam_update(streams, n, po, *HYPER, *want) == 0
    assert oracle.sparse_adam_update(sound, n, po, *HYPER, *rest) == 0
    packed = (False, True) if 3 in modes else (False,)
    for p in packed:
        assert _check_update(streams, n, pg, model, want, p) == 0
    for x, y in zip(want, rest):
        x[lo:hi] = y[lo:hi]
    for p in packed:
        assert _check_update(damaged, n, pg, model, want, p) == first


# about as many keys a group as where another way of decoding begins: more groups to a block than teams of four take side by side, and as many
@pytest.mark.parametrize("owned", [3, 6])
@pytest.mark.parametrize("workers,count", [(8, 27), (4, 64), (8, 45), (3, 140), (5, 199), (2, 580), (2, 900)])
def test_means_near_the_lines(owned, workers, count):
    n = owned * _blocks() * 2048 - 5
    streams, po, pg = _streams(n, 11, workers, count, count)
    binding.ensure_workspace(n, pg)
    rng = np.random.default_rng(count)
    dense0 = rng.standard_normal(n).astype(np.float32)
    want = dense0.copy()
    for s in streams:
        assert oracle.decompress_accumulate(s, n, po, want) == 0
    assert _check_decode(streams, n, po, pg, want, dense0) == 0
    model = [rng.standard_normal(n).astype(np.float32), (rng.standard_normal(n) * 1e-3).astype(np.float32), (rng.standard_normal(n) ** 2 * 1e-6).astype(np.float32)]
    want = [x.copy() for x in model]
    assert oracle.sparse_adam_update(streams, n, po, *HYPER, *want) == 0
    for p in (False, True):
        assert _check_update(streams, n, pg, model, want, p) == 0


# one stream: entries by the block or over the slice; by warps with two entries in flight or eight
@pytest.mark.parametrize("n,group_log2,count,routes", [(1160 << 14, 14, 960, ("block over the slice",)),
                                                        (13_000_001, 14, 1100, ("block",)),
                                                        (45_000_001, 13, 150, ("warp, two in flight",)),
                                                        (45_000_001, 13, 250, ("warp", "warp, two in flight"))])
def test_one_stream_of_many_groups(n, group_log2, count, routes):
    streams, po, pg = _streams(n, group_log2, 1, count, count)
    assert _routes(streams, n, group_log2, 0) == set(routes)
    binding.ensure_workspace(n, pg)
    dense0 = np.random.default_rng(count).standard_normal(n).astype(np.float32)
    want = dense0.copy()
    assert oracle.decompress_accumulate(streams[0], n, po, want) == 0
    assert _check_decode(streams, n, po, pg, want, dense0) == 0
