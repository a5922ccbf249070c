"""Workspaces of the least size a call takes, of other sizes than the call's, and too small ones."""
import numpy as np
import pytest
import torch

import gpu_util as G
import oracle
from paper_2112_04291_b200 import binding, workloads

pytestmark = pytest.mark.gpu

TILE = 16384
MIB = 1 << 20


@pytest.fixture
def workspace():
    """Registers a workspace of a given size and returns it with canaries behind; afterwards the next ensure_workspace allocates one of
    its own."""
    def register(nbytes):
        buf = G.Guarded(nbytes)
        binding.set_workspace(buf.view)
        return buf
    yield register
    binding.set_workspace(torch.empty(2 * MIB, dtype=torch.uint8, device=G.dev()))


def _least(n, group_log2):
    """What the header says one dense gradient takes."""
    return 3 * MIB + 2432 * -(-n >> 14) + 12 * -(-n >> group_log2)


def _streams_equal(outs, grads, po):
    for o, v in zip(outs, grads):
        rc, want = oracle.compress(v, po)
        total, d, status = binding.stream_info(o.view)
        assert status == rc == 0 and total == want.size and o.intact()
        assert np.array_equal(o.view[:total].cpu().numpy(), want)


def test_registered_for_a_larger_n(workspace):
    # (one gradient of half the GPU's entries a launch takes, and a little less: eight a launch instead of seven)
    p = binding.params(1.2)
    ws = workspace(binding.workspace_bytes(402_653_185, p))
    for n in (402_653_184, 1 << 20):
        grad = torch.zeros(n, dtype=torch.float32, device=G.dev())
        grad[::99_991] = 1.0
        out = torch.zeros(64 * MIB, dtype=torch.uint8, device=G.dev())
        assert binding.compress(grad, p, out) == 0
        total, d, status = binding.stream_info(out)
        assert status == 0 and d == -(-n // 99_991)
        assert binding.decompress_accumulate(out, total, n, p, grad.zero_()) == 0 and binding.decode_status() == 0
        assert int((grad != 0).sum()) == d
    assert ws.intact()


# dense input with the least workspace: the pool holds next to nothing, tiles and groups of which much is kept are read again, and blobs
# longer than their slots are packed where they belong in the stream
@pytest.mark.parametrize("group_log2", [8, 9, 12, 14, 16, 20])
@pytest.mark.parametrize("workers", [1, 3])
def test_least_workspace_of_the_encoder(workspace, workers, group_log2):
    n = 600 * TILE + 77
    rng = np.random.default_rng(group_log2)
    grads = []
    for w in range(workers):                               # tiles of which nothing, a little, a tenth, most and everything is kept
        v = (rng.standard_normal(n) * 1e-9).astype(np.float32)
        for t in range(0, 600, 1 + w):
            share = (0.0, 0.002, 0.1, 0.7, 1.0)[(t // 7) % 5]
            c = int(share * TILE)
            k = t * TILE + rng.choice(TILE, c, replace=False)
            v[k] = (rng.uniform(0.5, 2.0, c) * rng.choice([-1.0, 1.0], c)).astype(np.float32)
        grads.append(v)
    pg, po = binding.params(1.2, 128, 3, group_log2), oracle.params(1.2, 128, 3, group_log2)
    least = _least(n, group_log2)
    dev = [G.to_dev(v) for v in grads]
    outs = [G.Guarded((binding.compress_bound(n, pg) + 255) & ~255) for _ in grads]
    for size in (least, least + 20 * MIB):
        ws = workspace(size)
        for rep in range(2):
            assert binding.compress_batch(dev, pg, [o.view for o in outs]) == 0
            _streams_equal(outs, grads, po)
        assert ws.intact()


def test_other_calls_take_the_least_workspace(workspace):
    n = 3_000_017
    v = workloads.normal_outliers(n, seed=3)
    base = workloads.base_for_keep(v, n // 50)
    pg, po = binding.params(base), oracle.params(base)
    rc, want = oracle.compress(v, po)
    ws = workspace(2 * MIB + 8 * -(-n >> 14))
    # decoder and update: the fixed part
    stream = G.to_dev(np.concatenate([want, np.zeros(-want.size % 16 + 16, np.uint8)]))
    dense, odense = torch.zeros(n, dtype=torch.float32, device=G.dev()), np.zeros(n, np.float32)
    assert binding.decompress_accumulate(stream, want.size, n, pg, dense) == 0 and binding.decode_status() == 0
    assert oracle.decompress_accumulate(want, n, po, odense) == 0
    assert np.array_equal(dense.cpu().numpy(), odense)
    # key-value input: 8 bytes a group; the sum: 8 bytes a chunk
    keys = np.flatnonzero(odense).astype(np.uint32)
    sparse = np.zeros(n, np.float32)
    sparse[keys] = v[keys]
    rc, want = oracle.compress(sparse, po)
    out = G.Guarded((want.size + 4096 + 255) & ~255)
    assert binding.compress_kv(G.to_dev(keys.view(np.int32)), G.to_dev(v[keys]), n, pg, out.view) == 0
    _streams_equal([out], [sparse], po)
    total = torch.zeros(1, dtype=torch.float64, device=G.dev())
    assert binding.abs_sum(G.to_dev(v), total) == 0
    assert total.item() == oracle.abs_sum(v)
    # one dense gradient of this length needs more
    big = torch.zeros(n, dtype=torch.float32, device=G.dev())
    assert binding.compress(big, pg, out.view) == binding.E_NO_WORKSPACE
    assert ws.intact()


def late_blobs():
    torch.cuda.synchronize()
    return int(binding.workspace_u32("late_blobs", 1)[0].item())


def test_blobs_go_where_their_lists_were(workspace):
    # a tenth of the entries kept: a list takes 3.3 KB of the pool per unit, a blob 2.9 KB per tile and more than the tile's slots.  With room for
    # the lists and half of the blobs beside them no tile is packed twice
    n = 600 * TILE
    v = np.random.default_rng(8).standard_normal(n).astype(np.float32)
    base = workloads.base_for_keep(v, n // 10)
    pg, po = binding.params(base), oracle.params(base)
    ws = workspace(_least(n, 14) + 4 * 600 * 3300 + 600 * 1450)
    out = G.Guarded((binding.compress_bound(n, pg) + 255) & ~255)
    dev = G.to_dev(v)
    for rep in range(2):
        assert binding.compress(dev, pg, out.view) == 0
        _streams_equal([out], [v], po)
        assert binding.listed_tiles(1) == [0] and late_blobs() == 0
    assert ws.intact()


def test_lists_leave_room_for_the_blobs_of_tiles_without(workspace):
    # a tenth of the entries kept and room for two lists in three: the other tiles are read again, and none is packed twice
    n = 4000 * TILE
    v = np.random.default_rng(9).standard_normal(n).astype(np.float32)
    base = workloads.base_for_keep(v[::16], n // 160)
    base **= (1 + np.log(16) / (128 * np.log(base)))         # (the sum of all entries, not of every sixteenth)
    pg, po = binding.params(base), oracle.params(base)
    ws = workspace(_least(n, 14) + 36 * MIB)
    out = G.Guarded(4 * n)
    dev = G.to_dev(v)
    for rep in range(2):
        assert binding.compress(dev, pg, out.view) == 0
        _streams_equal([out], [v], po)
        assert binding.listed_tiles(1)[0] > 400 and late_blobs() == 0
    assert binding.stream_info(out.view)[1] > n // 12
    assert ws.intact()
