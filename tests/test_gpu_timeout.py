"""The kernels' bounded waits, made to run out on purpose -- without hanging, trapping or faulting anything.

Every wait of one thread block on another (the counts of arrived blocks, the tagged words of k_resident and of the list
encoder, the decoder's queue of large groups) has an iteration limit.  These tests shorten the limits
(fastsgd_debug_set_wait_limits), put a counter of the workspace where no block can ever complete it, or allow so few looks
that others cannot have published yet, and check that the launch ends by itself with FASTSGD_ST_TIMEOUT in every status
word, that nothing outside the output buffers was written, that the library refuses further work until the workspace is
registered again, and that it is exact again afterwards.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded
from paper_2112_04291_b200 import binding, workloads

pytestmark = pytest.mark.gpu


def _streams_equal_oracle(grads, pg, po, outs):
    for g, o in zip(grads, outs):
        total, d, status = binding.stream_info(o)
        orc, ostream = oracle.compress(g, po)
        assert status == orc == 0 and total == ostream.size
        assert np.array_equal(o[:total].cpu().numpy(), ostream)


@pytest.mark.parametrize("n,workers", [(5_000_011, 3), (1_000_003, 1)])
def test_grid_barrier_that_cannot_complete_ends_in_timeout(n, workers):
    # 3 gradients of 306 tiles: k_encode's check that all blocks of k_scan have finished; 1 gradient of 62: k_resident's count of tiles
    host = [workloads.student_t_layers(n, seed=40 + w, blocks=9) for w in range(workers)]
    base = workloads.base_for_keep(host[0], n // 300)
    pg, po = binding.params(base), oracle.params(base)
    ws = binding.ensure_workspace(n, pg)
    grads = [torch.from_numpy(g).cuda() for g in host]
    cap = (min(binding.compress_bound(n, pg), max(4 * n, 1 << 20)) + 255) & ~255
    bufs = [Guarded(cap, fill=0x11) for _ in range(workers)]
    outs = [b.view for b in bufs]
    try:
        assert binding.compress_batch(grads, pg, outs) == 0
        _streams_equal_oracle(host, pg, po, outs)
        # the first count of arrivals starts beyond reach: it never is what is waited for
        binding.debug_set_wait_limits(block_polls=4096, copy_tries=256)
        binding.workspace_u32("bar_count", 8)[0] = 0x40000000
        torch.cuda.synchronize()
        assert binding.compress_batch(grads, pg, outs) == 0          # the launch itself is accepted ...
        for o in outs:                                              # ... and ends by itself, every stream marked
            total, d, status = binding.stream_info(o)
            assert (total, d, status) == (64, 0, binding.ST_TIMEOUT)
        assert all(b.intact() for b in bufs)
        # the workspace's counters are not at rest: further work is refused until it is registered again
        assert binding.compress_batch(grads, pg, outs) == binding.E_NO_WORKSPACE
        dense = torch.zeros(n, dtype=torch.float32, device="cuda")
        assert binding.decompress_accumulate(outs[0], cap, n, pg, dense) == binding.E_NO_WORKSPACE
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(ws)
    assert binding.compress_batch(grads, pg, outs) == 0
    _streams_equal_oracle(host, pg, po, outs)
    assert all(b.intact() for b in bufs)


def test_decoder_queue_slot_that_is_never_filled_ends_in_timeout():
    n = 5_000_011
    host = workloads.normal_outliers(n, seed=3)
    base = workloads.base_for_keep(host, n // 20)            # 5 %: every group is decoded by a whole block
    pg, po = binding.params(base), oracle.params(base)
    ws = binding.ensure_workspace(n, pg)
    cap = (min(binding.compress_bound(n, pg), max(4 * n, 1 << 20)) + 255) & ~255
    out = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    assert binding.compress(torch.from_numpy(host).cuda(), pg, out) == 0
    orc, ostream = oracle.compress(host, po)
    odense = np.zeros(n, np.float32)
    assert orc == 0 and oracle.decompress_accumulate(ostream, n, po, odense) == 0
    buf = Guarded(4 * n)
    dense = buf.view.view(torch.float32)
    try:
        # five queue slots count as reserved although nothing will ever fill them: their takers' waits run out
        binding.debug_set_wait_limits(queue_polls=2000)
        binding.workspace_u32("queue_counters", 6)[4] = 5
        torch.cuda.synchronize()
        assert binding.decompress_accumulate(out, cap, n, pg, dense) == 0
        assert binding.decode_status() == binding.ST_TIMEOUT
        assert buf.intact()
        # the queue is back in its resting state all the same
        assert not bool(binding.workspace_u32("queue_counters", 6).any().item())
        assert not bool(binding.workspace_u32("queue_slots", 4096).any().item())
        assert binding.decompress_accumulate(out, cap, n, pg, dense) == binding.E_NO_WORKSPACE
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(ws)
    dense.zero_()
    assert binding.decompress_accumulate(out, cap, n, pg, dense) == 0
    assert binding.decode_status() == 0
    assert np.array_equal(dense.cpu().numpy(), odense) and buf.intact()


def test_other_group_sizes_after_an_error_end_in_timeout():
    # k_filter finds the count of k_scan's blocks beyond reach; k_groups and k_place leave, the headers say why
    n, workers = 5_000_011, 2
    host = [workloads.student_t_layers(n, seed=60 + w, blocks=9) for w in range(workers)]
    base = workloads.base_for_keep(host[0], n // 300)
    pg, po = binding.params(base, 128, 2, 10), oracle.params(base, 128, 2, 10)
    ws = binding.ensure_workspace(n, pg)
    grads = [torch.from_numpy(g).cuda() for g in host]
    bufs = [Guarded((min(binding.compress_bound(n, pg), 4 * n) + 255) & ~255, fill=0x11) for _ in range(workers)]
    outs = [b.view for b in bufs]
    try:
        binding.debug_set_wait_limits(block_polls=4096, copy_tries=256)
        binding.workspace_u32("bar_count", 8)[0] = 0x40000000
        torch.cuda.synchronize()
        assert binding.compress_batch(grads, pg, outs) == 0
        for o in outs:
            assert binding.stream_info(o) == (64, 0, binding.ST_TIMEOUT)
        assert all(b.intact() and bool((b.view[64:] == 0x11).all()) for b in bufs)
        assert binding.compress_batch(grads, pg, outs) == binding.E_NO_WORKSPACE
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(ws)
    assert binding.compress_batch(grads, pg, outs) == 0
    _streams_equal_oracle(host, pg, po, outs)


def _pairs():
    n = 3_000_017
    rng = np.random.default_rng(9)
    keys = np.sort(rng.choice(n, 30_000, replace=False)).astype(np.uint32)
    vals = rng.standard_normal(keys.size).astype(np.float32)
    dense = np.zeros(n, np.float32)
    dense[keys] = vals
    base = workloads.base_for_keep(dense, keys.size // 2)
    return n, dense, torch.from_numpy(keys.view(np.int32)).cuda(), torch.from_numpy(vals).cuda(), base


def test_list_encoder_barrier_that_cannot_complete_ends_in_timeout():
    n, dense, keys, vals, base = _pairs()
    pg, po = binding.params(base), oracle.params(base)
    ws = binding.ensure_workspace(n, pg)
    buf = Guarded(1 << 20)
    try:
        binding.debug_set_wait_limits(block_polls=4096)
        binding.workspace_u32("bar_count", 8)[0] = 0x40000000
        torch.cuda.synchronize()
        assert binding.compress_kv(keys, vals, n, pg, buf.view) == 0
        assert binding.stream_info(buf.view) == (64, 0, binding.ST_TIMEOUT) and buf.intact()
        assert binding.compress_kv(keys, vals, n, pg, buf.view) == binding.E_NO_WORKSPACE
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(ws)
    assert binding.compress_kv(keys, vals, n, pg, buf.view) == 0
    _streams_equal_oracle([dense], pg, po, [buf.view])


@pytest.mark.parametrize("kind", ["resident", "list"])
def test_exchange_with_a_single_look_ends_in_timeout(kind):
    # the first block to look for the others' words cannot find them all: it gives up, and so says the header, or (should they all have been
    # there) the stream is exact
    n, dense, keys, vals, base = _pairs()
    pg, po = binding.params(base), oracle.params(base)
    ws = binding.ensure_workspace(n, pg)
    buf = Guarded(1 << 20)
    grad = torch.from_numpy(dense).cuda()
    call = (lambda: binding.compress(grad, pg, buf.view)) if kind == "resident" else (lambda: binding.compress_kv(keys, vals, n, pg, buf.view))
    seen = 0
    try:
        binding.debug_set_wait_limits(block_polls=1)
        for rep in range(20):
            assert call() == 0
            status = binding.stream_info(buf.view)[2]
            assert buf.intact()
            if status == binding.ST_TIMEOUT:
                seen += 1
                assert call() == binding.E_NO_WORKSPACE
                binding.set_workspace(ws)
            else:
                _streams_equal_oracle([dense], pg, po, [buf.view])
    finally:
        binding.debug_set_wait_limits(0, 0, 0)
        binding.set_workspace(ws)
    assert seen > 0
    assert call() == 0
    _streams_equal_oracle([dense], pg, po, [buf.view])
