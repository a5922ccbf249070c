// C-ABI shim: argument checks, workspace bookkeeping and kernel launches on the caller's
// stream.  No computation of the path happens here except the parameter-only table b^k.
#include "../../include/fastsgd.h"
#include "../../include/fastsgd_debug.h"

#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "sum.cuh"
#include "bits.cuh"
#include "prims.cuh"
#include "encode.cuh"
#include "groups.cuh"
#include "place.cuh"
#include "keys_paper.cuh"
#include "kv.cuh"
#include "decode.cuh"

namespace {

using namespace fsg;

// Per device: the registered workspace and what the launches need to know about the GPU.
struct State {
    void*      ws = nullptr;
    uint64_t   ws_bytes = 0;
    int        sm_count = 0;
    int        sum_blocks_per_sm = 0;
    int        dec_blocks_per_sm = 0;
    int        res_blocks_per_sm = 0;
    int        enc_blocks_per_sm = 0;
    int        place_blocks_per_sm = 0;
    int        kv_blocks_per_sm = 0;
    bool       attrs_set = false;
    bool       timed_out = false;          // a status query saw FASTSGD_ST_TIMEOUT: the workspace's counters are not at rest
};
// Process-wide test settings (fastsgd_debug_*).
struct Tunables {
    uint32_t   grid_override = 0;          // blocks of the encoders' launches (0: as many as are resident); tests only
    uint32_t   wait_limit = kWaitLimit;    // bounded waits of the kernels (shortened only by fastsgd_debug_set_wait_limits)
    uint32_t   try_limit = kTryLimit;
    uint32_t   dec_spin_limit = kDecSpinLimit;
};
constexpr int kMaxDevices = 64;
std::mutex g_mu;                           // guards everything below (host side only: the calls of one device share its workspace)
State      g_states[kMaxDevices];
Tunables   g_tun;

// the state of the current device (caller holds g_mu)
State* device_state() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); dev = 0; }      // (no device at all: the argument checks still answer)
    if (dev < 0 || dev >= kMaxDevices) return nullptr;
    return &g_states[dev];
}
#define FSG_DEVICE_STATE() State* sp_ = device_state(); if (!sp_) return FASTSGD_E_CUDA; State& g_state = *sp_

std::atomic<uint64_t> g_launches{0};

// optional per-kernel timing (profiling aid)
struct TimedLaunch { int kernel; cudaEvent_t start, stop; };
bool g_timing = false;
std::vector<TimedLaunch> g_timed;
std::vector<std::pair<cudaEvent_t, cudaEvent_t>> g_event_pool;

struct LaunchTimer {
    bool active = false; TimedLaunch t{}; cudaStream_t st;
    LaunchTimer(int kernel, cudaStream_t s) : st(s) {
        if (!g_timing) return;
        if (g_event_pool.empty()) {
            if (cudaEventCreate(&t.start) != cudaSuccess || cudaEventCreate(&t.stop) != cudaSuccess) return;
        } else { t.start = g_event_pool.back().first; t.stop = g_event_pool.back().second; g_event_pool.pop_back(); }
        t.kernel = kernel; active = true;
        cudaEventRecord(t.start, st);
    }
    ~LaunchTimer() { if (active) { cudaEventRecord(t.stop, st); g_timed.push_back(t); } }
};

int check_params(const fastsgd_params* p, PowTable* pw) {
    if (!p) return FASTSGD_E_NULL;
    if (!(p->base > 1.0) || !std::isfinite(p->base)) return FASTSGD_E_BAD_PARAM;
    if (p->tau < 1 || p->tau > (uint32_t)kMaxTau) return FASTSGD_E_BAD_PARAM;
    if (p->flag_bits < 1 || p->flag_bits > 5) return FASTSGD_E_BAD_PARAM;
    if (p->group_log2 < 1 || p->group_log2 > 20) return FASTSGD_E_BAD_PARAM;
    if (p->reserved != 0) return FASTSGD_E_BAD_PARAM;
    PowTable local;
    PowTable& t = pw ? *pw : local;
    volatile double acc = 1.0;            // one rounded fp64 product per step
    t.P[0] = 1.0;
    for (uint32_t k = 1; k <= (uint32_t)kMaxTau; ++k) {
        if (k <= p->tau) { acc = acc * p->base; t.P[k] = acc; }
        else t.P[k] = t.P[p->tau];
    }
    if (!std::isfinite(t.P[p->tau])) return FASTSGD_E_BAD_PARAM;
    return FASTSGD_OK;
}

int check_n(uint64_t n) { return (n == 0 || n >= (1ull << 31)) ? FASTSGD_E_BAD_N : FASTSGD_OK; }

uint64_t groups_of(uint64_t n, uint32_t group_log2) { return (n + (1ull << group_log2) - 1) >> group_log2; }
uint64_t chunks_of(uint64_t n) { return (n + kChunk - 1) >> kChunkLog2; }

uint64_t bound_bytes(uint64_t n, const fastsgd_params* p) {
    const uint64_t T = 1ull << p->group_log2, G = groups_of(n, p->group_log2);
    const uint64_t per_group_words = (T * (8ull + p->flag_bits + p->group_log2) + 31ull) / 32ull;
    return kHeaderBytes + 8ull * G + 4ull * G * per_group_words;
}

// Gradients one encoder launch takes: up to eight, as long as they are no more than 3 * 2^30 entries together (the workspace has to
// hold all their lists).
uint32_t jobs_per_launch(uint64_t n) {
    const uint64_t j = (3ull << 30) / n;
    return j < 1ull ? 1u : j > (uint64_t)kEncMaxJobs ? (uint32_t)kEncMaxJobs : (uint32_t)j;
}

// The part of the workspace that an encoder launch of J gradients uses, as byte offsets: per unit (a quarter of a tile of 2^14 entries)
// its node of the sum tree, largest |v| and list; nodes of 512 units; per group (by default: tile) its descriptor and blob's place; per
// segment of groups its totals; the lists (a slot per unit and a pool for longer ones, which takes what is left of ws_bytes).
struct Layout {
    uint64_t partials, chunk, umax, info, desc, blob, seg, scratch, pool_begin, pool_bytes, end;      // end: bytes needed at least
    uint32_t J, tiles, groups, chunks, seg_log2, segments;
};
constexpr uint64_t kLeastPool = 32768;                             // bytes of each pool at least
Layout layout_of(uint64_t n, uint32_t group_log2, uint32_t J, uint64_t ws_bytes) {
    Layout y;
    y.J = J;
    y.tiles = (uint32_t)chunks_of(n);
    y.chunks = (4u * y.tiles + kChunkUnits - 1u) / kChunkUnits;
    y.groups = (uint32_t)groups_of(n, group_log2);
    y.seg_log2 = 6u;
    while ((uint64_t)y.J * ((y.groups + (1ull << y.seg_log2) - 1ull) >> y.seg_log2) > kMaxSegments) ++y.seg_log2;
    y.segments = (uint32_t)((y.groups + (1ull << y.seg_log2) - 1ull) >> y.seg_log2);
    const uint64_t T = (uint64_t)y.J * y.tiles, descs = (uint64_t)y.J * y.groups;
    uint64_t at = kPartialsOffset;
    auto take = [&](uint64_t bytes) { const uint64_t here = at; at = (at + bytes + 255ull) & ~255ull; return here; };
    y.partials = take(32ull * T);
    y.chunk = take(16ull * y.J * y.chunks);
    y.umax = take(16ull * T);
    y.info = take(4ull * sizeof(UnitInfo) * T);
    y.desc = take(8ull * descs);
    y.blob = take(4ull * descs);
    y.seg = take(8ull * y.J * y.segments);
    y.pool_begin = (uint64_t)kSlotBytes * T;
    y.scratch = take(y.pool_begin + kPools * kLeastPool);
    y.end = at;
    // (never more than every entry on a list)
    const uint64_t rest = ws_bytes > y.end ? ws_bytes - y.end : 0ull, most = 6ull * y.J * n;
    y.pool_bytes = kLeastPool + ((rest < most ? rest : most) / kPools & ~15ull);      // each
    return y;
}

// What fastsgd_workspace_bytes answers: enough for as many gradients of up to n entries as one launch takes, with a pool of a sixth of
// their entries, within 2^24 (or all of smaller gradients) and 2^27.  A launch never takes more than `all` entries, whatever the length of
// its gradients, so that every term here is at least the layout's for any shorter length and any number of gradients, and none
// falls as n grows.
uint64_t ws_bytes_for(uint64_t n, uint32_t group_log2) {
    const uint64_t most = 3ull << 30, all = n < most / (uint64_t)kEncMaxJobs ? (uint64_t)kEncMaxJobs * n : most;
    const uint64_t T = (all >> kChunkLog2) + kEncMaxJobs, descs = (all >> group_log2) + kEncMaxJobs, chunks = (4ull * T) / kChunkUnits + kEncMaxJobs;
    uint64_t pool = all / 6ull;
    if (pool < (1ull << 24)) pool = 1ull << 24;
    if (pool > (1ull << 27)) pool = 1ull << 27;
    if (pool > all) pool = all;
    const uint64_t parts = (32ull + 16ull + 4ull * sizeof(UnitInfo) + kSlotBytes) * T + 16ull * chunks + 12ull * descs + 8ull * kMaxSegments;
    return (kPartialsOffset + parts + 8ull * 256ull + kPools * kLeastPool + 6ull * pool + 255ull) & ~255ull;
}

// Gradients a launch takes with the workspace at hand: as many as it has room for, of those that are there; 0: too small for one.
uint32_t jobs_that_fit(uint64_t n, uint32_t group_log2, uint32_t num_grads, uint64_t ws_bytes) {
    uint32_t J = jobs_per_launch(n);
    if (J > num_grads) J = num_grads ? num_grads : 1u;
    while (J > 0u && layout_of(n, group_log2, J, 0ull).end > ws_bytes) --J;
    return J;
}

Control* control_of(void* ws) { return static_cast<Control*>(ws); }

int ensure_device_setup() {
    // caller holds g_mu; once per device
    FSG_DEVICE_STATE();
    if (g_state.attrs_set) return FASTSGD_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FASTSGD_E_CUDA;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ResShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_scan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScanShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_encode, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EncShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_place<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PlaceShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_place<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PlaceShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_groups, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GroupShared)) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_compress_kv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(KvSmem)) != cudaSuccess) return FASTSGD_E_CUDA;
    int b1 = 0, b2 = 0;
    {
        int x = 0, y = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_state.kv_blocks_per_sm, k_compress_kv, kKvThreads, sizeof(KvSmem)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_state.res_blocks_per_sm, k_resident, kEncThreads, sizeof(ResShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, k_encode, kEncThreads, sizeof(EncShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&y, k_place<true>, kEncThreads, sizeof(PlaceShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        g_state.enc_blocks_per_sm = x > 0 ? x : 1;
        g_state.place_blocks_per_sm = y > 0 ? y : 1;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b1, k_abs_sum, kSumThreads, 0) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<true, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<false, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    if (cudaFuncSetAttribute(k_decode_accumulate<true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecShared)) != cudaSuccess)
        return FASTSGD_E_CUDA;
    {   // every instantiation must be resident with the grid the launch uses (the queue of large groups relies on it)
        int b2x[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[0], k_decode_accumulate<false>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[1], k_decode_accumulate<true>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[2], k_decode_accumulate<false, 1>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[3], k_decode_accumulate<true, 1>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[4], k_decode_accumulate<false, 2>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[5], k_decode_accumulate<true, 2>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[6], k_decode_accumulate<false, 3>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b2x[7], k_decode_accumulate<true, 3>, kDecThreads, sizeof(DecShared)) != cudaSuccess) return FASTSGD_E_CUDA;
        b2 = b2x[0];
        for (int i = 1; i < 8; ++i) if (b2x[i] < b2) b2 = b2x[i];
    }
    g_state.sm_count = sms;
    g_state.sum_blocks_per_sm = b1 > 0 ? b1 : 1;
    g_state.dec_blocks_per_sm = b2 > 0 ? b2 : 1;
    g_state.attrs_set = true;
    return FASTSGD_OK;
}

// A launch whose blocks may move onto the GPU while the previous kernel of the stream drains (programmatic dependent launch): the
// kernel itself waits (wait_for_previous_kernels) before it reads or writes memory.
cudaError_t launch_overlapped(const void* fn, unsigned grid, unsigned threads, size_t smem, void** kargs, cudaStream_t st) {
    cudaLaunchConfig_t c;
    std::memset(&c, 0, sizeof(c));
    c.gridDim = dim3(grid); c.blockDim = dim3(threads); c.dynamicSmemBytes = smem; c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at; c.numAttrs = 1;
    return cudaLaunchKernelExC(&c, fn, kargs);
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// 1 / b^k (kernels multiply with it where that gives the quotient's rounding)
PowTable inverse_of(const PowTable& pw) {
    PowTable inv;
    for (int k = 0; k <= kMaxTau; ++k) inv.P[k] = 1.0 / pw.P[k];
    return inv;
}

int launch_sum(const float* grad, uint64_t n, Control* ctl, double* partials, double* sum_out, cudaStream_t st) {
    FSG_DEVICE_STATE();
    SumArgs sa;
    sa.grad = grad; sa.n = n; sa.chunks = (uint32_t)chunks_of(n);
    sa.ctl = ctl; sa.partials = partials; sa.sum_out = sum_out;
    uint64_t grid = (uint64_t)g_state.sm_count * g_state.sum_blocks_per_sm;
    if (grid > sa.chunks) grid = sa.chunks;
    { LaunchTimer lt(0, st); k_abs_sum<<<(unsigned)grid, kSumThreads, 0, st>>>(sa); }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? FASTSGD_OK : FASTSGD_E_CUDA;
}

}  // namespace

extern "C" {

int fastsgd_version(void) { return 1; }

int fastsgd_kernel_timing_enable(int enable) {
    std::lock_guard<std::mutex> lock(g_mu);
    g_timing = enable != 0;
    return FASTSGD_OK;
}

int fastsgd_kernel_timing_read(double ms_total[3], uint64_t launches[3]) {
    if (!ms_total || !launches) return FASTSGD_E_NULL;
    std::lock_guard<std::mutex> lock(g_mu);
    for (int i = 0; i < 3; ++i) { ms_total[i] = 0.0; launches[i] = 0; }
    int rc = FASTSGD_OK;
    for (const TimedLaunch& t : g_timed) {
        float ms = 0.f;
        if (cudaEventSynchronize(t.stop) != cudaSuccess || cudaEventElapsedTime(&ms, t.start, t.stop) != cudaSuccess) rc = FASTSGD_E_CUDA;
        else { ms_total[t.kernel] += ms; launches[t.kernel] += 1; }
        g_event_pool.emplace_back(t.start, t.stop);
    }
    g_timed.clear();
    return rc;
}

uint64_t fastsgd_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int fastsgd_debug_set_wait_limits(uint32_t block_polls, uint32_t copy_tries, uint32_t queue_polls) {
    std::lock_guard<std::mutex> lock(g_mu);
    g_tun.wait_limit = block_polls ? block_polls : kWaitLimit;
    g_tun.try_limit = copy_tries ? copy_tries : kTryLimit;
    g_tun.dec_spin_limit = queue_polls == 0xFFFFFFFFu ? 0u : (queue_polls ? queue_polls : kDecSpinLimit);
    return FASTSGD_OK;
}

int fastsgd_debug_set_grid(uint32_t blocks) {
    std::lock_guard<std::mutex> lock(g_mu);
    g_tun.grid_override = blocks;
    return FASTSGD_OK;
}

int fastsgd_debug_decoder_route(uint32_t mode, uint32_t streams, uint64_t n, uint32_t group_log2, uint32_t owned, uint32_t alike_mean, uint32_t keys, uint32_t words, int bulk) {
    if (mode > 3u || streams < 1u || streams > (uint32_t)kDecMaxStreams) return -1;
    if (streams == 1u) {
        if (keys <= warp_max(owned) && group_log2 <= 16u) return mode == 0u && two_in_flight(owned, n) && sparse_group(keys, 1u << group_log2) ? 7 : 0;
    } else {
        const TeamRule rule = team_rule((int)mode, group_log2, owned, alike_mean != 0u, alike_mean, bulk != 0, streams);
        const uint32_t team = team_for(rule, group_log2, keys, words);
        if (team < 3u) return team == 2u && !rule.table ? 3 : (int)team;
    }
    return group_log2 > 14u ? 6 : mode == 0u && keys >= slice_min(bulk != 0, streams == 1u, n) ? 5 : 4;
}

int fastsgd_debug_layout(uint64_t* offsets, uint32_t count) {
    if (!offsets) return FASTSGD_E_NULL;
    const uint64_t v[FASTSGD_DEBUG_LAYOUT_FIELDS] = {
        offsetof(Control, bar_count), offsetof(Control, ne_count), offsetof(Control, error),
        kEncStateOffset + offsetof(EncState, noblob), 0, 0, kQueueOffset, offsetof(Control, dq)};
    for (uint32_t i = 0; i < count && i < (uint32_t)FASTSGD_DEBUG_LAYOUT_FIELDS; ++i) offsets[i] = v[i];
    return FASTSGD_OK;
}

const char* fastsgd_strerror(int code) {
    switch (code) {
        case FASTSGD_OK: return "ok";
        case FASTSGD_E_NULL: return "null pointer argument";
        case FASTSGD_E_ALIGN: return "pointer not aligned as required";
        case FASTSGD_E_BAD_PARAM: return "invalid parameters";
        case FASTSGD_E_BAD_N: return "n must satisfy 1 <= n < 2^31";
        case FASTSGD_E_CAPACITY: return "output capacity smaller than header + directory";
        case FASTSGD_E_NO_WORKSPACE: return "no workspace registered or workspace too small";
        case FASTSGD_E_NOT_IMPLEMENTED: return "parameter combination not implemented in this build";
        case FASTSGD_E_CUDA: return "CUDA runtime error";
        case FASTSGD_E_TRUNCATED: return "stream shorter than its header";
        case FASTSGD_E_TOO_LARGE: return "n exceeds the built-in scratch of fastsgd_abs_sum_noalloc (2^28 entries)";
        case FASTSGD_ST_NONFINITE: return "sum of |v| is not finite";
        case FASTSGD_ST_CAPACITY: return "stream does not fit in the output buffer";
        case FASTSGD_ST_TIMEOUT: return "bounded wait between thread blocks ran out";
        case FASTSGD_ST_BAD_MAGIC: return "bad magic";
        case FASTSGD_ST_BAD_VERSION: return "bad version";
        case FASTSGD_ST_BAD_STATUS: return "stream carries an error status";
        case FASTSGD_ST_N_MISMATCH: return "n differs from the header";
        case FASTSGD_ST_PARAM_MISMATCH: return "parameters differ from the header";
        case FASTSGD_ST_TRUNCATED: return "stream truncated";
        case FASTSGD_ST_BAD_DIRECTORY: return "inconsistent directory";
        case FASTSGD_ST_BAD_KEY: return "decoded key out of range";
        case FASTSGD_ST_BAD_CODE: return "code byte out of range";
        default: return "unknown code";
    }
}

uint64_t fastsgd_compress_bound(uint64_t n, const fastsgd_params* params) {
    int rc = check_params(params, nullptr);
    if (rc != FASTSGD_OK || n == 0) return 0;
    return bound_bytes(n, params);
}

uint64_t fastsgd_workspace_bytes(uint64_t n, const fastsgd_params* params) {
    int rc = check_params(params, nullptr);
    if (rc != FASTSGD_OK || n == 0) return 0;
    return ws_bytes_for(n, params->group_log2);
}

int fastsgd_set_workspace(void* dev_ptr, uint64_t bytes, void* stream) {
    if (!dev_ptr) return FASTSGD_E_NULL;
    if (!aligned(dev_ptr, 256)) return FASTSGD_E_ALIGN;
    if (bytes < kPartialsOffset) return FASTSGD_E_NO_WORKSPACE;   // the fixed part: control block, encoder state, decoder queue, chunk sums of the list encoder
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    int rc = ensure_device_setup();
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(dev_ptr, 0, kPartialsOffset, st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaMemsetAsync(static_cast<unsigned char*>(dev_ptr) + offsetof(Control, decode_status), 0xFF, 8, st) != cudaSuccess)
        return FASTSGD_E_CUDA;
    g_state.ws = dev_ptr;
    g_state.ws_bytes = bytes;
    g_state.timed_out = false;
    return FASTSGD_OK;
}

int fastsgd_abs_sum(const float* grad, uint64_t n, double* sum_out, void* stream) {
    if (!grad || !sum_out) return FASTSGD_E_NULL;
    if (!aligned(grad, 16) || !aligned(sum_out, 8)) return FASTSGD_E_ALIGN;
    int rc = check_n(n);
    if (rc) return rc;
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    if (!g_state.ws || g_state.ws_bytes < kPartialsOffset + 8ull * chunks_of(n)) return FASTSGD_E_NO_WORKSPACE;
    rc = ensure_device_setup();
    if (rc) return rc;
    double* partials = reinterpret_cast<double*>(static_cast<unsigned char*>(g_state.ws) + kPartialsOffset);
    return launch_sum(grad, n, control_of(g_state.ws), partials, sum_out, static_cast<cudaStream_t>(stream));
}

namespace {
// The list encoder (kv.cuh).  Caller holds g_mu.  Of the workspace it uses the fixed part and 8 bytes per group.
int launch_list_encoder(const uint32_t* keys, const float* values, uint64_t count, uint64_t n,
                        const fastsgd_params* params, const PowTable& pw, void* out, uint64_t out_bytes, cudaStream_t st) {
    FSG_DEVICE_STATE();
    if (g_state.kv_blocks_per_sm < 1) return FASTSGD_E_CUDA;
    KvArgs ka;
    std::memset(&ka, 0, sizeof(ka));
    ka.keys = keys; ka.vals = values; ka.count = count; ka.n = n;
    ka.out = static_cast<uint8_t*>(out); ka.out_bytes = out_bytes; ka.ctl = control_of(g_state.ws);
    ka.partials = reinterpret_cast<double*>(static_cast<unsigned char*>(g_state.ws) + kKvPartialsOffset);
    ka.meta = reinterpret_cast<unsigned long long*>(static_cast<unsigned char*>(g_state.ws) + kPartialsOffset);
    ka.st = reinterpret_cast<EncState*>(static_cast<unsigned char*>(g_state.ws) + kEncStateOffset);
    ka.base = params->base; ka.G = (uint32_t)groups_of(n, params->group_log2); ka.chunks = (uint32_t)chunks_of(n);
    ka.tau = params->tau; ka.l = params->flag_bits; ka.group_log2 = params->group_log2;
    ka.wait_limit = g_tun.wait_limit;
    // all blocks are resident (they meet at grid barriers).  A warp per kKvSlice entries until the GPU is full: a warp works off its
    // chunks and groups one after the other, and the runs of a sparse gradient put a new one every few entries.
    uint64_t grid = (count + kKvSlice * kKvWarps - 1) / (kKvSlice * kKvWarps);
    const uint64_t cap = (uint64_t)g_state.sm_count * (uint64_t)(g_state.kv_blocks_per_sm > 2 ? 2 : g_state.kv_blocks_per_sm);
    if (grid > cap) grid = cap;
    if (grid > kKvMaxGrid) grid = kKvMaxGrid;
    if (g_tun.grid_override && g_tun.grid_override < grid) grid = g_tun.grid_override;
    if (grid < 1) grid = 1;
    const uint64_t warps = grid * kKvWarps;
    uint64_t slice = ((count + warps - 1) / warps + kKvSlice - 1) / kKvSlice * kKvSlice;
    if (slice < kKvSlice) slice = kKvSlice;
    ka.slice = (uint32_t)slice;
    PowTable pwc = pw;
    void* kargs[] = {&ka, &pwc};
    cudaError_t err;
    {
        LaunchTimer lt(1, st);
        err = cudaLaunchCooperativeKernel((const void*)k_compress_kv, dim3((unsigned)grid), dim3(kKvThreads), kargs, sizeof(KvSmem), st);
    }
    if (err != cudaSuccess) { cudaGetLastError(); return FASTSGD_E_CUDA; }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return FASTSGD_OK;
}

// The encoder's launches: num_grads dense gradients, up to 8 per launch.
int compress_launches(const float* const* grads, uint64_t n, const fastsgd_params* params,
                      void* const* outs, uint64_t out_bytes, uint32_t num_grads, void* stream) {
    if (!outs || !params || !grads) return FASTSGD_E_NULL;
    for (uint32_t i = 0; i < num_grads; ++i) {
        if (!grads[i] || !outs[i]) return FASTSGD_E_NULL;
        if (!aligned(grads[i], 16) || !aligned(outs[i], 16)) return FASTSGD_E_ALIGN;
    }
    PowTable pw;
    int rc = check_params(params, &pw);
    if (rc) return rc;
    rc = check_n(n);
    if (rc) return rc;
    const uint64_t G = groups_of(n, params->group_log2);
    if (out_bytes < kHeaderBytes + 8ull * G) return FASTSGD_E_CAPACITY;
    if (bound_bytes(n, params) / 4ull >= (1ull << 31)) return FASTSGD_E_BAD_N;   // descriptor fields are 31 bits
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    const uint32_t jobs = g_state.ws && !g_state.timed_out ? jobs_that_fit(n, params->group_log2, num_grads, g_state.ws_bytes) : 0u;
    if (!jobs) return FASTSGD_E_NO_WORKSPACE;
    rc = ensure_device_setup();
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (params->group_log2 < 8u) return FASTSGD_E_NOT_IMPLEMENTED;
    const bool tile_groups = params->group_log2 == (uint32_t)kGroupLog2;
    const Layout y = layout_of(n, params->group_log2, jobs, g_state.ws_bytes);
    unsigned char* wsb = static_cast<unsigned char*>(g_state.ws);
    PowTable inv = inverse_of(pw);
    for (uint32_t first = 0; first < num_grads; first += y.J) {
        EncArgs ea;
        std::memset(&ea, 0, sizeof(ea));
        ea.J = num_grads - first < y.J ? num_grads - first : y.J;
        for (uint32_t i = 0; i < ea.J; ++i) {
            ea.grad[i] = grads[first + i];
            ea.out[i] = static_cast<uint8_t*>(outs[first + i]);
        }
        ea.out_bytes = out_bytes; ea.n = n; ea.ctl = control_of(wsb);
        ea.st = reinterpret_cast<EncState*>(wsb + kEncStateOffset);
        ea.partials = reinterpret_cast<double*>(wsb + y.partials);
        ea.chunk = reinterpret_cast<unsigned long long*>(wsb + y.chunk); ea.chunks = y.chunks;
        ea.umax = reinterpret_cast<float*>(wsb + y.umax);
        ea.info = reinterpret_cast<UnitInfo*>(wsb + y.info);
        ea.desc = reinterpret_cast<unsigned long long*>(wsb + y.desc);
        ea.blob = reinterpret_cast<uint32_t*>(wsb + y.blob);
        ea.seg = reinterpret_cast<unsigned long long*>(wsb + y.seg); ea.seg_log2 = y.seg_log2; ea.segments = y.segments;
        ea.scratch = wsb + y.scratch; ea.pool_begin = y.pool_begin; ea.pool_bytes = y.pool_bytes; ea.pool_units = (4u * ea.J * y.tiles + kPools - 1u) / kPools;
        ea.base = params->base; ea.inv_ptau = inv.P[params->tau]; ea.G = y.tiles; ea.D = y.groups; ea.group_log2 = params->group_log2;
        ea.tau = params->tau; ea.l = params->flag_bits; ea.wait_limit = g_tun.wait_limit; ea.try_limit = g_tun.try_limit;
        const uint64_t tiles = (uint64_t)ea.J * ea.G;
        void* kargs[] = {&ea, &pw, &inv};
        // every tile on the GPU at once (a single block waits for nobody, so it need not be launched cooperatively)
        const uint64_t resident = (uint64_t)g_state.sm_count * (uint64_t)(g_state.res_blocks_per_sm > 0 ? g_state.res_blocks_per_sm : 0);
        if (tile_groups && tiles <= resident && tiles <= kMaxResident && (!g_tun.grid_override || tiles <= g_tun.grid_override)) {
            LaunchTimer lt(1, st);
            const cudaError_t err = tiles == 1u ? launch_overlapped((const void*)k_resident, 1u, kEncThreads, sizeof(ResShared), kargs, st)
                                                : cudaLaunchCooperativeKernel((const void*)k_resident, dim3((unsigned)tiles), dim3(kEncThreads), kargs, sizeof(ResShared), st);
            if (err != cudaSuccess) { cudaGetLastError(); return FASTSGD_E_CUDA; }
            g_launches.fetch_add(1, std::memory_order_relaxed);
            continue;
        }
        uint64_t g1 = (uint64_t)g_state.sm_count, g2 = (uint64_t)g_state.sm_count * g_state.enc_blocks_per_sm, g3 = (uint64_t)g_state.sm_count * g_state.place_blocks_per_sm;
        if (g_tun.grid_override) {
            if (g_tun.grid_override < g1) g1 = g_tun.grid_override;
            if (g_tun.grid_override < g2) g2 = g_tun.grid_override;
            if (g_tun.grid_override < g3) g3 = g_tun.grid_override;
        }
        if (g1 > tiles) g1 = tiles;
        if (g2 > tiles) g2 = tiles;
        if (g3 > tiles) g3 = tiles;
        ea.scan_blocks = (uint32_t)g1;
        ea.samplers = (uint32_t)g1 / ea.J < kSampleBlocks ? (uint32_t)g1 / ea.J : kSampleBlocks;      // (none: no estimate, every tile is read again)
        {
            LaunchTimer lt(1, st);
            cudaError_t err = launch_overlapped((const void*)k_scan, (unsigned)g1, kScanThreads, sizeof(ScanShared), kargs, st);
            if (tile_groups) {
                if (err == cudaSuccess) err = launch_overlapped((const void*)k_encode, (unsigned)g2, kEncThreads, sizeof(EncShared), kargs, st);
                if (err == cudaSuccess) err = launch_overlapped((const void*)k_place<true>, (unsigned)g3, kEncThreads, sizeof(PlaceShared), kargs, st);
            } else {
                if (err == cudaSuccess) err = launch_overlapped((const void*)k_filter, (unsigned)g2, kEncThreads, 0, kargs, st);
                if (err == cudaSuccess) err = launch_overlapped((const void*)k_groups, (unsigned)g2, kEncThreads, sizeof(GroupShared), kargs, st);
                if (err == cudaSuccess) err = launch_overlapped((const void*)k_place<false>, (unsigned)g3, kEncThreads, sizeof(PlaceShared), kargs, st);
            }
            if (err != cudaSuccess) { cudaGetLastError(); return FASTSGD_E_CUDA; }
        }
        g_launches.fetch_add(tile_groups ? 3 : 4, std::memory_order_relaxed);
    }
    return FASTSGD_OK;
}
}  // namespace

int fastsgd_compress_batch(const float* const* grads, uint64_t n, const fastsgd_params* params,
                           void* const* outs, uint64_t out_bytes, uint32_t num_grads, void* stream) {
    if (!grads) return FASTSGD_E_NULL;
    return compress_launches(grads, n, params, outs, out_bytes, num_grads, stream);
}

int fastsgd_compress_kv(const uint32_t* keys, const float* values, uint64_t count, uint64_t n,
                        const fastsgd_params* params, void* out, uint64_t out_bytes, void* stream) {
    if (!out || !params) return FASTSGD_E_NULL;
    if (count && (!keys || !values)) return FASTSGD_E_NULL;
    if (!aligned(keys, 4) || !aligned(values, 4) || !aligned(out, 16)) return FASTSGD_E_ALIGN;
    PowTable pw;
    int rc = check_params(params, &pw);
    if (rc) return rc;
    rc = check_n(n);
    if (rc) return rc;
    if (count > n) return FASTSGD_E_BAD_N;
    const uint64_t G = groups_of(n, params->group_log2);
    if (out_bytes < kHeaderBytes + 8ull * G) return FASTSGD_E_CAPACITY;
    if (bound_bytes(n, params) / 4ull >= (1ull << 31)) return FASTSGD_E_BAD_N;
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    if (!g_state.ws || g_state.timed_out || g_state.ws_bytes < kPartialsOffset + 8ull * G) return FASTSGD_E_NO_WORKSPACE;
    rc = ensure_device_setup();
    if (rc) return rc;
    return launch_list_encoder(keys, values, count, n, params, pw, out, out_bytes, static_cast<cudaStream_t>(stream));
}

int fastsgd_compress(const float* grad, uint64_t n, const fastsgd_params* params,
                     void* out, uint64_t out_bytes, void* stream) {
    if (!grad || !out) return FASTSGD_E_NULL;
    const float* g1[1] = {grad};
    void* o1[1] = {out};
    return fastsgd_compress_batch(g1, n, params, o1, out_bytes, 1u, stream);
}

namespace {
// The decoder's launches over a list of streams, 8 per launch.  adam == nullptr: aggregation into
// dense_out; else the model-update pass (dense_out holds the aggregated gradient), or, `fused` (one
// launch's worth of streams, dense_out all zero), aggregation and update in the same launch.
int decode_launches(const void* const* streams_in, const uint64_t* bytes, uint32_t num_streams, uint64_t n,
                    const fastsgd_params* params, float* dense_out, const fastsgd_adam* adam,
                    float* theta, float* m, float* v, void* stream, bool fused = false, bool packed = false) {
    if (fused && (!adam || num_streams > (uint32_t)kDecMaxStreams)) return FASTSGD_E_BAD_PARAM;
    if (packed && !fused) return FASTSGD_E_BAD_PARAM;
    if (!streams_in || !bytes || !dense_out || !params) return FASTSGD_E_NULL;
    if (!aligned(dense_out, 4)) return FASTSGD_E_ALIGN;
    PowTable pw;
    int rc = check_params(params, &pw);
    if (rc) return rc;
    rc = check_n(n);
    if (rc) return rc;
    // (the queue of groups that whole blocks decode has 2^17 slots)
    if (params->group_log2 < 8u || groups_of(n, params->group_log2) > (kQueueBytes >> 2)) return FASTSGD_E_NOT_IMPLEMENTED;
    for (uint32_t i = 0; i < num_streams; ++i) {
        if (!streams_in[i]) return FASTSGD_E_NULL;
        if (!aligned(streams_in[i], 16)) return FASTSGD_E_ALIGN;
        if (bytes[i] < kHeaderBytes) return FASTSGD_E_TRUNCATED;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    if (!g_state.ws || g_state.timed_out) return FASTSGD_E_NO_WORKSPACE;      // (the decoder uses its fixed part alone)
    rc = ensure_device_setup();
    if (rc) return rc;
    const uint64_t G = groups_of(n, params->group_log2);
    // a block per group until the GPU is full
    const uint64_t cap = (uint64_t)g_state.sm_count * g_state.dec_blocks_per_sm;
    const uint64_t grid = G < cap ? G : cap;
    PowTable inv = inverse_of(pw);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    for (uint32_t first = 0; first < num_streams; first += kDecMaxStreams) {
        DecArgs da;
        std::memset(&da, 0, sizeof(da));
        da.W = num_streams - first < (uint32_t)kDecMaxStreams ? num_streams - first : (uint32_t)kDecMaxStreams;
        for (uint32_t i = 0; i < da.W; ++i) {
            da.stream[i] = static_cast<const uint8_t*>(streams_in[first + i]);
            da.bytes[i] = bytes[first + i];
        }
        da.n = n; da.dense = dense_out;
        da.status = &control_of(g_state.ws)->decode_status;
        da.q_ctl = control_of(g_state.ws)->dq;
        da.q_list = reinterpret_cast<unsigned int*>(static_cast<unsigned char*>(g_state.ws) + kQueueOffset);
        da.base = params->base; da.G = (uint32_t)G; da.tau = params->tau; da.l = params->flag_bits;
        da.group_log2 = params->group_log2;
        da.spin_limit = g_tun.dec_spin_limit; da.try_limit = g_tun.try_limit;
        if (adam) {
            da.theta = theta; da.m = m; da.v = v;
            da.lr = adam->lr; da.beta1 = adam->beta1; da.beta2 = adam->beta2; da.eps = adam->eps;
        }
        {
            LaunchTimer lt(2, st);
            void* kargs[] = {&da, &pw, &inv};
            const bool one = da.W == 1u;
            const void* fn = packed ? (one ? (const void*)k_decode_accumulate<true, 3> : (const void*)k_decode_accumulate<false, 3>)
                             : fused ? (one ? (const void*)k_decode_accumulate<true, 2> : (const void*)k_decode_accumulate<false, 2>)
                             : adam ? (one ? (const void*)k_decode_accumulate<true, 1> : (const void*)k_decode_accumulate<false, 1>)
                                    : (one ? (const void*)k_decode_accumulate<true> : (const void*)k_decode_accumulate<false>);
            if (launch_overlapped(fn, (unsigned)grid, kDecThreads, sizeof(DecShared), kargs, st) != cudaSuccess) { cudaGetLastError(); return FASTSGD_E_CUDA; }
        }
        g_launches.fetch_add(1, std::memory_order_relaxed);
    }
    return FASTSGD_OK;
}
}  // namespace

int fastsgd_decompress_accumulate_batch(const void* const* streams_in, const uint64_t* bytes,
                                        uint32_t num_streams, uint64_t n, const fastsgd_params* params,
                                        float* dense_out, void* stream) {
    return decode_launches(streams_in, bytes, num_streams, n, params, dense_out, nullptr, nullptr, nullptr, nullptr, stream);
}

int fastsgd_sparse_adam_update_batch(const void* const* streams_in, const uint64_t* bytes,
                                     uint32_t num_streams, uint64_t n, const fastsgd_params* params,
                                     const fastsgd_adam* hyper, float* grad_scratch,
                                     float* theta, float* m, float* v, void* stream) {
    if (!hyper || !grad_scratch || !theta || !m || !v) return FASTSGD_E_NULL;
    if (!aligned(theta, 4) || !aligned(m, 4) || !aligned(v, 4)) return FASTSGD_E_ALIGN;
    // up to 8 streams: one launch, each group aggregated and its coordinates updated by the warp or block that decodes it
    if (num_streams <= (uint32_t)kDecMaxStreams)
        return decode_launches(streams_in, bytes, num_streams, n, params, grad_scratch, hyper, theta, m, v, stream, true);
    // more: pass 1, the aggregated gradient; pass 2, the same streams again, every key's coordinate updated once
    int rc = decode_launches(streams_in, bytes, num_streams, n, params, grad_scratch, nullptr, nullptr, nullptr, nullptr, stream);
    if (rc) return rc;
    return decode_launches(streams_in, bytes, num_streams, n, params, grad_scratch, hyper, theta, m, v, stream);
}

int fastsgd_sparse_adam_update_packed_batch(const void* const* streams_in, const uint64_t* bytes,
                                            uint32_t num_streams, uint64_t n, const fastsgd_params* params,
                                            const fastsgd_adam* hyper, float* state, void* stream) {
    if (!hyper || !state || !params) return FASTSGD_E_NULL;
    if (!aligned(state, 16)) return FASTSGD_E_ALIGN;
    // (the update of a group lives in the 64 KiB slice of shared memory of the block that decodes it: groups of up to 2^14
    //  indices, one launch's worth of streams)
    if (params->group_log2 > 14u || num_streams > (uint32_t)kDecMaxStreams) return FASTSGD_E_NOT_IMPLEMENTED;
    return decode_launches(streams_in, bytes, num_streams, n, params, state, hyper, nullptr, nullptr, nullptr, stream, true, true);
}

uint64_t fastsgd_key_encode_paper_bound(uint64_t d, uint32_t flag_bits) {
    if (flag_bits < 1 || flag_bits > 5 || d >= (1ull << 31)) return 0;
    const uint64_t blocks = (d + kBkBlockKeys - 1) / kBkBlockKeys;
    const uint64_t words = (d * (flag_bits + 32ull) + 31ull) / 32ull + 1ull;      // widest levels everywhere, and the padding word
    return 16ull + 8ull * blocks + 4ull * words;
}

int fastsgd_key_encode_paper(const uint32_t* keys, uint64_t d, uint32_t flag_bits,
                             void* out, uint64_t out_bytes, void* stream) {
    if (!out || (!keys && d)) return FASTSGD_E_NULL;
    if (!aligned(out, 16) || !aligned(keys, 4)) return FASTSGD_E_ALIGN;
    const uint64_t need = fastsgd_key_encode_paper_bound(d, flag_bits);
    if (!need) return FASTSGD_E_BAD_PARAM;
    if (out_bytes < need) return FASTSGD_E_CAPACITY;
    int sm_count = 0;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        FSG_DEVICE_STATE();
        const int rc = ensure_device_setup();
        if (rc) return rc;
        sm_count = g_state.sm_count;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    BkArgs a;
    a.keys = keys; a.d = d; a.l = flag_bits;
    a.blocks = (uint32_t)((d + kBkBlockKeys - 1) / kBkBlockKeys);
    a.header = static_cast<uint32_t*>(out);
    a.index = reinterpret_cast<unsigned long long*>(static_cast<unsigned char*>(out) + 16);
    a.bk = reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(out) + 16 + 8ull * a.blocks);
    if (cudaMemsetAsync(out, 0, 16, st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (a.blocks) {
        const unsigned cap = 8u * (unsigned)sm_count;
        const unsigned want = (unsigned)((d + kBkThreads - 1) / kBkThreads);
        k_bk_maxdelta<<<want < cap ? want : cap, kBkThreads, 0, st>>>(a);
        k_bk_sizes<<<a.blocks, kBkThreads, 0, st>>>(a);
    }
    k_bk_scan<<<1, kBkThreads, 0, st>>>(a);
    if (a.blocks) k_bk_pack<<<a.blocks, kBkThreads, 0, st>>>(a);
    g_launches.fetch_add(a.blocks ? 4 : 1, std::memory_order_relaxed);
    if (cudaGetLastError() != cudaSuccess) return FASTSGD_E_CUDA;
    return FASTSGD_OK;
}

int fastsgd_decompress_accumulate(const void* stream_in, uint64_t bytes, uint64_t n,
                                  const fastsgd_params* params, float* dense_out, void* stream) {
    if (!stream_in) return FASTSGD_E_NULL;
    const void* one[1] = {stream_in};
    return fastsgd_decompress_accumulate_batch(one, &bytes, 1u, n, params, dense_out, stream);
}

int fastsgd_stream_info(const void* stream_in, void* stream, uint64_t* total_bytes, uint64_t* d, int* status) {
    if (!stream_in) return FASTSGD_E_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char h[kHeaderBytes];
    if (cudaMemcpyAsync(h, stream_in, kHeaderBytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return FASTSGD_E_CUDA;
    uint32_t s32; uint64_t v;
    std::memcpy(&s32, h + 8, 4);
    if (status) *status = (int)s32;
    if (s32 == (uint32_t)FASTSGD_ST_TIMEOUT) {        // the launch that wrote this stream left the workspace's counters mid-way
        std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
        g_state.timed_out = true;
    }
    if (d) { std::memcpy(&v, h + 24, 8); *d = v; }
    if (total_bytes) { std::memcpy(&v, h + 32, 8); *total_bytes = v; }
    return FASTSGD_OK;
}

int fastsgd_decode_status(void* stream, int* status) {
    if (!status) return FASTSGD_E_NULL;
    std::lock_guard<std::mutex> lock(g_mu);
    FSG_DEVICE_STATE();
    if (!g_state.ws) return FASTSGD_E_NO_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned long long v = 0;
    unsigned char* p = static_cast<unsigned char*>(g_state.ws) + offsetof(Control, decode_status);
    if (cudaMemcpyAsync(&v, p, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return FASTSGD_E_CUDA;
    *status = (v == ~0ull) ? FASTSGD_ST_OK : (int)(v & 0xFFull);
    if (*status == FASTSGD_ST_TIMEOUT) g_state.timed_out = true;
    if (v != ~0ull) {
        if (cudaMemsetAsync(p, 0xFF, 8, st) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return FASTSGD_E_CUDA;
    }
    return FASTSGD_OK;
}

uint64_t fastsgd_host_scratch_bytes(uint64_t n, const fastsgd_params* params) {
    const uint64_t b = fastsgd_compress_bound(n, params);
    if (!b) return 0;
    return ((4ull * n + 255ull) & ~255ull) + ((b + 255ull) & ~255ull);
}

int fastsgd_compress_host(const float* grad_host, uint64_t n, const fastsgd_params* params,
                          void* out_host, uint64_t out_bytes, uint64_t* produced, int* status,
                          void* dev_scratch, uint64_t dev_scratch_bytes, void* stream) {
    if (!grad_host || !out_host || !dev_scratch || !params) return FASTSGD_E_NULL;
    if (!aligned(dev_scratch, 16)) return FASTSGD_E_ALIGN;
    const uint64_t need = fastsgd_host_scratch_bytes(n, params);
    if (!need) return FASTSGD_E_BAD_PARAM;
    if (dev_scratch_bytes < need) return FASTSGD_E_NO_WORKSPACE;
    if (out_bytes < kHeaderBytes) return FASTSGD_E_CAPACITY;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* dgrad = static_cast<float*>(dev_scratch);
    unsigned char* dout = static_cast<unsigned char*>(dev_scratch) + ((4ull * n + 255ull) & ~255ull);
    const uint64_t bound = fastsgd_compress_bound(n, params);
    const uint64_t cap = out_bytes < bound ? out_bytes : bound;
    if (cudaMemcpyAsync(dgrad, grad_host, 4ull * n, cudaMemcpyHostToDevice, st) != cudaSuccess) return FASTSGD_E_CUDA;
    int rc = fastsgd_compress(dgrad, n, params, dout, cap, stream);
    if (rc) return rc;
    uint64_t total = 0; int hst = 0;
    rc = fastsgd_stream_info(dout, stream, &total, nullptr, &hst);
    if (rc) return rc;
    if (total > cap) return FASTSGD_E_CUDA;
    if (cudaMemcpyAsync(out_host, dout, total, cudaMemcpyDeviceToHost, st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return FASTSGD_E_CUDA;
    if (produced) *produced = total;
    if (status) *status = hst;
    return FASTSGD_OK;
}

int fastsgd_decompress_accumulate_host(const void* const* streams_host, const uint64_t* bytes,
                                       uint32_t num_streams, uint64_t n, const fastsgd_params* params,
                                       float* dense_host, int accumulate, int* status,
                                       void* dev_scratch, uint64_t dev_scratch_bytes, void* stream) {
    if (!streams_host || !bytes || !dense_host || !dev_scratch || !params) return FASTSGD_E_NULL;
    if (!aligned(dev_scratch, 16)) return FASTSGD_E_ALIGN;
    const uint64_t need = fastsgd_host_scratch_bytes(n, params);
    if (!need) return FASTSGD_E_BAD_PARAM;
    const uint64_t dense_bytes = (4ull * n + 255ull) & ~255ull;
    if (dev_scratch_bytes < need) return FASTSGD_E_NO_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* ddense = static_cast<float*>(dev_scratch);
    unsigned char* dstream = static_cast<unsigned char*>(dev_scratch) + dense_bytes;
    if (accumulate) {
        if (cudaMemcpyAsync(ddense, dense_host, 4ull * n, cudaMemcpyHostToDevice, st) != cudaSuccess) return FASTSGD_E_CUDA;
    } else {
        if (cudaMemsetAsync(ddense, 0, 4ull * n, st) != cudaSuccess) return FASTSGD_E_CUDA;
    }
    // The streams are copied side by side into the staging area (16-byte aligned each) as long as they fit, then decoded
    // by one batched launch per 8; a stream that does not fit beside the others starts a new round (stream order keeps
    // the next round's copies behind this round's launch).
    const uint64_t room = need - dense_bytes;
    uint32_t i = 0;
    while (i < num_streams) {
        std::vector<const void*> ptrs;
        std::vector<uint64_t> sizes;
        uint64_t used = 0;
        while (i < num_streams) {
            if (!streams_host[i]) return FASTSGD_E_NULL;
            if (bytes[i] > room) return FASTSGD_E_NO_WORKSPACE;
            const uint64_t padded = (bytes[i] + 15ull) & ~15ull;
            if (used + padded > room) break;
            if (cudaMemcpyAsync(dstream + used, streams_host[i], bytes[i], cudaMemcpyHostToDevice, st) != cudaSuccess) return FASTSGD_E_CUDA;
            ptrs.push_back(dstream + used);
            sizes.push_back(bytes[i]);
            used += padded;
            ++i;
        }
        int rc2 = fastsgd_decompress_accumulate_batch(ptrs.data(), sizes.data(), (uint32_t)ptrs.size(), n, params, ddense, stream);
        if (rc2) return rc2;
    }
    if (cudaMemcpyAsync(dense_host, ddense, 4ull * n, cudaMemcpyDeviceToHost, st) != cudaSuccess) return FASTSGD_E_CUDA;
    int dst = 0;
    int rc = fastsgd_decode_status(stream, &dst);
    if (rc) return rc;
    if (status) *status = dst;
    return FASTSGD_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// fastsgd_abs_sum_noalloc: the sum kernel with its scratch inside the library image.
//
// Some callers have no way to give the library scratch memory: they may not call cudaMalloc
// (it synchronises the whole device and can fail when memory is tight), they do not own a
// framework allocator, they only receive an input and an output pointer.  For them the
// per-tile partials and the block counter of the sum kernel live in the array below: part of
// the loaded module on every GPU, 256-byte aligned, never allocated and never freed.
//
// In host code the name `g_noalloc_scratch` is only a handle for the symbol, not a device
// address; the address the kernel may use comes from cudaGetSymbolAddress, looked up once
// per device with that device current.
// ---------------------------------------------------------------------------------------------
namespace {

constexpr uint64_t kNoAllocMaxN      = FASTSGD_NOALLOC_MAX_N;                  // 2^28 entries = 1 GiB of fp32
constexpr uint64_t kNoAllocPartials  = kNoAllocMaxN >> fsg::kChunkLog2;        // 16384 fp64 partials
constexpr uint64_t kNoAllocCtlBytes  = 1024;                                   // control block + boundary table
constexpr uint64_t kNoAllocBytes     = kNoAllocCtlBytes + 8ull * kNoAllocPartials;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
struct NoAllocDevice {
    unsigned char* scratch = nullptr;     // device address of g_noalloc_scratch on this GPU
    int            grid_cap = 0;          // blocks that fit the GPU at once
};
std::mutex     g_noalloc_mu;
NoAllocDevice  g_noalloc_dev[kNoAllocMaxDevices];

// once per device, with that device current; allocates nothing
int noalloc_setup(int dev, NoAllocDevice** out) {
    if (dev < 0 || dev >= kNoAllocMaxDevices) return FASTSGD_E_CUDA;
    NoAllocDevice& d = g_noalloc_dev[dev];
    if (!d.scratch) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) { cudaGetLastError(); return FASTSGD_E_CUDA; }
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return FASTSGD_E_CUDA;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fsg::k_abs_sum, fsg::kSumThreads, 0) != cudaSuccess)
            return FASTSGD_E_CUDA;
        d.grid_cap = sms * (per_sm > 0 ? per_sm : 1);
        d.scratch = static_cast<unsigned char*>(p);
    }
    *out = &d;
    return FASTSGD_OK;
}

}  // namespace

extern "C" int fastsgd_abs_sum_noalloc(const float* grad, uint64_t n, double* sum_out, void* stream) {
    if (!grad || !sum_out) return FASTSGD_E_NULL;
    if (!aligned(grad, 16) || !aligned(sum_out, 8)) return FASTSGD_E_ALIGN;
    if (n == 0) return FASTSGD_E_BAD_N;
    if (n > kNoAllocMaxN) return FASTSGD_E_TOO_LARGE;              // would not fit the built-in scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FASTSGD_E_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocDevice* d = nullptr;
    int rc = noalloc_setup(dev, &d);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // The array keeps the previous call's contents.  Only the block counter has to start at zero
    // (the kernel leaves it at zero, but a call that was cut short might not have): clear the
    // control block on the stream.  Every partial that is read is written first by this call.
    if (cudaMemsetAsync(d->scratch, 0, sizeof(fsg::Control), st) != cudaSuccess) return FASTSGD_E_CUDA;
    fsg::SumArgs sa;
    sa.grad = grad; sa.n = n; sa.chunks = (uint32_t)((n + fsg::kChunk - 1) >> fsg::kChunkLog2);
    sa.ctl = reinterpret_cast<fsg::Control*>(d->scratch);
    sa.partials = reinterpret_cast<double*>(d->scratch + kNoAllocCtlBytes);
    sa.sum_out = sum_out;
    unsigned grid = (unsigned)d->grid_cap;
    if (grid > sa.chunks) grid = sa.chunks;
    fsg::k_abs_sum<<<grid, fsg::kSumThreads, 0, st>>>(sa);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? FASTSGD_OK : FASTSGD_E_CUDA;
}
