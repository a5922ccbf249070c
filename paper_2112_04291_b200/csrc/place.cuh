// k_place: the last of the dense encoder's launches, for every group size.
#pragma once

#include "encode.cuh"
#include "groups.cuh"

namespace fsg {

// ---- k_place -----------------------------------------------------------------------------------
constexpr uint32_t kRowTiles = 8;                              // tiles whose blobs a warp copies together: neighbours in the stream
struct PlaceShared {
    unsigned long long seg[kMaxSegments];                      // exclusive sums over the segments of each gradient (kept entries << 32 | words)
    unsigned long long total[kEncMaxJobs];
    unsigned long long scan64[kEncWarps];
    union {
        struct { float thr[132]; TeamScratch team; WorkArea::Block area; };
        GroupShared grp;
    };
};
static_assert(2 * (sizeof(PlaceShared) + 1024) <= 233472, "two blocks per SM (1 KiB per block is the system's)");

// kept entries and words of the tiles before `tile` in the gradient; one warp
__device__ __forceinline__ unsigned long long tile_prefix(const EncArgs& a, const unsigned long long* seg, uint32_t j, uint32_t tile, int lane) {
    const uint32_t sg = tile >> a.seg_log2, t0 = sg << a.seg_log2;
    unsigned long long x = 0ull;
    for (uint32_t i = t0 + (uint32_t)lane; i < tile; i += 32u) {
        const unsigned long long d = __ldcg(&a.desc[(uint64_t)j * a.D + i]);
        x += ((d & 0xFFFFFFull) << 32) | (d >> 32);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
    return seg[j * a.segments + sg] + x;
}

template <bool kTiles>                                         // groups are tiles
__global__ void __launch_bounds__(kEncThreads, 2)
k_place(const EncArgs a) {
    extern __shared__ __align__(128) unsigned char place_smem_raw[];
    PlaceShared& s = *reinterpret_cast<PlaceShared*>(place_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t B = gridDim.x, fixed_words = (kHeaderBytes + 8u * a.D) >> 2;
    allow_next_kernel();
    wait_for_previous_kernels();
    if (ld_acquire_u32(&a.ctl->error) != 0u) {                 // (the same answer in every block) some wait of the launch ran out
        if (blockIdx.x == 0 && tid < (int)a.J) enc_write_header(a, (uint32_t)tid, kStTimeout, 0ull, 0ull, 0.0);
        return;
    }
    // ---- exclusive sums over the segments (all gradients' in one scan, each gradient's start taken off afterwards)
    const uint32_t segs = a.J * a.segments;
    {
        constexpr uint32_t kPer = (kMaxSegments + kEncThreads - 1u) / kEncThreads;
        unsigned long long x[kPer], sum = 0ull;
#pragma unroll
        for (uint32_t i = 0; i < kPer; ++i) {
            const uint32_t e = (uint32_t)tid * kPer + i;
            x[i] = e < segs ? __ldcg(&a.seg[e]) : 0ull;
            sum += x[i];
        }
        unsigned long long incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s.scan64[warp] = incl;
        __syncthreads();
        unsigned long long w = lane < kEncWarps ? s.scan64[lane] : 0ull, wi = w;
#pragma unroll
        for (int o = 1; o < kEncWarps; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(kFullMask, wi, o);
            if (lane >= o) wi += u;
        }
        unsigned long long before = incl - sum + __shfl_sync(kFullMask, wi - w, warp);
#pragma unroll
        for (uint32_t i = 0; i < kPer; ++i) {
            const uint32_t e = (uint32_t)tid * kPer + i;
            if (e < segs) s.seg[e] = before;
            before += x[i];
            if (e < segs && (e + 1u) % a.segments == 0u) s.total[e / a.segments] = before;
        }
        __syncthreads();
        if (a.J > 1u) {
            unsigned long long start[kPer];
#pragma unroll
            for (uint32_t i = 0; i < kPer; ++i) {
                const uint32_t e = (uint32_t)tid * kPer + i;
                start[i] = e < segs ? s.seg[e / a.segments * a.segments] : 0ull;
            }
            if (tid < (int)a.J) s.total[tid] -= s.seg[(uint32_t)tid * a.segments];
            __syncthreads();
#pragma unroll
            for (uint32_t i = 0; i < kPer; ++i) {
                const uint32_t e = (uint32_t)tid * kPer + i;
                if (e < segs) s.seg[e] -= start[i];
            }
            __syncthreads();
        }
    }
    // ---- headers; a gradient whose sum is not finite or whose stream does not fit has nothing else
    auto total_bytes_of = [&](uint32_t j) -> uint64_t { return ((uint64_t)fixed_words + (uint32_t)s.total[j]) << 2; };
    auto fits = [&](uint32_t j) -> bool { return total_bytes_of(j) <= a.out_bytes; };
    const bool noblob = __ldcg(&a.st->noblob) != 0u;
    if (blockIdx.x == 0 && tid < (int)a.J) {
        const double S = __ldcg(&a.st->S[tid]);
        enc_write_header(a, (uint32_t)tid, !isfinite(S) ? kStNonfinite : !fits((uint32_t)tid) ? kStCapacity : kStOk, s.total[tid] >> 32, total_bytes_of((uint32_t)tid), S);
    }
    static_assert(kTicketGroups == (uint32_t)kEncMaxJobs, "reset together");
    if (blockIdx.x == 0 && tid < (int)kPools) a.st->pool_used[tid][0] = 0ull;
    if (blockIdx.x == 0 && tid < kEncMaxJobs) {                // at rest again
        a.ctl->bar_count[tid] = 0u; a.st->ticket[tid][0] = 0u;
        for (uint32_t i = 0; i < kSampleBlocks; ++i) a.st->sample[tid][i] = 0ull;
    }
    // ---- rows of eight tiles: directory entries and blobs.  When the rows are fewer than the warps, several warps share a row's words.
    const uint32_t rows = (a.D + kRowTiles - 1u) / kRowTiles, warps = B * (uint32_t)kEncWarps;
    const uint32_t parts = max(1u, min(32u, warps / (a.J * rows)));
    for (uint32_t x = blockIdx.x + B * (uint32_t)warp; x < a.J * rows * parts; x += warps) {
        const uint32_t part = x % parts, y = x / parts, j = y / rows, t0 = (y - j * rows) * kRowTiles, tile = t0 + (uint32_t)lane;
        if (!fits(j)) continue;
        const bool mine = (uint32_t)lane < kRowTiles && tile < a.D;
        const unsigned long long d = mine ? __ldcg(&a.desc[(uint64_t)j * a.D + tile]) : 0ull;
        const uint32_t place = mine ? __ldcg(&a.blob[(uint64_t)j * a.D + tile]) : 0u;
        const uint32_t before = fixed_words + (uint32_t)tile_prefix(a, s.seg, j, t0, lane);
        const uint32_t w = (uint32_t)(d >> 32), wi = warp_incl_scan(w, lane), we = wi - w;
        const uint32_t all = __shfl_sync(kFullMask, wi, 31);
        if (mine && part == 0u) *reinterpret_cast<uint2*>(a.out[j] + kHeaderBytes + 8ull * tile) = make_uint2((uint32_t)d, before + we);
        const uint32_t p0 = (uint32_t)((uint64_t)all * part / parts), p1 = (uint32_t)((uint64_t)all * (part + 1u) / parts);
        uint32_t* dst = reinterpret_cast<uint32_t*>(a.out[j]) + before;
        for (uint32_t i0 = p0; i0 < p1; i0 += 128u) {
            uint32_t v[4], ok = 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + 32u * (uint32_t)u + (uint32_t)lane;
                // which tile is word i of?  (the last one that starts at or before it)
                uint32_t at = 0u;
#pragma unroll
                for (uint32_t o = kRowTiles / 2u; o > 0u; o >>= 1) { const uint32_t e = __shfl_sync(kFullMask, we, at + o); if (e <= i) at += o; }
                const uint32_t e = __shfl_sync(kFullMask, we, at), pl = __shfl_sync(kFullMask, place, at);
                v[u] = 0u;
                if (i < p1 && pl != kNoPlace) { v[u] = __ldcg(reinterpret_cast<const uint32_t*>(a.scratch + 16ull * pl) + (i - e)); ok |= 1u << u; }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) if ((ok >> u) & 1u) dst[i0 + 32u * (uint32_t)u + (uint32_t)lane] = v[u];
        }
    }
    // ---- tiles for whose blobs there was no room: packed here (the pool holds a sixth of the entries; only where most of them are kept)
    if (noblob && !kTiles) {
        const uint32_t per = items_of(a);
        for (uint32_t x = blockIdx.x; x < a.J * per; x += B) {
            const uint32_t j = x / per;
            const Item it(a, x - j * per);
            bool without = false;                              // (all groups of an item or none)
            for (uint32_t g = (uint32_t)lane; g < it.groups; g += 32u) {
                const uint64_t t = (uint64_t)j * a.D + it.group0 + g;
                without = without || (__ldcg(&a.desc[t]) != 0ull && __ldcg(&a.blob[t]) == kNoPlace);
            }
            if (!__any_sync(kFullMask, without) || !fits(j)) continue;      // (the same in every warp)
            __syncthreads();
            block_item(a, s.grp, j, it, reinterpret_cast<uint32_t*>(a.out[j]) + fixed_words + (uint32_t)tile_prefix(a, s.seg, j, it.group0, lane), tid, lane, warp);
        }
    }
    if (noblob && kTiles) {
        for (uint32_t t = blockIdx.x; t < a.J * a.D; t += B) {
            const unsigned long long d = __ldcg(&a.desc[t]);
            const uint32_t j = t / a.D, tile = t - j * a.D;
            if (d == 0ull || __ldcg(&a.blob[t]) != kNoPlace || !fits(j)) continue;      // (uniform)
            __syncthreads();
            const double S = __ldcg(&a.st->S[j]);
            for (uint32_t k = (uint32_t)tid; k <= a.tau; k += kEncThreads) s.thr[k] = boundary(S, __ldcg(a.st->pw + k), __ldcg(a.st->inv + k));
            if (tid == kEncThreads - 1) table_hints(S, a.base, &s.thr[130]);
            __syncthreads();
            const uint32_t count = block_tile(a, j, tile, s.thr, s.area.key, s.area.blob, s.team, tid, lane, warp);
            team_pack<kEncWarps>(a.l, s.area.key, s.area.blob, count, s.team, warp, lane, 0, [](uint32_t) {});
            uint32_t* dst = reinterpret_cast<uint32_t*>(a.out[j]) + fixed_words + (uint32_t)tile_prefix(a, s.seg, j, tile, lane);
            for (uint32_t i = (uint32_t)tid; i < (uint32_t)(d >> 32); i += kEncThreads) dst[i] = bswap32(s.area.blob[i]);
            __syncthreads();
        }
    }
}

}  // namespace fsg
