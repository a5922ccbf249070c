// Group sizes other than the default tile (2^8 .. 2^20 indices): between k_scan and k_place two launches that work by units and groups
// instead of by tiles.
//
//   k_filter  the sum, the boundaries; every unit's list filtered and quantised in place: its kept keys and code bytes.  A warp per unit,
//             no shared memory, no barrier.  Units whose estimate was too high are read again.
//   k_groups  an item is a group of one or more units, or a unit with the groups in it.  Its kept entries are gathered in shared
//             memory and packed; a warp takes a short item, the block a long one (in pieces, the partly filled words carried on).
//
// Both are chains of a few L2 round trips per item, many items side by side.  Per call, before (sum kernel, a kernel that read the gradient
// twice more to list the kept entries, and the list encoder with a warp per group) and now: 16.8 M entries at 0.2 %, groups of 2^16,
// 67.7 -> 45.5; 60 M at 2 %, groups of 2^10 605 -> 181, of 2^13 370 -> 171, of 2^18 2345 -> 398 us.
#pragma once

#include "encode.cuh"

namespace fsg {

constexpr uint32_t kUnitLog2     = 12;
static_assert(kUnit == 1u << kUnitLog2, "units");
constexpr uint32_t kGroupWarpMax = 512;                        // kept entries of an item that a warp takes
constexpr uint32_t kGroupChunk   = 4096;                       // ... that the block takes at a time (a whole unit)
constexpr uint32_t kGroupUnits   = 256;                        // units of the largest group
constexpr uint32_t kGroupPad     = 256;                        // bytes of a unit's place for the gaps between its groups' blobs (16-byte places)

// Entries of unit `unit` of gradient j that reach thr_e, in order, by one warp: put(rank, key in the unit, value).  Returns their number.
template <typename F>
__device__ __forceinline__ uint32_t unit_again(const EncArgs& a, uint32_t j, uint32_t unit, float thr_e, int lane, F put) {
    uint32_t rank = 0u;
    const uint64_t e0 = (uint64_t)unit << kUnitLog2;
#pragma unroll 1
    for (uint32_t r0 = 0; r0 < kUnit / 128u; r0 += 4u) {
        float4 row[4];                                         // (asked for together: the scans below wait for each in turn)
#pragma unroll
        for (uint32_t r = 0; r < 4u; ++r) row[r] = load4_guarded(a.grad[j], e0 + 128u * (r0 + r) + 4u * (uint32_t)lane, a.n);
#pragma unroll
        for (uint32_t r = 0; r < 4u; ++r) {
            const uint32_t k = 128u * (r0 + r) + 4u * (uint32_t)lane;
            const float4 q = row[r];
            const uint32_t m = reach_mask(q, thr_e), own = (uint32_t)__popc(m), incl = warp_incl_scan(own, lane);
            uint32_t at = rank + incl - own;
            if (m & 1u) put(at++, k, q.x);
            if (m & 2u) put(at++, k + 1u, q.y);
            if (m & 4u) put(at++, k + 2u, q.z);
            if (m & 8u) put(at++, k + 3u, q.w);
            rank += __shfl_sync(kFullMask, incl, 31);
        }
    }
    return rank;
}

struct FilterShared {
    float    thr[kEncMaxJobs][132];
    double   S[kEncMaxJobs];
    double   nodes[kMaxChunks];
    uint32_t abort_flag;
};

__global__ void __launch_bounds__(kEncThreads, 2)
k_filter(const EncArgs a) {
    __shared__ FilterShared s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t units = 4u * a.G, U = a.J * units;
    if (tid == 0) s.abort_flag = 0u;
    allow_next_kernel();
    wait_for_previous_kernels();
    __syncthreads();
    if (!gradient_bounds(a, s, s.nodes, tid, lane, warp)) return;
    for (uint32_t u = blockIdx.x + gridDim.x * (uint32_t)warp; u < U; u += gridDim.x * (uint32_t)kEncWarps) {
        const uint32_t j = u / units;
        const float thr_e = s.thr[j][a.tau], most = __ldcg(a.umax + u);
        const UnitInfo in = load_info(a.info + u);
        uint32_t count = 0u, piece = in.piece, room = in.room;
        if (most >= thr_e && thr_e < __int_as_float(0x7f800000)) {
            if (in.sthr <= thr_e) {
                // in place: a code lies before its value, a key not behind its candidate's
                const List x = list_of(a, u, in);
                count = unit_list(x, in.count, s.thr[j], a.tau, const_cast<uint16_t*>(x.k), reinterpret_cast<uint8_t*>(const_cast<float*>(x.v)), lane);
            } else {
                count = unit_again(a, j, u - j * units, thr_e, lane, [](uint32_t, uint32_t, float) {});
                room = kSlotEntries;
                if (count > kSlotEntries) {
                    room = max(128u, ((count + 3u) / 4u + 31u) & ~31u);
                    if (lane == 0) piece = pool_take(a, room * 4u + count * 2u + kGroupPad);
                    piece = __shfl_sync(kFullMask, piece, 0);
                    if (piece == kNoPlace) room = 0u;          // (the entries are read again wherever they are needed)
                }
                if (room != 0u) {
                    UnitInfo to = in;
                    to.piece = piece; to.room = room;
                    const List x = list_of(a, u, to);
                    uint16_t* keys = const_cast<uint16_t*>(x.k);
                    uint8_t* codes = reinterpret_cast<uint8_t*>(const_cast<float*>(x.v));
                    const CodeTable ct(s.thr[j], a.tau);
                    unit_again(a, j, u - j * units, thr_e, lane, [&](uint32_t q, uint32_t k, float v) { keys[q] = (uint16_t)k; codes[q] = (uint8_t)code_byte_of(ct, v); });
                }
                if (lane == 0) atomicAdd(&a.ctl->ne_count[j], 1u);
            }
        }
        if (lane == 0) *reinterpret_cast<uint4*>(a.info + u) = make_uint4(count, piece, room, 0u);
    }
}

// ---- packing -----------------------------------------------------------------------------------
// A thread's run of consecutive entries (the groups' keys may need 20 bits and start anywhere); beyond its end delta 0.
struct WideRun {
    const uint32_t* keys; const uint8_t* codes; int left; uint32_t prev;
    // entries q0 .. of count; before: the key before entry 0
    __device__ __forceinline__ WideRun(const uint32_t* k, const uint8_t* c, uint32_t q0, uint32_t most, uint32_t count, uint32_t before)
        : keys(k + q0), codes(c + q0), left(q0 < count ? (int)min(most, count - q0) : 0), prev(q0 && q0 < count ? k[q0 - 1u] : before) {}
    __device__ __forceinline__ void next4(uint32_t (&d)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) { const uint32_t k = i < left ? keys[i] : prev; d[i] = k - prev; prev = k; }
        keys += 4; codes += 4; left -= 4;
    }
};
__device__ __forceinline__ uint32_t wide_max(WideRun r, uint32_t quads) {
    uint32_t top = 0u, d[4];
    if (r.left <= 0) quads = 0u;
    for (uint32_t c = 0; c < quads; ++c) { r.next4(d); top = max(max(top, max(d[0], d[1])), max(d[2], d[3])); }
    return __reduce_max_sync(kFullMask, top);
}
__device__ __forceinline__ uint32_t wide_bits(WideRun r, uint32_t quads, uint32_t shape, int least) {
    uint32_t bits = 0u, d[4];
    for (uint32_t c = 0; c < quads; ++c) {
        r.next4(d);
        if (r.left <= -4) { d[0] = d[1] = d[2] = d[3] = 0u; }
#pragma unroll
        for (int i = 0; i < 4; ++i) bits += __shfl_sync(kFullMask, shape, i ? top_bit(d[i]) : max(top_bit(d[0]), least)) & 0xFFFFu;
        least = -1;
    }
    return bits;
}
__device__ __forceinline__ void wide_write(WideRun r, uint32_t quads, uint32_t shape, int least, uint32_t l, BitRun bytes, BitRun flags, BitRun deltas) {
    uint32_t d[4];
    for (uint32_t c = 0; c < quads; ++c) {
        const int have = max(0, min(4, r.left));
        const uint8_t* codes = r.codes;
        r.next4(d);
        uint32_t f = 0u, b = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (have == 0) d[i] = 0u;
            const uint32_t x = __shfl_sync(kFullMask, shape, i ? top_bit(d[i]) : max(top_bit(d[0]), least));
            deltas.put(d[i], x & 0xFFFFu);
            if (i < have) { f = (f << l) | (x >> 16); b = (b << 8) | codes[i]; }
        }
        least = -1;
        flags.put(f, l * (uint32_t)have);
        bytes.put(b, 8u * (uint32_t)have);
    }
    deltas.close(); flags.close(); bytes.close();
}

// One group by one warp: count > 0 entries, keys from `start` (the group's first index) on.  The blob's place follows its size.
struct WarpGroup {
    uint32_t quads, q0, M, shape, dpos, words; int least;
    __device__ __forceinline__ WarpGroup(const uint32_t* keys, const uint8_t* codes, uint32_t count, uint32_t start, uint32_t l, int lane) {
        quads = (count + 127u) >> 7; q0 = 4u * quads * (uint32_t)lane;
        const WideRun r(keys, codes, q0, 4u * quads, count, start);
        M = max(1u, bit_length(wide_max(r, quads)));
        shape = delta_shape(l, M, lane); least = q0 == 0u ? 0 : -1;
        const uint32_t bits = wide_bits(r, quads, shape, least), incl = warp_incl_scan(bits, lane);
        dpos = (8u + l) * count + incl - bits;
        words = ((8u + l) * count + __shfl_sync(kFullMask, incl, 31) + 31u) >> 5;
    }
    __device__ __forceinline__ void write(const uint32_t* keys, const uint8_t* codes, uint32_t count, uint32_t start, uint32_t l, uint32_t* blob, int lane) const {
        for (uint32_t i = (uint32_t)lane; i < words; i += 32u) blob[i] = 0u;
        __syncwarp();
        wide_write(WideRun(keys, codes, q0, 4u * quads, count, start), quads, shape, least, l, BitRun(blob, 8u * q0), BitRun(blob, 8u * count + l * q0), BitRun(blob, dpos));
        __syncwarp();
    }
};

struct GroupShared {
    float    thr[132];
    uint32_t n_light, n_heavy, next_light, place, carry[3];
    uint16_t light[kEncThreads], heavy[kEncThreads];
    uint32_t warp_sum[kEncWarps], warp_max[kEncWarps];
    uint32_t off[kGroupUnits + 1];                             // kept entries before each unit of the item
    uint32_t sub_m[kEncWarps], sub_words[kEncWarps];
    struct Warp { uint32_t key[kGroupWarpMax]; uint8_t code[kGroupWarpMax]; uint32_t blob[(kGroupWarpMax * 33u + 31u) / 32u + 2u]; };
    struct Block { uint32_t key[kGroupChunk]; uint8_t code[kGroupChunk]; uint32_t bytes[kGroupChunk / 4 + 2], flags[kGroupChunk * 5 / 32 + 2], deltas[kGroupChunk * 20 / 32 + 2]; };
    union { Warp w[kEncWarps]; Block b; };
};
static_assert(2 * (sizeof(GroupShared) + 1024) <= 233472, "two blocks per SM (1 KiB per block is the system's)");

// What item i of gradient j is made of: its groups and units.
struct Item {
    uint32_t group0, groups, unit0, units;                     // (in the gradient)
    __device__ __forceinline__ Item(const EncArgs& a, uint32_t i) {
        if (a.group_log2 >= kUnitLog2) {
            const uint32_t up = a.group_log2 - kUnitLog2;
            group0 = i; groups = 1u; unit0 = i << up; units = min(1u << up, 4u * a.G - unit0);
        } else {
            const uint32_t down = kUnitLog2 - a.group_log2;
            group0 = i << down; groups = group0 < a.D ? min(1u << down, a.D - group0) : 0u; unit0 = i; units = 1u;
        }
    }
};
__device__ __forceinline__ uint32_t items_of(const EncArgs& a) { return a.group_log2 >= kUnitLog2 ? a.D : 4u * a.G; }

__device__ __forceinline__ void record_group(const EncArgs& a, uint32_t j, uint32_t group, uint32_t count, uint32_t M, uint32_t words, uint32_t place) {
    a.desc[(uint64_t)j * a.D + group] = count ? tile_desc(count, M, words) : 0ull;
    a.blob[(uint64_t)j * a.D + group] = place;
    if (count) atomicAdd(&a.seg[j * a.segments + (group >> a.seg_log2)], ((unsigned long long)count << 32) | words);
    if (count && place == kNoPlace) atomicAdd(&a.st->noblob, 1u);
}

// An item by the block.  dst == nullptr: sizes, the blobs to places of their own where there are any; else the blobs to dst and onwards.
__device__ __forceinline__ void block_item(const EncArgs& a, GroupShared& s, uint32_t j, const Item& it, uint32_t* dst, int tid, int lane, int warp) {
    const uint32_t ubase = 4u * a.G * j + it.unit0;
    // kept entries before each unit; units that have to be read again
    UnitInfo in; in.count = 0u; in.room = 1u; in.piece = 0u;
    if ((uint32_t)tid < it.units) in = load_info(a.info + ubase + tid);
    {
        const uint32_t incl = warp_incl_scan(in.count, lane);
        if (lane == 31) s.warp_sum[warp] = incl;
        __syncthreads();
        const uint32_t w = lane < kEncWarps ? s.warp_sum[lane] : 0u, wi = warp_incl_scan(w, lane);
        const uint32_t upto = __shfl_sync(kFullMask, wi - w, warp) + incl;
        if ((uint32_t)tid < it.units) s.off[tid + 1] = upto;
        if (tid == 0) { s.off[0] = 0u; s.carry[0] = 0u; s.carry[1] = 0u; s.carry[2] = 0u; }
    }
    const bool again = __syncthreads_or(in.count != 0u && in.room == 0u) != 0;
    const uint32_t count = s.off[it.units];
    if (again) {
        const double S = __ldcg(&a.st->S[j]);
        for (uint32_t k = (uint32_t)tid; k <= a.tau; k += kEncThreads) s.thr[k] = boundary(S, __ldcg(a.st->pw + k), __ldcg(a.st->inv + k));
        if (tid == kEncThreads - 1) table_hints(S, a.base, &s.thr[130]);
        __syncthreads();
    }
    // entries from r0 on, as many as the chunk holds (again: a unit's)
    uint32_t unit = 0u;
    auto load_chunk = [&](uint32_t r0) -> uint32_t {
        uint32_t r1 = min(count, r0 + kGroupChunk);
        if (again) {
            while (s.off[unit + 1u] <= r0) ++unit;             // (the same in every thread)
            r1 = s.off[unit + 1u];
            const UnitInfo x = load_info(a.info + ubase + unit);
            if (x.room == 0u) {
                const CodeTable ct(s.thr, a.tau);
                if (warp == 0) unit_again(a, j, it.unit0 + unit, s.thr[a.tau], lane, [&](uint32_t q, uint32_t k, float v) {
                    s.b.key[q] = (unit << kUnitLog2) + k; s.b.code[q] = (uint8_t)code_byte_of(ct, v);
                });
                __syncthreads();
                return r1 - r0;
            }
        }
        for (uint32_t e = r0 + (uint32_t)tid; e < r1; e += kEncThreads) {
            uint32_t lo = 0u, hi = it.units;                   // the last unit that starts at or before e
            while (hi - lo > 1u) { const uint32_t m = (lo + hi) >> 1; if (s.off[m] <= e) lo = m; else hi = m; }
            const UnitInfo x = load_info(a.info + ubase + lo);
            const List y = list_of(a, ubase + lo, x);
            s.b.key[e - r0] = (lo << kUnitLog2) + ((uint32_t)__ldcg(y.k + (e - s.off[lo])) & (kUnit - 1u));
            s.b.code[e - r0] = __ldcg(reinterpret_cast<const uint8_t*>(y.v) + (e - s.off[lo]));
        }
        __syncthreads();
        return r1 - r0;
    };
    if (a.group_log2 < kUnitLog2) {
        // the unit's groups, a warp each
        load_chunk(0u);
        static_assert(1u << (kUnitLog2 - 8u) == (uint32_t)kEncWarps, "a warp per group of a unit");
        const uint32_t p = (uint32_t)warp, start = p << a.group_log2;
        auto first_at = [&](uint32_t key) -> uint32_t {        // entries before `key`
            uint32_t lo = 0u, hi = count;
            while (lo < hi) { const uint32_t m = (lo + hi) >> 1; if (s.b.key[m] < key) lo = m + 1u; else hi = m; }
            return lo;
        };
        const bool mine = p < it.groups;
        const uint32_t q0 = mine ? first_at(start) : 0u, n = mine ? first_at(start + (1u << a.group_log2)) - q0 : 0u;
        const WarpGroup wg(s.b.key + q0, s.b.code + q0, n, start, a.l, lane);
        if (lane == 0) { s.sub_m[warp] = wg.M; s.sub_words[warp] = n ? wg.words : 0u; }
        __syncthreads();
        uint32_t at = 0u, all = 0u;                            // (in places of their own the blobs start at multiples of 16 bytes)
        for (uint32_t i = 0; i < (uint32_t)kEncWarps; ++i) {
            const uint32_t w = dst ? s.sub_words[i] : (s.sub_words[i] + 3u) & ~3u;
            if (i < p) at += w;
            all += w;
        }
        if (dst == nullptr && tid == 0) {
            const UnitInfo x = load_info(a.info + ubase);
            s.place = x.room == kSlotEntries ? (ubase * kUnitSlotBytes) / 16u : x.room ? x.piece : pool_take(a, all * 4u);
        }
        __syncthreads();
        const uint32_t place = dst ? 0u : s.place;
        if (n && place != kNoPlace) {
            uint32_t* blob = s.b.bytes + at;                   // (bytes, flags and deltas: one area; 24 bits an entry at most)
            wg.write(s.b.key + q0, s.b.code + q0, n, start, a.l, blob, lane);
            uint32_t* to = (dst ? dst : reinterpret_cast<uint32_t*>(a.scratch + 16ull * place)) + at;
            for (uint32_t i = (uint32_t)lane; i < wg.words; i += 32u) to[i] = bswap32(blob[i]);
        }
        if (dst == nullptr && mine && lane == 0) record_group(a, j, it.group0 + p, n, wg.M, wg.words, place == kNoPlace ? kNoPlace : place + at / 4u);
        __syncthreads();
        return;
    }
    // ---- one group: its largest delta (a group of one chunk stays where it is)
    uint32_t top = 0u, last = 0u, have = 0u;
    for (uint32_t r0 = 0; r0 < count; r0 += have) {
        have = load_chunk(r0);
        const uint32_t quads = (have + 4u * kEncThreads - 1u) / (4u * kEncThreads), q0 = 4u * quads * (uint32_t)tid;
        top = max(top, wide_max(WideRun(s.b.key, s.b.code, q0, 4u * quads, have, last), quads));
        last = s.b.key[have - 1u];
        if (have < count) __syncthreads();
    }
    const bool one = have == count;
    if (lane == 0) s.warp_max[warp] = top;
    __syncthreads();
    top = __reduce_max_sync(kFullMask, lane < kEncWarps ? s.warp_max[lane] : 0u);
    const uint32_t M = max(1u, bit_length(top)), shape = delta_shape(a.l, M, lane), delta0 = (8u + a.l) * count;
    // a place of its own: the units' slots (their entries have been read, if they are all here), or a piece of the pool
    const uint32_t bound = (count * (8u + a.l + M) + 31u) >> 5;
    if (dst == nullptr) {
        if (tid == 0) s.place = one && bound * 4u <= it.units * kUnitSlotBytes ? (ubase * kUnitSlotBytes) / 16u : pool_take(a, bound * 4u);
        __syncthreads();
    }
    const uint32_t place = dst ? 0u : s.place;
    uint32_t* to = dst ? dst : place != kNoPlace ? reinterpret_cast<uint32_t*>(a.scratch + 16ull * place) : nullptr;
    uint32_t dpos = delta0;
    last = 0u; unit = 0u;
    for (uint32_t r0 = 0; r0 < count; r0 += have) {
        if (!one) { __syncthreads(); have = load_chunk(r0); }
        const uint32_t quads = (have + 4u * kEncThreads - 1u) / (4u * kEncThreads), q0 = 4u * quads * (uint32_t)tid;
        const WideRun r(s.b.key, s.b.code, q0, 4u * quads, have, last);
        const int least = r0 + q0 == 0u ? 0 : -1;
        const uint32_t bits = wide_bits(r, quads, shape, least), incl = warp_incl_scan(bits, lane);
        if (lane == 31) s.warp_sum[warp] = incl;
        // three pieces of the blob, from the words on in which they start: what the piece before left in those words goes first
        const uint32_t p0 = 8u * r0, p1 = 8u * count + a.l * r0, e0 = p0 + 8u * have, e1 = p1 + a.l * have;
        for (uint32_t i = (uint32_t)tid; i < kGroupChunk / 4u + 2u; i += kEncThreads) s.b.bytes[i] = i ? 0u : s.carry[0];
        for (uint32_t i = (uint32_t)tid; i < kGroupChunk * 5u / 32u + 2u; i += kEncThreads) s.b.flags[i] = i ? 0u : s.carry[1];
        for (uint32_t i = (uint32_t)tid; i < kGroupChunk * 20u / 32u + 2u; i += kEncThreads) s.b.deltas[i] = i ? 0u : s.carry[2];
        __syncthreads();
        const uint32_t w = lane < kEncWarps ? s.warp_sum[lane] : 0u, wi = warp_incl_scan(w, lane);
        const uint32_t mine = __shfl_sync(kFullMask, wi - w, warp) + incl - bits, e2 = dpos + __shfl_sync(kFullMask, wi, 31);
        last = s.b.key[have - 1u];
        if (to != nullptr)
            wide_write(r, quads, shape, least, a.l, BitRun(s.b.bytes, (p0 & 31u) + 8u * q0), BitRun(s.b.flags, (p1 & 31u) + a.l * q0), BitRun(s.b.deltas, (dpos & 31u) + mine));
        __syncthreads();
        if (to != nullptr) {
            for (uint32_t i = (uint32_t)tid; i < (e0 >> 5) - (p0 >> 5); i += kEncThreads) to[(p0 >> 5) + i] = bswap32(s.b.bytes[i]);
            for (uint32_t i = (uint32_t)tid; i < (e1 >> 5) - (p1 >> 5); i += kEncThreads) to[(p1 >> 5) + i] = bswap32(s.b.flags[i]);
            for (uint32_t i = (uint32_t)tid; i < (e2 >> 5) - (dpos >> 5); i += kEncThreads) to[(dpos >> 5) + i] = bswap32(s.b.deltas[i]);
        }
        if (tid == 0) {
            s.carry[0] = (e0 & 31u) ? s.b.bytes[(e0 >> 5) - (p0 >> 5)] : 0u;
            s.carry[1] = (e1 & 31u) ? s.b.flags[(e1 >> 5) - (p1 >> 5)] : 0u;
            s.carry[2] = (e2 & 31u) ? s.b.deltas[(e2 >> 5) - (dpos >> 5)] : 0u;
        }
        dpos = e2;
    }
    __syncthreads();
    if (tid == 0) {
        if (to != nullptr) {
            // the words in which codes, flags and deltas end: with what the next parts put there
            const uint32_t end[3] = {8u * count, delta0, dpos};
            uint32_t word = 0u;
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const uint32_t at = end[x] >> 5;
                word |= s.carry[x];
                if (x < 2 && at == end[x + 1] >> 5) continue;  // (the next part ends in the same word)
                if (end[x] & 31u) to[at] = x < 2 ? bswap32(bswap32(to[at]) | word) : bswap32(word);
                word = 0u;
            }
        }
        if (dst == nullptr) record_group(a, j, it.group0, count, M, (dpos + 31u) >> 5, place);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kEncThreads, 2)
k_groups(const EncArgs a) {
    extern __shared__ __align__(128) unsigned char grp_smem_raw[];
    GroupShared& s = *reinterpret_cast<GroupShared*>(grp_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    allow_next_kernel();
    wait_for_previous_kernels();
    if (ld_acquire_u32(&a.ctl->error) != 0u) return;           // (the same answer in every block)
    const uint32_t per = items_of(a), I = a.J * per, B = gridDim.x, owned = blockIdx.x < I ? (I - blockIdx.x + B - 1u) / B : 0u;
    for (uint32_t first = 0; first < owned; first += kEncThreads) {
        if (tid == 0) { s.n_light = 0u; s.n_heavy = 0u; s.next_light = 0u; }
        __syncthreads();
        if (first + (uint32_t)tid < owned) {
            const uint32_t x = blockIdx.x + (first + (uint32_t)tid) * B, j = x / per;
            const Item it(a, x - j * per);
            uint32_t count = 0u;
            bool again = false;
#pragma unroll 8
            for (uint32_t u = 0; u < it.units; ++u) {
                const UnitInfo in = load_info(a.info + 4ull * a.G * j + it.unit0 + u);
                count += in.count;
                again = again || (in.count != 0u && in.room == 0u);
            }
            if (count == 0u) { for (uint32_t g = 0; g < it.groups; ++g) a.desc[(uint64_t)j * a.D + it.group0 + g] = 0ull; }
            else if (count <= kGroupWarpMax && !again) s.light[atomicAdd(&s.n_light, 1u)] = (uint16_t)tid;
            else s.heavy[atomicAdd(&s.n_heavy, 1u)] = (uint16_t)tid;
        }
        __syncthreads();
        for (uint32_t h = 0; h < s.n_heavy; ++h) {
            const uint32_t x = blockIdx.x + (first + s.heavy[h]) * B, j = x / per;
            block_item(a, s, j, Item(a, x - j * per), nullptr, tid, lane, warp);
        }
        for (;;) {
            uint32_t x = 0u;
            if (lane == 0) x = atomicAdd(&s.next_light, 1u);
            x = __shfl_sync(kFullMask, x, 0);
            if (x >= s.n_light) break;
            x = blockIdx.x + (first + s.light[x]) * B;
            const uint32_t j = x / per;
            const Item it(a, x - j * per);
            GroupShared::Warp& w = s.w[warp];
            const uint32_t ubase = 4u * a.G * j + it.unit0;
            // the item's entries, 32 units' at a time
            uint32_t count = 0u, place = ubase * kUnitSlotBytes / 16u;
            for (uint32_t u0 = 0; u0 < it.units; u0 += 32u) {
                UnitInfo in; in.count = 0u; in.piece = 0u; in.room = kSlotEntries;
                if (u0 + (uint32_t)lane < it.units) in = load_info(a.info + ubase + u0 + lane);
                if (it.units == 1u && __shfl_sync(kFullMask, in.room, 0) != kSlotEntries) place = __shfl_sync(kFullMask, in.piece, 0);
                const uint32_t incl = warp_incl_scan(in.count, lane), excl = incl - in.count, all = __shfl_sync(kFullMask, incl, 31);
                for (uint32_t e0 = 0; e0 < all; e0 += 32u) {
                    const uint32_t e = e0 + (uint32_t)lane;
                    uint32_t at = 0u;                          // the last unit that starts at or before e
#pragma unroll
                    for (uint32_t o = 16u; o > 0u; o >>= 1) { const uint32_t y = __shfl_sync(kFullMask, excl, at + o); if (y <= e) at += o; }
                    UnitInfo from;
                    from.piece = __shfl_sync(kFullMask, in.piece, at); from.room = __shfl_sync(kFullMask, in.room, at);
                    const uint32_t q = e - __shfl_sync(kFullMask, excl, at);
                    if (e < all) {
                        const List y = list_of(a, ubase + u0 + at, from);
                        w.key[count + e] = ((u0 + at) << kUnitLog2) + ((uint32_t)__ldcg(y.k + q) & (kUnit - 1u));
                        w.code[count + e] = __ldcg(reinterpret_cast<const uint8_t*>(y.v) + q);
                    }
                }
                count += all;
            }
            __syncwarp();
            if (a.group_log2 >= kUnitLog2) {
                const WarpGroup wg(w.key, w.code, count, 0u, a.l, lane);
                wg.write(w.key, w.code, count, 0u, a.l, w.blob, lane);
                // the units' slots, where the blob fits (a unit's own piece does): nothing in them is needed any more
                if (place == ubase * kUnitSlotBytes / 16u && wg.words * 4u > it.units * kUnitSlotBytes) {
                    if (lane == 0) place = pool_take(a, wg.words * 4u);
                    place = __shfl_sync(kFullMask, place, 0);
                }
                if (place != kNoPlace) {
                    uint32_t* to = reinterpret_cast<uint32_t*>(a.scratch + 16ull * place);
                    for (uint32_t i = (uint32_t)lane; i < wg.words; i += 32u) to[i] = bswap32(w.blob[i]);
                }
                if (lane == 0) record_group(a, j, it.group0, count, wg.M, wg.words, place);
            } else {
                // the unit's groups one after the other, their blobs in the place of the unit's list
                uint32_t q0 = 0u, total = 0u;
                for (uint32_t p = 0; p < it.groups; ++p) {
                    const uint32_t start = p << a.group_log2, end = start + (1u << a.group_log2);
                    uint32_t n = 0u;
                    for (uint32_t e = q0 + (uint32_t)lane;; e += 32u) {
                        const uint32_t m = __ballot_sync(kFullMask, e < count && w.key[min(e, kGroupWarpMax - 1u)] < end);
                        n += (uint32_t)__popc(m);
                        if (m != kFullMask) break;
                    }
                    uint32_t M = 0u, words = 0u;
                    if (n) {
                        const WarpGroup wg(w.key + q0, w.code + q0, n, start, a.l, lane);
                        wg.write(w.key + q0, w.code + q0, n, start, a.l, w.blob, lane);
                        M = wg.M; words = wg.words;
                        uint32_t* to = reinterpret_cast<uint32_t*>(a.scratch + 16ull * place);
                        for (uint32_t i = (uint32_t)lane; i < words; i += 32u) to[i] = bswap32(w.blob[i]);
                    }
                    if (lane == 0) {
                        a.desc[(uint64_t)j * a.D + it.group0 + p] = n ? tile_desc(n, M, words) : 0ull;
                        a.blob[(uint64_t)j * a.D + it.group0 + p] = place;
                    }
                    q0 += n; total += words; place += (words + 3u) / 4u;
                    __syncwarp();
                }
                // (a unit's groups lie in one segment)
                if (lane == 0) atomicAdd(&a.seg[j * a.segments + (it.group0 >> a.seg_log2)], ((unsigned long long)count << 32) | total);
            }
            __syncwarp();
        }
        __syncthreads();
    }
}

}  // namespace fsg
