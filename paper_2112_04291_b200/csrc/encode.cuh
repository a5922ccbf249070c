// The encoder for dense gradients: Algorithm 1 and, per group of 2^14 entries (a tile), Algorithm 2, for up to eight
// gradients of the same length.
//
// The threshold B_tau = sum / b^tau is known only when every entry has been read, so the definition reads a gradient twice.  Here
// it comes from memory once.
//
// k_resident: gradients that fit the GPU's shared memory, a tile per block (up to two blocks per SM).  The blocks exchange
// their tiles' sums and, later, sizes through tagged words of the workspace, everyone reading what it needs; one launch.
//
// Larger ones take three launches that overlap at their edges:
//   k_scan    streams the gradient.  A sample gives an estimate of the sum; every unit (a quarter of a tile) leaves its node of the
//             fixed fp64 tree, its largest |v|, and the list (key, value) of the entries that reach the estimated threshold,
//             lowered by a margin for the sampling error.
//   k_encode  the sum from the units' nodes (same tree), the exact boundaries.  A tile whose estimate was not above the threshold
//             has all its kept entries in its units' lists: filter, quantisation, delta keys, M, bit-packing; the blob
//             replaces the lists.  Where it was too high (or missing) the tile itself is read again, unless its largest |v| is
//             below the threshold.
//   k_place   the tiles' places in the stream by exclusive sums, directory, header, and the blobs copied there.
// The estimate steers only what is read again: which entries are kept and every bit of the stream follow from the exact sum.
#pragma once

#include "common.cuh"
#include "sum.cuh"
#include "bits.cuh"
#include "prims.cuh"

namespace fsg {

constexpr int      kEncThreads   = 512;
constexpr int      kEncWarps     = kEncThreads / 32;
constexpr uint32_t kTile         = 1u << kGroupLog2;           // entries per tile = per group
constexpr uint32_t kSlab         = kTile / kEncWarps;          // entries a warp takes at a time
static_assert(kSlab == 1024u, "eight rows of 128 entries per slab");
constexpr int      kEncMaxJobs   = 8;                          // gradients (simulated workers) one launch can take
constexpr uint32_t kMaxResident  = 320;                        // tiles k_resident can take (its exchange words in the workspace)

constexpr uint32_t kUnit         = 4u * kSlab;                 // entries of a unit, the quarter of a tile: what a warp of k_scan leaves a list of
constexpr uint32_t kSlotEntries  = 96;                         // candidates a unit may have in its own slot of the workspace; longer lists go to the pool
constexpr uint32_t kUnitSlotBytes = kSlotEntries * 6u;
constexpr uint32_t kSlotBytes    = 4u * kUnitSlotBytes;        // of a tile
constexpr uint32_t kSlotWords    = kSlotBytes / 4u;
constexpr uint32_t kListMost     = 2048;                       // units that promise more candidates are not listed: from half of the entries on, a list (8 bytes a candidate with its spare room, written and read) is more traffic than the unit's 16 KB once more
constexpr uint32_t kNoPlace      = 0xFFFFFFFFu;                // no room in the pool
constexpr uint32_t kSampleBlocks = 32;                         // blocks that sample one gradient, four entries at 768 places each
constexpr uint32_t kSamplePolls  = 64;                         // looks (0.7 us each) a block takes for another block's sample
constexpr uint32_t kTicketGroups = 8;
constexpr uint32_t kPools        = 32;
constexpr uint32_t kChunkUnits   = 512;                        // units under one node of the upper part of the sum tree
constexpr uint32_t kMaxChunks    = 1552;                       // such nodes in a launch
constexpr uint32_t kMaxSegments  = 1600;                       // segments of tiles (64 or more) whose sizes k_place scans
constexpr uint32_t kWarpListMax  = 4u * kSlotEntries, kUnitListMax = 768;      // candidates of a tile that one warp (all in slots), of a unit that one warp of four take

// Encoder state in the workspace's fixed part (zero between launches, except S and the tables; k_resident's exchange words are told
// apart by their tags).
struct EncState {
    alignas(16) unsigned long long res_node[2 * kMaxResident]; // k_resident: a tile's node, tag
    unsigned long long res_size[kMaxResident];                 // tag << 32 | kept entries << 16 | words
    unsigned long long sample[kEncMaxJobs][kSampleBlocks];     // a block's sum and sum of squares (two floats, the latter not 0); 0: not there yet
    uint32_t ticket[kTicketGroups][32];                        // k_scan: units handed out beyond each warp's first
    double   S[kEncMaxJobs];
    double   pw[132], inv[132];                                // b^k, 1 / b^k
    unsigned long long pool_used[kPools][16];                  // bytes in use of each pool
    uint32_t noblob;                                           // tiles (groups) k_place has to pack; stays until the next launch
};
static_assert(kEncStateOffset + sizeof(EncState) <= kQueueOffset, "fits before the decoder's queue");

struct alignas(16) UnitInfo { uint32_t count, piece, room; float sthr; };      // list: candidates, piece of the pool (16-byte units), entries it has room for (kSlotEntries: it is in the slot), what it was made with (+inf: no list)

struct EncArgs {
    const float*        grad[kEncMaxJobs];
    uint8_t*            out[kEncMaxJobs];
    uint64_t            out_bytes;
    uint64_t            n;
    Control*            ctl;
    EncState*           st;
    double*             partials;        // [J][4 G] units' nodes
    unsigned long long* chunk;           // [J][chunks] pairs: node of 512 units, 1 when it is there
    float*              umax;            // [J][4 G] largest |v|
    UnitInfo*           info;            // [J][4 G]
    unsigned long long* desc;            // [J][G] words << 32 | M << 24 | count
    uint32_t*           blob;            // [J][G] the packed blob's place in the scratch (16-byte units)
    unsigned long long* seg;             // [J][segments] kept entries << 32 | words of the segment's tiles
    unsigned char*      scratch;         // [J G] slots, then the pool
    uint64_t            pool_begin, pool_bytes;     // bytes: of one of the pools (below 2^32)
    uint32_t            pool_units;      // units that share a pool
    double              base;
    double              inv_ptau;        // 1 / b^tau (steers the estimate only)
    uint32_t            J, G;            // gradients; tiles of one
    uint32_t            D, group_log2;   // groups of one (the tiles, for the default size)
    uint32_t            chunks;          // of a gradient
    uint32_t            seg_log2, segments;
    uint32_t            scan_blocks, samplers;      // blocks of k_scan; blocks that sample each gradient
    uint32_t            tau, l;
    uint32_t            wait_limit, try_limit;      // polls before a wait on another block, tries before a wait on a bulk copy gives up
};

__device__ __forceinline__ unsigned long long tile_desc(uint32_t count, uint32_t M, uint32_t words) {
    return ((unsigned long long)words << 32) | (M << 24) | count;
}
__device__ __forceinline__ UnitInfo load_info(const UnitInfo* p) {
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(p));
    UnitInfo in;
    in.count = q.x; in.piece = q.y; in.room = q.z; in.sthr = __uint_as_float(q.w);
    return in;
}
// A piece of the pool (16-byte units), or kNoPlace.  The pool is 32 pools, a block's own first: atomics on one address go at 0.3 a
// nanosecond, which was 10 us when the first slabs of 3000 units asked at once and 55 us of the 65 us scan of 2^26 entries.
// A piece may not reach beyond a pool's first `limit` bytes.  What a refusal adds to a counter is lost to others: pools other than the
// block's own, and (look) that one too, are asked only after a look.  fill: how far the piece's pool is used.
__device__ __forceinline__ uint32_t pool_take(const EncArgs& a, uint32_t bytes, uint64_t limit, bool look, uint64_t& fill) {
    const unsigned long long b = (bytes + 15u) & ~15u;
#pragma unroll 1                                               // (unrolled, its code costs the kernels around it 5 to 10 %)
    for (uint32_t i = 0; i < kPools; ++i) {
        const uint32_t p = (blockIdx.x + i) % kPools;
        if ((i || look) && ld_relaxed_u64(&a.st->pool_used[p][0]) + b > limit) continue;
        const unsigned long long at = atomicAdd(&a.st->pool_used[p][0], b);
        fill = at + b;
        if (at + b <= limit) return (uint32_t)((a.pool_begin + p * a.pool_bytes + at) >> 4);
    }
    return kNoPlace;
}
__device__ __forceinline__ uint32_t pool_take(const EncArgs& a, uint32_t bytes) { uint64_t fill; return pool_take(a, bytes, a.pool_bytes, false, fill); }
// How far lists of `entries` candidates a unit may fill a pool: so far that the tiles that then have none find room for their blobs
// there, unless these fit the tiles' slots.  A list takes about 8 bytes a candidate, a blob at most 2.25 (up to 18 bits an entry): with x
// units listed of the U that share a pool, 8 e x + 2.25 e (U - x) <= pool bytes.  Eight gradients of 335 M, a tenth kept: lists
// without a limit filled the pool, and four tiles in five were packed twice.
__device__ __forceinline__ uint32_t lists_limit(const EncArgs& a, uint32_t entries) {
    const uint32_t pool = (uint32_t)a.pool_bytes, blobs = entries * a.pool_units / 4u * 9u;
    if (8u * entries <= kSlotBytes) return pool;
    const uint32_t rest = pool > blobs ? pool - blobs : 0u;
    return min(pool, rest + rest / 3u);
}

// RU32(B_k) for one gradient: |v| >= B_k on an fp32 |v| equals |v| >= RU32(B_k); never below the smallest denormal, because an entry
// must also be non-zero to be kept; nothing is kept of an all-zero gradient or one whose sum is not finite.  The quotient is
// formed as a product with the reciprocal (within 2^-51 of it) whenever everything within 2^-50 of the product rounds alike.
__device__ __forceinline__ float boundary(double S, double pk, double inv_pk) {
    if (!isfinite(S) || S == 0.0) return __int_as_float(0x7f800000);
    const double q = __dmul_rn(S, inv_pk);
    const float lo = __double2float_ru(__dmul_rn(q, 1.0 - 0x1p-50)), hi = __double2float_ru(__dmul_rn(q, 1.0 + 0x1p-50));
    return fmaxf(lo == hi ? lo : __double2float_ru(__ddiv_rn(S, pk)), __int_as_float(1));
}

__device__ __forceinline__ uint32_t reach_mask(float4 q, float thr) {
    return (fabsf(q.x) >= thr ? 1u : 0u) | (fabsf(q.y) >= thr ? 2u : 0u) | (fabsf(q.z) >= thr ? 4u : 0u) | (fabsf(q.w) >= thr ? 8u : 0u);
}

// A warp's slab in shared memory: lane l holds entries 32 l .. 32 l + 31, eight 16-byte pieces of which the r-th it reads is piece
// r ^ (l & 7): free of bank conflicts, and siblings of the sum tree stay siblings (addition commutes).  Node of the slab:
__device__ __forceinline__ double slab_node(const float4 (&v)[8]) {
    double x[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) x[r] = abs_sum4(v[r]);
    return warp_tree(__dadd_rn(__dadd_rn(__dadd_rn(x[0], x[1]), __dadd_rn(x[2], x[3])), __dadd_rn(__dadd_rn(x[4], x[5]), __dadd_rn(x[6], x[7]))));
}
__device__ __forceinline__ void slab_read(const float* slab, float4 (&v)[8], int lane) {
    const float4* mine = reinterpret_cast<const float4*>(slab) + 8 * lane;
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = mine[r ^ (lane & 7)];
}
// ... and which of the lane's entries reach thr: bit i <-> entry 32 l + i
__device__ __forceinline__ uint32_t slab_mask(const float4 (&v)[8], float thr, int lane) {
    uint32_t m = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r) m |= reach_mask(v[r], thr) << (4 * r);
    if (lane & 1) m = ((m & 0x0F0F0F0Fu) << 4) | ((m >> 4) & 0x0F0F0F0Fu);        // pieces into index order
    if (lane & 2) m = __byte_perm(m, 0u, 0x2301);
    if (lane & 4) m = __byte_perm(m, 0u, 0x1032);
    return m;
}

// ---- teams: one, four or sixteen warps on one tile ------------------------------------------------------
// The kept entries' keys stand in shared memory in index order, their code bytes already in the blob (big-endian valued words); flags
// and deltas are packed behind the codes.
struct TeamScratch { uint32_t cnt[kEncWarps], maxd[kEncWarps], first[4], last[4], bits[kEncWarps], room[4], piece[4], word; };

template <int W> __device__ __forceinline__ void team_sync(int id) {
    if constexpr (W == 1) __syncwarp();
    else if constexpr (W == 4) asm volatile("bar.sync %0, 128;" ::"r"(id + 1) : "memory");
    else __syncthreads();
}

__device__ __forceinline__ void put_code(uint32_t* blob, uint32_t q, uint32_t code) { reinterpret_cast<uint8_t*>(blob)[q ^ 3u] = (uint8_t)code; }

// Appends bit fields to a zeroed blob from any bit position on (its first and last words are shared with neighbours).
struct BitRun {
    uint32_t *at, cur, fill;
    __device__ __forceinline__ BitRun(uint32_t* blob, uint32_t pos) : at(blob + (pos >> 5)), cur(0u), fill(pos & 31u) {}
    // a value of `width` (0 to 32) bits; width 0: value 0
    __device__ __forceinline__ void put(uint32_t value, uint32_t width) {
        const uint32_t x = value << ((32u - width) & 31u), end = fill + width;
        cur |= x >> fill;
        if (end >= 32u) {
            atomicOr(at++, cur);
            cur = __funnelshift_r(0u, x, fill);
        }
        fill = end & 31u;
    }
    __device__ __forceinline__ void close() { if (cur) atomicOr(at, cur); }
};

// A thread's run of consecutive entries, taken four at a time (keys ascend: two deltas to a register without a borrow from one to the
// other); entries beyond the run's end have delta 0.
struct KeyRun {
    const uint16_t* keys;                                      // 8-byte aligned
    int left;                                                  // entries not yet taken (0 or less: none)
    uint32_t prev;                                             // the key before them
    __device__ __forceinline__ uint2 next4() {
        uint2 d = make_uint2(0u, 0u);
        if (left > 0) {
            uint2 k = *reinterpret_cast<const uint2*>(keys);
            if (left < 4) {                                    // (the last run's last entries)
                const uint32_t last = keys[left - 1];
                if (left == 1) k.x = last * 0x10001u;
                k.y = last * 0x10001u;
            }
            d.x = k.x - __byte_perm(prev, k.x, 0x5410);
            d.y = k.y - __byte_perm(k.x, k.y, 0x5432);
            prev = k.y >> 16;
        }
        keys += 4;
        left -= 4;
        return d;
    }
};

// The largest delta of the warp's runs (of up to 4 `quads` entries).
__device__ __forceinline__ uint32_t runs_max(KeyRun r, uint32_t quads) {
    uint32_t top = 0u;
    for (uint32_t c = 0; c < quads; ++c) {
        const uint2 d = r.next4();
        top = __vmaxu2(top, __vmaxu2(d.x, d.y));
    }
    return __reduce_max_sync(kFullMask, max(top & 0xFFFFu, top >> 16));
}

// Width in bits and flag of a delta of b bits, held by lane b - 1: flag << 16 | width.  0 bits (lane 31): no entry (the only delta of 0,
// that of a first key 0, goes by 1 bit: the same flag).
__device__ __forceinline__ uint32_t delta_shape(uint32_t l, uint32_t M, int lane) {
    if (lane == 31) return 0u;
    const uint32_t flag = flag_of((2u << lane) - 1u, l, c_inv_m[M]);
    return (flag << 16) | (((flag + 1u) * M + (1u << l) - 1u) >> l);
}
__device__ __forceinline__ uint32_t bit_length(uint32_t x) { return 32u - (uint32_t)__clz((int)x); }
// position of the highest bit; -1 (for a shuffle: lane 31) for 0
__device__ __forceinline__ int top_bit(uint32_t x) {
    int r;
    asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// Bits of the lane's run.  least: 0 where the run starts the group, else -1.
__device__ __forceinline__ uint32_t run_bits(KeyRun r, uint32_t quads, uint32_t shape, int least) {
    uint32_t bits = 0u;
    for (uint32_t c = 0; c < quads; ++c) {
        const uint2 d = r.next4();
        bits += __shfl_sync(kFullMask, shape, max(top_bit(d.x & 0xFFFFu), least)) + __shfl_sync(kFullMask, shape, top_bit(d.x >> 16));
        bits += __shfl_sync(kFullMask, shape, top_bit(d.y & 0xFFFFu)) + __shfl_sync(kFullMask, shape, top_bit(d.y >> 16));
        least = -1;
    }
    return bits & 0xFFFFu;
}

// Flags, deltas and (where codes is set: 4-byte aligned, a byte per entry) codes of the lane's run, which starts with entry q0 of count
// and with bit dpos of the blob.
template <bool kCodes>
__device__ __forceinline__ void write_runs(KeyRun r, uint32_t quads, uint32_t shape, int least, uint32_t l, uint32_t* blob, uint32_t count,
                                           uint32_t q0, uint32_t dpos, const uint8_t* codes) {
    BitRun deltas(blob, dpos), flags(blob, 8u * count + l * q0), bytes(blob, 8u * q0);
    for (uint32_t c = 0; c < quads; ++c) {
        const uint32_t have = (uint32_t)max(0, min(4, r.left));
        const uint2 d = r.next4();
        const uint32_t d0 = d.x & 0xFFFFu, d1 = d.x >> 16, d2 = d.y & 0xFFFFu, d3 = d.y >> 16;
        const uint32_t x0 = __shfl_sync(kFullMask, shape, max(top_bit(d0), least)), x1 = __shfl_sync(kFullMask, shape, top_bit(d1));
        const uint32_t x2 = __shfl_sync(kFullMask, shape, top_bit(d2)), x3 = __shfl_sync(kFullMask, shape, top_bit(d3));
        static_assert(kGroupLog2 <= 16, "two deltas to a word");
        deltas.put((d0 << (x1 & 0xFFFFu)) | d1, (x0 + x1) & 0xFFFFu);
        deltas.put((d2 << (x3 & 0xFFFFu)) | d3, (x2 + x3) & 0xFFFFu);
        const uint32_t f = ((((((x0 >> 16) << l) | (x1 >> 16)) << l) | (x2 >> 16)) << l) | (x3 >> 16);
        least = -1;
        if (have) {                                            // (a part of four only at the end of the last run)
            flags.put(f >> (l * (4u - have)), l * have);
            if constexpr (kCodes) bytes.put(bswap32(reinterpret_cast<const uint32_t*>(codes)[c]) >> (8u * (4u - have)), 8u * have);
        }
    }
    deltas.close();
    flags.close();
    if constexpr (kCodes) bytes.close();
}

// Packs flags and deltas of count > 0 entries whose keys (ascending; behind a barrier) and codes (W > 1: with or without) the team has
// written; sized(words) is called by every thread as soon as the size is known.  The blob is complete when the call returns M.  A thread
// takes a run of consecutive entries: widths and bits are added up in registers, one scan over the threads gives each run its place.
template <int W, typename F>
__device__ __forceinline__ uint32_t team_pack(uint32_t l, const uint16_t* keys, uint32_t* blob, uint32_t count, TeamScratch& s, int w, int lane, int id, F sized) {
    const uint32_t quads = (count + 128u * W - 1u) / (128u * W), q0 = 4u * quads * (uint32_t)(32 * w + lane);
    KeyRun r;
    r.keys = keys + q0; r.left = q0 < count ? (int)min(4u * quads, count - q0) : 0; r.prev = q0 && q0 < count ? (uint32_t)keys[q0 - 1u] : 0u;
    uint32_t top = runs_max(r, quads);
    if constexpr (W > 1) {
        if (lane == 0) s.maxd[w] = top;
        team_sync<W>(id);
        top = __reduce_max_sync(kFullMask, lane < W ? s.maxd[lane] : 0u);
    }
    const uint32_t M = max(1u, bit_length(top)), shape = delta_shape(l, M, lane);
    const int least = q0 == 0u ? 0 : -1;
    const uint32_t bits = run_bits(r, quads, shape, least), incl = warp_incl_scan(bits, lane);
    if (W > 1 && lane == 31) s.bits[w] = incl;
    // zeroes behind the codes
    if (w == 0 && lane == 0 && (count & 3u)) blob[count >> 2] &= 0xFFFFFFFFu << (32u - 8u * (count & 3u));
    const uint32_t bound = (count * (8u + l + M) + 31u) >> 5, delta0 = (8u + l) * count;
    for (uint32_t i = ((count + 3u) >> 2) + (uint32_t)(w * 32 + lane); i <= bound; i += 32u * W) blob[i] = 0u;
    team_sync<W>(id);
    uint32_t dpos = delta0 + incl - bits, all = __shfl_sync(kFullMask, incl, 31);
    if constexpr (W > 1) {
        const uint32_t x = lane < W ? s.bits[lane] : 0u, xi = warp_incl_scan(x, lane);
        dpos += __shfl_sync(kFullMask, xi - x, w);
        all = __shfl_sync(kFullMask, xi, 31);
    }
    sized((delta0 + all + 31u) >> 5);
    write_runs<false>(r, __any_sync(kFullMask, r.left > 0) ? quads : 0u, shape, least, l, blob, count, q0, dpos, nullptr);
    team_sync<W>(id);
    return M;
}

__device__ __forceinline__ void enc_write_header(const EncArgs& a, uint32_t j, int status, uint64_t d, uint64_t total_bytes, double S) {
    uint32_t* outw = reinterpret_cast<uint32_t*>(a.out[j]);
    if (status != kStOk) { d = 0ull; total_bytes = kHeaderBytes; }
    if (status == kStNonfinite || status == kStTimeout) S = 0.0;
    const unsigned long long sb = (unsigned long long)__double_as_longlong(S), bb = (unsigned long long)__double_as_longlong(a.base);
    outw[0] = kMagic;                   outw[1] = kVersion;
    outw[2] = (uint32_t)status;         outw[3] = a.tau;
    outw[4] = (uint32_t)a.n;            outw[5] = (uint32_t)(a.n >> 32);
    outw[6] = (uint32_t)d;              outw[7] = (uint32_t)(d >> 32);
    outw[8] = (uint32_t)total_bytes;    outw[9] = (uint32_t)(total_bytes >> 32);
    outw[10] = (uint32_t)sb;            outw[11] = (uint32_t)(sb >> 32);
    outw[12] = (uint32_t)bb;            outw[13] = (uint32_t)(bb >> 32);
    outw[14] = a.l | (a.group_log2 << 8);
    outw[15] = a.D;
}

// A unit's list of candidates: in its slot, or in a piece of the pool.
struct List { const float* v; const uint16_t* k; };
__device__ __forceinline__ List list_of(const EncArgs& a, uint32_t u, const UnitInfo& in) {
    List x;
    x.v = reinterpret_cast<const float*>(a.scratch + (in.room == kSlotEntries ? (uint64_t)u * kUnitSlotBytes : 16ull * in.piece));
    x.k = reinterpret_cast<const uint16_t*>(x.v + in.room);
    return x;
}

// Kept keys and codes of a tile from its units' lists, by the block: warp w takes its share of unit w / 4; returns the number of kept
// entries.
template <int W>
__device__ __forceinline__ uint32_t team_list(const EncArgs& a, uint32_t t, const float* thr, uint16_t* keys, uint32_t* blob, TeamScratch& s, int w, int lane, int id) {
    const float thr_e = thr[a.tau];
    const CodeTable ct(thr, a.tau);
    const uint32_t u = 4u * t + (uint32_t)w / (W / 4), part = (uint32_t)w % (W / 4);
    const UnitInfo in = load_info(a.info + u);
    const List x = list_of(a, u, in);
    const uint32_t cnt = __ldcg(a.umax + u) >= thr_e ? in.count : 0u;
    const uint32_t nb = (cnt + 31u) >> 5, b0 = nb * part / (W / 4), b1 = nb * (part + 1u) / (W / 4);
    const uint32_t end = min(cnt, 32u * b1);
    // how many are kept
    uint32_t n = 0u;
    for (uint32_t b = b0; b < b1; b += 4u) {
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = 32u * (b + i) + (uint32_t)lane < end ? __ldcg(x.v + 32u * (b + i) + lane) : 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) n += fabsf(v[i]) >= thr_e ? 1u : 0u;
    }
    n = __reduce_add_sync(kFullMask, n);
    if (lane == 0) s.cnt[w] = n;
    auto value = [&](uint32_t b) -> float { return 32u * b + (uint32_t)lane < end ? __ldcg(x.v + 32u * b + lane) : 0.0f; };
    auto key = [&](uint32_t b) -> uint32_t { return 32u * b + (uint32_t)lane < end ? __ldcg(x.k + 32u * b + lane) : 0u; };
    float v0 = value(b0), v1 = value(b0 + 1u);
    uint32_t k0 = key(b0), k1 = key(b0 + 1u);
    team_sync<W>(id);
    const uint32_t c = lane < W ? s.cnt[lane] : 0u, ci = warp_incl_scan(c, lane);
    uint32_t rank = __shfl_sync(kFullMask, ci - c, w);
    const uint32_t count = __shfl_sync(kFullMask, ci, 31), below = (1u << lane) - 1u;
    for (uint32_t b = b0; b < b1; ++b) {
        const float v2 = value(b + 2u);
        const uint32_t k2 = key(b + 2u);
        const bool kept = fabsf(v0) >= thr_e;
        const uint32_t km = __ballot_sync(kFullMask, kept);
        if (kept) {
            const uint32_t q = rank + (uint32_t)__popc(km & below);
            keys[q] = (uint16_t)k0;
            put_code(blob, q, code_byte_of(ct, v0));
        }
        rank += (uint32_t)__popc(km);
        v0 = v1; k0 = k1; v1 = v2; k1 = k2;
    }
    team_sync<W>(id);
    return count;
}

// The same by one warp for a whole unit, without ranks among the other units: keys and code bytes in the unit's own place (which may be
// that of its list).
__device__ __forceinline__ uint32_t unit_list(const List& x, uint32_t cnt, const float* thr, uint32_t tau, uint16_t* keys, uint8_t* codes, int lane) {
    const float thr_e = thr[tau];
    const CodeTable ct(thr, tau);
    uint32_t rank = 0u;
    const uint32_t below = (1u << lane) - 1u;
    auto value = [&](uint32_t e) -> float { return e + (uint32_t)lane < cnt ? __ldcg(x.v + e + lane) : 0.0f; };
    auto key = [&](uint32_t e) -> uint32_t { return e + (uint32_t)lane < cnt ? __ldcg(x.k + e + lane) : 0u; };
    float v[4]; uint32_t k[4];
#pragma unroll
    for (uint32_t i = 0; i < 4u; ++i) { v[i] = value(32u * i); k[i] = key(32u * i); }
    for (uint32_t e = 0; e < cnt; e += 128u) {
        float nv[4]; uint32_t nk[4];
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) { nv[i] = value(e + 128u + 32u * i); nk[i] = key(e + 128u + 32u * i); }
        __syncwarp();                                          // (keys and codes may go where the list is: all of it up to here has been read)
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            const bool kept = fabsf(v[i]) >= thr_e;
            const uint32_t km = __ballot_sync(kFullMask, kept);
            if (kept) {
                const uint32_t q = rank + (uint32_t)__popc(km & below);
                keys[q] = (uint16_t)k[i];
                codes[q] = (uint8_t)code_byte_of(ct, v[i]);
            }
            rank += (uint32_t)__popc(km);
            v[i] = nv[i]; k[i] = nk[i];
        }
    }
    return rank;
}

// The same by one warp, all candidates (off[q]: those of the units before unit q) in the units' slots.
__device__ __forceinline__ uint32_t warp_list(const EncArgs& a, uint32_t t, const uint32_t (&off)[5], const float* thr, uint16_t* keys, uint32_t* blob, int lane) {
    const float thr_e = thr[a.tau];
    const CodeTable ct(thr, a.tau);
    const unsigned char* slots = a.scratch + (uint64_t)t * kSlotBytes;
    auto load = [&](uint32_t e, float& v, uint32_t& k) {
        v = 0.0f; k = 0u;
        if (e >= off[4]) return;
        const uint32_t q = (e >= off[1] ? 1u : 0u) + (e >= off[2] ? 1u : 0u) + (e >= off[3] ? 1u : 0u);
        const uint32_t i = e - (q == 0u ? 0u : q == 1u ? off[1] : q == 2u ? off[2] : off[3]);
        const unsigned char* slot = slots + q * kUnitSlotBytes;
        v = __ldcg(reinterpret_cast<const float*>(slot) + i);
        k = __ldcg(reinterpret_cast<const uint16_t*>(slot + 4u * kSlotEntries) + i);
    };
    uint32_t rank = 0u, k0, k1, k2; float v0, v1, v2;
    const uint32_t below = (1u << lane) - 1u;
    load((uint32_t)lane, v0, k0);
    load(32u + (uint32_t)lane, v1, k1);
    for (uint32_t e = 0; e < off[4]; e += 32u) {
        load(e + 64u + (uint32_t)lane, v2, k2);
        const bool kept = fabsf(v0) >= thr_e;
        const uint32_t km = __ballot_sync(kFullMask, kept);
        if (kept) {
            const uint32_t q = rank + (uint32_t)__popc(km & below);
            keys[q] = (uint16_t)k0;
            put_code(blob, q, code_byte_of(ct, v0));
        }
        rank += (uint32_t)__popc(km);
        v0 = v1; k0 = k1; v1 = v2; k1 = k2;
    }
    __syncwarp();
    return rank;
}

// The same from the tile itself, by the whole block: the kept keys of warp w's slab, then the codes.
__device__ __forceinline__ uint32_t block_tile(const EncArgs& a, uint32_t j, uint32_t tile, const float* thr, uint16_t* keys, uint32_t* blob, TeamScratch& s,
                                               int tid, int lane, int warp) {
    const float* g = a.grad[j] + ((uint64_t)tile << kGroupLog2);
    const uint64_t left = a.n - ((uint64_t)tile << kGroupLog2);
    const float thr_e = thr[a.tau];
    const CodeTable ct(thr, a.tau);
    // (32 loads of consecutive entries: row i of the slab's 32 rows of 32; sixteen in flight, each needed by a ballot only when all of them
    // have been asked for)
    uint32_t mine = 0u, mask = 0u;
#pragma unroll 1
    for (int i0 = 0; i0 < 32; i0 += 16) {
        float x[16];
        const uint32_t e0 = (uint32_t)warp * kSlab + 32u * (uint32_t)i0 + (uint32_t)lane;
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = e0 + 32u * (uint32_t)i < left ? g[e0 + 32u * (uint32_t)i] : 0.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t b = __ballot_sync(kFullMask, fabsf(x[i]) >= thr_e);      // (thr_e > 0)
            if (lane == i0 + i) mask = b;                      // lane i: row i
            mine += (uint32_t)__popc(b);
        }
    }
    if (lane == 0) s.cnt[warp] = mine;
    __syncthreads();
    const uint32_t c = lane < kEncWarps ? s.cnt[lane] : 0u, ci = warp_incl_scan(c, lane);
    const uint32_t count = __shfl_sync(kFullMask, ci, 31);
    const uint32_t own = (uint32_t)__popc(mask), incl = warp_incl_scan(own, lane);
    uint32_t pos = __shfl_sync(kFullMask, ci - c, warp) + incl - own;
    for (; mask != 0u; mask &= mask - 1u, ++pos) keys[pos] = (uint16_t)((uint32_t)warp * kSlab + 32u * (uint32_t)lane + (uint32_t)__ffs((int)mask) - 1u);
    __syncthreads();
    for (uint32_t q = (uint32_t)tid; q < count; q += 4u * kEncThreads) {
        float x[4];
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) x[i] = q + i * kEncThreads < count ? g[keys[q + i * kEncThreads]] : 0.0f;
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) if (q + i * kEncThreads < count) put_code(blob, q + i * kEncThreads, code_byte_of(ct, x[i]));
    }
    return count;
}

// ---- k_resident ----------------------------------------------------------------------------------
struct ResShared {
    union alignas(128) {
        float    tile[kTile];
        uint32_t blob[kTile];            // 27 bits an entry at most; grows over the tile, whose values behind it are still needed
    };
    alignas(16) uint16_t key[kTile];
    unsigned long long mbar[kEncWarps];
    float    thr[132];
    double   node[kEncWarps], s_tree[kEncWarps];
    unsigned long long scan64[kEncWarps];
    TeamScratch team;
    uint32_t abort_flag, gen;
};
static_assert(2 * (sizeof(ResShared) + 1024) <= 233472, "two blocks per SM (1 KiB per block is the system's)");

// All blocks of the launch are resident (cooperative launch, or a single block).  A launch is a chain: start, copy, node, exchange,
// filter, sizes, exchange, pack, store; every link about a microsecond.  Per call, before (two grid barriers, the last block to arrive
// working for everybody) and now: 5003 entries 16.4 -> 9.6 us, 2^20 at 1 % 18.5 -> 13.0, 4.8 M at 10 % 27.0 -> 21.6.
__global__ void __launch_bounds__(kEncThreads, 2)
k_resident(const EncArgs a, const __grid_constant__ PowTable pw, const __grid_constant__ PowTable inv) {
    extern __shared__ __align__(128) unsigned char res_smem_raw[];
    ResShared& s = *reinterpret_cast<ResShared*>(res_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t t = blockIdx.x, j = t / a.G, tile = t - j * a.G;
    const uint64_t first = (uint64_t)tile << kGroupLog2;
    allow_next_kernel();
    if (lane == 0) {
        mbar_init(&s.mbar[warp], 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) s.abort_flag = 0u;
    __syncthreads();
    wait_for_previous_kernels();
    // ---- the warp's slab
    const uint64_t slab0 = first + (uint64_t)warp * kSlab;
    const uint32_t valid = slab0 < a.n ? (uint32_t)min((uint64_t)kSlab, a.n - slab0) : 0u;
    float* slab = s.tile + (uint32_t)warp * kSlab;
    if (valid == kSlab) {
        if (lane == 0) {
            mbar_expect_tx(&s.mbar[warp], kSlab * 4u);
            bulk_load(slab, a.grad[j] + slab0, kSlab * 4u, &s.mbar[warp]);
        }
    } else {
        for (uint32_t i = lane; i < kSlab; i += 32u) slab[i] = i < valid ? a.grad[j][slab0 + i] : 0.0f;
        __syncwarp();
    }
    if (tid == 0) s.gen = ld_acquire_u32(&a.ctl->bar_gen) + 1u;      // before this block lets others go on
    if (valid == kSlab && !mbar_wait(&s.mbar[warp], 0u, a.try_limit)) s.abort_flag = 1u;
    float4 v[8];
    slab_read(slab, v, lane);
    const double u = slab_node(v);
    if (lane == 0) s.node[warp] = u;
    __syncthreads();
    const uint32_t gen = s.gen;
    if (warp == 0) {
        const double T = warp_tree(lane < kEncWarps ? s.node[lane] : 0.0, kEncWarps);
        if (lane == 0) {
            st_relaxed_pair(a.st->res_node + 2u * t, (unsigned long long)__double_as_longlong(T), gen);
            atomicAdd(&a.ctl->bar_count[j], 1u);
        }
    }
    // ---- everybody reduces the gradient's tiles by itself (same tree)
    double y = 0.0;
    if ((uint32_t)tid < a.G) {
        unsigned long long lo, hi;
        uint32_t spin = 0;
        for (;;) {
            ld_relaxed_pair(a.st->res_node + 2u * (j * a.G + (uint32_t)tid), lo, hi);
            if (hi == gen) break;
            if (++spin > a.wait_limit) { s.abort_flag = 1u; break; }
        }
        y = __longlong_as_double((long long)lo);
    }
    const double S = block_tree(y, s.s_tree, lane, warp);
    for (uint32_t k = (uint32_t)tid; k <= a.tau; k += kEncThreads) s.thr[k] = boundary(S, pw.P[k], inv.P[k]);
    if (tid == kEncThreads - 1) table_hints(S, a.base, &s.thr[130]);
    __syncthreads();
    // ---- filter; keys in order
    const float thr_e = s.thr[a.tau];
    const CodeTable ct(s.thr, a.tau);
    uint32_t m = slab_mask(v, thr_e, lane);
    const uint32_t own = (uint32_t)__popc(m), incl = warp_incl_scan(own, lane);
    if (lane == 31) s.team.cnt[warp] = incl;
    __syncthreads();
    const uint32_t c = lane < kEncWarps ? s.team.cnt[lane] : 0u, ci = warp_incl_scan(c, lane);
    const uint32_t count = __shfl_sync(kFullMask, ci, 31);
    for (uint32_t pos = __shfl_sync(kFullMask, ci - c, warp) + incl - own; m != 0u; m &= m - 1u, ++pos)
        s.key[pos] = (uint16_t)((uint32_t)warp * kSlab + 32u * (uint32_t)lane + (uint32_t)__ffs((int)m) - 1u);
    __syncthreads();
    // ---- codes: those of a round replace entries of the tile whose codes have been formed (rank <= key: a code lies before its value)
    for (uint32_t q0 = 0; q0 < count; q0 += kEncThreads) {
        const uint32_t q = q0 + (uint32_t)tid;
        uint32_t code = 0u;
        if (q < count) code = code_byte_of(ct, s.tile[s.key[q]]);
        __syncthreads();
        if (q < count) put_code(s.blob, q, code);
    }
    uint32_t words = 0u, M = 0u;
    auto publish = [&](uint32_t w) {
        words = w;
        if (tid == 0) st_relaxed_u64(a.st->res_size + t, ((unsigned long long)gen << 32) | (count << 16) | w);
    };
    if (count) M = team_pack<kEncWarps>(a.l, s.key, s.blob, count, s.team, warp, lane, 0, publish);
    else publish(0u);
    // ---- the tile's place: the sizes of the gradient's tiles before it
    unsigned long long z = 0ull;
    if ((uint32_t)tid < tile) {
        unsigned long long x;
        uint32_t spin = 0;
        for (;;) {
            x = ld_relaxed_u64(a.st->res_size + j * a.G + (uint32_t)tid);
            if ((uint32_t)(x >> 32) == gen) break;
            if (++spin > a.wait_limit) { s.abort_flag = 1u; break; }
        }
        z = ((x & 0xFFFF0000ull) << 16) | (x & 0xFFFFull);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(kFullMask, z, o);
    if (lane == 0) s.scan64[warp] = z;
    __syncthreads();
    z = lane < kEncWarps ? s.scan64[lane] : 0ull;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(kFullMask, z, o);
    z = __shfl_sync(kFullMask, z, 0);
    const uint32_t fixed_words = (kHeaderBytes + 8u * a.G) >> 2, off = fixed_words + (uint32_t)z;
    const uint64_t end_bytes = ((uint64_t)off + words) << 2;
    uint32_t* outw = reinterpret_cast<uint32_t*>(a.out[j]);
    if (!s.abort_flag) {
        if (end_bytes <= a.out_bytes)
            for (uint32_t i = (uint32_t)tid; i < words; i += kEncThreads) outw[off + i] = bswap32(s.blob[i]);
        if (tid == 0) *reinterpret_cast<uint2*>(outw + (kHeaderBytes >> 2) + 2u * tile) = make_uint2(count ? (count | (M << 24)) : 0u, off);
        if (tile == a.G - 1u && tid == 0) {
            uint32_t spin = 0;                                // (every tile has been summed: true since the first exchange)
            while (ld_acquire_u32(&a.ctl->bar_count[j]) != a.G) if (++spin > a.wait_limit) { s.abort_flag = 1u; break; }
            enc_write_header(a, j, !isfinite(S) ? kStNonfinite : end_bytes > a.out_bytes ? kStCapacity : kStOk, (z >> 32) + count, end_bytes, S);
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (s.abort_flag) {
            atomicExch(&a.ctl->error, (unsigned)kStTimeout);
            for (uint32_t i = 0; i < a.J; ++i) enc_write_header(a, i, kStTimeout, 0ull, 0ull, 0.0);
        }
        // the last block out readies the workspace for the next launch and has the final word on a timeout
        if (atom_add_acq_rel_u32(&a.ctl->exit_count, 1u) == gridDim.x - 1u) {
            if (ld_acquire_u32(&a.ctl->error) != 0u) for (uint32_t i = 0; i < a.J; ++i) enc_write_header(a, i, kStTimeout, 0ull, 0ull, 0.0);
            for (uint32_t i = 0; i < a.J; ++i) { a.ctl->bar_count[i] = 0u; a.ctl->ne_count[i] = 0u; }
            a.ctl->exit_count = 0u;
            st_release_u32(&a.ctl->bar_gen, gen);
        }
    }
}

// ---- k_scan ------------------------------------------------------------------------------------
// A warp takes whole units, slab after slab, through a ring of its own in shared memory: bulk copies of two slabs (8 KB a warp, 192 KB
// an SM) are in flight, no warp waits for another, and a unit's list is written in order as it goes.
//
// What bounds it is instructions and the latency of their chains: at 7 TB/s an SM has 160 cycles per slab.  A lane takes 32 consecutive
// entries (slab_read), so that five levels of the tree need no shuffles and the kept mask is in index order.  Measured on 1 GiB: rows of
// 128 entries across the warp 209 us; 32 warps that load into registers, slabs asked for in L2 ahead of time, 300 us; a fence and an
// atomic per tile 207 us; the rings alone, without arithmetic, 159 us.
constexpr int kScanThreads = 768;
constexpr int kScanWarps   = kScanThreads / 32;
constexpr int kRing        = 2;                                // slabs in flight per warp
struct ScanShared {
    alignas(128) float ring[kScanWarps][kRing][kSlab];
    unsigned long long mbar[kScanWarps][kRing];
    float samp[2][kScanWarps];
    float est[kEncMaxJobs];
    uint32_t refused;                                          // bytes of the shortest list the pools have refused one of the block's warps
    uint32_t nearly;                                           // the pools are close to their limit
};
static_assert(sizeof(ScanShared) <= 232448, "shared memory of one block");

__global__ void __launch_bounds__(kScanThreads, 1)
k_scan(const EncArgs a, const __grid_constant__ PowTable pw, const __grid_constant__ PowTable inv) {
    extern __shared__ __align__(128) unsigned char scan_smem_raw[];
    ScanShared& s = *reinterpret_cast<ScanShared*>(scan_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t units = 4u * a.G, T = a.J * units;
    allow_next_kernel();
    if (tid == 0) { s.refused = 0xFFFFFFFFu; s.nearly = 0u; }
    if (lane == 0) {
        for (int i = 0; i < kRing; ++i) mbar_init(&s.mbar[warp][i], 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    wait_for_previous_kernels();
    // unit k: unit k / J of gradient k % J (gradients interleaved).  Lane 0 starts the copy of one of its slabs; one that reaches beyond n
    // is read by its consumer instead.
    struct Where { const float* g; uint64_t left; };           // the unit's first entry, entries from there to the gradient's end
    auto where = [&](uint32_t k) -> Where {
        const uint32_t i = k / a.J;
        const uint64_t e = (uint64_t)i * kUnit;
        Where w;
        w.g = a.grad[k - i * a.J] + e; w.left = e < a.n ? a.n - e : 0ull;
        return w;
    };
    auto issue = [&](const Where& w, uint32_t slab, uint32_t slot) {
        if (w.left >= (slab + 1u) * kSlab) {
            mbar_expect_tx(&s.mbar[warp][slot], kSlab * 4u);
            bulk_load(s.ring[warp][slot], w.g + slab * kSlab, kSlab * 4u, &s.mbar[warp][slot]);
        } else {
            mbar_arrive(&s.mbar[warp][slot]);
        }
    };
    // ---- sample: blocks j, j + J, ... of the first J * samplers take gradient j; their loads go first, the rings are only half filled until
    // the estimate is there (behind full rings the sample took 20 us)
    const uint32_t sj = blockIdx.x % a.J, si = blockIdx.x / a.J;
    const bool sampler = si < a.samplers;
    float sx = 0.0f, sy = 0.0f;
    if (sampler) {
        const uint32_t places = (uint32_t)(a.n >> 2), count = a.samplers * (uint32_t)kScanThreads, step = places / count, at = si * (uint32_t)kScanThreads + (uint32_t)tid;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (places) q = reinterpret_cast<const float4*>(a.grad[sj])[step ? at * step + (step >> 1) : at % places];
        sx = fabsf(q.x) + fabsf(q.y) + fabsf(q.z) + fabsf(q.w);
        sy = sx * sx;
    }
    uint32_t cur = (uint32_t)warp * gridDim.x + blockIdx.x;
    Where here = where(min(cur, T - 1u));
    if (lane == 0 && cur < T) issue(here, 0u, 0u);
    if (sampler) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { sx += __shfl_xor_sync(kFullMask, sx, o); sy += __shfl_xor_sync(kFullMask, sy, o); }
        if (lane == 0) { s.samp[0][warp] = sx; s.samp[1][warp] = sy; }
        __syncthreads();
        if (warp == 0) {
            sx = lane < kScanWarps ? s.samp[0][lane] : 0.0f; sy = lane < kScanWarps ? s.samp[1][lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) { sx += __shfl_xor_sync(kFullMask, sx, o); sy += __shfl_xor_sync(kFullMask, sy, o); }
            if (lane == 0) st_relaxed_u64(&a.st->sample[sj][si], ((unsigned long long)__float_as_uint(sx) << 32) | max(__float_as_uint(sy), 1u));
        }
    }
    if (warp < (int)a.J) {
        // every block forms the estimates by itself: warp <-> gradient, lane <-> sampling block.  Margin: 2 % and three standard errors of the
        // mean of k samples
        static_assert(kSampleBlocks == 32u && kEncMaxJobs < kScanWarps, "a lane per sampling block, a warp per gradient");
        unsigned long long v = 1ull;
        if ((uint32_t)lane < a.samplers)
            for (uint32_t p = 0; p < kSamplePolls; ++p) if ((v = ld_relaxed_u64(&a.st->sample[warp][lane])) != 0ull) break;
        const bool all = __all_sync(kFullMask, v != 0ull);
        float x = __uint_as_float((uint32_t)(v >> 32)), y = __uint_as_float((uint32_t)v);
        if ((uint32_t)lane >= a.samplers) x = y = 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { x += __shfl_xor_sync(kFullMask, x, o); y += __shfl_xor_sync(kFullMask, y, o); }
        const float k = (float)(a.samplers * (uint32_t)kScanThreads), mean = x / k, var = fmaxf(y / k - mean * mean, 0.0f), margin = 0.02f + 3.0f * sqrtf(var / k) / mean;
        const float e = (float)((double)(mean * (1.0f - margin)) * (double)a.n * 0.25 * a.inv_ptau);
        if (lane == 0) s.est[warp] = all && margin < 0.75f && e > 0.0f ? e : -1.0f;
    } else {
        // (what k_encode adds to, exchanges and reads)
        const uint32_t others = (uint32_t)kScanThreads - 32u * a.J, x = (uint32_t)tid - 32u * a.J;
        for (uint32_t i = blockIdx.x * others + x; i < a.J * max(a.segments, 2u * a.chunks); i += gridDim.x * others) {
            if (i < a.J * a.segments) a.seg[i] = 0ull;
            if (i < 2u * a.J * a.chunks) a.chunk[i] = 0ull;
        }
        if (blockIdx.x == 0) {
            if (x < (uint32_t)kEncMaxJobs) a.ctl->ne_count[x] = 0u;
            if (x == 0u) a.st->noblob = 0u;
            if (x <= (uint32_t)kMaxTau) { a.st->pw[x] = pw.P[x]; a.st->inv[x] = inv.P[x]; }
        }
    }
    __syncthreads();
    if (lane == 0 && cur < T)
        for (uint32_t i = 1; i < (uint32_t)kRing; ++i) issue(here, i, i);

    const uint32_t groups = min(kTicketGroups, gridDim.x), tg = blockIdx.x % groups;
    uint32_t slot = 0u, parity = 0u;                           // bit i: the parity the next wait on slot i expects
    bool failed = false;
    while (cur < T && !failed) {
        const uint32_t i = cur / a.J, j = cur - i * a.J, t = j * units + i;
        uint32_t nxt = T, tk = 0u;
        Where there = here;
        // what follows, asked for now and needed when its first copies start.  (Eight counters, each for every eighth block: SMs differ
        // by a quarter in the bandwidth they get, so that units cannot be shared out beforehand, and one counter for all gives 0.3
        // tickets a nanosecond: 240 us for 65536 units.)
        if (lane == 0) tk = atomicAdd(&a.st->ticket[tg][0], 1u);
        const float est = s.est[j], thr = est > 0.0f ? est : __int_as_float(0x7f800000);
        float* lv = reinterpret_cast<float*>(a.scratch + (uint64_t)t * kUnitSlotBytes);
        uint16_t* lk = reinterpret_cast<uint16_t*>(lv + kSlotEntries);
        bool listing = true;
        uint32_t n_list = 0u, piece = 0u, room = kSlotEntries;
        float mx = 0.0f;
        double mynode = 0.0;
#pragma unroll 1
        for (uint32_t slab = 0; slab < 4u; ++slab) {
            if (!__all_sync(kFullMask, mbar_wait(&s.mbar[warp][slot], (parity >> slot) & 1u, a.try_limit))) { failed = true; break; }
            parity ^= 1u << slot;
            float* ring = s.ring[warp][slot];
            const bool whole = here.left >= (slab + 1u) * kSlab;
            if (!whole) {                                      // the gradient's last entries
                for (uint32_t q = lane; q < kSlab; q += 32u) ring[q] = slab * kSlab + q < here.left ? here.g[slab * kSlab + q] : 0.0f;
                __syncwarp();
            }
            float4 v[8];
            slab_read(ring, v, lane);
            float f[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) f[r] = fmaxf(fmaxf(fabsf(v[r].x), fabsf(v[r].y)), fmaxf(fabsf(v[r].z), fabsf(v[r].w)));
            const float fm = fmaxf(fmaxf(fmaxf(f[0], f[1]), fmaxf(f[2], f[3])), fmaxf(fmaxf(f[4], f[5]), fmaxf(f[6], f[7])));
            mx = fmaxf(mx, fm);
            if (__any_sync(kFullMask, fm >= thr) && listing) { // (uniform)
                uint32_t m = slab_mask(v, thr, lane);
                const uint32_t own = (uint32_t)__popc(m), incl = warp_incl_scan(own, lane), cnt = __shfl_sync(kFullMask, incl, 31);
                if (n_list + cnt > room || (slab == 0u && 4u * cnt > kSlotEntries)) {
                    // a piece of the pool instead of the slot: what the unit so far promises, and a quarter more
                    const uint32_t promise = (n_list + cnt) * 4u / (slab + 1u);
                    listing = room == kSlotEntries && promise <= kListMost;
                    if (listing) {
                        room = min(kUnit, (promise * 5u / 4u + 63u) & ~31u);
                        piece = kNoPlace;
                        // (32 pools in turn take 20 us: not again for as long a list)
                        if (lane == 0 && room * 6u < *const_cast<volatile uint32_t*>(&s.refused)) {
                            const uint32_t limit = lists_limit(a, promise);
                            uint64_t fill = 0ull;
                            piece = pool_take(a, room * 6u, limit, *const_cast<volatile uint32_t*>(&s.nearly) != 0u, fill);
                            if (fill > limit - limit / 8u) s.nearly = 1u;
                            if (piece == kNoPlace) atomicMin(&s.refused, room * 6u);
                        }
                        piece = __shfl_sync(kFullMask, piece, 0);
                        listing = piece != kNoPlace;
                        if (listing) {
                            float* pv = reinterpret_cast<float*>(a.scratch + 16ull * piece);
                            uint16_t* pk = reinterpret_cast<uint16_t*>(pv + room);
                            for (uint32_t q = lane; q < n_list; q += 32u) { pv[q] = lv[q]; pk[q] = lk[q]; }
                            lv = pv; lk = pk;
                        }
                    }
                }
                if (listing) {
                    const uint32_t key0 = (i & 3u) * kUnit + slab * kSlab + 32u * (uint32_t)lane;
                    uint32_t pos = n_list + incl - own;
                    for (; m != 0u; m &= m - 1u, ++pos) {
                        const uint32_t b = (uint32_t)__ffs((int)m) - 1u;
                        lv[pos] = ring[32u * (uint32_t)lane + b];
                        lk[pos] = (uint16_t)(key0 + b);
                    }
                    n_list += cnt;
                }
            }
            __syncwarp();                                      // the slab has been read: its place takes the slab two further on
            if (slab + (uint32_t)kRing == 4u) {
                nxt = min(__shfl_sync(kFullMask, tk, 0), T) * groups + tg + gridDim.x * (uint32_t)kScanWarps;
                there = where(min(nxt, T - 1u));
            }
            if (lane == 0) {
                // (generic writes to the place only where the gradient ends: ordered before the copy that follows)
                if (!whole) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (slab + (uint32_t)kRing < 4u) issue(here, slab + (uint32_t)kRing, slot);
                else if (nxt < T) issue(there, slab + (uint32_t)kRing - 4u, slot);
            }
            slot = slot + 1u == (uint32_t)kRing ? 0u : slot + 1u;
            const double u = slab_node(v);
            if (lane == (int)slab) mynode = u;
        }
        if (failed) break;
        const double node = warp_tree(mynode, 4);
        const uint32_t um = __reduce_max_sync(kFullMask, __float_as_uint(mx));      // (non-negative floats order like their bits; a NaN shows in the sum)
        if (lane == 0) {
            a.partials[t] = node;
            a.umax[t] = __uint_as_float(um);
            *reinterpret_cast<uint4*>(a.info + t) = make_uint4(n_list, piece, room, __float_as_uint(listing ? thr : __int_as_float(0x7f800000)));
        }
        here = there;
        cur = nxt;
    }
    if (failed && lane == 0) {                                 // (a copy never came: give up; the others' copies are waited for, bounded)
        atomicExch(&a.ctl->error, (unsigned)kStTimeout);
        for (int i = 0; i < kRing; ++i) mbar_wait(&s.mbar[warp][i], (parity >> i) & 1u, a.try_limit);
    }
    __syncthreads();
    if (tid == 0) atomicAdd(&a.ctl->bar_count[0], 1u);         // (k_encode checks that all blocks were there)
}

// ---- k_encode ----------------------------------------------------------------------------------
struct WorkArea {                                              // shared memory of one team: [16 warps], [4 quads] or [the block]
    static constexpr uint32_t kWarpWords = (kWarpListMax * 27u + 31u) / 32u + 4u, kQuadWords = (4u * kUnitListMax * 27u + 31u) / 32u + 4u,
                              kBlockWords = (kTile * 27u + 31u) / 32u + 4u;
    struct Warp { alignas(16) uint16_t key[kWarpListMax]; uint32_t blob[kWarpWords]; };
    struct Quad { union { struct { alignas(16) uint16_t key[4][kUnitListMax]; uint8_t code[4][kUnitListMax]; uint32_t blob[kQuadWords]; }; Warp w[4]; }; };
    struct Block { alignas(16) uint16_t key[kTile]; uint32_t blob[kBlockWords]; };
    union { Quad q[kEncWarps / 4]; Block b; };
};

struct EncShared {
    float    thr[kEncMaxJobs][132];
    double   S[kEncMaxJobs];
    uint32_t n_light, n_mid, n_heavy, next_light, next_mid, abort_flag, grab[4];
    TeamScratch team[4];
    uint16_t light[kEncThreads], mid[kEncThreads], heavy[kEncThreads];      // heavy: bit 15: the tile is read again
    WorkArea area;
};
static_assert(2 * (sizeof(EncShared) + 1024) <= 233472, "two blocks per SM (1 KiB per block is the system's)");

// The gradients' sums from the units' nodes (same tree).  The first blocks form the nodes of 512 units, a warp each, and publish them;
// every block takes them all and forms the rest of the tree for itself.  Nobody depends on another block: one that is not given a
// node within kNodePolls looks (0.7 us each; they come within 3 us when the GPU runs the first blocks at all) forms it from the units'
// nodes, which the launch before this one has left.
constexpr uint32_t kNodePolls = 256;
// node c of the launch, by one warp
__device__ __forceinline__ double form_node(const double* partials, uint32_t units, uint32_t chunks, uint32_t c, int lane) {
    const uint32_t j = c / chunks, p = c - j * chunks;
    double x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const uint32_t e = kChunkUnits * p + 32u * (uint32_t)i + (uint32_t)lane;
        x[i] = e < units ? __ldcg(partials + (uint64_t)j * units + e) : 0.0;
    }
    return warp_rows16_tree(x, lane);
}
// the nodes below 0, by the block (hardly ever called: kept out of the kernels' code and registers)
__device__ __noinline__ void form_missing_nodes(const double* partials, uint32_t units, uint32_t chunks, double* nodes, uint32_t C) {
    const int lane = threadIdx.x & 31;
    for (uint32_t c = threadIdx.x >> 5; c < C; c += kEncWarps) {
        if (nodes[c] != -1.0) continue;
        const double node = form_node(partials, units, chunks, c, lane);
        __syncwarp();
        if (lane == 0) nodes[c] = node;
    }
}
template <typename Shared>
__device__ __forceinline__ void gradient_sums(const EncArgs& a, Shared& s, double* nodes, int tid, int lane, int warp) {
    const uint32_t units = 4u * a.G, C = a.J * a.chunks, R = min(gridDim.x, 32u), polls = min(kNodePolls, a.wait_limit);
    if (blockIdx.x < R) {
        for (uint32_t c = blockIdx.x + R * (uint32_t)warp; c < C; c += R * (uint32_t)kEncWarps) {
            const double node = form_node(a.partials, units, a.chunks, c, lane);
            if (lane == 0) st_relaxed_pair(a.chunk + 2u * c, (unsigned long long)__double_as_longlong(node), 1ull);
        }
    }
    bool missing = false;
    for (uint32_t c = (uint32_t)tid; c < C; c += kEncThreads) {
        unsigned long long lo, hi;
        uint32_t spin = 0;
        for (;;) {
            ld_relaxed_pair(a.chunk + 2u * c, lo, hi);
            if (hi != 0ull) break;
            if (++spin > polls) { missing = true; break; }
            if (spin > 16u) __nanosleep(32);
        }
        nodes[c] = hi != 0ull ? __longlong_as_double((long long)lo) : -1.0;      // (no sum of |v| is negative)
    }
    if (__syncthreads_or(missing ? 1 : 0)) {
        form_missing_nodes(a.partials, units, a.chunks, nodes, C);
        __syncthreads();
    }
    if ((uint32_t)warp < a.J) {
        const double* p = nodes + (uint32_t)warp * a.chunks;
        double S = 0.0;
        for (uint32_t h = 0; h < (a.chunks > 512u ? 2u : 1u); ++h) {      // (at most 1024 nodes for n < 2^31)
            double x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) { const uint32_t e = 512u * h + 32u * (uint32_t)i + (uint32_t)lane; x[i] = e < a.chunks ? p[e] : 0.0; }
            const double y = warp_rows16_tree(x, lane);
            S = h ? __dadd_rn(S, y) : y;
        }
        if (lane == 0) { s.S[warp] = S; if (blockIdx.x == 0) a.st->S[warp] = S; }
    }
    __syncthreads();
}

// Sums and boundary tables (s.thr) of all gradients; false (in every thread) when a wait has run out.
template <typename Shared>
__device__ __forceinline__ bool gradient_bounds(const EncArgs& a, Shared& s, double* nodes, int tid, int lane, int warp) {
    if (tid == kEncThreads - 1) {                              // all blocks of k_scan have finished (they have: the launch before this one)
        uint32_t spin = 0;
        while (ld_acquire_u32(&a.ctl->bar_count[0]) != a.scan_blocks) if (++spin > a.wait_limit) { s.abort_flag = 1u; break; }
        if (ld_acquire_u32(&a.ctl->error) != 0u) s.abort_flag = 1u;
    }
    gradient_sums(a, s, nodes, tid, lane, warp);
    if (s.abort_flag) {                                        // (every stream of the launch reports it)
        if (tid == 0) atomicExch(&a.ctl->error, (unsigned)kStTimeout);
        return false;
    }
    for (uint32_t i = (uint32_t)tid; i < a.J * 132u; i += kEncThreads) {
        const uint32_t j = i / 132u, k = i - j * 132u;
        if (k <= a.tau) s.thr[j][k] = boundary(s.S[j], __ldcg(a.st->pw + k), __ldcg(a.st->inv + k));
        if (k == 131u) table_hints(s.S[j], a.base, &s.thr[j][130]);
    }
    __syncthreads();
    return true;
}

__global__ void __launch_bounds__(kEncThreads, 2)
k_encode(const EncArgs a) {
    extern __shared__ __align__(128) unsigned char enc_smem_raw[];
    EncShared& s = *reinterpret_cast<EncShared*>(enc_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t T = a.J * a.G, B = gridDim.x;
    if (tid == 0) s.abort_flag = 0u;
    allow_next_kernel();
    wait_for_previous_kernels();
    __syncthreads();
    // ---- the first batch's tiles, requested before the sums are known
    const uint32_t owned = blockIdx.x < T ? (T - blockIdx.x + B - 1u) / B : 0u;
    float4 um; UnitInfo in[4];
    auto load_tile = [&](uint32_t i) {
        if (i < owned) {
            const uint32_t t = blockIdx.x + i * B;
            um = __ldcg(reinterpret_cast<const float4*>(a.umax) + t);
#pragma unroll
            for (int q = 0; q < 4; ++q) in[q] = load_info(a.info + 4ull * t + q);
        }
    };
    load_tile((uint32_t)tid);
    static_assert(sizeof(s.area) >= kMaxChunks * sizeof(double), "the nodes fit the work area");
    if (!gradient_bounds(a, s, reinterpret_cast<double*>(&s.area), tid, lane, warp)) return;

    // (few tiles per block: a list is better shared out among more warps)
    const uint32_t warp_max = owned >= (uint32_t)kEncWarps ? kWarpListMax : 64u;
    for (uint32_t first = 0; first < owned; first += kEncThreads) {
        // ---- which of the block's tiles hold anything, and where it is
        if (tid == 0) { s.n_light = 0u; s.n_mid = 0u; s.n_heavy = 0u; s.next_light = 0u; s.next_mid = 0u; }
        if (first) load_tile(first + (uint32_t)tid);
        __syncthreads();
        if (first + (uint32_t)tid < owned) {
            const uint32_t t = blockIdx.x + (first + (uint32_t)tid) * B, j = t / a.G;
            const float thr_e = s.thr[j][a.tau];
            uint32_t cnt = 0u;
            bool again = false, any = false, slots = true, units = true;      // (a unit that does not reach the threshold counts for nothing)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float x = q == 0 ? um.x : q == 1 ? um.y : q == 2 ? um.z : um.w;
                if (x >= thr_e) { any = true; cnt += in[q].count; again = again || !(in[q].sthr <= thr_e); slots = slots && in[q].room == kSlotEntries; units = units && in[q].count <= kUnitListMax; }
            }
            if (!(thr_e < __int_as_float(0x7f800000)) || !any) a.desc[t] = 0ull;      // nothing is kept here
            else if (again) {
                s.heavy[atomicAdd(&s.n_heavy, 1u)] = (uint16_t)(tid | 0x8000);
                atomicAdd(&a.ctl->ne_count[j], 1u);
            } else if (slots && cnt <= warp_max) s.light[atomicAdd(&s.n_light, 1u)] = (uint16_t)tid;
            else if (units) s.mid[atomicAdd(&s.n_mid, 1u)] = (uint16_t)tid;
            else s.heavy[atomicAdd(&s.n_heavy, 1u)] = (uint16_t)tid;
        }
        __syncthreads();
        // (the first lane of a team records the tile's sizes)
        auto record = [&](uint32_t t, uint32_t j, uint32_t count, uint32_t M, uint32_t words, uint32_t place) {
            a.desc[t] = count ? tile_desc(count, M, words) : 0ull;
            a.blob[t] = place;
            if (count) atomicAdd(&a.seg[j * a.segments + ((t - j * a.G) >> a.seg_log2)], ((unsigned long long)count << 32) | words);
        };
        // Where the tile's lists were, which by now are in shared memory: the slots of its units or the largest of their pieces of the
        // pool (a quarter of the candidates at 6 bytes holds all entries at up to 12 bits); else a new piece.  (One gradient of 2^30, a
        // tenth kept: lists and blobs together did not fit the pool, and most tiles were packed twice: 5.9 ms, now 1.8.)
        auto piece_of = [&](const UnitInfo& in, TeamScratch& ts, uint32_t q) {
            ts.room[q] = in.room != kSlotEntries && in.piece != kNoPlace ? in.room : 0u;
            ts.piece[q] = in.piece;
        };
        auto place_of = [&](const TeamScratch& ts, uint32_t t, uint32_t words) -> uint32_t {
            if (words <= kSlotWords) return t * (kSlotBytes / 16u);
            uint32_t room = 0u, p = kNoPlace;
#pragma unroll
            for (int q = 0; q < 4; ++q) if (ts.room[q] > room) { room = ts.room[q]; p = ts.piece[q]; }
            if (4u * words > 6u * room) p = pool_take(a, words * 4u);
            if (p == kNoPlace) atomicAdd(&a.st->noblob, 1u);
            return p;
        };
        // ---- by the whole block
        for (uint32_t h = 0; h < s.n_heavy; ++h) {
            const uint32_t x = s.heavy[h];
            const uint32_t t = blockIdx.x + (first + (x & 0x7FFFu)) * B, j = t / a.G, tile = t - j * a.G;
            uint32_t M = 0u, words = 0u, place = 0u;
            if (tid < 4) piece_of(load_info(a.info + 4ull * t + tid), s.team[0], (uint32_t)tid);
            const uint32_t count = (x & 0x8000u) != 0u ? block_tile(a, j, tile, s.thr[j], s.area.b.key, s.area.b.blob, s.team[0], tid, lane, warp)
                                                               : team_list<kEncWarps>(a, t, s.thr[j], s.area.b.key, s.area.b.blob, s.team[0], warp, lane, 0);
            if (count) {
                M = team_pack<kEncWarps>(a.l, s.area.b.key, s.area.b.blob, count, s.team[0], warp, lane, 0, [&](uint32_t w_) {
                    words = w_;
                    if (tid == 0) s.team[0].word = place_of(s.team[0], t, w_);
                });
                place = s.team[0].word;
                if (place != kNoPlace) {
                    uint32_t* dst = reinterpret_cast<uint32_t*>(a.scratch + 16ull * place);
                    for (uint32_t i = (uint32_t)tid; i < words; i += kEncThreads) dst[i] = bswap32(s.area.b.blob[i]);
                }
            }
            if (tid == 0) record(t, j, count, M, words, place);
            __syncthreads();
        }
        // ---- by four warps
        const int quad = warp >> 2, qw = warp & 3;
        if (qw == 0 && lane == 0) s.grab[quad] = atomicAdd(&s.next_mid, 1u);
        team_sync<4>(quad);
        // (a warp per unit; three barriers a tile; the next tile's entries of the tables are asked for while this one is packed)
        uint32_t x = s.grab[quad], t = 0u;
        UnitInfo ui;
        float ux = 0.0f;
        auto next_unit = [&]() {
            if (x >= s.n_mid) return;
            t = blockIdx.x + (first + s.mid[x]) * B;
            ui = load_info(a.info + 4ull * t + qw);
            ux = __ldcg(a.umax + 4ull * t + qw);
        };
        next_unit();
        while (x < s.n_mid) {
            const uint32_t here = t, j = t / a.G;
            WorkArea::Quad& ar = s.area.q[quad];
            TeamScratch& ts = s.team[quad];
            const uint16_t* keys = ar.key[qw];
            const uint32_t n = ux >= s.thr[j][a.tau] ? unit_list(list_of(a, 4u * t + (uint32_t)qw, ui), ui.count, s.thr[j], a.tau, ar.key[qw], ar.code[qw], lane) : 0u;
            __syncwarp();
            const uint32_t quads = (n + 127u) >> 7, q0 = 4u * quads * (uint32_t)lane;
            KeyRun r;
            r.keys = keys + q0; r.left = q0 < n ? (int)min(4u * quads, n - q0) : 0; r.prev = q0 < n ? (uint32_t)keys[q0 ? q0 - 1u : 0u] : 0u;
            const uint32_t top = runs_max(r, quads);           // (within the unit)
            if (lane == 0) { piece_of(ui, ts, (uint32_t)qw); ts.cnt[qw] = n; ts.maxd[qw] = top; ts.first[qw] = n ? (uint32_t)keys[0] : 0u; ts.last[qw] = n ? (uint32_t)keys[n - 1u] : 0u; }
            team_sync<4>(quad);
            // from one unit's last key to the next one's first; the unit's rank
            uint32_t M = 0u, count = 0u, rank = 0u, last = 0u, before = 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t c = ts.cnt[q];
                if (q == qw) { rank = count; before = last; }
                if (c) { M = max(M, max(ts.maxd[q], ts.first[q] - last)); last = ts.last[q]; }
                count += c;
            }
            if (count == 0u) {                                 // (the same in the four warps)
                if (qw == 0 && lane == 0) { record(here, j, 0u, 0u, 0u, 0u); s.grab[quad] = atomicAdd(&s.next_mid, 1u); }
                team_sync<4>(quad);
                x = s.grab[quad];
                next_unit();
                continue;
            }
            M = max(1u, bit_length(M));
            if (lane == 0) r.prev = before;
            const uint32_t shape = delta_shape(a.l, M, lane);
            const int least = rank + q0 == 0u ? 0 : -1;
            const uint32_t bits = run_bits(r, quads, shape, least), incl = warp_incl_scan(bits, lane);
            if (lane == 31) ts.bits[qw] = incl;
            if (qw == 0 && lane == 0) s.grab[quad] = atomicAdd(&s.next_mid, 1u);
            const uint32_t bound = (count * (8u + a.l + M) + 31u) >> 5, delta0 = (8u + a.l) * count;
            for (uint32_t i = (uint32_t)(qw * 32 + lane); i <= bound; i += 128u) ar.blob[i] = 0u;
            team_sync<4>(quad);
            x = s.grab[quad];
            next_unit();
            uint32_t dpos = delta0 + incl - bits, words = delta0;
#pragma unroll
            for (int q = 0; q < 4; ++q) { const uint32_t y = ts.bits[q]; if (q < qw) dpos += y; words += y; }
            words = (words + 31u) >> 5;
            if (qw == 0 && lane == 0) ts.word = place_of(ts, here, words);
            write_runs<true>(r, quads, shape, least, a.l, ar.blob, count, rank + q0, dpos, ar.code[qw] + q0);
            team_sync<4>(quad);
            const uint32_t place = ts.word;
            if (place != kNoPlace) {
                uint32_t* dst = reinterpret_cast<uint32_t*>(a.scratch + 16ull * place);
                for (uint32_t i = (uint32_t)(qw * 32 + lane); i < words; i += 128u) dst[i] = bswap32(ar.blob[i]);
            }
            if (qw == 0 && lane == 0) record(here, j, count, M, words, place);
        }
        team_sync<4>(quad);
        // ---- by single warps
        for (;;) {
            uint32_t x = 0u;
            if (lane == 0) x = atomicAdd(&s.next_light, 1u);
            x = __shfl_sync(kFullMask, x, 0);
            if (x >= s.n_light) break;
            const uint32_t t = blockIdx.x + (first + s.light[x]) * B, j = t / a.G;
            const float thr_e = s.thr[j][a.tau];
            uint32_t off[5];
            {
                uint32_t c = 0u;
                if (lane < 4) c = __ldcg(a.umax + 4ull * t + lane) >= thr_e ? __ldcg(&a.info[4ull * t + lane].count) : 0u;
                const uint32_t ci = warp_incl_scan(c, lane);
                off[0] = 0u;
#pragma unroll
                for (int q = 0; q < 4; ++q) off[q + 1] = __shfl_sync(kFullMask, ci, q);
            }
            WorkArea::Warp& ar = s.area.q[quad].w[qw];
            uint32_t M = 0u, words = 0u;
            const uint32_t place = t * (kSlotBytes / 16u);      // (27 bits an entry at most: the blob fits the slots)
            const uint32_t count = warp_list(a, t, off, s.thr[j], ar.key, ar.blob, lane);
            if (count) {
                M = team_pack<1>(a.l, ar.key, ar.blob, count, s.team[quad], 0, lane, 0, [&](uint32_t w_) { words = w_; });
                uint32_t* dst = reinterpret_cast<uint32_t*>(a.scratch + 16ull * place);
                for (uint32_t i = lane; i < words; i += 32u) dst[i] = bswap32(ar.blob[i]);
            }
            if (lane == 0) record(t, j, count, M, words, place);
            __syncwarp();
        }
        __syncthreads();
    }
}

}  // namespace fsg
