// Decoder (decoder phases 1-4) and aggregation, for one stream or for several workers' streams
// of the same gradient in one launch.
//
// Phase 1: the length flags give every delta's width; an exclusive scan of the widths gives
// its bit offset.  Phase 2: an inclusive scan of the deltas, started at g*T, gives the keys
// back.  Phases 3-4: code L -> sum / b^L (the boundary B_L rounded to fp32), signed.  The
// aggregation adds the value into dense_out[key].  Keys are unique within a stream, and the values
// that several streams hold for one key are added in the streams' order by one thread (or behind
// block barriers), so the read-modify-write needs no atomics and the result equals that of one call
// per stream.
//
// Work split.  A block owns groups blockIdx.x, blockIdx.x + gridDim.x, ... and reads their
// directory entries first, one entry per thread.  One stream: groups of up to kDecWarpMax keys (kDecWarpFew
// where a block has few groups) are decoded by one warp each, larger ones by the whole block.  Several streams: groups go to
// teams of one, two or four warps or to the block (team_rule).  Either way the streams are parsed side
// by side (the team's lanes or the block's threads are shared out among them, a thread owns a run of
// consecutive keys), into lists of keys in shared memory; a stream's group is validated in full
// before any of it is applied; then the lists are applied with neighbouring threads on neighbouring keys
// and all of a batch's memory accesses in flight together.
//
// What bounds it.  With few groups per block, the latency of the chain launch - directory - blob - parse - entries of
// dense_out (about 3 + 5 us); with many scattered keys, DRAM transactions: a bare kernel that only reads and writes 2.7 M
// floats at ascending random places of a 1 GiB array takes 100 us, the decoder 121.  So what counts is warps in
// flight and few instructions per key: 512 threads per block and two blocks per SM at 64 registers are 32 warps (256 threads
// with longer register-resident runs, 16 warps, took 149 us there); parsing side by side with independent fetches instead of a
// bit reader per thread halved the parse; the table of distinct keys or their ranks (teams) and the slice (blocks) give each coordinate one
// round trip to memory however many streams hold it (one per stream before).  Measured before and after: four
// streams of 128 K keys over 25.6 M entries 28.8 -> 25.0 us, eight streams of 33 K keys over 33.5 M 26.7 -> 16.8, one stream of
// 1.3 M over 67 M 97.8 -> 59.5; model update of the first 68.6 -> 50.5, of eight streams of 671 K keys over 67 M on the
// packed state 510 -> 216.
#pragma once

#include <cstddef>

#include "common.cuh"
#include "bits.cuh"
#include "prims.cuh"

namespace fsg {

constexpr int      kDecThreads     = 512;
constexpr int      kDecWarps       = kDecThreads / 32;
constexpr int      kDecMaxStreams  = 8;       // streams per launch
constexpr uint32_t kDecWarpMax     = 1024;    // groups with more keys go to the whole block (one stream, many groups per block)
constexpr uint32_t kDecWarpFew     = 256;     // the same when a block has only a few groups: its other warps would stand idle
constexpr uint32_t kTeamBytes      = 6144;    // launch with several streams: shared memory of a team, for each of its warps
constexpr uint32_t kTeamSlotsLog2  = 10, kTeamSlots = 1u << kTeamSlotsLog2;      // ... of which slots (16 bits each) of the table of distinct keys
constexpr uint32_t kDecWarpWords   = kDecWarpMax * (8u + 5u + 16u) / 32u + 4u;    // words of one stream's blob on the warp path (16: largest group_log2 it takes)
constexpr uint32_t kBlockStageWords = 4096;   // blobs larger than this in total are parsed from global memory
constexpr uint32_t kBlockListMax   = 8192;    // keys of a group (all streams together) the block path lists in shared memory
constexpr uint32_t kWideListMax    = 1u << 14;      // ... of a group wider than the tile, in the tile's place
// From this many keys on the group's whole slice of dense_out goes through shared memory: scattered over 2048 sectors of 32 bytes
// they touch a third of it, and a bulk copy moves whole pages (7.5 % of 2^26 entries, one stream: 96 us with, 111 without the slice).
constexpr uint32_t kTileMinKeys    = 768;
// ... where no bulk copy moves it, but words (dense_out not 16-byte aligned, or the ragged last group; 2^25 entries, one stream, 800, 1100, 1450 keys a
// group: entry by entry 57, 59, 65 us, over the slice 89, 88, 89)
constexpr uint32_t kTileMinWords   = 1536;
// Several streams whose groups have about as many keys: from this many a group on ranks by bits (four warps) instead of the table of keys, up to as
// many as the slice is for (team_rule).  Eight streams over 2^25 entries, us by table and by ranks (slice), at keys a group:
//   aggregation  180: 22, 27; 290: 27, 31; 420: 38, 37; 650: 59, 56; 850: 75, 68 (78); 980: 77 by ranks (78); 1310: 94 by ranks (78)
//   update       180: 64, 63; 290: 97, 84; 420: 131, 102; 650: 183, 126; 1310: 182 over the slice of g, 164; 1770: 186, 174
//   (two streams over as many entries: aggregation 450: 45, 43; 930: 70, 59; update 450: 124, 99; 700: 164, 127; packed 450: 61, 54; 930: 114, 90)
//   packed       180: 25, 28; 290: 34, 35; 420: 51, 50; 650: 85, 76; 850: 112, 90; 1770: 196 over the slice, 139
__host__ __device__ constexpr uint32_t ranked_mean(int mode) { return mode == 2 ? 256u : 400u; }
constexpr uint32_t kSliceMean      = 1000;
constexpr uint32_t kFewGroups      = 4;       // groups of a block that teams of four take side by side
// From this many keys on the model update by a block goes over the slice of g, four neighbouring coordinates at a time, instead of key by key
// (eight streams, 5 % of 2^24 entries: 292 -> 125 us); on the packed state, where a key is one access anyway, later (235 -> 132 us).
constexpr uint32_t kSweepMinKeys   = 768;
constexpr uint32_t kSweepMinPacked = 2048;
constexpr uint64_t kL2Entries      = 1u << 25;      // entries of dense_out that fill the L2
constexpr uint32_t kDecSpinLimit   = 1u << 20;

struct DecArgs {
    const uint8_t*      stream[kDecMaxStreams];
    uint64_t            bytes[kDecMaxStreams];
    uint64_t            n;
    float*              dense;
    unsigned long long* status;     // sticky minimum of (group << 32 | key index << 8 | status)
    unsigned int*       q_ctl;      // {-, taken, done, exited, reserved}: queue of groups for whole blocks, shared by the grid
    unsigned int*       q_list;     // its slots (group + 1; 0: empty)
    double              base;
    uint32_t            W;          // streams in this launch
    uint32_t            G;
    uint32_t            tau;
    uint32_t            l;
    uint32_t            group_log2;
    uint32_t            spin_limit; // polls before a wait on the queue of large groups gives up (kDecSpinLimit unless a test shortens it)
    uint32_t            try_limit;  // tries before a wait on a bulk copy gives up
    // model update on the decoded coordinates (modes 1 to 3)
    float*              theta;
    float*              m;
    float*              v;
    float               lr, beta1, beta2, eps;
};

// Modes of the decoder (template parameter MODE): 0 aggregation into dense_out; 1 model update as a pass of its own
// (dense_out holds the aggregated gradient, left there by mode-0 launches over the same streams); 2 both in one launch
// (dense_out: all zero, and left so); 3 both in one launch on the packed state (theta, m, v, g per coordinate).
__host__ __device__ constexpr bool mode_fused(int mode) { return mode == 2 || mode == 3; }

// Scattered entries: loads that bring 64 bytes of a line from memory, not all 128.
__device__ __forceinline__ float load_entry(const float* p) {
    float x;
    asm volatile("ld.global.L2::64B.f32 %0, [%1];" : "=f"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ float4 load_entry(const float4* p) {
    float4 x;
    asm volatile("ld.global.L2::64B.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "l"(p) : "memory");
    return x;
}

// One Adam step (the experimental set-up's equations, no bias correction; one IEEE fp32 operation at a time) on up to K
// coordinates kk[i] with aggregated gradient g[i]; nothing happens where g[i] == 0 (kk[i] is then not looked at).  All loads
// are issued before the first of them is needed.  PACKED: one 16-byte entry (theta, m, v, g) per coordinate.  ASCENDING: neighbouring threads
// have neighbouring coordinates (what shares a line is asked for together).
template <bool PACKED, int K, bool ASCENDING = false>
__device__ __forceinline__ void adam_run(const DecArgs& a, const uint32_t (&kk)[K], const float (&g)[K]) {
    if constexpr (PACKED) {
        float4* state = reinterpret_cast<float4*>(a.dense);
        float4 st[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            st[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (g[k] != 0.0f) st[k] = ASCENDING ? load_entry(state + kk[k]) : state[kk[k]];
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (g[k] != 0.0f) {
                const float mk = __fadd_rn(__fmul_rn(a.beta1, st[k].y), __fmul_rn(__fsub_rn(1.0f, a.beta1), g[k]));
                const float vk = __fadd_rn(__fmul_rn(a.beta2, st[k].z), __fmul_rn(__fsub_rn(1.0f, a.beta2), __fmul_rn(g[k], g[k])));
                const float step = __fdiv_rn(a.lr, __fsqrt_rn(__fadd_rn(vk, a.eps)));
                state[kk[k]] = make_float4(__fsub_rn(st[k].x, __fmul_rn(step, mk)), mk, vk, 0.0f);
            }
        }
    } else {
        float pm[K], pv[K], pt[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool on = g[k] != 0.0f;
            pm[k] = !on ? 0.0f : ASCENDING ? load_entry(a.m + kk[k]) : a.m[kk[k]];
            pv[k] = !on ? 0.0f : ASCENDING ? load_entry(a.v + kk[k]) : a.v[kk[k]];
            pt[k] = !on ? 0.0f : ASCENDING ? load_entry(a.theta + kk[k]) : a.theta[kk[k]];
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (g[k] != 0.0f) {
                const float mk = __fadd_rn(__fmul_rn(a.beta1, pm[k]), __fmul_rn(__fsub_rn(1.0f, a.beta1), g[k]));
                const float vk = __fadd_rn(__fmul_rn(a.beta2, pv[k]), __fmul_rn(__fsub_rn(1.0f, a.beta2), __fmul_rn(g[k], g[k])));
                const float step = __fdiv_rn(a.lr, __fsqrt_rn(__fadd_rn(vk, a.eps)));
                a.m[kk[k]] = mk;
                a.v[kk[k]] = vk;
                a.theta[kk[k]] = __fsub_rn(pt[k], __fmul_rn(step, mk));
            }
        }
    }
}

__device__ __forceinline__ void adam_step(const DecArgs& a, float g, float& theta, float& m, float& v) {
    if (g == 0.0f) return;
    m = __fadd_rn(__fmul_rn(a.beta1, m), __fmul_rn(__fsub_rn(1.0f, a.beta1), g));
    v = __fadd_rn(__fmul_rn(a.beta2, v), __fmul_rn(__fsub_rn(1.0f, a.beta2), __fmul_rn(g, g)));
    theta = __fsub_rn(theta, __fmul_rn(__fdiv_rn(a.lr, __fsqrt_rn(__fadd_rn(v, a.eps))), m));
}

// The model update of a group with many keys from its slice of g in shared memory: four neighbouring coordinates per thread,
// 16-byte accesses wherever one of the four has a gradient (a warp's access then covers a run of lines, where key by key every
// lane's is a line of its own).  theta, m and v are 16-byte aligned.
__device__ __forceinline__ void adam_sweep(const DecArgs& a, const float* tile, uint32_t lo, uint32_t span, int tid, int threads) {
#pragma unroll 1
    for (uint32_t q = (uint32_t)tid * 4u; q < span; q += 4u * (uint32_t)threads) {
        const float4 g = *reinterpret_cast<const float4*>(tile + q);
        if (g.x == 0.0f && g.y == 0.0f && g.z == 0.0f && g.w == 0.0f) continue;
        if (q + 4u <= span) {
            float4 t = *reinterpret_cast<const float4*>(a.theta + lo + q), m = *reinterpret_cast<const float4*>(a.m + lo + q),
                   v = *reinterpret_cast<const float4*>(a.v + lo + q);
            adam_step(a, g.x, t.x, m.x, v.x);
            adam_step(a, g.y, t.y, m.y, v.y);
            adam_step(a, g.z, t.z, m.z, v.z);
            adam_step(a, g.w, t.w, m.w, v.w);
            *reinterpret_cast<float4*>(a.theta + lo + q) = t;
            *reinterpret_cast<float4*>(a.m + lo + q) = m;
            *reinterpret_cast<float4*>(a.v + lo + q) = v;
        } else {                                                        // the gradient's last few entries
            for (uint32_t k = q; k < span; ++k) adam_step(a, tile[k], a.theta[lo + k], a.m[lo + k], a.v[lo + k]);
        }
    }
}

__device__ __forceinline__ void dec_fail(const DecArgs& a, uint32_t g, uint32_t j, int st) {
    atomicMin(a.status, ((unsigned long long)g << 32) | ((unsigned long long)(j & 0xFFFFFFu) << 8) | (unsigned)st);
}

__device__ __forceinline__ int check_header(const DecArgs& a, uint64_t bytes, const uint32_t* w, uint64_t* total_out, double* sum_out) {
    if (w[0] != kMagic) return kStBadMagic;
    if (w[1] != kVersion) return kStBadVersion;
    if (w[2] != (uint32_t)kStOk) return kStBadStatus;
    const uint64_t n = (uint64_t)w[4] | ((uint64_t)w[5] << 32);
    if (n != a.n) return kStNMismatch;
    const unsigned long long bb = (unsigned long long)w[12] | ((unsigned long long)w[13] << 32);
    if (bb != (unsigned long long)__double_as_longlong(a.base) || w[3] != a.tau ||
        (w[14] & 0xFFu) != a.l || ((w[14] >> 8) & 0xFFu) != a.group_log2 || w[15] != a.G)
        return kStParamMismatch;
    const uint64_t total = (uint64_t)w[8] | ((uint64_t)w[9] << 32);
    const uint64_t fixed = (uint64_t)kHeaderBytes + 8ull * a.G;
    if (total > bytes || total < fixed || (total & 3ull)) return kStTruncated;
    *total_out = total;
    *sum_out = __longlong_as_double((long long)((unsigned long long)w[10] | ((unsigned long long)w[11] << 32)));
    return kStOk;
}

// A warp's working memory on the warp path (overlays the block path's).
struct DecWarpOne {
    uint32_t blob[kDecWarpWords];
    uint16_t key[kDecWarpMax];       // group-relative keys
};
constexpr uint32_t kTeamFew        = 249;     // groups of fewer keys go to a warp where groups differ much
constexpr uint32_t kTeamShared     = 200;     // from this many keys on two warps (four) are quicker than one (eight streams of 16 keys: 18 us, by two 21)
// Bytes that a group of several streams takes of its team's memory beside the table: 4 for a coordinate's value and 2 for a key of each
// entry, the blobs, two words behind them that the parse may look at, and one of flags.
__host__ __device__ constexpr uint32_t team_bytes(uint32_t entries, uint32_t words) { return 6u * ((entries + 1u) & ~1u) + 4u * (words + 3u); }

// The same for a team of four warps: a bit and the share of a 16-bit count for each index of the group, 8 for each entry (a sum, a key, a place in
// a list), the blobs, two words behind them that the parse may look at, and five more.
__host__ __device__ constexpr uint32_t ranked_bytes(uint32_t entries, uint32_t words, uint32_t group_log2) {
    return 6u * ((1u << group_log2) / 32u) + 8u * ((entries + 1u) & ~1u) + 4u * (words + 2u + 5u);
}

// Who decodes the groups of several streams (mode as below): those of fewer than `below` keys teams of at least `least` (0, 1, 2: one, two, four
// warps), the others the block.  table: teams of four by the table of keys, not by ranks.  two: there are teams of two (not in the update in one launch: four
// streams of 230 keys a group over 20 M and 33 M entries 55 and 82 us, by ranks 49 and 71).
// Where most of a block's groups have about as many keys (alike), they all go to teams (of the same size: ranked_mean), up to as many keys as the
// slice is for (kSliceMean); with few groups to a block to larger teams, so that its warps have work.  Else (layers of different scales) and in a
// block with one group, those of many keys are for whole blocks, which share them through a queue: teams of several sizes work one after
// the other, and nobody helps a block that has many (four streams of 25.6 M: 33 to 42 us, so 24).
// bulk: dense_out (the update: theta, m and v) is 16-byte aligned, as the slice wants it (else, eight streams over 2^25 entries, 1100, 1450, 1800 keys a group: by teams 83, 98, 111 us, by
// blocks 119, 120, 121).
// The update goes over the slice of g (sweep_all) from a mean on that grows with the streams, whose lists the block adds up one after the other (2^25 entries;
// us by ranks and over the slice at 1200, 1600, 2000 keys a group: two streams 157, 172, 181 and 164, 165, 167; four 155, 166, 176 and 168, 170,
// 174; eight 161, 172, 182 and 182, 184, 188, 2050 keys 212 and 189).
// (Groups wider than the slice have no slice: eight streams over 2^25 entries in groups of 2^15, 1050, 1500, 1750 keys a group: by teams 51, 70, 80 us, by
// blocks 70, 85, 95.)
// Aggregation by the table in teams of four too where a block's few groups stand side by side: what counts then is the shorter chain (550 groups
// of 790 keys, four streams: 19.6 us, by ranks 20.8).
struct TeamRule { uint32_t below, least; bool table, two; };
__host__ __device__ constexpr TeamRule team_rule(int mode, uint32_t group_log2, uint32_t owned, bool alike, uint32_t mean, bool bulk, uint32_t W) {
    const bool few = owned <= kFewGroups;
    TeamRule r{kTeamFew, 0u, mode == 0 && few, mode != 2};
    if (alike) {
        const uint32_t slice = mode == 0 ? kSliceMean : mode == 2 ? (W < 5u ? 1000u + 200u * W : 2000u) : 0xFFFFFFFFu;
        r.below = mean >= slice && group_log2 <= 14u && bulk ? kTeamFew : 0xFFFFFFFFu;      // (as many as the memory of four warps holds)
        r.least = mean >= ranked_mean(mode) ? 2u : mean < kTeamShared ? 0u : few ? 2u : owned <= 8u ? (r.two ? 1u : 2u) : 0u;
    }
    if (group_log2 > 15u) r.below = 0u;
    return r;
}
// ... and a group of so many keys, with blobs of so many words: 0, 1, 2 as above, or 3, the block
__host__ __device__ constexpr uint32_t team_for(const TeamRule& r, uint32_t group_log2, uint32_t keys, uint32_t words) {
    if (keys >= r.below) return 3u;
    const uint32_t bytes = team_bytes(keys, words), room = kTeamBytes - 2u * kTeamSlots;
    const uint32_t fits = bytes <= room ? 0u : bytes <= 2u * room && r.two ? 1u : 2u, team = fits < r.least ? r.least : fits;
    if (team == 2u && (r.table ? bytes > 4u * room : ranked_bytes(keys, words, group_log2) > 4u * kTeamBytes)) return 3u;
    return team;
}
// One stream: the most keys of a group that one warp decodes.
__host__ __device__ constexpr uint32_t warp_max(uint32_t owned) { return owned >= (uint32_t)kDecWarps / 2u ? kDecWarpMax : kDecWarpFew; }
// ... and whether it keeps two entries a lane in flight when it adds them up, not eight.  Where every warp has several groups, entries are further apart than
// a line and dense_out is more than the L2 holds, memory is the bound, and more in flight only make it switch between reading and writing
// more often (a bare kernel that updates 2.7 M floats at ascending random places of 1 GiB, a group a warp: eight a lane 113 us, four 107, two 101, and 8 us
// more with whole lines fetched; 268 M entries, 1 % kept: 131.5, now 121).  Else it is the latency.  us with two and with eight at keys a group: groups of
// 2^14, 140 M entries 400: 120, 121; 600: 153, 150; 900: 185, 183; of 2^12, 20 M entries 900: 52.5, 47.1; of 2^10, 6 M 400: 17.4, 15.8.
__host__ __device__ constexpr bool two_in_flight(uint32_t owned, uint64_t n) { return owned > (uint32_t)kDecWarps && n > kL2Entries; }
__host__ __device__ constexpr bool sparse_group(uint32_t keys, uint32_t span) { return 32u * keys < span; }
// Aggregation by the block: over the group's whole slice of dense_out from this many keys on.  One stream (a warp takes up to 1024 keys where the block
// has 8 groups): what fits the L2 is read there entry by entry, and the slice's 64 KiB both ways are 8 bytes an entry of the vector at 5 TB/s.  us entry by entry
// and over the slice at 800, 1000, 1250 keys a group: 12 M entries 18.6, 19.4, 20.5 and 23.6, 22.2, 23.2; 16.8 M 29.4, 31.9, 33.7 and 31.6, 31.2,
// 31.3; 25 M 44.4, 46.3, 47.4 and 42.5, 42.0, 42.3; 36 M 61, 66, 67 and 60, 62, 57.
__host__ __device__ constexpr uint32_t slice_min(bool bulk, bool one, uint64_t n) {
    return !bulk ? kTileMinWords : !one || n > 20000000u ? kTileMinKeys : n > 15000000u ? 900u : kTileMinWords;
}

struct DecShared {
    float              val[kDecMaxStreams][132];
    uint32_t           hdr[kDecMaxStreams][16];
    double             sum[kDecMaxStreams];
    uint32_t           total_words[kDecMaxStreams];
    uint32_t           ok[kDecMaxStreams];
    // the directory entries of the block's groups, kDecThreads (group, stream) pairs at a time
    uint32_t           e_cm[kDecThreads], e_off[kDecThreads], e_nw[kDecThreads];
    uint32_t           gtot[kDecThreads];           // keys of each of these groups over all streams; several streams: from kDecThreads / 2 on their words
    uint16_t           light[kDecThreads], heavy[kDecThreads];      // groups for a warp, and from the end on for four; for the block, and from the end on for two
    uint32_t           n_light[3], n_heavy, next_light[3], grab[kDecWarps], mean;
    uint32_t           scan[2][kDecWarps];
    uint32_t           got;           // answer of thread 0 to the block
    uint32_t           bad[kDecMaxStreams];
    // the group the block works on, per stream
    uint32_t           g_count[kDecMaxStreams], g_M[kDecMaxStreams], g_off[kDecMaxStreams], g_nwords[kDecMaxStreams],
                       g_base[kDecMaxStreams], g_list[kDecMaxStreams];
    unsigned long long tile_bar;      // mbarrier of the bulk copy that loads the tile
    union alignas(128) {               // (bulk copies need 16-byte aligned shared addresses)
        DecWarpOne     one[kDecWarps];
        uint8_t        team[kDecWarps][kTeamBytes];
        struct {                                 // block path
            float      tile[1u << 14];           // the group's slice of dense_out (or of g)
            uint32_t   bstage[kBlockStageWords + 4];
            alignas(16) uint16_t lkey[kBlockListMax];
        };
    } u;
};
static_assert(2 * (sizeof(DecShared) + 1024) <= 233472, "two blocks per SM (1 KiB per block is the system's)");
static_assert(offsetof(DecShared, u) % 128 == 0, "tile alignment");

// Directory entry of group g in one stream (its two words and the offset that follows, or the stream's end), checked.
// Returns false (and records the status) if it is inconsistent.  count = 0 for an empty group.
__device__ __forceinline__ bool check_dir(const DecArgs& a, uint32_t g, uint32_t total_words, uint32_t e0, uint32_t o, uint32_t next_off,
                                          uint32_t* nwords) {
    const uint32_t fixed_words = (kHeaderBytes + 8u * a.G) >> 2;
    const uint32_t c = e0 & 0xFFFFFFu, m = e0 >> 24;
    *nwords = 0;
    if ((g == 0 && o != fixed_words) || next_off < o || next_off > total_words || o < fixed_words) {
        dec_fail(a, g, 0u, kStBadDirectory);
        return false;
    }
    if (c == 0) {
        if (e0 != 0u || next_off != o) { dec_fail(a, g, 0u, kStBadDirectory); return false; }
        return true;
    }
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    const uint32_t nw = next_off - o;
    // (a blob is never longer than count * (8 + l + M) bits rounded up to words: also bounds the staging copy)
    if (c > span || m < 1u || m > a.group_log2 || (uint64_t)(8u + a.l) * c > 32ull * nw ||
        (uint64_t)nw > ((uint64_t)c * (8u + a.l + m) + 31ull) / 32ull) {
        dec_fail(a, g, 0u, kStBadDirectory);
        return false;
    }
    *nwords = nw;
    return true;
}

// exclusive scan of one value per thread over its team: `tn` consecutive lanes (BLOCK = false: tn <= 32) or tn / 32 consecutive
// warps of the block (BLOCK = true; one barrier, every thread of the block calls it); also the team's total.  `which`
// alternates between the two shared arrays.
template <bool BLOCK>
__device__ __forceinline__ uint32_t team_scan(uint32_t v, uint32_t* total, DecShared& s, uint32_t tn, int lane, int warp, int which) {
    if constexpr (!BLOCK) {
        uint32_t incl = v;
#pragma unroll
        for (uint32_t o = 1; o < 32u; o <<= 1) {
            if (o < tn) {            // (uniform)
                const uint32_t t = __shfl_up_sync(kFullMask, incl, o, tn);
                if (((uint32_t)lane & (tn - 1u)) >= o) incl += t;
            }
        }
        *total = __shfl_sync(kFullMask, incl, tn - 1u, tn);
        return incl - v;
    } else {
        const uint32_t incl = warp_incl_scan(v, lane);
        if (lane == 31) s.scan[which][warp] = incl;
        __syncthreads();
        const uint32_t wt = tn >> 5, w0 = (uint32_t)warp & ~(wt - 1u);
        const uint32_t x = (uint32_t)lane < wt ? s.scan[which][w0 + lane] : 0u;
        uint32_t xi = x;
#pragma unroll
        for (int o = 1; o < kDecWarps; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFullMask, xi, o);
            if (lane >= o) xi += t;
        }
        *total = __shfl_sync(kFullMask, xi, kDecWarps - 1);
        return __shfl_sync(kFullMask, xi - x, (uint32_t)warp - w0) + incl - v;
    }
}

// One group's blob of one stream.  STAGED: in shared memory, its words already most significant byte first, at least two words
// of the stage behind it; else in global memory, as it stands in the stream.
struct Blob {
    const uint32_t* words;
    uint32_t nwords, count, M;
};
// the 32 bits from bit `pos` on (beyond the blob: anything, but no access outside the stage or the stream)
template <bool STAGED>
__device__ __forceinline__ uint32_t bits_at(const Blob& b, uint32_t pos) {
    uint32_t w0, w1;
    if constexpr (STAGED) {
        const uint32_t wi = min(pos >> 5, b.nwords);
        w0 = b.words[wi]; w1 = b.words[wi + 1u];
    } else {
        const uint32_t wi = pos >> 5;
        w0 = wi < b.nwords ? bswap32(b.words[wi]) : 0u; w1 = (wi + 1u) < b.nwords ? bswap32(b.words[wi + 1u]) : 0u;
    }
    return __funnelshift_l(w1, w0, pos);
}
template <bool STAGED>
__device__ __forceinline__ uint32_t code_at(const Blob& b, uint32_t j) {
    return reinterpret_cast<const uint8_t*>(b.words)[STAGED ? j ^ 3u : j];
}

// One round of a team's parse: K consecutive keys per thread, from key j0 + K t on.  All fields a thread needs are fetched
// independently of one another (the flags of its keys at once, then every delta at its own bit position), so that a
// round's chain is one fetch, one scan of the widths, one fetch, one scan of the deltas; about 20 instructions per key
// (a run of get-next-field steps took 60 and made the parse of a 2700-key group 3.6 us instead of 1.9).
// f(j, m, keys): the thread's keys j .. j + m - 1, relative to the group's start.
template <bool BLOCK, bool STAGED, int K, typename F>
__device__ __forceinline__ void parse_round(const DecArgs& a, DecShared& s, const Blob& b, uint32_t span, uint32_t j0, uint32_t t, uint32_t tn,
                                            uint32_t& bitpos, uint32_t& keybase, unsigned long long& bad, int lane, int warp, F f) {
    const uint32_t levels_m1 = (1u << a.l) - 1u;
    const uint32_t jb = j0 + t * (uint32_t)K;
    const int m = jb < b.count ? (int)min(b.count - jb, (uint32_t)K) : 0;
    uint32_t v[K], wsum = 0u, wtotal, dtotal;
    {
        uint32_t top[2];
        const uint32_t fpos = 8u * b.count + a.l * jb;
        top[0] = m > 0 ? bits_at<STAGED>(b, fpos) : 0u;
        top[1] = (K > 4 && a.l > 4u) ? (m > 4 ? bits_at<STAGED>(b, fpos + 4u * a.l) : 0u) : top[0] << (4u * a.l & 31u);
        const uint32_t c0 = b.M + levels_m1;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t fk = (top[k >> 2] >> (32u - a.l * (uint32_t)((k & 3) + 1))) & levels_m1;
            v[k] = k < m ? (fk * b.M + c0) >> a.l : 0u;
            wsum += v[k];
        }
    }
    uint32_t pos = bitpos + team_scan<BLOCK>(wsum, &wtotal, s, tn, lane, warp, 0);
    uint32_t dsum = 0u;
    bool zero = false;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t w = v[k];
        v[k] = __funnelshift_rc(bits_at<STAGED>(b, pos), 0u, 32u - w);  // (width 0 beyond the run: 0)
        pos += w;
        zero = zero || (v[k] == 0u && k < m && (k > 0 || jb > 0u));
        dsum += v[k];
    }
    uint32_t key = keybase + team_scan<BLOCK>(min(dsum, 1u << 21), &dtotal, s, tn, lane, warp, 1);      // (saturates only when already invalid)
#pragma unroll
    for (int k = 0; k < K; ++k) { key += v[k]; v[k] = key; }
    // keys ascend: the last one tells whether all lie inside the group
    bool suspect = zero || (m > 0 && key >= span);
    if (a.tau < (uint32_t)kMaxTau) {
#pragma unroll
        for (int k = 0; k < K; ++k) suspect = suspect || (k < m && (code_at<STAGED>(b, jb + k) & 0x7Fu) + 1u > a.tau);
    }
    if (suspect) {                                                      // the first failure of the run
        uint32_t prev = key - dsum;
#pragma unroll
        for (int k = K - 1; k >= 0; --k) {
            if (k < m) {
                int st = 0;
                if ((jb + k > 0u && v[k] == (k ? v[k ? k - 1 : 0] : prev)) || v[k] >= span) st = kStBadKey;
                else if ((code_at<STAGED>(b, jb + k) & 0x7Fu) + 1u > a.tau) st = kStBadCode;
                if (st) bad = min(bad, ((unsigned long long)(jb + k) << 8) | (unsigned)st);
            }
        }
    }
    if (m > 0) f(jb, m, v);
    bitpos += wtotal;
    keybase = min(keybase + dtotal, 0x7FFF0000u);                       // (saturates only when already invalid)
}

// One group of one stream, parsed by a team of `tn` threads (this one: t; several teams of a warp or block parse different
// streams at the same time), in `rounds` rounds of four (small = true) or eight keys per thread, the same in all teams that
// share a barrier.  Returns the first failure this thread has seen (key index << 8 | status; the blob's length, which
// the flags imply, counts as key 0), ~0 if none.
template <bool BLOCK, bool STAGED, typename F>
__device__ __forceinline__ unsigned long long parse_team(const DecArgs& a, DecShared& s, const Blob& b, uint32_t span, uint32_t t, uint32_t tn,
                                                         bool small, uint32_t rounds, int lane, int warp, F f) {
    uint32_t bitpos = (8u + a.l) * b.count, keybase = 0u;
    unsigned long long bad = ~0ull;
    if (small) {
        for (uint32_t r = 0; r < rounds; ++r) parse_round<BLOCK, STAGED, 4>(a, s, b, span, r * 4u * tn, t, tn, bitpos, keybase, bad, lane, warp, f);
    } else {
        for (uint32_t r = 0; r < rounds; ++r) parse_round<BLOCK, STAGED, 8>(a, s, b, span, r * 8u * tn, t, tn, bitpos, keybase, bad, lane, warp, f);
    }
    if (t == 0u && b.count != 0u && ((bitpos + 31u) >> 5) != b.nwords) bad = (unsigned long long)kStBadDirectory;
    return bad;
}

__device__ __forceinline__ float code_value(const float* val, uint32_t code) {
    const float mag = val[(code & 0x7Fu) + 1u];
    return (code & 0x80u) ? -mag : mag;
}

// 4 bytes from global into shared memory, asynchronously (any 4-byte aligned addresses)
__device__ __forceinline__ void copy_word_async(void* dst_smem, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// the same for a scattered entry: 64 bytes of its line from memory, not all 128
__device__ __forceinline__ void copy_entry_async(void* dst_smem, const void* src) {
    asm volatile("cp.async.ca.shared.global.L2::64B [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(__cvta_generic_to_global(src)) : "memory");
}

constexpr uint32_t kNoKey = 0xFFFFu;               // (in a list of keys) an entry of a stream that failed

// One group of a single stream by one warp; entry eb of the block's table is its directory entry; two: as in two_in_flight.
template <int MODE>
__device__ __forceinline__ void warp_group(const DecArgs& a, DecShared& s, uint32_t g, uint32_t eb, bool two, int lane, int warp) {
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t lo = (uint32_t)lo64, span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    uint32_t* blob = s.u.one[warp].blob;
    uint16_t* keys = s.u.one[warp].key;
    Blob b;
    b.words = blob; b.nwords = s.e_nw[eb]; b.count = s.e_cm[eb] & 0xFFFFFFu; b.M = s.e_cm[eb] >> 24;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(a.stream[0]) + s.e_off[eb];
    for (uint32_t i = lane; i < b.nwords; i += 32u) copy_word_async(&blob[i], src + i);
    copies_wait();
    __syncwarp();
    for (uint32_t i = lane; i < b.nwords; i += 32u) blob[i] = bswap32(blob[i]);
    __syncwarp();
    const bool small = b.count <= 128u;
    const unsigned long long bad = parse_team<false, true>(a, s, b, span, (uint32_t)lane, 32u, small, small ? 1u : (b.count + 255u) / 256u, lane, warp,
                                                           [&](uint32_t j, int m, const auto& v) {
        constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
        for (int k = 0; k < K; ++k) if (k < m) keys[j + (uint32_t)k] = (uint16_t)v[k];
    });
    if (bad != ~0ull) dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
    const uint32_t c0 = __any_sync(kFullMask, bad != ~0ull) ? 0u : b.count;       // a failed group is left out as a whole
    __syncwarp();
    if constexpr (MODE == 0) {
        auto add = [&](auto flight) {                          // so many entries in flight a lane
            constexpr int K = (int)(sizeof(flight) / sizeof(uint32_t));
#pragma unroll 1
            for (uint32_t e0 = 0; e0 < c0; e0 += 32u * K) {
                uint32_t kk[K]; float x[K];
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const uint32_t e = e0 + 32u * i + lane;
                    kk[i] = 0xFFFFFFFFu; x[i] = 0.0f;
                    if (e < c0) { kk[i] = lo + keys[e]; x[i] = load_entry(a.dense + kk[i]); }
                }
#pragma unroll
                for (int i = 0; i < K; ++i)
                    if (kk[i] != 0xFFFFFFFFu) a.dense[kk[i]] = __fadd_rn(x[i], code_value(s.val[0], code_at<true>(b, e0 + 32u * i + lane)));
            }
        };
        struct Two { uint32_t x[2]; };
        struct Eight { uint32_t x[8]; };
        if (two && sparse_group(c0, span)) add(Two()); else add(Eight());
    } else {
        for (uint32_t e0 = 0; e0 < c0; e0 += 128u) {
            uint32_t kk[4]; float gg[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t e = e0 + 32u * i + lane;
                kk[i] = e < c0 ? lo + keys[e] : 0u;
                // (a single stream: g is the decoded value; 0 + value is the value)
                if constexpr (MODE == 1) gg[i] = e < c0 ? atomicExch(a.dense + kk[i], 0.0f) : 0.0f;
                else gg[i] = e < c0 ? code_value(s.val[0], code_at<true>(b, e)) : 0.0f;
            }
            adam_run<MODE == 3, 4, true>(a, kk, gg);
        }
    }
    __syncwarp();                                                       // (the list is rewritten by the warp's next group)
}

template <int NW> __device__ __forceinline__ void dec_team_sync(int team) {
    if constexpr (NW == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(32 * NW) : "memory");
}
// Lane w: stream w's directory entry in the block's table (entries eb + w), and where its blob and its list begin among the group's.
struct TeamEntries {
    uint32_t count, M, off, nw, wbase, lbase, words, total;
    __device__ __forceinline__ TeamEntries(const DecShared& s, uint32_t W, uint32_t eb, int lane) {
        uint32_t cm = 0u;
        off = nw = 0u;
        if (lane < (int)W) { cm = s.e_cm[eb + lane]; off = s.e_off[eb + lane]; nw = s.e_nw[eb + lane]; }
        count = cm & 0xFFFFFFu; M = cm >> 24;
        const uint32_t wincl = warp_incl_scan(nw, lane), lincl = warp_incl_scan(count, lane);
        wbase = wincl - nw; lbase = lincl - count;
        words = __shfl_sync(kFullMask, wincl, 31); total = __shfl_sync(kFullMask, lincl, 31);
    }
};

// The streams' blobs into shared memory and parsed into lists of keys, side by side, by a team of NW warps (tl: thread of the team).  prepare(): what
// else is to be done before the first barrier, while the copies are in flight; each(k): every key as it is found.  Returns the streams that failed (bit w).
template <int NW, typename P, typename E>
__device__ __forceinline__ uint32_t team_lists(const DecArgs& a, DecShared& s, const TeamEntries& q, uint32_t W, uint32_t g, uint32_t span, uint32_t* blob,
                                               uint16_t* lists, uint32_t tl, int lane, int warp, P prepare, E each) {
    constexpr uint32_t threads = 32u * NW, nw_log2 = NW == 1 ? 0u : NW == 2 ? 1u : 2u;
    const int team = warp / NW;
    uint32_t* failed = blob + q.words + 2u;                             // bit w: stream w
    for (uint32_t w = 0; w < W; ++w) {                                  // all copies in flight together
        const uint32_t n_w = __shfl_sync(kFullMask, q.nw, w), o_w = __shfl_sync(kFullMask, q.off, w), b_w = __shfl_sync(kFullMask, q.wbase, w);
        const uint32_t* src = reinterpret_cast<const uint32_t*>(a.stream[w]) + o_w;
        for (uint32_t i = tl; i < n_w; i += threads) copy_word_async(&blob[b_w + i], src + i);
    }
    prepare();
    if (NW > 1 && tl == 0u) *failed = 0u;
    copies_wait();
    dec_team_sync<NW>(team);
    for (uint32_t i = tl; i < q.words; i += threads) blob[i] = bswap32(blob[i]);
    dec_team_sync<NW>(team);
    // ---- parse: the threads shared out among the streams, within a warp
    const uint32_t tn_log2 = min(5u, (W <= 2u ? 4u : (W <= 4u ? 3u : 2u)) + nw_log2), tn = 1u << tn_log2;
    const uint32_t mine = tl >> tn_log2;                                // (beyond W - 1: a stream without keys)
    Blob b;
    b.count = __shfl_sync(kFullMask, q.count, mine);
    b.nwords = __shfl_sync(kFullMask, q.nw, mine);
    b.M = __shfl_sync(kFullMask, q.M, mine);
    b.words = blob + __shfl_sync(kFullMask, q.wbase, mine);
    uint16_t* keys = lists + __shfl_sync(kFullMask, q.lbase, mine);
    const uint32_t most = __reduce_max_sync(kFullMask, b.count);
    const bool small = most <= 4u * tn;
    const unsigned long long bad = parse_team<false, true>(a, s, b, span, (uint32_t)lane & (tn - 1u), tn, small, small ? 1u : (most + 8u * tn - 1u) / (8u * tn),
                                                           lane, warp, [&](uint32_t j, int m, const auto& v) {
        constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
        for (int k = 0; k < K; ++k) if (k < m) { keys[j + (uint32_t)k] = (uint16_t)v[k]; each(v[k]); }
    });
    if (bad != ~0ull) {
        dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
        if (NW > 1) atomicOr(failed, 1u << mine);
    }
    uint32_t out;
    if constexpr (NW == 1) {
        out = __any_sync(kFullMask, bad != ~0ull) ? __reduce_or_sync(kFullMask, bad != ~0ull ? 1u << mine : 0u) : 0u;
        __syncwarp();
    } else {
        dec_team_sync<NW>(team);
        out = *failed;
    }
    return out;
}

// Several streams: one group by a team of NW warps (1, 2 or 4); entries eb + w of the block's table are stream w's directory entry.  One
// entry stands for every distinct key; it collects the streams' values in stream order, so that each coordinate takes one round
// trip to memory.  keys: a key, or kSharedKey | the entry that stands for it.
//
// A group is a chain of about ten steps (copy, flags, deltas, table, one addition a stream, memory) of which few fill a block's 512
// threads.  Groups of 250 to 1500 keys by the whole block took 10 us each, two at a time on an SM; by teams (32, 16 or 8 groups
// at a time) eight streams of 47 keys a group take 51 us instead of 100 (2781 groups), of 98 keys 104 instead of 136.
constexpr uint32_t kSharedKey = 0x8000u;
template <int MODE, int NW>
__device__ __forceinline__ void team_group(const DecArgs& a, DecShared& s, uint32_t W, uint32_t g, uint32_t eb, int lane, int warp) {
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t lo = (uint32_t)lo64, span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    const int team = warp / NW;
    const uint32_t tl = 32u * (uint32_t)(warp % NW) + (uint32_t)lane;   // thread of the team
    constexpr uint32_t threads = 32u * NW;
    const TeamEntries q(s, W, eb, lane);
    const uint32_t total = q.total;
    uint32_t count = q.count;
    uint8_t* mem = s.u.team[team * NW];
    uint16_t* slot = reinterpret_cast<uint16_t*>(mem);                  // table of distinct keys: the entry that stands for the key; 0xFFFF: free
    // (four times the entries as far as the memory's share goes; never less than 1.5 times)
    const uint32_t slots_log2 = min(32u - (uint32_t)__clz((int)(4u * total + 31u)), kTeamSlotsLog2 + (NW == 1 ? 0u : NW == 2 ? 1u : 2u)), slots = 1u << slots_log2;
    float* acc = reinterpret_cast<float*>(slot + kTeamSlots * NW);
    uint16_t* keys = reinterpret_cast<uint16_t*>(acc + ((total + 1u) & ~1u));
    uint32_t* blob = reinterpret_cast<uint32_t*>(keys + ((total + 1u) & ~1u));
    const uint32_t out = team_lists<NW>(a, s, q, W, g, span, blob, keys, tl, lane, warp,
        [&]() { for (uint32_t i = tl; i < slots / 2u; i += threads) reinterpret_cast<uint32_t*>(slot)[i] = 0xFFFFFFFFu; }, [](uint32_t) {});
    if (out) {                                                          // a failed stream is left out as a whole
        for (uint32_t w = 0; w < W; ++w) {
            const uint32_t b_w = __shfl_sync(kFullMask, q.lbase, w), c_w = __shfl_sync(kFullMask, count, w);
            if ((out >> w) & 1u) for (uint32_t j = tl; j < c_w; j += threads) keys[b_w + j] = kNoKey;
        }
        if ((out >> lane) & 1u) count = 0u;
        dec_team_sync<NW>(team);
    }
    // ---- who stands for each key (open addressing)
    for (uint32_t e0 = 0; e0 < total; e0 += threads) {
        const uint32_t e = e0 + tl;
        const uint32_t key = e < total ? keys[e] : kNoKey;
        bool open = key != kNoKey;
        uint32_t h = (key * 0x9E3779B1u) >> (32u - slots_log2), owner = e;
        if (MODE == 1) open = false;                                    // (g is exchanged out of dense_out: no matter how often a key comes)
        if constexpr (NW == 1) {                                        // (a lane writes its entry into a free slot and looks who is there)
            while (__any_sync(kFullMask, open)) {
                if (open && slot[h] == 0xFFFFu) slot[h] = (uint16_t)e;
                __syncwarp();
                if (open) {
                    const uint32_t r = slot[h];
                    if (r == e || keys[r] == key) { owner = r; open = false; }
                    else h = (h + 1u) & (slots - 1u);
                }
                __syncwarp();
            }
        } else {
            while (open) {
                const uint32_t r = atomicCAS(reinterpret_cast<unsigned short*>(&slot[h]), (unsigned short)0xFFFFu, (unsigned short)e);
                if (r == 0xFFFFu) open = false;
                else if (keys[r] == key) { owner = r; open = false; }
                else h = (h + 1u) & (slots - 1u);
            }
            __syncwarp();
        }
        if (key != kNoKey) {
            if (owner != e) keys[e] = (uint16_t)(kSharedKey | owner);   // (nobody looks at the key of an entry that is in no slot)
            else if constexpr (MODE == 0) copy_word_async(&acc[e], a.dense + lo + key);
            else if constexpr (MODE == 1) acc[e] = atomicExch(a.dense + lo + key, 0.0f);
            else acc[e] = 0.0f;
        }
    }
    if constexpr (MODE == 0) copies_wait();
    dec_team_sync<NW>(team);
    if constexpr (MODE != 1) {
        for (uint32_t w = 0; w < W; ++w) {
            const uint32_t b_w = __shfl_sync(kFullMask, q.lbase, w), c_w = __shfl_sync(kFullMask, count, w), s_w = __shfl_sync(kFullMask, q.wbase, w);
            const uint8_t* codes = reinterpret_cast<const uint8_t*>(blob + s_w);
            for (uint32_t j = tl; j < c_w; j += threads) {
                const uint32_t k = keys[b_w + j], at = k & kSharedKey ? k & (kSharedKey - 1u) : b_w + j;
                acc[at] = __fadd_rn(acc[at], code_value(s.val[w], codes[j ^ 3u]));
            }
            dec_team_sync<NW>(team);
        }
    }
    for (uint32_t e0 = 0; e0 < total; e0 += 4u * threads) {
        uint32_t kk[4]; float gg[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t e = e0 + threads * (uint32_t)i + tl;
            const uint32_t key = e < total ? keys[e] : kNoKey;
            const bool on = (key & kSharedKey) == 0u;                   // (a key below 2^15; not one that another entry stands for, nor kNoKey)
            kk[i] = lo + key;
            gg[i] = on ? acc[e] : 0.0f;
            if constexpr (MODE == 0) if (on) a.dense[kk[i]] = gg[i];
        }
        if constexpr (MODE != 0) adam_run<MODE == 3, 4>(a, kk, gg);
    }
    dec_team_sync<NW>(team);                                            // (the memory is rewritten for the team's next group)
}

// The same by a team of four warps, for groups of many keys: a bit for every index of the group and counts of the bits before each word give
// every distinct key its rank, and the sums go to memory in the order of the coordinates, so that what shares a line is asked for together.
// (With the table, coordinates came in the streams' order, and it was a third of the instructions: eight streams of 671 K keys over 67 M, the update on the packed
// state 285 us, now 216.  Of few keys a group the bits cost more than the table: 29 keys of each of four streams 12.9 us, so 14.4.)
template <int MODE>
__device__ __forceinline__ void ranked_group(const DecArgs& a, DecShared& s, uint32_t W, uint32_t g, uint32_t eb, int lane, int warp) {
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t lo = (uint32_t)lo64, span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    constexpr uint32_t threads = 128u;
    const int team = warp / 4;
    const uint32_t tl = 32u * (uint32_t)(warp % 4) + (uint32_t)lane;    // thread of the team
    const TeamEntries q(s, W, eb, lane);
    const uint32_t total = q.total, even = (total + 1u) & ~1u;
    uint32_t count = q.count;
    const uint32_t map_words = (1u << a.group_log2) / 32u;
    uint32_t* bits = reinterpret_cast<uint32_t*>(s.u.team[team * 4]);
    uint16_t* before = reinterpret_cast<uint16_t*>(bits + map_words);   // bits set in the words before
    float* acc = reinterpret_cast<float*>(before + map_words);          // per rank: the sum
    uint16_t* key_of = reinterpret_cast<uint16_t*>(acc + even);         // ... and the key
    uint16_t* list = key_of + even;                                     // the streams' keys, then their ranks
    uint32_t* blob = reinterpret_cast<uint32_t*>(list + even);
    uint32_t* sums = blob + q.words + 3u;                               // (behind the failed streams' bits) bits set in the words of each warp
    auto clear = [&]() { for (uint32_t i = tl; i < map_words / 4u; i += threads) reinterpret_cast<uint4*>(bits)[i] = make_uint4(0u, 0u, 0u, 0u); };
    auto mark = [&](uint32_t k) { if (k < span) atomicOr(&bits[k >> 5], 1u << (k & 31u)); };      // (beyond: the stream fails)
    const uint32_t out = team_lists<4>(a, s, q, W, g, span, blob, list, tl, lane, warp, clear, mark);
    if (out) {                                                          // a failed stream is left out as a whole: the others' keys again
        clear();
        if ((out >> lane) & 1u) count = 0u;
        dec_team_sync<4>(team);
        for (uint32_t w = 0; w < W; ++w) {
            const uint32_t b_w = __shfl_sync(kFullMask, q.lbase, w), c_w = __shfl_sync(kFullMask, q.count, w);
            for (uint32_t j = tl; j < c_w; j += threads) {
                if ((out >> w) & 1u) list[b_w + j] = kNoKey; else mark(list[b_w + j]);
            }
        }
        dec_team_sync<4>(team);
    }
    // ---- counts of the bits before each word
    uint32_t distinct;
    {
        const uint32_t per = max(1u, map_words / 512u), w0 = tl * per;      // in fours of words
        const uint4* fours = reinterpret_cast<const uint4*>(bits);
        const bool any = 4u * w0 < map_words;
        uint32_t c = 0u;
        if (any) for (uint32_t i = 0; i < per; ++i) { const uint4 q = fours[w0 + i]; c += (uint32_t)(__popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w)); }
        const uint32_t incl = warp_incl_scan(c, lane);
        uint32_t at = incl - c;
        if (lane == 31) sums[tl >> 5] = incl;
        dec_team_sync<4>(team);
        distinct = 0u;
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) { if (i == (tl >> 5)) at += distinct; distinct += sums[i]; }
        if (any) for (uint32_t i = 0; i < per; ++i) {
            const uint4 q = fours[w0 + i];
            const uint32_t x = at + (uint32_t)__popc(q.x), y = x + (uint32_t)__popc(q.y), z = y + (uint32_t)__popc(q.z);
            reinterpret_cast<uint2*>(before)[w0 + i] = make_uint2(at | (x << 16), y | (z << 16));
            at = z + (uint32_t)__popc(q.w);
        }
    }
    dec_team_sync<4>(team);
    // ---- ranks, and what their sums start from (a key of several streams: the same every time)
    for (uint32_t e0 = tl; e0 < total; e0 += 4u * threads) {
        uint32_t k[4], word[4], r[4];
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) k[i] = e0 + threads * i < total ? (uint32_t)list[e0 + threads * i] : (uint32_t)kNoKey;
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) { word[i] = 0u; r[i] = 0u; if (k[i] != kNoKey) { word[i] = bits[k[i] >> 5]; r[i] = before[k[i] >> 5]; } }
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            if (k[i] == kNoKey) continue;
            r[i] += (uint32_t)__popc(word[i] & ((1u << (k[i] & 31u)) - 1u));
            list[e0 + threads * i] = (uint16_t)r[i];
            key_of[r[i]] = (uint16_t)k[i];
            if constexpr (MODE == 0) copy_entry_async(&acc[r[i]], a.dense + lo + k[i]);
            else acc[r[i]] = 0.0f;
        }
    }
    if constexpr (MODE == 0) copies_wait();
    dec_team_sync<4>(team);
    if constexpr (MODE != 1) {
        for (uint32_t w = 0; w < W; ++w) {
            const uint32_t b_w = __shfl_sync(kFullMask, q.lbase, w), c_w = __shfl_sync(kFullMask, count, w), s_w = __shfl_sync(kFullMask, q.wbase, w);
            if (c_w == 0u) continue;
            const uint8_t* codes = reinterpret_cast<const uint8_t*>(blob + s_w);
            for (uint32_t j = tl; j < c_w; j += threads) {
                const uint32_t r = list[b_w + j];
                acc[r] = __fadd_rn(acc[r], code_value(s.val[w], codes[j ^ 3u]));
            }
            dec_team_sync<4>(team);
        }
    }
    for (uint32_t r0 = 0; r0 < distinct; r0 += 4u * threads) {
        uint32_t kk[4]; float gg[4];
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            const uint32_t r = r0 + threads * i + tl;
            const bool on = r < distinct;
            kk[i] = on ? lo + key_of[r] : 0u;
            gg[i] = 0.0f;
            if (on) {
                if constexpr (MODE == 0) a.dense[kk[i]] = acc[r];
                else if constexpr (MODE == 1) { gg[i] = a.dense[kk[i]]; a.dense[kk[i]] = 0.0f; }
                else gg[i] = acc[r];
            }
        }
        if constexpr (MODE != 0) adam_run<MODE == 3, 4, true>(a, kk, gg);
    }
    dec_team_sync<4>(team);                                       // (the memory is rewritten for the team's next group)
}

// entry x of the list of groups for one (list 0), two or four (2) warps
__device__ __forceinline__ uint16_t& team_list_entry(DecShared& s, uint32_t list, uint32_t x) {
    return list == 0u ? s.light[x] : list == 1u ? s.heavy[kDecThreads - 1u - x] : s.light[kDecThreads - 1u - x];
}

// The block's groups for teams of NW warps, one after the other to whichever team is free.  table (teams of four, aggregation): as in TeamRule.
template <int MODE, int NW>
__device__ __forceinline__ void team_groups(const DecArgs& a, DecShared& s, uint32_t W, uint32_t first, int lane, int warp, bool table = false) {
    constexpr uint32_t kList = NW == 1 ? 0u : NW == 2 ? 1u : 2u;
    const uint32_t n = s.n_light[kList];
    const int team = warp / NW;
    for (;;) {
        uint32_t x = 0u;
        if (warp % NW == 0 && lane == 0) { x = atomicAdd(&s.next_light[kList], 1u); if (NW > 1) s.grab[team] = x; }
        if constexpr (NW == 1) x = __shfl_sync(kFullMask, x, 0);
        else { dec_team_sync<NW>(team); x = s.grab[team]; }
        if (x >= n) break;
        const uint32_t i = team_list_entry(s, kList, x);
        const uint32_t g = blockIdx.x + (first + i) * gridDim.x;
        if (NW < 4 || (MODE == 0 && table)) team_group<MODE, NW>(a, s, W, g, i * W, lane, warp);
        else ranked_group<MODE>(a, s, W, g, i * W, lane, warp);
    }
}

// index of coordinate k's aggregated gradient (or entry of dense_out) as a float
template <int MODE> __device__ __forceinline__ uint64_t dense_at(uint32_t k) { return MODE == 3 ? 4ull * k + 3ull : (uint64_t)k; }

// The model update of all coordinates of a group with a gradient in its slice of g, coordinate by coordinate.
template <int MODE>
__device__ __forceinline__ void update_slice(const DecArgs& a, const float* tile, uint32_t lo, uint32_t span, int tid) {
    for (uint32_t i0 = 0; i0 < span; i0 += 4u * (uint32_t)kDecThreads) {
        uint32_t kk[4]; float gg[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t idx = i0 + (uint32_t)i * kDecThreads + tid;
            kk[i] = lo + idx;
            gg[i] = idx < span ? tile[idx] : 0.0f;
        }
        adam_run<MODE == 3, 4>(a, kk, gg);
    }
}

// K entries of stream w (those whose bit of `on` is set) straight in memory, all accesses of a step in flight together: added into
// dense_out, or (update) their coordinates updated once with the g that the streams have left there (one stream: with its value).
template <bool ONE, int MODE, int K>
__device__ __forceinline__ void entries_in_memory(const DecArgs& a, const DecShared& s, uint32_t w, uint32_t lo, bool update, uint32_t on, const uint32_t (&key)[K], const uint32_t (&code)[K]) {
    uint32_t kk[K]; float x[K];
#pragma unroll
    for (int i = 0; i < K; ++i) { kk[i] = lo + key[i]; x[i] = 0.0f; }
    if (MODE == 0 || (MODE == 2 && !update)) {
#pragma unroll
        for (int i = 0; i < K; ++i) if ((on >> i) & 1u) x[i] = a.dense[kk[i]];
#pragma unroll
        for (int i = 0; i < K; ++i) if ((on >> i) & 1u) a.dense[kk[i]] = __fadd_rn(x[i], code_value(s.val[w], code[i]));
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) if ((on >> i) & 1u) x[i] = ONE && mode_fused(MODE) ? code_value(s.val[w], code[i]) : atomicExch(a.dense + dense_at<MODE>(kk[i]), 0.0f);
        adam_run<MODE == 3, K>(a, kk, x);
    }
}

// A group's blobs for the block: all streams' together in the stage, or (together = false) one in each half of it, or (staged = false) where
// they are in memory.
struct Stage {
    uint32_t words, listed; bool together, staged;                     // (listed: entries of the lists, each padded to a multiple of 8)
    __device__ __forceinline__ Stage(const DecShared& s, uint32_t W) : words(0u), listed(0u), staged(true) {
        for (uint32_t w = 0; w < W; ++w) { words += s.g_nwords[w]; listed += (s.g_count[w] + 7u) & ~7u; }
        together = words <= kBlockStageWords;
        for (uint32_t w = 0; w < W; ++w) staged = staged && (together || s.g_nwords[w] <= kBlockStageWords / 2u);
    }
    __device__ __forceinline__ void copy(const DecArgs& a, DecShared& s, uint32_t w, uint32_t at, int tid) const {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(a.stream[w]) + s.g_off[w];
        for (uint32_t i = tid; i < s.g_nwords[w]; i += kDecThreads) copy_word_async(&s.u.bstage[at + i], src + i);
    }
    __device__ __forceinline__ void swap(DecShared& s, uint32_t w, uint32_t at, int tid) const {      // (every thread the words it has copied itself)
        for (uint32_t i = tid; i < s.g_nwords[w]; i += kDecThreads) s.u.bstage[at + i] = bswap32(s.u.bstage[at + i]);
    }
    __device__ __forceinline__ Blob blob(const DecArgs& a, const DecShared& s, uint32_t w) const {
        Blob b;
        b.words = staged ? s.u.bstage + s.g_base[w] : reinterpret_cast<const uint32_t*>(a.stream[w]) + s.g_off[w];
        b.nwords = s.g_nwords[w]; b.count = s.g_count[w]; b.M = s.g_M[w];
        return b;
    }
};

// One group wider than the tile by the whole block, in memory.  (A function of its own, so that its registers do not weigh on the groups of
// the default size: inlined, these took 3 % longer.)
template <bool ONE, int MODE>
__device__ __noinline__ void block_wide(const DecArgs& a, DecShared& s, uint32_t W, uint32_t g) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t lo = (uint32_t)lo64, span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    const Stage st(s, W);
    {
        uint32_t used = 0u, list = 0u;
        for (uint32_t w = 0; w < W; ++w) {
            if (tid == 0) { s.g_base[w] = st.together ? used : (w & 1u) * (kBlockStageWords / 2u + 2u); s.g_list[w] = list; s.bad[w] = 0u; }
            if (st.together) st.copy(a, s, w, used, tid);
            used += s.g_nwords[w]; list += (s.g_count[w] + 7u) & ~7u;
        }
        if (st.together) {
            copies_wait();
            used = 0u;
            for (uint32_t w = 0; w < W; ++w) { st.swap(s, w, used, tid); used += s.g_nwords[w]; }
        }
    }
    __syncthreads();
    uint32_t* wkey = reinterpret_cast<uint32_t*>(s.u.tile);             // a list of 32-bit keys
    const int sweeps = MODE == 2 && !ONE ? 2 : 1;                       // (the update in one launch: g first, from all streams)
    auto code_of = [&](const Blob& b, uint32_t j) -> uint32_t { return st.staged ? code_at<true>(b, j) : code_at<false>(b, j); };
    auto apply_list = [&](uint32_t w, const Blob& b, uint32_t l0, bool update) {      // neighbouring threads on neighbouring keys
        for (uint32_t j0 = (uint32_t)tid; j0 < b.count; j0 += 4u * kDecThreads) {
            uint32_t key[4], code[4], on = 0u;
#pragma unroll
            for (uint32_t i = 0; i < 4u; ++i) {
                const uint32_t j = j0 + i * kDecThreads;
                key[i] = 0u; code[i] = 0u;
                if (j < b.count) { on |= 1u << i; key[i] = wkey[l0 + j]; code[i] = code_of(b, j); }
            }
            entries_in_memory<ONE, MODE, 4>(a, s, w, lo, update, on, key, code);
        }
    };
    if (st.listed <= kWideListMax && st.together) {
        // ---- all streams parsed side by side into lists, then applied one after the other.  (Before, each stream was parsed twice, the second
        // time by threads that took runs of consecutive keys one access at a time: 442 groups of 2^15, eight streams of 200 keys, 87 us, now
        // 38; 12.8 M entries in groups of 2^17, five streams, the update 60, now 21.)
        const uint32_t tn = ONE ? (uint32_t)kDecThreads : (W <= 2u ? kDecThreads / 2u : (W <= 4u ? kDecThreads / 4u : kDecThreads / 8u));
        const uint32_t mine = ONE ? 0u : (uint32_t)tid / tn;
        uint32_t most = 0u;
        for (uint32_t w = 0; w < W; ++w) most = max(most, s.g_count[w]);
        const bool small = most <= 4u * tn;
        Blob b = st.blob(a, s, mine < W ? mine : 0u);
        if (mine >= W) b.count = 0u;
        const uint32_t list = mine < W ? s.g_list[mine] : 0u;
        const unsigned long long bad = parse_team<true, true>(a, s, b, span, (uint32_t)tid & (tn - 1u), tn, small, small ? 1u : (most + 8u * tn - 1u) / (8u * tn),
                                                              lane, warp, [&](uint32_t j, int m, const auto& v) {
            constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
            for (int k = 0; k < K; ++k) if (k < m) wkey[list + j + (uint32_t)k] = v[k];
        });
        if (bad != ~0ull) {
            s.bad[mine] = 1u;
            dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
        }
        __syncthreads();
        for (int sweep = 0; sweep < sweeps; ++sweep) {
            for (uint32_t w = 0; w < W; ++w) {
                if (!s.bad[w]) apply_list(w, st.blob(a, s, w), s.g_list[w], MODE == 1 || (MODE == 2 && sweep + 1 == sweeps));      // (a failed stream is left out as a whole)
                __syncthreads();                                        // this stream's updates before the next stream's
            }
        }
    } else {
        // ---- stream by stream; one that has more keys than the list holds is parsed once to validate and once to apply
        for (int sweep = 0; sweep < sweeps; ++sweep) {
            const bool update = MODE == 1 || (MODE == 2 && sweep + 1 == sweeps);
            if (st.staged && !st.together) st.copy(a, s, 0u, s.g_base[0], tid);
            for (uint32_t w = 0; w < W; ++w) {
                const Blob b = st.blob(a, s, w);
                if (st.staged && !st.together) {
                    copies_wait();
                    st.swap(s, w, s.g_base[w], tid);
                    __syncthreads();
                    if (w + 1u < W) st.copy(a, s, w + 1u, s.g_base[w + 1u], tid);
                }
                if (b.count == 0u) continue;                            // (uniform; the next stream's copy goes to the other half of the stage)
                const bool fits = b.count <= kWideListMax, small = b.count <= 4u * kDecThreads;
                const uint32_t rounds = small ? 1u : (b.count + 8u * kDecThreads - 1u) / (8u * kDecThreads);
                auto put = [&](uint32_t j, int m, const auto& v) {
                    constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
                    for (int k = 0; k < K; ++k) if (fits && k < m) wkey[j + (uint32_t)k] = v[k];
                };
                const unsigned long long bad = st.staged ? parse_team<true, true>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, put)
                                                         : parse_team<true, false>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, put);
                if (bad != ~0ull) dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
                if (!__syncthreads_or(bad != ~0ull ? 1 : 0)) {          // validated in full before any of it is applied
                    auto apply_run = [&](uint32_t j, int m, const auto& v) {
                        constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
                        for (int k0 = 0; k0 < K; k0 += 4) {
                            uint32_t key[4], code[4], on = 0u;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                key[k] = v[k0 + k]; code[k] = 0u;
                                if (k0 + k < m) { on |= 1u << k; code[k] = code_of(b, j + (uint32_t)(k0 + k)); }
                            }
                            entries_in_memory<ONE, MODE, 4>(a, s, w, lo, update, on, key, code);
                        }
                    };
                    if (fits) apply_list(w, b, 0u, update);
                    else if (st.staged) parse_team<true, true>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, apply_run);
                    else parse_team<true, false>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, apply_run);
                }
                __syncthreads();                                        // this stream's updates before the next stream's
            }
        }
    }
    __syncthreads();
}

// One group of up to 2^14 indices by the whole block; s.g_* hold its directory entries.
template <bool ONE, int MODE>
__device__ __forceinline__ void block_group(const DecArgs& a, DecShared& s, uint32_t W, uint32_t g, uint32_t& tile_parity, int tid, int lane, int warp) {
    const uint64_t lo64 = (uint64_t)g << a.group_log2;
    const uint64_t hi64 = lo64 + (1ull << a.group_log2);
    const uint32_t lo = (uint32_t)lo64, span = (uint32_t)((hi64 < a.n ? hi64 : a.n) - lo64);
    uint32_t total = 0u, words = 0u;
    uint32_t listed = 0u;                                               // entries of the lists (each padded to a multiple of 8)
    for (uint32_t w = 0; w < W; ++w) { total += s.g_count[w]; words += s.g_nwords[w]; listed += (s.g_count[w] + 7u) & ~7u; }
    const bool lists = listed <= kBlockListMax && words <= kBlockStageWords;      // (else: stream by stream)
    const bool bulk_ok = ((reinterpret_cast<uintptr_t>(a.dense) & 15u) == 0u) && ((span & 3u) == 0u);
    // aggregation of many keys: the slice of dense_out goes through shared memory as a whole
    const bool slice = MODE == 0 && (total >= slice_min(bulk_ok, ONE, a.n) || !lists);
    if (tid == 0) {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // the last write-back has read the tile
        if (slice && bulk_ok) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(&s.tile_bar, span * 4u);
            bulk_load(s.u.tile, a.dense + lo, span * 4u, &s.tile_bar);
        }
    }
    // (all streams' blobs together, or, where that is too much, one after the other, the next one's copy under way meanwhile)
    const bool together = words <= kBlockStageWords;
    bool staged = true;
    for (uint32_t w = 0; w < W; ++w) staged = staged && (together || s.g_nwords[w] <= kBlockStageWords / 2u);
    auto stage_copy = [&](uint32_t w, uint32_t at) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(a.stream[w]) + s.g_off[w];
        for (uint32_t i = tid; i < s.g_nwords[w]; i += kDecThreads) copy_word_async(&s.u.bstage[at + i], src + i);
    };
    auto stage_swap = [&](uint32_t w, uint32_t at) {                     // (every thread the words it has copied itself)
        for (uint32_t i = tid; i < s.g_nwords[w]; i += kDecThreads) s.u.bstage[at + i] = bswap32(s.u.bstage[at + i]);
    };
    {
        uint32_t used = 0u, listed = 0u;
        for (uint32_t w = 0; w < W; ++w) {
            const uint32_t nw = s.g_nwords[w], c = s.g_count[w];
            if (tid == 0) { s.g_base[w] = together ? used : (w & 1u) * (kBlockStageWords / 2u + 2u); s.g_list[w] = listed; s.bad[w] = 0u; }
            if (together) stage_copy(w, used);
            // (a stream's list starts at a multiple of 8 entries: a thread's eight keys are stored at once)
            if (lists && tid < (int)(-c & 7u)) s.u.lkey[listed + c + tid] = kNoKey;
            used += nw; listed += (c + 7u) & ~7u;
        }
        if (together) {
            copies_wait();
            used = 0u;
            for (uint32_t w = 0; w < W; ++w) { stage_swap(w, used); used += s.g_nwords[w]; }
        }
    }
    __syncthreads();
    auto blob_of = [&](uint32_t w) -> Blob {
        Blob b;
        b.words = staged ? s.u.bstage + s.g_base[w] : reinterpret_cast<const uint32_t*>(a.stream[w]) + s.g_off[w];
        b.nwords = s.g_nwords[w]; b.count = s.g_count[w]; b.M = s.g_M[w];
        return b;
    };
    auto code_of = [&](const Blob& b, uint32_t j) -> uint32_t { return staged ? code_at<true>(b, j) : code_at<false>(b, j); };
    auto wait_slice = [&]() -> bool {                     // the slice is in shared memory (bounded wait); false: the group is skipped
        if (bulk_ok) {
            if (tid == 0) s.got = mbar_wait(&s.tile_bar, tile_parity, a.try_limit) ? 1u : 0u;
            tile_parity ^= 1u;
        } else {
            for (uint32_t i = tid; i < span; i += kDecThreads) s.u.tile[i] = a.dense[lo + i];
            if (tid == 0) s.got = 1u;
        }
        __syncthreads();
        if (s.got == 0u && tid == 0) dec_fail(a, g, 0u, kStTimeout);
        return s.got != 0u;
    };
    auto store_slice = [&]() {
        if (bulk_ok) {
            if (tid == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the updates above, before the copy reads them
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(__cvta_generic_to_global(a.dense + lo)), "r"(smem_u32(s.u.tile)), "r"(span * 4u) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        } else {
            for (uint32_t i = tid; i < span; i += kDecThreads) a.dense[lo + i] = s.u.tile[i];
        }
    };

    // model update of many keys: a sweep over the slice of g
    const bool sweep_all = mode_fused(MODE) && (total >= (MODE == 2 ? kSweepMinKeys : kSweepMinPacked) || !lists) &&
                           (MODE == 3 || ((reinterpret_cast<uintptr_t>(a.theta) | reinterpret_cast<uintptr_t>(a.m) | reinterpret_cast<uintptr_t>(a.v)) & 15u) == 0u);
    if (lists) {
        // ---- all streams parsed side by side into the lists
        const uint32_t tn = ONE ? (uint32_t)kDecThreads : (W <= 2u ? kDecThreads / 2u : (W <= 4u ? kDecThreads / 4u : kDecThreads / 8u));
        const uint32_t mine = ONE ? 0u : (uint32_t)tid / tn;
        uint32_t most = 0u;
        for (uint32_t w = 0; w < W; ++w) most = max(most, s.g_count[w]);
        const bool small = most <= 4u * tn;
        Blob b = blob_of(mine < W ? mine : 0u);
        if (mine >= W) b.count = 0u;
        const uint32_t list = mine < W ? s.g_list[mine] : 0u;
        const unsigned long long bad = parse_team<true, true>(a, s, b, span, (uint32_t)tid & (tn - 1u), tn, small, small ? 1u : (most + 8u * tn - 1u) / (8u * tn),
                                                              lane, warp, [&](uint32_t j, int m, const auto& v) {
            constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
            uint32_t p[K / 2];
#pragma unroll
            for (int k = 0; k < K; k += 2) p[k / 2] = (k < m ? v[k] & 0xFFFFu : (uint32_t)kNoKey) | (k + 1 < m ? v[k + 1] << 16 : (uint32_t)kNoKey << 16);
            if constexpr (K == 8) *reinterpret_cast<uint4*>(&s.u.lkey[list + j]) = make_uint4(p[0], p[1], p[2], p[3]);
            else *reinterpret_cast<uint2*>(&s.u.lkey[list + j]) = make_uint2(p[0], p[1]);
        });
        if (bad != ~0ull) {
            s.bad[mine] = 1u;
            dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
        }
        if (__syncthreads_or(bad != ~0ull ? 1 : 0)) {                   // a failed stream is left out as a whole
            for (uint32_t w = 0; w < W; ++w)
                if (s.bad[w]) for (uint32_t j = tid; j < s.g_count[w]; j += kDecThreads) s.u.lkey[s.g_list[w] + j] = kNoKey;
            __syncthreads();
        }
        auto keys_of = [&](uint32_t w) -> uint32_t { return s.bad[w] ? 0u : s.g_count[w]; };
        if (MODE == 0 && slice) {
            if (!wait_slice()) return;
        } else if (sweep_all) {
            for (uint32_t i = tid; i < ((span + 3u) >> 2); i += kDecThreads)
                reinterpret_cast<float4*>(s.u.tile)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
        } else if constexpr (!ONE && MODE != 1) {
            // few enough keys that touching them alone is less than the whole slice: the entries at the lists' keys are brought into
            // the tile (a key of several streams: the same value every time), updated there stream by stream and taken back
            for (uint32_t e = tid; e < listed; e += kDecThreads) {
                const uint32_t k = s.u.lkey[e];
                if (k != kNoKey) {
                    if constexpr (MODE == 0) copy_word_async(&s.u.tile[k], a.dense + lo + k);
                    else s.u.tile[k] = 0.0f;
                }
            }
            if constexpr (MODE == 0) copies_wait();
            __syncthreads();
        }
        if constexpr (MODE != 1) {
            if (!ONE || (MODE == 0 && slice) || sweep_all) {
                for (uint32_t w = 0; w < W; ++w) {
                    const uint32_t c = keys_of(w), l0 = s.g_list[w];
                    const Blob bw = blob_of(w);
                    for (uint32_t j = tid; j < c; j += kDecThreads) {
                        const uint32_t k = s.u.lkey[l0 + j];
                        s.u.tile[k] = __fadd_rn(s.u.tile[k], code_value(s.val[w], code_at<true>(bw, j)));
                    }
                    __syncthreads();
                }
            }
        }
        if (MODE == 0 && slice) {
            store_slice();
        } else if (sweep_all) {
            if constexpr (MODE == 2) adam_sweep(a, s.u.tile, lo, span, tid, kDecThreads);
            else if constexpr (MODE == 3) update_slice<MODE>(a, s.u.tile, lo, span, tid);
        } else {
            // all lists in one sweep, neighbouring threads on neighbouring keys, the loads of four keys per thread in flight together
            const Blob b0 = blob_of(0);
            for (uint32_t e0 = 0; e0 < listed; e0 += 4u * kDecThreads) {
                uint32_t kk[4]; float x[4]; bool on[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t e = e0 + (uint32_t)i * kDecThreads + tid;
                    const uint32_t k = e < listed ? s.u.lkey[e] : kNoKey;
                    on[i] = k != kNoKey;
                    kk[i] = lo + k;
                    x[i] = 0.0f;
                    if (on[i]) {
                        if constexpr (MODE == 0) x[i] = ONE ? a.dense[kk[i]] : s.u.tile[k];
                        else if constexpr (MODE == 1) x[i] = atomicExch(a.dense + kk[i], 0.0f);
                        else if constexpr (ONE) x[i] = code_value(s.val[0], code_at<true>(b0, e));
                        else x[i] = atomicExch(&s.u.tile[k], 0.0f);     // (the first to take a key's g updates it, the others find 0)
                    }
                }
                if constexpr (MODE == 0) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (on[i]) a.dense[kk[i]] = ONE ? __fadd_rn(x[i], code_value(s.val[0], code_at<true>(b0, e0 + (uint32_t)i * kDecThreads + tid))) : x[i];
                } else {
                    adam_run<MODE == 3, 4>(a, kk, x);
                }
            }
        }
    } else {
        // ---- more keys than the lists hold: stream by stream, the whole block on each
        if (slice) { if (!wait_slice()) return; }
        if constexpr (mode_fused(MODE)) {
            for (uint32_t i = tid; i < ((span + 3u) >> 2); i += kDecThreads)
                reinterpret_cast<float4*>(s.u.tile)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
        }
        if (staged && !together) stage_copy(0u, s.g_base[0]);
        for (uint32_t w = 0; w < W; ++w) {
            const Blob b = blob_of(w);
            if (staged && !together) {
                copies_wait();
                stage_swap(w, s.g_base[w]);
                __syncthreads();
                if (w + 1u < W) stage_copy(w + 1u, s.g_base[w + 1u]);
            }
            if (b.count == 0u) continue;                            // (uniform; the next stream's copy goes to the other half of the stage)
            // (one stream at a time fits the list far more often than all of them: parsed once then, else once to validate and once to apply)
            const bool fits = b.count <= kBlockListMax;
            const bool small = b.count <= 4u * kDecThreads;
            const uint32_t rounds = small ? 1u : (b.count + 8u * kDecThreads - 1u) / (8u * kDecThreads);
            auto put = [&](uint32_t j, int m, const auto& v) {
                constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
                for (int k = 0; k < K; ++k) if (fits && k < m) s.u.lkey[j + (uint32_t)k] = (uint16_t)v[k];
            };
            const unsigned long long bad = staged ? parse_team<true, true>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, put)
                                                  : parse_team<true, false>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, put);
            if (bad != ~0ull) dec_fail(a, g, (uint32_t)(bad >> 8), (int)(bad & 0xFFull));
            if (!__syncthreads_or(bad != ~0ull ? 1 : 0)) {          // validated in full before any of it is applied
                auto apply = [&](uint32_t j, uint32_t key) {
                    if constexpr (MODE != 1) s.u.tile[key] = __fadd_rn(s.u.tile[key], code_value(s.val[w], code_of(b, j)));
                    else {
                        const uint32_t kk[1] = {lo + key};
                        const float gg[1] = {atomicExch(a.dense + lo + key, 0.0f)};
                        adam_run<false, 1>(a, kk, gg);
                    }
                };
                auto apply_run = [&](uint32_t j, int m, const auto& v) {
                    constexpr int K = (int)(sizeof(v) / sizeof(v[0]));
#pragma unroll
                    for (int k = 0; k < K; ++k) if (k < m) apply(j + (uint32_t)k, v[k]);
                };
                if (fits) for (uint32_t j = tid; j < b.count; j += kDecThreads) apply(j, s.u.lkey[j]);
                else if (staged) parse_team<true, true>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, apply_run);
                else parse_team<true, false>(a, s, b, span, (uint32_t)tid, (uint32_t)kDecThreads, small, rounds, lane, warp, apply_run);
            }
            __syncthreads();                                        // this stream's updates before the next stream's
        }
        if (MODE == 0 && slice) {
            store_slice();
        } else if (sweep_all) {
            if constexpr (MODE == 2) adam_sweep(a, s.u.tile, lo, span, tid, kDecThreads);
            else if constexpr (MODE == 3) update_slice<MODE>(a, s.u.tile, lo, span, tid);
        } else if constexpr (mode_fused(MODE)) {
            update_slice<MODE>(a, s.u.tile, lo, span, tid);
        }
    }
    __syncthreads();
}

// ONE: the launch holds a single stream (its own instantiation, so that the code of the many-stream paths does not weigh on it).
template <bool ONE, int MODE = 0>
__global__ void __launch_bounds__(kDecThreads, 2)
k_decode_accumulate(const __grid_constant__ DecArgs a, const __grid_constant__ PowTable pw, const __grid_constant__ PowTable inv) {
    extern __shared__ __align__(128) unsigned char dec_smem_raw[];
    DecShared& s = *reinterpret_cast<DecShared*>(dec_smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t W = ONE ? 1u : a.W;
    const uint32_t B = gridDim.x;
    const uint32_t owned = blockIdx.x < a.G ? (a.G - blockIdx.x + B - 1u) / B : 0u;      // groups blockIdx.x + i B
    const uint32_t per_batch = (uint32_t)kDecThreads / W;
    const uint64_t fixed_bytes = (uint64_t)kHeaderBytes + 8ull * a.G;

    uint32_t tile_parity = 0;

    if (tid == 0) {
        mbar_init(&s.tile_bar, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    wait_for_previous_kernels();
    // (The next kernel's blocks may move in from here on, not before: else, with few blocks to a launch, those of several launches in a row
    // stand on the GPU at once, and two that work share an SM while others wait with one to themselves.  64 groups of 2^20 entries, two
    // streams, launches in a row: 214 us, now 144.)
    allow_next_kernel();
    // ---- headers and the first batch of directory entries, requested together
    static_assert(16 * kDecMaxStreams <= kDecThreads, "a thread per header word");
    if (tid < (int)(16u * W)) s.hdr[tid >> 4][tid & 15] = reinterpret_cast<const uint32_t*>(a.stream[tid >> 4])[tid & 15];
    const uint32_t my_w = ONE ? 0u : (uint32_t)tid % W, my_i = ONE ? (uint32_t)tid : (uint32_t)tid / W;
    uint32_t d0 = 0u, d1 = 0u, d2 = 0u;
    auto load_dir = [&](uint32_t i) {
        // (a stream too short for its directory is not looked into: its header fails the check)
        if (my_i < per_batch && i < owned && a.bytes[my_w] >= fixed_bytes) {
            const uint32_t g = blockIdx.x + i * B;
            const uint32_t* e = reinterpret_cast<const uint32_t*>(a.stream[my_w]) + (kHeaderBytes >> 2) + 2u * g;
            const uint2 x = *reinterpret_cast<const uint2*>(e);
            d0 = x.x; d1 = x.y; d2 = g + 1u < a.G ? e[3] : 0u;
        }
    };
    load_dir(my_i);
    __syncthreads();
    if (tid < (int)W) {
        uint64_t total = 0; double S = 0.0;
        const int st = check_header(a, a.bytes[tid], s.hdr[tid], &total, &S);
        s.ok[tid] = st == kStOk ? 1u : 0u;
        s.total_words[tid] = (uint32_t)(total >> 2);
        s.sum[tid] = S;
        if (st != kStOk && blockIdx.x == 0) dec_fail(a, 0u, 0u, st);
    }
    __syncthreads();
    // several streams: keys of a group on average (what the headers say: it steers who decodes a group, nothing else)
    if (!ONE && tid == kDecThreads - 1) {
        float keys = 0.0f;
        for (uint32_t w = 0; w < W; ++w) keys += (float)s.hdr[w][6];
        s.mean = (uint32_t)fminf(__fdividef(keys, (float)a.G), 65535.0f);
    }
    // phases 3-4 as a table per stream: value[L] = (float)(sum / b^L).  The division is a multiplication by the reciprocal
    // (within 2^-51 of the quotient) whenever everything within 2^-50 of the product rounds to the same float.
    for (uint32_t idx = tid; idx < W * 132u; idx += kDecThreads) {
        const uint32_t w = idx / 132u, k = idx % 132u;
        if (k <= a.tau && s.ok[w]) {
            const double q = __dmul_rn(s.sum[w], inv.P[k]);
            const float lo = __double2float_rn(__dmul_rn(q, 1.0 - 0x1p-50)), hi = __double2float_rn(__dmul_rn(q, 1.0 + 0x1p-50));
            s.val[w][k] = lo == hi ? lo : __double2float_rn(__ddiv_rn(s.sum[w], pw.P[k]));
        }
    }

    unsigned int* q_taken = a.q_ctl + 1, *q_done = a.q_ctl + 2, *q_exited = a.q_ctl + 3, *q_reserved = a.q_ctl + 4;
    const bool queue = a.G > B;
    for (uint32_t first = 0; first < owned; first += per_batch) {
        if (first > 0u) { __syncthreads(); d0 = d1 = d2 = 0u; load_dir(first + my_i); }
        // ---- classify the batch's groups
        s.gtot[tid] = 0u;
        if (tid < 3) { s.n_light[tid] = 0u; s.next_light[tid] = 0u; }
        if (tid == 0) s.n_heavy = 0u;
        __syncthreads();
        const uint32_t in_batch = min(per_batch, owned - first);
        if (my_i < in_batch) {
            const uint32_t g = blockIdx.x + (first + my_i) * B;
            uint32_t nw = 0u;
            const bool sound = s.ok[my_w] && check_dir(a, g, s.total_words[my_w], d0, d1, g + 1u < a.G ? d2 : s.total_words[my_w], &nw);
            const uint32_t cm = sound ? d0 : 0u;
            s.e_cm[tid] = cm; s.e_off[tid] = d1; s.e_nw[tid] = nw;
            if (ONE) s.gtot[tid] = cm & 0xFFFFFFu;
            else if (cm) { atomicAdd(&s.gtot[my_i], cm & 0xFFFFFFu); atomicAdd(&s.gtot[kDecThreads / 2 + my_i], nw); }
        }
        __syncthreads();
        TeamRule rule{};
        if constexpr (!ONE) {
            const uint32_t x = tid < (int)in_batch ? s.gtot[tid] : 0u;
            const uint32_t alike = (uint32_t)__syncthreads_count(x != 0u && 2u * x >= s.mean && x <= 2u * s.mean);
            const uintptr_t at = MODE == 2 ? reinterpret_cast<uintptr_t>(a.theta) | reinterpret_cast<uintptr_t>(a.m) | reinterpret_cast<uintptr_t>(a.v)
                                           : reinterpret_cast<uintptr_t>(a.dense);
            rule = team_rule(MODE, a.group_log2, owned, in_batch > 1u && 4u * alike >= 3u * in_batch, s.mean, (at & 15u) == 0u, W);
        }
        if (tid < (int)in_batch) {
            const uint32_t tot = s.gtot[tid];
            if (tot != 0u) {
                uint32_t list = 3u;
                if (ONE) { if (tot <= warp_max(owned) && a.group_log2 <= 16u) list = 0u; }
                else list = team_for(rule, a.group_log2, tot, s.gtot[kDecThreads / 2 + tid]);
                if (list < 3u) team_list_entry(s, list, atomicAdd(&s.n_light[list], 1u)) = (uint16_t)tid;
                else s.heavy[atomicAdd(&s.n_heavy, 1u)] = (uint16_t)tid;
            }
        }
        __syncthreads();
        // Groups for whole blocks: the block's own; where only some groups are large (layers of different scales) a block that
        // found several of them hands up to three to a queue shared by all blocks, where the blocks that found none take them
        // (four streams of 25.6 M entries: the unluckiest block had five, 35 us against 16 for the median one).
        // With one group per block there is nothing to share, and the queue is left alone.
        const uint32_t n_heavy = s.n_heavy;
        const uint32_t keep = n_heavy == in_batch ? n_heavy : (n_heavy <= 4u ? min(n_heavy, 1u) : n_heavy - 3u);
        if (tid >= (int)keep && tid < (int)n_heavy) {
            const uint32_t slot = atomicAdd(q_reserved, 1u);
            __threadfence();
            *reinterpret_cast<volatile unsigned int*>(a.q_list + slot) = blockIdx.x + (first + s.heavy[tid]) * B + 1u;
        }
        if (queue && first + per_batch >= owned) {        // nothing more comes from this block
            if (keep < n_heavy) __syncthreads();
            if (tid == 0) { __threadfence(); atomicAdd(q_done, 1u); }
        }
        for (uint32_t h = 0; h < keep; ++h) {
            const uint32_t i = s.heavy[h];
            if (tid < (int)W) {
                const uint32_t e = i * W + (uint32_t)tid, cm = s.e_cm[e];
                s.g_count[tid] = cm & 0xFFFFFFu; s.g_M[tid] = cm >> 24; s.g_off[tid] = s.e_off[e]; s.g_nwords[tid] = s.e_nw[e];
            }
            __syncthreads();
            if (MODE != 3 && a.group_log2 > 14u) block_wide<ONE, MODE>(a, s, W, blockIdx.x + (first + i) * B);
            else block_group<ONE, MODE>(a, s, W, blockIdx.x + (first + i) * B, tile_parity, tid, lane, warp);
        }
        if (keep > 0u) {                                  // (the tile becomes the warps' memory)
            if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncthreads();
        }
        // ---- groups for teams of warps
        if constexpr (ONE) {
            const uint32_t n_light = s.n_light[0];
            for (;;) {
                uint32_t x = 0u;
                if (lane == 0) x = atomicAdd(&s.next_light[0], 1u);
                x = __shfl_sync(kFullMask, x, 0);
                if (x >= n_light) break;
                const uint32_t i = s.light[x];
                warp_group<MODE>(a, s, blockIdx.x + (first + i) * B, i, two_in_flight(owned, a.n), lane, warp);
            }
        } else {
            // (The update in one launch takes the single warps' first: the compiler then spills less; four streams of 25.6 M entries 51.4 us, so 50.4, of
            // 5 M 16.8 and 16.4.  The others are quicker with the long ones in front: packed 216 us, else 220.)
            if constexpr (MODE == 2) {
                team_groups<MODE, 1>(a, s, W, first, lane, warp);
                if (s.n_light[2]) { __syncthreads(); team_groups<MODE, 4>(a, s, W, first, lane, warp); }
            } else {
                if (s.n_light[2]) { team_groups<MODE, 4>(a, s, W, first, lane, warp, MODE == 0 && owned <= kFewGroups); __syncthreads(); }
                if (s.n_light[1]) { team_groups<MODE, 2>(a, s, W, first, lane, warp); __syncthreads(); }
                team_groups<MODE, 1>(a, s, W, first, lane, warp);
            }
        }
    }

    // ---- the queue: slots are filled as the groups are found; a taker waits (bounded) for its slot, or leaves once every
    //      block has pushed what it had and the slot lies beyond the last reservation.
    while (queue) {
        __syncthreads();
        if (tid == 0) {
            uint32_t got = 0xFFFFFFFFu;
            const uint32_t done = *reinterpret_cast<volatile unsigned int*>(q_done), taken = *reinterpret_cast<volatile unsigned int*>(q_taken),
                           reserved = *reinterpret_cast<volatile unsigned int*>(q_reserved);
            if (done < gridDim.x || taken < reserved) {
                const uint32_t i = atomicAdd(q_taken, 1u);
                uint32_t spin = 0;
                for (;;) {
                    if (i < a.G) {
                        const uint32_t e = *reinterpret_cast<volatile unsigned int*>(a.q_list + i);
                        if (e != 0u) { got = e - 1u; *reinterpret_cast<volatile unsigned int*>(a.q_list + i) = 0u; break; }
                    }
                    if (*reinterpret_cast<volatile unsigned int*>(q_done) >= gridDim.x &&
                        i >= *reinterpret_cast<volatile unsigned int*>(q_reserved)) break;      // nothing will fill it
                    if (i >= a.G) break;
                    if (++spin > a.spin_limit) {         // reserved and never filled in time: the group it stands for is lost
                        dec_fail(a, 0u, 0u, kStTimeout);
                        break;
                    }
                    __nanosleep(100);
                }
            }
            s.got = got;
        }
        __syncthreads();
        const uint32_t g = s.got;
        if (g == 0xFFFFFFFFu) break;
        if (tid < (int)W) {
            uint32_t cm = 0u, nw = 0u, o = 0u;
            if (s.ok[tid]) {
                const uint32_t* e = reinterpret_cast<const uint32_t*>(a.stream[tid]) + (kHeaderBytes >> 2) + 2u * g;
                cm = e[0]; o = e[1];
                if (!check_dir(a, g, s.total_words[tid], cm, o, g + 1u < a.G ? e[3] : s.total_words[tid], &nw)) { cm = 0u; nw = 0u; }
            }
            s.g_count[tid] = cm & 0xFFFFFFu; s.g_M[tid] = cm >> 24; s.g_off[tid] = o; s.g_nwords[tid] = nw;
        }
        __syncthreads();
        if (MODE != 3 && a.group_log2 > 14u) block_wide<ONE, MODE>(a, s, W, g);
        else block_group<ONE, MODE>(a, s, W, g, tile_parity, tid, lane, warp);
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");        // write-backs complete before the block leaves
    // the last block to leave clears the counters for the next launch.  The slots were cleared as they were taken; a
    // slot whose taker gave up (status TIMEOUT) was filled afterwards with nobody to take it: cleared here, so that
    // the queue is back in its resting state whatever happened.
    if (queue && tid == 0) {
        if (atomicAdd(q_exited, 1u) == gridDim.x - 1u) {
            const uint32_t reserved = *reinterpret_cast<volatile unsigned int*>(q_reserved);
            if (reserved != 0u && *reinterpret_cast<volatile unsigned long long*>(a.status) != ~0ull)
                for (uint32_t i = 0; i < reserved && i < a.G; ++i) a.q_list[i] = 0u;
            *q_taken = 0u; *q_done = 0u; *q_reserved = 0u;
            *q_exited = 0u;
        }
    }
}

}  // namespace fsg
