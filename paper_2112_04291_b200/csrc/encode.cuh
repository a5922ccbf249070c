// The encoder for dense gradients: Algorithm 1 and, per group of 2^14 entries (a tile), Algorithm 2, for up to eight
// gradients of the same length.
//
// k_resident: gradients that fit the GPU's shared memory, a tile per block (up to two blocks per SM).  Every entry is read
// from memory once; the blocks exchange their tiles' sums and, later, sizes through tagged words of the workspace, everyone
// reading what it needs; one launch.
#pragma once

#include "common.cuh"
#include "sum.cuh"
#include "bits.cuh"
#include "compress.cuh"     // copy and ordering primitives, table search, flag rule

namespace fsg {

constexpr int      kEncThreads   = 512;
constexpr int      kEncWarps     = kEncThreads / 32;
constexpr uint32_t kSlab         = kTile / kEncWarps;          // entries a warp takes at a time
static_assert(kSlab == 1024u, "eight rows of 128 entries per slab");
constexpr int      kEncMaxJobs   = 8;                          // gradients (simulated workers) one launch can take
constexpr uint32_t kMaxResident  = 320;                        // tiles k_resident can take (its exchange words in the workspace)

// Encoder state in the workspace's fixed part (the exchange words are told apart by their tags).
struct EncState {
    alignas(16) unsigned long long res_node[2 * kMaxResident]; // k_resident: a tile's node, tag
    unsigned long long res_size[kMaxResident];                 // tag << 32 | kept entries << 16 | words
};
static_assert(kEncStateOffset + sizeof(EncState) <= kQueueOffset, "fits before the decoder's queue");

struct EncArgs {
    const float*        grad[kEncMaxJobs];
    uint8_t*            out[kEncMaxJobs];
    uint64_t            out_bytes;
    uint64_t            n;
    Control*            ctl;
    EncState*           st;
    double              base;
    uint32_t            J, G;
    uint32_t            tau, l;
    uint32_t            wait_limit, try_limit;      // polls before a wait on another block, tries before a wait on a bulk copy gives up
};

// a pair of words that travels as one
__device__ __forceinline__ void ld_relaxed_pair(const unsigned long long* p, unsigned long long& lo, unsigned long long& hi) {
    asm volatile("{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_relaxed_pair(unsigned long long* p, unsigned long long lo, unsigned long long hi) {
    asm volatile("{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}

// log2 S and 1 / log2 b only steer the table search (its result does not depend on them): single precision, and the exponent of
// S taken from its bits so that sums beyond the fp32 range still give a finite estimate.  hints: thr + 130.
__device__ __forceinline__ void table_hints(double S, double base, float* hints) {
    const unsigned long long sb = (unsigned long long)__double_as_longlong(S);
    const int ex = (int)((sb >> 52) & 0x7FFull) - 1023;
    const float mant = __uint_as_float(0x3F800000u | (uint32_t)((sb >> 29) & 0x7FFFFFull));      // [1, 2)
    hints[0] = (float)ex + __log2f(mant);
    hints[1] = 1.0f / __log2f((float)base);
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
struct TeamScratch { uint32_t cnt[kEncWarps], first[kEncWarps], last[kEncWarps], maxd[kEncWarps], bits[kEncWarps], word; };

template <int W> __device__ __forceinline__ void team_sync(int id) {
    if constexpr (W == 1) __syncwarp();
    else if constexpr (W == 4) asm volatile("bar.sync %0, 128;" ::"r"(id + 1) : "memory");
    else __syncthreads();
}

__device__ __forceinline__ void put_code(uint32_t* blob, uint32_t q, uint32_t code) { reinterpret_cast<uint8_t*>(blob)[q ^ 3u] = (uint8_t)code; }

// M from the threads' largest deltas; a barrier of the team (keys and codes are complete behind it)
template <int W>
__device__ __forceinline__ uint32_t team_width(uint32_t maxd, TeamScratch& s, int w, int lane, int id) {
    maxd = __reduce_max_sync(kFullMask, maxd);
    if (W > 1 && lane == 0) s.maxd[w] = maxd;
    team_sync<W>(id);
    if (W > 1) maxd = __reduce_max_sync(kFullMask, lane < W ? s.maxd[lane] : 0u);
    return maxd ? 32u - (uint32_t)__clz((int)maxd) : 1u;
}

// Packs flags and deltas of count > 0 entries (all written before a barrier of the team); sized(words) is called by every thread as
// soon as the size is known.  The blob is complete when the call returns.
template <int W, typename F>
__device__ __forceinline__ void team_pack(uint32_t l, const uint16_t* keys, uint32_t* blob, uint32_t count, uint32_t M, TeamScratch& s,
                                          int w, int lane, int id, F sized) {
    const uint32_t inv_m = c_inv_m[M], up = (1u << l) - 1u;
    // zeroes behind the codes
    if (w == 0 && lane == 0 && (count & 3u)) blob[count >> 2] &= 0xFFFFFFFFu << (32u - 8u * (count & 3u));
    const uint32_t bound = (count * (8u + l + M) + 31u) >> 5;
    for (uint32_t i = ((count + 3u) >> 2) + (uint32_t)(w * 32 + lane); i <= bound; i += 32u * W) blob[i] = 0u;
    auto delta_of = [&](uint32_t q) -> uint32_t { return (uint32_t)keys[q] - (q ? (uint32_t)keys[q - 1u] : 0u); };
    const uint32_t nb = (count + 31u) >> 5, b0 = nb * (uint32_t)w / W, b1 = nb * (uint32_t)(w + 1) / W;
    const uint32_t delta0 = (8u + l) * count;
    uint32_t dpos = delta0;
    if (W > 1) {
        uint32_t bits = 0u;
        for (uint32_t q = 32u * b0 + (uint32_t)lane; q < min(count, 32u * b1); q += 32u) bits += ((flag_of(delta_of(q), l, inv_m) + 1u) * M + up) >> l;
        bits = __reduce_add_sync(kFullMask, bits);
        if (lane == 0) s.bits[w] = bits;
        team_sync<W>(id);
        const uint32_t x = lane < W ? s.bits[lane] : 0u, xi = warp_incl_scan(x, lane);
        dpos += __shfl_sync(kFullMask, xi - x, w);
        sized((delta0 + __shfl_sync(kFullMask, xi, 31) + 31u) >> 5);
    } else {
        __syncwarp();
    }
    // deltas: a field per lane
    for (uint32_t b = b0; b < b1; ++b) {
        const uint32_t q = 32u * b + (uint32_t)lane;
        uint32_t d = 0u, wd = 0u;
        if (q < count) { d = delta_of(q); wd = ((flag_of(d, l, inv_m) + 1u) * M + up) >> l; }
        const uint32_t wi = warp_incl_scan(wd, lane), pos = dpos + wi - wd, end = (pos & 31u) + wd;
        if (q < count) {                                                // (wd is 1 to 20)
            if (end <= 32u) atomicOr(&blob[pos >> 5], d << (32u - end));
            else { atomicOr(&blob[pos >> 5], d >> (end - 32u)); atomicOr(&blob[(pos >> 5) + 1u], d << (64u - end)); }
        }
        dpos += __shfl_sync(kFullMask, wi, 31);
    }
    // flags: a word per lane, from the deltas of the entries whose flags lie in it
    const uint32_t f0 = 8u * count, f1 = delta0;
    for (uint32_t i = (f0 >> 5) + (uint32_t)(w * 32 + lane); i <= (f1 - 1u) >> 5; i += 32u * W) {
        const uint32_t lo = max(32u * i, f0) - f0, q0 = lo / l, q1 = min(count, (32u * i + 32u - f0 + l - 1u) / l);
        uint32_t word = 0u, prev = q0 ? (uint32_t)keys[q0 - 1u] : 0u;
        int sh = (int)(32u * i + 32u) - (int)(f0 + l * q0 + l);          // where the flag's last bit lies in the word
        for (uint32_t q = q0; q < q1; ++q, sh -= (int)l) {
            const uint32_t k = keys[q], f = flag_of(k - prev, l, inv_m);
            word |= sh >= 0 ? f << sh : f >> -sh;
            prev = k;
        }
        if (word) atomicOr(&blob[i], word);
    }
    if (W == 1) sized((dpos + 31u) >> 5);
    team_sync<W>(id);
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
    outw[14] = a.l | ((uint32_t)kGroupLog2 << 8);
    outw[15] = a.G;
}

// ---- k_resident ----------------------------------------------------------------------------------
struct ResShared {
    union alignas(128) {
        float    tile[kTile];
        uint32_t blob[kTile];            // 27 bits an entry at most; grows over the tile, whose values behind it are still needed
    };
    uint16_t key[kTile];
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
        for (uint32_t i = lane; i < kSlab; i += 32u) slab[i] = i < valid ? __ldg(a.grad[j] + slab0 + i) : 0.0f;
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
    uint32_t maxd = 0u;
    for (uint32_t q0 = 0; q0 < count; q0 += kEncThreads) {
        const uint32_t q = q0 + (uint32_t)tid;
        uint32_t code = 0u;
        if (q < count) {
            const uint32_t k = s.key[q];
            maxd = max(maxd, k - (q ? (uint32_t)s.key[q - 1u] : 0u));
            code = code_byte_of(s.thr, a.tau, s.tile[k]);
        }
        __syncthreads();
        if (q < count) put_code(s.blob, q, code);
    }
    uint32_t words = 0u, M = 0u;
    auto publish = [&](uint32_t w) {
        words = w;
        if (tid == 0) st_relaxed_u64(a.st->res_size + t, ((unsigned long long)gen << 32) | (count << 16) | w);
    };
    if (count) {
        M = team_width<kEncWarps>(maxd, s.team, warp, lane, 0);
        team_pack<kEncWarps>(a.l, s.key, s.blob, count, M, s.team, warp, lane, 0, publish);
    } else {
        publish(0u);
    }
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

}  // namespace fsg
