// Device helpers shared by the encoders and the decoder: bulk copies, memory-ordering accesses, the final reduction of the sum
// tree, the flag rule and the table search.  sm_100a only.
#pragma once

#include "common.cuh"
#include "sum.cuh"
#include "bits.cuh"

namespace fsg {

constexpr int      kBlockThreads = 512;                       // the block size the block-wide helpers below are written for
constexpr int      kBlockWarps   = kBlockThreads / 32;
constexpr uint32_t kWaitLimit    = 1u << 22;                  // polls before a wait on another block gives up

// ---- mbarrier / bulk-copy primitives (sm_90+ PTX) -------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait: the hardware suspends the thread for up to about the hinted time per try, so a
// wait costs a handful of instructions; false when every try ran out.
constexpr uint32_t kTryHintNs = 10000u;
constexpr uint32_t kTryLimit  = 1u << 18;
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity, uint32_t tries = kTryLimit) {
    const uint32_t addr = smem_u32(bar);
    for (uint32_t t = 0; t < tries; ++t) {
        uint32_t ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(ok) : "r"(addr), "r"(parity), "r"(kTryHintNs) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src_global, uint32_t bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst_smem)), "l"(__cvta_generic_to_global(src_global)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Words that carry their whole payload: relaxed accesses are enough.
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// a pair of words that travels as one
__device__ __forceinline__ void ld_relaxed_pair(const unsigned long long* p, unsigned long long& lo, unsigned long long& hi) {
    asm volatile("{\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%2];\n mov.b128 {%0, %1}, q;\n}" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_relaxed_pair(unsigned long long* p, unsigned long long lo, unsigned long long hi) {
    asm volatile("{\n .reg .b128 q;\n mov.b128 q, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], q;\n}" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}

__device__ __forceinline__ void st_release_u32(unsigned int* p, unsigned int v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// counter increment that publishes this thread's earlier writes and, for whoever comes last, makes the others' visible
__device__ __forceinline__ unsigned int atom_add_acq_rel_u32(unsigned int* p, unsigned int v) {
    unsigned int old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
// The node of the block's values on the tree (positions: lanes, then warps), in every thread.
__device__ __forceinline__ double block_tree(double x, double* s_tree, int lane, int warp) {
    x = warp_tree(x);
    __syncthreads();                                   // s_tree may still be read from the last use
    if (lane == 0) s_tree[warp] = x;
    __syncthreads();
    double t = lane < kBlockWarps ? s_tree[lane] : 0.0;
    t = warp_tree(t, kBlockWarps);                       // lanes 0..15 of every warp hold the root
    return __shfl_sync(kFullMask, t, 0);
}

// Tree reduction of up to 2^17 partials by one block, 512 to a node: a warp forms a node by itself (16 partials per lane, all in flight
// at once, consecutive across the warp), the block the rest.  (A run of 8 per thread instead, 64 bytes apart across a warp: 5 us
// slower with all blocks at it.)
__device__ __forceinline__ double reduce_partials(const double* partials, uint32_t chunks, double* s_tree,
                                                  double* s_nodes, int tid, int lane, int warp) {
    const uint32_t passes = (chunks + kBlockThreads - 1) / kBlockThreads;       // <= 256 for n < 2^31
    if (passes <= 1u) return block_tree((uint32_t)tid < chunks ? __ldcg(partials + tid) : 0.0, s_tree, lane, warp);
    for (uint32_t p = (uint32_t)warp; p < passes; p += kBlockWarps) {
        double x[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const uint64_t idx = (uint64_t)p * kBlockThreads + 32u * (uint32_t)j + (uint32_t)lane;
            x[j] = idx < chunks ? __ldcg(partials + idx) : 0.0;
        }
        const double node = warp_rows16_tree(x, lane);
        if (lane == 0) s_nodes[p] = node;
    }
    __syncthreads();
    // the nodes of the passes, zero-padded to 512 positions, reduced on the same tree
    const double y = (uint32_t)tid < passes ? s_nodes[tid] : 0.0;
    return block_tree(y, s_tree, lane, warp);
}

// ceil(2^16 / M) for M = 1..20
__device__ __constant__ uint32_t c_inv_m[21] = {0, 65536, 32768, 21846, 16384, 13108, 10923, 9363, 8192, 7282, 6554, 5958,
                                                5462, 5042, 4682, 4370, 4096, 3856, 3641, 3450, 3277};

// flag of a delta with bit length bl: least f with ceil((f+1) M / 2^l) >= bl, which is
// floor((bl-1) 2^l / M) for bl >= 1; the division is a multiplication by ceil(2^16 / M)
__device__ __forceinline__ uint32_t flag_of(uint32_t delta, uint32_t l, uint32_t inv_m) {
    const uint32_t bl = delta ? 32u - __clz(delta) : 0u;
    return bl ? ((((bl - 1u) << l) * inv_m) >> 16) : 0u;
}

// L = least k in [0, tau] with |v| >= B_k (Eq. 2-3 as a table search; holds for k = tau), raised
// to 1, and the sign: the code byte.  The search starts from an estimate of log_b(S / |v|)
// (thr[130] = log2 S, thr[131] = 1 / log2 b, both approximate) and walks the non-increasing
// table from there, so the result does not depend on how good the estimate is.
// (The estimate is off by one a few times in a million; the two hints are kept in registers.)
struct CodeTable {
    const float* thr; int tau; float h0, h1;
    __device__ __forceinline__ CodeTable(const float* thr_, uint32_t tau_) : thr(thr_), tau((int)tau_), h0(thr_[130] * thr_[131]), h1(-thr_[131]) {}
};
__device__ __forceinline__ uint32_t code_byte_of(const CodeTable& t, float val) {
    const float av = fabsf(val);
    float lg;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(av));
    uint32_t L = (uint32_t)max(1, min(t.tau, __float2int_rd(fmaf(lg, t.h1, t.h0)) + 1));
    const float* thr = t.thr;
    if (av >= thr[L - 1u] || av < thr[L]) {
        while (L > 0u && av >= thr[L - 1u]) --L;
        while (L < (uint32_t)t.tau && av < thr[L]) ++L;
        L = L < 1u ? 1u : L;
    }
    return ((__float_as_uint(val) >> 24) & 0x80u) | (L - 1u);
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

}  // namespace fsg
