// Shared definitions of the CUDA side: stream constants, the workspace layout and small
// device helpers.  sm_100a only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fsg {

constexpr uint32_t kMagic       = 0x31475346u;   // "FSG1"
constexpr uint32_t kVersion     = 1u;
constexpr uint32_t kHeaderBytes = 64u;
constexpr int      kMaxTau      = 128;

// The sum tree is cut into aligned chunks of 2^14 entries: one fp64 partial per chunk.
constexpr int      kChunkLog2   = 14;
constexpr uint32_t kChunk       = 1u << kChunkLog2;

constexpr int kStOk = 0, kStNonfinite = 1, kStCapacity = 2, kStTimeout = 3;
constexpr int kStBadMagic = 16, kStBadVersion = 17, kStBadStatus = 18, kStNMismatch = 19,
              kStParamMismatch = 20, kStTruncated = 21, kStBadDirectory = 22, kStBadKey = 23,
              kStBadCode = 24;

// b^k, k = 0..tau, by the recurrence P_k = P_{k-1} * b in fp64 (a function of the
// parameters alone; passed to the kernels by value).
struct PowTable {
    double P[kMaxTau + 1];
};

// Control block at the start of the workspace.
struct Control {
    unsigned int       done;           // blocks of the sum kernel that have finished (self-resetting)
    unsigned int       pad0;
    unsigned int       error;          // encode: non-zero once a bounded wait ran out
    unsigned int       pad1;
    unsigned long long decode_status;  // min over failures of (group << 32 | key index << 8 | status)
    double             sum;            // S
    unsigned int       bar_gen;        // launches of the kernels whose blocks wait for one another that have finished
    unsigned int       exit_count;     // blocks of the running one that have finished (self-resetting)
    unsigned int       dq[6];          // decoder work queue: -, taken, done, exited, reserved (zero between launches)
    unsigned int       pad2[24];
    unsigned int       bar_count[8];   // k_resident: tiles of each gradient that have been summed; [0] k_scan: blocks that have finished; list encoder: arrivals at its grid barrier (zero between launches)
    unsigned int       pad3[8];
    unsigned int       ne_count[8];    // tiles of each gradient that the last encoder launch read a second time
};
static_assert(sizeof(Control) == 256, "control block is 256 bytes");

constexpr uint64_t kEncStateOffset = 1024;   // EncState (encode.cuh)
constexpr uint64_t kQueueOffset    = 32768;  // u32 queue[2^17]: decoder's grid-wide queue of groups (zero between launches)
constexpr uint64_t kQueueBytes     = 4ull << 17;
constexpr uint64_t kKvPartialsOffset = kQueueOffset + kQueueBytes;   // double [2^17]: chunk nodes of the key-value encoder's sum (zero between launches)
constexpr uint64_t kKvPartialsBytes  = 8ull << 17;
constexpr uint64_t kPartialsOffset = kKvPartialsOffset + kKvPartialsBytes;     // from here on the layout depends on n (api.cu)

__host__ __device__ inline uint64_t ceil_div_u64(uint64_t a, uint64_t b) { return (a + b - 1) / b; }

// Programmatic dependent launch: the next kernel of the stream may be brought onto the GPU from here on (it waits below before it
// touches memory) ...
__device__ __forceinline__ void allow_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// ... and: everything the kernels before this one in the stream have written is there.  What they may have written (gradients, streams,
// the workspace) is not read-only for the lifetime of such a kernel, which began before: never __ldg or __restrict__ for it.
__device__ __forceinline__ void wait_for_previous_kernels() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t bswap32(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

}  // namespace fsg
