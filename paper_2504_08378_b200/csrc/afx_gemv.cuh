// What the sparse operators share: block shape, staging area, cluster barrier, epilogue and list arguments.
#pragma once

#include <cooperative_groups.h>

#include "afx_common.cuh"

namespace afx {

namespace cg = cooperative_groups;

constexpr int kGemvWarps = 16;
constexpr int kGemvThreads = 32 * kGemvWarps;
constexpr int kMaxCluster = 8;

// Split cluster barrier.  Every block arrives once when it starts and waits just before its
// first store into a peer's shared memory: by then every block of the cluster is running.
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// How a finished sum leaves the kernel.
enum { EP_STORE = 0, EP_ACCUM = 1, EP_SILU = 2 };

struct EpilogueArgs {
    float* y;            // EP_STORE / EP_ACCUM: [T][N] fp32
    uint16_t* out_bits;  // EP_SILU: [T][N/2] 16-bit floats
    int N;               // outputs of the operator (columns of Wt)
    const float* scale;  // EP_STORE / EP_ACCUM: DEVICE factor applied to the finished sum (an
                         // expert's routing weight), or NULL for 1
};

// A staged list entry holds its row's offset from the start of the weights in 16-byte units, in 32 bits; the place inside
// the row is added in 64 bits, so that only the offset itself has to fit.  (An operator of K rows whose K * ldw / 8 is at
// most 2^32, 64 GB, has no row whose offset does not.)
constexpr uint32_t kSkippedEntry = 0xFFFFFFFFu;  // of an entry that takes no part
__device__ __forceinline__ bool row_offset_fits(uint64_t off) { return off < kSkippedEntry; }

struct GemvListArgs {
    const uint16_t* Wt;
    int64_t ldw;
    int K, N, T;
    const uint16_t* x;
    const int32_t* idx;
    const int32_t* count;
    const int32_t* slot;
    int accumulate;   // 0: y = sum, 1: y += sum
    int silu;         // 1: gate|up columns, out_bits = round(silu(gate) * up) instead of y
    EpilogueArgs ep;
    int32_t* status;  // device status word or NULL
};

// afx_sparse_gemv's launcher (afx_gemv.cu), also used by the layer step over host-resident weights.
afx_status launch_list_gemv(int dtype, const GemvListArgs& a, cudaStream_t st);

}  // namespace afx
