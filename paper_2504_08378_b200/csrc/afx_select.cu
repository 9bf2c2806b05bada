// afx_select_active / afx_diff_active: stand-alone selection and cross-layer set difference.
#include "afx_launch.cuh"
#include "afx_fused.cuh"
#include "afx_select.cuh"

namespace afx {

constexpr int kSelectThreads = 1024;

// Dynamic shared memory of the kernel for K > kSelectFastMaxK: flag words.
static size_t select_dyn_smem(int K) { return (static_cast<size_t>((K + 31) >> 5) * 4 + 15) / 16 * 16; }

template <int DT>
__global__ void __launch_bounds__(kSelectThreads, 1)
select_kernel(const uint16_t* __restrict__ x, int K, int T, int mode, int k, float tau,
              int32_t* __restrict__ idx, int32_t* __restrict__ count, uint32_t* __restrict__ bitmap) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ SelectScratch scratch;
    const int nwords = (K + 31) >> 5;
    uint32_t* s_flags = reinterpret_cast<uint32_t*>(s_dyn);
    const int lane = lane_id();
    int w0, w1;
    warp_word_range(nwords, w0, w1);
    int mine = 0;
    block_select_flags_large<DT>(x, K, T, mode, k, tau, s_flags, &scratch);
    for (int w = w0 + lane; w < w1; w += 32) mine += __popc(s_flags[w]);
    mine = warp_sum(mine);
    int total;
    int base = warp_prefix(mine, scratch.wtot[1], total);
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (int w = w0; w < w1; ++w) {
        const uint32_t bits = s_flags[w];
        if ((bits >> lane) & 1u) idx[base + __popc(bits & lt_mask)] = (w << 5) + lane;
        base += __popc(bits);
    }
    if (threadIdx.x == 0) *count = total;
    if (bitmap != nullptr)
        for (int w = w0 + lane; w < w1; w += 32) bitmap[w] = s_flags[w];
}

// miss = A \ P (ascending), hit = |A & P|.  One block; in passes of 8192 entries each warp owns a contiguous run of
// list positions so that the output keeps A's order.  An entry outside [0, K) is neither a
// hit nor a miss; the status word reports it.
//
// What bounds it is latency: of the dependency wait, the count, the list and P, one behind the other.  All entries of a
// pass are on their way together and stay in registers until they are written; P is in shared memory by then, where it
// fits.  A warp that took its chunks one after the other, twice, needed two loads in a row for each (selection,
// difference of 4096 entries and list operator 8192 -> 57344: 89.3 us, now 87.7).  A short list is done in a pass with
// room for one chunk per warp, or four: the instructions of eight cost more than the loads.  us in a graph, one
// after the other, with eight always, and now: 51 of 512 entries 2.1, 2.7, 1.7; 2048 of 4096 2.8, 3.0, 2.1; 7372 of 8192
// 5.6, 3.4, 3.1; 100000 of 200000 60.0, 28.7, 25.8.
constexpr int kDiffChunks = 8;                     // chunks of 32 entries per warp and pass
constexpr int kDiffWords = kSelectFastMaxK / 32;   // words of P in shared memory

struct DiffArgs {
    const int32_t* idxA;
    const uint32_t* bitmapP;
    int32_t* miss;
    int K, n;
};
// The chunks c_lo .. of the list, `per` <= CH of them per warp: writes their misses from position n_miss on; the number
// of misses, and of entries out of range above bit 16.  Every thread calls it; a block barrier is part of it.
template <int CH, bool STAGED>
__device__ __forceinline__ int diff_pass(const DiffArgs& a, int c_lo, int per, const uint32_t* words, bool first, int* scan, int n_miss) {
    const int lane = lane_id();
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int p0 = ((c_lo + warp_id() * per) << 5) + lane;  // (a position beyond the run of another warp is beyond n as well)
    int j[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) j[c] = c < per && p0 + 32 * c < a.n ? __ldg(a.idxA + p0 + 32 * c) : 0;
    if (first) __syncthreads();  // P is in place
    uint32_t m[CH];
    int mine = 0;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        const bool here = c < per && p0 + 32 * c < a.n, ok = static_cast<unsigned>(j[c]) < static_cast<unsigned>(a.K);
        uint32_t w = 0xFFFFFFFFu;
        if (here && ok) w = STAGED ? words[j[c] >> 5] : __ldg(a.bitmapP + (j[c] >> 5));
        m[c] = __ballot_sync(0xFFFFFFFFu, here && ok && ((w >> (j[c] & 31)) & 1u) == 0u);
        mine += __popc(m[c]) + (__popc(__ballot_sync(0xFFFFFFFFu, here && !ok)) << 16);
    }
    int total;
    int at = n_miss + (warp_prefix(mine, scan, total) & 0xFFFF);
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        if ((m[c] >> lane) & 1u) a.miss[at + __popc(m[c] & lt_mask)] = j[c];
        at += __popc(m[c]);
    }
    return total;
}

__global__ void __launch_bounds__(kSelectThreads, 1)
diff_kernel(DiffArgs a, const int32_t* __restrict__ cntA, int32_t* __restrict__ miss_count, int32_t* __restrict__ hit_count,
            int32_t* __restrict__ status) {
    __shared__ int scan[2][33];
    __shared__ uint32_t words[kDiffWords];
    constexpr int kWarps = kSelectThreads / 32;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (ordering rule of the library)
    const bool staged = a.K <= kSelectFastMaxK;
    int n = *cntA;
    if (staged)
        for (int w = threadIdx.x; w < (a.K + 31) / 32; w += kSelectThreads) words[w] = a.bitmapP[w];
    if (n < 0 || n > a.K) {
        if (threadIdx.x == 0) report_status(status, AFX_ERR_CAPACITY);
        n = max(0, min(n, a.K));
    }
    a.n = n;
    const int nchunks = (n + 31) >> 5;
    int n_miss = 0, n_bad = 0;
    for (int pass = 0, c_lo = 0; c_lo < nchunks; ++pass, c_lo += kWarps * kDiffChunks) {
        const int per = min(kDiffChunks, (nchunks - c_lo + kWarps - 1) / kWarps);
        int* const sc = scan[pass & 1];
        int total;
        if (!staged)
            total = diff_pass<kDiffChunks, false>(a, c_lo, per, words, false, sc, n_miss);
        else if (per == 1)
            total = diff_pass<1, true>(a, c_lo, per, words, pass == 0, sc, n_miss);
        else if (per <= 4)
            total = diff_pass<4, true>(a, c_lo, per, words, pass == 0, sc, n_miss);
        else
            total = diff_pass<kDiffChunks, true>(a, c_lo, per, words, pass == 0, sc, n_miss);
        n_miss += total & 0xFFFF;
        n_bad += total >> 16;
    }
    if (threadIdx.x == 0) {
        *miss_count = n_miss;
        *hit_count = n - n_miss - n_bad;
        if (n_bad > 0) report_status(status, AFX_ERR_INVALID_ARG);
    }
}

}  // namespace afx

extern "C" afx_status afx_select_active(const void* x, int dtype, int K, int T, int mode, int k,
                                        float tau, int32_t* idx, int32_t* count, uint32_t* bitmap,
                                        void* stream) {
    using namespace afx;
    if (x == nullptr || idx == nullptr || count == nullptr) return AFX_ERR_INVALID_ARG;
    if (K <= 0 || K > (1 << 20) || T < 1 || T > AFX_MAX_T) return AFX_ERR_INVALID_ARG;
    if (dtype != AFX_F16 && dtype != AFX_BF16) return AFX_ERR_UNSUPPORTED;
    if (mode != AFX_MODE_TOPK && mode != AFX_MODE_THRESHOLD) return AFX_ERR_UNSUPPORTED;
    if (mode == AFX_MODE_TOPK && (k < 0 || k > K)) return AFX_ERR_INVALID_ARG;
    if (mode == AFX_MODE_THRESHOLD && tau != tau) return AFX_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x) & 1u) || (reinterpret_cast<uintptr_t>(idx) & 3u) ||
        (reinterpret_cast<uintptr_t>(count) & 3u) || (reinterpret_cast<uintptr_t>(bitmap) & 3u))
        return AFX_ERR_ALIGNMENT;
    if (K <= kSelectFastMaxK) {
        FusedArgs a = {};
        a.K = K;
        a.T = T;
        a.x = static_cast<const uint16_t*>(x);
        a.mode = mode;
        a.k = k;
        a.tau = tau;
        a.idx_out = idx;
        a.count_out = count;
        a.bitmap_out = bitmap;
        return launch_select_tokens(dtype, false, a, static_cast<cudaStream_t>(stream));
    }
    const size_t smem = select_dyn_smem(K);
    auto kern = dtype == AFX_F16 ? select_kernel<AFX_F16> : select_kernel<AFX_BF16>;
    if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), smem)) {
        cudaGetLastError();
        return AFX_ERR_CUDA;
    }
    kern<<<1, kSelectThreads, smem, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint16_t*>(x), K, T, mode, k, tau, idx, count, bitmap);
    return launch_status();
}

extern "C" afx_status afx_diff_active(const int32_t* idxA, const int32_t* cntA,
                                      const uint32_t* bitmapP, int K, int32_t* miss,
                                      int32_t* miss_count, int32_t* hit_count, int32_t* dev_status,
                                      void* stream) {
    using namespace afx;
    if (idxA == nullptr || cntA == nullptr || bitmapP == nullptr || miss == nullptr ||
        miss_count == nullptr || hit_count == nullptr)
        return AFX_ERR_INVALID_ARG;
    if (K <= 0 || K > (1 << 20)) return AFX_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(idxA) & 3u) || (reinterpret_cast<uintptr_t>(cntA) & 3u) ||
        (reinterpret_cast<uintptr_t>(bitmapP) & 3u) || (reinterpret_cast<uintptr_t>(miss) & 3u) ||
        (reinterpret_cast<uintptr_t>(miss_count) & 3u) || (reinterpret_cast<uintptr_t>(hit_count) & 3u) ||
        (reinterpret_cast<uintptr_t>(dev_status) & 3u))
        return AFX_ERR_ALIGNMENT;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, 1, 1);
    cfg.blockDim = dim3(kSelectThreads, 1, 1);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, diff_kernel, DiffArgs{idxA, bitmapP, miss, K, 0}, cntA, miss_count, hit_count, dev_status) == cudaSuccess
               ? AFX_OK
               : AFX_ERR_CUDA;
}
