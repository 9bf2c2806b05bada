// afx_sparse_gemv: host-side shape selection and launch.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "afx_launch.cuh"
#include "afx_list.cuh"
#include "afx_mtlist.cuh"

namespace afx {

template <int DT, int PW>
__global__ void __launch_bounds__(kGemvThreads, 2) sparse_gemv_kernel(GemvListArgs a) {
    __shared__ ListSmem<1, 1024> sm;
    __shared__ GemvRecv<1> recv;
    gemv_list_block<DT, 1, PW, 1024>(a, &sm, &recv);
}

// A few tokens at once: the tensor-core kernel (afx_mtlist.cuh), two blocks per SM.
template <int DT>
__global__ void __launch_bounds__(kGemvThreads, 2) sparse_gemm_mt_kernel(GemvListArgs a) {
    extern __shared__ __align__(16) unsigned char ml_dyn[];
    mt_list_block<DT>(a, ml_dyn);
}

// Clusters of s blocks of the kernel above that are resident at once; its shared memory is never what bounds them.
// (Asked once per device and size: a call looks through all sizes.)
template <int DT>
static int ml_resident(int s) {
    static std::atomic<int> known[64][kMlMaxCluster + 1];  // + 1, 0: not asked yet
    const void* kern = reinterpret_cast<const void*>(sparse_gemm_mt_kernel<DT>);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = known[dev][s].load(std::memory_order_relaxed) - 1;
    if (n < 0) {
        if (s > kMaxCluster && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        n = max_active_clusters(kern, s, ml_dyn_smem(AFX_MAX_T, kMlMaxGranules, s));
        known[dev][s].store(n + 1, std::memory_order_relaxed);
    }
    return n;
}

// Granules g per tile and blocks s per cluster.  Of every cluster size that keeps all clusters resident at once, with room
// for two clusters and eight blocks more (the occupancy query counts what fits an empty GPU; behind another kernel
// clusters were seen to run as a second wave without it), the narrowest tile; of these the shape of least cost.  The cost
// is that of a block, in parts that were fitted to 207 calls of 1024 to 13824 channels on 1024 to 57344 outputs with two,
// four and eight tokens, each in 5 to 25 shapes: the entries that a warp multiplies (16 / g warps share a granule's
// list, so that three, five, six or seven granules leave warps idle), the entries that it stages, and the rows and peers
// that its sums meet.  It is within 1 % of the best resident shape in the mean and 18 % at worst; the fewest granules per
// block, the nearest to five blocks of equals, were within 4 % and 38 %.  By that rule and now, us: eight tokens
// 1024 -> 16384 14.3 and 11.6, 2048 -> 20480 25.2 and 19.9, 5120 -> 24576 43.0 and 40.9, 5120 -> 16384 31.0 and 29.3;
// four tokens 5120 -> 14336 27.1 and 26.5, 1024 -> 10240 9.9 and 8.8; two tokens 2048 -> 10240 11.4 and 10.4.
// Sizes above eight only where whole GPCs hold several of them, and not nine (28 of 30 clusters of nine ran as one wave or
// two from call to call).  No block with less than a step or so of the list per warp (1024 -> 1024, three tokens: 1 x 10
// 6.1; the rule's 1 x 5 5.0, 2048 -> 1024 with four tokens 5.6).
template <int DT>
static afx_status launch_gemm_mt(const GemvListArgs& a, cudaStream_t st) {
    constexpr int kSpare = 8, kMinEntries = 192;
    const int n = (a.N + kMlGranule - 1) / kMlGranule;
    int best_s = 1, best_g = kMlMaxGranules;
    float least = INFINITY;
    for (const int s : {1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 16}) {
        if (s > 1 && a.K < s * kMinEntries) break;
        const int resident = ml_resident<DT>(s), clusters = resident - std::max(2, (kSpare + s - 1) / s);
        if (clusters < 1) continue;
        const int g = (n + clusters - 1) / clusters;  // the narrowest tile that leaves no more clusters
        if (g > kMlMaxGranules) continue;
        const float T = static_cast<float>(a.T), warps = static_cast<float>(kGemvWarps / g);  // that share a granule's list
        const float cost = static_cast<float>(a.K) / s * (100.0f / warps + T) + T * (300.0f * g + 100.0f * s);
        if (cost >= least) continue;
        least = cost;
        best_s = s;
        best_g = g;
    }
    const int tiles = (n + best_g - 1) / best_g;
    if (tiles > 65535) return AFX_ERR_CAPACITY;
    return launch_clustered(sparse_gemm_mt_kernel<DT>, best_s, tiles, ml_dyn_smem(a.T, best_g, best_s), a, st);
}

int sm_count() {
    static int cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cached[dev] = n;
    }
    return cached[dev];
}

#ifdef AFX_EXPERIMENT
int g_force_pw = 0, g_force_s = 0;  // experiment knobs, 0 = automatic
int g_cluster_margin = -1;          // experiment knob, < 0 = automatic
#endif

template <int DT>
static afx_status launch_gemv(const GemvListArgs& a, cudaStream_t st) {
    if (a.T > 1) return launch_gemm_mt<DT>(a, st);
    const void* kerns[3] = {reinterpret_cast<const void*>(sparse_gemv_kernel<DT, 256>),
                            reinterpret_cast<const void*>(sparse_gemv_kernel<DT, 128>),
                            reinterpret_cast<const void*>(sparse_gemv_kernel<DT, 64>)};
    const GemvShapeChoice c = choose_gemv_shape(a.N, kerns, 0);
    switch (c.pw) {
        case 256: return launch_clustered(sparse_gemv_kernel<DT, 256>, c.S, c.tiles, 0, a, st);
        case 128: return launch_clustered(sparse_gemv_kernel<DT, 128>, c.S, c.tiles, 0, a, st);
        default: return launch_clustered(sparse_gemv_kernel<DT, 64>, c.S, c.tiles, 0, a, st);
    }
}

afx_status launch_list_gemv(int dtype, const GemvListArgs& a, cudaStream_t st) {
    return dtype == AFX_F16 ? launch_gemv<AFX_F16>(a, st) : launch_gemv<AFX_BF16>(a, st);
}

}  // namespace afx

#ifdef AFX_EXPERIMENT
// Experiment builds only (not part of the ABI): force tile width / cluster size / margin.
extern "C" void afx_internal_tune_gemv(int pw, int s) {
    afx::g_force_pw = pw;
    afx::g_force_s = s;
}
extern "C" void afx_internal_cluster_margin(int margin) { afx::g_cluster_margin = margin; }
#endif

extern "C" size_t afx_workspace_bytes(int K_max, int N_max, int T_max) {
    (void)K_max;
    (void)N_max;
    (void)T_max;
    return 0;  // partial sums meet in (distributed) shared memory: no entry point needs scratch
}

extern "C" afx_status afx_sparse_gemv(const void* Wt, int dtype, int K, int N, int64_t ldw,
                                      const void* x, int T, const int32_t* idx, const int32_t* count,
                                      const int32_t* slot, float* y, int accumulate, int32_t* dev_status,
                                      void* stream) {
    using namespace afx;
    if (Wt == nullptr || x == nullptr || idx == nullptr || count == nullptr || y == nullptr)
        return AFX_ERR_INVALID_ARG;
    if (K <= 0 || N <= 0 || T < 1 || T > AFX_MAX_T || ldw < N) return AFX_ERR_INVALID_ARG;
    if (dtype != AFX_F16 && dtype != AFX_BF16) return AFX_ERR_UNSUPPORTED;
    if ((N & 7) != 0 || (ldw & 7) != 0 || !aligned16(Wt) || !aligned16(y) ||
        (reinterpret_cast<uintptr_t>(x) & 1u) != 0 || (reinterpret_cast<uintptr_t>(idx) & 3u) != 0 ||
        (reinterpret_cast<uintptr_t>(count) & 3u) != 0 || (reinterpret_cast<uintptr_t>(slot) & 3u) != 0 ||
        (reinterpret_cast<uintptr_t>(dev_status) & 3u) != 0)
        return AFX_ERR_ALIGNMENT;
    if ((N + 63) / 64 > 65535) return AFX_ERR_CAPACITY;
    GemvListArgs a;
    a.Wt = static_cast<const uint16_t*>(Wt);
    a.ldw = ldw;
    a.K = K;
    a.N = N;
    a.T = T;
    a.x = static_cast<const uint16_t*>(x);
    a.idx = idx;
    a.count = count;
    a.slot = slot;
    a.accumulate = accumulate ? 1 : 0;
    a.silu = 0;
    a.ep.y = y;
    a.ep.out_bits = nullptr;
    a.ep.N = N;
    a.ep.scale = nullptr;
    a.status = dev_status;
    return launch_list_gemv(dtype, a, static_cast<cudaStream_t>(stream));
}
