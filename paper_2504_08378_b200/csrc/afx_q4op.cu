// Launcher of the one-token operator over 4-bit rows (afx_q4op.cuh).
#include "afx_launch.cuh"
#include "afx_q4op.cuh"
#include "afx_slice.cuh"

namespace afx {

template <int DT, int NT, int NW, int CH, int W, int IN, int EP, bool SPLIT>
__global__ void __launch_bounds__(NT, W == 2 ? 1024 / NT : 1) q4_op_kernel(FusedArgs a) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ RegSelScratch s;
    __shared__ float recv[SPLIT ? NT + 2 * kQoSplit : 1];
    q4op_block<DT, NT, NW, CH, W, IN, EP, SPLIT>(a, dyn, &s, recv);
}

template <int DT, int NT, int NW, int CH, int W, int IN, int EP, bool SPLIT>
static afx_status launch_q4op(const FusedArgs& a, cudaStream_t st) {
    FusedArgs b = a;
    b.side_cluster = a.idx_out != nullptr || a.count_out != nullptr || a.bitmap_out != nullptr || a.xnorm_out != nullptr ||
                     a.bitmap_pred != nullptr || a.kth_slot != nullptr;
    size_t dyn = q4op_dyn_smem(NT, W, a.K, a.idx_in != nullptr);
    if (NT == 512 && dyn < kSlAlone) dyn = kSlAlone;
    auto kern = q4_op_kernel<DT, NT, NW, CH, W, IN, EP, SPLIT>;
    if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), dyn)) {
        cudaGetLastError();
        return AFX_ERR_CUDA;
    }
    // one tile per SM (split: per kQoSplit SMs), one SM left for the side outputs where there are any; more tiles, in
    // waves, only where one would exceed the widest a block can finish
    const int blocks = a.N / 32, sms = sm_count() > 0 ? sm_count() : 148;
    const int split = SPLIT ? kQoSplit : 1;
    int room = sms - b.side_cluster;
    if (SPLIT) {
        // All clusters that the occupancy query counts (32 on 148 SMs): one, two or three spare ones make the tiles wider
        // and a layer slower, 8192 channels 122.7 and 125.5 us, 4096 58.3 and 59.2, 2048 37.3 and 38.4.
        const int fit = max_active_clusters(reinterpret_cast<const void*>(kern), split, dyn, NT) - b.side_cluster;
        room = fit < 1 ? 1 : fit;
    }
    int per = (blocks + room - 1) / room;
    if (per > q4op_max_blocks(NT)) per = q4op_max_blocks(NT);
    b.slices = (blocks + per - 1) / per;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((b.slices + b.side_cluster) * split, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SPLIT ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, b) == cudaSuccess ? AFX_OK : AFX_ERR_CUDA;
}

// Rows of many channels on few outputs: clusters of four blocks share the list of a tile four times as wide, which costs
// a cluster barrier and touches a quarter of the rows.  A layer of 1000 to 2048 positions, half of the channels kept,
// down projection without and with: 5504 -> 2048 40.1 and 39.3 us, 11008 -> 4096 61.5 and 59.7, 13824 -> 5120 71.9 and
// 70.0; but 2816 -> 1024 33.0 and 34.8, and the o projections 4096 -> 4096 59.9 and 59.7, 5120 -> 5120 71.9 and 73.8.
constexpr int kQoSplitMinK = 4096;
// Blocks of 512 threads that hold 32 outputs per thread take more than half of the registers of an SM, and no block of the
// attention fits beside them; with 16 outputs per thread and 64 registers one does.  q | k | v at 4096 -> 12288: layer
// 61.9 and 59.9 us, 2048 -> 6144 40.6 and 40.3, 1024 -> 3072 33.2 and 33.1; above K = 4096 the registers are worth more
// (5120 -> 15360 72.0 and 72.8, 8192 -> 10240 117.4 and 119.3).  Away from the attention 16 outputs cost 1 to 3 us
// (4096 -> 22016 59.8 and 62.2).
constexpr int kQoBesideMaxK = 4096;

template <int DT, int IN, int EP>
static afx_status launch_q4op_dt(const FusedArgs& a, cudaStream_t st) {
    if (static_cast<uint64_t>(a.K) * static_cast<uint64_t>(a.ldw >> 3) > 0x100000000ull) return AFX_ERR_CAPACITY;
    if constexpr (IN == IN_X) {
        if (a.K >= kQoSplitMinK && a.K >= 2 * static_cast<int64_t>(a.N)) {
            if (a.K <= 16384) return launch_q4op<DT, 512, 16, 8, 4, IN, EP, true>(a, st);
            if (a.K <= 32768) return launch_q4op<DT, 1024, 32, 8, 2, IN, EP, true>(a, st);
            return AFX_ERR_CAPACITY;
        }
    }
    if constexpr (EP != EP_SILU) {
        if (a.beside_attention && a.K <= kQoBesideMaxK) return launch_q4op<DT, 512, 8, 4, 2, IN, EP, false>(a, st);
    }
    if (a.K <= 4096) return launch_q4op<DT, 512, 8, 4, 4, IN, EP, false>(a, st);
    if (a.K <= 16384) return launch_q4op<DT, 512, 16, 8, 4, IN, EP, false>(a, st);
    if (a.K <= 32768) return launch_q4op<DT, 1024, 32, 8, 2, IN, EP, false>(a, st);
    return AFX_ERR_CAPACITY;
}

template <int DT>
static afx_status launch_q4_operator_dt(int in, int ep, const FusedArgs& a, cudaStream_t st) {
    if (in == IN_NORM && ep == EP_STORE) return launch_q4op_dt<DT, IN_NORM, EP_STORE>(a, st);
    if (in == IN_NORM && ep == EP_SILU) return launch_q4op_dt<DT, IN_NORM, EP_SILU>(a, st);
    if (in == IN_X && ep == EP_ACCUM) return launch_q4op_dt<DT, IN_X, EP_ACCUM>(a, st);
    return AFX_ERR_UNSUPPORTED;
}

afx_status launch_q4_operator(int dtype, int in, int ep, const FusedArgs& a, cudaStream_t st) {
    return dtype == AFX_F16 ? launch_q4_operator_dt<AFX_F16>(in, ep, a, st) : launch_q4_operator_dt<AFX_BF16>(in, ep, a, st);
}

}  // namespace afx
