// Launcher of the stand-alone selection (afx_seltok.cuh).
#include "afx_launch.cuh"
#include "afx_seltok.cuh"

namespace afx {

template <int DT, int NW, int CH, int IN>
__global__ void __launch_bounds__(kStThreads, 1) select_tokens_kernel(FusedArgs a) {
    __shared__ SelTokSmem sm;
    select_tokens_block<DT, NW, CH, IN>(a, &sm);
}

template <int DT, int IN>
static afx_status launch_select_tokens_dt(const FusedArgs& a, cudaStream_t st) {
    auto go = [&](auto kern) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(a.T, 1, 1);
        cfg.blockDim = dim3(kStThreads, 1, 1);
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = a.T;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = a.T > 1 ? 2 : 1;
        return cudaLaunchKernelEx(&cfg, kern, a) == cudaSuccess ? AFX_OK : AFX_ERR_CUDA;
    };
    // as few selecting warps as leave a lane enough registers (see afx_topk.cuh)
    if (a.K <= 4096) return go(select_tokens_kernel<DT, 8, 4, IN>);
    if (a.K <= 8192) return go(select_tokens_kernel<DT, 16, 4, IN>);
    if (a.K <= 16384) return go(select_tokens_kernel<DT, 16, 8, IN>);
    if (a.K <= kSelectFastMaxK) return go(select_tokens_kernel<DT, 32, 8, IN>);
    return AFX_ERR_CAPACITY;
}

afx_status launch_select_tokens(int dtype, bool norm, const FusedArgs& a, cudaStream_t st) {
    if (dtype == AFX_F16)
        return norm ? launch_select_tokens_dt<AFX_F16, IN_NORM>(a, st) : launch_select_tokens_dt<AFX_F16, IN_X>(a, st);
    return norm ? launch_select_tokens_dt<AFX_BF16, IN_NORM>(a, st) : launch_select_tokens_dt<AFX_BF16, IN_X>(a, st);
}

}  // namespace afx
