// Launcher of the decoding-step attention (afx_attn.cuh, afx_attn_mma.cuh).
#include "afx_attn_mma.cuh"
#include "afx_launch.cuh"

namespace afx {

// One query head per kv head: dot products on the fp32 pipe, U cache rows in flight per half warp.
template <int DT, int U>
__global__ void __launch_bounds__(kAttnThreads, U == 8 ? 2 : 3) attention_kernel(AttnArgs a) {
    __shared__ AttnSmem sm;
    attention_block<DT, U>(a, &sm);
}

template <int DT>
__global__ void __launch_bounds__(kAttnMmaThreads, 1) attention_mma_kernel(AttnArgs a) {
    extern __shared__ __align__(16) unsigned char dyn[];
    attention_mma_block<DT>(a, reinterpret_cast<AttnMmaSmem*>(dyn));
}

// The largest cluster of at most `most` blocks that keeps all `groups` clusters resident at once.
static int attn_mma_cluster(const void* kern, size_t dyn, int groups, int most) {
    if (most > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        most = 8;
    }
    for (int S = most; S > 1; --S)
        if (max_active_clusters(kern, S, dyn, kAttnMmaThreads) >= groups + (groups + 15) / 16) return S;
    return 1;
}

template <int DT>
static afx_status launch_attention_dt(const AttnArgs& a, cudaStream_t st) {
    const int groups = a.kv_heads * a.T;
    // Several query heads share a cache row: the tensor cores, whose work does not grow with them (kv 16,
    // rep 2, 2048 positions: 13.4 us on the fp32 pipe, 8.5 here; kv 8, rep 8, 8000 positions: 100 and 15.7).
    // One query head uses an eighth of their rows, and the fp32 pipe keeps up (kv 32, 2048 positions: 11.3
    // and 12.3 us; kv 40, four tokens: 47.1 and 52.6).
    const bool mma = a.q_heads > a.kv_heads;
    // one query head: split the cached positions so that kv_heads * T * S blocks fill the machine, S <= 8
    int S = (2 * sm_count() + groups - 1) / groups;
    S = S < 1 ? 1 : (S > 8 ? 8 : S);
    // Two blocks per SM with 8 cache rows of K and V in flight per half warp, where all of them are resident that
    // way; where some would stream alone in a second wave, three per SM with 4 rows (kv 40, four tokens, 2048
    // positions, 320 blocks: 45.8 and 32.5 us).
    const bool deep = groups * S <= 2 * sm_count();
    const void* kern = mma ? reinterpret_cast<const void*>(attention_mma_kernel<DT>)
                           : deep ? reinterpret_cast<const void*>(attention_kernel<DT, 8>)
                                  : reinterpret_cast<const void*>(attention_kernel<DT, 4>);
    size_t dyn = 0;
    if (mma) {
        // as many blocks as find a tile for every warp, at most what is resident in one wave
        const int useful = (a.pos + kAttnTile * kAttnMmaWarps - 1) / (kAttnTile * kAttnMmaWarps);
        dyn = sizeof(AttnMmaSmem);
        if (!ensure_dyn_smem(kern, dyn)) {
            cudaGetLastError();
            return AFX_ERR_CUDA;
        }
        S = attn_mma_cluster(kern, dyn, groups, useful < 1 ? 1 : useful > kAttnMaxCluster ? kAttnMaxCluster : useful);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, a.kv_heads, a.T);
    cfg.blockDim = dim3(mma ? kAttnMmaThreads : kAttnThreads, 1, 1);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = mma ? cudaLaunchKernelEx(&cfg, attention_mma_kernel<DT>, a)
                       : deep ? cudaLaunchKernelEx(&cfg, attention_kernel<DT, 8>, a)
                              : cudaLaunchKernelEx(&cfg, attention_kernel<DT, 4>, a);
    return e == cudaSuccess ? AFX_OK : AFX_ERR_CUDA;
}

afx_status launch_attention(int dtype, const AttnArgs& a, cudaStream_t st) {
    return dtype == AFX_F16 ? launch_attention_dt<AFX_F16>(a, st) : launch_attention_dt<AFX_BF16>(a, st);
}

}  // namespace afx
