// Launcher of the one-token sparse operator (afx_slice.cuh).
#include "afx_launch.cuh"
#include "afx_slice.cuh"

namespace afx {

template <int DT, int NT, int NW, int CH, int IN, int EP, bool GRP, int FORM>
__global__ void __launch_bounds__(NT, 1024 / NT) slice_op_kernel(FusedArgs a) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ RegSelScratch s;
    __shared__ float recv[FORM == SLICE_SPLIT ? kSlMaxSplit * kSlSplitOutputs : 1];
    slice_op_block<DT, NT, NW, CH, IN, EP, GRP, FORM>(a, dyn, &s, recv);
}

// split: blocks (a cluster) that share the list of a granule; a.N is then at most as wide as there is room for
// one granule per cluster.
template <int DT, int NT, int NW, int CH, int IN, int EP, bool GRP, int FORM = SLICE_PLAIN>
static afx_status launch_slice(const FusedArgs& a, cudaStream_t st, int split = 1) {
    constexpr bool SPLIT = FORM == SLICE_SPLIT;
    if (static_cast<uint64_t>(a.K) * static_cast<uint64_t>(a.ldw >> 3) > 0x100000000ull) return AFX_ERR_CAPACITY;
    FusedArgs b = a;
    b.side_cluster = a.idx_out != nullptr || a.count_out != nullptr || a.bitmap_out != nullptr ||
                     a.xnorm_out != nullptr || a.bitmap_pred != nullptr || a.kth_slot != nullptr;
    // one slice per SM, one SM left for the side outputs where there are any; more slices (in waves) only
    // where one would exceed the widest a block can finish
    const int groups = GRP ? a.groups : 1;
    const int sms = sm_count() > 0 ? sm_count() : 148;
    int nb = (sms - b.side_cluster - (GRP && a.x_early ? 1 : 0)) / groups;  // (that kernel's block keeps one SM busy)
    b.granule = kSlGranule;
    if (FORM == SLICE_FINE)
        while (b.granule > (EP == EP_SILU ? 2 : 1) && 2 * ((a.N / 8 + b.granule - 1) / b.granule) <= nb) b.granule >>= 1;
    const int most = slice_max_pieces(NT) / b.granule;  // granules per slice
    const int granules = (a.N / 8 + b.granule - 1) / b.granule;
    if (nb > granules) nb = granules;
    if (nb < 1) nb = 1;
    if ((granules + nb - 1) / nb > most) nb = ((granules + most - 1) / most + nb - 1) / nb * nb;
    if (static_cast<int64_t>(nb) * granules >= 0x7FFFFFFF) return AFX_ERR_CAPACITY;
    b.slices = nb;
    size_t dyn = slice_dyn_smem(NT, a.K, a.idx_in != nullptr);
    if (NT == 512 && dyn < kSlAlone) dyn = kSlAlone;
    auto kern = slice_op_kernel<DT, NT, NW, CH, IN, EP, GRP, FORM>;
    if (!ensure_dyn_smem(reinterpret_cast<const void*>(kern), dyn)) {
        cudaGetLastError();
        return AFX_ERR_CUDA;
    }
    cudaLaunchConfig_t cfg = {};
    const int units = nb * groups + b.side_cluster;
    // clusters that the occupancy query counts and that are then placed behind another kernel differ by a few
    while (SPLIT && split > 1 && max_active_clusters(reinterpret_cast<const void*>(kern), split, dyn, NT) < units + 2) split >>= 1;
    cfg.gridDim = dim3(units * split, 1, 1);
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

// Blocks of 512 threads beside the attention: its blocks become resident next to them, request their first
// rows before the wait and start as soon as the operator's last block ends (4096 -> 12288, attention over
// 2048 positions, 4096 -> 4096: 35.0 us, with 1024 threads 39.7).  Small operators too, which wait less
// for fewer warps (1024 -> 5632: 6.2 us, with 1024 threads 8.0).  Elsewhere 1024 threads keep twice
// the loads in flight (4096 -> 22016: 20.0 us, with 512 threads 24.1), and above K = 4096 that is worth
// more than the overlap (a layer over 2048 positions, 1024 and 512 threads beside the attention: 4608 channels
// 77.3 and 78.3 us, 5120 97.0 and 99.8, 6144 119.2 and 123.3, 8192 with 8 kv heads 93.7 and 100.0).
constexpr int kSlNarrowMaxK = 4096;
// From here on clusters share a granule's list, where at least four blocks find an SM for each granule.  One block and
// a cluster per granule, half of the channels kept, in a graph: 5120 -> 256 6.9 and 6.4 us, 5120 -> 1024 7.1 and 7.3,
// 8192 -> 512 8.2 and 6.9, 8192 -> 1024 9.7 and 8.2, 16384 -> 256 12.9 and 8.2, 28672 -> 512 20.8 and 15.0; two
// blocks per granule do not pay (8192 -> 2048 9.4 and 9.7).
constexpr int kSlSplitMinK = 6144;
// From here on slices of two pieces of a row, or one, where that puts twice as many SMs to work (a gate | up pair needs two
// pieces); neighbouring SMs then share the sectors of L2.  Half of the channels kept, in a graph, four pieces, two and one:
// 2048 -> 1024 5.3, 4.7, 4.8 us, 2816 -> 1024 5.6, 5.2, 5.1, 4096 -> 512 6.5, 5.9, 5.5, 5504 -> 1024 8.2, 7.1, 6.8,
// 2048 -> 2048 5.5, 5.0, 4096 -> 2048 7.4, 7.0, 16384 -> 2048 15.9, 15.2; below, a list is short enough for few SMs:
// 512 -> 1376 3.9, 4.0, 1024 -> 1024 4.2, 4.2, 4.3.
constexpr int kSlFineMinK = 1536, kSlFineMaxN = 2336;  // (73 granules of four pieces and the block of the side outputs)
// Top-k operators of 16-bit inputs on 1024 threads where a thread takes seven or eight rows: all of them in flight instead
// of six and then the rest.  us, eight rows in flight always, six, and now, half of the channels kept: 2048 -> 5632 7.0,
// 7.2, 6.7, 4096 -> 4096 8.0, 8.1, 7.7, 2048 -> 8192 7.4, 7.7, 7.2; 40 %: 4096 -> 4096 7.5, 7.6, 7.3.  More rows than
// eight lose with two passes of eight what three of six cost (13 rows, 4096 -> 6144: 9.6 and 9.1).
// Selecting warps and slots: as few warps as leave a lane enough registers.
template <int DT, int IN, int EP, bool GRP>
static afx_status launch_slice_k(const FusedArgs& a, cudaStream_t st) {
    if (a.K >= kSlSplitMinK) {
        const int clusters = (a.N / 8 + kSlGranule - 1) / kSlGranule * (GRP ? a.groups : 1) + 1;  // (one for the side outputs)
        const int fit = (sm_count() > 0 ? sm_count() : 148) / clusters;
        const int split = fit >= 8 ? 8 : 4;
        if (fit >= 4 && a.K <= 16384) return launch_slice<DT, 512, 16, 8, IN, EP, GRP, SLICE_SPLIT>(a, st, split);
        if (fit >= 4 && a.K <= 32768) return launch_slice<DT, 1024, 32, 8, IN, EP, GRP, SLICE_SPLIT>(a, st, split);
    }
    const bool narrow = (a.beside_attention && a.K <= kSlNarrowMaxK) || static_cast<int64_t>(a.K) * a.N <= (8 << 20);
    if constexpr (!GRP) {
        if (a.K >= kSlFineMinK && a.N <= kSlFineMaxN) {
            if (narrow && a.K <= 4096) return launch_slice<DT, 512, 8, 4, IN, EP, GRP, SLICE_FINE>(a, st);
            if (narrow && a.K <= 12288) return launch_slice<DT, 512, 16, 6, IN, EP, GRP, SLICE_FINE>(a, st);
            if (a.K <= 16384) return launch_slice<DT, 1024, 16, 8, IN, EP, GRP, SLICE_FINE>(a, st);
        }
    }
    if (narrow && a.K <= 4096) return launch_slice<DT, 512, 8, 4, IN, EP, GRP>(a, st);
    if (narrow && a.K <= 12288) return launch_slice<DT, 512, 16, 6, IN, EP, GRP>(a, st);
    if constexpr (!GRP && IN == IN_X && EP != EP_SILU) {
        const int granules = (a.N / 8 + kSlGranule - 1) / kSlGranule, sms = (sm_count() > 1 ? sm_count() : 148) - 1;
        const int rows = 1024 / (kSlGranule * ((granules + sms - 1) / sms));  // list entries the widest slice takes at once
        if (a.idx_in == nullptr && a.mode == AFX_MODE_TOPK && a.k > 6 * rows && a.k <= kSlDeepRows * rows) {
            if (a.K <= 4096) return launch_slice<DT, 1024, 8, 4, IN, EP, GRP, SLICE_DEEP>(a, st);
            if (a.K <= 12288) return launch_slice<DT, 1024, 16, 6, IN, EP, GRP, SLICE_DEEP>(a, st);
        }
    }
    if (a.K <= 4096) return launch_slice<DT, 1024, 8, 4, IN, EP, GRP>(a, st);
    if (a.K <= 12288) return launch_slice<DT, 1024, 16, 6, IN, EP, GRP>(a, st);
    if (a.K <= 16384) return launch_slice<DT, 1024, 16, 8, IN, EP, GRP>(a, st);
    if (a.K <= 32768) return launch_slice<DT, 1024, 32, 8, IN, EP, GRP>(a, st);
    return AFX_ERR_CAPACITY;
}

template <int DT>
static afx_status launch_one_token_dt(int in, int ep, OneTokenForm form, const FusedArgs& a, cudaStream_t st) {
    if (form == ONE_TOKEN_FAMILY) {
        if (a.T != 1 || a.groups < 1 || a.wt_table == nullptr || a.wt_sel == nullptr) return AFX_ERR_INVALID_ARG;
        return ep == EP_SILU ? launch_slice_k<DT, IN_X, EP_SILU, true>(a, st)
                             : launch_slice_k<DT, IN_X, EP_STORE, true>(a, st);
    }
    if (in == IN_NORM && ep == EP_STORE) return launch_slice_k<DT, IN_NORM, EP_STORE, false>(a, st);
    if (in == IN_NORM && ep == EP_SILU) return launch_slice_k<DT, IN_NORM, EP_SILU, false>(a, st);
    if (in == IN_X && ep == EP_ACCUM) return launch_slice_k<DT, IN_X, EP_ACCUM, false>(a, st);
    if (in == IN_X && ep == EP_SILU) return launch_slice_k<DT, IN_X, EP_SILU, false>(a, st);
    if (in == IN_X && ep == EP_STORE) return launch_slice_k<DT, IN_X, EP_STORE, false>(a, st);
    return AFX_ERR_UNSUPPORTED;
}

afx_status launch_one_token(int dtype, int in, int ep, OneTokenForm form, const FusedArgs& a, cudaStream_t st) {
    return dtype == AFX_F16 ? launch_one_token_dt<AFX_F16>(in, ep, form, a, st)
                            : launch_one_token_dt<AFX_BF16>(in, ep, form, a, st);
}

}  // namespace afx
