// What a fused sparse operator is given (FusedArgs), and the form of it for several tokens in one kernel, whose clusters
// select over a shared-memory histogram: where the caller has no room for the list between two launches
// (afx_seltok.cuh, afx_mtlist.cuh).  (One token: afx_slice.cuh, afx_q4op.cuh.)
// Active-channel selection, sparse GEMV, epilogue in one kernel; every cluster repeats the exact selection on its own
// (the activation vectors are a few KB and L2 resident).
#pragma once

#include "afx_gemv.cuh"
#include "afx_mma.cuh"
#include "afx_select.cuh"

namespace afx {

enum { IN_X = 0, IN_NORM = 1 };

constexpr int kFusedMtRows = 64;  // channels per pipeline stage of the several-token operator

struct FusedArgs {
    const uint16_t* Wt;
    // mixture of experts (one-token operator): if wt_table is given, the weights are wt_table[wt_sel[g]] (both DEVICE;
    // the choice is made on the device by the router kernel earlier in the stream)
    const uint16_t* const* wt_table;
    const int32_t* wt_sel;
    int64_t ldw;
    int K, N, T;
    // ---- input: IN_X reads x; IN_NORM computes x = round(h / rms(h) * gain) ----
    const uint16_t* x;  // [T][K] 16-bit floats
    const float* h;     // [T][K] fp32
    const float* gain;  // [K] fp32
    float eps;
    // ---- selection: own selection, or (idx_in != NULL) a list decided earlier ----
    int mode, k;
    float tau;
    const int32_t* idx_in;
    const int32_t* count_in;
    EpilogueArgs ep;
    // ---- side outputs, written by one block; each may be NULL ----
    int32_t* idx_out;        // the active list used (capacity K)
    int32_t* count_out;
    uint32_t* bitmap_out;    // the same set as a bitmap (own selection only)
    uint16_t* xnorm_out;     // IN_NORM: the normalised, rounded input [T][K]
    const uint32_t* bitmap_pred;  // cross-layer bookkeeping: predicted set P ...
    int32_t* miss_out;            // ... A \ P ascending (capacity K)
    int32_t* miss_count;
    int32_t* hit_count;           // |A & P|
    // ---- top-k search hint (may be NULL): 0x10000 | k-th key of this operator's last top-k
    // selection with T == 1; read before the selection, rewritten after it by the block of the side outputs ----
    int32_t* kth_slot;
    // ---- the same for several tokens (T > 1; may be NULL): T consecutive slots, one per token ----
    int32_t* kth_multi;
    // ---- set by the launcher (several-token operators): column tiles per cluster, 0 or 1 = one ----
    int tiles_per_cluster;
    // ---- set by the launcher: 1 if the grid has one more cluster (slice operator: block) than its outputs need; its block 0
    // repeats input stage and selection only to write the side outputs, off the path of the
    // clusters that stream (its other blocks leave at once) ----
    int side_cluster;
    // ---- several operators of one family in one grid (one-token operator; groups > 1, no side outputs):
    // the slices are `groups` equal runs, run g being an operator of the same shape with
    // weights wt_table[wt_sel[g]], input x + g * x_stride, outputs ep.y / ep.out_bits +
    // g * out_stride (elements) and factor ep.scale[g] ----
    int groups;
    // ---- one-token operator: the kernel before or after it is the attention ----
    int beside_attention;
    // ---- family: x was written before the kernel in front of this one started (that one decides wt_sel) ----
    int x_early;
    int slices;  // set by the launcher: slices per operator
    int granule;  // set by the launcher (16-bit rows): 16-byte pieces of a row that a slice holds together
    int64_t x_stride, out_stride;
};

// The one-token operator (afx_onetok.cu): a plain operator or `groups` operators of one family.
enum OneTokenForm { ONE_TOKEN_PLAIN, ONE_TOKEN_FAMILY };
afx_status launch_one_token(int dtype, int in, int ep, OneTokenForm form, const FusedArgs& a, cudaStream_t st);

// The same over 4-bit rows (afx_q4op.cu): a.Wt = the rows, a.ldw = their stride in units of 2 bytes, a.N % 32 == 0.
afx_status launch_q4_operator(int dtype, int in, int ep, const FusedArgs& a, cudaStream_t st);

// Input stage and selection of a.T tokens with the side outputs, as a kernel of its own (afx_seltok.cu).
afx_status launch_select_tokens(int dtype, bool norm, const FusedArgs& a, cudaStream_t st);

// Dynamic shared memory: [16-bit inputs of one token, padded to a multiple of 8 elements] [T bitmaps of ceil(K/32) flag
// words, each padded to 16 bytes: where the blocks of a cluster exchange the per-token sets they decided] [work area:
// the key histogram during the selection, then the staging and pipeline buffers].
__host__ __device__ inline size_t fused_input_smem(int K) { return (static_cast<size_t>(K) + 7) / 8 * 16; }
__host__ __device__ inline size_t fused_flag_smem(int K, int T = 1) {
    return static_cast<size_t>(T) * ((static_cast<size_t>((K + 31) / 32) * 4 + 15) / 16 * 16);
}
// work = bytes of the work area: the key histogram, or more where the streaming stage needs more
__host__ __device__ inline size_t fused_dyn_smem(int K, int T, size_t work) {
    return fused_input_smem(K) + fused_flag_smem(K, T) + (work > kKeyHistBytes ? work : kKeyHistBytes);
}

// Reads a.x, a.mode, a.k, a.tau; a.idx_out and a.count_out are the only side outputs.  The streaming stage runs on the
// tensor cores (afx_mma.cuh) with STAGES pipeline stages: the work area holds an MtSmem<CAP, STAGES> once the
// selection is over.
template <int DT, int TMAX, int CAP, int EP, int STAGES>
__device__ __forceinline__ void fused_op_block(const FusedArgs& a, unsigned char* dyn, SelectScratch* sel) {
    const int tid = threadIdx.x;
    // CS blocks form a cluster; S of them split the active list of one column tile.  CS == S
    // except for operators with few tiles: there a cluster covers CS / S adjacent
    // tiles, so that more blocks share the per-token selections (a.tiles_per_cluster).
    const int CS = gridDim.x, cs = blockIdx.x;
    const int tpc = a.tiles_per_cluster > 1 ? a.tiles_per_cluster : 1;
    const int S = tpc > 1 ? CS / tpc : CS, s = tpc > 1 ? cs % S : cs;
    const int T = a.T, K = a.K;
    const bool side = a.side_cluster != 0 && blockIdx.y == gridDim.y - 1;  // the cluster without a tile
    const int tile = tpc > 1 ? blockIdx.y * tpc + cs / S : blockIdx.y;
    if (side && blockIdx.x != 0) return;  // (a block that has left no longer holds back the next grid)

    uint16_t* xs = reinterpret_cast<uint16_t*>(dyn);
    unsigned char* work = dyn + fused_input_smem(K) + fused_flag_smem(K, T);
    uint32_t* hist = reinterpret_cast<uint32_t*>(work);

    const uint32_t ld16 = static_cast<uint32_t>(a.ldw >> 3);  // row stride in 16-byte units (the launcher checked the range)
    AFX_TRACE_REGION(EP == EP_SILU ? 2 : (K > a.N ? 3 : 4));
    AFX_MARK(0);
    if (!side) cluster_arrive();  // the side cluster never meets
    if (a.mode == AFX_MODE_TOPK && a.k > 0 && a.k < K) block_clear_key_hist<kGemvThreads>(hist);  // does not depend on the previous kernel

    // Ordering rule of every kernel of this library: a grid lets its successor be scheduled
    // only AFTER its own dependency wait.  When a grid runs its prologue, its predecessor has
    // therefore passed its wait, i.e. the grid before that one is complete: whatever is read
    // before the wait below must have been written at least two grids earlier (weights and
    // gains: never; the predicted set: by the same operator of an earlier layer, at least five
    // grids back).  The search hint is the exception: it may be rewritten while it is read.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    AFX_MARK(2);

    // ---- selection ----------------------------------------------------------------------
    unsigned long long fl = 0ull;  // this thread's active flags
    // The blocks of a cluster share the work -- block s decides the sets of the
    // tokens t with t % CS == cs and writes their flags into every block's table of per-token
    // bitmaps (distributed shared memory); after one cluster barrier every thread reads the
    // union for its own chunks.  (The side cluster works alone and decides every token.)
    const bool share = !side && CS > 1;
    uint8_t* const ftab = dyn + fused_input_smem(K);
    const size_t fstride = fused_flag_smem(K);
    int q_lo, q_hi;
    thread_chunk_range(K, q_lo, q_hi);
    if (share) cluster_wait();  // pairs with the cluster_arrive() at kernel start: the peers are running
    bool first = true;
    for (int t = 0; t < T; ++t) {
        if (share && t % CS != cs) continue;
        if (!first) __syncthreads();  // the previous token's keys are still being read
        block_stage_token(a.x + static_cast<size_t>(t) * K, K, xs);
        const unsigned long long ft = block_token_flags<DT, kGemvThreads>(xs, K, a.mode, a.k, a.tau, hist, first, sel);
        if (share) {
            for (int q = 0; q < CS; ++q) {
                uint8_t* dst = cg::this_cluster().map_shared_rank(ftab + static_cast<size_t>(t) * fstride, q);
                for (int c = q_lo; c < q_hi; ++c) dst[c] = static_cast<uint8_t>(ft >> (8 * (c - q_lo)));
            }
        } else {
            fl |= ft;
        }
        first = false;
    }
    if (share) {
        cluster_arrive();  // the flags written above are visible to the peers after their wait
        cluster_wait();
        for (int t = 0; t < T; ++t)
            for (int c = q_lo; c < q_hi; ++c)
                fl |= static_cast<unsigned long long>(ftab[static_cast<size_t>(t) * fstride + c]) << (8 * (c - q_lo));
    }
    int cnt = 0;
    const int pos0 = block_prefix(__popcll(fl), sel->wtot[2], cnt);  // list position of this thread's first active channel
    // ---- side outputs ----
    if (side) {
        if (a.idx_out != nullptr) for_each_owned_active(fl, K, pos0, [&](int j, int pos) { a.idx_out[pos] = j; });
        if (tid == 0 && a.count_out != nullptr) *a.count_out = cnt;
        return;
    }
    AFX_MARK(3);
    const int c_lo = s * cnt / S;  // S <= 8, cnt <= 2^20: no overflow
    const int c_hi = (s + 1) * cnt / S;

    const int n_mine = __popcll(fl);
    using MtT = MtSmem<CAP, STAGES, kFusedMtRows>;
    MtT* mt = reinterpret_cast<MtT*>(work);
    float c4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const uint4* wtile16 = reinterpret_cast<const uint4*>(a.Wt + static_cast<size_t>(tile) * kMtTile);
    const int n_chunks = max(0, min(kMtTile, a.N - tile * kMtTile)) >> 3;
    // (the last cluster of a grid with several tiles per cluster may hold a block without a
    // tile: it only shares the selections and meets the barriers)
    for (int c0 = c_lo; n_chunks > 0 && c0 < c_hi; c0 += CAP) {
        const int staged = min(CAP, c_hi - c0);
        __syncthreads();  // the work area is free: the histogram / the previous pass has been read
        if (pos0 < c0 + staged && pos0 + n_mine > c0) {
            for_each_owned_active(fl, K, pos0, [&](int j, int pos) {
                const int p = pos - c0;
                if (p >= 0 && p < staged) {
                    uint16_t xv[TMAX];  // (all on their way before the first store)
#pragma unroll
                    for (int t = 0; t < TMAX; ++t)
                        if (t < T) xv[t] = a.x[static_cast<size_t>(t) * K + j];
                    mt->col[p] = static_cast<uint32_t>(j) * ld16;
#pragma unroll
                    for (int t = 0; t < TMAX; ++t)
                        if (t < T) mt->xb[t][p] = xv[t];
                }
            });
        }
        mt_pad_inputs(mt, T, staged);
        __syncthreads();
        mt_stream_pass<DT>(wtile16, mt, staged, n_chunks, c4);
    }
    if (!share) cluster_wait();  // pairs with the cluster_arrive() at kernel start
    mt_finish<DT>(c4, mt, T, tile, a.N, EP, a.ep, S, s, cs - s);
    AFX_MARK(7);
}

}  // namespace afx
