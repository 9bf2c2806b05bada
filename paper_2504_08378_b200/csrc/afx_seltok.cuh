// Selection on its own: the active list of one to eight tokens and the side outputs of a layer operator,
// one block of 1024 threads per token, the tokens' blocks in one cluster.
//
// A block holds its token's keys in the registers of NW warps (afx_topk.cuh) and leaves the token's set as a
// bitmap in shared memory; after one cluster barrier every block has the union of all bitmaps, a word per
// thread, and writes its share of the list.  What bounds it is latency: of a chain of search steps, not of
// the tokens, which one block used to take one after the other (eight tokens of 5120 channels with the
// operator on their list, 5120 -> 27648: 91 us, with the list kernel of that time 67, now 59).
#pragma once

#include <cooperative_groups.h>

#include "afx_fused.cuh"
#include "afx_topk.cuh"

namespace afx {

constexpr int kStThreads = 1024;
constexpr int kStWords = kSelectFastMaxK / 32;

struct SelTokSmem {
    RegSelScratch sel;
    uint32_t set[kStWords];   // this token's active channels
    uint32_t all[kStWords];   // the union
    int32_t pos[kStWords];    // list position of a word's first channel
    int wtot[2][33];
};

// Writes the channels of the words w = rank, rank + T, ... of `words` (positions in `pos`) to `out`.
__device__ __forceinline__ void write_words(const uint32_t* words, const int32_t* pos, int nwords, int rank, int T, int32_t* out) {
    const int lane = lane_id();
    const uint32_t lt = (1u << lane) - 1u;
    for (int w = rank + T * warp_id(); w < nwords; w += T * (kStThreads / 32)) {
        const uint32_t u = words[w];
        if ((u >> lane) & 1u) out[pos[w] + __popc(u & lt)] = 32 * w + lane;
    }
}

// grid = cluster = (T, 1, 1).  Reads a.h / a.gain / a.eps (IN_NORM) or a.x, mode, k, tau and the hints; with a list
// decided earlier (a.idx_in) only the normed input, the copy of the list and its length are written.
template <int DT, int NW, int CH, int IN>
__device__ __forceinline__ void select_tokens_block(const FusedArgs& a, SelTokSmem* sm) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int T = gridDim.x, t = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int K = a.K, m = sel_slots<NW>(K), nwords = (K + 31) >> 5;
    const bool selects = NW == kStThreads / 32 || warp_id() < NW;
    const bool own = a.idx_in == nullptr;
    const bool topk = a.mode == AFX_MODE_TOPK && a.k > 0 && a.k < K;
    // Read before the dependency wait: gains never change; the hint may be rewritten meanwhile by an earlier launch
    // of the operator, and either value gives the same selection.
    constexpr bool kEarlyGain = IN == IN_NORM && CH < 8;
    float4 gv[kEarlyGain ? CH : 1];
    if constexpr (kEarlyGain) {
        if (selects) sel_load_gain<CH>(a.gain, K, m, gv);
    }
    int32_t* const slot = T == 1 ? a.kth_slot : a.kth_multi != nullptr ? a.kth_multi + t : nullptr;
    if (own) sel_prepare<NW>(slot, &sm->sel);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (ordering rule)

    int cnt = 0;
    if (selects) {
        uint32_t kw[2 * CH];
        if (IN == IN_NORM)
            sel_norm_keys<DT, NW, CH, kEarlyGain>(a.h + static_cast<size_t>(t) * K, a.gain, gv, a.eps, K, m, &sm->sel,
                                                  a.xnorm_out != nullptr ? a.xnorm_out + static_cast<size_t>(t) * K : nullptr, kw);
        else if (own)
            sel_load_keys<CH>(a.x + static_cast<size_t>(t) * K, K, m, kw);
        if (own) {
            if (IN == IN_X) sel_barrier<NW>();  // the hint is there (IN_NORM: since the norm's barrier)
            int kth, at;
            const uint32_t fl = sel_flags<DT, NW, CH>(kw, m, K, a.mode, a.k, a.tau, sm->sel.hint, &sm->sel, kth, at, cnt);
            if (tid == 0 && topk && slot != nullptr) *slot = 0x10000 | kth;
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                uint32_t bits = 0;  // of 8 lanes: 32 channels
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (fl & sel_bit(i, e)) bits |= 1u << (4 * (lane & 7) + e);
                bits |= __shfl_xor_sync(0xFFFFFFFFu, bits, 1);
                bits |= __shfl_xor_sync(0xFFFFFFFFu, bits, 2);
                bits |= __shfl_xor_sync(0xFFFFFFFFu, bits, 4);
                const int j = sel_channel(m, i);
                if (i < m && (lane & 7) == 0 && j < K) sm->set[j >> 5] = bits;
            }
        }
    }
    if (!own) {  // (any block of the cluster may do this: no barrier)
        cnt = max(0, min(*a.count_in, K));
        if (a.idx_out != nullptr && a.idx_out != a.idx_in)
            for (int i = t * kStThreads + tid; i < cnt; i += T * kStThreads) a.idx_out[i] = a.idx_in[i];
        if (t == 0 && tid == 0 && a.count_out != nullptr) *a.count_out = cnt;
        return;
    }
    if (T > 1) cluster.sync(); else __syncthreads();  // every token's set is in place
    uint32_t u = 0;
    if (tid < nwords) {
        u = sm->set[tid];
        for (int q = 1; q < T; ++q) u |= *cluster.map_shared_rank(&sm->set[tid], (t + q) % T);
    }
    const int first = block_prefix(__popc(u), sm->wtot[0], cnt);
    if (tid < nwords) {
        sm->all[tid] = u;
        sm->pos[tid] = first;
        if (a.bitmap_out != nullptr && tid % T == t) a.bitmap_out[tid] = u;
    }
    __syncthreads();
    if (a.idx_out != nullptr) write_words(sm->all, sm->pos, nwords, t, T, a.idx_out);
    if (t == 0 && tid == 0 && a.count_out != nullptr) *a.count_out = cnt;
    if (a.bitmap_pred != nullptr) {  // A \ P in ascending order, |A & P|
        const uint32_t miss = tid < nwords ? u & ~__ldcg(a.bitmap_pred + tid) : 0u;
        int n_miss;
        const int at = block_prefix(__popc(miss), sm->wtot[1], n_miss);
        __syncthreads();  // the list has been written
        if (tid < nwords) {
            sm->all[tid] = miss;
            sm->pos[tid] = at;
        }
        __syncthreads();
        if (a.miss_out != nullptr) write_words(sm->all, sm->pos, nwords, t, T, a.miss_out);
        if (t == 0 && tid == 0) {
            if (a.miss_count != nullptr) *a.miss_count = n_miss;
            if (a.hit_count != nullptr) *a.hit_count = cnt - n_miss;
        }
    }
    if (T > 1) cluster.sync();  // the peers have read this block's set
}

}  // namespace afx
