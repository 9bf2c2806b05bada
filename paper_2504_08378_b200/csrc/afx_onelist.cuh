// The front of the one-token operators (16-bit rows: afx_slice.cuh, 4-bit rows: afx_q4op.cuh): input stage with
// optional RMSNorm, selection in registers, the active list in shared memory, and the side outputs.
#pragma once

#include "afx_fused.cuh"
#include "afx_gemv.cuh"
#include "afx_topk.cuh"

namespace afx {

template <int DT>
__device__ __forceinline__ float list_x(uint32_t entry) {
    return DT == AFX_BF16 ? __uint_as_float(entry & 0xFFFF0000u) : bits_to_float<DT>(static_cast<uint16_t>(entry >> 16));
}

// Input stage and selection of a one-token operator: the active list, staged as entries (16-bit channel, 16-bit
// input) at `dyn`, and its length.  `early`: the input is older than the kernel before this one, and the dependency
// wait is left to the caller.  xs_at: where in `dyn` the inputs of a list decided earlier are staged.  The first NW of
// the NT / 32 warps select, with up to CH slots of 4 channels per lane (K <= 128 NW CH).  Every thread calls it; a
// block barrier is its last step.
template <int DT, int NT, int NW, int CH, int IN>
__device__ __forceinline__ int one_token_list(const FusedArgs& a, const uint16_t* x, bool early, bool scribe, unsigned char* dyn,
                                              size_t xs_at, RegSelScratch* sc) {
    const int tid = threadIdx.x;
    const int K = a.K, m = sel_slots<NW>(K);
    const bool selects = NW == NT / 32 || (tid >> 5) < NW;
    uint32_t* list = reinterpret_cast<uint32_t*>(dyn);
    const bool own = a.idx_in == nullptr;
    // What the prologue reads before the dependency wait was written at least two grids earlier (the
    // ordering rule stated at fused_op_block): gains never.  The hint may be rewritten meanwhile (by the launch
    // before, or by this launch's own scribe): either value gives the same selection.
    constexpr bool kEarlyGain = IN == IN_NORM && CH < 8;
    float4 gv[kEarlyGain ? CH : 1];
    if constexpr (kEarlyGain) {
        if (selects) sel_load_gain<CH>(a.gain, K, m, gv);
    }
    if (own) sel_prepare<NW>(a.kth_slot, sc);
    if (!early) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (ordering rule)
    }
    AFX_MARK(1);

    // ---- input and selection: the active list, staged as (channel, 16-bit input) ----
    uint16_t* xs = reinterpret_cast<uint16_t*>(dyn + xs_at);
    constexpr int kGiven = 4;  // entries of a given list that are requested together with the input
    int32_t given[kGiven];
    int cnt = 0;
    if (!own) {
        cnt = *a.count_in;
#pragma unroll
        for (int u = 0; u < kGiven; ++u)
            if (tid + u * NT < K) given[u] = a.idx_in[tid + u * NT];  // (the list's capacity is K)
    }
    if (selects) {
        uint32_t kw[2 * CH];
        if (IN == IN_NORM)
            sel_norm_keys<DT, NW, CH, kEarlyGain>(a.h, a.gain, gv, a.eps, K, m, sc, scribe ? a.xnorm_out : nullptr, kw);
        else
            sel_load_keys<CH>(x, K, m, kw);
        AFX_MARK(2);
        if (own) {
            if (IN == IN_X) sel_barrier<NW>();  // sc->hint is there (IN_NORM: since the norm's barrier)
            int kth, at, n;
            const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(list));
            const uint32_t fl = sel_flags<DT, NW, CH>(kw, m, K, a.mode, a.k, a.tau, sc->hint, sc, kth, at, n);
            sel_emit<CH>(fl, m, kw, base + 4u * static_cast<uint32_t>(at));
            if (tid == 0) {
                sc->count = n;
                if (scribe && a.kth_slot != nullptr && a.mode == AFX_MODE_TOPK && a.k > 0 && a.k < K)
                    *a.kth_slot = 0x10000 | kth;
            }
        } else {
#pragma unroll
            for (int i = 0; i < CH; ++i)
                if (i < m && sel_channel(m, i) < K)
                    *reinterpret_cast<uint2*>(xs + sel_channel(m, i)) = make_uint2(kw[2 * i], kw[2 * i + 1]);
        }
    }
    if (!own) {
        __syncthreads();
        cnt = max(0, min(cnt, K));
#pragma unroll
        for (int u = 0; u < kGiven; ++u) {
            const int i = tid + u * NT;
            if (i < cnt) list[i] = (static_cast<uint32_t>(xs[given[u]]) << 16) | static_cast<uint32_t>(given[u]);
        }
        for (int i = tid + kGiven * NT; i < cnt; i += NT) {
            const uint32_t j = static_cast<uint32_t>(a.idx_in[i]);
            list[i] = (static_cast<uint32_t>(xs[j]) << 16) | j;
        }
    }
    __syncthreads();
    if (own) cnt = sc->count;
    AFX_MARK(3);
    return cnt;
}

// What a layer operator leaves besides its outputs, from the staged list of `cnt` entries: the block that writes the side
// outputs selects like the others and does nothing else.
template <int NT>
__device__ __forceinline__ void one_token_side_outputs(const FusedArgs& a, const uint32_t* list, int cnt, RegSelScratch* sc) {
    const int tid = threadIdx.x, K = a.K;
    const bool own = a.idx_in == nullptr;
    if (own) {
        if (a.idx_out != nullptr)
            for (int i = tid; i < cnt; i += NT) a.idx_out[i] = static_cast<int32_t>(list[i] & 0xFFFFu);
        if (a.bitmap_pred != nullptr) {
            // A \ P in ascending order, |A & P|: thread t looks at a contiguous run of the list
            const int per = (cnt + NT - 1) / NT;  // <= 32
            const int i0 = min(cnt, tid * per), i1 = min(cnt, i0 + per);
            uint32_t miss = 0;
            for (int i = i0; i < i1; ++i) {
                const uint32_t j = list[i] & 0xFFFFu;
                if (((__ldcg(a.bitmap_pred + (j >> 5)) >> (j & 31u)) & 1u) == 0u) miss |= 1u << (i - i0);
            }
            int n_miss;
            int at = block_prefix(__popc(miss), reinterpret_cast<int*>(&sc->part[0][0][0]), n_miss);
            if (a.miss_out != nullptr)
                for (int i = i0; i < i1; ++i)
                    if ((miss >> (i - i0)) & 1u) a.miss_out[at++] = static_cast<int32_t>(list[i] & 0xFFFFu);
            if (tid == 0) {
                if (a.miss_count != nullptr) *a.miss_count = n_miss;
                if (a.hit_count != nullptr) *a.hit_count = cnt - n_miss;
            }
        }
        if (a.bitmap_out != nullptr) {
            // word w = the list's channels 32 w .. 32 w + 31: a run of the ascending list
            for (int w = tid; w < (K + 31) / 32; w += NT) {
                int lo = 0, hi = cnt;  // first entry at or behind channel 32 w
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (static_cast<int>(list[mid] & 0xFFFFu) < 32 * w) lo = mid + 1; else hi = mid;
                }
                uint32_t bits = 0;
                for (; lo < cnt && static_cast<int>(list[lo] & 0xFFFFu) < 32 * w + 32; ++lo) bits |= 1u << (list[lo] & 31u);
                a.bitmap_out[w] = bits;
            }
        }
    } else if (a.idx_out != nullptr && a.idx_out != a.idx_in) {
        for (int i = tid; i < cnt; i += NT) a.idx_out[i] = a.idx_in[i];
    }
    if (tid == 0 && a.count_out != nullptr) *a.count_out = cnt;
}

}  // namespace afx
