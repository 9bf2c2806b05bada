// The one-token sparse operator of a decoder layer as a single kernel: input stage (optional
// RMSNorm), selection, sparse GEMV, epilogue, on one block per SM.
//
// The outputs are cut into one slice per SM, equal to within one granule of 32 outputs (64 bytes of a row:
// one DRAM access), and a block streams the WHOLE active list for its slice: sums meet inside the block
// only, every SM carries the same bytes, and the input stage and the selection run once per SM.  A
// row's piece of a slice is P 16-byte loads; thread t takes piece t mod P of the list entries t div P,
// t div P + rows, ..., eight of them in flight.
//
// What bounds it: HBM while it streams (a 4096 -> 22016 operator at 50 %: 6.1 TB/s between the first load and
// the last), and before and after that a chain of latencies in which HBM is idle: dependency wait 1.0 us,
// input and norm 1.5, search 1.3, list 1.0, sums 0.8 at K = 4096.  Clusters of 3 to 8 blocks of 512 threads,
// two per SM, that shared a tile ran the input stage and the selection twice per SM, bound by instruction
// issue, left 6 to 14 SMs without a block and needed a cluster barrier for the sums.  Alone in a
// graph, before and after: 4096 -> 22016 21.8 and 20.0 us, 4096 -> 4096 9.6 and 8.5, 11008 -> 4096
// 17.2 and 15.3, 28672 -> 8192 70.9 and 52.0, 1024 -> 3072 7.7 and 5.7 us.
// Sharing the selection among the eight blocks of a cluster lost again: a cluster barrier with pushed
// operands costs 0.75 to 1 us, five of them more than the selection takes.
// Narrow operators of many channels have fewer granules than there are SMs and long lists: there the blocks of
// a cluster share the list of one granule (SPLIT, see launch_slice_k).
#pragma once

#include "afx_fused.cuh"
#include "afx_gemv.cuh"
#include "afx_topk.cuh"

namespace afx {

constexpr int kSlGranule = 4;  // pieces (16-byte loads of a row) that one slice holds together
// Shared memory that at least one block of 512 threads asks for, so that an SM takes one such block and
// what it leaves free goes to a block of another kernel.
constexpr size_t kSlAlone = 116 * 1024;

// Blocks that share a granule's list at most, and outputs of a granule.
constexpr int kSlMaxSplit = 8;
constexpr int kSlSplitOutputs = kSlGranule * 8;

// Widest slice in pieces: one output per thread in the epilogue.
__host__ __device__ constexpr int slice_max_pieces(int threads) { return threads / 8; }

// Dynamic shared memory: the staged list (16-bit channel, 16-bit input), later the sums; behind it the
// 16-bit inputs where a list decided earlier is staged.
__host__ __device__ inline size_t slice_list_bytes(int threads, int K) {
    const size_t list = (static_cast<size_t>(K) * 4 + 15) / 16 * 16;
    const size_t sums = static_cast<size_t>(threads) * 9 * 4;
    return list > sums ? list : sums;
}
__host__ __device__ inline size_t slice_dyn_smem(int threads, int K, bool list_given) {
    return slice_list_bytes(threads, K) + (list_given ? (static_cast<size_t>(K) + 7) / 8 * 16 : 0);
}

template <int DT>
__device__ __forceinline__ float list_x(uint32_t entry) {
    return DT == AFX_BF16 ? __uint_as_float(entry & 0xFFFF0000u) : bits_to_float<DT>(static_cast<uint16_t>(entry >> 16));
}

// Streams list entries [0, cnt) for one piece: acc += x * W[channel][8 outputs].
template <int DT>
__device__ __forceinline__ void slice_stream(const uint16_t* Wt, int64_t ldw, int piece, const uint32_t* list, int cnt, int g,
                                             int groups, f32x2 (&acc)[4]) {
    constexpr int U = 8;
    const char* base = reinterpret_cast<const char*>(Wt + static_cast<size_t>(piece) * 8);
    const uint64_t row = static_cast<uint64_t>(ldw) * 2;
    auto consume = [&](const uint4& raw, uint32_t e) {
        f32x2 w[4];
        unpack8_pairs<DT>(raw, w);
        const float xv = list_x<DT>(e);
        const f32x2 x2 = pack_f32x2(xv, xv);
#pragma unroll
        for (int i = 0; i < 4; ++i) fma_f32x2(acc[i], w[i], x2);
    };
    int p = g;
    for (; p + (U - 1) * groups < cnt; p += U * groups) {
        uint4 raw[U];
#pragma unroll
        for (int u = 0; u < U; ++u) raw[u] = ld_stream_16B(base + (list[p + u * groups] & 0xFFFFu) * row);
#pragma unroll
        for (int u = 0; u < U; ++u) consume(raw[u], list[p + u * groups]);
    }
    if (p < cnt) {
        uint4 raw[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (p + u * groups < cnt) raw[u] = ld_stream_16B(base + (list[p + u * groups] & 0xFFFFu) * row);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (p + u * groups < cnt) consume(raw[u], list[p + u * groups]);
    }
}

// Stores v to the shared-memory word at `at` where `on` holds; never a branch.
__device__ __forceinline__ void st_shared_if(uint32_t at, uint32_t v, bool on) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p st.shared.u32 [%0], %1; }" ::"r"(at), "r"(v), "r"(on ? 1u : 0u) : "memory");
}

// The row sets' sums (thread `tid` holds row set g = tid / P, piece tid - g P, of `rows` sets) meet and leave
// as outputs 8 piece0 .. of the operator: `parts` threads per output add every parts-th set, then in order.
// SPLIT: the blocks of the cluster (all have arrived once at its barrier) push their sums into block 0's `recv`,
// which adds them in rank order.
template <int DT, int NT, int EP, bool SPLIT>
__device__ __forceinline__ void slice_finish(const f32x2 (&acc)[4], int g, int rows, int P, int piece0, unsigned char* dyn, float* recv,
                                             float* y, uint16_t* out_bits, float scale, float y_old) {
    const int tid = threadIdx.x, nout = P * 8;
    const int parts = NT / nout, part = tid / nout, out = tid - part * nout;
    __syncthreads();  // the list has been read
    AFX_MARK(6);
    float* red = reinterpret_cast<float*>(dyn);
    if (g < rows) {
        float4* d4 = reinterpret_cast<float4*>(red + tid * 8);
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            float4 v;
            unpack_f32x2(acc[i], v.x, v.y);
            unpack_f32x2(acc[i + 1], v.z, v.w);
            d4[i / 2] = v;
        }
    }
    __syncthreads();
    float* red2 = red + NT * 8;
    if (part < parts) {
        float sum = 0.0f;
#pragma unroll 4
        for (int r = part; r < rows; r += parts) sum += red[r * nout + out];
        red2[tid] = sum;
    }
    __syncthreads();
    auto own = [&](int o) {
        float v = red2[o];
#pragma unroll 4
        for (int q = 1; q < parts; ++q) v += red2[q * nout + o];
        return v;
    };
    const int split = SPLIT ? static_cast<int>(cg::this_cluster().num_blocks()) : 1;
    if (SPLIT) {
        const int rank = static_cast<int>(cg::this_cluster().block_rank());
        cluster_wait();  // block 0 is running
        if (tid < nout) cg::this_cluster().map_shared_rank(recv, 0)[rank * kSlSplitOutputs + tid] = own(tid);
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        if (rank != 0) return;
    }
    auto total = [&](int o) {
        if (!SPLIT) return own(o);
        float v = recv[o];
        for (int q = 1; q < split; ++q) v += recv[q * kSlSplitOutputs + o];
        return v;
    };
    if (EP == EP_SILU) {
        // pair r of the slice: 8 gate then 8 up outputs per 16 columns
        if (tid < nout / 2) {
            const int o = (tid >> 3) * 16 + (tid & 7);
            const float gate = total(o), up = total(o + 8);
            out_bits[piece0 * 4 + tid] = float_to_bits<DT>(gate / (1.0f + expf(-gate)) * up);
        }
    } else if (tid < nout) {
        const float v = total(tid) * scale;
        y[piece0 * 8 + tid] = EP == EP_ACCUM ? y_old + v : v;
    }
}

// GRP: the grid may hold several operators of one family (FusedArgs::groups).  The first NW of the NT / 32
// warps select, with up to CH slots of 4 channels per lane (K <= 128 NW CH).
template <int DT, int NT, int NW, int CH, int IN, int EP, bool GRP, bool SPLIT>
__device__ __forceinline__ void slice_op_block(const FusedArgs& a, unsigned char* dyn, RegSelScratch* sc, float* recv) {
    const int tid = threadIdx.x, warp = tid >> 5;
    const int K = a.K, m = sel_slots<NW>(K);
    const bool selects = NW == NT / 32 || warp < NW;
    const int split = SPLIT ? static_cast<int>(cg::this_cluster().num_blocks()) : 1;  // blocks that share a list
    const int rank = SPLIT ? static_cast<int>(cg::this_cluster().block_rank()) : 0;
    const int unit = SPLIT ? static_cast<int>(blockIdx.x) / split : static_cast<int>(blockIdx.x);
    const int units = SPLIT ? static_cast<int>(gridDim.x) / split : static_cast<int>(gridDim.x);
    const int nb = a.slices, grp = GRP ? unit / nb : 0, b = unit - grp * nb;
    const bool scribe = a.side_cluster != 0 && unit == units - 1;  // selects only, writes the side outputs
    if (SPLIT) {
        if (scribe && rank != 0) return;
        if (!scribe) cluster_arrive();  // (the scribe's cluster never meets)
    }
    const uint16_t* x = GRP ? a.x + grp * a.x_stride : a.x;
    uint32_t* list = reinterpret_cast<uint32_t*>(dyn);
    const bool own = a.idx_in == nullptr;
    AFX_TRACE_REGION(IN == IN_NORM ? (EP == EP_SILU ? 2 : 1) : (K > a.N ? 3 : 4));
    AFX_MARK(0);

    // ---- this block's slice: granules [g_lo, g_hi) of the operator, P pieces per row ----
    const int pieces = a.N / 8, granules = (pieces + kSlGranule - 1) / kSlGranule;
    const int g_lo = b * granules / nb, g_hi = (b + 1) * granules / nb;  // (the launcher keeps the products below 2^31)
    const int piece0 = g_lo * kSlGranule, P = max(1, min(g_hi * kSlGranule, pieces) - piece0);  // 1 <= P <= slice_max_pieces
    const int nout = P * 8;
    const int rows = NT / P;                  // list entries the block takes at once
    const int g = tid / P, piece = tid - g * P;

    // What the prologue reads before the dependency wait was written at least two grids earlier (the
    // ordering rule stated at fused_op_block): gains never.  The hint may be rewritten meanwhile (by the launch
    // before, or by this launch's own scribe): either value gives the same selection.
    constexpr bool kEarlyGain = IN == IN_NORM && CH < 8;
    float4 gv[kEarlyGain ? CH : 1];
    if constexpr (kEarlyGain) {
        if (selects) sel_load_gain<CH>(a.gain, K, m, gv);
    }
    if (own) sel_read_hint(a.kth_slot, sc);
    const bool early = GRP && a.x_early != 0;  // the input is older than the kernel before this one: select first
    if (!early) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (ordering rule)
    }
    AFX_MARK(1);

    // ---- input and selection: the active list, staged as (channel, 16-bit input) ----
    uint16_t* xs = reinterpret_cast<uint16_t*>(dyn + slice_list_bytes(NT, K));
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
            sel_emit<CH>(fl, m, at, [&](int i, int e, int pos, bool on) {
                st_shared_if(base + 4 * pos, __byte_perm(kw[2 * i + (e >> 1)], static_cast<uint32_t>(sel_channel(m, i) + e), (e & 1) ? 0x3254 : 0x1054), on);
            });
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

    if (scribe) {
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
        return;
    }

    if (early) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    // where the sums leave
    const uint16_t* Wt = a.wt_table != nullptr ? a.wt_table[a.wt_sel[grp]] : a.Wt;
    float* y = a.ep.y;
    uint16_t* out_bits = a.ep.out_bits;
    float scale = 1.0f;
    if (GRP) {
        if (y != nullptr) y += grp * a.out_stride;
        if (out_bits != nullptr) out_bits += grp * a.out_stride;
    }
    if (EP != EP_SILU && a.ep.scale != nullptr) scale = a.ep.scale[grp];
    float y_old = 0.0f;
    if (EP == EP_ACCUM && tid < nout) y_old = y[piece0 * 8 + tid];  // long before it is added to

    f32x2 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = pack_f32x2(0.0f, 0.0f);
    const int c_lo = SPLIT ? rank * cnt / split : 0, c_hi = SPLIT ? (rank + 1) * cnt / split : cnt;
    if (g < rows) slice_stream<DT>(Wt, a.ldw, piece0 + piece, list + c_lo, c_hi - c_lo, g, rows, acc);
    AFX_MARK(5);

    slice_finish<DT, NT, EP, SPLIT>(acc, g, rows, P, piece0, dyn, recv, y, out_bits, scale, y_old);
    AFX_MARK(7);
}

}  // namespace afx
