// The one-token sparse operator of a decoder layer as a single kernel: input stage (optional
// RMSNorm), selection, sparse GEMV, epilogue, on one block per SM.
//
// The outputs are cut into one slice per SM, equal to within one granule of 32 outputs (64 bytes of a row:
// one DRAM access), and a block streams the WHOLE active list for its slice: sums meet inside the block
// only, every SM carries the same bytes, and the input stage and the selection run once per SM.  A
// row's piece of a slice is P 16-byte loads; thread t takes piece t mod P of the list entries t div P,
// t div P + rows, ..., six of them in flight (eight spill at 64 registers: 7B-shaped decode step 2312 and 2244 us; four
// 2299, five 2257, seven 2271).
//
// What bounds it: HBM while it streams (a 4096 -> 22016 operator at 50 %: 6.1 TB/s between the first load and
// the last), and before and after that a chain of latencies in which HBM is idle: dependency wait 0.2 us,
// input and norm 1.1, search 0.9, list 0.6, first load 1, sums 0.6 to 1.2 at K = 4096.  Clusters of 3 to 8 blocks of 512 threads,
// two per SM, that shared a tile ran the input stage and the selection twice per SM, bound by instruction
// issue, left 6 to 14 SMs without a block and needed a cluster barrier for the sums.  Alone in a
// graph, before and after: 4096 -> 22016 21.8 and 20.0 us, 4096 -> 4096 9.6 and 8.5, 11008 -> 4096
// 17.2 and 15.3, 28672 -> 8192 70.9 and 52.0, 1024 -> 3072 7.7 and 5.7 us.
// Sharing the selection among the eight blocks of a cluster lost again: a cluster barrier with pushed
// operands costs 0.75 to 1 us, five of them more than the selection takes.
// Narrow operators of many channels have fewer granules than there are SMs and long lists: there the blocks of
// a cluster share the list of one granule (SPLIT, see launch_slice_k).
#pragma once

#include "afx_onelist.cuh"

namespace afx {

constexpr int kSlGranule = 4;  // pieces (16-byte loads of a row) that one slice holds together
// SLICE_SPLIT: the blocks of a cluster share a granule's list; SLICE_FINE: granules of fewer pieces (FusedArgs::granule);
// SLICE_DEEP: kSlDeepRows rows in flight.
constexpr int kSlDeepRows = 8;
enum { SLICE_PLAIN = 0, SLICE_SPLIT = 1, SLICE_FINE = 2, SLICE_DEEP = 3 };
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

// Streams list entries [0, cnt) for one piece, U of them in flight: acc += x * W[channel][8 outputs].
template <int DT, int U>
__device__ __forceinline__ void slice_stream(const uint16_t* Wt, int64_t ldw, int piece, const uint32_t* list, int cnt, int g,
                                             int groups, f32x2 (&acc)[4]) {
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

// The row sets' sums (thread `tid` holds row set g = tid / P, piece tid - g P, of `rows` sets) meet and leave
// as outputs 8 piece0 .. of the operator: `parts` threads per output add every parts-th set, then in order.
// SPLIT: the blocks of the cluster (all have arrived once at its barrier) push their sums into block 0's `recv`,
// which adds them in rank order.
template <int DT, int NT, int EP, bool SPLIT, bool FINE>
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
    // Slices of one or two pieces leave many parts per output: those of a warp meet first.
    const bool narrow = FINE && (nout == 8 || nout == 16);
    if (narrow) {
        float sum = 0.0f;
        for (int r = part; r < rows; r += parts) sum += red[r * nout + out];  // (nout divides the block: every thread has a part)
        if (nout == 8) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 8);
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 16);
        if ((tid & 31) < nout) red2[(tid >> 5) * nout + out] = sum;
    } else if (part < parts) {
        float sum = 0.0f;
#pragma unroll 4
        for (int r = part; r < rows; r += parts) sum += red[r * nout + out];
        red2[tid] = sum;
    }
    __syncthreads();
    const int sums = narrow ? NT / 32 : parts;
    auto own = [&](int o) {
        float v = red2[o];
#pragma unroll 4
        for (int q = 1; q < sums; ++q) v += red2[q * nout + o];
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

// GRP: the grid may hold several operators of one family (FusedArgs::groups).
template <int DT, int NT, int NW, int CH, int IN, int EP, bool GRP, int FORM>
__device__ __forceinline__ void slice_op_block(const FusedArgs& a, unsigned char* dyn, RegSelScratch* sc, float* recv) {
    constexpr bool SPLIT = FORM == SLICE_SPLIT, FINE = FORM == SLICE_FINE;
    const int tid = threadIdx.x;
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
    AFX_TRACE_REGION(IN == IN_NORM ? (EP == EP_SILU ? 2 : 1) : (a.K > a.N ? 3 : 4));
    AFX_MARK(0);

    // ---- this block's slice: granules [g_lo, g_hi) of the operator, P pieces per row ----
    const int gran = FINE ? a.granule : kSlGranule;
    const int pieces = a.N / 8, granules = (pieces + gran - 1) / gran;
    const int g_lo = b * granules / nb, g_hi = (b + 1) * granules / nb;  // (the launcher keeps the products below 2^31)
    const int piece0 = g_lo * gran, P = max(1, min(g_hi * gran, pieces) - piece0);  // 1 <= P <= slice_max_pieces
    const int nout = P * 8;
    const int rows = NT / P;                  // list entries the block takes at once
    const int g = tid / P, piece = tid - g * P;

    const bool early = GRP && a.x_early != 0;  // the input is older than the kernel before this one: select first
    const int cnt = one_token_list<DT, NT, NW, CH, IN>(a, x, early, scribe, dyn, slice_list_bytes(NT, a.K), sc);
    if (scribe) {
        one_token_side_outputs<NT>(a, list, cnt, sc);
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
    if (g < rows) slice_stream<DT, FORM == SLICE_DEEP ? kSlDeepRows : 6>(Wt, a.ldw, piece0 + piece, list + c_lo, c_hi - c_lo, g, rows, acc);
    AFX_MARK(5);

    slice_finish<DT, NT, EP, SPLIT, FINE>(acc, g, rows, P, piece0, dyn, recv, y, out_bits, scale, y_old);
    AFX_MARK(7);
}

}  // namespace afx
