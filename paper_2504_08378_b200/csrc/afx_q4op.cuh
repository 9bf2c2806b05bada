// The one-token sparse operator of a decoder layer over 4-bit rows (afx_sparse_gemv_q4's layout) as a single kernel:
// the front of the one-token operators (afx_onelist.cuh), then the rows of the active channels.
//
// The outputs are cut into tiles of whole blocks of 32, one tile per SM, and a block streams the whole active list for its
// tile (few outputs of many channels: a cluster shares the list of a wider tile, see afx_q4op.cu).  A row's piece
// of a tile is its codes, 16 bytes per block of 32 outputs, and its scales; a thread takes W words of codes (8 W
// outputs) of every (NT / threads per piece)-th entry, five (W = 4) or four (W = 2) entries in flight (six and eight: 1 % more).
//
// What bounds it: the same chain of latencies as over 16-bit rows (afx_slice.cuh) and, while it streams, instruction
// issue: three per weight, of which codes to fp32 take 1.4 and the products 0.5.  (Over a whole launch, chain included,
// a gate | up operator of 4096 and 11008 channels issues in 40 % of its cycles, 4.5 instructions per weight.)  It replaced clusters of two blocks
// per SM that each selected over a shared-memory histogram, two thirds of all instructions; a layer of 4096 and 11008
// channels over 2048 positions, one token: 81 and 60 us.  Loading an entry's registers again as soon as it has been
// multiplied, instead of some entries together: 63.
#pragma once

#include "afx_onelist.cuh"
#include "afx_q4.cuh"

namespace afx {

constexpr int kQoSplit = 4;  // blocks that share a list
constexpr int kQoPad = 36;  // floats per (row set, block of 32 outputs) where the sums meet

// Widest tile in blocks of 32 outputs: one output per thread in the epilogue.
__host__ __device__ constexpr int q4op_max_blocks(int threads) { return threads / 32; }

// Dynamic shared memory: the staged list, later the sums; behind it the inputs of a list decided earlier.
// W = 4-byte words of codes per thread and row: a thread holds 8 W outputs.
__host__ __device__ inline size_t q4op_list_bytes(int threads, int W, int K) {
    const size_t list = (static_cast<size_t>(K) * 4 + 15) / 16 * 16;
    const size_t sums = static_cast<size_t>(threads) * W / 4 * kQoPad * 4 + static_cast<size_t>(threads) * 4;
    return list > sums ? list : sums;
}
__host__ __device__ inline size_t q4op_dyn_smem(int threads, int W, int K, bool list_given) {
    return q4op_list_bytes(threads, W, K) + (list_given ? (static_cast<size_t>(K) + 7) / 8 * 16 : 0);
}

template <int W>
struct Q4Raw {
    uint32_t w[W];
};
template <int W>
__device__ __forceinline__ Q4Raw<W> ld_codes(const unsigned char* p) {
    Q4Raw<W> r;
    if constexpr (W == 4) {
        const uint4 v = ld_stream_16B(p);
        r.w[0] = v.x;
        r.w[1] = v.y;
        r.w[2] = v.z;
        r.w[3] = v.w;
    } else {
        const uint2 v = ld_stream_8B(p);
        r.w[0] = v.x;
        r.w[1] = v.y;
    }
    return r;
}

// Streams list entries g, g + groups, .. below cnt: acc += x * scale * (code - 8) for the 8 W outputs of the W words
// at `codes` + channel * ldq, whose scale is at `scales` + channel * ldq.  acc: pairs of the low-nibble outputs, then
// of the high-nibble ones, in byte order.
template <int DT, int W, int U>
__device__ __forceinline__ void q4op_stream(const unsigned char* codes, const unsigned char* scales, uint64_t ldq, const uint32_t* list,
                                            int cnt, int g, int groups, f32x2 (&acc)[4 * W]) {
    auto consume = [&](const Q4Raw<W>& raw, uint16_t sc, uint32_t e) {
        const float s = list_x<DT>(e) * __half2float(__ushort_as_half(sc));
        const f32x2 s2 = pack_f32x2(s, s);
#pragma unroll
        for (int q = 0; q < W; ++q) {
            f32x2 a, b;
            nibbles_to_pairs(raw.w[q] & 0x0F0F0F0Fu, a, b);
            fma_f32x2(acc[2 * q], a, s2);
            fma_f32x2(acc[2 * q + 1], b, s2);
            nibbles_to_pairs((raw.w[q] >> 4) & 0x0F0F0F0Fu, a, b);
            fma_f32x2(acc[2 * W + 2 * q], a, s2);
            fma_f32x2(acc[2 * W + 2 * q + 1], b, s2);
        }
    };
    auto batch = [&](int p, bool guarded) {
        Q4Raw<W> raw[U];
        uint16_t sc[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (!guarded || p + u * groups < cnt) {
                const uint64_t off = (list[p + u * groups] & 0xFFFFu) * ldq;
                raw[u] = ld_codes<W>(codes + off);
                sc[u] = __ldg(reinterpret_cast<const uint16_t*>(scales + off));
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (!guarded || p + u * groups < cnt) consume(raw[u], sc[u], list[p + u * groups]);
    };
    int p = g;
    for (; p + (U - 1) * groups < cnt; p += U * groups) batch(p, false);
    if (p < cnt) batch(p, true);
}

// Tile u of a.slices is the blocks of 32 outputs [u n / slices, (u + 1) n / slices); the blocks of a cluster (SPLIT)
// share the list of one tile, each finishing every split-th output.
template <int DT, int NT, int NW, int CH, int W, int IN, int EP, bool SPLIT>
__device__ __forceinline__ void q4op_block(const FusedArgs& a, unsigned char* dyn, RegSelScratch* sc, float* recv) {
    constexpr int kPerBlock = 4 / W;  // threads per block of 32 outputs
    constexpr int U = W == 4 ? 5 : 4;
    const int tid = threadIdx.x;
    const int split = SPLIT ? static_cast<int>(cg::this_cluster().num_blocks()) : 1;
    const int rank = SPLIT ? static_cast<int>(cg::this_cluster().block_rank()) : 0;
    const int unit = static_cast<int>(blockIdx.x) / split, units = static_cast<int>(gridDim.x) / split;
    const bool scribe = a.side_cluster != 0 && unit == units - 1;  // selects only, writes the side outputs
    if (SPLIT) {
        if (scribe && rank != 0) return;
        if (!scribe) cluster_arrive();  // (the scribe's cluster never meets)
    }
    uint32_t* list = reinterpret_cast<uint32_t*>(dyn);
    AFX_TRACE_REGION(IN == IN_NORM ? (EP == EP_SILU ? 2 : 1) : (a.K > a.N ? 3 : 4));
    AFX_MARK(0);

    const int blocks = a.N / 32;
    const int b_lo = static_cast<int>(static_cast<int64_t>(unit) * blocks / a.slices);
    const int P = max(1, static_cast<int>(static_cast<int64_t>(unit + 1) * blocks / a.slices) - b_lo);  // <= q4op_max_blocks
    const int nout = P * 32, lanes = P * kPerBlock;
    const int rows = NT / lanes;  // list entries the block takes at once
    const int g = tid / lanes, piece = tid - g * lanes;

    const int cnt = one_token_list<DT, NT, NW, CH, IN>(a, a.x, false, scribe, dyn, q4op_list_bytes(NT, W, a.K), sc);
    if (scribe) {
        one_token_side_outputs<NT>(a, list, cnt, sc);
        return;
    }
    // the output this thread will add to (split: rank owns every split-th output of the tile)
    float y_old = 0.0f;
    const int mine = SPLIT ? tid * split + rank : tid;
    if (EP == EP_ACCUM && mine < nout) y_old = a.ep.y[b_lo * 32 + mine];

    f32x2 acc[4 * W];
#pragma unroll
    for (int i = 0; i < 4 * W; ++i) acc[i] = pack_f32x2(0.0f, 0.0f);
    const int c_lo = SPLIT ? rank * cnt / split : 0, c_hi = SPLIT ? (rank + 1) * cnt / split : cnt;
    if (g < rows) {
        const unsigned char* rows4 = reinterpret_cast<const unsigned char*>(a.Wt);
        q4op_stream<DT, W, U>(rows4 + b_lo * 16 + piece * (4 * W), rows4 + (a.N >> 1) + (b_lo + piece / kPerBlock) * 2,
                              static_cast<uint64_t>(a.ldw) * 2, list + c_lo, c_hi - c_lo, g, rows, acc);
    }
    AFX_MARK(5);

    // ---- the sums meet: row sets in shared memory, then the cluster's blocks in rank order ----
    __syncthreads();  // the list has been read
    AFX_MARK(6);
    float* red = reinterpret_cast<float*>(dyn);
    if (g < rows) {
        // bytes 4 W h .. of the block: outputs 4 W h .. (low nibbles) and 16 + 4 W h .. (high)
        float* at = red + (g * P + piece / kPerBlock) * kQoPad + (piece % kPerBlock) * (4 * W);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            float4 lo, hi;
            unpack_f32x2(acc[2 * i], lo.x, lo.y);
            unpack_f32x2(acc[2 * i + 1], lo.z, lo.w);
            unpack_f32x2(acc[2 * W + 2 * i], hi.x, hi.y);
            unpack_f32x2(acc[2 * W + 2 * i + 1], hi.z, hi.w);
            *reinterpret_cast<float4*>(at + 4 * i) = lo;
            *reinterpret_cast<float4*>(at + 16 + 4 * i) = hi;
        }
    }
    __syncthreads();
    float* red2 = red + NT * W / 4 * kQoPad;
    const int parts = NT / nout, part = tid / nout, out = tid - part * nout;
    if (part < parts) {
        const float* col = red + (out >> 5) * kQoPad + (out & 31);
        float sum = 0.0f;
#pragma unroll 4
        for (int r = part; r < rows; r += parts) sum += col[r * P * kQoPad];
        red2[tid] = sum;
    }
    __syncthreads();
    auto own = [&](int o) {
        float v = red2[o];
#pragma unroll 4
        for (int q = 1; q < parts; ++q) v += red2[q * nout + o];
        return v;
    };
    auto silu = [&](int pair, float gate, float up) {
        a.ep.out_bits[b_lo * 16 + pair] = float_to_bits<DT>(gate / (1.0f + expf(-gate)) * up);
    };
    if (SPLIT) {
        // output o goes to block o % split; a gate | up pair (16 apart inside a block of 32) to block pair % split
        const int per = EP == EP_SILU ? (nout / 2 + split - 1) / split * 2 : (nout + split - 1) / split;
        cluster_wait();  // the peers are running
        if (tid < nout) {
            const int pair = (tid >> 5) * 16 + (tid & 15);
            const int owner = EP == EP_SILU ? pair % split : tid % split;
            const int slot = EP == EP_SILU ? pair / split * 2 + ((tid >> 4) & 1) : tid / split;
            cg::this_cluster().map_shared_rank(recv, owner)[rank * per + slot] = own(tid);
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        auto total = [&](int slot) {
            float v = recv[slot];
            for (int q = 1; q < split; ++q) v += recv[q * per + slot];
            return v;
        };
        if (EP == EP_SILU) {
            if (mine < nout / 2) silu(mine, total(2 * tid), total(2 * tid + 1));
        } else if (mine < nout) {
            const float v = total(tid);
            a.ep.y[b_lo * 32 + mine] = EP == EP_ACCUM ? y_old + v : v;
        }
    } else if (EP == EP_SILU) {
        if (tid < nout / 2) {
            const int o = (tid >> 4) * 32 + (tid & 15);
            silu(tid, own(o), own(o + 16));
        }
    } else if (tid < nout) {
        const float v = own(tid);
        a.ep.y[b_lo * 32 + tid] = EP == EP_ACCUM ? y_old + v : v;
    }
    AFX_MARK(7);
}

}  // namespace afx
