// Sparse GEMV of 2 to 8 tokens over an active-channel list, on the tensor cores without a trip through shared memory.
//
// D[outputs][tokens] = W^T[outputs][channels] . X[channels][tokens], a dense contraction over the ACTIVE channels.  The
// fragments of `mma` hold neighbouring channels in one register, memory holds neighbouring outputs; a lane therefore
// loads the same 16 bytes (8 outputs) of four list entries and pairs their halves with two byte permutes per two
// words, which gives it the A fragments of four tiles of 16 outputs:
//   granule of 64 outputs, step of 16 list entries; lane = 4 g + t: piece g of the entries 4 t .. 4 t + 3;
//   tile j (0..3): rows r < 8 are outputs 8 r + 2 j, rows r + 8 outputs 8 r + 2 j + 1.
// Which entries of a step stand for which k of the product is free, as long as the B fragment (the inputs of token g at the
// entries 4 t ..) agrees.  Products of two 16-bit floats are exact; the sums are fp32 inside the tensor core, in a
// fixed order: the same inputs give the same bits.
//
// A cluster of S blocks owns a tile of up to kMlMaxGranules granules and splits the active list; the warps of a
// block take a granule each and share its part of the list.
//
// What bounds it: HBM.  A warp has one step in flight, 2 KB; 32 warps per SM that drift apart keep the loads coming.  Two
// steps per warp, together or one ahead of the other, cost registers that 64 do not hold (5120 -> 27648, four tokens: 57
// to 68 us; with one block per SM and 128 registers 55 to 70; one step 47).  It replaced stages of 16 channels
// in shared memory (cp.async, ldmatrix.trans, a block barrier per stage): four tokens 5120 -> 27648 53.6 and 47.1 us,
// 5120 -> 5120 16.9 and 14.5, 13824 -> 5120 33.1 and 29.1, 5120 -> 15360 (4096 entries) 27.5 and 27.8; eight tokens
// 5120 -> 27648 61.8 and 53.7; two tokens 8192 -> 57344 132.7 and 122.8; three tokens 5003 -> 7208 17.4 and 15.7.  It
// loses where few channels meet many outputs, whose blocks have little to stream beside the sums of many granules: eight
// tokens 2048 -> 20480 17.4 and 19.9, 1024 -> 20480 12.1 and 14.3.
#pragma once

#include "afx_gemv.cuh"
#include "afx_mma.cuh"

namespace afx {

constexpr int kMlGranule = 64;       // outputs a warp works on
constexpr int kMlMaxGranules = 8;    // of a tile
constexpr int kMlMaxCluster = 16;
constexpr int kMlCap = 2048;         // staged list entries per pass
constexpr int kMlXStride = kMlCap + 16;  // (32 bytes more per token: 8-byte reads of a warp in two passes)
constexpr int kMlRedStride = 72;     // floats per (warp, token) where the sums meet: 8-byte stores without conflicts

__host__ __device__ inline size_t ml_stage_bytes(int T) {
    const size_t stage = static_cast<size_t>(kMlCap) * 4 + static_cast<size_t>(T) * kMlXStride * 2;
    const size_t red = static_cast<size_t>(kGemvWarps) * T * kMlRedStride * 4;
    return stage > red ? stage : red;
}
// rows of 64 sums (token, granule) that one block of the cluster finishes
__host__ __device__ inline int ml_rows_per_block(int T, int granules, int S) { return (T * granules + S - 1) / S; }
__host__ __device__ inline size_t ml_dyn_smem(int T, int granules, int S) {
    return ml_stage_bytes(T) + static_cast<size_t>(S) * ml_rows_per_block(T, granules, S) * kMlGranule * 4;
}

// Steps st, st + stride, .. below n_steps of the staged entries [0, staged): c[j] += tile j.
template <int DT>
__device__ __forceinline__ void ml_stream(const unsigned char* base, const uint32_t* col, const uint16_t* x, bool has_token, bool has_piece,
                                          int staged, int st, int stride, float (&c)[4][4]) {
    const int tig = lane_id() & 3;
    const int n_steps = (staged + 15) >> 4;
    auto load = [&](int s, bool guarded, uint4 (&raw)[4]) {
        const int p = 16 * s + 4 * tig;
        const uint4 at = *reinterpret_cast<const uint4*>(col + p);
        const uint32_t r[4] = {at.x, at.y, at.z, at.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (guarded) raw[e] = make_uint4(0u, 0u, 0u, 0u);
            if (!guarded || (has_piece && p + e < staged)) raw[e] = ld_stream_16B(base + static_cast<uint64_t>(r[e]) * 16u);
        }
    };
    auto multiply = [&](int s, const uint4 (&raw)[4]) {
        uint2 b = make_uint2(0u, 0u);
        if (has_token) b = *reinterpret_cast<const uint2*>(x + 16 * s + 4 * tig);
        const uint32_t w[4][4] = {{raw[0].x, raw[0].y, raw[0].z, raw[0].w}, {raw[1].x, raw[1].y, raw[1].z, raw[1].w},
                                  {raw[2].x, raw[2].y, raw[2].z, raw[2].w}, {raw[3].x, raw[3].y, raw[3].z, raw[3].w}};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t a[4] = {__byte_perm(w[0][j], w[1][j], 0x5410), __byte_perm(w[0][j], w[1][j], 0x7632),
                                   __byte_perm(w[2][j], w[3][j], 0x5410), __byte_perm(w[2][j], w[3][j], 0x7632)};
            mt_mma<DT>(c[j], a, b.x, b.y);
        }
    };
    const int full = __all_sync(0xFFFFFFFFu, has_piece) ? staged >> 4 : 0;  // steps whose loads need no guard
    int s = st;
    for (; s < full; s += stride) {
        uint4 raw[4];
        load(s, false, raw);
        multiply(s, raw);
    }
#pragma unroll 1
    for (; s < n_steps; s += stride) {
        uint4 raw[4];
        load(s, true, raw);
        multiply(s, raw);
    }
}

// grid = (S, tiles), cluster = (S, 1, 1), 512 threads.
template <int DT>
__device__ __forceinline__ void mt_list_block(const GemvListArgs& a, unsigned char* dyn) {
    cg::cluster_group cluster = cg::this_cluster();
    const int S = gridDim.x, rank = blockIdx.x, tile = blockIdx.y, T = a.T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    cluster_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (ordering rule of the library)
    int cnt = *a.count;
    if (cnt < 0 || cnt > a.K) {
        if (tid == 0 && rank == 0 && tile == 0) report_status(a.status, AFX_ERR_CAPACITY);
        cnt = max(0, min(cnt, a.K));
    }
    const int c_lo = static_cast<int>(static_cast<int64_t>(rank) * cnt / S);
    const int c_hi = static_cast<int>(static_cast<int64_t>(rank + 1) * cnt / S);
    const uint64_t ld16 = static_cast<uint64_t>(a.ldw >> 3);
    // this tile's granules; a warp's granule and its share of the list
    const int all_granules = (a.N + kMlGranule - 1) / kMlGranule;
    const int g_lo = static_cast<int>(static_cast<int64_t>(tile) * all_granules / gridDim.y);
    const int G = static_cast<int>(static_cast<int64_t>(tile + 1) * all_granules / gridDim.y) - g_lo;  // 1 .. kMlMaxGranules
    const int subs = kGemvWarps / G, sub = warp / G, gr = warp - sub * G;
    const int gid = lane >> 2;
    const int out0 = (g_lo + gr) * kMlGranule + gid * 8;
    const bool has_piece = out0 < a.N;
    const unsigned char* base = reinterpret_cast<const unsigned char*>(a.Wt + (has_piece ? out0 : 0));

    uint32_t* col = reinterpret_cast<uint32_t*>(dyn);
    uint16_t* xb = reinterpret_cast<uint16_t*>(dyn + static_cast<size_t>(kMlCap) * 4);
    float c[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[j][i] = 0.0f;
    __shared__ int first_ok;

    for (int c0 = c_lo; c0 < c_hi; c0 += kMlCap) {
        int staged = min(kMlCap, c_hi - c0);
        __syncthreads();  // the previous pass has been multiplied
        bool skipped = false;
        for (int i = tid; i < staged; i += kGemvThreads) {
            // as in the fp32 kernel: an entry outside [0, K) or with a negative cache slot takes no part
            const int j = a.idx[c0 + i];
            const int cl = a.slot != nullptr ? a.slot[c0 + i] : j;
            const bool in_range = static_cast<unsigned>(j) < static_cast<unsigned>(a.K);
            const uint64_t off = static_cast<uint64_t>(cl < 0 ? 0 : cl) * ld16;
            const bool ok = in_range && cl >= 0 && row_offset_fits(off);
            if (!ok && tile == 0) report_status(a.status, in_range ? AFX_ERR_CAPACITY : AFX_ERR_INVALID_ARG);
            skipped |= !ok;
            col[i] = ok ? static_cast<uint32_t>(off) : kSkippedEntry;
            for (int t = 0; t < T; ++t) xb[t * kMlXStride + i] = ok ? a.x[static_cast<size_t>(t) * a.K + j] : uint16_t(0);
        }
        for (int i = staged + tid; i < (staged + 15) / 16 * 16; i += kGemvThreads)  // inputs of the last step's missing entries
            for (int t = 0; t < T; ++t) xb[t * kMlXStride + i] = 0;
        if (__syncthreads_or(skipped)) {  // rare: a skipped entry reads the row of one that takes part (x = 0)
            if (tid == 0) first_ok = staged;
            __syncthreads();
            for (int i = tid; i < staged; i += kGemvThreads)
                if (col[i] != kSkippedEntry) atomicMin(&first_ok, i);
            __syncthreads();
            const int f = first_ok;
            if (f < staged) {
                const uint32_t safe = col[f];
                __syncthreads();
                for (int i = tid; i < staged; i += kGemvThreads)
                    if (col[i] == kSkippedEntry) col[i] = safe;
            } else {
                staged = 0;
            }
            __syncthreads();
        }
        if (sub < subs) ml_stream<DT>(base, col, xb + min(gid, T - 1) * kMlXStride, gid < T, has_piece, staged, sub, subs, c);
    }

    // ---- the sums meet: warps of a granule, then the cluster's blocks in rank order ----
    __syncthreads();  // the staged entries have been read
    float* red = reinterpret_cast<float*>(dyn);
    if (sub < subs) {
        const int t0 = 2 * (lane & 3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // output 8 g + 2 j + h of the granule at place 16 j + 2 g + h
            float* at = red + (warp * T + t0) * kMlRedStride + 16 * j + 2 * gid;
            if (t0 < T) *reinterpret_cast<float2*>(at) = make_float2(c[j][0], c[j][2]);
            if (t0 + 1 < T) *reinterpret_cast<float2*>(at + kMlRedStride) = make_float2(c[j][1], c[j][3]);
        }
    }
    float* recv = reinterpret_cast<float*>(dyn + ml_stage_bytes(T));
    const int per = ml_rows_per_block(T, G, S);
    // the value that this thread's first output is added to, long before it is
    const int mine = tid >> 6, place = tid & 63;
    const int o_in = 8 * ((place >> 1) & 7) + 2 * (place >> 4) + (place & 1);
    auto output = [&](int r) { return (g_lo + r % G) * kMlGranule + o_in; };
    float y_old = 0.0f;
    {
        const int r = mine * S + rank;
        if (a.accumulate && r < T * G && output(r) < a.N) y_old = a.ep.y[static_cast<size_t>(r / G) * a.N + output(r)];
    }
    cluster_wait();  // the peers are running (and every warp's sums are in place)
    __syncthreads();
    for (int r = mine; r < T * G; r += kGemvThreads / kMlGranule) {
        const float* at = red + ((r % G) * T + r / G) * kMlRedStride + place;
        float v = 0.0f;
        for (int q = 0; q < subs; ++q) v += at[q * G * T * kMlRedStride];
        float* to = S > 1 ? cluster.map_shared_rank(recv, r % S) : recv;
        to[(rank * per + r / S) * kMlGranule + place] = v;
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    const float scale = !a.silu && a.ep.scale != nullptr ? *a.ep.scale : 1.0f;
    for (int i = mine; i < per; i += kGemvThreads / kMlGranule) {
        const int r = i * S + rank;
        if (r >= T * G) break;
        const int t = r / G, out = output(r);
        const float* at = recv + i * kMlGranule + place;
        float v = 0.0f;
        for (int q = 0; q < S; ++q) v += at[q * per * kMlGranule];
        if (a.silu) {
            // pieces in pairs, gate then up: the up output is two places on
            const float up = __shfl_down_sync(0xFFFFFFFFu, v, 2);
            if (((place >> 1) & 1) == 0 && out < a.N)
                a.ep.out_bits[static_cast<size_t>(t) * (a.N / 2) + (out >> 4) * 8 + (out & 7)] = float_to_bits<DT>(v / (1.0f + expf(-v)) * up);
        } else if (out < a.N) {
            float* p = a.ep.y + static_cast<size_t>(t) * a.N + out;
            v *= scale;
            *p = a.accumulate ? (i == mine ? y_old : *p) + v : v;
        }
    }
}

}  // namespace afx
