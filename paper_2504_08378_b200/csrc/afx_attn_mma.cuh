// Dense single-query attention over an fp16 KV cache for one decoding step (support op of
// the decoder layer; the paper keeps attention dense and so does this kernel).
//
// grid = (S, kv_heads, T), cluster = (S,1,1): the S blocks of a cluster split the past positions of one
// (token, kv head) in tiles of 16, a warp takes every NW-th tile of its block.  A tile is two matrix
// products on the tensor cores, whose operands come straight from 16-byte global loads:
//   scores[head][position] = Q . K^T   (16 x 8 x 16 products: a lane loads the row of ONE position)
//   O[head][dim]          += P . V     (a lane loads the same 8 dims of four positions and pairs them up)
// The 16 rows of a product are the up to 8 query heads of the kv head twice: the high and the low half
// of their fp32 values (two fp16 numbers, within 2^-23), so that neither the queries nor the
// probabilities lose the precision of the fp32 pipe; both are scaled by powers of two into fp16's range.
// Softmax is online and in base 2.  The warps of a block and the blocks of a cluster meet in a fixed
// order.  head_dim is fixed at 128.
//
// 16 positions cost a warp 8 KB of K and V and about 200 instructions whatever the number of query heads,
// where dot products on the fp32 pipe cost 45 instructions per position and query head (64 heads, kv 8, 8000
// positions: 100 -> 15.7 us, and 0.7 since the scores are summed on the fp32 pipe).  Bound by the latency of a warp's tile of loads: one block of 8 warps per SM
// with a whole tile of K and V in flight each (206 registers) beats two or three blocks of 4 (23.8, 43.2 us).
#pragma once

#include "afx_attn.cuh"

namespace afx {

constexpr int kAttnMaxCluster = 16;  // blocks per cluster (above 8: where few kv heads leave SMs idle)
constexpr int kAttnMmaWarps = 8;
constexpr int kAttnMmaThreads = kAttnMmaWarps * 32;
constexpr int kAttnTile = 16;        // positions
constexpr int kAttnQRow = 160;       // fp16 values per staged query row (128 + padding: no bank conflicts)

struct AttnMmaSmem {
    __align__(16) uint16_t q_hi[kAttnMaxRep][kAttnQRow];  // rotated queries times scale * log2(e), times 1 / q_unit
    __align__(16) uint16_t q_lo[kAttnMaxRep][kAttnQRow];
    float q_unit[kAttnMaxRep];                            // power of two
    __align__(16) float acc[kAttnMmaWarps + 1][kAttnMaxRep][kHeadDim];  // the warps' partial outputs; the last one: the new position
    float m[kAttnMmaWarps + 1][kAttnMaxRep];
    float l[kAttnMmaWarps + 1][kAttnMaxRep];
    // the cluster's partials, pushed by its blocks: every S-th value of the heads, and what goes with them
    float recv_acc[kAttnMaxRep * kHeadDim + kAttnMaxCluster];
    float recv_m[kAttnMaxCluster][kAttnMaxRep];
    float recv_l[kAttnMaxCluster][kAttnMaxRep];
};

// c += A . B, 16 x 8 x 16, fp16 in, fp32 out
__device__ __forceinline__ void attn_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the pair (a, b) as fp16, and what that rounding left out as fp16
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
    hi = pack2_bits<AFX_F16>(a, b);
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hi));
    lo = pack2_bits<AFX_F16>(a - f.x, b - f.y);
}

// A product's sums of the high and the low halves.  An infinity in the cache makes the high one what the product is
// (infinite, or NaN); the low one may then be of the other sign, or 0 times infinity, and says nothing.
__device__ __forceinline__ float whole(float hi, float lo) { return fabsf(hi) <= 3.402823466e38f ? hi + lo : hi; }

template <int DT>
__device__ __forceinline__ void attention_mma_block(const AttnArgs& a, AttnMmaSmem* sm) {
    constexpr int NW = kAttnMmaWarps, NT = kAttnMmaThreads;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = static_cast<int>(cluster.num_blocks());
    const int rank = static_cast<int>(cluster.block_rank());
    const int hk = blockIdx.y, t = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gid = lane >> 2, tig = lane & 3;
    const int rep = a.q_heads / a.kv_heads;
    const int tiles = (a.pos + 15) >> 4;  // of past positions; the new one is apart
    const int t_lo = static_cast<int>(static_cast<int64_t>(rank) * tiles / S);
    const int t_hi = static_cast<int>(static_cast<int64_t>(rank + 1) * tiles / S);
    const bool newest = rank == S - 1;  // this block also takes (and stores) the new position

    AFX_TRACE_REGION(0);
    AFX_MARK(0);
    cluster_arrive();
    const size_t row_stride = static_cast<size_t>(a.kv_heads) * kHeadDim;
    uint16_t* kc = a.k_cache + (static_cast<size_t>(t) * a.max_seq * a.kv_heads + hk) * kHeadDim;
    uint16_t* vc = a.v_cache + (static_cast<size_t>(t) * a.max_seq * a.kv_heads + hk) * kHeadDim;

    // Key rows behind the last past position are read as the last one, and their scores masked below; value rows are
    // zero there (a probability of 0 times an infinity of the last row would be NaN).
    uint4 kr[2][4], vr[2][2][2];
    auto row_of = [&](int p) { return static_cast<size_t>(min(p, a.pos - 1)) * row_stride; };
    auto fetch_k = [&](int tile) {  // tile half h: the lane's position 8 h + gid, 16-byte pieces 4 j + tig
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4* r = reinterpret_cast<const uint4*>(kc + row_of(tile * 16 + 8 * h + gid));
#pragma unroll
            for (int j = 0; j < 4; ++j) kr[h][j] = r[4 * j + tig];
        }
    };
    auto fetch_v = [&](int tile) {  // tile half h: positions 8 h + 2 tig + e, dims 64 q + 8 gid .. + 7
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int p = tile * 16 + 8 * h + 2 * tig + e;
                const uint4* r = reinterpret_cast<const uint4*>(vc + row_of(p));
#pragma unroll
                for (int q = 0; q < 2; ++q) vr[h][e][q] = p < a.pos ? r[8 * q + gid] : make_uint4(0u, 0u, 0u, 0u);
            }
    };
    // Inside a layer step the first tile's rows are requested before the wait for q, k, v.
    const bool any = t_lo + warp < t_hi;
    if (any && a.past_final) {
        fetch_k(t_lo + warp);
        fetch_v(t_lo + warp);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // only after the wait (see fused_op_block)
    AFX_MARK(1);
    if (any && !a.past_final) {
        fetch_k(t_lo + warp);
        fetch_v(t_lo + warp);
    }

    const float* row = a.qkv + static_cast<size_t>(t) * a.n_qkv;
    const float2* cs = reinterpret_cast<const float2*>(a.rope_cos + static_cast<size_t>(a.pos) * (kHeadDim / 2));
    const float2* sn = reinterpret_cast<const float2*>(a.rope_sin + static_cast<size_t>(a.pos) * (kHeadDim / 2));
    const float qscale = rsqrtf(static_cast<float>(kHeadDim)) * 1.4426950408889634f;
    // A lane owns dims 4 lane .. + 3 (rotary pairs 2 lane, 2 lane + 1).
    const float2 c2 = cs[lane], s2 = sn[lane];
    auto rotated = [&](const float* head, float (&v)[4]) {
        const float4 x = reinterpret_cast<const float4*>(head)[lane];
        v[0] = x.x * c2.x - x.y * s2.x;
        v[1] = x.x * s2.x + x.y * c2.x;
        v[2] = x.z * c2.y - x.w * s2.y;
        v[3] = x.z * s2.y + x.w * c2.y;
    };
    float kn[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // the new position's key as the cache stores it
    uint2 kb = make_uint2(0u, 0u);
    if (newest) {
        float v[4];
        rotated(row + static_cast<size_t>(a.q_heads + hk) * kHeadDim, v);
        kb = make_uint2(pack2_bits<AFX_F16>(v[0], v[1]), pack2_bits<AFX_F16>(v[2], v[3]));
        const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&kb.x));
        const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&kb.y));
        kn[0] = f0.x;
        kn[1] = f0.y;
        kn[2] = f1.x;
        kn[3] = f1.y;
    }
    for (int r = warp; r < kAttnMaxRep; r += NW) {
        uint2 hi = make_uint2(0u, 0u), lo = make_uint2(0u, 0u);
        if (r < rep) {
            float q[4];
            rotated(row + static_cast<size_t>(hk * rep + r) * kHeadDim, q);
            float big = 0.0f, dot = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                q[i] *= qscale;
                big = fmaxf(big, fabsf(q[i]));
                dot = fmaf(q[i], kn[i], dot);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xFFFFFFFFu, big, o));
            // the head's largest value lands in [2^9, 2^10); exponents are kept away from the ends of fp32's range
            const int e = min(max(static_cast<int>((__float_as_uint(big) >> 23) & 0xFFu) - 127, -100), 110);
            const float up = __uint_as_float(static_cast<uint32_t>(127 + 9 - e) << 23);
            split_pair(q[0] * up, q[1] * up, hi.x, lo.x);
            split_pair(q[2] * up, q[3] * up, hi.y, lo.y);
            if (newest) dot = warp_sum(dot);
            if (lane == 0) {
                sm->q_unit[r] = __uint_as_float(static_cast<uint32_t>(127 - 9 + e) << 23);
                sm->m[NW][r] = newest ? dot : -INFINITY;
                sm->l[NW][r] = newest ? 1.0f : 0.0f;
            }
            // (its value rows count once per query head)
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (newest) {
                const float4 x = reinterpret_cast<const float4*>(row + static_cast<size_t>(a.q_heads + a.kv_heads + hk) * kHeadDim)[lane];
                const uint2 vb = make_uint2(pack2_bits<AFX_F16>(x.x, x.y), pack2_bits<AFX_F16>(x.z, x.w));
                const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&vb.x));
                const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&vb.y));
                v = make_float4(f0.x, f0.y, f1.x, f1.y);
                if (r == 0) {
                    reinterpret_cast<uint2*>(kc + static_cast<size_t>(a.pos) * row_stride)[lane] = kb;
                    reinterpret_cast<uint2*>(vc + static_cast<size_t>(a.pos) * row_stride)[lane] = vb;
                }
            }
            reinterpret_cast<float4*>(sm->acc[NW][r])[lane] = v;
        } else if (lane == 0) {
            sm->q_unit[r] = 0.0f;
        }
        reinterpret_cast<uint2*>(sm->q_hi[r])[lane] = hi;
        reinterpret_cast<uint2*>(sm->q_lo[r])[lane] = lo;
    }
    __syncthreads();
    AFX_MARK(2);

    // Probabilities are carried times 2^10: an exact product.  (10 added to the exponent instead would round them to 2^-21.)
    constexpr float kUp = 1024.0f;
    float m_run = -INFINITY, l_run = 0.0f;  // of query head gid (l: this lane's positions)
    float o[2][8][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int x = 0; x < 4; ++x) o[q][i][x] = 0.0f;
    const float unit = sm->q_unit[gid];

    for (int tile = t_lo + warp; tile < t_hi; tile += NW) {
        float s[2][2];
        {
            float c[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 qh = reinterpret_cast<const uint4*>(sm->q_hi[gid])[4 * j + tig];
                const uint4 ql = reinterpret_cast<const uint4*>(sm->q_lo[gid])[4 * j + tig];
                const uint32_t a0[4] = {qh.x, ql.x, qh.y, ql.y}, a1[4] = {qh.z, ql.z, qh.w, ql.w};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // Sums of 32 products leave the tensor core, which truncates what it adds, and are rounded together here
                    // (f16 outputs that are not the nearest ones, q ~ N(0, 1): 1.1e-3, with chains of 128 products
                    // 1.5e-3, on the fp32 pipe 1.2e-3; 8 kv heads of 8, 8000 positions: 17.0 us, with chains 16.4).
                    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    attn_mma(d, a0, kr[h][j].x, kr[h][j].y);
                    attn_mma(d, a1, kr[h][j].z, kr[h][j].w);
#pragma unroll
                    for (int x = 0; x < 4; ++x) c[h][x] += d[x];
                }
            }
            if (tile + NW < t_hi) fetch_k(tile + NW);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    s[h][e] = tile * 16 + 8 * h + 2 * tig + e < a.pos ? whole(c[h][e], c[h][2 + e]) * unit : -INFINITY;
        }
        float mn = fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1]));
        mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 1));
        mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 2));
        mn = fmaxf(mn, m_run);  // (-inf while every score has been)
        const float ref = mn == -INFINITY ? 0.0f : mn;
        if (__any_sync(0xFFFFFFFFu, mn > m_run)) {
            const float f = fast_exp2(m_run - ref);  // 0 on the first visit (m_run = -inf)
            m_run = mn;
            l_run *= f;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int x = 0; x < 4; ++x) o[q][i][x] *= f;
        }
        uint32_t p[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float p0 = fast_exp2(s[h][0] - ref) * kUp, p1 = fast_exp2(s[h][1] - ref) * kUp;
            l_run += p0 + p1;
            split_pair(p0, p1, p[2 * h], p[2 * h + 1]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t w00[4] = {vr[0][0][q].x, vr[0][0][q].y, vr[0][0][q].z, vr[0][0][q].w};
            const uint32_t w01[4] = {vr[0][1][q].x, vr[0][1][q].y, vr[0][1][q].z, vr[0][1][q].w};
            const uint32_t w10[4] = {vr[1][0][q].x, vr[1][0][q].y, vr[1][0][q].z, vr[1][0][q].w};
            const uint32_t w11[4] = {vr[1][1][q].x, vr[1][1][q].y, vr[1][1][q].z, vr[1][1][q].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                attn_mma(o[q][2 * i], p, __byte_perm(w00[i], w01[i], 0x5410), __byte_perm(w10[i], w11[i], 0x5410));
                attn_mma(o[q][2 * i + 1], p, __byte_perm(w00[i], w01[i], 0x7632), __byte_perm(w10[i], w11[i], 0x7632));
            }
        }
        if (tile + NW < t_hi) fetch_v(tile + NW);
    }
    AFX_MARK(3);

    // this warp's partial: query head gid, dims 64 q + 16 tig + 8 c + i
    l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 1);
    l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 2);
    if (gid < rep) {
        if (tig == 0) {
            sm->m[warp][gid] = m_run;
            sm->l[warp][gid] = l_run * (1.0f / kUp);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float4* d = reinterpret_cast<float4*>(&sm->acc[warp][gid][64 * q + 16 * tig + 8 * c]);
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = whole(o[q][i][c], o[q][i][2 + c]) * (1.0f / kUp);
                d[0] = make_float4(v[0], v[1], v[2], v[3]);
                d[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
    }
    __syncthreads();
    // Block e % S of the cluster finishes value e of the heads: the partial sums are pushed there, behind one cluster barrier.
    const int per = (rep * kHeadDim + S - 1) / S;
    cluster_wait();  // the peers are running
    for (int e = tid; e < rep * kHeadDim; e += NT) {
        const int r = e / kHeadDim, d = e - r * kHeadDim;
        float M = -INFINITY;
#pragma unroll
        for (int g = 0; g <= NW; ++g) M = fmaxf(M, sm->m[g][r]);
        float acc = 0.0f, l = 0.0f;
#pragma unroll
        for (int g = 0; g <= NW; ++g) {
            // a warp that saw no position has m = -inf, l = 0, acc = 0
            const float w = sm->m[g][r] == -INFINITY ? 0.0f : fast_exp2(sm->m[g][r] - M);
            acc = fmaf(w, sm->acc[g][r][d], acc);
            l = fmaf(w, sm->l[g][r], l);
        }
        cluster.map_shared_rank(&sm->recv_acc[0], e % S)[rank * per + e / S] = acc;
        if (d < S) {
            cluster.map_shared_rank(&sm->recv_m[0][0], d)[rank * kAttnMaxRep + r] = M;
            cluster.map_shared_rank(&sm->recv_l[0][0], d)[rank * kAttnMaxRep + r] = l;
        }
    }
    AFX_MARK(4);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    AFX_MARK(5);
    for (int i = tid; rank + S * i < rep * kHeadDim; i += NT) {
        const int e = rank + S * i, r = e / kHeadDim, d = e - r * kHeadDim;
        // the merge in block order
        float M = -INFINITY;
        for (int q = 0; q < S; ++q) M = fmaxf(M, sm->recv_m[q][r]);
        float num = 0.0f, den = 0.0f;
        for (int q = 0; q < S; ++q) {
            const float w = sm->recv_m[q][r] == -INFINITY ? 0.0f : fast_exp2(sm->recv_m[q][r] - M);
            num = fmaf(w, sm->recv_acc[q * per + i], num);
            den = fmaf(w, sm->recv_l[q][r], den);
        }
        a.out[static_cast<size_t>(t) * a.q_heads * kHeadDim + static_cast<size_t>(hk * rep + r) * kHeadDim + d] =
            float_to_bits<DT>(num / den);
    }
    AFX_MARK(7);
}

}  // namespace afx
