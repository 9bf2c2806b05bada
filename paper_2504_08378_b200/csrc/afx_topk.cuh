// Active-channel selection with the keys in registers.
//
// The first NW warps of the block own the channels: slot s of warp w holds channels (w m + s) 128 + 4
// lane .. + 3.  The k-th largest 15-bit magnitude key is found by a seven-way search: a step counts the
// keys at or above six candidates (two keys per operation), adds the counts over warp and block (three
// `redux` before and three shuffles behind one barrier of the NW warps) and keeps a seventh of the interval.
// With a hint of the answer two steps suffice in bf16 and three in f16; without one a sample of the keys gives it.  There are no
// atomics and no histogram, hence no shared memory to clear and no serialisation on popular keys.
//
// What bounds it is the issue rate of integer instructions and the latency of a step's barrier and
// reductions.  What every warp repeats behind the barrier counts NW times, so few warps with many keys
// each beat many warps with few: K = 4096, bf16, hinted: 1.3 us for the search on 8 warps of 16 keys per
// lane; 2.2 us where all 32 warps of an SM's two blocks searched a histogram of the same keys.
#pragma once

#include "afx_select.cuh"

namespace afx {

constexpr uint32_t kNoHint = 0xFFFFFFFFu;
constexpr int kRegSelMaxWarps = 32;

struct RegSelScratch {
    __align__(16) uint32_t part[2][kRegSelMaxWarps][4];  // per-warp counts of a search step (double-buffered)
    uint32_t scan[kRegSelMaxWarps];
    int count;      // the list's length, for the warps that did not select
    uint32_t hint;  // where the search starts (sel_read_hint)
    __align__(16) float sum[kRegSelMaxWarps];
};

// Barrier of the block's first NW warps.
template <int NW>
__device__ __forceinline__ void sel_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory");
}

// The search hint in `slot` (NULL: none) for the whole block: ONE thread of the first warp reads it and leaves it in
// sc->hint, which the others read behind a barrier of the selecting warps.  Another launch of the operator, or
// another block of this one, may be rewriting the word: threads that read it for themselves could start with
// different hints, take different numbers of search steps, and wait at different barriers for each other.
__device__ __forceinline__ void sel_read_hint(const int32_t* slot, RegSelScratch* sc) {
    if (threadIdx.x == 0) {
        const uint32_t v = slot != nullptr ? static_cast<uint32_t>(__ldcg(slot)) : 0u;
        sc->hint = (v & 0x10000u) ? v & 0x7FFFu : kNoHint;
    }
}

// Slots per lane for K channels on NW warps.
template <int NW>
__device__ __forceinline__ int sel_slots(int K) { return (K + NW * 128 - 1) / (NW * 128); }
// First channel of slot s of the calling lane.
__device__ __forceinline__ int sel_channel(int m, int s) { return (warp_id() * m + s) * 128 + 4 * lane_id(); }

// The lane's channels of a 16-bit vector in global memory: word 2s = the first two channels of slot s,
// word 2s+1 = the next two; zero behind K.
template <int CH>
__device__ __forceinline__ void sel_load_keys(const uint16_t* x, int K, int m, uint32_t (&kw)[2 * CH]) {
    const bool wide = (reinterpret_cast<uintptr_t>(x) & 7u) == 0;
#pragma unroll
    for (int s = 0; s < CH; ++s) {
        kw[2 * s] = 0u;
        kw[2 * s + 1] = 0u;
        const int j = sel_channel(m, s);
        if (s < m && j < K) {
            if (wide && j + 4 <= K) {
                const uint2 v = *reinterpret_cast<const uint2*>(x + j);
                kw[2 * s] = v.x;
                kw[2 * s + 1] = v.y;
            } else {
                uint32_t b[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) b[e] = j + e < K ? x[j + e] : 0u;
                kw[2 * s] = b[0] | (b[1] << 16);
                kw[2 * s + 1] = b[2] | (b[3] << 16);
            }
        }
    }
}

// 1 in each half whose 15-bit key is >= v (nv = both halves 1 - v, v in 1..32768).
__device__ __forceinline__ uint32_t sel_ge(uint32_t keys, uint32_t nv) {
    return __viaddmin_s16x2_relu(keys, nv, 0x00010001u);
}
__device__ __forceinline__ uint32_t sel_neg(int v) { return (static_cast<uint32_t>(1 - v) & 0xFFFFu) * 0x00010001u; }
constexpr uint32_t kMagnitudes = 0x7FFF7FFFu;

// The k-th largest key (1 <= k <= K) of the NW warps' channels: `thr`; how many channels with exactly
// that key belong to the top k: `need_eq`.  Same values in every thread.  `hint` only shortens the
// search.  Zero padding behind K is never counted (candidates are >= 1).
template <int DT, int NW, int CH>
__device__ __forceinline__ void sel_kth_key(const uint32_t (&kw)[2 * CH], int m, int K, int k, uint32_t hint, RegSelScratch* sc,
                                            int& thr, int& need_eq) {
    constexpr int C = 6;
    // first step: candidates this far apart around the hint: +-17 keys (about +-13 % in magnitude) in
    // bf16, +-122 (+-12 to 24 %) in f16; successive tokens' keys for one operator lie within a few percent
    constexpr int D = DT == AFX_BF16 ? 7 : 49;
    const int lane = lane_id(), warp = warp_id();
    int lo = 0, hi = 32768, above = 0;  // count(keys >= lo) >= k > count(keys >= hi) = above
    int base = 4682, stride = 4682, stage = 2;
    if (hint == kNoHint && K >= 128 * m * 4) {
        // No hint: every warp that is full takes the like order statistic of one key per lane, and their mean is
        // the hint (500 samples at 16 warps: within 2 % of the rank).
        const uint32_t v = kw[0] & 0x7FFFu;
        const int r = max(1, min(32, (32 * k + K / 2) / K));
        uint32_t est = 0;
#pragma unroll
        for (int b = 14; b >= 0; --b) {
            const uint32_t c = est | (1u << b);
            if (__popc(__ballot_sync(0xFFFFFFFFu, v >= c)) >= r) est = c;
        }
        if (lane == 0) sc->scan[warp] = (warp + 1) * m * 128 <= K ? est : kNoHint;
        sel_barrier<NW>();
        const uint32_t e = lane < NW ? sc->scan[lane] : kNoHint;
        const uint32_t full = __popc(__ballot_sync(0xFFFFFFFFu, e != kNoHint));  // >= 4
        hint = __reduce_add_sync(0xFFFFFFFFu, e != kNoHint ? e : 0u) / full;
    }
    if (hint != kNoHint) {
        base = static_cast<int>(hint) - 5 * D / 2;
        stride = D;
        stage = 0;
    }
    for (int it = 0;; ++it) {
        int cand[C];
        uint32_t nv[C], n[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            cand[j] = max(lo + 1, min(base + j * stride, hi));
            nv[j] = sel_neg(cand[j]);
            n[j] = 0;
        }
#pragma unroll
        for (int s = 0; s < CH; ++s) {
            if (s < m) {
                const uint32_t a = kw[2 * s] & kMagnitudes, b = kw[2 * s + 1] & kMagnitudes;
#pragma unroll
                for (int j = 0; j < C; ++j) n[j] += sel_ge(a, nv[j]) + sel_ge(b, nv[j]);
            }
        }
        uint32_t p[C / 2];  // counts of candidates 2q and 2q + 1, packed 16 : 16
#pragma unroll
        for (int q = 0; q < C / 2; ++q)
            p[q] = __reduce_add_sync(0xFFFFFFFFu, __byte_perm(n[2 * q], n[2 * q + 1], 0x5410) + __byte_perm(n[2 * q], n[2 * q + 1], 0x7632));
        if (lane == 0) *reinterpret_cast<uint4*>(sc->part[it & 1][warp]) = make_uint4(p[0], p[1], p[2], 0u);
        sel_barrier<NW>();
        // lane l adds word l % 4 of the warps l / 4, l / 4 + 8, ..
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < NW; w += 8) tot += sc->part[it & 1][w + (lane >> 2)][lane & 3];
        tot += __shfl_xor_sync(0xFFFFFFFFu, tot, 4);
        tot += __shfl_xor_sync(0xFFFFFFFFu, tot, 8);
        tot += __shfl_xor_sync(0xFFFFFFFFu, tot, 16);  // at most 32768 in either half
        // counts fall as the candidates rise: the first c have at least k keys at or above them
        const uint32_t ev = __ballot_sync(0xFFFFFFFFu, static_cast<int>(tot & 0xFFFFu) >= k) & 7u;
        const uint32_t od = __ballot_sync(0xFFFFFFFFu, static_cast<int>(tot >> 16) >= k) & 7u;
        const int c = __popc(ev | (od << 3));
        const uint32_t t = __shfl_sync(0xFFFFFFFFu, tot, c >> 1);
        const bool none = c == 0, all = c == C;
        const int next = max(lo + 1, min(base + c * stride, hi));
        if (!none) lo = max(lo + 1, min(base + (c - 1) * stride, hi));
        if (!all) {
            hi = next;
            above = static_cast<int>((c & 1) ? t >> 16 : t & 0xFFFFu);
        }
        if (hi - lo <= 1) break;
        if (stage == 0 && (none || all)) {  // the hint was off: wider steps on that side of it
            stage = 1;
            stride = 8 * D;
            base = all ? lo + stride : hi - C * stride;
        } else {
            stage = 2;
            stride = (hi - lo + C) / (C + 1);
            base = lo + stride;
        }
    }
    thr = lo;
    need_eq = k - above;
    AFX_MARK(8);
}

// Flags of the lane's channels whose key is >= v (v in 1..32768): bit w for the low half of word w, bit
// 16 + w for the high half.
template <int CH>
__device__ __forceinline__ uint32_t sel_flags_ge(const uint32_t (&kw)[2 * CH], int m, int v) {
    const uint32_t nv = sel_neg(v);
    uint32_t f = 0;
#pragma unroll
    for (int s = 0; s < CH; ++s)
        if (s < m) f += (sel_ge(kw[2 * s] & kMagnitudes, nv) << (2 * s)) + (sel_ge(kw[2 * s + 1] & kMagnitudes, nv) << (2 * s + 1));
    return f;
}
// Bit of channel e (0..3) of slot s.
__device__ __forceinline__ constexpr uint32_t sel_bit(int s, int e) { return 1u << (2 * s + (e >> 1) + 16 * (e & 1)); }

// Key above which |x| > tau holds (tau >= 0): the largest 16-bit magnitude not above tau.
template <int DT>
__device__ __forceinline__ int tau_key(float tau) {
    if (DT == AFX_F16) return __half_as_ushort(__float2half_rd(tau)) & 0x7FFF;
    return static_cast<int>((__float_as_uint(tau) >> 16) & 0x7FFFu);
}

// Flags (sel_bit) of the lane's active channels; `at` = the list position of the warp's first one,
// `count` = the list's length.  Every thread of the NW warps calls it.  `kth` receives the k-th key where
// one was searched (top-k with 0 < k < K), else 0.
template <int DT, int NW, int CH>
__device__ __forceinline__ uint32_t sel_flags(const uint32_t (&kw)[2 * CH], int m, int K, int mode, int k, float tau,
                                              uint32_t hint, RegSelScratch* sc, int& kth, int& at, int& count) {
    static_assert(CH <= 8, "flags of one lane in a word");
    const int lane = lane_id(), warp = warp_id();
    const uint32_t lt = (1u << lane) - 1u;
    auto valid = [&]() {  // flags of the lane's channels below K
        uint32_t f = 0;
#pragma unroll
        for (int s = 0; s < CH; ++s)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (s < m && sel_channel(m, s) + e < K) f |= sel_bit(s, e);
        return f;
    };
    uint32_t fl, fe = 0;  // certainly in; at the boundary, in channel order until need_eq of them are in
    int need_eq = 0;
    kth = 0;
    if (mode == AFX_MODE_TOPK) {
        if (k <= 0 || k >= K) {
            fl = k <= 0 ? 0u : valid();
        } else {
            sel_kth_key<DT, NW, CH>(kw, m, K, k, hint, sc, kth, need_eq);
            fl = sel_flags_ge<CH>(kw, m, kth + 1);
            fe = (kth == 0 ? valid() : sel_flags_ge<CH>(kw, m, kth)) & ~fl;
        }
    } else if (tau < 0.0f) {
        fl = valid();
    } else {
        constexpr int kInf = DT == AFX_F16 ? 0x7C00 : 0x7F80;  // NaN patterns lie above and never pass
        fl = sel_flags_ge<CH>(kw, m, tau_key<DT>(tau) + 1) & ~sel_flags_ge<CH>(kw, m, kInf + 1);
    }
    AFX_MARK(9);
    // counts of the warps before this one, (certain, boundary) packed 16 : 16
    const uint32_t mine = __reduce_add_sync(0xFFFFFFFFu, (static_cast<uint32_t>(__popc(fl)) << 16) | static_cast<uint32_t>(__popc(fe)));
    if (lane == 0) sc->scan[warp] = mine;
    sel_barrier<NW>();
    const uint32_t wt = lane < NW ? sc->scan[lane] : 0u;
    const uint32_t pre = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wt : 0u);
    const uint32_t tot = __reduce_add_sync(0xFFFFFFFFu, wt);
    const int pre_e = static_cast<int>(pre & 0xFFFFu), my_e = static_cast<int>(mine & 0xFFFFu);
    const int room = need_eq - pre_e;  // boundary channels of this warp that are in
    if (room >= my_e) {
        fl |= fe;
    } else if (room > 0) {  // the boundary runs through this warp: its first `room` of them
        int seen = 0;
#pragma unroll
        for (int s = 0; s < CH; ++s) {
            if (s < m) {
                int before = seen;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t b = __ballot_sync(0xFFFFFFFFu, fe & sel_bit(s, e));
                    before += __popc(b & lt);
                    seen += __popc(b);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (fe & sel_bit(s, e)) {
                        if (before < room) fl |= sel_bit(s, e);
                        ++before;
                    }
            }
        }
    }
    AFX_MARK(10);
    at = static_cast<int>(pre >> 16) + min(pre_e, need_eq);
    count = static_cast<int>(tot >> 16) + need_eq;
    return fl;
}

// Calls emit(slot, element, position, active) for the lane's channels; the active ones' positions ascend with
// the channel, from `at` for the warp's first.
template <int CH, class Emit>
__device__ __forceinline__ void sel_emit(uint32_t fl, int m, int at, Emit emit) {
    const int lane = lane_id();
    // Active channels per slot, four slots to a word (bytes 0..3 = slots 0, 2, 1, 3, then 4, 6, 5, 7), and
    // their prefix over the lanes (a slot of a warp has at most 128).
    const uint32_t pairs = (fl & 0x55555555u) + ((fl >> 1) & 0x55555555u);
    uint32_t ev = pairs & 0x33333333u, od = (pairs >> 2) & 0x33333333u;  // slots 0, 2, 4, 6 and 1, 3, 5, 7
    ev += ev >> 16;
    od += od >> 16;
#pragma unroll
    for (int h = 0; h < (CH + 3) / 4; ++h) {
        if (4 * h < m) {
            const uint32_t e2 = ev >> (8 * h), o2 = od >> (8 * h);
            const uint32_t cnt4 = (e2 & 15u) | ((e2 & 0xF0u) << 4) | ((o2 & 15u) << 16) | ((o2 & 0xF0u) << 20);
            uint32_t incl = cnt4;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += n;
            }
            const uint32_t whole = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - cnt4;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s = 4 * h + q, sh = q == 0 ? 0 : q == 1 ? 16 : q == 2 ? 8 : 24;
                if (s < CH) {
                    int pos = at + static_cast<int>((excl >> sh) & 0xFFu);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t in = fl & sel_bit(s, e);
                        emit(s, e, pos, in != 0u);
                        pos += in != 0u ? 1 : 0;
                    }
                    at += static_cast<int>((whole >> sh) & 0xFFu);
                }
            }
        }
    }
}

// What a layer operator reads: x = round(h / rms(h) * gain), the lane's channels as sel_load_keys leaves them
// (K % 8 == 0).  gv: the gains (sel_load_gain), or, with EARLY false, nothing: they are read here.
template <int CH>
__device__ __forceinline__ void sel_load_gain(const float* gain, int K, int m, float4 (&gv)[CH]) {
#pragma unroll
    for (int i = 0; i < CH; ++i)
        if (i < m && sel_channel(m, i) < K) gv[i] = *reinterpret_cast<const float4*>(gain + sel_channel(m, i));
}
template <int DT, int NW, int CH, bool EARLY>
__device__ __forceinline__ void sel_norm_keys(const float* h, const float* gain, const float4 (&gv)[EARLY ? CH : 1], float eps,
                                              int K, int m, RegSelScratch* sc, uint16_t* xnorm_out, uint32_t (&kw)[2 * CH]) {
    float4 hv[CH];
    float ss = 0.0f;
#pragma unroll
    for (int i = 0; i < CH; ++i) {
        hv[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (i < m && sel_channel(m, i) < K) hv[i] = *reinterpret_cast<const float4*>(h + sel_channel(m, i));
    }
#pragma unroll
    for (int i = 0; i < CH; ++i) {
        ss = fmaf(hv[i].x, hv[i].x, ss);
        ss = fmaf(hv[i].y, hv[i].y, ss);
        ss = fmaf(hv[i].z, hv[i].z, ss);
        ss = fmaf(hv[i].w, hv[i].w, ss);
    }
    ss = warp_sum(ss);
    if (lane_id() == 0) sc->sum[warp_id()] = ss;
    sel_barrier<NW>();
    float tot = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; w += 4) {
        const float4 v = *reinterpret_cast<const float4*>(sc->sum + w);
        tot += (v.x + v.y) + (v.z + v.w);
    }
    const float inv = 1.0f / sqrtf(tot / static_cast<float>(K) + eps);
#pragma unroll
    for (int i = 0; i < CH; ++i) {
        kw[2 * i] = 0u;
        kw[2 * i + 1] = 0u;
        const int j = sel_channel(m, i);
        if (i < m && j < K) {
            const float4 gn = EARLY ? gv[EARLY ? i : 0] : *reinterpret_cast<const float4*>(gain + j);
            kw[2 * i] = pack2_bits<DT>(hv[i].x * inv * gn.x, hv[i].y * inv * gn.y);
            kw[2 * i + 1] = pack2_bits<DT>(hv[i].z * inv * gn.z, hv[i].w * inv * gn.w);
            if (xnorm_out != nullptr) *reinterpret_cast<uint2*>(xnorm_out + j) = make_uint2(kw[2 * i], kw[2 * i + 1]);
        }
    }
}

}  // namespace afx
