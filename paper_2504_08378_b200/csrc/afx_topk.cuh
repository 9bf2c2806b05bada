// Active-channel selection with the keys in registers.
//
// The first NW warps of the block own the channels: slot s of warp w holds channels (w m + s) 128 + 4
// lane .. + 3.  The k-th largest 15-bit magnitude key is found from a hint of it, the last k-th key or, without one, a
// sample of the keys: every key of a window around the hint has a counter in shared memory, the keys above the
// window are counted two per operation, and behind ONE barrier every warp sums the counters from the top.  Where the
// k-th key is outside the window a seven-way search of the rest follows, from the window outwards: a step counts the keys
// at or above six candidates, adds the counts over warp and block (three `redux` before and three shuffles behind one
// barrier of the NW warps) and keeps the interval between two of them.
//
// What bounds it is the latency of barriers and reductions and the rate of shared-memory atomics (about one in ten keys
// is in the window; all of them on one counter cost no more: one token of 28672 equal magnitudes 8.8 us, of Laplace ones
// 9.6).  Clocks for the k-th key, the seven-way search alone from the same hint and now: bf16 K = 4096 on 8
// warps 2050 and 1560, K = 11008 on 16 warps 3850 and 2340; f16 K = 4096 3030 and 1640, K = 1024 2470 and 1030.  What
// every warp repeats behind the barrier counts NW times, so few warps with many keys each beat many warps with few.
#pragma once

#include "afx_select.cuh"

namespace afx {

constexpr uint32_t kNoHint = 0xFFFFFFFFu;
constexpr int kRegSelMaxWarps = 32;

constexpr int kSelBins = 256;

struct RegSelScratch {
    __align__(16) uint32_t win[kSelBins];  // keys around the hint, counted one by one (cleared by sel_prepare)
    __align__(16) uint32_t part[2][kRegSelMaxWarps][4];  // per-warp counts of a search step (double-buffered)
    uint32_t scan[kRegSelMaxWarps], top[kRegSelMaxWarps];
    int count;      // the list's length, for the warps that did not select
    uint32_t hint;  // where the search starts (sel_prepare)
    __align__(16) float sum[kRegSelMaxWarps];
};

// Barrier of the block's first NW warps.
template <int NW>
__device__ __forceinline__ void sel_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory");
}

// Before the selection: clears the counters, and leaves the search hint in `slot` (NULL: none) for the whole block.  ONE
// thread of the first warp reads the hint, and the others take it from sc->hint behind a barrier of the selecting warps:
// another launch of the operator, or another block of this one, may be rewriting the word, and threads that read it for
// themselves could start with different hints, take different numbers of search steps, and wait at different barriers.
template <int NW>
__device__ __forceinline__ void sel_prepare(const int32_t* slot, RegSelScratch* sc) {
    if (threadIdx.x < NW * 32)
        for (int i = threadIdx.x; i < kSelBins / 4; i += NW * 32) reinterpret_cast<uint4*>(sc->win)[i] = make_uint4(0u, 0u, 0u, 0u);
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

// ++win[d] where d < N; never a branch (sixteen of them, as branches, cost 250 of the search's clocks).
template <int N>
__device__ __forceinline__ void count_below(uint32_t win, uint32_t d) {
    asm volatile("{ .reg .pred p; .reg .b32 t; setp.lt.u32 p, %1, %2; mad.lo.u32 t, %1, 4, %0; @p red.shared.add.u32 [t], 1; }" ::"r"(win), "r"(d), "n"(N) : "memory");
}

// The k-th largest key (1 <= k <= K) of the NW warps' channels: `thr`; how many channels with exactly
// that key belong to the top k: `need_eq`.  Same values in every thread.  `hint` only shortens the
// search.  Zero padding behind K is never counted (candidates are >= 1).
template <int DT, int NW, int CH>
__device__ __forceinline__ void sel_kth_key(const uint32_t (&kw)[2 * CH], int m, int K, int k, uint32_t hint, RegSelScratch* sc,
                                            int& thr, int& need_eq) {
    constexpr int C = 6;
    // A counter for every key of a window around the hint: +-32 keys in bf16 (+-12 to 25 % in magnitude), +-128 in f16
    // (+-6 to 12 %); successive tokens' keys for one operator lie within a few percent.
    constexpr int kWin = DT == AFX_BF16 ? 64 : 256;
    static_assert(kWin <= kSelBins, "counters");
    const int lane = lane_id(), warp = warp_id();
    int lo = 0, hi = 32768, above = 0;  // count(keys >= lo) >= k > count(keys >= hi) = above
    // The candidates of a search step are a seventh of the interval apart.  Behind a missed window they are a power of seven
    // apart, next to it, since that is where the k-th key usually is: two steps are left in bf16, three in f16, instead of
    // five (a hint off by more than a factor of four pays one step more).  From below the farthest one is key 1: more than
    // half of some inputs are zeros.  us, the whole selection, a missed window behind which the search took sevenths at
    // once, and now: one token of 4096 4-bit values 5.1 and 4.7, half of 4096 zeros 6.1 and 4.5; f16, four tokens of 4096
    // 7.1 and 6.6, one of 11008 values half of them zeros 11.0 and 7.4.
    constexpr int kNear = DT == AFX_BF16 ? 49 : 343;
    int stride = (32768 + C) / (C + 1), from = stride;
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
        const uint32_t base = static_cast<uint32_t>(max(1, min(static_cast<int>(hint) - kWin / 2, 32768 - kWin)));
        const uint32_t nv = sel_neg(static_cast<int>(base) + kWin);
        const uint32_t win = static_cast<uint32_t>(__cvta_generic_to_shared(sc->win));
        uint32_t n = 0;
#pragma unroll
        for (int w = 0; w < 2 * CH; ++w) {
            if (w < 2 * m) {
                const uint32_t a = kw[w] & kMagnitudes;
                n += sel_ge(a, nv);
                count_below<kWin>(win, (a & 0xFFFFu) - base);
                count_below<kWin>(win, (a >> 16) - base);
            }
        }
        n = __reduce_add_sync(0xFFFFFFFFu, (n & 0xFFFFu) + (n >> 16));
        if (lane == 0) sc->top[warp] = n;
        sel_barrier<NW>();
        // lane l: counters kLane l .. of the window
        constexpr int kLane = kWin / 32;
        uint32_t c[kLane], sum = 0;
#pragma unroll
        for (int j = 0; j < kLane; j += 2) {
            const uint2 v = *reinterpret_cast<const uint2*>(sc->win + kLane * lane + j);
            c[j] = v.x;
            c[j + 1] = v.y;
            sum += v.x + v.y;
        }
        const uint32_t top = __reduce_add_sync(0xFFFFFFFFu, lane < NW ? sc->top[lane] : 0u);
        uint32_t ge = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_down_sync(0xFFFFFFFFu, ge, o);
            if (lane + o < 32) ge += v;
        }
        ge += top;  // keys at or above the lane's first one
        const uint32_t at = __ballot_sync(0xFFFFFFFFu, ge >= static_cast<uint32_t>(k));  // lanes 0 .. of the one that holds it
        uint32_t run = ge - sum, key = 0, over = 0;
        bool found = false;
#pragma unroll
        for (int j = kLane - 1; j >= 0; --j) {
            if (!found) {
                over = run;
                key = j;
                run += c[j];
                found = run >= static_cast<uint32_t>(k);
            }
        }
        if (at != 0u && top < static_cast<uint32_t>(k)) {
            const uint32_t got = __shfl_sync(0xFFFFFFFFu, ((base + kLane * lane + key) << 16) | over, 31 - __clz(at));
            thr = static_cast<int>(got >> 16);
            need_eq = k - static_cast<int>(got & 0xFFFFu);
            AFX_MARK(8);
            return;
        }
        // the hint was off: the interval on that side of the window
        if (at == 0u) {
            hi = static_cast<int>(base);
            above = static_cast<int>(__shfl_sync(0xFFFFFFFFu, ge, 0));
            from = hi - C * kNear;
        } else {
            lo = static_cast<int>(base) + kWin;
            from = lo + kNear;
        }
        stride = kNear;
    }
    int it = 0;
    while (hi - lo > 1) {
        const bool zeros = it == 0 && stride == kNear && lo == 0;
        uint32_t nv[C], n[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            nv[j] = sel_neg(j == 0 && zeros ? 1 : max(lo + 1, min(from + j * stride, hi)));
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
        const int next = c == 0 && zeros ? 1 : max(lo + 1, min(from + c * stride, hi));
        if (c > 0) lo = c == 1 && zeros ? 1 : max(lo + 1, min(from + (c - 1) * stride, hi));
        if (c < C) {
            hi = next;
            above = static_cast<int>((c & 1) ? t >> 16 : t & 0xFFFFu);
        }
        stride = (hi - lo + C) / (C + 1);
        from = lo + stride;
        ++it;
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

// Stores v to the shared-memory word at `at` and moves on to the next one where `fl` has `BIT`; never a branch.
template <uint32_t BIT>
__device__ __forceinline__ void st_shared_next(uint32_t& at, uint32_t v, uint32_t fl) {
    asm volatile("{ .reg .pred p; .reg .b32 t; and.b32 t, %2, %3; setp.ne.u32 p, t, 0; @p st.shared.u32 [%0], %1; @p add.u32 %0, %0, 4; }"
                 : "+r"(at)
                 : "r"(v), "r"(fl), "n"(BIT)
                 : "memory");
}

// Writes the lane's active channels (flags of sel_flags, words of sel_load_keys) as list entries (16-bit channel, 16-bit
// value) to shared memory, `list` the address of the warp's first entry; entries ascend with the channel.
template <int CH>
__device__ __forceinline__ void sel_emit(uint32_t fl, int m, const uint32_t (&kw)[2 * CH], uint32_t list) {
    const int lane = lane_id();
    // Active channels per slot, four slots to a word (bytes 0..3 = slots 0, 2, 1, 3, then 4, 6, 5, 7), and
    // their prefix over the lanes (a slot of a warp has at most 128).
    const uint32_t pairs = (fl & 0x55555555u) + ((fl >> 1) & 0x55555555u);
    uint32_t ev = pairs & 0x33333333u, od = (pairs >> 2) & 0x33333333u;  // slots 0, 2, 4, 6 and 1, 3, 5, 7
    ev += ev >> 16;
    od += od >> 16;
    constexpr int NH = (CH + 3) / 4;
    uint32_t cnt4[NH], incl[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const uint32_t e2 = ev >> (8 * h), o2 = od >> (8 * h);
        cnt4[h] = (e2 & 15u) | ((e2 & 0xF0u) << 4) | ((o2 & 15u) << 16) | ((o2 & 0xF0u) << 20);
        incl[h] = cnt4[h];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl[h], o);
            if (lane >= o) incl[h] += n;
        }
    }
    uint32_t chan = static_cast<uint32_t>(sel_channel(m, 0));
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const uint32_t whole = __shfl_sync(0xFFFFFFFFu, incl[h], 31), excl = incl[h] - cnt4[h];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            constexpr int kShift[4] = {0, 16, 8, 24};
            const int s = 4 * h + q;
            if (s < CH) {
                uint32_t at = list + 4u * ((excl >> kShift[q]) & 0xFFu);
                const uint32_t f = fl >> (2 * s);
                st_shared_next<0x00001u>(at, __byte_perm(kw[2 * s], chan, 0x1054), f);
                st_shared_next<0x10000u>(at, __byte_perm(kw[2 * s], chan + 1u, 0x3254), f);
                st_shared_next<0x00002u>(at, __byte_perm(kw[2 * s + 1], chan + 2u, 0x1054), f);
                st_shared_next<0x20000u>(at, __byte_perm(kw[2 * s + 1], chan + 3u, 0x3254), f);
                list += 4u * ((whole >> kShift[q]) & 0xFFu);
                chan += 128u;
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
