// Device code shared by the kernels that score templates exactly (k_sparse.cu, k_score.cu): the
// correlation C(s) of one template for all its shifts over polar rows staged in shared memory, in
// the three row layouts that k_sparse.cu describes, and the order of the results.
#pragma once

#include <float.h>
#include <limits.h>

#include "tm_internal.h"

namespace tmgb {

// Shift blocks per template are rounded up to one of a few unrolled kernels.
__host__ __device__ constexpr int round_nb(int nb) {
    return nb <= 4 ? nb : nb <= 6 ? 6 : nb <= 8 ? 8 : nb <= 12 ? 12 : nb <= 16 ? 16 : nb <= 24 ? 24 : 32;
}

__device__ __forceinline__ bool better(float qa, int ka, float qb, int kb) {
    return qa > qb || (qa == qb && ka < kb);
}

// Order-preserving integer key of a float (for atomicMax on scores).
__device__ __forceinline__ unsigned score_key(float x) {
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_score(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// ---------------------------------------------------------------- per-layout spot updates
// acc holds V values per lane (V = 2 NB for the dual layout, NB otherwise); value v of lane L
// is shift shift_of(v, L).  FIRST initialises instead of accumulating.

template <int LAYOUT>
__device__ __forceinline__ int shift_of(int v, int lane) {
    return LAYOUT == TM_LAYOUT_DUAL ? 64 * (v >> 1) + 2 * lane + (v & 1) : 32 * v + lane;
}

// Dual and wrap-free layouts: px holds the spot's shared-memory offset (bits 0..15 dual,
// 16..31 wrap-free).
template <int V, int LAYOUT, bool FIRST>
__device__ __forceinline__ void add_spot(float (&acc)[V], const float* __restrict__ sP, int px, float I, int lane) {
    if (LAYOUT == TM_LAYOUT_DUAL) {
        const float2* p = reinterpret_cast<const float2*>(sP + (px & 0xffff)) + lane;
#pragma unroll
        for (int b = 0; b < V / 2; ++b) {
            const float2 v = p[32 * b];
            acc[2 * b] = FIRST ? I * v.x : fmaf(I, v.x, acc[2 * b]);
            acc[2 * b + 1] = FIRST ? I * v.y : fmaf(I, v.y, acc[2 * b + 1]);
        }
    } else {
        const float* p = sP + ((unsigned)px >> 16) + lane;
#pragma unroll
        for (int b = 0; b < V; ++b) acc[b] = FIRST ? I * p[32 * b] : fmaf(I, p[32 * b], acc[b]);
    }
}

// Wrapped layout: px = t | row << 11 | w << 24, w the first 32-wide block past the wrap.
template <int V, bool FIRST>
__device__ __forceinline__ void add_spot_wrapped(float (&acc)[V], const float* __restrict__ sP, int px, float I,
                                                 int pitch, int n_theta, int lane) {
    const int t = px & 0x7ff;
    const int row = (px >> 11) & 0x1fff;
    const int w = (int)((unsigned)px >> 24);
    const float* p1 = sP + row * pitch + t + lane;
    const float* p2 = p1 - n_theta;                           // blocks b >= w: wrapped
#pragma unroll
    for (int b = 0; b < V; ++b) {
        const float v = (b < w ? p1 : p2)[32 * b];
        acc[b] = FIRST ? I * v : fmaf(I, v, acc[b]);
    }
}

// Correlation C(s) of one template for all its shifts (warp-collective).  NB = shift blocks
// (64 wide for the dual layout, else 32).  Returns the warp-wide maximum; when it reaches
// thr_c, shift_out is the lowest shift attaining it and `resolved` is set.  FULL: the
// template is slid over all n_theta shifts.  `mine`: the lane's spot of the first 32 (lane_spot).
__device__ __forceinline__ int2 lane_spot(const int2* __restrict__ spots, int beg, int cnt, int lane) {
    return lane < min(32, cnt) ? __ldg(spots + beg + lane) : make_int2(0, 0);   // one lane-parallel load
}

template <int NB, int LAYOUT, bool FULL>
__device__ __forceinline__ float score_template(const float* __restrict__ sP, const int2* __restrict__ spots, int beg,
                                                int cnt_all, int2 mine, int S, int n_theta, int pitch, int lane,
                                                float thr_c, int& shift_out, bool& resolved) {
    constexpr int V = LAYOUT == TM_LAYOUT_DUAL ? 2 * NB : NB;
    resolved = false;
    int cnt = min(32, cnt_all);
    float acc[V];
    if (cnt <= 0) {                                               // no spot on the grid: C = 0, no read
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.0f;
        cnt = 0;
    }
    if (cnt > 0) {
        const int px = __shfl_sync(0xffffffffu, mine.x, 0);
        const float I = __int_as_float(__shfl_sync(0xffffffffu, mine.y, 0));
        if (LAYOUT == TM_LAYOUT_WRAP) add_spot_wrapped<V, true>(acc, sP, px, I, pitch, n_theta, lane);
        else add_spot<V, LAYOUT, true>(acc, sP, px, I, lane);
    }
    const int end = beg + cnt_all;
    for (int i0 = beg, j = 1;;) {
        for (; j < cnt; ++j) {
            const int px = __shfl_sync(0xffffffffu, mine.x, j);
            const float I = __int_as_float(__shfl_sync(0xffffffffu, mine.y, j));
            if (LAYOUT == TM_LAYOUT_WRAP) add_spot_wrapped<V, false>(acc, sP, px, I, pitch, n_theta, lane);
            else add_spot<V, LAYOUT, false>(acc, sP, px, I, lane);
        }
        i0 += 32;
        if (i0 >= end) break;
        cnt = min(32, end - i0);
        if (lane < cnt) mine = __ldg(spots + i0 + lane);
        j = 0;
    }
    // Every value holds C(shift mod Nθ), computed by the same operations as the shift it
    // repeats (column c of a row holds P'[c mod Nθ]); so for a template slid over all Nθ
    // shifts the maximum needs no lane mask.  Otherwise shifts >= S are masked.
    float best = -FLT_MAX;
    if (FULL) {
#pragma unroll
        for (int v = 0; v < V; ++v) best = fmaxf(best, acc[v]);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (shift_of<LAYOUT>(v, lane) < S) best = fmaxf(best, acc[v]);
    }
    if (!__any_sync(0xffffffffu, best >= thr_c)) return best;    // cannot enter the top-N
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (best >= thr_c) {
        int s = INT_MAX;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const int sv = shift_of<LAYOUT>(v, lane);
            if (sv < S && acc[v] == best) s = min(s, sv);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s = min(s, __shfl_xor_sync(0xffffffffu, s, o));
        shift_out = s;
        resolved = true;
    }
    return best;
}

template <int NBMAX, int LAYOUT>
__device__ __forceinline__ float score_dispatch(const float* sP, const int2* spots, int beg, int cnt, int2 mine, int S,
                                                int n_theta, int pitch, int lane, float thr_c, int& s, bool& res) {
    constexpr int W = LAYOUT == TM_LAYOUT_DUAL ? 64 : 32;
    res = false;
    if (S == n_theta && round_nb((n_theta + W - 1) / W) == NBMAX)   // the common case, tested first
        return score_template<NBMAX, LAYOUT, true>(sP, spots, beg, cnt, mine, S, n_theta, pitch, lane, thr_c, s, res);
    const int nb = (S + W - 1) / W;
#define TMGB_SCORE(NBV)                                                                                          \
    return score_template<(NBMAX >= NBV ? NBV : 1), LAYOUT, false>(sP, spots, beg, cnt, mine, S, n_theta, pitch, \
                                                                   lane, thr_c, s, res)
    if (nb <= 1) TMGB_SCORE(1);
    if (nb <= 2) TMGB_SCORE(2);
    if (nb <= 3) TMGB_SCORE(3);
    if (nb <= 4) TMGB_SCORE(4);
    if (NBMAX >= 6 && nb <= 6) TMGB_SCORE(6);
    if (NBMAX >= 8 && nb <= 8) TMGB_SCORE(8);
    if (NBMAX >= 12 && nb <= 12) TMGB_SCORE(12);
    if (NBMAX >= 16 && nb <= 16) TMGB_SCORE(16);
    if (NBMAX >= 24 && nb <= 24) TMGB_SCORE(24);
    TMGB_SCORE(32);
#undef TMGB_SCORE
}

}  // namespace tmgb
