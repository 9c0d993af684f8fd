// enomr_select.cuh -- the ENO-MR selection of a window and the value on a
// selected stencil, from the differences of neighbouring cells in float.
//
// arXiv 2311.15504: Sec. 3.2 (Steps 1-3), Eq. (Baseline_IS), Eq. (CurrentIS),
// Eq. (ReconstructedFlux).
//
// Why.  GB300 has two FP64 lanes per SM and cycle against 128 FP32 lanes: one
// FP64 warp instruction takes the time of 64 FP32 ones, and the path's
// FP64 work is mostly this: the indicators |sum b_l v_l| and the
// reconstructions sum a_l v_l.  Both depend on the window through
// differences e_j = v_{j+1} - v_j alone (sum b_l = 0, sum a_l = 1), and a
// difference, formed once in FP64, needs far fewer than 53 bits.
//
// Selection.  Every comparison IS_t < IS_0 and every minmod decision is taken
// on float values with a bound on their distance from the values that the
// FP64 evaluation (mr_select) compares: the float rounding of the
// differences and sums, relative to sum |b'_j| |e_j|, and the rounding of the
// FP64 evaluation itself, relative to the size of the window's values.  A
// comparison that the bound does not decide leaves the window to the FP64
// evaluation, so the selection is the one of the FP64 evaluation always.
// Differences below 2^-60 and values above 2^90 are out of the floats' range and
// go to FP64 too.
//
// Value.  With e_j as a pair of floats (48 bits) and weights w_j as pairs,
// v_c + sum w_j e_j is a compensated float sum and one FP64 addition.  Its
// error against exact arithmetic, measured over random windows with
// |e_j| <= 2^-k |v_c| (rms / max, ulp): order 9, k = 6: 0.35 / 1.5 (FP64
// sum: 0.66 / 2.9); order 17: 0.39 / 2.7 (0.87 / 3.6).  Whole right-hand sides
// against 113-bit arithmetic, rms: advection, N = 1 048 573, order 9, 6.4e-17
// (FP64 sums 1.36e-16); Burgers, N = 2^22, order 13, 5.9e-17 (1.17e-16).  It is
// taken for windows with |e_j| <= 2^-6 |v_c| only, and not for those that are
// selected in FP64.
#pragma once

#include "enomr_float.cuh"
#include "enomr_kernels.cuh"

namespace enomr {

// ---- compensated sum of products of float pairs (error-free sum and product:
// Knuth's TwoSum, the product's rest by a fused multiply-add)
struct PairSum {
    float s, c;
    __device__ __forceinline__ void first(float2 w, float2 e)
    {
        s = __fmul_rn(w.x, e.x);
        c = __fmaf_rn(w.y, e.x, __fmaf_rn(w.x, e.y, __fmaf_rn(w.x, e.x, -s)));
    }
    __device__ __forceinline__ void add(float2 w, float2 e)
    {
        const float p = __fmul_rn(w.x, e.x);
        const float r = __fmaf_rn(w.y, e.x, __fmaf_rn(w.x, e.y, __fmaf_rn(w.x, e.x, -p)));
        const float t = __fadd_rn(s, p), b = __fsub_rn(t, s);
        const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(p, b));
        c = __fadd_rn(c, __fadd_rn(d, r));
        s = t;
    }
};

// Largest |e_j| over |v_c| for which the pair sum is taken.
constexpr float PAIR_RANGE = 0x1p-6f;

template <int R, int t>
__device__ __forceinline__ void select_walk(const float *e, float S, float lo, float hi, int &sel)
{
    constexpr int g = (R + 1) / 2, c = g - 1, T = Tab<R>::T;
    if constexpr (t < T) {
        constexpr int K = Cand<R, t>::m + Cand<R, t>::n, j0 = c - Cand<R, t>::m;
        float s = 0.0f, a = 0.0f;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const float b = ((K - 1 - i) & 1) ? -binomial(K - 1, i) : binomial(K - 1, i);
            s = i == 0 ? __fmul_rn(b, e[j0 + i]) : __fmaf_rn(b, e[j0 + i], s);
            a = i == 0 ? fabsf(b) * fabsf(e[j0 + i]) : __fmaf_rn(fabsf(b), fabsf(e[j0 + i]), a);
        }
        const float err = __fmaf_rn(a, float_error(K), S * fp64_error(K));
        s = fabsf(s);
        if (s + err < lo) {
            sel = t;
        } else if (s - err > hi) {
            select_walk<R, t + 1>(e, S, lo, hi, sel);
        } else {
            sel = SEL_OPEN;
        }
    }
}

// Selection of the window with differences e_j (j = 0 .. 2g-3); S: size of the
// centre value.  left0, right0: the three cells ending / starting at the
// centre are bitwise equal.  Returns 0 .. T+2 or SEL_OPEN.
template <int R>
__device__ __forceinline__ int select_float(const float *e, float S, bool left0, bool right0)
{
    constexpr int g = (R + 1) / 2, c = g - 1, T = Tab<R>::T;
    if (left0 || right0) return T + 2;  // IS_0 = 0: no candidate passes, minmod(a, b) = 0
    const float l1 = e[c - 1], l2 = e[c - 2], r1 = e[c], r2 = e[c + 1];
    const float al = fabsf(l1), ar = fabsf(r1), sv = S * fp64_error(2);
    const float el = __fmaf_rn(al + fabsf(l2), float_error(2), sv);
    const float er = __fmaf_rn(ar + fabsf(r2), float_error(2), sv);
    const float L = fmaxf(al, fabsf(l1 - l2)), Q = fmaxf(ar, fabsf(r2 - r1));
    const float lo = fminf(L - el, Q - er), hi = fminf(L + el, Q + er);
    int sel = T;
    if (!(S <= 0x1p90f) || !(el + er <= 0x1p90f)) return SEL_OPEN;  // NaN or out of range
    select_walk<R, 0>(e, S, lo, hi, sel);
    if (sel != T) return sel;
    // every candidate failed: minmod(f_{j+1} - f_j, f_j - f_{j-1})
    const float e1 = __fmaf_rn(al, float_error(2), sv), e2 = __fmaf_rn(ar, float_error(2), sv);
    if (!(al > e1) || !(ar > e2)) return SEL_OPEN;
    if ((l1 < 0.0f) != (r1 < 0.0f)) return T + 2;
    if (ar + e2 < al - e1) return T;
    if (al + e1 < ar - e2) return T + 1;
    return SEL_OPEN;
}

}  // namespace enomr
