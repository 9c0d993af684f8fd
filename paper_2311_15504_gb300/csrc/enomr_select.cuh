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
//
// Value.  With e_j as a pair of floats (48 bits) and weights w_j as pairs,
// v_c + sum w_j e_j is a compensated float sum and one FP64 addition.  Its
// error against exact arithmetic, measured over random windows with
// |e_j| <= 2^-k |v_c| (rms / max, ulp): order 9, k = 6: 0.35 / 1.5 (FP64
// sum: 0.66 / 2.9); order 17: 0.39 / 2.7 (0.87 / 3.6).  It is taken for
// windows with |e_j| <= 2^-6 |v_c| only.
#pragma once

#include "enomr_kernels.cuh"

namespace enomr {

// ---- conversions on the integer ALU (a double conversion instruction runs
// at the FP64 rate).  split_pair: high 24 bits (truncated) and rest of x.
// Outside 2^-60 <= |x| < 2^100 (and x = 0, exact) the pair is NaN, which no
// test below accepts.
__device__ __forceinline__ float2 split_pair(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned m = hi & 0x7fffffffu, sg = hi & 0x80000000u, ex = m >> 20;
    if ((m | lo) == 0u) return make_float2(0.0f, 0.0f);
    if (ex < 1023u - 60u || ex >= 1023u + 100u)
        return make_float2(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff));
    const float h = __uint_as_float(sg | __funnelshift_l(lo, m - 0x38000000u, 3));
    const float sc = __uint_as_float(sg | ((ex - (1023u + 52u - 127u)) << 23));
    return make_float2(h, __uint2float_rn(lo & 0x1fffffffu) * sc);
}

// the high part alone (relative error below 2^-23)
__device__ __forceinline__ float to_float(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned m = hi & 0x7fffffffu, ex = m >> 20;
    if ((m | lo) == 0u) return 0.0f;
    if (ex < 1023u - 60u || ex >= 1023u + 100u) return __int_as_float(0x7fffffff);
    return __uint_as_float((hi & 0x80000000u) | __funnelshift_l(lo, m - 0x38000000u, 3));
}

// a float as a double (subnormal floats, below 2^-126, as zero)
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    const unsigned hi = m < 0x00800000u ? 0u : (m >> 3) + 0x38000000u;
    return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(m < 0x00800000u ? 0u : m << 29));
}

// ---- compensated sum of products of float pairs
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

constexpr int SEL_OPEN = -1;  // the float comparisons do not decide

__host__ __device__ constexpr float binomial(int n, int k)
{
    double r = 1.0;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return (float)r;  // at most C(15, 7) = 6435: exact
}

// Bound units.  EPS: relative error of a difference e_j against its
// magnitude m_j, in 2^-24 (scalar: the truncation to float, m_j = |e_j|).
// OPS: FP64 roundings of a window value.
template <int EPS, int OPS>
struct SelBound {
    // K terms: K fused products, one rounding each
    __host__ __device__ static constexpr float terms(int K) { return 0x1p-24f * (EPS + K + 2); }
    // FP64 evaluation: 2^K coefficients' sum, K + 1 roundings and those of the values
    __host__ __device__ static constexpr float values(int K)
    {
        return 0x1.2p-53f * (float)(1 << K) * (float)(K + 2 + OPS);
    }
};

template <int R, int t, class B, bool REV>
__device__ __forceinline__ void select_walk(const float *e, const float *m, float S, float lo,
                                            float hi, int &sel)
{
    constexpr int g = (R + 1) / 2, c = g - 1, N = 2 * g - 2, T = Tab<R>::T;
    if constexpr (t < T) {
        constexpr int K = Cand<R, t>::m + Cand<R, t>::n, j0 = c - Cand<R, t>::m;
        float s = 0.0f, a = 0.0f;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const float b = ((K - 1 - i) & 1) ? -binomial(K - 1, i) : binomial(K - 1, i);
            const int j = REV ? N - 1 - (j0 + i) : j0 + i;
            s = i == 0 ? __fmul_rn(b, e[j]) : __fmaf_rn(b, e[j], s);
            a = i == 0 ? fabsf(b) * fabsf(m[j]) : __fmaf_rn(fabsf(b), fabsf(m[j]), a);
        }
        const float err = __fmaf_rn(a, B::terms(K), S * B::values(K));
        s = fabsf(s);
        if (s + err < lo) {
            sel = t;
        } else if (s - err > hi) {
            select_walk<R, t + 1, B, REV>(e, m, S, lo, hi, sel);
        } else {
            sel = SEL_OPEN;
        }
    }
}

// Selection of the window with differences e_j (j = 0 .. 2g-3) and their
// magnitudes m_j >= the size of the terms that formed e_j; S: bound of the
// size of the terms that formed the centre value.  REV: e and m run against
// the window (window difference i is entry 2g-3-i; the sign of all of them
// is immaterial).  left0, right0: the three cells ending / starting at the
// centre are bitwise equal.  Returns 0 .. T+2 or SEL_OPEN.
template <int R, class B, bool REV>
__device__ __forceinline__ int select_float(const float *e, const float *m, float S, bool left0,
                                            bool right0)
{
    constexpr int g = (R + 1) / 2, c = g - 1, N = 2 * g - 2, T = Tab<R>::T;
    if (left0 || right0) return T + 2;  // IS_0 = 0: no candidate passes, minmod(a, b) = 0
    auto at = [&](const float *p, int j) { return p[REV ? N - 1 - j : j]; };
    const float l1 = at(e, c - 1), l2 = at(e, c - 2), r1 = at(e, c), r2 = at(e, c + 1);
    const float ml = fabsf(at(m, c - 1)), mr = fabsf(at(m, c));
    const float sv = S * B::values(2);
    const float el = __fmaf_rn(ml + fabsf(at(m, c - 2)), B::terms(2), sv);
    const float er = __fmaf_rn(mr + fabsf(at(m, c + 1)), B::terms(2), sv);
    const float L = fmaxf(fabsf(l1), fabsf(l1 - l2)), Q = fmaxf(fabsf(r1), fabsf(r2 - r1));
    const float lo = fminf(L - el, Q - er), hi = fminf(L + el, Q + er);
    int sel = T;
    if (!(S <= 0x1p90f) || !(el + er <= 0x1p90f)) return SEL_OPEN;  // NaN or out of range
    select_walk<R, 0, B, REV>(e, m, S, lo, hi, sel);
    if (sel != T) return sel;
    // every candidate failed: minmod(f_{j+1} - f_j, f_j - f_{j-1})
    const float e1 = __fmaf_rn(ml, B::terms(2), sv), e2 = __fmaf_rn(mr, B::terms(2), sv);
    const float al = fabsf(l1), ar = fabsf(r1);
    if (!(al > e1) || !(ar > e2)) return SEL_OPEN;
    if ((l1 < 0.0f) != (r1 < 0.0f)) return T + 2;
    if (ar + e2 < al - e1) return T;
    if (al + e1 < ar - e2) return T + 1;
    return SEL_OPEN;
}

}  // namespace enomr
