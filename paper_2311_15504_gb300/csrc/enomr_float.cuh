// enomr_float.cuh -- floats of doubles on the integer ALU, and the bounds of
// the float form of the selection (select_float, mr_select).
#pragma once

#include <cuda_runtime.h>

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

constexpr int SEL_OPEN = -1;  // the float comparisons do not decide

__host__ __device__ constexpr float binomial(int n, int k)
{
    double r = 1.0;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return (float)r;  // at most C(15, 7) = 6435: exact
}

// Bounds of the float form of an indicator of order K = m + n against the value
// that the FP64 evaluation compares: float_error(K) * sum |b'_j| |e_j| +
// fp64_error(K) * |v_c|.

// K fused products, one rounding each, of differences truncated to float (twice
// 2^-24), and the final additions
__host__ __device__ constexpr float float_error(int K) { return 0x1p-24f * (float)(K + 4); }

// the FP64 evaluation: one rounding per term of the partial sums of alternating
// binomials, +-C(K-1, i) times the centre value up to terms of the size of the
// differences: 2^(K-1) in all
__host__ __device__ constexpr float fp64_error(int K) { return 0x1.1p-54f * (float)(1 << K); }

}  // namespace enomr
