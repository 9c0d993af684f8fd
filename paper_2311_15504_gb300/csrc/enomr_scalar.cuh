// enomr_scalar.cuh -- scalar conservation laws: linear advection and the
// inviscid Burgers equation (arXiv 2311.15504, Sec. 4.1, Sec. 4.2).
// One thread per interface; a CTA stages TP + 2g - 1 split flux values.
#pragma once

#include <cooperative_groups.h>

#include "enomr_select.cuh"

namespace enomr {

// ENO-MR value of the window that starts at v0 and runs with stride DIRN (+1
// or -1) through the split fluxes; e0: the pair of the difference of its
// first two cells as stored (e[s] = f[s+1] - f[s]; a mirrored window meets
// them in the opposite order and sign, which the caller's pointer and DIRN
// express).  All 32 lanes of the warp call it together.  The FP64 pipe binds
// these kernels: the selection runs in float (select_float), and a window on
// a tested stencil whose differences are small against its centre takes the
// float-pair sum; the others take the FP64 sums.  Measured (GB300, smooth data
// with a square pulse): order 9, N = 1 048 573: 82 -> 34 us per launch, FP64
// pipe 59 % busy; Burgers, order 13, N = 2^22: 387 -> 165 us.
template <int R, int DIRN>
__device__ __forceinline__ double scalar_value(const double *v0, const float2 *e0,
                                               const double *sA, const float2 *sW, bool valid,
                                               int &sel)
{
    constexpr int g = (R + 1) / 2, W = 2 * g - 1, T = Tab<R>::T, c = g - 1, N = W - 1;
    float e[N];
    float emax = 0.0f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        e[j] = e0[DIRN * j].x;
        emax = fmaxf(emax, fabsf(e[j]));
    }
    const float vc = fabsf(to_float(v0[DIRN * c]));
    const bool left0 = e[c - 1] == 0.0f && e[c - 2] == 0.0f;
    const bool right0 = e[c] == 0.0f && e[c + 1] == 0.0f;
    // a warp of which every window is constant up to rounding or exactly: mr_select
    const bool none = left0 || right0;
    const float near = fmaxf(fmaxf(fabsf(e[c - 2]), fabsf(e[c - 1])), fmaxf(fabsf(e[c]), fabsf(e[c + 1])));
    const bool noise = !none && near <= vc * (0x1p-52f * (float)NOISE_ULP<R>);
    if (__all_sync(FULL, noise || none || !valid))
        sel = none ? T + 2 : SEL_OPEN;
    else
        sel = select_float<R>(e, vc, left0, right0);
    const bool open = valid && sel == SEL_OPEN;
    if (__any_sync(FULL, open)) {
        double v[W];
#pragma unroll
        for (int j = 0; j < W; ++j) v[j] = v0[DIRN * j];
        int s64;
        mr_select64<R>(v, open, s64);
        if (open) sel = s64;
    }
    // NaN differences do not enter emax: the float selection was open then.  An
    // open window has spent its FP64 time already and takes the FP64 sum; so does
    // one that may have been left open for the sake of its warp.
    bool small = emax <= PAIR_RANGE * vc && sel < T && valid && !open && !noise;
#pragma unroll
    for (int j = 0; j < N; ++j) small = small && e[j] == e[j];
    // the form is each lane's own choice: the face shared by two tiles takes
    // the same one in both
    auto rest = [&](int j) { return DIRN > 0 ? e0[j] : make_float2(-e0[-j].x, -e0[-j].y); };
    double value = 0.0;
    const unsigned pairs = __ballot_sync(FULL, small);
    if (pairs == 0) {
        // none
    } else if (__all_sync(FULL, !small || sel == 0)) {
        PairSum q;
        q.first(Coef<R>::w()[0], rest(0));
#pragma unroll
        for (int j = 1; j < N; ++j) q.add(Coef<R>::w()[j], rest(j));
        value = v0[DIRN * c] + (widen(q.s) + widen(q.c));
    } else if (small) {
        const float2 *w = sW + sel * N;
        PairSum q;
        q.first(w[0], rest(0));
#pragma unroll
        for (int j = 1; j < N; ++j) q.add(w[j], rest(j));
        value = v0[DIRN * c] + (widen(q.s) + widen(q.c));
    }
    if (__any_sync(FULL, valid && !small)) {
        double v[W];
#pragma unroll
        for (int j = 0; j < W; ++j) v[j] = v0[DIRN * j];
        const double w = mr_recon<R>(v, sA, valid ? sel : 0);
        if (!small) value = w;
    }
    return value;
}

// From global memory: a warp reads constant memory one address at a time (order
// 17, 416 entries: 2e6 cells, one right-hand side 83 -> 55 us; 300 000 cells with a
// square pulse 22.6 -> 17.2 us).
template <int R>
__device__ __forceinline__ void load_w_table(float2 *sW, int tid, int nthreads)
{
    constexpr int N = R - 1;
    for (int i = tid; i < Tab<R>::T * N; i += nthreads) sW[i] = Coef<R>::w_table()[i];
}

// Resident CTAs (of 256 threads) per SM of the scalar kernels.  Long lines,
// eight of 32 registers: between the FP64 operations lie long float sums, and
// more warps fill the FP64 pipe's gaps although the sums spill.  Burgers, N =
// 2^22, order 9 / 13 / 17: 123 / 167 / 277 us a launch unbounded (58 to 84
// registers), 117 / 141 / 196 with five, 114 / 127 / 181 with eight; advection,
// N = 1 048 573, order 17: 65 -> 52.  Lines of at most two CTAs per SM, whose
// launches last as long as one CTA: unbounded, without the spills (Burgers, order
// 17, 3000 cells, five stages of the linear SSP family: 90 -> 79 us; 300 000 cells,
// 1177 CTAs: 137 with eight, 157 unbounded).
constexpr int SCALAR_CTAS = 8;
constexpr long long SCALAR_FEW_TILES = 2 * 152;

// ---------------------------------------------------------------------------
// Scalar advection f(u) = a u, alpha = |a|: f^+ = a u, f^- = 0 for a >= 0
// (mirror for a < 0).  One thread per interface.
// ---------------------------------------------------------------------------
template <int R, int TP, int MINB>
__global__ void __launch_bounds__(TP, MINB) k_advection(AdvArgs A)
{
    constexpr int g = (R + 1) / 2, W = 2 * g - 1, S = TP + 2 * g - 1, T = Tab<R>::T;
    __shared__ double sf[S];
    __shared__ float2 se[S];  // e[s] = f[s+1] - f[s]
    __shared__ double sFh[TP];
    __shared__ double sA[T * W];
    __shared__ float2 sW[T * (W - 1)];
    const int p = threadIdx.x;
    const long long x0 = (long long)blockIdx.x * (TP - 1);
    load_a_table<R>(sA, p, TP);
    load_w_table<R>(sW, p, TP);
    for (int s = p; s < S; s += TP) sf[s] = A.a * A.U[ghost(x0 - g + s, A.n, A.bc)];
    __syncthreads();
    for (int s = p; s < S - 1; s += TP) se[s] = split_pair(sf[s + 1] - sf[s]);
    __syncthreads();
    const long long k = x0 + p;  // interface x_{k-1/2}
    const bool valid = k <= A.n;
    int sel;
    const double fh = A.a >= 0.0 ? scalar_value<R, 1>(sf + p, se + p, sA, sW, valid, sel)
                                 : scalar_value<R, -1>(sf + p + 2 * g - 1, se + p + 2 * g - 2, sA,
                                                       sW, valid, sel);
    sFh[p] = fh;
    if (A.sel && valid) {
        const long long NI = A.n + 1;
        A.sel[(A.a >= 0.0 ? 0 : NI) + k] = (uint8_t)sel;
        A.sel[(A.a >= 0.0 ? NI : 0) + k] = (uint8_t)(T + 2);
    }
    __syncthreads();
    if (p < TP - 1) {
        const long long i = x0 + p;
        if (i < A.n) {
            with_epilogue_form(A.epi, [&](auto M, auto P) {
                epilogue_form<decltype(M)::value, decltype(P)::value != 0, false>(
                    A.epi, i, sFh[p + 1] - sFh[p], A.inv_h, A.U[i], false, 0.0);
            });
        }
    }
}

// ---------------------------------------------------------------------------
// Inviscid Burgers f(u) = u^2/2 (Sec. 4.2).  f'(u) = u: where u keeps one
// sign over the line the flux is not split (f^+ = f, f^- = 0, or the
// mirror); otherwise the global Lax-Friedrichs split with alpha = max |u|.
// The case is uniform over the launch (read from the speed reduction of
// the same state), so a warp never diverges on it.  One thread per
// interface; split values are formed as written, 1/2 (f +- alpha u).
// ---------------------------------------------------------------------------
template <int R, int TP, int MINB>
__global__ void __launch_bounds__(TP, MINB) k_burgers(AdvArgs A)
{
    constexpr int g = (R + 1) / 2, W = 2 * g - 1, S = TP + 2 * g - 1, T = Tab<R>::T;
    __shared__ double sp[S];
    __shared__ double sm[S];
    __shared__ float2 ep[S], em[S];  // differences of neighbouring split fluxes
    __shared__ double sFh[TP];
    __shared__ double sA[T * W];
    __shared__ float2 sW[T * (W - 1)];
    const int p = threadIdx.x;
    const long long x0 = (long long)blockIdx.x * (TP - 1);
    load_a_table<R>(sA, p, TP);
    load_w_table<R>(sW, p, TP);
    const double alpha = A.speed[0];
    const unsigned long long flags = (unsigned long long)__double_as_longlong(A.speed[1]);
    const int mode = !(flags & SGN_NEG) ? 0 : (!(flags & SGN_POS) ? 1 : 2);
    for (int s = p; s < S; s += TP) {
        const double u = A.U[ghost(x0 - g + s, A.n, A.bc)];
        const double f = 0.5 * __dmul_rn(u, u);
        double fp, fm;
        if (mode == 0) {
            fp = f;
            fm = 0.0;
        } else if (mode == 1) {
            fp = 0.0;
            fm = f;
        } else {
            const double au = __dmul_rn(alpha, u);
            fp = 0.5 * __dadd_rn(f, au);
            fm = 0.5 * __dsub_rn(f, au);
        }
        sp[s] = fp;
        sm[s] = fm;
    }
    __syncthreads();
    for (int s = p; s < S - 1; s += TP) {
        if (mode != 1) ep[s] = split_pair(sp[s + 1] - sp[s]);
        if (mode != 0) em[s] = split_pair(sm[s + 1] - sm[s]);
    }
    __syncthreads();
    const long long k = x0 + p;  // interface x_{k-1/2}
    const bool valid = k <= A.n;
    int selp = T + 2, selm = T + 2;
    double hp = 0.0, hm = 0.0;
    if (mode != 1)  // f^+ at cell k-1+l
        hp = scalar_value<R, 1>(sp + p, ep + p, sA, sW, valid, selp);
    if (mode != 0)  // f^- at cell k-l
        hm = scalar_value<R, -1>(sm + p + 2 * g - 1, em + p + 2 * g - 2, sA, sW, valid, selm);
    sFh[p] = __dadd_rn(hp, hm);
    if (A.sel && valid) {
        A.sel[k] = (uint8_t)selp;
        A.sel[A.n + 1 + k] = (uint8_t)selm;
    }
    __syncthreads();
    unsigned long long m = 0, fl = 0;
    if (p < TP - 1) {
        const long long i = x0 + p;
        if (i < A.n) {
            double o = 0.0;
            with_epilogue_form(A.epi, [&](auto M, auto P) {
                o = epilogue_form<decltype(M)::value, decltype(P)::value != 0, false>(
                    A.epi, i, sFh[p + 1] - sFh[p], A.inv_h, A.U[i], false, 0.0);
            });
            if (A.speed_next) {
                const long long b = __double_as_longlong(o);
                m = (unsigned long long)(b & 0x7fffffffffffffffLL);
                fl = m == 0 ? 0 : ((b < 0) ? SGN_NEG : SGN_POS);
                if (!below_1e300(o)) atomicOr(A.status, ST_NONPHYS_CELL);
            }
        }
    }
    if (!A.speed_next) return;
    // the next stage's speed and signs (k_scalar_speed): integer work only,
    // which the FP64 pipe hides, instead of a launch that reads the state again
    __shared__ unsigned long long red[TP / 32][2];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(FULL, m, o);
        m = m > x ? m : x;
        fl |= __shfl_xor_sync(FULL, fl, o);
    }
    if ((p & 31) == 0) {
        red[p >> 5][0] = m;
        red[p >> 5][1] = fl;
    }
    __syncthreads();
    if (p == 0) {
        for (int w = 1; w < TP / 32; ++w) {
            m = m > red[w][0] ? m : red[w][0];
            fl |= red[w][1];
        }
        atomicMax((unsigned long long *)A.speed_next, m);
        if (fl) atomicOr((unsigned long long *)(A.speed_next + 1), fl);
    }
}

}  // namespace enomr

namespace enomr {

// ---------------------------------------------------------------------------
// One SSP-RK3 step of a short scalar line in one launch: a cluster of CTAs, each
// with up to SMALL_TILE cells, their interfaces one per thread.  Every CTA holds
// the state of the whole line in shared memory; a stage's new cells go to all of
// them (distributed shared memory), one cluster barrier a stage.  The same
// operations per cell and interface as k_advection and k_burgers, and as many
// cells on an SM, so that the FP64 work of windows that the float form leaves
// open is spread as in their launches.  A line of n <= SMALL_CELLS is a few warps
// of work; launched one stage at a time it costs four (Burgers: seven) launches
// of about 5 us each.  A step, by launches of one stage each / in one CTA / over a
// cluster: advection, order 5, 1024 cells, smooth 23.8 / 21.5 / 14.1 us, constant
// up to rounding 27 / 58 / 20; order 17, random cells 92 / 56 / 20, constant up to
// rounding 92 / 325 / 77; Burgers, order 9, smooth 43 / 25 / 16; 200 cells, one CTA,
// order 5, bound by the host: 23.7 / 15.7 / 15.8, on the device alone - / 7.4 / 7.1.
// ---------------------------------------------------------------------------
template <int R, bool BURGERS>
struct SmallSmem {
    static constexpr int g = (R + 1) / 2, W = 2 * g - 1, T = Tab<R>::T, S = SMALL_TILE + 2 * g;
    double u[2][SMALL_CELLS];               // the stage's state, the next one's
    double fh[SMALL_TILE + 1];
    double f[BURGERS ? 2 : 1][S];           // f^+ (advection: the flux), f^-
    float2 e[BURGERS ? 2 : 1][S];
    double a[T * W];
    float2 w[T * (W - 1)];
    double dt, alpha;
    unsigned long long red[SMALL_THREADS / 32][2];
    int mode;
};

template <int R, bool BURGERS>
__global__ void __launch_bounds__(SMALL_THREADS) k_scalar_step(SmallArgs A)
{
    constexpr int g = (R + 1) / 2, T = Tab<R>::T;
    using SM = SmallSmem<R, BURGERS>;
    __shared__ SM sm;
    auto cluster = cooperative_groups::this_cluster();
    const int tid = threadIdx.x, n = (int)A.n;
    const int ctas = (int)gridDim.x, rank = (int)blockIdx.x;  // one cluster
    const int chunk = (n + ctas - 1) / ctas, c0 = rank * chunk;
    const int m = chunk < n - c0 ? chunk : n - c0;            // this CTA's cells: c0 ..
    load_a_table<R>(sm.a, tid, SMALL_THREADS);
    load_w_table<R>(sm.w, tid, SMALL_THREADS);
    for (int i = tid; i < n; i += SMALL_THREADS) sm.u[0][i] = A.U[i];
    if (tid == 0) {
        sm.dt = A.dt_fixed;
        sm.mode = A.a >= 0.0 ? 0 : 1;  // advection: the upwind side
    }
    // the line is read by all and every CTA has started: it may be written
    cluster.sync();
    const double u0 = tid < m ? sm.u[0][c0 + tid] : 0.0;
    for (int stage = 0; stage < 3; ++stage) {
        const double *u = sm.u[stage & 1];
        if constexpr (BURGERS) {
            // k_scalar_speed: max |u|, and which signs occur
            unsigned long long mx = 0, fl = 0;
            for (int i = tid; i < n; i += SMALL_THREADS) {
                const long long b = __double_as_longlong(u[i]);
                const unsigned long long x = (unsigned long long)(b & 0x7fffffffffffffffLL);
                if (!below_1e300(u[i])) atomicOr(A.status, ST_NONPHYS_CELL);
                mx = mx > x ? mx : x;
                if (x != 0) fl |= (b < 0) ? SGN_NEG : SGN_POS;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long x = __shfl_xor_sync(FULL, mx, o);
                mx = mx > x ? mx : x;
                fl |= __shfl_xor_sync(FULL, fl, o);
            }
            if ((tid & 31) == 0) {
                sm.red[tid >> 5][0] = mx;
                sm.red[tid >> 5][1] = fl;
            }
            __syncthreads();
            if (tid == 0) {
                for (int i = 1; i < SMALL_THREADS / 32; ++i) {
                    mx = mx > sm.red[i][0] ? mx : sm.red[i][0];
                    fl |= sm.red[i][1];
                }
                sm.alpha = __longlong_as_double((long long)mx);
                sm.mode = !(fl & SGN_NEG) ? 0 : (!(fl & SGN_POS) ? 1 : 2);
                if (stage == 0)
                    sm.dt = step_size(__dmul_rn(sm.alpha, A.inv_h), A.cfl, A.dt_fixed);
                if (rank == 0) {
                    A.speed[0] = sm.alpha;
                    A.speed[1] = __longlong_as_double((long long)fl);
                }
            }
            __syncthreads();
        }
        const int mode = sm.mode;
        // split fluxes with their ghost cells, then their differences
        for (int s = tid; s < m + 2 * g; s += SMALL_THREADS) {
            const double us = u[ghost(c0 + s - g, n, A.bc)];
            if constexpr (BURGERS) {
                const double f = 0.5 * __dmul_rn(us, us);
                double fp = f, fm = f;
                if (mode == 2) {
                    const double au = __dmul_rn(sm.alpha, us);
                    fp = 0.5 * __dadd_rn(f, au);
                    fm = 0.5 * __dsub_rn(f, au);
                }
                sm.f[0][s] = fp;
                sm.f[BURGERS ? 1 : 0][s] = fm;
            } else {
                sm.f[0][s] = A.a * us;
            }
        }
        __syncthreads();
        for (int s = tid; s < m + 2 * g - 1; s += SMALL_THREADS) {
            if (!BURGERS || mode != 1) sm.e[0][s] = split_pair(sm.f[0][s + 1] - sm.f[0][s]);
            if (BURGERS && mode != 0)
                sm.e[BURGERS ? 1 : 0][s] = split_pair(sm.f[BURGERS ? 1 : 0][s + 1] - sm.f[BURGERS ? 1 : 0][s]);
        }
        __syncthreads();
        if ((tid & ~31) <= m) {  // interface x_{c0+tid-1/2}
            const bool valid = tid <= m;
            const int p = valid ? tid : m;
            int sel = T + 2;
            double hp = 0.0, hm = 0.0;
            if (mode != 1)
                hp = scalar_value<R, 1>(sm.f[0] + p, sm.e[0] + p, sm.a, sm.w, valid, sel);
            if (mode != 0) {
                const int q = BURGERS ? 1 : 0;
                hm = scalar_value<R, -1>(sm.f[q] + p + 2 * g - 1, sm.e[q] + p + 2 * g - 2, sm.a, sm.w,
                                         valid, sel);
            }
            if (valid) sm.fh[tid] = BURGERS ? __dadd_rn(hp, hm) : (mode != 1 ? hp : hm);
        }
        __syncthreads();
        if (tid < m) {
            const double D = __dmul_rn(-(sm.fh[tid + 1] - sm.fh[tid]), A.inv_h);
            const double w = fma(sm.dt, D, u[c0 + tid]);
            const double o = stage == 0 ? w : fma(A.c0[stage], u0, A.c1[stage] * w);
            if (stage == 2) {
                A.U[c0 + tid] = o;
            } else {
                double *next = &sm.u[(stage + 1) & 1][c0 + tid];
                for (int r = 0; r < ctas; ++r) *cluster.map_shared_rank(next, r) = o;
            }
        }
        // every CTA has the next state, and none reads this one's any more; after
        // the last stage nothing of another CTA is written
        if (stage < 2) cluster.sync();
    }
    if (rank == 0 && tid == 0) *A.dt = sm.dt;
}

template <int R> cudaError_t launch_scalar_step(const SmallArgs &a, bool burgers, cudaStream_t s)
{
    static_assert(SMALL_CELLS <= 8 * SMALL_TILE, "a portable cluster");
    static_assert(SMALL_THREADS > SMALL_TILE, "one interface per thread");
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)((a.n + SMALL_TILE - 1) / SMALL_TILE);
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(attr.val.clusterDim.x);
    cfg.blockDim = dim3(SMALL_THREADS);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = a.n > SMALL_TILE ? 1 : 0;  // one CTA: 0.5 us less than as a cluster of one
    return burgers ? cudaLaunchKernelEx(&cfg, k_scalar_step<R, true>, a)
                   : cudaLaunchKernelEx(&cfg, k_scalar_step<R, false>, a);
}

}  // namespace enomr
