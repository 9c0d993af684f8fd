// enomr_line.cuh -- the 1D Euler sweep of one problem, its windows spread over
// warps, and the wave-speed reduction with the CFL step in one launch.
//
// arXiv 2311.15504: Sec. 2.1 (Eq. 1DWENOFD, Eq. LF_Flux_Split), Sec. 3.2,
// Sec. 4, Eq. TVD3rdRK.
//
// A line of a few thousand cells leaves the chip nearly empty: its launches
// last as long as one tile, and a tile as long as its longest chain of FP64
// warp instructions (64 cycles each on an SM sub-partition, however many lanes
// they carry).  With one lane per interface that chain holds the cell, the
// Roe average, three projections and six windows.  Here a CTA takes 32
// interfaces with six warps: warp w evaluates field w % 3, side w / 3 of all
// of them, so the six windows run side by side on the four sub-partitions
// (their projections are formed once per side, a fifth more FP64 work), and
// one warp each does the Roe averages and the back-projection.  The stage's
// epilogue also takes the new state's wave speeds for the next stage.
// Same operations per cell, interface and window as sweep_tile.
// Measured (GB300, shock / entropy wave, a launch / an SSP-RK3 step): order 9,
// 400 cells: 41 -> 18 us / 155 -> 57 us; order 17, 6400 cells: 109 -> 45 us /
// 362 -> 137 us.
#pragma once

#include "enomr_sweep.cuh"

namespace enomr {

constexpr int LINE_TP = 32, LINE_THREADS = 192;

// Longest line that runs here; above, where the chip is full, k_sweep, which
// forms a window's projections once for both sides.  A step on the shock /
// entropy wave, this over k_sweep (the same with random cells): order 9, 20 000
// cells 0.81 (0.72), 40 000 0.99 (1.00), 65 000 1.10 (1.22), 131 072 1.17
// (1.22); order 5 0.85, 0.97, 1.09, 1.16; order 11, 40 000 0.84 (0.86), 65 000
// 0.99 (1.03), 100 000 1.15 (1.19); order 17 0.75 (0.84), 0.92 (0.98), 1.06 (1.13).
template <int R>
constexpr long long LINE_MAX_CELLS = R <= 9 ? 40000 : 65000;

template <int R>
__global__ void __launch_bounds__(LINE_THREADS) k_line(SweepArgs A)
{
    constexpr int g = (R + 1) / 2, W = 2 * g - 1, S = LINE_TP + 2 * g - 1, T = Tab<R>::T;
    constexpr int c = g - 1;
    static_assert(S <= 64, "two warps stage the cells");
    __shared__ double sU[3][S], sF[3][S], sP[3][S];  // P: sqrt(rho), u, H
    __shared__ double sRoe[7][LINE_TP];              // u, H, hq, c, kappa, c2g, b1
    __shared__ double sV[6][LINE_TP];                // value of (side, field)
    __shared__ double sFh[3][LINE_TP], sO[3][LINE_TP];
    __shared__ unsigned char sClass[LINE_TP];
    __shared__ double sA[T * W];
    enum : int { ONE_STATE = 0, FLAT = 1, WINDOW = 2 };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long n = A.nx, x0 = (long long)blockIdx.x * (LINE_TP - 1);
    const long long k = x0 + lane;  // interface x_{k-1/2} of this lane
    const bool valid = k <= n;
    const int sl = lane + g - 1, sr = lane + g;

    // ---- cells, and the table
    if (tid < S) {
        const long long cell = ghost(x0 - g + tid, n, A.bc);
        const double rho = A.U[cell], m = A.U[n + cell], E = A.U[2 * n + cell];
        const StagedCell<3> sc = stage_cell<3>(rho, m, 0.0, E, A.gm1);
        if (!positive(rho) || !positive(sc.p) || !below_1e300(E)) atomicOr(A.status, ST_NONPHYS_CELL);
        sU[0][tid] = rho;
        sU[1][tid] = m;
        sU[2][tid] = E;
#pragma unroll
        for (int q = 0; q < 3; ++q) sF[q][tid] = sc.F[q];
        sP[0][tid] = sc.sq;
        sP[1][tid] = sc.un;
        sP[2][tid] = sc.H;
    } else {
        load_a_table<R>(sA, tid - S, LINE_THREADS - S);
    }
    __syncthreads();
    // ---- Roe averages; flat interfaces (sweep_tile)
    if (warp == 0) {
        auto same = [&](int a, int b) {
            bool e = true;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                e = e && __double_as_longlong(sU[q][a]) == __double_as_longlong(sU[q][b]);
            return e;
        };
        const bool e0 = same(sl - 2, sl - 1), e1 = same(sl - 1, sl), e2 = same(sl, sr),
                   e3 = same(sr, sr + 1), e4 = same(sr + 1, sr + 2);
        const bool flat = ((e0 && e1) || (e2 && e3)) && ((e3 && e4) || (e1 && e2));
        const int cls = !flat ? WINDOW : (e2 && !A.ft_out ? ONE_STATE : FLAT);
        sClass[lane] = (unsigned char)cls;
        if (__any_sync(FULL, valid && cls != ONE_STATE)) {
            const RoeFace rf = roe_face(e2, sP[0][sl], sP[1][sl], 0.0, sP[2][sl], sP[0][sr],
                                        sP[1][sr], 0.0, sP[2][sr], false, A.gm1, A.inv_gm1);
            if (valid && cls != ONE_STATE && !positive(rf.c2)) atomicOr(A.status, ST_NONPHYS_ROE);
            sRoe[0][lane] = rf.uh;
            sRoe[1][lane] = rf.Hh;
            sRoe[2][lane] = rf.hq;
            sRoe[3][lane] = rf.cs;
            sRoe[4][lane] = rf.kap;
            sRoe[5][lane] = rf.c2g;
            sRoe[6][lane] = rf.b1;
        }
    }
    __syncthreads();
    const int cls = sClass[lane];
    // ---- windows: warp = (side, field)
    {
        const int f = warp % 3, side = warp / 3;
        const bool window = valid && cls == WINDOW;
        int sel = T + 2;
        if (__any_sync(FULL, valid && cls != ONE_STATE)) {
            const double uh = sRoe[0][lane], hq = sRoe[2][lane], kap = sRoe[4][lane];
            const double l0 = f == 0 ? fma(uh, kap, hq)
                                     : (f == 2 ? fma(-uh, kap, hq) : hq - sRoe[5][lane]);
            const double l1 = f == 0 ? -(uh + kap) : (f == 2 ? -(uh - kap) : -uh);
            const double a = side ? -A.alpha[f] : A.alpha[f];
            auto value = [&](int s) {
                const double w = fma(l0, sU[0][s], fma(l1, sU[1][s], sU[2][s]));
                const double q = fma(l0, sF[0][s], fma(l1, sF[1][s], sF[2][s]));
                return fma(a, w, q);
            };
            double r;
            if (__any_sync(FULL, window)) {
                double v[W];
#pragma unroll
                for (int j = 0; j < W; ++j) v[j] = value(side ? lane + 2 * g - 1 - j : lane + j);
                int s;
                mr_select<R>(v, window, s);
                r = mr_recon<R>(v, sA, s);
                if (window)
                    sel = s;
                else
                    r = v[c];
            } else {
                r = value(side ? sr : sl);
            }
            sV[warp][lane] = r;
        }
        if (A.sel && valid) A.sel[(side * 3 + f) * (n + 1) + k] = (uint8_t)sel;
    }
    __syncthreads();
    // ---- back-projection
    if (warp == 0) {
        double Fh[3];
        if (cls == ONE_STATE) {
#pragma unroll
            for (int q = 0; q < 3; ++q) Fh[q] = sF[q][sr];
        } else {
            double ft[3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                ft[f] = sV[f][lane] + sV[3 + f][lane];
                if (A.ft_out && valid) A.ft_out[f * (n + 1) + k] = ft[f];
            }
            back_project3(sRoe[0][lane], sRoe[1][lane], sRoe[2][lane], sRoe[3][lane],
                          sRoe[6][lane], ft, Fh);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) sFh[q][lane] = Fh[q];
    }
    __syncthreads();
    // ---- stage update: warp q takes component q of the 31 cells
    const bool mine = lane < LINE_TP - 1 && k < n;
    if (warp < 3 && mine) {
        double o = 0.0;
        with_epilogue_form(A.epi, [&](auto M, auto P) {
            o = epilogue_form<decltype(M)::value, decltype(P)::value != 0, false>(
                A.epi, warp * n + k, sFh[warp][lane + 1] - sFh[warp][lane], A.inv_h,
                sU[warp][lane + g], false, 0.0);
        });
        sO[warp][lane] = o;
    }
    if (!A.alpha_next) return;
    __syncthreads();
    if (warp == 0) {
        unsigned long long ws[3] = {0, 0, 0};
        if (mine) {
            double w3[3];
            wave_speeds3(sO[0][lane], sO[1][lane], sO[2][lane], A.gm1, A.gamma, w3, A.status);
#pragma unroll
            for (int i = 0; i < 3; ++i) ws[i] = (unsigned long long)__double_as_longlong(w3[i]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long w = __shfl_xor_sync(FULL, ws[i], o);
                ws[i] = ws[i] > w ? ws[i] : w;
            }
            if (lane == i) atomicMax((unsigned long long *)(A.alpha_next + i), ws[i]);
        }
    }
}

template <int R> cudaError_t launch_line(const SweepArgs &a, cudaStream_t s)
{
    const long long tiles = (a.nx + LINE_TP - 2) / (LINE_TP - 1);
    k_line<R><<<(unsigned)tiles, LINE_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace enomr
