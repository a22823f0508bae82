// Device helpers shared by the forward and adjoint predictor-corrector kernels: geometry,
// radial stencils on global / shared columns, and the banded substitutions with the
// pivoted LU factors of Sec. 3.2.
#pragma once

#include "tc_internal.cuh"
#include "tc_fx.cuh"

namespace tc {

struct Geo {
    int N, M, K, nk, nmode, K1, M1K1;
    int mlo, mhi;            // modes [mlo, mhi) handled by a launch (default: all)
    int sh;                  // fused steps 2-5: systems cut at row sh into two partitions (0: uncut)
    size_t S;
    double mp, kz, dt, c1;   // c1 = 1 / (2 dt)
};

static inline Geo geo(const tc_plan* p) {
    Geo g;
    g.N = p->N_r; g.M = p->M; g.K = p->K; g.nk = 2 * p->K + 1; g.nmode = p->nmode;
    g.K1 = p->K + 1; g.M1K1 = (p->M + 1) * (p->K + 1); g.S = p->S;
    g.mlo = 0; g.mhi = g.nmode;
    g.sh = 0;
    g.mp = (double)p->m_p; g.kz = p->k_z; g.dt = p->dt; g.c1 = 1.0 / (2.0 * p->dt);
    return g;
}

// first and second radial derivative of column `mode` of a scalar field at row j
__device__ __forceinline__ double2 drow(const double2* __restrict__ f, const double* __restrict__ w,
                                        const int* __restrict__ col0, int j, int nmode, int mode) {
    const int c0 = col0[j];
    double2 s = make_double2(0.0, 0.0);
    stencil_taps<true>(c0, [&](int t) {
        const double wt = __ldg(&w[j * kStencil + t]);
        const double2 v = f[(size_t)(c0 + t) * nmode + mode];
        s.x += wt * v.x;
        s.y += wt * v.y;
    });
    return s;
}

// (Lap u)_r = ((L_+ u_+) + (L_- u_-)) / 2 at row j, L_pm = Lap_h - 1/r^2 -+ 2 m m_p / r^2
static __device__ double2 lap_r(const double2* __restrict__ u, const double* __restrict__ w1,
                         const double* __restrict__ w2, const int* __restrict__ col0,
                         double r, int j, int mode, double mm, double kk, const Geo& g) {
    double2 acc = make_double2(0.0, 0.0);
    const double ir = 1.0 / r, ir2 = ir * ir;
    for (int c = 0; c < 2; ++c) {
        const double2* f = u + (size_t)c * g.S;
        const double2 d1 = drow(f, w1, col0, j, g.nmode, mode);
        const double2 d2 = drow(f, w2, col0, j, g.nmode, mode);
        const double2 v = f[(size_t)j * g.nmode + mode];
        const double sgn = c == 0 ? -1.0 : 1.0;
        const double diag = -mm * mm * ir2 - kk * kk - ir2 + sgn * 2.0 * mm * ir2;
        acc.x += d2.x + ir * d1.x + diag * v.x;
        acc.y += d2.y + ir * d1.y + diag * v.y;
    }
    acc.x *= 0.5;
    acc.y *= 0.5;
    return acc;
}

// ---------------------------------------------------------------- fused steps 2-5
// One block owns T consecutive modes (all N_r rows).  Shared memory holds four complex
// columns per mode, row-major [j][t]: C0 = b_p -> p* -> div u* -> phi, C1..C3 = u*_c.
// X = (2N - N_prev)_r (pressure stage) is staged in C1 before C1 receives u*_+.

// In-place banded substitution on one real part (part = 0: re, 1: im) of column t of a
// [N][T] complex smem array, with the pivoted LU of Sec. 3.2 stored for (set, m, |k|).
// The factors of the next D rows are kept in flight in a register ring: the few long
// substitution chains of a block wait on each row's factors otherwise (they come from DRAM:
// a step streams more than L2 holds between two uses), and one row of arithmetic does not
// cover that latency.
template <int D = 1>
__device__ __forceinline__ void smem_band_solve(double2* col, int T, int off, int N,
                                                const double* __restrict__ F, const uint8_t* __restrict__ P,
                                                int M1K1) {
    double* x = reinterpret_cast<double*>(col) + off;   // x[j] at x[2 T j]
    const int st = 2 * T;
    const size_t rs = (size_t)kBands * M1K1;                      // one row of factors
    // forward: rows j .. j+4 live in w0..w4
    double w0 = x[0], w1 = N > 1 ? x[st] : 0.0, w2 = N > 2 ? x[2 * st] : 0.0,
           w3 = N > 3 ? x[3 * st] : 0.0, w4 = N > 4 ? x[4 * st] : 0.0;
    double lr[D][4];
    int pr[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        pr[d] = 0;
        lr[d][0] = lr[d][1] = lr[d][2] = lr[d][3] = 0.0;
        if (d < N) {
            const double* Fr = F + (size_t)d * rs;
            pr[d] = P[(size_t)d * M1K1];
#pragma unroll
            for (int q = 0; q < 4; ++q) lr[d][q] = __ldg(&Fr[(size_t)q * M1K1]);
        }
    }
    for (int j0 = 0; j0 < N; j0 += D) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int j = j0 + d;
            if (j < N) {
                const int pj = pr[d];
                const double l1 = lr[d][0], l2 = lr[d][1], l3 = lr[d][2], l4 = lr[d][3];
                if (j + D < N) {   // refill this slot with row j + D
                    const double* Fr = F + (size_t)(j + D) * rs;
                    pr[d] = P[(size_t)(j + D) * M1K1];
#pragma unroll
                    for (int q = 0; q < 4; ++q) lr[d][q] = __ldg(&Fr[(size_t)q * M1K1]);
                }
                if (pj == 1) { double q = w0; w0 = w1; w1 = q; }
                else if (pj == 2) { double q = w0; w0 = w2; w2 = q; }
                else if (pj == 3) { double q = w0; w0 = w3; w3 = q; }
                else if (pj == 4) { double q = w0; w0 = w4; w4 = q; }
                x[(size_t)j * st] = w0;
                w1 = fma(-l1, w0, w1);
                w2 = fma(-l2, w0, w2);
                w3 = fma(-l3, w0, w3);
                w4 = fma(-l4, w0, w4);
                w0 = w1; w1 = w2; w2 = w3; w3 = w4;
                w4 = (j + 5 < N) ? x[(size_t)(j + 5) * st] : 0.0;
            }
        }
    }
    // backward: x_{j+1..j+8} in v1..v8.  Row-oriented.  A column-oriented variant (each x_j
    // taken out of the rows above at once: two dependent operations per row instead of nine,
    // same results bit for bit) measured slower on GB300 (k_pc 0.547 against 0.286 ms at
    // N_r = 64): each FP64 instruction costs its warp the same issue time whatever the chain,
    // so the substitution is bound by the count of FP64 instructions, not by their latency
    double v1 = 0.0, v2 = 0.0, v3 = 0.0, v4 = 0.0, v5 = 0.0, v6 = 0.0, v7 = 0.0, v8 = 0.0;
    double ur[D][9];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const int j = N - 1 - d;
#pragma unroll
        for (int q = 0; q < 9; ++q) ur[d][q] = j >= 0 ? __ldg(&F[(size_t)j * rs + (size_t)(4 + q) * M1K1]) : 0.0;
    }
    for (int j0 = N - 1; j0 >= 0; j0 -= D) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int j = j0 - d;
            if (j >= 0) {
                double uc[9];
#pragma unroll
                for (int q = 0; q < 9; ++q) uc[q] = ur[d][q];
                if (j - D >= 0) {   // refill this slot with row j - D
#pragma unroll
                    for (int q = 0; q < 9; ++q) ur[d][q] = __ldg(&F[(size_t)(j - D) * rs + (size_t)(4 + q) * M1K1]);
                }
                double s = x[(size_t)j * st];
                s = fma(-uc[8], v8, s);
                s = fma(-uc[7], v7, s);
                s = fma(-uc[6], v6, s);
                s = fma(-uc[5], v5, s);
                s = fma(-uc[4], v4, s);
                s = fma(-uc[3], v3, s);
                s = fma(-uc[2], v2, s);
                s = fma(-uc[1], v1, s);
                const double xj = s * uc[0];
                x[(size_t)j * st] = xj;
                v8 = v7; v7 = v6; v6 = v5; v5 = v4; v4 = v3; v3 = v2; v2 = v1; v1 = xj;
            }
        }
    }
}

// The same substitution with the factors fetched in chunks, CF rows (forward) and CB rows
// (backward) ahead in a second register buffer.  A ring that is refilled row by row leaves the
// loads of several rows on one scoreboard, and waiting for a row then waits for the youngest of
// them, a memory latency per row; a chunk's loads are waited for once, a chunk later.
// INIT: set the buffers first, for a call within a loop, around which ptxas otherwise keeps them live and spills.
template <int CF, int CB, bool INIT>
__device__ __forceinline__ void smem_band_solve_c(double2* col, int T, int off, int N,
                                                  const double* __restrict__ F, const uint8_t* __restrict__ P,
                                                  int M1K1) {
    double* x = reinterpret_cast<double*>(col) + off;   // x[j] at x[2 T j]
    const int st = 2 * T;
    const size_t rs = (size_t)kBands * M1K1;
    double w0 = x[0], w1 = N > 1 ? x[st] : 0.0, w2 = N > 2 ? x[2 * st] : 0.0,
           w3 = N > 3 ? x[3 * st] : 0.0, w4 = N > 4 ? x[4 * st] : 0.0;
    {
        double lr[2][CF][4];
        int pr[2][CF];
        if (INIT) {
#pragma unroll
            for (int i = 0; i < 2 * CF; ++i) {
                pr[i / CF][i % CF] = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) lr[i / CF][i % CF][q] = 0.0;
            }
        }
        auto load = [&](double (&l)[CF][4], int (&p)[CF], int c) {
#pragma unroll
            for (int d = 0; d < CF; ++d) {
                const int j = min(c * CF + d, N - 1);
                p[d] = __ldg(&P[(size_t)j * M1K1]);
#pragma unroll
                for (int q = 0; q < 4; ++q) l[d][q] = __ldg(&F[(size_t)j * rs + (size_t)q * M1K1]);
            }
        };
        load(lr[0], pr[0], 0);
        const int nc = (N + CF - 1) / CF;
        for (int c0 = 0; c0 < nc; c0 += 2) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                if (c0 + b < nc) {
                    load(lr[b ^ 1], pr[b ^ 1], c0 + b + 1);
#pragma unroll
                    for (int d = 0; d < CF; ++d) {
                        const int j = (c0 + b) * CF + d;
                        if (j < N) {
                            const int pj = pr[b][d];
                            if (pj == 1) { double q = w0; w0 = w1; w1 = q; }
                            else if (pj == 2) { double q = w0; w0 = w2; w2 = q; }
                            else if (pj == 3) { double q = w0; w0 = w3; w3 = q; }
                            else if (pj == 4) { double q = w0; w0 = w4; w4 = q; }
                            x[(size_t)j * st] = w0;
                            w1 = fma(-lr[b][d][0], w0, w1);
                            w2 = fma(-lr[b][d][1], w0, w2);
                            w3 = fma(-lr[b][d][2], w0, w3);
                            w4 = fma(-lr[b][d][3], w0, w4);
                            w0 = w1; w1 = w2; w2 = w3; w3 = w4;
                            w4 = (j + 5 < N) ? x[(size_t)(j + 5) * st] : 0.0;
                        }
                    }
                }
            }
        }
    }
    double v1 = 0.0, v2 = 0.0, v3 = 0.0, v4 = 0.0, v5 = 0.0, v6 = 0.0, v7 = 0.0, v8 = 0.0;
    double ur[2][CB][9];
    if (INIT) {
#pragma unroll
        for (int i = 0; i < 2 * CB; ++i)
#pragma unroll
            for (int q = 0; q < 9; ++q) ur[i / CB][i % CB][q] = 0.0;
    }
    auto load = [&](double (&u)[CB][9], int c) {
#pragma unroll
        for (int d = 0; d < CB; ++d) {
            const int j = max(N - 1 - (c * CB + d), 0);
#pragma unroll
            for (int q = 0; q < 9; ++q) u[d][q] = __ldg(&F[(size_t)j * rs + (size_t)(4 + q) * M1K1]);
        }
    };
    load(ur[0], 0);
    const int nc = (N + CB - 1) / CB;
    for (int c0 = 0; c0 < nc; c0 += 2) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            if (c0 + b < nc) {
                load(ur[b ^ 1], c0 + b + 1);
#pragma unroll
                for (int d = 0; d < CB; ++d) {
                    const int j = N - 1 - ((c0 + b) * CB + d);
                    if (j >= 0) {
                        double s = x[(size_t)j * st];
                        s = fma(-ur[b][d][8], v8, s);
                        s = fma(-ur[b][d][7], v7, s);
                        s = fma(-ur[b][d][6], v6, s);
                        s = fma(-ur[b][d][5], v5, s);
                        s = fma(-ur[b][d][4], v4, s);
                        s = fma(-ur[b][d][3], v3, s);
                        s = fma(-ur[b][d][2], v2, s);
                        s = fma(-ur[b][d][1], v1, s);
                        const double xj = s * ur[b][d][0];
                        x[(size_t)j * st] = xj;
                        v8 = v7; v7 = v6; v6 = v5; v5 = v4; v4 = v3; v3 = v2; v2 = v1; v1 = xj;
                    }
                }
            }
        }
    }
}

// The element loops of k_pc with a radial stencil: body(j, i, d, pre(j)) for the real
// and imaginary parts of all rows of the block's modes, i the index of the part's double in the
// [N][T] arrays in shared memory, d the stencil at row j of F (of F + F2 with pair).  pre: the body's
// load from device memory, issued ahead of the stencil.  slow(j, c): the FP64 sum at row j of column c.
// slow's last argument: whether to guard the rows below 0 (N < kStencil).
// FX: all but the ZONE rows next to each wall in tiles of kTileRows rows per thread in fixed point
// (weights fw, few; rows beyond the limit far in FP64, see fx::Tile), the others one per thread, by the
// other half of the block first.  A tile's FP64 sums share one copy in a rolled loop: 9 to 18 instructions
// a row unrolled four times are most of a stage's code, and they are rarely taken.
// Otherwise all in FP64, two rows at a time: a warp may issue an FP64 instruction every 64 cycles, and one
// chain of dependent FMAs does not fill that (N_r = 160, M = 8, K = 16: k_pc 229 -> 225 us; N_r = 64,
// M = 64, K = 128: 903 -> 873 us).
constexpr int kTileRows = 4;   // rows per thread, here and in the split path
template <int ZONE, bool FX, bool PAIR, class Slow, class Pre, class Body>
__device__ __forceinline__ void stencil_rows(const int2* __restrict__ fw, const int2* __restrict__ few, int far, const double2* F,
                                             const double2* F2, int N, int T, Slow slow, Pre pre, Body body) {
    using namespace fx;
    const int c = threadIdx.x % (2 * T), step = blockDim.x / (2 * T), st = 2 * T;
    if (FX) {
        const double* f = reinterpret_cast<const double*>(F) + c;
        const double* f2 = reinterpret_cast<const double*>(F2) + c;
#pragma unroll 1
        for (int j0 = ZONE + kTileRows * (threadIdx.x / st); j0 < N - ZONE; j0 += kTileRows * step) {
            double d[kTileRows], g[kTileRows];
#pragma unroll
            for (int i = 0; i < kTileRows; ++i) g[i] = pre(min(j0 + i, N - 1));
            unsigned fp64;
            {
                Tile<kTileRows> X;
                double v[kTileRows + 8], v2[kTileRows + 8];
#pragma unroll
                for (int i = 0; i < kTileRows + 8; ++i) {
                    const int j = j0 - 4 + i;
                    v[i] = j < N ? f[j * st] : 0.0;
                    if (PAIR) v2[i] = j < N ? f2[j * st] : 0.0;
                }
                auto near = [&](int i) { return (unsigned)__ldg(&few[min(j0 + i, N - ZONE - 1)].y); };
                if (PAIR) X.load(v, v2, far, near);
                else X.load(v, far, near);
                fp64 = X.fp64;
#pragma unroll
                for (int i = 0; i < kTileRows; ++i) {
                    const int j = min(j0 + i, N - ZONE - 1);
                    d[i] = X.row(i, fw + j * kStencil, __ldg(&few[j].x));
                }
            }
            if (fp64) {
#pragma unroll 1
                for (int i = 0; i < kTileRows; ++i)
                    if ((fp64 >> i) & 1) {
                        const double o = slow(min(j0 + i, N - ZONE - 1), c, std::false_type{});
#pragma unroll
                        for (int q = 0; q < kTileRows; ++q) d[q] = i == q ? o : d[q];
                    }
            }
#pragma unroll
            for (int i = 0; i < kTileRows; ++i)
                if (j0 + i < N - ZONE) body(j0 + i, (j0 + i) * st + c, d[i], g[i]);
        }
    }
    if (FX) {
        for (int i = (threadIdx.x ^ (blockDim.x >> 1)) / st; i < min(N, 2 * ZONE); i += step) {
            const int j = N < 2 * ZONE || i < ZONE ? i : N - 2 * ZONE + i;
            const double g = pre(j);
            body(j, j * st + c, slow(j, c, std::false_type{}), g);
        }
        return;
    }
    int j = threadIdx.x / st;
    if (N >= kStencil) {
        for (; j + step < N; j += 2 * step) {
            const double g = pre(j), g2 = pre(j + step);
            const double o = slow(j, c, std::false_type{}), o2 = slow(j + step, c, std::false_type{});
            body(j, j * st + c, o, g);
            body(j + step, (j + step) * st + c, o2, g2);
        }
    }
    for (; j < N; j += step) {
        const double g = pre(j);
        body(j, j * st + c, slow(j, c, std::true_type{}), g);
    }
}

}  // namespace tc
