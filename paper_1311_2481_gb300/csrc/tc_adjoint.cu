// Adjoint of the AB2BD2 step (differentiation form; the paper has no adjoint).  The step maps
// (u^i, u^{i-1}, N^{i-1}) -> (u^{i+1}, u^i, N^i) and is affine except for N(u) = u . grad u,
// so its adjoint is the transposed chain of the linear part (steps 2-5 of Sec. 3.2:
// transposed banded solves, transposed stencils) plus the transposed linearised nonlinear
// term about the forward state (transposed forward transforms = unscaled inverse transforms
// and vice versa, the transposed pointwise products, the transposed radial stencil).  The
// inner product is the Euclidean one on the stored (Re, Im) pairs.
#include "tc_solve_core.cuh"

namespace tc {

static int ablocks(size_t n, int bs) { return (int)((n + bs - 1) / bs); }

// x <- A^{-T} x on one real part of column t of a [N][T] smem array, for A = P L U stored
// as in smem_band_solve: first U^T y = x (forward), then for j = N-1..0 the transposed
// elimination x_j -= sum_q l_q(j) x_{j+q} followed by the row interchange j <-> j + piv_j.
// The factors come in chunks of CB (U) and CF (L) rows, as in smem_band_solve_c.
template <int CF, int CB>
__device__ __forceinline__ void smem_band_solve_T(double2* col, int T, int t, int part, int N,
                                                  const double* __restrict__ F,
                                                  const uint8_t* __restrict__ P, int M1K1) {
    double* x = reinterpret_cast<double*>(col) + 2 * t + part;
    const int st = 2 * T;
    // U^T y = b: y_j = (b_j - sum_{q=1..8} U(j-q, j) y_{j-q}) / U_jj, column-oriented: p0..p7
    // hold the partial sums of rows j .. j+7, and y_j is taken out of rows j+1 .. j+8 as soon
    // as it is known, with U(j, j+q) = band 4+q of row j (one FMA and one multiply between
    // consecutive y)
    const size_t rs = (size_t)kBands * M1K1;
    double p0 = N > 0 ? x[0] : 0.0, p1 = N > 1 ? x[(size_t)st] : 0.0, p2 = N > 2 ? x[(size_t)2 * st] : 0.0;
    double p3 = N > 3 ? x[(size_t)3 * st] : 0.0, p4 = N > 4 ? x[(size_t)4 * st] : 0.0;
    double p5 = N > 5 ? x[(size_t)5 * st] : 0.0, p6 = N > 6 ? x[(size_t)6 * st] : 0.0;
    double p7 = N > 7 ? x[(size_t)7 * st] : 0.0;
    {
        double ur[2][CB][9];
        auto load = [&](double (&u)[CB][9], int c) {
#pragma unroll
            for (int d = 0; d < CB; ++d) {
                const int j = min(c * CB + d, N - 1);
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
                        const int j = (c0 + b) * CB + d;
                        if (j < N) {
                            const double* u = ur[b][d];
                            const double yj = p0 * u[0];
                            x[(size_t)j * st] = yj;
                            const double p8 = j + 8 < N ? x[(size_t)(j + 8) * st] : 0.0;
                            p0 = fma(-u[1], yj, p1);
                            p1 = fma(-u[2], yj, p2);
                            p2 = fma(-u[3], yj, p3);
                            p3 = fma(-u[4], yj, p4);
                            p4 = fma(-u[5], yj, p5);
                            p5 = fma(-u[6], yj, p6);
                            p6 = fma(-u[7], yj, p7);
                            p7 = fma(-u[8], yj, p8);
                        }
                    }
                }
            }
        }
    }
    // transposed eliminations and interchanges, j = N-1 .. 0; w1..w4 hold x_{j+1..j+4}
    double w1 = 0.0, w2 = 0.0, w3 = 0.0, w4 = 0.0;
    double lr[2][CF][4];
    int pr[2][CF];
    auto load = [&](double (&l)[CF][4], int (&p)[CF], int c) {
#pragma unroll
        for (int d = 0; d < CF; ++d) {
            const int j = max(N - 1 - (c * CF + d), 0);
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
                    const int j = N - 1 - ((c0 + b) * CF + d);
                    if (j >= 0) {
                        const int pj = pr[b][d];
                        double w0 = x[(size_t)j * st];
                        // oldest values first: without an interchange at row j+1 only w1 is new
                        w0 = fma(-lr[b][d][3], w4, w0);
                        w0 = fma(-lr[b][d][2], w3, w0);
                        w0 = fma(-lr[b][d][1], w2, w0);
                        w0 = fma(-lr[b][d][0], w1, w0);
                        if (pj == 1) { double q = w0; w0 = w1; w1 = q; }
                        else if (pj == 2) { double q = w0; w0 = w2; w2 = q; }
                        else if (pj == 3) { double q = w0; w0 = w3; w3 = q; }
                        else if (pj == 4) { double q = w0; w0 = w4; w4 = q; }
                        if (j + 4 < N) x[(size_t)(j + 4) * st] = w4;   // x_{j+4} is final
                        w4 = w3; w3 = w2; w2 = w1; w1 = w0;
                    }
                }
            }
        }
    }
    // flush the window: x_0..x_3
    if (N > 0) x[0] = w1;
    if (N > 1) x[(size_t)st] = w2;
    if (N > 2) x[(size_t)2 * st] = w3;
    if (N > 3) x[(size_t)3 * st] = w4;
}

constexpr int kAdjChunkF = 4, kAdjChunkB = 2;

struct PCAdjArgs {
    const double2* ubar_new;   // adjoint of u^{i+1}
    const double2* ubar_cur;   // adjoint of u^i from the later step (may be null: zero)
    const double2* Nbar_cur;   // adjoint of N^i from the later step (may be null: zero)
    double2* u_out;            // ubar_cur + linear-part adjoint of u^i (nonlinear part added later)
    double2* up_out;           // adjoint of u^{i-1}
    double2* N_out;            // total adjoint of N^i (input of the transposed nonlinear term)
    double2* Np_out;           // adjoint of N^{i-1}
    const double* ir;   // 1 / r_j
    const double* w1;
    const double* w2;
    const int* col0;
    const int* trow;
    const double* tw;
    int ntab;
    const double* fac;
    const uint8_t* piv;
};

// Adjoint of k_pc (steps 2-5 of Sec. 3.2), phases in reverse order.  Shared memory as in
// k_pc: C0 scalar column, C1..C3 vector columns, [N][T] each.
// Bound by latency and the FP64 pipe in turn (three substitutions of N rows, one DFMA per 64 cycles
// and warp).  The element loops run over the real and imaginary parts, each thread staying with its
// mode, divisions by dt are taken once, and ubar and u_prev's adjoint are written by the warps that
// idle during the last substitution: 561 -> 419 us at N_r = 96, M = 32, K = 64.  The transposed
// stencils stay FP64 sums in table order: the Poisson substitutions that follow magnify a rounding
// of their input by up to 10^7, so fixed point (391 us) moves the wall rows of the result by 1e-9.
template <int NTH>
__global__ void __launch_bounds__(NTH, 512 / NTH) k_pc_adj(PCAdjArgs a, Geo g, int T) {
    extern __shared__ double2 sm[];
    const int N = g.N;
    const int items = N * T;
    double2* C0 = sm;
    double2* C1 = sm + items;
    double2* C2 = C1 + items;
    double2* C3 = C2 + items;
    double2* Cv[3] = {C1, C2, C3};
    double *D0 = reinterpret_cast<double*>(C0), *D1 = D0 + 2 * items, *D2 = D1 + 2 * items, *D3 = D2 + 2 * items;
    const int mode0 = blockIdx.x * T;
    const int nT = min(T, g.nmode - mode0);
    const size_t per_set = (size_t)N * kBands * g.M1K1;
    const double dt = g.dt;
    auto minfo = [&](int t, int& m, int& k) {
        const int mode = mode0 + t;
        m = mode / g.nk;
        k = mode - m * g.nk - g.K;
    };
    // T divides the block size (k_pc): the modes of this thread in the element loops (tq) and in
    // the stencil loops (ts, part)
    const int tq = threadIdx.x % T, jstep = blockDim.x / T;
    const bool in = tq < nT;
    const int ts = threadIdx.x % (2 * T) >> 1, part = threadIdx.x & 1;
    const bool ins = ts < nT;
    int ms, ks;
    minfo(ts, ms, ks);
    const double mms = g.mp * ms, kks = (part ? 1 : -1) * (g.kz * ks);   // i k of the other part: kks times it

    // G': u*bar = ubar_new; phibar = -grad_h^T ubar_new
    for (int j = threadIdx.x / T; j < N; j += jstep) {
        const int idx = j * T + tq;
        double2 v0 = make_double2(0.0, 0.0), v1 = v0, v2 = v0;
        if (in) {
            const size_t e = (size_t)j * g.nmode + mode0 + tq;
            v0 = a.ubar_new[e];
            v1 = a.ubar_new[g.S + e];
            v2 = a.ubar_new[2 * g.S + e];
        }
        C1[idx] = v0;
        C2[idx] = v1;
        C3[idx] = v2;
    }
    __syncthreads();
    // (D1^T f)(c) on the real or imaginary part i of this thread: gather over the rows whose stencil
    // holds c, from the host-built table (row, weight) padded with zero weights
    auto dT = [&](const double* f, int c) {
        double o = 0.0;
        for (int e = 0; e < a.ntab; ++e)
            o = fma(__ldg(&a.tw[c * a.ntab + e]), f[__ldg(&a.trow[c * a.ntab + e]) * 2 * T], o);
        return o;
    };
    const int cs = threadIdx.x % (2 * T), sstep = blockDim.x / (2 * T);
    // grad_h^T g = D1^T(g_+ + g_-) - m m_p (g_+ - g_-)/r - i k k_z g_z, negated, into C0
    auto gradT = [&] {
        for (int j = threadIdx.x / (2 * T); j < N; j += sstep) {
            const int i = j * 2 * T + cs;
            double o = 0.0;
            if (ins) o = -(dT(D1 + cs, j) + dT(D2 + cs, j) - mms * __ldg(&a.ir[j]) * (D1[i] - D2[i]) - kks * D3[i ^ 1]);
            D0[i] = o;
        }
    };
    gradT();
    __syncthreads();
    // F': bbar = P^{-T} phibar, wall rows carry no dependence
    if (threadIdx.x < 2 * nT) {
        const int t = threadIdx.x >> 1, part = threadIdx.x & 1;
        int m, k;
        minfo(t, m, k);
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        smem_band_solve_T<kAdjChunkF, kAdjChunkB>(C0, T, t, part, N, a.fac + (size_t)kSetP * per_set + mk,
                                                  a.piv + (size_t)kSetP * N * g.M1K1 + mk, g.M1K1);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        C0[t] = make_double2(0.0, 0.0);
        C0[(N - 1) * T + t] = make_double2(0.0, 0.0);
    }
    __syncthreads();
    // E': u*bar += div_h^T bbar:  t = D1^T b + b/r;  +: t/2 + m m_p b/(2r), -: t/2 - .., z: -i k k_z b
    if (ins)
        for (int j = threadIdx.x / (2 * T); j < N; j += sstep) {
            const int i = j * 2 * T + cs;
            const double ir = __ldg(&a.ir[j]), b = D0[i], tt = dT(D0 + cs, j) + b * ir, mm = 0.5 * mms * ir;
            D1[i] += 0.5 * tt + mm * b;
            D2[i] += 0.5 * tt - mm * b;
            D3[i] -= kks * D0[i ^ 1];
        }
    __syncthreads();
    // D': rhsbar_c = H_c^{-T} u*bar_c; wall rows of rhs are constants
    if (threadIdx.x < 6 * nT) {
        const int c = threadIdx.x / (2 * nT), rem = threadIdx.x - c * 2 * nT;
        const int t = rem >> 1, part = rem & 1;
        int m, k;
        minfo(t, m, k);
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        const int set = kSetHp + c;
        smem_band_solve_T<kAdjChunkF, kAdjChunkB>(Cv[c], T, t, part, N, a.fac + (size_t)set * per_set + mk,
                                                  a.piv + (size_t)set * N * g.M1K1 + mk, g.M1K1);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < T; t += blockDim.x)
        for (int c = 0; c < 3; ++c) {
            Cv[c][t] = make_double2(0.0, 0.0);
            Cv[c][(N - 1) * T + t] = make_double2(0.0, 0.0);
        }
    __syncthreads();
    // C': ubar += (4/(2dt)) rhsbar, up_bar = -rhsbar/(2dt); p*bar = -grad_h^T rhsbar (C0)
    gradT();
    __syncthreads();
    // B': bpbar = P^{-T} p*bar.  Meanwhile the warps without a substitution write ubar and up_bar.
    const int helper0 = ((2 * nT + 31) / 32) * 32;
    if (threadIdx.x < 2 * nT) {
        const int t = threadIdx.x >> 1, part = threadIdx.x & 1;
        int m, k;
        minfo(t, m, k);
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        smem_band_solve_T<kAdjChunkF, kAdjChunkB>(C0, T, t, part, N, a.fac + (size_t)kSetP * per_set + mk,
                                                  a.piv + (size_t)kSetP * N * g.M1K1 + mk, g.M1K1);
    } else if (threadIdx.x >= helper0 && in) {   // helper0 < blockDim.x, and a multiple of T
        const double c2 = 2.0 / dt, ch = 1.0 / (2.0 * dt);
        for (int j = (threadIdx.x - helper0) / T; j < N; j += ((int)blockDim.x - helper0) / T) {
            const size_t e = (size_t)j * g.nmode + mode0 + tq;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const size_t ec = (size_t)c * g.S + e;
                const double2 rb = Cv[c][j * T + tq];
                double2 ub = a.ubar_cur ? a.ubar_cur[ec] : make_double2(0.0, 0.0);
                ub.x += c2 * rb.x;
                ub.y += c2 * rb.y;
                a.u_out[ec] = ub;
                a.up_out[ec] = make_double2(-rb.x * ch, -rb.y * ch);
            }
        }
    }
    __syncthreads();
    // A': interior rows b_p = div_h(-NN): NNbar = -rhsbar + div_h^T(-bpbar_interior);
    //     wall rows b_p = -NN_r + 2 Lap_r(u) - Lap_r(u_prev) (not the (0,0) row at r_o)
    if (ins)
        for (int j = threadIdx.x / (2 * T); j < N; j += sstep) {
            const int i = j * 2 * T + cs;
            const bool wall = j == 0 || j == N - 1;
            double d = 0.0;
            for (int e = 0; e < a.ntab; ++e) {
                const int row = __ldg(&a.trow[j * a.ntab + e]);
                if (row == 0 || row == N - 1) continue;
                d = fma(-__ldg(&a.tw[j * a.ntab + e]), D0[row * 2 * T + cs], d);
            }
            const double ir = __ldg(&a.ir[j]), b = D0[i], v = wall ? 0.0 : -b, o = wall ? 0.0 : D0[i ^ 1];
            const double tt = d + v * ir, mm = 0.5 * mms * ir;
            double p = 0.5 * tt + mm * v - D1[i], m = 0.5 * tt - mm * v - D2[i];
            if (wall && !(j == N - 1 && ms == 0 && ks == 0)) {
                p -= 0.5 * b;
                m -= 0.5 * b;
            }
            D1[i] = p;
            D2[i] = m;
            D3[i] = kks * o - D3[i];
        }
    __syncthreads();
    // wall Laplacian transposes: column c of the wall stencils receives, for wall row jw with
    // value w: 1/2 (D2[jw][c] + D1[jw][c]/r_jw) w (+ 1/2 diag_pm w at c = jw), times 2 into
    // ubar and -1 into up_bar.  One thread per (column, mode) of the two wall stencils.
    for (int idx = threadIdx.x; idx < 2 * kStencil * T; idx += blockDim.x) {
        const int side = idx / (kStencil * T);
        const int rem = idx - side * kStencil * T;
        const int q = rem / T, t = rem - (rem / T) * T;
        if (t >= nT) continue;
        int m, k;
        minfo(t, m, k);
        const int jw = side == 0 ? 0 : N - 1;
        if (jw == N - 1 && m == 0 && k == 0) continue;
        const int c = a.col0[jw] + q;
        const double ir = a.ir[jw], ir2 = ir * ir;
        const double wq = 0.5 * (a.w2[jw * kStencil + q] + ir * a.w1[jw * kStencil + q]);
        const double2 w = C0[jw * T + t];
        const double mm = g.mp * m, kk = g.kz * k;
        const size_t e = (size_t)c * g.nmode + mode0 + t;
        for (int cc = 0; cc < 2; ++cc) {
            double coef = wq;
            if (c == jw) {
                const double sgn = cc == 0 ? -1.0 : 1.0;
                coef += 0.5 * (-mm * mm * ir2 - kk * kk - ir2 + sgn * 2.0 * mm * ir2);
            }
            if (coef == 0.0) continue;
            const size_t ec = (size_t)cc * g.S + e;
            // rows of the two wall stencils may share a column only when N_r < 10; the
            // two sides then run in sequence below to keep the read-modify-write race free
            if (side == 1 && N < 2 * kStencil) continue;
            double2 ub = a.u_out[ec], pb = a.up_out[ec];
            ub.x += 2.0 * coef * w.x; ub.y += 2.0 * coef * w.y;
            pb.x -= coef * w.x; pb.y -= coef * w.y;
            a.u_out[ec] = ub;
            a.up_out[ec] = pb;
        }
    }
    __syncthreads();
    if (N < 2 * kStencil) {   // second wall for small N_r, after the first
        for (int idx = threadIdx.x; idx < kStencil * T; idx += blockDim.x) {
            const int q = idx / T, t = idx - (idx / T) * T;
            if (t >= nT) continue;
            int m, k;
            minfo(t, m, k);
            const int jw = N - 1;
            if (m == 0 && k == 0) continue;
            const int c = a.col0[jw] + q;
            const double ir = a.ir[jw], ir2 = ir * ir;
            const double wq = 0.5 * (a.w2[jw * kStencil + q] + ir * a.w1[jw * kStencil + q]);
            const double2 w = C0[jw * T + t];
            const double mm = g.mp * m, kk = g.kz * k;
            const size_t e = (size_t)c * g.nmode + mode0 + t;
            for (int cc = 0; cc < 2; ++cc) {
                double coef = wq;
                if (c == jw) {
                    const double sgn = cc == 0 ? -1.0 : 1.0;
                    coef += 0.5 * (-mm * mm * ir2 - kk * kk - ir2 + sgn * 2.0 * mm * ir2);
                }
                if (coef == 0.0) continue;
                const size_t ec = (size_t)cc * g.S + e;
                double2 ub = a.u_out[ec], pb = a.up_out[ec];
                ub.x += 2.0 * coef * w.x; ub.y += 2.0 * coef * w.y;
                pb.x -= coef * w.x; pb.y -= coef * w.y;
                a.u_out[ec] = ub;
                a.up_out[ec] = pb;
            }
        }
        __syncthreads();
    }
    // NN = 2N - N_prev:  Nbar = Nbar_cur + 2 NNbar,  Np_bar = -NNbar
    for (int idx = threadIdx.x; idx < 3 * items; idx += blockDim.x) {
        const int c = idx / items, rem = idx - c * items;
        const int j = rem / T, t = rem - (rem / T) * T;
        if (t >= nT) continue;
        const size_t ec = (size_t)c * g.S + (size_t)j * g.nmode + mode0 + t;
        const double2 nn = Cv[c][rem];
        double2 nb = a.Nbar_cur ? a.Nbar_cur[ec] : make_double2(0.0, 0.0);
        nb.x += 2.0 * nn.x;
        nb.y += 2.0 * nn.y;
        a.N_out[ec] = nb;
        a.Np_out[ec] = make_double2(-nn.x, -nn.y);
    }
}

// ---------------------------------------------------------------- transposed steps 2-5, per stage
// The same phases as k_pc_adj as one kernel per stage over all modes, for large N_r: each
// column lives in global memory, so every transposed substitution runs on its own thread
// (mode, real / imaginary part) with full warps, where k_pc_adj would hold few modes per
// block.  Scratch: US (3 fields), PH and PS (one each), the forward split path's buffers.
// A wall row of PH, US or PS holds no dependence after its solve and is read as zero.

struct AdjT {
    const double* ir;
    const int* trow;
    const double* tw;
    int ntab;
};

// sum_e D1[row_e][j] f(row_e) over the rows whose stencil holds column j; wall rows of f
// dropped when `walls` is false
__device__ __forceinline__ double2 growT(const double2* __restrict__ f, const AdjT& a, int j, int nmode,
                                         int mode, int N, bool walls) {
    double2 s = make_double2(0.0, 0.0);
    for (int e = 0; e < a.ntab; ++e) {
        const int row = __ldg(&a.trow[j * a.ntab + e]);
        if (!walls && (row == 0 || row == N - 1)) continue;
        const double w = __ldg(&a.tw[j * a.ntab + e]);
        const double2 v = f[(size_t)row * nmode + mode];
        s.x = fma(w, v.x, s.x);
        s.y = fma(w, v.y, s.y);
    }
    return s;
}

// grad_h^T of the vector field v at (j, mode), negated: -(D1^T(v_+ + v_-) - m m_p (v_+ - v_-)/r
// - i k k_z v_z); wall rows of v read as zero unless `walls`
__device__ __forceinline__ double2 neg_gradT(const double2* __restrict__ v, const AdjT& a, const Geo& g, int j,
                                             int mode, bool walls) {
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const double2 dp = growT(v, a, j, g.nmode, mode, g.N, walls);
    const double2 dm = growT(v + g.S, a, j, g.nmode, mode, g.N, walls);
    const bool wall = j == 0 || j == g.N - 1;
    const size_t e = (size_t)j * g.nmode + mode;
    const double2 z0 = make_double2(0.0, 0.0);
    const double2 gp = (walls || !wall) ? v[e] : z0, gm = (walls || !wall) ? v[g.S + e] : z0;
    const double2 gz = (walls || !wall) ? v[2 * g.S + e] : z0;
    const double mm = g.mp * m * a.ir[j], kk = g.kz * k;
    return make_double2(-(dp.x + dm.x - mm * (gp.x - gm.x) + kk * gz.y),
                        -(dp.y + dm.y - mm * (gp.y - gm.y) - kk * gz.x));
}

// G': PH = -grad_h^T ubar_new
__global__ void k_adjT_phi(const double2* __restrict__ ubn, double2* __restrict__ PH, AdjT a, Geo g) {
    const int mode = blockIdx.y * blockDim.x + threadIdx.x;   // x = radial row
    if (mode >= g.nmode) return;
    const int j = blockIdx.x;
    PH[(size_t)j * g.nmode + mode] = neg_gradT(ubn, a, g, j, mode, true);
}

// E': US = ubar_new + div_h^T PH (PH's wall rows zero)
__global__ void k_adjT_ustar(const double2* __restrict__ ubn, const double2* __restrict__ PH,
                             double2* __restrict__ US, AdjT a, Geo g) {
    const int mode = blockIdx.y * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int j = blockIdx.x;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const size_t e = (size_t)j * g.nmode + mode;
    const double ir = a.ir[j];
    const double2 d = growT(PH, a, j, g.nmode, mode, g.N, false);
    const double2 b = (j == 0 || j == g.N - 1) ? make_double2(0.0, 0.0) : PH[e];
    const double2 tt = make_double2(d.x + b.x * ir, d.y + b.y * ir);
    const double mm = 0.5 * g.mp * m * ir, kk = g.kz * k;
    double2 v;
    v = ubn[e]; v.x += 0.5 * tt.x + mm * b.x; v.y += 0.5 * tt.y + mm * b.y; US[e] = v;
    v = ubn[g.S + e]; v.x += 0.5 * tt.x - mm * b.x; v.y += 0.5 * tt.y - mm * b.y; US[g.S + e] = v;
    v = ubn[2 * g.S + e]; v.x += kk * b.y; v.y -= kk * b.x; US[2 * g.S + e] = v;
}

// C': with rb = US (wall rows zero): u_out = ubar_cur + (2/dt) rb, up_out = -rb/(2 dt),
// PS = -grad_h^T rb.  u_out may alias ubar_new (no longer read) and up_out ubar_cur (read
// first, by the same thread).
__global__ void k_adjT_rhs(const double2* __restrict__ US, const double2* ubc, double2* u_out, double2* up_out,
                           double2* __restrict__ PS, AdjT a, Geo g) {
    const int mode = blockIdx.y * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int j = blockIdx.x;
    const size_t e = (size_t)j * g.nmode + mode;
    const bool wall = j == 0 || j == g.N - 1;
    const double dt = g.dt;
    for (int c = 0; c < 3; ++c) {
        const size_t ec = (size_t)c * g.S + e;
        const double2 rb = wall ? make_double2(0.0, 0.0) : US[ec];
        double2 ub = ubc ? ubc[ec] : make_double2(0.0, 0.0);
        ub.x += 2.0 / dt * rb.x;
        ub.y += 2.0 / dt * rb.y;
        u_out[ec] = ub;
        up_out[ec] = make_double2(-rb.x / (2.0 * dt), -rb.y / (2.0 * dt));
    }
    PS[e] = neg_gradT(US, a, g, j, mode, false);
}

// A': NNbar = -rb + div_h^T(-bpbar on interior rows) and the wall-row terms of Eq. ppBC;
// N_out = Nbar_cur + 2 NNbar, Np_out = -NNbar (Np_out may alias Nbar_cur: same thread)
__global__ void k_adjT_nn(const double2* __restrict__ US, const double2* __restrict__ PS, const double2* Nbc,
                          double2* N_out, double2* Np_out, AdjT a, Geo g) {
    const int mode = blockIdx.y * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int j = blockIdx.x;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const size_t e = (size_t)j * g.nmode + mode;
    const int N = g.N;
    const bool wall = j == 0 || j == N - 1;
    const double ir = a.ir[j];
    const double2 dd = growT(PS, a, j, g.nmode, mode, N, false);
    const double2 d = make_double2(-dd.x, -dd.y);
    const double2 bp = PS[e];
    const double2 v = wall ? make_double2(0.0, 0.0) : make_double2(-bp.x, -bp.y);
    const double2 tt = make_double2(d.x + v.x * ir, d.y + v.y * ir);
    const double mm = 0.5 * g.mp * m * ir, kk = g.kz * k;
    const bool wterm = j == 0 || (j == N - 1 && !(m == 0 && k == 0));
    double2 q[3];
    for (int c = 0; c < 3; ++c) {
        const double2 rb = wall ? make_double2(0.0, 0.0) : US[(size_t)c * g.S + e];
        q[c] = make_double2(-rb.x, -rb.y);
    }
    q[0].x += 0.5 * tt.x + mm * v.x; q[0].y += 0.5 * tt.y + mm * v.y;
    q[1].x += 0.5 * tt.x - mm * v.x; q[1].y += 0.5 * tt.y - mm * v.y;
    if (wterm) {
        q[0].x -= 0.5 * bp.x; q[0].y -= 0.5 * bp.y;
        q[1].x -= 0.5 * bp.x; q[1].y -= 0.5 * bp.y;
    }
    q[2].x += kk * v.y; q[2].y -= kk * v.x;
    for (int c = 0; c < 3; ++c) {
        const size_t ec = (size_t)c * g.S + e;
        double2 nb = Nbc ? Nbc[ec] : make_double2(0.0, 0.0);
        nb.x += 2.0 * q[c].x;
        nb.y += 2.0 * q[c].y;
        N_out[ec] = nb;
        Np_out[ec] = make_double2(-q[c].x, -q[c].y);
    }
}

// Wall Laplacian transposes of Eq. ppBC's wall rows (side 0: r_i, 1: r_o; `sides` of them
// from `side0`): column c of the wall stencil receives 1/2 (D2 + D1/r)[jw][c] bpbar(jw)
// (+ the diagonal terms at c = jw), times 2 into u_out and -1 into up_out, for the + and -
// components.  One thread per (side, stencil column, mode); the two sides touch the same
// columns only when N_r < 18, and then run as two launches.
__global__ void k_adjT_wall(const double2* __restrict__ PS, double2* u_out, double2* up_out,
                            const double* __restrict__ w1, const double* __restrict__ w2,
                            const int* __restrict__ col0, AdjT a, Geo g, int side0) {
    const int mode = blockIdx.x * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int q = blockIdx.y;
    const int side = side0 + blockIdx.z;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const int jw = side == 0 ? 0 : g.N - 1;
    if (jw == g.N - 1 && m == 0 && k == 0) return;
    const int c = col0[jw] + q;
    const double ir = a.ir[jw], ir2 = ir * ir;
    const double wq = 0.5 * (w2[jw * kStencil + q] + ir * w1[jw * kStencil + q]);
    const double2 w = PS[(size_t)jw * g.nmode + mode];
    const double mm = g.mp * m, kk = g.kz * k;
    const size_t e = (size_t)c * g.nmode + mode;
    for (int cc = 0; cc < 2; ++cc) {
        double coef = wq;
        if (c == jw) {
            const double sgn = cc == 0 ? -1.0 : 1.0;
            coef += 0.5 * (-mm * mm * ir2 - kk * kk - ir2 + sgn * 2.0 * mm * ir2);
        }
        if (coef == 0.0) continue;
        const size_t ec = (size_t)cc * g.S + e;
        double2 ub = u_out[ec], pb = up_out[ec];
        ub.x += 2.0 * coef * w.x; ub.y += 2.0 * coef * w.y;
        pb.x -= coef * w.x; pb.y -= coef * w.y;
        u_out[ec] = ub;
        up_out[ec] = pb;
    }
}

// x <- A^{-T} x for every mode of nfields consecutive fields (sets set0, set0 + 1, ...):
// thread (field, mode, part) runs the transposed substitution down its global column
__global__ void k_band_solve_gT(double2* __restrict__ x, const double* __restrict__ fac,
                                const uint8_t* __restrict__ piv, int set0, Geo g) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;   // (mode, part); y = field
    if (t >= 2 * g.nmode) return;
    const int part = t & 1;
    const int mode = t >> 1;
    const int fld = blockIdx.y;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
    const size_t per_set = (size_t)g.N * kBands * g.M1K1;
    const int set = set0 + fld;
    smem_band_solve_T<kAdjChunkF, kAdjChunkB>(x + (size_t)fld * g.S, g.nmode, mode, part, g.N, fac + (size_t)set * per_set + mk,
                      piv + (size_t)set * g.N * g.M1K1 + mk, g.M1K1);
}

// ---------------------------------------------------------------- transposed nonlinear term
// ubar(c, j, mode) += sum over the staged rows i = r0 .. r0 + nh - 1 of D1[i][j] Rhat(c, i, mode)
// for the columns j = j0 .. j0 + gridDim.x - 1 (the columns those rows' stencils reach)
__global__ void k_drT(double2* __restrict__ ub, const double2* __restrict__ Rh, const int* __restrict__ trow,
                      const double* __restrict__ tw, int ntab, Geo g, int r0, int nh, int j0) {
    // grid: x = radial column (fastest: the gathered rows stay in cache), y over modes, z = component
    const int mode = blockIdx.y * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int j = j0 + blockIdx.x, c = blockIdx.z;
    const size_t e = (size_t)c * g.S + (size_t)j * g.nmode + mode;
    const size_t Sh = (size_t)nh * g.nmode;
    double2 s = ub[e];
    for (int q = 0; q < ntab; ++q) {
        const int i = __ldg(&trow[j * ntab + q]) - r0;
        if (i < 0 || i >= nh) continue;
        const double w = __ldg(&tw[j * ntab + q]);
        const double2 v = Rh[(size_t)c * Sh + (size_t)i * g.nmode + mode];
        s.x = fma(w, v.x, s.x);
        s.y = fma(w, v.y, s.y);
    }
    ub[e] = s;
}

tc_status launch_adjoint_advance(tc_plan* p, const double2* ubar_new, const double2* ubar_cur,
                                 const double2* Nbar_cur, double2* u_out, double2* up_out,
                                 double2* N_out, double2* Np_out, char* ws, cudaStream_t s) {
    Geo g = geo(p);
    if (p->pc_split) {
        // per-stage transposed steps 2-5 (the forward split path's scratch)
        double2* PS = reinterpret_cast<double2*>(ws + p->ws.pstar);
        double2* US = reinterpret_cast<double2*>(ws + p->ws.ustar);
        double2* PH = reinterpret_cast<double2*>(ws + p->ws.phi);
        AdjT a{p->d_ir, p->d_d1t_row, p->d_d1t_w, p->d1t_n};
        const dim3 g1(g.N, ablocks(g.nmode, 128));
        auto sgrid = [&](int nf) { return dim3(ablocks((size_t)2 * g.nmode, 128), nf); };
        const int slot = prof_begin(p, kKPCAdj, s);
        k_adjT_phi<<<g1, 128, 0, s>>>(ubar_new, PH, a, g);
        k_band_solve_gT<<<sgrid(1), 128, 0, s>>>(PH, p->d_fac, p->d_piv, kSetP, g);
        k_adjT_ustar<<<g1, 128, 0, s>>>(ubar_new, PH, US, a, g);
        k_band_solve_gT<<<sgrid(3), 128, 0, s>>>(US, p->d_fac, p->d_piv, kSetHp, g);
        k_adjT_rhs<<<g1, 128, 0, s>>>(US, ubar_cur, u_out, up_out, PS, a, g);
        k_band_solve_gT<<<sgrid(1), 128, 0, s>>>(PS, p->d_fac, p->d_piv, kSetP, g);
        k_adjT_nn<<<g1, 128, 0, s>>>(US, PS, Nbar_cur, N_out, Np_out, a, g);
        if (g.N >= 2 * kStencil) {
            k_adjT_wall<<<dim3(ablocks(g.nmode, 128), kStencil, 2), 128, 0, s>>>(PS, u_out, up_out, p->d_w1, p->d_w2,
                                                                                p->d_col0, a, g, 0);
        } else {
            for (int side = 0; side < 2; ++side)
                k_adjT_wall<<<dim3(ablocks(g.nmode, 128), kStencil, 1), 128, 0, s>>>(PS, u_out, up_out, p->d_w1,
                                                                                    p->d_w2, p->d_col0, a, g, side);
        }
        prof_end(p, slot, s);
        TC_LAUNCHED(p, "k_adjT");
        return TC_OK;
    }
    const int T = pc_modes(p, g.nmode);
    PCAdjArgs a;
    a.ubar_new = ubar_new; a.ubar_cur = ubar_cur; a.Nbar_cur = Nbar_cur;
    a.u_out = u_out; a.up_out = up_out; a.N_out = N_out; a.Np_out = Np_out;
    a.ir = p->d_ir; a.w1 = p->d_w1; a.w2 = p->d_w2; a.col0 = p->d_col0;
    a.trow = p->d_d1t_row; a.tw = p->d_d1t_w; a.ntab = p->d1t_n;
    a.fac = p->d_fac; a.piv = p->d_piv;
    const size_t sm = (size_t)4 * p->N_r * T * sizeof(double2);
    const int slot = prof_begin(p, kKPCAdj, s);
    auto run = [&](auto kern, int nth) -> tc_status {
        TC_CUDA(p, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        kern<<<ablocks(g.nmode, T), nth, sm, s>>>(a, g, T);
        return TC_OK;
    };
    TC_TRY_STATUS(T <= 8 ? run(k_pc_adj<128>, 128) : run(k_pc_adj<256>, 256));
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_pc_adj");
    return TC_OK;
}

// ubar += N'(u)^T Nbar, slab by slab of p->stage_rows radial rows: the transposed transforms of
// a row read only that row's staging, and the transposed radial stencil of a slab's Rhat rows
// is added before the next slab overwrites them
tc_status launch_nonlinear_adjoint(tc_plan* p, const double2* u, const double2* Nbar, double2* ubar,
                                   char* ws, cudaStream_t s) {
    Geo g = geo(p);
    double2* Rh = reinterpret_cast<double2*>(ws + p->ws.Rhat);
    for (int r0 = 0; r0 < p->N_r; r0 += p->stage_rows) {
        const int nh = p->N_r - r0 < p->stage_rows ? p->N_r - r0 : p->stage_rows;
        TC_TRY_STATUS(launch_adjoint_rows_fx(p, u, Nbar, ubar, Rh, ws, s, r0, nh));
        // columns reached by the stencils of rows r0 .. r0 + nh - 1
        int jlo = p->N_r, jhi = -1;
        for (int i = r0; i < r0 + nh; ++i) {
            jlo = p->col0[i] < jlo ? p->col0[i] : jlo;
            jhi = p->col0[i] + kStencil - 1 > jhi ? p->col0[i] + kStencil - 1 : jhi;
        }
        if (jlo < 0) jlo = 0;
        if (jhi > p->N_r - 1) jhi = p->N_r - 1;
        const int slot = prof_begin(p, kKDrT, s);
        k_drT<<<dim3(jhi - jlo + 1, ablocks(g.nmode, 128), 3), 128, 0, s>>>(ubar, Rh, p->d_d1t_row, p->d_d1t_w,
                                                                            p->d1t_n, g, r0, nh, jlo);
        prof_end(p, slot, s);
        TC_LAUNCHED(p, "k_drT");
    }
    return TC_OK;
}

// gradient of J = 1/2 sum_j w_j r_j sum c_m (|u'_+|^2/2 + |u'_-|^2/2 + |u'_z|^2), u' = u - Couette
__global__ void k_energy_grad(const double2* __restrict__ u, double2* __restrict__ gr,
                              const double* __restrict__ rn, double C1, double C2, Geo g) {
    const int mode = blockIdx.x * blockDim.x + threadIdx.x;
    if (mode >= g.nmode) return;
    const int j = blockIdx.y, c = blockIdx.z;
    const size_t e = (size_t)c * g.S + (size_t)j * g.nmode + mode;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const double r = rn[j];
    double wr = 0.0;
    if (j > 0) wr += 0.5 * (r - rn[j - 1]);
    if (j < g.N - 1) wr += 0.5 * (rn[j + 1] - r);
    double2 d = u[e];
    if (m == 0 && k == 0 && c < 2) d.y -= (c == 0 ? 1.0 : -1.0) * (C1 * r + C2 / r);
    const double f = wr * r * (m == 0 ? 1.0 : 2.0) * (c < 2 ? 0.5 : 1.0);
    gr[e] = make_double2(f * d.x, f * d.y);
}

tc_status launch_energy_gradient(tc_plan* p, const double2* u, double2* gr, cudaStream_t s) {
    Geo g = geo(p);
    const double eta = p->eta;
    const double C1 = (p->Re_o - eta * p->Re_i) / (1.0 + eta);
    const double C2 = eta * (p->Re_i - eta * p->Re_o) / ((1.0 - eta) * (1.0 - eta * eta));
    k_energy_grad<<<dim3(ablocks(g.nmode, 128), g.N, 3), 128, 0, s>>>(u, gr, p->d_r, C1, C2, g);
    TC_LAUNCHED(p, "k_energy_grad");
    return TC_OK;
}

}  // namespace tc

using namespace tc;

namespace {

tc_status adj_ready(tc_plan* p, void* ws) {
    if (!p) return TC_ERR_ARG;
    if (p->host_only) return TC_ERR_STATE;
    if (!p->adjoint) {
        snprintf(p->err, sizeof(p->err), "plan created with no_adjoint: its workspace has no adjoint regions");
        return TC_ERR_STATE;
    }
    int dev = -1;
    TC_CUDA(p, cudaGetDevice(&dev));
    if (dev != p->device) return TC_ERR_STATE;
    if (!ws || reinterpret_cast<uintptr_t>(ws) % 256 != 0) return TC_ERR_ARG;
    return check_device_ptr(p, ws, "ws", p->ws.total);
}

#define TC_TRY2(x)                   \
    do {                             \
        tc_status s_ = (x);          \
        if (s_ != TC_OK) return s_;  \
    } while (0)

}  // namespace

extern "C" {

tc_status tc_adjoint_step(tc_plan* plan, const tc_state* fwd, tc_state_bar* bar, void* ws, void* stream) {
    TC_TRY2(adj_ready(plan, ws));
    if (!fwd || !bar) return TC_ERR_ARG;
    if (!fwd->started) {
        snprintf(plan->err, sizeof(plan->err), "tc_adjoint_step needs a started forward state (use tc_adjoint_start for the cold start)");
        return TC_ERR_STATE;
    }
    const size_t vb = 3 * plan->S * sizeof(double2);
    TC_TRY2(check_device_ptr(plan, fwd->u, "fwd->u", vb));
    TC_TRY2(check_device_ptr(plan, bar->u, "bar->u", vb));
    TC_TRY2(check_device_ptr(plan, bar->u_prev, "bar->u_prev", vb));
    TC_TRY2(check_device_ptr(plan, bar->N_prev, "bar->N_prev", vb));
    if (bar->u == bar->u_prev || bar->u == bar->N_prev || bar->u_prev == bar->N_prev) return TC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    double2* ub = static_cast<double2*>(bar->u);
    double2* upb = static_cast<double2*>(bar->u_prev);
    double2* Npb = static_cast<double2*>(bar->N_prev);
    double2* Nb = reinterpret_cast<double2*>(w + plan->ws.Nbar);
    TC_TRY2(launch_adjoint_advance(plan, ub, upb, Npb, ub, upb, Nb, Npb, w, s));
    return launch_nonlinear_adjoint(plan, static_cast<const double2*>(fwd->u), Nb, ub, w, s);
}

tc_status tc_adjoint_start(tc_plan* plan, const void* u0, const tc_state_bar* bar, void* u0_bar,
                           void* ws, void* stream) {
    TC_TRY2(adj_ready(plan, ws));
    if (!bar) return TC_ERR_ARG;
    const size_t vb = 3 * plan->S * sizeof(double2);
    TC_TRY2(check_device_ptr(plan, u0, "u0", vb));
    TC_TRY2(check_device_ptr(plan, u0_bar, "u0_bar", vb));
    TC_TRY2(check_device_ptr(plan, bar->u, "bar->u", vb));
    TC_TRY2(check_device_ptr(plan, bar->u_prev, "bar->u_prev", vb));
    TC_TRY2(check_device_ptr(plan, bar->N_prev, "bar->N_prev", vb));
    if (u0_bar == u0 || u0_bar == bar->u_prev || u0_bar == bar->N_prev) return TC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* w = static_cast<char*>(ws);
    const size_t n3 = 3 * plan->S;
    const double2* u = static_cast<const double2*>(u0);
    double2* out = static_cast<double2*>(u0_bar);
    double2* Nc = reinterpret_cast<double2*>(w + plan->ws.Ncur);
    double2* uE = reinterpret_cast<double2*>(w + plan->ws.uE);
    double2* Nb = reinterpret_cast<double2*>(w + plan->ws.Nbar);
    double2* um1 = reinterpret_cast<double2*>(w + plan->ws.abar);
    double2* m1b = um1 + n3;
    double2* uEb = m1b + n3;
    // forward recomputation of the start-up: N0 = N(u0), u_E, u^{-1}
    TC_TRY2(launch_nonlinear(plan, u, Nc, w, s));
    TC_TRY2(launch_advance(plan, u, const_cast<double2*>(u), Nc, Nc, nullptr, uE, w, false, s));
    TC_TRY2(launch_axpby(plan, um1, u, 2.5, uE, -1.5, n3, s));
    // m1_bar = ubar_prev + N'(u^{-1})^T Nbar_prev
    TC_CUDA(plan, cudaMemcpyAsync(m1b, bar->u_prev, n3 * sizeof(double2), cudaMemcpyDeviceToDevice, s));
    TC_TRY2(launch_nonlinear_adjoint(plan, um1, static_cast<const double2*>(bar->N_prev), m1b, w, s));
    // u_E bar = -1.5 m1_bar; adjoint of the Euler step (u, u_prev, N, N_prev all = u0 / N0)
    TC_TRY2(launch_axpby(plan, uEb, m1b, -1.5, m1b, 0.0, n3, s));
    double2* a_u = out;   // adjoint of its u input
    double2* a_up = uE;   // adjoint of its u_prev input
    double2* a_N = Nb;    // adjoint of its N input
    double2* a_Np = Nc;   // adjoint of its N_prev input
    TC_TRY2(launch_adjoint_advance(plan, uEb, nullptr, nullptr, a_u, a_up, a_N, a_Np, w, s));
    // u0_bar = ubar + 2.5 m1_bar + a_u + a_up + N'(u0)^T (a_N + a_Np)
    TC_TRY2(launch_axpby(plan, out, out, 1.0, a_up, 1.0, n3, s));
    TC_TRY2(launch_axpby(plan, out, out, 1.0, m1b, 2.5, n3, s));
    TC_TRY2(launch_axpby(plan, out, out, 1.0, static_cast<const double2*>(bar->u), 1.0, n3, s));
    TC_TRY2(launch_axpby(plan, a_N, a_N, 1.0, a_Np, 1.0, n3, s));
    return launch_nonlinear_adjoint(plan, u, a_N, out, w, s);
}

tc_status tc_energy_gradient(tc_plan* plan, const void* u, void* g, void* stream) {
    if (!plan) return TC_ERR_ARG;
    if (plan->host_only) return TC_ERR_STATE;
    TC_TRY2(check_device_ptr(plan, u, "u", 3 * plan->S * sizeof(double2)));
    TC_TRY2(check_device_ptr(plan, g, "g", 3 * plan->S * sizeof(double2)));
    return launch_energy_gradient(plan, static_cast<const double2*>(u), static_cast<double2*>(g),
                                  static_cast<cudaStream_t>(stream));
}

}  // extern "C"
