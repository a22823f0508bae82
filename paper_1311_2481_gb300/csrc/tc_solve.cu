// Linear part of the AB2BD2 step (Sec. 3.2 steps 2-5): right-hand sides, the five banded
// solves per Fourier mode with precomputed LU factors (forward / backward substitution,
// O(N_r) per system), and the update.  Two paths:
//
//   k_pc     (N_r up to 192) one block per T consecutive modes, all five solves and their
//            right-hand sides in shared memory.  Each system is solved in two partitions
//            (rows [0, N_r/2) and [N_r/2, N_r), each with its own pivoted LU factors, on
//            separate threads), coupled through an 8 x 8 reduced system and a fix-up; one
//            real part per thread, consecutive modes on consecutive threads.
//   split    (larger N_r) one kernel per stage; the solves walk one column per thread in
//            global memory with the full-system factors.
//
// Threads of a warp own consecutive k, so every access to a field [r][m][k] or to the
// factors [j][band][m][|k|] is coalesced.
#include <algorithm>

#include "tc_internal.cuh"
#include "tc_solve_core.cuh"

namespace tc {

struct PCArgs {
    const double2* u;   // u^i
    const double2* up;  // u^{i-1}
    const double2* Nc;  // N^i
    const double2* Np;  // N^{i-1}
    double2* u_out;     // commit: u (in place); otherwise the result u^{i+1} only
    double2* up_out;    // commit: u_prev <- u^i
    double2* Np_out;    // commit: N_prev <- N^i
    double2* p;         // commit: p <- p^{i+1}
    const double* ir;   // 1 / r_j
    const double* w1;
    const double* w2;
    const int* col0;
    const int2* fw;       // fixed-point stencil weights, their exponents and near ones (fx::Tile)
    const int2* few;
    const double* fac;
    const uint8_t* piv;
    const double* fac2;   // two-partition form (g.sh > 0): factors of the diagonal blocks,
    const uint8_t* piv2;  // spikes [set][j][q][m][ka] and inverse reduced matrices
    const double* spk;    // [set][8 i + l][m][ka]
    const double* rinv;
    int* nonfinite;       // set to 1 when a NaN/Inf is written into the state
    double Re_i, Re_o;
    int commit;
    int far;              // rows left to FP64 sums by the fixed-point stencils (fx::Tile): limit
    int sum;              // the block has a fifth column, for C1 + C2
};

constexpr int kChunkF = 4, kChunkB = 2;   // rows of factors per register chunk (3, 2: 2 % and 4, 3: 9 % slower k_pc)

// CH: chunks; the row by row ring of kPCDepth rows reaches further ahead, which counts where a launch
// has few warps and nothing else covers a load (N_r = 160, M = 8, K = 16: k_pc 223 against 239 us).
template <bool CH, bool LOOP>
__device__ __forceinline__ void band_solve(double2* col, int off, int T, int N, const double* __restrict__ F,
                                           const uint8_t* __restrict__ P, int M1K1) {
    if (CH) smem_band_solve_c<kChunkF, kChunkB, LOOP>(col, T, off, N, F, P, M1K1);
    else smem_band_solve<kPCDepth>(col, T, off, N, F, P, M1K1);
}

// Thread lt of the threads of one system (its column X in shared memory).  With two partitions
// (g.sh > 0) 4 nT threads, each with one half of it for one (mode, part): threads [0, 2nT) rows [0, sh),
// threads [2nT, 4nT) rows [sh, N), with the pivoted LU factors of the diagonal block; the column then
// holds g = (A1^{-1} b1, A2^{-1} b2).  Otherwise 2 nT threads with the factors of the whole system.
template <bool CH, bool LOOP>
__device__ __forceinline__ void system_solve(const PCArgs& a, const Geo& g, double2* X, int set, int T, int nT, int mode0, int lt) {
    const bool sp = g.sh > 0;
    const int half = lt >= 2 * nT ? 1 : 0;
    const int r = lt - half * 2 * nT;
    const int t = r >> 1, part = r & 1;
    const int mode = mode0 + t, m = mode / g.nk, k = mode - m * g.nk - g.K;
    const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
    const size_t per_set = (size_t)g.N * kBands * g.M1K1;
    const int r0 = half ? g.sh : 0, n = half ? g.N - g.sh : sp ? g.sh : g.N;
    band_solve<CH, LOOP>(X + (size_t)r0 * T, 2 * t + part, T, n,
                   (sp ? a.fac2 : a.fac) + (size_t)set * per_set + (size_t)r0 * kBands * g.M1K1 + mk,
                   (sp ? a.piv2 : a.piv) + ((size_t)set * g.N + r0) * g.M1K1 + mk, g.M1K1);
}

// Couple the halves of nsys systems (columns X0 + s N T, factor sets set0 + s), block-wide:
// the interface unknowns x[sh-4 .. sh+3] = R^{-1} g[sh-4 .. sh+3] per (mode, part) into Xr,
// then x = g - V x[sh .. sh+3] on rows < sh and x = g - W x[sh-4 .. sh-1] on rows >= sh.
// Starts after a barrier that follows the half solves; ends with one.
__device__ __forceinline__ void spike_combine(const PCArgs& a, const Geo& g, double2* X0, int nsys, int set0,
                                              int T, int nT, int mode0, double* Xr) {
    const int N = g.N, h = g.sh, items = N * T, st = 2 * T;
    for (int task = threadIdx.x; task < nsys * nT * 16; task += blockDim.x) {
        const int s = task / (nT * 16), rem = task - s * nT * 16;
        const int t = rem >> 4, part = (rem >> 3) & 1, i = rem & 7;
        const int mode = mode0 + t, m = mode / g.nk, k = mode - m * g.nk - g.K;
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        const double* x = reinterpret_cast<const double*>(X0 + (size_t)s * items) + 2 * t + part;
        const double* R = a.rinv + ((size_t)(set0 + s) * 64 + 8 * i) * g.M1K1 + mk;
        double acc = 0.0;
#pragma unroll
        for (int l = 0; l < 8; ++l) acc = fma(__ldg(&R[(size_t)l * g.M1K1]), x[(size_t)(h - 4 + l) * st], acc);
        Xr[(s * T + t) * 16 + part * 8 + i] = acc;
    }
    __syncthreads();
    // fix-up: T divides the block size, so a thread's elements all belong to mode t = tid % T;
    // rows step by blockDim / T, four in flight per iteration
    const int t = threadIdx.x % T;
    if (t < nT) {
        const int mode = mode0 + t, m = mode / g.nk, k = mode - m * g.nk - g.K;
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        const int jstep = blockDim.x / T;
        for (int s = 0; s < nsys; ++s) {
            const double* Vs = a.spk + (size_t)(set0 + s) * N * 4 * g.M1K1 + mk;
            const double* xs = Xr + (s * T + t) * 16;
            double2* Xs = X0 + (size_t)s * items + t;
#pragma unroll 4
            for (int j = threadIdx.x / T; j < N; j += jstep) {
                const double* V = Vs + (size_t)j * 4 * g.M1K1;
                const double* xr = xs + (j < h ? 4 : 0);
                double2 v = Xs[(size_t)j * T];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double w = __ldg(&V[(size_t)q * g.M1K1]);
                    v.x = fma(-w, xr[q], v.x);
                    v.y = fma(-w, xr[8 + q], v.y);
                }
                Xs[(size_t)j * T] = v;
            }
        }
    }
    __syncthreads();
}

// L_pm v (c = 0, 1 for +, -) at row j of component c of u: one half of lap_r
__device__ __forceinline__ double2 lap_pm(const double2* __restrict__ u, const PCArgs& a, int c, int j, int mode, double mm,
                                          double kk, const Geo& g) {
    const double2* f = u + (size_t)c * g.S;
    const double ir = a.ir[j], ir2 = ir * ir;
    double2 d1 = make_double2(0.0, 0.0), d2 = d1;
    const int c0 = a.col0[j];
    stencil_taps<true>(c0, [&](int t) {
        const double2 x = f[(size_t)(c0 + t) * g.nmode + mode];
        const double p = __ldg(&a.w1[j * kStencil + t]), q = __ldg(&a.w2[j * kStencil + t]);
        d1.x += p * x.x;
        d1.y += p * x.y;
        d2.x += q * x.x;
        d2.y += q * x.y;
    });
    const double2 v = f[(size_t)j * g.nmode + mode];
    const double diag = -mm * mm * ir2 - kk * kk - ir2 + (c == 0 ? -2.0 : 2.0) * mm * ir2;
    return make_double2(d2.x + ir * d1.x + diag * v.x, d2.y + ir * d1.y + diag * v.y);
}

// Steps 2-5 of Sec. 3.2 for the T modes of this block: pressure prediction (Eq. pressure
// with the Neumann rows of Eq. ppBC), velocity prediction (Eq. vel), correction potential
// (Eq. correction) and update (Eq. update).
// The stages run as iterations of a loop around one copy of the substitution, of its coupling and of
// the work beside it.  Once a launch takes several waves its blocks are at different stages, and
// with a copy per stage they waited for instructions (1.6 warps per issue, 0.7 in the loop's smaller
// code): N_r = 64, M = 64, K = 128, fixed-point stencils: 969 -> 908 us; one wave, N_r = 64, M = 32,
// K = 64: 224 -> 221.
template <int NTH, bool FX>
__global__ void __launch_bounds__(NTH, 512 / NTH) k_pc(PCArgs a, Geo g, int T) {
    extern __shared__ double2 sm[];
    const int N = g.N;
    const int items = N * T;
    double2* C0 = sm;
    double2* C1 = sm + items;
    double2* C2 = C1 + items;
    double2* C3 = C2 + items;
    const int mode0 = g.mlo + blockIdx.x * T;
    const int nT = min(T, g.mhi - mode0);
    const double c1 = g.c1;   // 1 / (2 dt)
    // T divides the block size, so every element a thread visits in the element loops below
    // belongs to the same mode t = threadIdx.x % T: its row index steps by blockDim / T, and
    // m, k and the FP64 factors m m_p, k k_z are computed once (an int -> double conversion
    // takes the FP64 pipe like an arithmetic instruction)
    const int tq = threadIdx.x % T;
    const int jstep = blockDim.x / T;
    const int modeq = mode0 + tq;
    const int mq = modeq / g.nk;
    const int kq = modeq - mq * g.nk - g.K;
    const double mmq = g.mp * mq, kkq = g.kz * kq;

    const bool in = tq < nT;
    double2* Lw = C3 + items;   // scratch of the spikes, free until then: L_pm u at the walls
    double2* C4 = Lw + 24 * T;   // a.sum: C1 + C2

    // A1: (2N - N_prev)_+, _-, _z into C1, C2, C3; the halves of the wall Laplacians of u and
    // u_prev, one (field, component, wall, mode) per thread
#pragma unroll 2
    for (int j = threadIdx.x / T; j < N; j += jstep) {
        const int idx = j * T + tq;
        double2 n[3] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
        if (in) {
            const size_t e = (size_t)j * g.nmode + modeq;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 n1 = __ldg(&a.Nc[c * g.S + e]), n0 = __ldg(&a.Np[c * g.S + e]);
                n[c] = make_double2(2.0 * n1.x - n0.x, 2.0 * n1.y - n0.y);
            }
        }
        C1[idx] = n[0];
        C2[idx] = n[1];
        C3[idx] = n[2];
        if (!FX && a.sum) C4[idx] = make_double2(n[0].x + n[1].x, n[0].y + n[1].y);
    }
    for (int i = threadIdx.x / T; i < 8; i += jstep)
        if (in) Lw[i * T + tq] = lap_pm(i & 4 ? a.up : a.u, a, i & 1, i & 2 ? N - 1 : 0, modeq, mmq, kkq, g);
    __syncthreads();
    // the columns as doubles; the mode and part of this thread in the stencil loops
    double *D0 = reinterpret_cast<double*>(C0), *D1 = D0 + 2 * items, *D2 = D1 + 2 * items, *D3 = D2 + 2 * items;
    const int ts = threadIdx.x % (2 * T) >> 1, part = threadIdx.x & 1, modes = mode0 + ts, ms = modes / g.nk;
    const int ks = modes - ms * g.nk - g.K;
    const bool ins = ts < nT;
    const double mms = g.mp * ms, kks = (part ? 1 : -1) * (g.kz * ks);   // i k of the other part: kks times it
    const bool sp = g.sh > 0;
    double* Xr = reinterpret_cast<double*>(C3 + items);
    const double c3 = 3.0 * c1;   // 3 / (2 dt)
    double* pw = a.commit && ins ? reinterpret_cast<double*>(a.p) + 2 * (size_t)modes + part : nullptr;
    bool bad = false;
    int stage = 0;
    const int far = modes == g.K ? fx::kFar : a.far;   // the mean mode (0, 0) rounds as in FP64
    auto ir = [&](int j) { return __ldg(&a.ir[j]); };
    auto p0 = [&](int j) { return pw ? pw[2 * (size_t)j * g.nmode] : 0.0; };
    auto slow0 = [&](int j, int c, auto guard) {   // FP64 stencil at row j of C0
        const int c0 = __ldg(&a.col0[j]);
        double o = 0.0;
        stencil_taps<decltype(guard)::value>(c0, [&](int q) { o = fma(__ldg(&a.w1[j * kStencil + q]), D0[c + (c0 + q) * 2 * T], o); });
        return o;
    };
    auto slow12 = [&](int j, int c, auto guard) {   // of C1 + C2
        const int c0 = __ldg(&a.col0[j]);
        double o = 0.0;
        if (!FX && a.sum) {
            const double* D4 = reinterpret_cast<const double*>(C4);
            stencil_taps<decltype(guard)::value>(c0, [&](int q) { o = fma(__ldg(&a.w1[j * kStencil + q]), D4[c + (c0 + q) * 2 * T], o); });
            return o;
        }
        stencil_taps<decltype(guard)::value>(c0, [&](int q) {
            const int n = c + (c0 + q) * 2 * T;
            o = fma(__ldg(&a.w1[j * kStencil + q]), D1[n] + D2[n], o);
        });
        return o;
    };
    // div_h of (p, m, D3), given dr = 2 d_r v_r + 2 v_r / r of v_r = (p + m) / 2: one halving, which is
    // exact, for three terms
    auto div = [&](double p, double m, double dr, double irj, int i) {
        return fma(kks, D3[i ^ 1], 0.5 * fma(mms * irj, p - m, dr));
    };
    auto stencils = [&] {
        if (stage == 0) {         // A2: pressure right-hand side into C0
            stencil_rows<4, FX, true>(a.fw, a.few, far, C1, C2, N, T, slow12, ir, [&](int j, int i, double d, double irj) {
                double out = 0.0;
                const double n = D1[i], m = D2[i];
                if (j == 0 || j == N - 1) {
                    if (ins && !(j == N - 1 && ms == 0 && ks == 0)) {
                        const double* L = reinterpret_cast<const double*>(Lw + (j == 0 ? 0 : 2 * T) + ts) + part;
                        out = -0.5 * (n + m) + (L[0] + L[2 * T]) - 0.5 * (L[8 * T] + L[10 * T]);
                    }
                } else {
                    out = -div(n, m, fma(n + m, irj, d), irj, i);
                }
                D0[i] = out;
            });
        } else if (stage == 1) {  // C: velocity right-hand sides: subtract grad_h p* on interior rows; p <- p* (commit)
            stencil_rows<4, FX, false>(a.fw, a.few, far, C0, nullptr, N, T, slow0, ir, [&](int j, int i, double d, double irj) {
                if (!ins) return;
                const double pv = D0[i];
                if (pw) pw[2 * (size_t)j * g.nmode] = pv;
                if (j == 0 || j == N - 1) return;
                const double tp = mms * irj * pv;
                D1[i] -= d - tp;
                D2[i] -= d + tp;
                D3[i] -= kks * D0[i ^ 1];
            });
        } else if (stage == 2) {  // E: div_h u* into C0 (homogeneous Neumann / Dirichlet rows)
            if (!FX && a.sum) {
                for (int i = threadIdx.x; i < items; i += blockDim.x) C4[i] = make_double2(C1[i].x + C2[i].x, C1[i].y + C2[i].y);
                __syncthreads();
            }
            stencil_rows<4, FX, true>(a.fw, a.few, far, C1, C2, N, T, slow12, ir, [&](int j, int i, double d, double irj) {
                double out = 0.0;
                if (ins && j > 0 && j < N - 1) out = div(D1[i], D2[i], __dadd_rn(d, __dmul_rn(D1[i] + D2[i], irj)), irj, i);
                D0[i] = out;
            });
        } else {                  // G: u^{i+1} = u* - grad_h phi, p^{i+1} = p* + 3 phi / (2 dt)
            stencil_rows<4, FX, false>(a.fw, a.few, far, C0, nullptr, N, T, slow0, p0, [&](int j, int i, double d, double p) {
                if (!ins) return;
                const size_t e = 2 * ((size_t)j * g.nmode + modes) + part;
                const double f = D0[i], tf = mms * __ldg(&a.ir[j]) * f;
                const double un[3] = {D1[i] - (d - tf), D2[i] - (d + tf), D3[i] - kks * D0[i ^ 1]};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    reinterpret_cast<double*>(a.u_out)[2 * c * g.S + e] = un[c];
                    bad |= nonfinite1(un[c]);
                }
                if (pw) pw[2 * (size_t)j * g.nmode] = fma(c3, f, p);
            });
        }
    };
    // the warps without a substitution, from thread `first` (a multiple of T) on
    auto beside = [&](int first) {
        const int j0 = ((int)threadIdx.x - first) / T, dj = ((int)blockDim.x - first) / T;
        if (stage == 0) {
            // beside P: the part of the velocity right-hand sides that does not depend on p*,
            // (4u - u_prev)/(2dt) - (2N - N_prev), in place of the latter, and the Dirichlet rows
            for (int j = j0; j < N; j += dj) {
                const int idx = j * T + tq;
                double2 o[3] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
                if (in) {
                    if (j == 0 || j == N - 1) {
                        if (mq == 0 && kq == 0) {
                            const double Re = j == 0 ? a.Re_i : a.Re_o;
                            o[0].y = Re;
                            o[1].y = -Re;
                        }
                    } else {
                        const size_t e = (size_t)j * g.nmode + modeq;
                        o[0] = C1[idx];
                        o[1] = C2[idx];
                        o[2] = C3[idx];
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const size_t ec = (size_t)c * g.S + e;
                            const double2 uu = a.u[ec], q = a.up[ec];
                            o[c].x = (4.0 * uu.x - q.x) * c1 - o[c].x;
                            o[c].y = (4.0 * uu.y - q.y) * c1 - o[c].y;
                        }
                    }
                }
                C1[idx] = o[0];
                C2[idx] = o[1];
                C3[idx] = o[2];
            }
        } else if (stage == 1 && a.commit && in) {
            // beside H: rotate the history (nothing reads u_prev or N_prev any more):
            // u_prev <- u^i, N_prev <- N^i
            for (int j = j0; j < N; j += dj)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const size_t ec = (size_t)c * g.S + (size_t)j * g.nmode + modeq;
                    a.up_out[ec] = a.u[ec];
                    a.Np_out[ec] = a.Nc[ec];
                }
        }
    };
#pragma unroll 1
    for (;; ++stage) {
        stencils();
        if (stage == 3) break;
        __syncthreads();
        // B: p* = P^{-1} b_p;  D: the three Helmholtz solves;  F: phi = P^{-1} div_h u* (real and
        // imaginary parts by separate threads, two per (mode, part) with two partitions)
        const int nsys = stage == 1 ? 3 : 1, set0 = stage == 1 ? kSetHp : kSetP, per = (sp ? 4 : 2) * nT;
        const int helper = (nsys * per + 31) / 32 * 32;
        const bool spare = helper < (int)blockDim.x;
        double2* X0 = stage == 1 ? C1 : C0;
        if ((int)threadIdx.x < nsys * per) {
            const int c = nsys == 1 ? 0 : threadIdx.x / per;
            system_solve<FX, true>(a, g, X0 + (size_t)c * items, set0 + c, T, nT, mode0, threadIdx.x - c * per);
        } else if (spare && (int)threadIdx.x >= helper) {
            beside(helper);
        }
        __syncthreads();
        if (!spare) {   // with no spare warp the whole block does it
            beside(0);
            __syncthreads();
        }
        if (sp) spike_combine(a, g, X0, nsys, set0, T, nT, mode0, Xr);
    }
    if (bad && a.nonfinite) *a.nonfinite = 1;
}

// ---------------------------------------------------------------- split path (large N_r)
// With few modes per block in shared memory the fused kernel leaves most lanes idle during
// the substitutions; at large N_r there are enough modes to run each stage as its own
// kernel instead: elementwise right-hand sides and update, and one thread per (system,
// mode, real/imaginary part) walking its column in global memory.

// X = (2N - N_prev)_r = ((2N - N_prev)_+ + (2N - N_prev)_-) / 2, once per element (the
// pressure right-hand side applies the radial stencil to it).
__global__ void k_nn_r(const double2* __restrict__ Nc, const double2* __restrict__ Np, double2* __restrict__ X, Geo g) {
    const int mode = g.mlo + blockIdx.y * blockDim.x + threadIdx.x;   // x = radial row
    if (mode >= g.mhi) return;
    const size_t e = (size_t)blockIdx.x * g.nmode + mode;
    const double2 n1 = Nc[e], n0 = Np[e], m1 = Nc[g.S + e], m0 = Np[g.S + e];
    X[e] = make_double2((n1.x - 0.5 * n0.x) + (m1.x - 0.5 * m0.x), (n1.y - 0.5 * n0.y) + (m1.y - 0.5 * m0.y));
}

// The stages below take the radial stencil of kTileRows consecutive rows of the real or imaginary
// part of one mode per thread in fixed point (fx::Tile; FP64 next to the walls); the two threads of
// a mode then trade halves, and each has both parts of half the rows for the rest, in FP64.  With
// FP64 stencils the FP64 pipe bounded these kernels; now memory and what FP64 is left do.  N_r = 256,
// M = 64, K = 128, before and after: right-hand sides of step 2 478 -> 270 us, of step 3 443 -> 312,
// of step 4 438 -> 178, update 301 -> 277.
struct Stencil {
    const double* w1;
    const int* col0;
    const int2* fw;
    const int2* few;
    int far;   // limit of the rows left to FP64 sums
};
struct Cols {
    int mode, part, m, k, j0;
    bool in;
};

// grid: x over the parts of the modes, y = row tile
__device__ __forceinline__ Cols cols(const Geo& g) {
    Cols c;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    c.mode = g.mlo + (t >> 1);
    c.part = t & 1;
    c.in = c.mode < g.mhi;
    c.m = c.mode / g.nk;
    c.k = c.mode - c.m * g.nk - g.K;
    c.j0 = blockIdx.y * kTileRows;
    return c;
}

// body(j, e, d) for half of the tile's rows: d the radial derivative of F (of F + F2) at row j of
// the thread's mode, e the index of the element
template <bool PAIR, class Body>
__device__ __forceinline__ void tile_rows(const Cols& c, const Stencil& s, const Geo& g, const double2* __restrict__ F,
                                          const double2* __restrict__ F2, Body body) {
    using namespace fx;
    constexpr int H = kTileRows / 2;
    const int N = g.N;
    const size_t st = 2 * (size_t)g.nmode;
    const double* f = reinterpret_cast<const double*>(F) + 2 * (size_t)c.mode + c.part;
    const double* f2 = reinterpret_cast<const double*>(F2) + 2 * (size_t)c.mode + c.part;
    double d[kTileRows];
    {
        double v[kTileRows + 8], v2[kTileRows + 8];
#pragma unroll
        for (int i = 0; i < kTileRows + 8; ++i) {
            const int j = c.j0 - 4 + i;
            const bool on = c.in && j >= 0 && j < N;
            v[i] = on ? __ldg(&f[(size_t)j * st]) : 0.0;
            if (PAIR) v2[i] = on ? __ldg(&f2[(size_t)j * st]) : 0.0;
        }
        Tile<kTileRows> X;
        auto near = [&](int i) { return (unsigned)__ldg(&s.few[min(c.j0 + i, N - 1)].y); };
        const int far = c.mode == g.K ? kFar : s.far;
        if (PAIR) X.load(v, v2, far, near);
        else X.load(v, far, near);
#pragma unroll
        for (int i = 0; i < kTileRows; ++i) {
            const int j = c.j0 + i;
            d[i] = 0.0;
            if (!c.in || j >= N) continue;
            if (j < 4 || j > N - 5 || X.far(i)) {
                const int c0 = __ldg(&s.col0[j]);
                stencil_taps<true>(c0, [&](int t) {
                    const size_t o = (size_t)(c0 + t) * st;
                    const double w = __ldg(&s.w1[j * kStencil + t]), x = __ldg(&f[o]);
                    d[i] = fma(w, PAIR ? x + __ldg(&f2[o]) : x, d[i]);
                });
            } else {
                d[i] = X.row(i, s.fw + j * kStencil, __ldg(&s.few[j].x));
            }
        }
    }
    double2 q[H];   // rows j0 + H part .. + H - 1
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const double give = c.part ? d[i] : d[i + H], keep = c.part ? d[i + H] : d[i];
        const double got = __shfl_xor_sync(0xffffffffu, give, 1);
        q[i] = c.part ? make_double2(got, keep) : make_double2(keep, got);
    }
    if (!c.in) return;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const int j = c.j0 + H * c.part + i;
        if (j < N) body(j, (size_t)j * g.nmode + c.mode, q[i]);
    }
}

// Step 2 right-hand side on the interior rows: div_h(-(2N - N_prev)) (the wall rows:
// k_rhs_pressure_walls).
__global__ void __launch_bounds__(128) k_rhs_pressure(const double2* __restrict__ Nc, const double2* __restrict__ Np,
                                                      const double2* __restrict__ X, double2* __restrict__ b,
                                                      const double* __restrict__ irn, Stencil s, Geo g) {
    const Cols c = cols(g);
    const double mm = g.mp * c.m, kk = g.kz * c.k;
    tile_rows<false>(c, s, g, X, nullptr, [&](int j, size_t e, double2 d) {
        if (j == 0 || j == g.N - 1) return;
        const double2 x = __ldg(&X[e]), n1 = __ldg(&Nc[e]), n0 = __ldg(&Np[e]);
        const double2 z1 = __ldg(&Nc[2 * g.S + e]), z0 = __ldg(&Np[2 * g.S + e]);
        const double ir = __ldg(&irn[j]), mr = mm * ir;
        // (2N - N_prev)_+ - x = ((2N - N_prev)_+ - (2N - N_prev)_-) / 2
        b[e] = make_double2(-(d.x + x.x * ir + mr * ((2.0 * n1.x - n0.x) - x.x) - kk * (2.0 * z1.y - z0.y)),
                            -(d.y + x.y * ir + mr * ((2.0 * n1.y - n0.y) - x.y) + kk * (2.0 * z1.x - z0.x)));
    });
}

// Step 2 right-hand side on the two wall rows: the consistent Neumann value of Eq. ppBC
// (the wall Laplacian of u and u_prev), or the Dirichlet value 0 for (0,0) at r_o; kept apart
// from the interior rows, whose kernel then needs far fewer registers
__global__ void k_rhs_pressure_walls(const double2* __restrict__ u, const double2* __restrict__ up,
                                     const double2* __restrict__ X, double2* __restrict__ b,
                                     const double* __restrict__ rn, const double* __restrict__ w1,
                                     const double* __restrict__ w2, const int* __restrict__ col0, Geo g) {
    const int mode = g.mlo + blockIdx.x * blockDim.x + threadIdx.x;   // y = wall (0: r_i, 1: r_o)
    if (mode >= g.mhi) return;
    const int j = blockIdx.y == 0 ? 0 : g.N - 1;
    const size_t e = (size_t)j * g.nmode + mode;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    double2 out = make_double2(0.0, 0.0);
    if (!(j == g.N - 1 && m == 0 && k == 0)) {
        const double mm = g.mp * m, kk = g.kz * k;
        const double r = rn[j];
        const double2 x = X[e];
        const double2 l0 = lap_r(u, w1, w2, col0, r, j, mode, mm, kk, g);
        const double2 l1 = lap_r(up, w1, w2, col0, r, j, mode, mm, kk, g);
        out.x = -x.x + 2.0 * l0.x - l1.x;
        out.y = -x.y + 2.0 * l0.y - l1.y;
    }
    b[e] = out;
}

// Step 3 right-hand sides, all three components together so that the radial stencil of p* is
// applied once: (4u - u_prev)/(2dt) - (2N - N_prev) - grad_h p*; Dirichlet rows.
// commit: p <- p* (p^{i+1} is completed in the update).
__global__ void __launch_bounds__(128) k_rhs_velocity(const double2* __restrict__ u, const double2* __restrict__ up,
                                                      const double2* __restrict__ Nc, const double2* __restrict__ Np,
                                                      const double2* __restrict__ ps, double2* __restrict__ rhs,
                                                      double2* __restrict__ p_out, const double* __restrict__ irn,
                                                      double Re_i, double Re_o, Stencil s, Geo g) {
    const Cols c = cols(g);
    const double mm = g.mp * c.m, kk = g.kz * c.k;
    tile_rows<false>(c, s, g, ps, nullptr, [&](int j, size_t e, double2 d) {
        const double2 pv = __ldg(&ps[e]);
        if (p_out) p_out[e] = pv;
        if (j == 0 || j == g.N - 1) {
            const double Re = (c.m == 0 && c.k == 0) ? (j == 0 ? Re_i : Re_o) : 0.0;
            rhs[e] = make_double2(0.0, Re);
            rhs[g.S + e] = make_double2(0.0, -Re);
            rhs[2 * g.S + e] = make_double2(0.0, 0.0);
            return;
        }
        const double tt = mm * __ldg(&irn[j]);
        const double2 gp[3] = {make_double2(d.x - tt * pv.x, d.y - tt * pv.y),
                               make_double2(d.x + tt * pv.x, d.y + tt * pv.y),
                               make_double2(-kk * pv.y, kk * pv.x)};
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const size_t ec = f * g.S + e;
            const double2 a = __ldg(&u[ec]), q = __ldg(&up[ec]), n1 = __ldg(&Nc[ec]), n0 = __ldg(&Np[ec]);
            rhs[ec] = make_double2((4.0 * a.x - q.x) * g.c1 - (2.0 * n1.x - n0.x) - gp[f].x,
                                   (4.0 * a.y - q.y) * g.c1 - (2.0 * n1.y - n0.y) - gp[f].y);
        }
    });
}

// Step 4 right-hand side: div_h u* on interior rows, homogeneous Neumann / Dirichlet rows.
__global__ void __launch_bounds__(128) k_rhs_div(const double2* __restrict__ us, double2* __restrict__ b,
                                                 const double* __restrict__ irn, Stencil s, Geo g) {
    const Cols c = cols(g);
    const double mm = g.mp * c.m, kk = g.kz * c.k;
    tile_rows<true>(c, s, g, us, us + g.S, [&](int j, size_t e, double2 d) {
        if (j == 0 || j == g.N - 1) {
            b[e] = make_double2(0.0, 0.0);
            return;
        }
        const double hr = 0.5 * __ldg(&irn[j]), mr = mm * hr;
        const double2 vp = __ldg(&us[e]), vm = __ldg(&us[g.S + e]), vz = __ldg(&us[2 * g.S + e]);
        b[e] = make_double2(0.5 * d.x + (vp.x + vm.x) * hr + mr * (vp.x - vm.x) - kk * vz.y,
                            0.5 * d.y + (vp.y + vm.y) * hr + mr * (vp.y - vm.y) + kk * vz.x);
    });
}

// Step 5, all components together: u^{i+1} = u* - grad_h phi; p^{i+1} = p* + 3 phi/(2dt).
// commit: rotate the history in place (u_prev <- u^i, u <- u^{i+1}, N_prev <- N^i, p += 3 phi/(2dt));
// otherwise write u^{i+1} to u_out only.
__global__ void __launch_bounds__(128) k_update(double2* __restrict__ u, double2* __restrict__ up,
                                                const double2* __restrict__ Nc, double2* __restrict__ Np,
                                                double2* __restrict__ p, const double2* __restrict__ us,
                                                const double2* __restrict__ phi, double2* __restrict__ u_out,
                                                const double* __restrict__ irn, int commit,
                                                int* __restrict__ nonfinite, Stencil s, Geo g) {
    const Cols c = cols(g);
    const double mm = g.mp * c.m, kk = g.kz * c.k, q = 3.0 * g.c1;
    bool bad = false;
    tile_rows<false>(c, s, g, phi, nullptr, [&](int j, size_t e, double2 d) {
        const double2 f = __ldg(&phi[e]);
        const double tt = mm * __ldg(&irn[j]);
        const double2 gph[3] = {make_double2(d.x - tt * f.x, d.y - tt * f.y),
                                make_double2(d.x + tt * f.x, d.y + tt * f.y),
                                make_double2(-kk * f.y, kk * f.x)};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const size_t ec = i * g.S + e;
            const double2 v = __ldg(&us[ec]), un = make_double2(v.x - gph[i].x, v.y - gph[i].y);
            bad |= nonfinite2(un);
            if (commit) {
                up[ec] = u[ec];
                u[ec] = un;
                Np[ec] = __ldg(&Nc[ec]);
            } else {
                u_out[ec] = un;
            }
        }
        if (commit) {
            const double2 a = p[e];
            p[e] = make_double2(a.x + q * f.x, a.y + q * f.y);
        }
    });
    if (bad && nonfinite) *nonfinite = 1;
}

// smem_band_solve on a column in global memory, in the same arithmetic: the right-hand side's
// rows come in through the ring with the factors, D rows ahead.  Used while a launch has few
// warps (launch_advance_split): there each row waited one memory latency.
constexpr int kGD = 6;   // ring depth (2, 3, 4, 5, 6, 8: 325, 325, 290, 275, 267, 267 us for a Poisson solve, N_r = 256, M = 64, K = 128)
template <int D>
__device__ __forceinline__ void gmem_band_solve(double* __restrict__ x, size_t st, int N, const double* __restrict__ F,
                                                const uint8_t* __restrict__ P, int M1K1) {
    const size_t rs = (size_t)kBands * M1K1;
    double w0 = x[0], w1 = N > 1 ? x[st] : 0.0, w2 = N > 2 ? x[2 * st] : 0.0, w3 = N > 3 ? x[3 * st] : 0.0,
           w4 = N > 4 ? x[4 * st] : 0.0;
    double lr[D][4], br[D];
    int pr[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        pr[d] = d < N ? P[(size_t)d * M1K1] : 0;
        br[d] = d + 5 < N ? x[(size_t)(d + 5) * st] : 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) lr[d][q] = d < N ? __ldg(&F[(size_t)d * rs + (size_t)q * M1K1]) : 0.0;
    }
    for (int j0 = 0; j0 < N; j0 += D) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int j = j0 + d;
            if (j < N) {
                const int pj = pr[d];
                const double l1 = lr[d][0], l2 = lr[d][1], l3 = lr[d][2], l4 = lr[d][3], b = br[d];
                if (j + D < N) {
                    const double* Fr = F + (size_t)(j + D) * rs;
                    pr[d] = P[(size_t)(j + D) * M1K1];
#pragma unroll
                    for (int q = 0; q < 4; ++q) lr[d][q] = __ldg(&Fr[(size_t)q * M1K1]);
                }
                br[d] = j + D + 5 < N ? x[(size_t)(j + D + 5) * st] : 0.0;
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
                w4 = b;
            }
        }
    }
    double v1 = 0.0, v2 = 0.0, v3 = 0.0, v4 = 0.0, v5 = 0.0, v6 = 0.0, v7 = 0.0, v8 = 0.0;
    double ur[D][9];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const int j = N - 1 - d;
        br[d] = j >= 0 ? x[(size_t)j * st] : 0.0;
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
                double s = br[d];
                if (j - D >= 0) {
                    br[d] = x[(size_t)(j - D) * st];
#pragma unroll
                    for (int q = 0; q < 9; ++q) ur[d][q] = __ldg(&F[(size_t)(j - D) * rs + (size_t)(4 + q) * M1K1]);
                }
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

// x <- A^{-1} x for every mode of nfields consecutive fields (system sets set0, set0+1, ...):
// thread (field, mode, part) runs the register-window substitution down its global column.
template <int D>
__global__ void k_band_solve_g(double2* __restrict__ x, const double* __restrict__ fac,
                               const uint8_t* __restrict__ piv, int set0, int nfields, Geo g) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;   // (mode, part); y = field
    if (t >= 2 * (g.mhi - g.mlo)) return;
    const int part = t & 1;
    const int mode = g.mlo + (t >> 1);
    const int fld = blockIdx.y;
    const int m = mode / g.nk;
    const int k = mode - m * g.nk - g.K;
    const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
    const size_t per_set = (size_t)g.N * kBands * g.M1K1;
    const int set = set0 + fld;
    const double* F = fac + (size_t)set * per_set + mk;
    const uint8_t* P = piv + (size_t)set * g.N * g.M1K1 + mk;
    if (D > 1) gmem_band_solve<D>(reinterpret_cast<double*>(x + (size_t)fld * g.S + mode) + part, (size_t)2 * g.nmode, g.N, F, P, g.M1K1);
    else smem_band_solve(x + (size_t)fld * g.S + mode, g.nmode, part, g.N, F, P, g.M1K1);
}

// Stand-alone solves of one system set for all modes (tc_helmholtz_solve): columns staged in shared
// memory, real and imaginary parts by separate threads.  rhs may be x: a block reads its columns
// before it writes them.
// In two partitions, T modes per block (as in k_pc's solve phases):
__global__ void __launch_bounds__(128) k_band_solve_s2(const double2* rhs, double2* x, PCArgs a, int set, Geo g, int T) {
    extern __shared__ double2 sm[];
    const int N = g.N, mode0 = blockIdx.x * T, nT = min(T, g.nmode - mode0), t = threadIdx.x % T;
    for (int j = threadIdx.x / T; j < N; j += blockDim.x / T)
        sm[j * T + t] = t < nT ? rhs[(size_t)j * g.nmode + mode0 + t] : make_double2(0.0, 0.0);
    __syncthreads();
    if (threadIdx.x < 4 * nT) system_solve<true, false>(a, g, sm, set, T, nT, mode0, threadIdx.x);
    __syncthreads();
    spike_combine(a, g, sm, 1, set, T, nT, mode0, reinterpret_cast<double*>(sm + (size_t)N * T));
    if (t < nT)
        for (int j = threadIdx.x / T; j < N; j += blockDim.x / T) x[(size_t)j * g.nmode + mode0 + t] = sm[j * T + t];
}

// In one:
__global__ void __launch_bounds__(256) k_band_solve_s(const double2* rhs, double2* x, const double* __restrict__ fac,
                                                      const uint8_t* __restrict__ piv, int set, Geo g, int T) {
    extern __shared__ double2 sm[];
    const int N = g.N;
    const int mode0 = g.mlo + blockIdx.x * T;
    const int nT = min(T, g.mhi - mode0);
    for (int idx = threadIdx.x; idx < N * T; idx += blockDim.x) {
        const int j = idx / T, t = idx - (idx / T) * T;
        sm[idx] = t < nT ? rhs[(size_t)j * g.nmode + mode0 + t] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (threadIdx.x < 2 * nT) {
        const int t = threadIdx.x >> 1, part = threadIdx.x & 1;
        const int mode = mode0 + t, m = mode / g.nk, k = mode - m * g.nk - g.K;
        const size_t mk = (size_t)m * g.K1 + (k < 0 ? -k : k);
        const size_t per_set = (size_t)N * kBands * g.M1K1;
        smem_band_solve<kPCDepth>(sm, T, 2 * t + part, N, fac + (size_t)set * per_set + mk, piv + (size_t)set * N * g.M1K1 + mk, g.M1K1);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < N * T; idx += blockDim.x) {
        const int j = idx / T, t = idx - (idx / T) * T;
        if (t < nT) x[(size_t)j * g.nmode + mode0 + t] = sm[idx];
    }
}

__global__ void k_axpby(double2* __restrict__ y, const double2* __restrict__ a, double ca,
                        const double2* __restrict__ b, double cb, size_t n) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const double2 x = a[e], z = b[e];
    y[e] = make_double2(ca * x.x + cb * z.x, ca * x.y + cb * z.y);
}

// Diagnostics: red[1] = max |div_h u| (as ordered bits), red[2] += non-finite, and each
// block's energy sum in red[kDiagPartials + block]; k_diag_sum adds those in a fixed order into
// red[0], so the energy does not depend on the order in which blocks finish.
constexpr int kDiagPartials = 8;
__global__ void k_diag(const double2* __restrict__ u, double* __restrict__ red,
                       const double* __restrict__ rn, const double* __restrict__ w1,
                       const int* __restrict__ col0, double C1, double C2, Geo g) {
    __shared__ double s_e[256];
    __shared__ unsigned long long s_d[256];
    __shared__ int s_n[256];
    const int mode = blockIdx.x * blockDim.x + threadIdx.x;   // y = radial row
    const int j = blockIdx.y;
    const size_t e = (size_t)j * g.nmode + mode;
    double en = 0.0, dv = 0.0;
    int bad = 0;
    if (mode < g.nmode) {
        const int m = mode / g.nk;
        const int k = mode - m * g.nk - g.K;
        const double r = rn[j];
        double2 a = u[e], b = u[g.S + e], z = u[2 * g.S + e];
        bad = !(isfinite(a.x) && isfinite(a.y) && isfinite(b.x) && isfinite(b.y) && isfinite(z.x) && isfinite(z.y));
        if (m == 0 && k == 0) {
            const double U = C1 * r + C2 / r;
            a.y -= U;
            b.y += U;
        }
        double wr = 0.0;
        if (j > 0) wr += 0.5 * (r - rn[j - 1]);
        if (j < g.N - 1) wr += 0.5 * (rn[j + 1] - r);
        const double cm = m == 0 ? 1.0 : 2.0;
        en = 0.5 * wr * r * cm * (0.5 * (a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y) + z.x * z.x + z.y * z.y);
        if (j > 0 && j < g.N - 1) {
            const int c0 = col0[j];
            double2 d = make_double2(0.0, 0.0);
            for (int t = 0; t < kStencil; ++t) {
                if (!stencil_row(c0, t)) continue;
                const double wt = w1[j * kStencil + t];
                const size_t o = (size_t)(c0 + t) * g.nmode + mode;
                const double2 p1 = u[o], p2 = u[g.S + o];
                d.x += wt * 0.5 * (p1.x + p2.x);
                d.y += wt * 0.5 * (p1.y + p2.y);
            }
            const double2 vp = u[e], vm = u[g.S + e], vz = u[2 * g.S + e];
            const double mm = g.mp * m, kk = g.kz * k, ir = 1.0 / r;
            const double dx = d.x + 0.5 * (vp.x + vm.x) * ir + mm * (vp.x - vm.x) * 0.5 * ir - kk * vz.y;
            const double dy = d.y + 0.5 * (vp.y + vm.y) * ir + mm * (vp.y - vm.y) * 0.5 * ir + kk * vz.x;
            dv = sqrt(dx * dx + dy * dy);
        }
        if (!isfinite(en)) en = 0.0;
        if (!isfinite(dv)) dv = 0.0;
    }
    s_e[threadIdx.x] = en;
    s_d[threadIdx.x] = (unsigned long long)__double_as_longlong(dv);
    s_n[threadIdx.x] = bad;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            s_e[threadIdx.x] += s_e[threadIdx.x + w];
            s_d[threadIdx.x] = max(s_d[threadIdx.x], s_d[threadIdx.x + w]);
            s_n[threadIdx.x] += s_n[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        red[kDiagPartials + (size_t)blockIdx.y * gridDim.x + blockIdx.x] = s_e[0];
        atomicMax(reinterpret_cast<unsigned long long*>(&red[1]), s_d[0]);
        atomicAdd(reinterpret_cast<unsigned long long*>(&red[2]), (unsigned long long)s_n[0]);
    }
}

// red[0] = sum of the n block partials: each thread a contiguous run, then a tree (one block)
__global__ void __launch_bounds__(1024) k_diag_sum(double* __restrict__ red, int n) {
    __shared__ double s[1024];
    const int per = (n + 1023) / 1024;
    double a = 0.0;
    for (int i = threadIdx.x * per; i < (threadIdx.x + 1) * per && i < n; ++i) a += red[kDiagPartials + i];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) red[0] = s[0];
}

static int blocks_for(size_t n, int bs) { return (int)((n + bs - 1) / bs); }

// doubles of the diagnostics reduction buffer: the fixed slots and one partial per k_diag block
size_t diag_red_doubles(const tc_plan* p) {
    return kDiagPartials + (size_t)blocks_for((size_t)p->nmode, 256) * p->N_r;
}

// Modes per block of the fused kernel (a power of two): the most (up to 16) that still give every SM a block,
// within 96 KB of shared memory for the four columns.  Each block's time is its substitution
// chain, so more modes per block cost little while the blocks fit one wave.
int pc_modes(const tc_plan* p, int nmode) {
    int T = 16;
    if (p->pc_modes > 0)
        while (T > p->pc_modes) T /= 2;   // a power of two: it divides the block size
    else
        while (T > 4 && (nmode + T - 1) / T < p->num_sms) T /= 2;
    while (T > 1 && (size_t)4 * p->N_r * T * sizeof(double2) > 96 * 1024) T /= 2;
    return T;
}

// x = A^{-1} rhs of the factor set for every mode (rhs may be x)
tc_status launch_solve(tc_plan* p, int set, const double2* rhs, double2* x, cudaStream_t s) {
    Geo g = geo(p);
    const int prof = set == kSetP ? kKSolveP : kKSolveH;
    if (p->part_h > 0 && g.nmode <= 64 * p->num_sms) {
        // two partitions: half the chain of substitutions, which bounds a launch of few modes per SM
        // (55: 103 against 127 us, N_r = 128); with many the coupling's work counts (110: 53 against
        // 41 us, N_r = 32)
        g.sh = p->part_h;
        PCArgs a{};
        a.fac2 = p->d_fac2; a.piv2 = p->d_piv2; a.spk = p->d_spk; a.rinv = p->d_rinv;
        int T = 16;   // a power of two: it divides the block size
        while (T > 1 && (size_t)p->N_r * T * sizeof(double2) > 96 * 1024) T /= 2;
        const size_t sm = (size_t)p->N_r * T * sizeof(double2) + (size_t)T * 16 * sizeof(double);
        TC_CUDA(p, cudaFuncSetAttribute(k_band_solve_s2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        const int slot = prof_begin(p, prof, s);
        k_band_solve_s2<<<blocks_for(g.nmode, T), 128, sm, s>>>(rhs, x, a, set, g, T);
        prof_end(p, slot, s);
        TC_LAUNCHED(p, "k_band_solve_s2");
        return TC_OK;
    }
    int T = 32;
    while (T > 1 && (size_t)p->N_r * T * sizeof(double2) > 96 * 1024) T /= 2;
    const size_t sm = (size_t)p->N_r * T * sizeof(double2);
    TC_CUDA(p, cudaFuncSetAttribute(k_band_solve_s, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int slot = prof_begin(p, prof, s);
    k_band_solve_s<<<blocks_for(g.nmode, T), 64, sm, s>>>(rhs, x, p->d_fac, p->d_piv, set, g, T);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_band_solve_s");
    return TC_OK;
}

// Limit of the rows that the fixed-point stencils of a mixed plan leave to FP64 sums: its transforms are in FP32, and
// its stencils were double-FP32 dot products, good to 2^-46 of sum |w f|; this limit keeps them at 2^-47.
// The mean mode keeps fx::kFar.  k_pc with fx::kFar throughout: 895 against 854 us (N_r = 64, M = 64,
// K = 128).
constexpr int kFarMixed = 12;

static tc_status launch_advance_split(tc_plan* p, const double2* u, double2* u_prev, const double2* Ncur,
                                      double2* N_prev, double2* p_out, double2* u_out, char* ws, bool commit,
                                      cudaStream_t s, int ma, int mb) {
    Geo g = geo(p);
    g.mlo = ma * g.nk;
    g.mhi = mb * g.nk;
    const int nm = g.mhi - g.mlo;
    double2* ps = reinterpret_cast<double2*>(ws + p->ws.pstar);
    double2* us = reinterpret_cast<double2*>(ws + p->ws.ustar);
    double2* phi = reinterpret_cast<double2*>(ws + p->ws.phi);   // also holds X before phi
    const dim3 g1(g.N, blocks_for(nm, 128));
    // nf substitutions with the factor sets set ..: the ring while a launch has fewer than 24 warps
    // per SM (20.6 warps: 680 against 706 us), the plain one beyond, where other warps cover the
    // latency and 40 registers more per thread do not pay (27 warps: 793 against 1008 us)
    auto split_solve = [&](double2* x, int set, int nf) {
        const dim3 grid(blocks_for((size_t)2 * nm, 128), nf);
        const bool ring = (size_t)2 * nm * nf < (size_t)24 * 32 * p->num_sms;
        (ring ? k_band_solve_g<kGD> : k_band_solve_g<1>)<<<grid, 128, 0, s>>>(x, p->d_fac, p->d_piv, set, nf, g);
    };
    const Stencil st{p->d_w1, p->d_col0, p->d_fx_w1, p->d_fx_ew, p->precision == TC_MIXED ? kFarMixed : fx::kFar};
    const dim3 gt(blocks_for((size_t)2 * nm, 128), blocks_for(g.N, kTileRows));
    int slot = prof_begin(p, kKRhsPressure, s);
    k_nn_r<<<g1, 128, 0, s>>>(Ncur, N_prev, phi, g);
    k_rhs_pressure<<<gt, 128, 0, s>>>(Ncur, N_prev, phi, ps, p->d_ir, st, g);
    k_rhs_pressure_walls<<<dim3(blocks_for(nm, 128), 2), 128, 0, s>>>(u, u_prev, phi, ps, p->d_r, p->d_w1, p->d_w2,
                                                                     p->d_col0, g);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_rhs_pressure");
    slot = prof_begin(p, kKSolveP, s);
    split_solve(ps, kSetP, 1);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_band_solve_g");
    slot = prof_begin(p, kKRhsVelocity, s);
    k_rhs_velocity<<<gt, 128, 0, s>>>(u, u_prev, Ncur, N_prev, ps, us, commit ? p_out : nullptr, p->d_ir, p->Re_i,
                                      p->Re_o, st, g);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_rhs_velocity");
    slot = prof_begin(p, kKSolveH, s);
    split_solve(us, kSetHp, 3);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_band_solve_g");
    slot = prof_begin(p, kKRhsDiv, s);
    k_rhs_div<<<gt, 128, 0, s>>>(us, phi, p->d_ir, st, g);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_rhs_div");
    slot = prof_begin(p, kKSolveP, s);
    split_solve(phi, kSetP, 1);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_band_solve_g");
    slot = prof_begin(p, kKUpdate, s);
    k_update<<<gt, 128, 0, s>>>(const_cast<double2*>(u), u_prev, Ncur, N_prev, p_out, us, phi, u_out, p->d_ir,
                                commit ? 1 : 0, p->d_nonfinite, st, g);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_update");
    return TC_OK;
}

// Fixed-point stencils in a launch of blocks of T modes.  With up to 8 warps per SM, one block of 256
// threads, their conversions take longer than the FP64 FMAs (N_r = 160, M = 8, K = 16: 273 against 225 us;
// N_r = 64, M = 24, K = 48, 152 blocks: 184 against 160 in the mixed form).  With more
// they are the faster form from some 76 rows on: below, two blocks with a fifth column for the sum of
// u_+ and u_- (launch_advance) fit an SM, and the tiles of 4 rows do not spread evenly over the warps.
// M = 64, K = 128, fixed point against FP64: N_r = 48 756 and 674 us, 64 909 and 890, 72 1017 and 1009;
// M = K = 64: N_r = 80 556 and 563, 96 652 and 729.  In the mixed form, which leaves fewer rows to FP64
// (kFarMixed), from 56 on: 48 696 and 674, 56 783 and 784, 64 874 and 890.
static bool fx_stencils(const tc_plan* p, int nmode, int T) {
    return p->N_r >= (p->precision == TC_MIXED ? 56 : 76) &&
           (size_t)blocks_for(nmode, T) * (T <= 8 ? 128 : 256) > (size_t)256 * p->num_sms;
}

tc_status launch_advance(tc_plan* p, const double2* u, double2* u_prev, const double2* Ncur,
                         double2* N_prev, double2* p_out, double2* u_out, char* ws, bool commit,
                         cudaStream_t s, int ma, int mb) {
    if (mb < 0) mb = p->M + 1;
    if (p->pc_split) return launch_advance_split(p, u, u_prev, Ncur, N_prev, p_out, u_out, ws, commit, s, ma, mb);
    Geo g = geo(p);
    g.mlo = ma * g.nk;
    g.mhi = mb * g.nk;
    const int T = pc_modes(p, g.mhi - g.mlo);
    PCArgs a;
    a.u = u; a.up = u_prev; a.Nc = Ncur; a.Np = N_prev;
    a.u_out = commit ? const_cast<double2*>(u) : u_out;
    a.up_out = commit ? u_prev : nullptr;
    a.Np_out = commit ? N_prev : nullptr;
    a.p = commit ? p_out : nullptr;
    a.ir = p->d_ir; a.w1 = p->d_w1; a.w2 = p->d_w2; a.col0 = p->d_col0;
    a.fw = p->d_fx_w1; a.few = p->d_fx_ew;
    a.fac = p->d_fac; a.piv = p->d_piv;
    a.fac2 = p->d_fac2; a.piv2 = p->d_piv2; a.spk = p->d_spk; a.rinv = p->d_rinv;
    a.nonfinite = p->d_nonfinite;
    a.Re_i = p->Re_i; a.Re_o = p->Re_o;
    a.commit = commit ? 1 : 0;
    // two partitions while the 12 T substitution threads of the Helmholtz phase fit the block
    g.sh = (p->part_h > 0 && 12 * T <= (T <= 8 ? 128 : 256)) ? p->part_h : 0;
    size_t sm = (size_t)4 * p->N_r * T * sizeof(double2) + (size_t)3 * T * 16 * sizeof(double);
    // 128 threads up to 8 modes per block, 256 beyond (6T substitution threads plus helpers)
    const int slot = prof_begin(p, kKPC, s);
    auto run = [&](auto kern, int nth) -> tc_status {
        TC_CUDA(p, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        kern<<<blocks_for(g.mhi - g.mlo, T), nth, sm, s>>>(a, g, T);
        return TC_OK;
    };
    const bool fxs = fx_stencils(p, g.mhi - g.mlo, T);
    a.far = p->precision == TC_MIXED ? kFarMixed : fx::kFar;
    // A fifth column for C1 + C2, whose FP64 stencils then take 9 operations less a row (N_r = 48, M = 64,
    // K = 128: 716 -> 660 us), where it costs no block its place:
    // per_sm blocks of an SM that the registers allow and the launch has.
    const size_t col = (size_t)p->N_r * T * sizeof(double2);
    const int per_sm = std::min(T <= 8 ? 4 : 2, (blocks_for(g.mhi - g.mlo, T) + p->num_sms - 1) / p->num_sms);
    a.sum = !fxs && (sm + col + 1024) * per_sm <= (size_t)228 * 1024 ? 1 : 0;
    if (a.sum) sm += col;
    if (T <= 8) TC_TRY_STATUS(fxs ? run(k_pc<128, true>, 128) : run(k_pc<128, false>, 128));
    else TC_TRY_STATUS(fxs ? run(k_pc<256, true>, 256) : run(k_pc<256, false>, 256));
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_pc");
    return TC_OK;
}

tc_status launch_axpby(tc_plan* p, double2* y, const double2* a, double ca, const double2* b,
                       double cb, size_t n, cudaStream_t s) {
    { const int slot_ = prof_begin(p, kKAxpby, s); k_axpby<<<blocks_for(n, 256), 256, 0, s>>>(y, a, ca, b, cb, n); prof_end(p, slot_, s); }
    TC_LAUNCHED(p, "k_axpby");
    return TC_OK;
}

tc_status launch_diagnostics(tc_plan* p, const double2* u, double* red, cudaStream_t s) {
    Geo g = geo(p);
    const double eta = p->eta;
    const double C1 = (p->Re_o - eta * p->Re_i) / (1.0 + eta);
    const double C2 = eta * (p->Re_i - eta * p->Re_o) / ((1.0 - eta) * (1.0 - eta * eta));
    TC_CUDA(p, cudaMemsetAsync(red, 0, 4 * sizeof(double), s));
    const dim3 grid(blocks_for(g.nmode, 256), g.N);
    const int slot = prof_begin(p, kKDiag, s);
    k_diag<<<grid, 256, 0, s>>>(u, red, p->d_r, p->d_w1, p->d_col0, C1, C2, g);
    k_diag_sum<<<1, 1024, 0, s>>>(red, (int)(grid.x * grid.y));
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_diag");
    return TC_OK;
}

}  // namespace tc
