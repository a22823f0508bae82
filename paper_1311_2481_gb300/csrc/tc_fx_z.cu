// FP64 form of the nonlinear term N(u) = u . grad u (Sec. 3.2 step 1, Eq. NS_cyl) on the
// P_theta x P_z dealiased grid (Sec. 3.1), in 64-bit fixed point (tc_fx.cuh).  Four kernels, the
// staging lines H1 and H2 in the workspace between them (the single-GPU counterpart of the
// paper's global transposes, Sec. 4):
//
//   k_fx_dr     per (c, mode, 8 rows): d_r u by the FD stencil (Sec. 3.1), to FP64, into the H2
//               region, which is free until the theta pass
//   k_fx_zinv   per (r, m, c): the lines of u, d_r u and d_z u = i k k_z u, zero-padded inverse
//               transforms along z                                     -> H1[9][r][m][z]
//   k_fx_theta  per (r, z tile): the 12 real fields as 6 complex inverse transforms along theta
//               (two real fields per line; d_theta = i m m_p applied here), the products with
//               the curvature terms, and the forward transforms of N_r + i N_theta (giving N_+
//               and N_- directly) and of N_z (two z per line)           -> H2[3][r][m][z]
//   k_fx_zfwd   per (r, m): forward transforms along z, truncation, 1/(P_theta P_z), to FP64.
//
// Exponents.  Every H1 line has its own (chosen from the sum of the moduli of its input, so
// that no partial sum overflows), with a bound of its largest value; from these each theta
// block takes the exponents of its six line kinds.  Products are taken from lines shifted up
// to their true maximum, and N's line to the sum of its moduli before the forward transform.
// A NaN or Inf anywhere in a row of u makes N of that row NaN, as the FP64 transforms did.
#include <algorithm>

#include "tc_fx_nl.cuh"

namespace tc {

using namespace fx;

namespace {

constexpr int kDrRows = 8;      // rows per thread of k_fx_dr
constexpr int kZThreads = 512;  // most threads of a transform block (128 registers each)

// exponent arrays of nh staged rows, in the fxe region: e1[9][nh][M+1] (exponent, largest
// |re| + |im| in units of 2^32), e2max[nh][2], e2[nh][tiles][2]; behind them s2[nh][tiles], the sums of N_t
struct Exps {
    int2* e1;
    int* e2;
    int* e2max;
    longlong2* s2;
};

// ---------------------------------------------------------------- radial derivative
// Rows j0 .. j0 + 7 of the real or imaginary part of one column per thread (fx::Tile).  Tiles
// start at multiples of kDrRows whatever r0, so that a row's result does not depend on the slab
// it is staged in.
__global__ void __launch_bounds__(128) k_fx_dr(const double* __restrict__ u, double* __restrict__ du,
                                               const int2* __restrict__ w, const int2* __restrict__ ew,
                                               const double* __restrict__ w1, const int* __restrict__ col0, int N,
                                               int ncol, int r0, int nh) {
    const int c = blockIdx.z, tile = (r0 / kDrRows + blockIdx.y) * kDrRows - r0, j0 = r0 + tile;
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= ncol) return;
    const double* src = u + (size_t)c * N * ncol + col;
    double d[kDrRows + 8];
#pragma unroll
    for (int i = 0; i < kDrRows + 8; ++i) {
        const int j = j0 - 4 + i;
        d[i] = j >= 0 && j < N ? __ldg(&src[(size_t)j * ncol]) : 0.0;
    }
    Tile<kDrRows> x;
    x.load(d, kFar, [&](int i) { return (unsigned)__ldg(&ew[min(max(j0 + i, 0), N - 1)].y); });
#pragma unroll
    for (int i = 0; i < kDrRows; ++i) {
        const int j = j0 + i;
        if (tile + i >= nh) break;
        if (tile + i < 0) continue;
        double o = 0.0;
        if (j < 4 || j > N - 5 || x.far(i)) {
            const int c0 = __ldg(&col0[j]);
            double v[kStencil];
#pragma unroll
            for (int t = 0; t < kStencil; ++t) v[t] = stencil_row(c0, t) ? __ldg(&src[(ptrdiff_t)(c0 + t) * ncol]) : 0.0;
#pragma unroll
            for (int t = 0; t < kStencil; ++t) o = fma(__ldg(&w1[j * kStencil + t]), v[t], o);
        } else {
            o = x.row(i, w + j * kStencil, __ldg(&ew[j].x));
        }
        du[((size_t)c * nh + tile + i) * ncol + col] = o;
    }
}

// s[line] = max / sum over the threads of a line, tl consecutive threads per line (line < 0 or
// >= NL: none).  From 32 threads per line on, a warp holds at most two lines and reduces each
// in registers; 32 atomics on one address would take turns.
template <int NL, bool MAX> __device__ __forceinline__ void line_reduce(unsigned* s, int line, unsigned v, int tl) {
    if (tl < 32) {
        if (line < NL) {
            if (MAX) atomicMax(&s[line], v);
            else atomicAdd(&s[line], v);
        }
        return;
    }
    const int first = __shfl_sync(0xffffffffu, line, 0), last = __shfl_sync(0xffffffffu, line, 31);
    const unsigned a = line == first ? v : 0u, b = line == first ? 0u : v;
    const unsigned ra = MAX ? __reduce_max_sync(0xffffffffu, a) : __reduce_add_sync(0xffffffffu, a);
    const unsigned rb = first == last ? 0u : MAX ? __reduce_max_sync(0xffffffffu, b) : __reduce_add_sync(0xffffffffu, b);
    if ((threadIdx.x & 31) == 0) {
        if (first < NL) {
            if (MAX) atomicMax(&s[first], ra);
            else atomicAdd(&s[first], ra);
        }
        if (last != first && last < NL) {
            if (MAX) atomicMax(&s[last], rb);
            else atomicAdd(&s[last], rb);
        }
    }
}

// ---------------------------------------------------------------- inverse z pass
// NL lines per block, out of the nine (d, c) of an (r, m), d = 0, 1, 2 for u, d_r u, d_z u.  tl
// threads per line hold its entries (at most 8 each) from the load to the fixed-point line.
// ADJ: the three lines of the adjoint field Nbar = u instead, (s_r, s_t, s_z) = c_m scale (Nbar_+ +
// Nbar_-, -i (Nbar_+ - Nbar_-), Nbar_z) with c_m = 1 for m = 0 and 1/2 beyond (kz: the scale).
template <class PL, int NL, bool ADJ>
__global__ void __launch_bounds__(kZThreads) k_fx_zinv(const double2* __restrict__ u, const double2* __restrict__ du,
                                                       cx* __restrict__ H1, int2* __restrict__ e1, int N, int M, int K,
                                                       double kz, int r0, int nh, FxPlan f, const int4* __restrict__ tw,
                                                       int tl, unsigned mtl, int* __restrict__ e2max,
                                                       const double* __restrict__ w1, const int* __restrict__ col0) {
    extern __shared__ cx buf[];
    __shared__ unsigned s_e[NL], s_l1[NL], s_mx[NL];
    const PL pl(f);
    const int P = pl.size(), lp = line_pitch(P), nk = 2 * K + 1, nmode = (M + 1) * nk;
    int t = blockIdx.x;
    constexpr int NF = ADJ ? 3 : 9;
    const int f0 = t % (NF / NL) * NL;   // lines in the order 3 c + d: a block reads few lines of u
    t /= NF / NL;
    const int rl = t % nh, m = t / nh;   // rows fastest: neighbouring blocks share cache lines of u
    constexpr int NE = ADJ ? 6 : 2;      // the theta pass takes maxima here
    if (m == 0 && f0 == 0 && threadIdx.x < NE) e2max[rl * NE + threadIdx.x] = 4 * kExpZero;
    if (threadIdx.x < NL) {
        s_e[threadIdx.x] = 0;
        s_l1[threadIdx.x] = 0;
        s_mx[threadIdx.x] = 0;
    }
    __syncthreads();
    const int line = NL == 1 ? 0 : udiv(threadIdx.x, mtl), i0 = threadIdx.x - line * tl;
    const bool on = line < NL;
    const int c = ADJ ? f0 + line : (f0 + line) / 3, d = ADJ ? 0 : f0 + line - 3 * c;
    double2 x[8];
    int e = 0;
    if (ADJ && on) {
        const double2* a = u + (size_t)(r0 + rl) * nmode + (size_t)m * nk;
        const size_t S = (size_t)N * nmode;
        const double cm = (m == 0 ? 1.0 : 0.5) * kz;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = i0 + i * tl;
            x[i] = make_double2(0.0, 0.0);
            if (k < nk) {
                if (c == 2) {
                    const double2 v = __ldg(&a[2 * S + k]);
                    x[i] = make_double2(cm * v.x, cm * v.y);
                } else {
                    const double2 p = __ldg(&a[k]), n = __ldg(&a[S + k]);
                    x[i] = c == 0 ? make_double2(cm * (p.x + n.x), cm * (p.y + n.y)) : make_double2(cm * (p.y - n.y), -cm * (p.x - n.x));
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) e = max(e, max(bexp(x[i].x), bexp(x[i].y)));
    }
    if (!ADJ && on) {
        const double2* src = d == 1 && du ? du + ((size_t)c * nh + rl) * nmode + (size_t)m * nk
                                          : u + ((size_t)c * N + r0 + rl) * nmode + (size_t)m * nk;
        if (NL == 9 && d == 1 && !du) {   // d_r u here, in FP64
            const int j0 = __ldg(&col0[r0 + rl]);
            const double2* a = u + ((ptrdiff_t)c * N + j0) * nmode + (ptrdiff_t)m * nk;
            double w[kStencil];
#pragma unroll
            for (int q = 0; q < kStencil; ++q) w[q] = __ldg(&w1[(r0 + rl) * kStencil + q]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                x[i] = make_double2(0.0, 0.0);
                if (i0 + i * tl < nk) {
                    double2 y = make_double2(0.0, 0.0);   // two sums: half the chain of dependent FMAs
#pragma unroll
                    for (int q = 0; q < kStencil; ++q) {
                        const double2 v = stencil_row(j0, q) ? __ldg(&a[(ptrdiff_t)q * nmode + i0 + i * tl]) : make_double2(0.0, 0.0);
                        double2& o = q & 1 ? y : x[i];
                        o.x = fma(w[q], v.x, o.x);
                        o.y = fma(w[q], v.y, o.y);
                    }
                    x[i].x += y.x;
                    x[i].y += y.y;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = i0 + i * tl < nk ? __ldg(&src[i0 + i * tl]) : make_double2(0.0, 0.0);
        }
        if (d == 2) {   // the FP64 pipe is otherwise idle here
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const double kk = kz * (i0 + i * tl - K);
                x[i] = make_double2(-kk * x[i].y, kk * x[i].x);
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) e = max(e, max(bexp(x[i].x), bexp(x[i].y)));
    }
    line_reduce<NL, true>(s_e, line, (unsigned)e, tl);
    zero_band(pl, buf, lp, NL, K + 1, P - K);
    __syncthreads();
    cx v[8];
    unsigned l1 = 0;
    if (on) {
        e = (int)s_e[line];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] = mk(fix(x[i].x, e), fix(x[i].y, e));
            l1 += ((mag_hi(v[i].x) + mag_hi(v[i].y)) >> 11) + 1;
        }
    }
    line_reduce<NL, false>(s_l1, line, l1, tl);
    __syncthreads();
    if (on) {
        // sum of moduli < s_l1 2^43: shifted to below 2^62
        const int s = max(0, bits(s_l1[line]) - 19);
        const long long h = half_of(s);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = i0 + i * tl - K;
            if (k <= K) buf[line * lp + (k >= 0 ? k : k + P)] = mk((v[i].x + h) >> s, (v[i].y + h) >> s);
        }
    }
    __syncthreads();
    transform(pl, buf, lp, NL, tw, true);
    unsigned mx = 0;
    if (on) {
        cx* dst = H1 + (((size_t)(3 * d + c) * nh + rl) * (M + 1) + m) * P;
        for (int p = i0; p < P; p += tl) {
            const cx o = buf[line * lp + pd(p)];
            dst[p] = o;
            mx = max(mx, mag_hi(o.x) + mag_hi(o.y) + 2);
        }
    }
    line_reduce<NL, true>(s_mx, line, mx, tl);
    __syncthreads();
    if (on && i0 == 0) {
        const int s = max(0, bits(s_l1[line]) - 19);
        e1[((size_t)(3 * d + c) * nh + rl) * (M + 1) + m] =
            e == 0 ? make_int2(kExpZero, 0) : e == 2047 ? make_int2(kExpNaN, 0) : make_int2(e - 1022 + s, (int)s_mx[line]);
    }
}

// ---------------------------------------------------------------- forward z pass
// Lines of H2 (the three components of N), or (ADJ) of H3: A, R, Z of one component, of which
// ubar += A - i k k_z Z and Rhat = R.  NL = 3 lines per block, or one: then line l0 of each
// component (ADJ), or each component in its own block.
struct ZfwdOut {
    double2* out;    // N, or ubar
    double2* Rh;     // Rhat of the staged rows
    const longlong2* s2;   // of N: sums of N_t over the theta blocks
    double scale;    // of N
    double kz;
    int l0;
};

template <class PL, int NL, bool ADJ>
__global__ void __launch_bounds__(kZThreads) k_fx_zfwd(const cx* __restrict__ H2, ZfwdOut w, const int* __restrict__ e2,
                                                       const int* __restrict__ e2max, int N, int M, int K, int r0, int nh, int zt,
                                                       unsigned mzt, FxPlan f, const int4* __restrict__ tw, int tl, unsigned mtl) {
    extern __shared__ cx buf[];
    __shared__ unsigned s_l1[NL];
    __shared__ double s_mean;
    const PL pl(f);
    constexpr int NE = ADJ ? 6 : 2;
    const int P = pl.size(), lp = line_pitch(P), nk = 2 * K + 1, nmode = (M + 1) * nk;
    int t = blockIdx.x;
    constexpr int NB = ADJ ? 3 : 3 / NL;   // blocks per (r, m)
    const int b = t % NB;
    t /= NB;
    const int m = t % (M + 1), rl = t / (M + 1);
    if (threadIdx.x < NL) s_l1[threadIdx.x] = 0;
    __syncthreads();
    const int line = NL == 1 ? 0 : udiv(threadIdx.x, mtl), i0 = threadIdx.x - line * tl;
    const bool on = line < NL;
    // component and kind (A, R, Z) of this thread's line, its field and exponent
    const int c = ADJ ? b : b * NL + line, l = ADJ ? (NL == 1 ? w.l0 : line) : 0;
    // the - component of m = 0 is the mirrored conjugate of the + one: taken from the same line, so that
    // it is that exactly
    const bool mirror = m == 0 && c == 1;
    const int field = 3 * l + (mirror ? 0 : c), ie = 2 * l + (c == 2);
    const int E = on ? e2max[rl * NE + ie] : 0;
    cx v[8];
    unsigned l1 = 0;
    if (on) {
        const cx* h = H2 + (((size_t)field * nh + rl) * (M + 1) + m) * P;
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = i0 + i * tl < P ? h[i0 + i * tl] : mk(0, 0);
    }
    if (!ADJ && m == 0 && threadIdx.x < 32) {
        // (0, 0): N_t from the sums over the theta blocks, while the line comes in
        double y = 0.0;
        for (int i = threadIdx.x; i < P / zt; i += 32) y += block_sum(__ldg(&w.s2[rl * (P / zt) + i]));
        for (int o = 16; o; o >>= 1)
            if (o < P / zt) y += __shfl_xor_sync(0xffffffffu, y, o);
        if (threadIdx.x == 0) s_mean = y;
    }
    if (on) {
        const int* er = e2 + (size_t)rl * (P / zt) * NE + ie;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i0 + i * tl < P) {
                const int te = E - __ldg(&er[udiv(i0 + i * tl, mzt) * NE]);
                v[i] = mk(shr(v[i].x, te), shr(v[i].y, te));
                l1 += ((mag_hi(v[i].x) + mag_hi(v[i].y)) >> 11) + 1;
            }
    }
    line_reduce<NL, false>(s_l1, line, l1, tl);
    __syncthreads();
    if (on) {
        const int s = max(0, bits(s_l1[line]) - 19);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i0 + i * tl < P) buf[line * lp + i0 + i * tl] = mk(v[i].y >> s, v[i].x >> s);   // exchanged
    }
    __syncthreads();
    transform(pl, buf, lp, NL, tw, false);
    // line q's value of mode k (index kk = k + K), from its own exponent
    auto value = [&](int q, int kk, int Eq) {
        const cx o = buf[q * lp + pd(kk >= K ? kk - K : kk - K + P)];
        const int s = Eq + max(0, bits(s_l1[q]) - 19) - 62;
        return Eq > kExpNaN / 2 ? make_double2(nan64(), nan64()) : make_double2(to_double(o.y, s), to_double(o.x, s));
    };
    const size_t e0 = ((size_t)c * N + r0 + rl) * nmode + (size_t)m * nk, h0 = ((size_t)c * nh + rl) * nmode + (size_t)m * nk;
    if (!ADJ) {
        if (!on) return;
        if (m == 0) {   // of a real field: k < 0 is the conjugate of k > 0
            for (int kk = i0; kk < nk; kk += tl) {
                const bool flip = c == 1 || (c == 2 && kk < K);
                double2 o = value(line, flip ? 2 * K - kk : kk, E);
                if (flip) o.y = -o.y;
                if (c < 2 && kk == K) o.y = c == 0 ? s_mean : -s_mean;
                w.out[e0 + kk] = make_double2(o.x * w.scale, o.y * w.scale);
            }
            return;
        }
        for (int kk = i0; kk < nk; kk += tl) {
            const double2 o = value(line, kk, E);
            w.out[e0 + kk] = make_double2(o.x * w.scale, o.y * w.scale);
        }
        return;
    }
    const int* em = e2max + rl * NE + (c == 2);
    auto coeff = [&](int q, int kk, int Eq) {   // with m = 0 of real fields as above (c is the block's)
        const bool flip = m == 0 && (c == 1 || (c == 2 && kk < K));
        double2 o = value(q, flip ? 2 * K - kk : kk, Eq);
        if (flip) o.y = -o.y;
        return o;
    };
    for (int kk = threadIdx.x; kk < nk; kk += blockDim.x) {
        const double kzk = w.kz * (kk - K);
        if (NL == 3 || w.l0 != 1) {
            double2 u = w.out[e0 + kk];
            if (NL == 3 || w.l0 == 0) {
                const double2 A = coeff(0, kk, em[0]);
                u.x += A.x;
                u.y += A.y;
            }
            if (NL == 3 || w.l0 == 2) {
                const double2 Z = coeff(NL == 3 ? 2 : 0, kk, em[4]);
                u.x += kzk * Z.y;
                u.y -= kzk * Z.x;
            }
            w.out[e0 + kk] = u;
        }
        if (NL == 3 || w.l0 == 1) w.Rh[h0 + kk] = coeff(NL == 3 ? 1 : 0, kk, em[2]);
    }
}

// bytes of e1, e2max and e2 of so many rows, up to the 16-byte boundary of s2
size_t fx_s2_offset(const tc_plan* p, int rows) {
    return ((size_t)rows * ((size_t)9 * (p->M + 1) * sizeof(int2) + 2 * sizeof(int) + (size_t)2 * p->P_z * sizeof(int)) + 15) & ~(size_t)15;
}

Exps exps(tc_plan* p, char* ws) {
    Exps e;
    e.e1 = reinterpret_cast<int2*>(ws + p->ws.fxe);
    e.e2max = reinterpret_cast<int*>(e.e1 + (size_t)9 * p->stage_rows * (p->M + 1));
    e.e2 = e.e2max + 2 * p->stage_rows;
    e.s2 = reinterpret_cast<longlong2*>(reinterpret_cast<char*>(e.e1) + fx_s2_offset(p, p->stage_rows));
    return e;
}

}  // namespace

size_t fx_exp_bytes(const tc_plan* p, int rows) {
    return fx_s2_offset(p, rows) + (size_t)rows * p->P_z * sizeof(longlong2);
}

namespace {

// What a z pass does: the inverse one of u (or of Nbar), the forward one into N (or into ubar
// and Rhat).
struct ZPass {
    bool inverse, adj;
    const double2* in;    // u or Nbar
    const double2* du;    // d_r u (nullptr: taken by the pass)
    cx* H;                // lines written or read
    int2* e1;             // exponents of the lines of an inverse pass
    int* e2max;
    const int* e2;
    ZfwdOut out;
    int r0, nh, zt;
};

// Launch shapes: as many of the lines of an (r, m) per block as give it about 128 threads at
// n / 8 each (L9 of nine, L3 of three).
template <class PL, int L9, int L3>
tc_status z_pass(tc_plan* p, const ZPass& a, const int4* tw, cudaStream_t s) {
    // at least a thread for 8 entries of a line; 4 in the short ones, where latency counts
    const int P = p->P_z, nl = a.inverse && !a.adj ? L9 : L3, thr = round32(nl * (P <= 48 ? (P + 3) / 4 : (P + 7) / 8)), tl = thr / nl;
    const size_t sm = (size_t)nl * line_pitch(P) * sizeof(cx);
    const int rm = a.nh * (p->M + 1);
    const double scale = 1.0 / ((double)p->P_t * (double)P);
    auto inv = [&](auto k, int lines) -> tc_status {
        TC_CUDA(p, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        k<<<rm * (lines / nl), thr, sm, s>>>(a.in, a.du, a.H, a.e1, p->N_r, p->M, p->K, a.adj ? scale : p->k_z, a.r0, a.nh, p->fx_z, tw, tl,
                                             magic(tl), a.e2max, p->d_w1, p->d_col0);
        TC_LAUNCHED(p, "k_fx_zinv");
        return TC_OK;
    };
    auto fwd = [&](auto k, int blocks, int l0) -> tc_status {
        ZfwdOut o = a.out;
        o.scale = scale;
        o.kz = p->k_z;
        o.l0 = l0;
        TC_CUDA(p, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        k<<<rm * blocks, thr, sm, s>>>(a.H, o, a.e2, a.e2max, p->N_r, p->M, p->K, a.r0, a.nh, a.zt, magic(a.zt), p->fx_z, tw, tl, magic(tl));
        TC_LAUNCHED(p, "k_fx_zfwd");
        return TC_OK;
    };
    if (a.inverse) return a.adj ? inv(k_fx_zinv<PL, L3, true>, 3) : inv(k_fx_zinv<PL, L9, false>, 9);
    if (!a.adj) return fwd(k_fx_zfwd<PL, L3, false>, 3 / L3, 0);
    if (L3 == 3) return fwd(k_fx_zfwd<PL, L3, true>, 3, 0);
    for (int l = 0; l < 3; ++l) TC_TRY_STATUS(fwd(k_fx_zfwd<PL, L3, true>, 3, l));
    return TC_OK;
}

tc_status run_z(tc_plan* p, const ZPass& a, cudaStream_t s);

// lengths with a compile-time plan
bool static_z(int P) {
    switch (P) {
        case 12: case 24: case 36: case 48: case 72: case 96: case 144: case 192: case 288: case 384: case 576: case 768: case 1152:
        case 1536: case 2304: return true;
    }
    return false;
}
}  // namespace

const int* fx_static_radices(int n) {
    switch (n) {
#define TC_FX_R(P) case P: return Radix<P>::r;
        TC_FX_R(12) TC_FX_R(24) TC_FX_R(36) TC_FX_R(48) TC_FX_R(72) TC_FX_R(96) TC_FX_R(144) TC_FX_R(192) TC_FX_R(288) TC_FX_R(384) TC_FX_R(576)
        TC_FX_R(768) TC_FX_R(1152) TC_FX_R(1536) TC_FX_R(2304)
#undef TC_FX_R
    }
    return nullptr;
}

namespace {

tc_status run_z(tc_plan* p, const ZPass& a, cudaStream_t s) {
    const bool st = p->theta_zt_forced == 0 && static_z(p->P_z) && 3 * p->K <= p->P_z;
    const int4* tw = p->d_fx_tw_z + (st ? p->fx_z.table : 0);
    switch (st ? p->P_z : 0) {
#define TC_FX_Z(P, A, B) case P: return z_pass<Ct<P>, A, B>(p, a, tw, s);
        TC_FX_Z(12, 9, 3) TC_FX_Z(24, 9, 3) TC_FX_Z(36, 9, 3) TC_FX_Z(48, 9, 3) TC_FX_Z(72, 9, 3) TC_FX_Z(96, 9, 3) TC_FX_Z(144, 3, 3)
        TC_FX_Z(192, 3, 3) TC_FX_Z(288, 3, 3) TC_FX_Z(384, 3, 3) TC_FX_Z(576, 3, 3) TC_FX_Z(768, 3, 3) TC_FX_Z(1152, 1, 1)
        TC_FX_Z(1536, 1, 1) TC_FX_Z(2304, 1, 1)
#undef TC_FX_Z
    }
    if (p->P_z <= 96) return z_pass<Rt, 9, 3>(p, a, tw, s);
    if (p->P_z <= 768) return z_pass<Rt, 3, 3>(p, a, tw, s);
    return z_pass<Rt, 1, 1>(p, a, tw, s);
}

// inverse z pass of u with its derivatives, rows r0 .. r0 + nh - 1; du: scratch of 3 nh (M+1)(2K+1)
tc_status zinv_u(tc_plan* p, const double2* u, double2* du, cx* H1, const Exps& e, cudaStream_t s, int r0, int nh) {
    const int slot = prof_begin(p, kKZinv, s);
    if (p->P_z <= 96 && p->S <= 65536) {
        // small problems: the inverse z pass takes d_r u itself, in FP64.  Its 18 FMAs per value
        // then cost less than a launch (S = 5000: 0.4 us of the FP64 pipe against 7 us).
        du = nullptr;
    } else {
        k_fx_dr<<<dim3((2 * p->nmode + 127) / 128, (r0 + nh + kDrRows - 1) / kDrRows - r0 / kDrRows, 3), 128, 0, s>>>(
            reinterpret_cast<const double*>(u), reinterpret_cast<double*>(du), p->d_fx_w1, p->d_fx_ew, p->d_w1, p->d_col0, p->N_r,
            2 * p->nmode, r0, nh);
        TC_LAUNCHED(p, "k_fx_dr");
    }
    TC_TRY_STATUS(run_z(p, ZPass{true, false, u, du, H1, e.e1, e.e2max, nullptr, {}, r0, nh, 1}, s));
    prof_end(p, slot, s);
    return TC_OK;
}

// The transforms of rows r0 .. r0 + nh - 1.
tc_status fx_rows(tc_plan* p, const double2* u, double2* Nh, char* ws, cudaStream_t s, int r0, int nh) {
    cx* H1 = reinterpret_cast<cx*>(ws + p->ws.H1);
    cx* H2 = reinterpret_cast<cx*>(ws + p->ws.H2);
    const Exps e = exps(p, ws);
    TC_TRY_STATUS(zinv_u(p, u, reinterpret_cast<double2*>(H2), H1, e, s, r0, nh));
    int slot = prof_begin(p, kKTheta, s);
    ThetaArgs a{H1, H2, e.e1, e.e2, e.e2max, e.s2, p->d_fx_ir, p->d_fx_mm, p->d_fx_tw_t, r0, nh, p->M, p->P_z, p->fx_zt, p->fx_emm,
                magic(p->fx_zt), magic(p->P_t), (long long)p->m_p};
    TC_TRY_STATUS(launch_fx_theta(p, a, s));
    prof_end(p, slot, s);
    slot = prof_begin(p, kKZfwd, s);
    TC_TRY_STATUS(run_z(p, ZPass{false, false, nullptr, nullptr, H2, nullptr, e.e2max, e.e2, {Nh, nullptr, e.s2, 0, 0, 0}, r0, nh, p->fx_zt}, s));
    prof_end(p, slot, s);
    return TC_OK;
}

}  // namespace

// exponents of the transposed term's lines: e1a[3][stage_rows][M+1], e2max[stage_rows][6], e2[stage_rows][P_z][6]
size_t fx_adj_exp_bytes(const tc_plan* p) {
    return (size_t)p->stage_rows * ((size_t)3 * (p->M + 1) * sizeof(int2) + 6 * sizeof(int) + (size_t)6 * p->P_z * sizeof(int));
}

// ubar += (the transposed transforms and products of Nbar about u), rows r0 .. r0 + nh - 1, but
// for the radial stencil: Rhat takes the part that k_drT brings in
tc_status launch_adjoint_rows_fx(tc_plan* p, const double2* u, const double2* Nbar, double2* ubar, double2* Rh, char* ws, cudaStream_t s,
                                 int r0, int nh) {
    cx* H1 = reinterpret_cast<cx*>(ws + p->ws.H1a);
    cx* Ha = reinterpret_cast<cx*>(ws + p->ws.Ha);
    cx* H3 = reinterpret_cast<cx*>(ws + p->ws.H3);
    const Exps e = exps(p, ws);
    int2* e1a = reinterpret_cast<int2*>(ws + p->ws.fxa);
    int* e2max = reinterpret_cast<int*>(e1a + (size_t)3 * p->stage_rows * (p->M + 1));
    int* e2 = e2max + (size_t)6 * p->stage_rows;
    TC_TRY_STATUS(zinv_u(p, u, Rh, H1, e, s, r0, nh));   // Rhat is free until the forward z pass
    int slot = prof_begin(p, kKZinvAdj, s);
    TC_TRY_STATUS(run_z(p, ZPass{true, true, Nbar, nullptr, Ha, e1a, e2max, nullptr, {}, r0, nh, 1}, s));
    prof_end(p, slot, s);
    slot = prof_begin(p, kKThetaAdj, s);
    const int zt = fx_zt_adj(p, p->theta_zt_forced);
    ThetaAdjArgs a{H1, Ha, H3, e.e1, e1a, e2, e2max, p->d_fx_ir, p->d_fx_mm, p->d_fx_tw_t, r0, nh, p->M, p->P_z, zt, p->fx_emm,
                   magic(zt), magic(p->P_t), (long long)p->m_p};
    TC_TRY_STATUS(launch_fx_theta_adj(p, a, s));
    prof_end(p, slot, s);
    slot = prof_begin(p, kKZfwdAdj, s);
    TC_TRY_STATUS(run_z(p, ZPass{false, true, nullptr, nullptr, H3, nullptr, e2max, e2, {ubar, Rh, nullptr, 0, 0, 0}, r0, nh, zt}, s));
    prof_end(p, slot, s);
    return TC_OK;
}

// N(u) in FP64, slab by slab of p->stage_rows radial rows (a row's transforms read no other
// row's staging)
tc_status launch_nonlinear_fx(tc_plan* p, const double2* u, double2* Nh, char* ws, cudaStream_t s) {
    for (int r0 = 0; r0 < p->N_r; r0 += p->stage_rows)
        TC_TRY_STATUS(fx_rows(p, u, Nh, ws, s, r0, std::min(p->stage_rows, p->N_r - r0)));
    return TC_OK;
}

}  // namespace tc
