// Theta pass of the transposed nonlinear term in 64-bit fixed point (tc_fx.cuh, tc_fx_z.cu).
//
// Per (r, z tile), two lines per z resident at a time.  Inverse phases (kinds L0; L1):
//   0: (s_r, s_t); (u_r, u_t)                    1: s_z, two z per line; (u_z, d_r u_z)
//   2: (d_r u_r, d_r u_t); (d_t u_r, d_t u_t)    3: (d_z u_r, d_z u_t); (d_t u_z, d_z u_z)
// with n the physical fields of s.  Per physical point (n_r, n_t), (u_r, u_t / r), n_z, u_z and
// the products that need the gradient lines stay in shared memory:
//   b_r = n_r d_r u_r + n_t (d_r u_t + u_t / r) + n_z d_r u_z,
//   r b_t = n_r (d_t u_r - 2 u_t) + n_t (d_t u_t + u_r) + n_z d_t u_z,
//   b_z = n_r d_z u_r + n_t d_z u_t + n_z d_z u_z.
// Forward phases transform six pairs, two per z, grouped so that each group alone fixes the H3
// fields it writes: (d_r u_r, d_r u_t), (d_z u_r, d_z u_t) -> R_+-, Z_+-; (u_r, u_t), (d_t u_r,
// d_t u_t) -> A_+-; (u_z, d_r u_z), (d_t u_z, d_z u_z) -> A_z, R_z, Z_z.  A has -i m m_p of the
// d_t part folded in.  As FP64 arithmetic this pass kept the FP64 pipe 86% busy (1.25 ms at
// N_r = 96, M = 32, K = 64).
#include "tc_fx_nl.cuh"

namespace tc {

using namespace fx;

namespace {

// per point: Nv, Uu, Ac (two parts each), Nz, Uz, Bz
constexpr int kAdjPoint = 9 * (int)sizeof(long long);

template <class PL, int ZT, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_fx_theta_adj(ThetaAdjArgs a, FxPlan f) {
    extern __shared__ cx buf[];
    __shared__ int s_E[11];
    __shared__ float s_bound[NT / 32][11];
    __shared__ unsigned s_mx[4][4];
    __shared__ unsigned long long s_sum[NT / 32][4];
    const PL pl(f);
    const int P = pl.size(), M = a.M, Pz = a.Pz, zt = ZT ? ZT : a.zt, lp = line_pitch(P), nl = 2 * zt, npt = zt * P;
    const int nt = PL::kStatic ? NT : (int)blockDim.x, nw = nt / 32, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto divz = [&](int i) { return ZT ? i / (ZT ? ZT : 1) : udiv(i, a.mzt); };
    auto divp = [&](int i) { return PL::kStatic ? i / P : udiv(i, a.mP); };
    cx* Nv = buf + nl * lp;
    cx* Uu = Nv + npt;
    cx* Ac = Uu + npt;
    long long* Nz = reinterpret_cast<long long*>(Ac + npt);
    long long* Uz = Nz + npt;
    long long* Bz = Uz + npt;
    const int tiles = Pz / zt;
    const int r = blockIdx.x / tiles, tile = blockIdx.x - r * tiles, z0 = tile * zt;
    const size_t fs = (size_t)a.nh * (M + 1) * Pz, es = (size_t)a.nh * (M + 1);
    const cx* h = a.H1 + (size_t)r * (M + 1) * Pz + z0;
    const cx* ha = a.Ha + (size_t)r * (M + 1) * Pz + z0;
    const int2* eh = a.e1 + (size_t)r * (M + 1);
    const int2* ea = a.e1a + (size_t)r * (M + 1);
    // line kinds 0 .. 7 as in the forward pass; 8 s_r, 9 s_t, 10 s_z
    auto bound = [&](auto f) {
        f(0, 0, false); f(0, 1, false); f(1, 2, false); f(2, 5, false); f(3, 3, false); f(3, 4, false);
        f(4, 0, true); f(4, 1, true); f(5, 6, false); f(5, 7, false); f(6, 2, true); f(7, 8, false);
        f(8, 9, false); f(9, 10, false); f(10, 11, false);
    };
    constexpr unsigned half = 0x7c6u;
    int er[11];
    float sum[11];
    line_bounds<12, 11, NT>([&](int q, int m) { return q < 9 ? __ldg(&eh[q * es + m]) : __ldg(&ea[(q - 9) * es + m]); }, bound, half, M,
                            a.mp, nt, s_E, s_bound, er, sum);
    if (threadIdx.x < 16) s_mx[threadIdx.x >> 2][threadIdx.x & 3] = 0;
    auto kind = [&](int s) { return kind_exponent(er[s], sum[s], s == 4 || s == 6, (half >> s) & 1, a.emm); };
    const int E0 = kind(0), E1x = kind(1), E1y = kind(2), E2 = kind(3), E3 = kind(4), E4 = kind(5), E5x = kind(6), E5y = kind(7);
    const int Esr = kind(8), Est = kind(9), Esz = kind(10);
    if (max(max(max(max(E0, E1x), max(E1y, E2)), max(max(E3, E4), max(E5x, E5y))), max(Esr, max(Est, Esz))) > kExpNaN / 2) {
        if (threadIdx.x < 6) {
            a.e2[(r * tiles + tile) * 6 + threadIdx.x] = kExpNaN;
            atomicMax(&a.e2max[r * 6 + threadIdx.x], kExpNaN);
        }
        return;
    }
    const int4 irv = a.ir[a.r0 + r];
    const lim ir = {irv.x, irv.y};
    const int eir = irv.z;
    int Enr = 0, Ent = 0, Enz = 0, Eu = 0, Eut = 0, Euz = 0, Ebr = 0, Ebt = 0, Ebz = 0;

    // ---- inverse phases
    auto fill = [&](auto phc) {
        constexpr int PH = decltype(phc)::value;
        for (int i = threadIdx.x; i < zt * (M + 1); i += nt) {
            const int m = divz(i), z = i - m * zt;
            const size_t o = (size_t)m * Pz + z;
            cx *l0 = buf + z * lp, *l1 = buf + (zt + z) * lp;
            auto H = [&](int q) { return h[q * fs + o]; };
            auto e = [&](int q) { return eh[q * es + m].x; };
            if (PH == 0) {
                put_real2(l0, P, m, shr2(ha[o], Esr - ea[m].x), shr2(ha[fs + o], Est - ea[es + m].x));
                put_pair(l1, P, m, shr2(H(0), E0 - e(0)), shr2(H(1), E0 - e(1)));
            } else if (PH == 1) {
                // line z / 2 takes s_z of z (even) and z + 1 as its two real fields
                if ((z & 1) == 0) {
                    const int t = Esz - ea[2 * es + m].x;
                    const cx y = z + 1 < zt ? ha[2 * fs + o + 1] : mk(0, 0);
                    put_real2(buf + (z / 2) * lp, P, m, shr2(ha[2 * fs + o], t), shr2(y, t));
                }
                put_real2(l1, P, m, shr2(H(2), E1x - e(2)), shr2(H(5), E1y - e(5)));
            } else if (PH == 2) {
                put_pair(l0, P, m, shr2(H(3), E2 - e(3)), shr2(H(4), E2 - e(4)));
                put_pair(l1, P, m, imul(H(0), a.mm[m], a.emm, E3, e(0)), imul(H(1), a.mm[m], a.emm, E3, e(1)));
            } else {
                put_pair(l0, P, m, shr2(H(6), E4 - e(6)), shr2(H(7), E4 - e(7)));
                put_real2(l1, P, m, imul(H(2), a.mm[m], a.emm, E5x, e(2)), shr2(H(8), E5y - e(8)));
            }
        }
        if (PH == 1 && (zt + 1) / 2 < zt) {   // lines of phase 1 that hold nothing
            for (int i = threadIdx.x; i < (zt - (zt + 1) / 2) * lp; i += nt) buf[(zt + 1) / 2 * lp + i] = mk(0, 0);
        }
    };
    auto products = [&](auto phc) {
        constexpr int PH = decltype(phc)::value;
        const int n0x = 30 - bits(s_mx[PH][0]), n0y = 30 - bits(s_mx[PH][1]), n1x = 30 - bits(s_mx[PH][2]), n1y = 30 - bits(s_mx[PH][3]);
        const int nz = PH == 1 ? min(n0x, n0y) : 0;
        Sum sa, sb, sc;
        if (PH == 0) {
            Enr = Esr - n0x;
            Ent = Est - n0y;
            Eu = E0 - n1x;
            const int et = E0 - n1y;
            Eut = et + eir;
            Ebr = Ent + Eut + 2;
            Ebt = kExpZero * 8;   // nothing yet
            sb.set(Ebt, Ent + Eu, Enr + et + 1);
        } else if (PH == 1) {
            Enz = Esz - nz;
            Euz = E1x - n1x;
            sa.set(Ebr, Enz + E1y - n1y, Enz + E1y - n1y);
        } else if (PH == 2) {
            sa.set(Ebr, Enr + E2 - n0x, Ent + E2 - n0y);
            sb.set(Ebt, Enr + E3 - n1x, Ent + E3 - n1y);
        } else {
            Ebz = kExpZero * 8;
            sa.set(Ebz, Enr + E4 - n0x, Ent + E4 - n0y);
            sc.set(Ebz, Enz + E5y - n1y, Enz + E5y - n1y);
            sb.set(Ebt, Enz + E5x - n1x, Enz + E5x - n1x);
        }
#pragma unroll 1
        for (int pt = threadIdx.x; pt < npt; pt += nt) {
            const int z = divp(pt), i = pd(pt - z * P);
            const cx p = buf[(PH == 1 ? z / 2 : z) * lp + i], q = buf[(zt + z) * lp + i];
            const long long qx = shl(q.x, n1x), qy = shl(q.y, n1y);
            const lim qxl = split(qx), qyl = split(qy);
            if (PH == 0) {
                const long long nr = shl(p.x, n0x), ntv = shl(p.y, n0y), utr = mulq(qyl, ir);
                const lim nrl = split(nr), ntl = split(ntv);
                Nv[pt] = mk(nr, ntv);
                Uu[pt] = mk(qx, utr);
                Ac[pt] = mk(mulhi(ntl, split(utr), 0, kHalf32), sb.first(ntl, qxl) - sb.second(nrl, qyl));
            } else if (PH == 1) {
                const long long n = shl(z & 1 ? p.y : p.x, nz);
                Nz[pt] = n;
                Uz[pt] = qx;
                Ac[pt].x = sa.old(Ac[pt].x) + sa.first(split(n), qyl);
            } else {
                const cx n = Nv[pt];
                const lim nrl = split(n.x), ntl = split(n.y), px = split(shl(p.x, n0x)), py = split(shl(p.y, n0y));
                if (PH == 2) {
                    const cx c = Ac[pt];
                    Ac[pt] = mk(sa.old(c.x) + sa.first(nrl, px) + sa.second(ntl, py), sb.old(c.y) + sb.first(nrl, qxl) + sb.second(ntl, qyl));
                } else {
                    const lim nzl = split(Nz[pt]);
                    Bz[pt] = sc.old(sa.first(nrl, px) + sa.second(ntl, py)) + sc.first(nzl, qyl);
                    Ac[pt].y = sb.old(Ac[pt].y) + sb.first(nzl, qxl);
                }
            }
        }
    };

    // ---- forward phases: values of the two lines of a z, exchanged parts as the transform wants
    // them; exponents e[0..3] of (L0.x, L0.y, L1.x, L1.y)
    int e[4] = {0, 0, 0, 0};
    InShift in;
    auto fill_forward = [&](auto fpc) {
        constexpr int FP = decltype(fpc)::value;
        if (FP == 0) {
            e[0] = Eu + Enr + 2; e[1] = Eu + Ent + 2; e[2] = Euz + Enr + 2; e[3] = Euz + Ent + 2;
        } else if (FP == 1) {
            e[0] = Ebr; e[1] = Ebt + eir; e[2] = Eut + Enr + 2; e[3] = Eut + Ent + 2;
        } else {
            e[0] = Ebz; e[1] = Eu + Enz + 2; e[2] = Eut + Enz + 2; e[3] = Euz + Enz + 2;
        }
        unsigned long long s[4] = {0, 0, 0, 0};
#pragma unroll 1
        for (int pt = threadIdx.x; pt < npt; pt += nt) {
            const int z = divp(pt), i = pt - z * P;
            cx A, B;
            auto mul = [](lim x, lim y) { return mulhi(x, y, 0, kHalf32); };
            if (FP == 2) {
                const lim nzl = split(Nz[pt]);
                const cx uu = Uu[pt];
                A = mk(Bz[pt], mul(split(uu.x), nzl));
                B = mk(mul(split(uu.y), nzl), mul(split(Uz[pt]), nzl));
            } else {
                const cx n = Nv[pt], uu = Uu[pt];
                const lim nrl = split(n.x), ntl = split(n.y);
                if (FP == 0) {
                    const lim ur = split(uu.x), uz = split(Uz[pt]);
                    A = mk(mul(ur, nrl), mul(ur, ntl));
                    B = mk(mul(uz, nrl), mul(uz, ntl));
                } else {
                    const cx c = Ac[pt];
                    const lim ut = split(uu.y);
                    A = mk(c.x, mulq(c.y, ir));
                    B = mk(mul(ut, nrl), mul(ut, ntl));
                }
            }
            s[0] += ((unsigned long long)llabs(A.x) >> 12) + 1;
            s[1] += ((unsigned long long)llabs(A.y) >> 12) + 1;
            s[2] += ((unsigned long long)llabs(B.x) >> 12) + 1;
            s[3] += ((unsigned long long)llabs(B.y) >> 12) + 1;
            buf[z * lp + i] = mk(A.y, A.x);
            buf[(zt + z) * lp + i] = mk(B.y, B.x);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int o = 16; o; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) s_sum[wid][q] = s[q];
        }
    };
    // exponents of the group's lines and the shifts into them: each part's sum below 2^59
    auto forward_shifts = [&](int fp) {
        int b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            unsigned long long t = 0;
            for (int w = 0; w < nw; ++w) t += s_sum[w][q];
            b[q] = e[q] + max(0, bits64(t) + 12 - 59);   // exponent this part needs
        }
        // the two parts of a pair of components (r, t) share theirs
        if (fp < 2) {
            b[0] = b[1] = max(b[0], b[1]);
            b[2] = b[3] = max(b[2], b[3]);
        }
        in.on = true;
        in.y0 = b[0] - e[0]; in.x0 = b[1] - e[1]; in.y1 = b[2] - e[2]; in.x1 = b[3] - e[3];   // exchanged
#pragma unroll
        for (int q = 0; q < 4; ++q) e[q] = b[q];
    };
    // output fields of a group: exponents go to e2 in the order A_+-, A_z, R_+-, R_z, Z_+-, Z_z
    auto write_e = [&](int i, int E) {
        a.e2[(r * tiles + tile) * 6 + i] = E;
        atomicMax(&a.e2max[r * 6 + i], E);
    };
    auto store = [&](auto fpc) {
        constexpr int FP = decltype(fpc)::value;
        const int EA = FP == 1 ? max(e[0], e[2] + a.emm) + 1 : FP == 2 ? max(e[0], e[2] + a.emm) + 1 : 0;
        if (threadIdx.x == 0) {
            if (FP == 0) { write_e(2, e[0]); write_e(4, e[2]); }
            else if (FP == 1) write_e(0, EA);
            else { write_e(1, EA); write_e(3, e[1]); write_e(5, e[3]); }
        }
        for (int i = threadIdx.x; i < zt * (M + 1); i += nt) {
            const int m = divz(i), z = i - m * zt, ip = pd(m), in_ = pd(m ? P - m : 0);
            // spectra of the two real parts of each line, times c_m = 2 (1 at m = 0)
            cx X[2], Y[2];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                const cx* L = buf + (l * zt + z) * lp;
                const cx c = mk(L[ip].y, L[ip].x), d = mk(L[in_].y, -L[in_].x);
                X[l] = m ? add(c, d) : mk(c.x, 0);
                Y[l] = m ? mk(c.y - d.y, d.x - c.x) : mk(c.y, 0);
            }
            const size_t o = ((size_t)r * (M + 1) + m) * Pz + z0 + z;
            auto plus = [](cx p, cx q) { return mk((p.x - q.y) >> 1, (p.y + q.x) >> 1); };
            auto minus = [](cx p, cx q) { return mk((p.x + q.y) >> 1, (p.y - q.x) >> 1); };
            auto less = [&](cx p, int ep, cx q, int eq) { return sub(shr2(p, EA - ep), imul(q, a.mm[m], a.emm, EA, eq)); };
            if (FP == 0) {
                a.H3[3 * fs + o] = plus(X[0], Y[0]);
                a.H3[4 * fs + o] = minus(X[0], Y[0]);
                a.H3[6 * fs + o] = plus(X[1], Y[1]);
                a.H3[7 * fs + o] = minus(X[1], Y[1]);
            } else if (FP == 1) {
                const cx Ar = less(X[0], e[0], X[1], e[2]), At = less(Y[0], e[0], Y[1], e[2]);
                a.H3[o] = plus(Ar, At);
                a.H3[fs + o] = minus(Ar, At);
            } else {
                a.H3[2 * fs + o] = less(X[0], e[0], X[1], e[2]);
                a.H3[5 * fs + o] = Y[0];
                a.H3[8 * fs + o] = Y[1];
            }
        }
    };
    auto each = [&](int i, auto fn) {
        if (i == 0) fn(std::integral_constant<int, 0>{});
        else if (i == 1) fn(std::integral_constant<int, 1>{});
        else if (i == 2) fn(std::integral_constant<int, 2>{});
        else fn(std::integral_constant<int, 3>{});
    };
#pragma unroll 1
    for (int ph = 0; ph < 7; ++ph) {
        if (ph < 4) {
            each(ph, fill);
            zero_band(pl, buf, lp, nl, M + 1, P - M);
        } else {
            if (ph == 4) fill_forward(std::integral_constant<int, 0>{});
            else if (ph == 5) fill_forward(std::integral_constant<int, 1>{});
            else fill_forward(std::integral_constant<int, 2>{});
        }
        __syncthreads();
        if (ph >= 4) forward_shifts(ph - 4);
        uint4 mx = transform(pl, buf, lp, nl, a.tw, ph < 4, ph < 4, zt, in);
        if (ph < 4) {
            mx.x = __reduce_max_sync(0xffffffffu, mx.x);
            mx.y = __reduce_max_sync(0xffffffffu, mx.y);
            mx.z = __reduce_max_sync(0xffffffffu, mx.z);
            mx.w = __reduce_max_sync(0xffffffffu, mx.w);
            if (lane < 4) atomicMax(&s_mx[ph][lane], lane == 0 ? mx.x : lane == 1 ? mx.y : lane == 2 ? mx.z : mx.w);
            __syncthreads();
            each(ph, products);
        } else if (ph == 4) {
            store(std::integral_constant<int, 0>{});
        } else if (ph == 5) {
            store(std::integral_constant<int, 1>{});
        } else {
            store(std::integral_constant<int, 2>{});
        }
        __syncthreads();   // the next fill overwrites the lines
    }
}

template <class PL, int ZT, int NT, int MINB>
tc_status theta_adj_pass(tc_plan* p, const ThetaAdjArgs& a, cudaStream_t s) {
    const size_t sm = (size_t)2 * a.zt * line_pitch(p->P_t) * sizeof(cx) + (size_t)a.zt * p->P_t * kAdjPoint;
    auto k = k_fx_theta_adj<PL, ZT, NT, MINB>;
    TC_CUDA(p, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int thr = PL::kStatic ? NT : round32(2 * a.zt * ((p->P_t + 7) / 8));
    k<<<a.nh * (p->P_z / a.zt), thr, sm, s>>>(a, p->fx_t);
    TC_LAUNCHED(p, "k_fx_theta_adj");
    return TC_OK;
}

// z values of the blocks of the lengths with a compile-time plan (0: none)
int static_zt_adj(int P) {
    switch (P) {
        case 12: case 24: case 36: case 48: case 72: case 96: case 144: return 4;
        case 192: case 288: case 384: return 2;
        case 576: case 768: case 1152: return 1;
    }
    return 0;
}

}  // namespace

// z values per block of the transposed theta pass
int fx_zt_adj(const tc_plan* p, int forced) {
    const int z = static_zt_adj(p->P_t);
    if (forced == 0 && z > 0 && p->P_z % z == 0 && 3 * p->M <= p->P_t) return z;
    auto fits = [&](int t) {
        const size_t sm = (size_t)2 * t * line_pitch(p->P_t) * sizeof(cx) + (size_t)t * p->P_t * kAdjPoint;
        return p->P_z % t == 0 && 2 * t * ((p->P_t + 7) / 8) <= 320 && (t == 1 || sm <= 100 * 1024);
    };
    int zt = forced > 0 ? std::min(forced, 8) : 4;
    while (zt > 1 && !fits(zt)) --zt;
    return zt;
}

tc_status fx::launch_fx_theta_adj(tc_plan* p, ThetaAdjArgs a, cudaStream_t s) {
    const bool st = p->theta_zt_forced == 0 && a.zt == static_zt_adj(p->P_t) && 3 * p->M <= p->P_t;
    if (st) a.tw += p->fx_t.table;
    switch (st ? p->P_t : 0) {
        case 12: return theta_adj_pass<Ct<12>, 4, 32, 12>(p, a, s);
        case 24: return theta_adj_pass<Ct<24>, 4, 32, 16>(p, a, s);
        case 36: return theta_adj_pass<Ct<36>, 4, 64, 8>(p, a, s);
        case 48: return theta_adj_pass<Ct<48>, 4, 64, 8>(p, a, s);
        case 72: return theta_adj_pass<Ct<72>, 4, 96, 6>(p, a, s);
        case 96: return theta_adj_pass<Ct<96>, 4, 96, 5>(p, a, s);
        case 144: return theta_adj_pass<Ct<144>, 4, 160, 3>(p, a, s);
        case 192: return theta_adj_pass<Ct<192>, 2, 96, 5>(p, a, s);
        case 288: return theta_adj_pass<Ct<288>, 2, 160, 3>(p, a, s);
        case 384: return theta_adj_pass<Ct<384>, 2, 192, 2>(p, a, s);
        case 576: return theta_adj_pass<Ct<576>, 1, 160, 3>(p, a, s);
        case 768: return theta_adj_pass<Ct<768>, 1, 192, 2>(p, a, s);
        case 1152: return theta_adj_pass<Ct<1152>, 1, 288, 1>(p, a, s);
    }
    if (2 * a.zt * ((p->P_t + 7) / 8) <= 128) return theta_adj_pass<Rt, 0, 128, 4>(p, a, s);
    return theta_adj_pass<Rt, 0, 320, 2>(p, a, s);
}

}  // namespace tc
