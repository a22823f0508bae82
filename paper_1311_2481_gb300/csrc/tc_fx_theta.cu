// Theta pass and products of the FP64 nonlinear term in 64-bit fixed point (see tc_fx_z.cu for
// the passes along z and the exponents of the lines).
#include "tc_fx_nl.cuh"

namespace tc {

using namespace fx;

namespace {

// H1 fields f = 3 d + c, c in {+, -, z}, d in {u, d_r u, d_z u}.  A block holds zt values of z
// of one r; in each of three phases two lines per z (kinds L0 and L1):
//   phase 0: (u_r, u_t) and (u_z, d_r u_z);  1: (d_r u_r, d_r u_t) and (d_t u_r, d_t u_t);
//   phase 2: (d_z u_r, d_z u_t) and (d_t u_z, d_z u_z).
// Per physical point Ua = (u_r, u_t / r), Ub = (u_z, N_z), Nn = (N_r, N_t) stay in shared
// memory.  After the last pass of a phase the products of its lines are added, a point per thread.
// The sum of N_t over the block goes out beside the lines: its mean drives the mean flow and is
// far smaller than N_r, with which it shares the exponent of a line from there on.

template <class PL, int ZT, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_fx_theta(ThetaArgs a, FxPlan f) {
    extern __shared__ cx buf[];
    __shared__ int s_E[8];               // largest exponents of the line kinds
    __shared__ float s_bound[NT / 32][8];
    __shared__ unsigned s_mx[3][4];   // largest parts of phase, {L0.x, L0.y, L1.x, L1.y}
    __shared__ unsigned long long s_sum[2][NT / 32];
    __shared__ long long s_t[2][NT / 32];   // sum of N_t over a warp, in units of 2^52 and of 1
    const PL pl(f);
    const int P = pl.size(), M = a.M, Pz = a.Pz, zt = ZT ? ZT : a.zt, lp = line_pitch(P), nl = 2 * zt;
    auto divz = [&](int i) { return ZT ? i / (ZT ? ZT : 1) : udiv(i, a.mzt); };
    auto divp = [&](int i) { return PL::kStatic ? i / P : udiv(i, a.mP); };
    cx* Ua = buf + nl * lp;
    cx* Ub = Ua + zt * P;
    cx* Nn = Ub + zt * P;
    const int tiles = Pz / zt;
    const int r = blockIdx.x / tiles, tile = blockIdx.x - r * tiles, z0 = tile * zt;
    const size_t fs = (size_t)a.nh * (M + 1) * Pz;
    const cx* h = a.H1 + (size_t)r * (M + 1) * Pz + z0;
    const size_t es = (size_t)a.nh * (M + 1);
    const int2* eh = a.e1 + (size_t)r * (M + 1);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nt = PL::kStatic ? NT : (int)blockDim.x, nw = nt / 32;
    // Exponents of the line kinds: the sum over m of the lines' largest values bounds every sum of
    // a theta line.  Kinds: 0 (u+-), 1 u_z, 2 d_r u_z, 3 (d_r u+-), 4 m (u+-), 5 (d_z u+-),
    // 6 m u_z, 7 d_z u_z.
    auto bound = [&](auto f) {   // f(kind, field, weighted by m m_p)
        f(0, 0, false); f(0, 1, false); f(1, 2, false); f(2, 5, false); f(3, 3, false); f(3, 4, false);
        f(4, 0, true); f(4, 1, true); f(5, 6, false); f(5, 7, false); f(6, 2, true); f(7, 8, false);
    };
    int er[8];
    float sum[8];
    line_bounds<9, 8, NT>([&](int q, int m) { return __ldg(&eh[q * es + m]); }, bound, 0xc6u, M, a.mp, nt, s_E, s_bound, er, sum);
    if (threadIdx.x < 12) s_mx[threadIdx.x >> 2][threadIdx.x & 3] = 0;   // barriers follow before its use
    auto kind = [&](int s) { return kind_exponent(er[s], sum[s], s == 4 || s == 6, (0xc6u >> s) & 1, a.emm); };
    const int E0 = kind(0), E1x = kind(1), E1y = kind(2), E2 = kind(3), E3 = kind(4), E4 = kind(5), E5x = kind(6), E5y = kind(7);
    if (max(max(max(E0, E1x), max(E1y, E2)), max(max(E3, E4), max(E5x, E5y))) > kExpNaN / 2) {
        if (threadIdx.x < 2) {
            a.e2[(r * tiles + tile) * 2 + threadIdx.x] = kExpNaN;
            atomicMax(&a.e2max[r * 2 + threadIdx.x], kExpNaN);
        }
        if (threadIdx.x == 0) a.s2[r * tiles + tile] = make_longlong2(0, kExpNaN);
        return;
    }
    const int4 irv = a.ir[a.r0 + r];
    const lim ir = {irv.x, irv.y};
    const int eir = irv.z;
    int Eu = 0, Eut = 0, Euz = 0, ENr = 0, ENt = 0, ENz = 0;   // exponents of Ua, Ub.x, Nn, Ub.y

    auto fill = [&](auto ph) {
        constexpr int PH = decltype(ph)::value;
        // spectra of the two lines of each z (lines z and zt + z); z fastest over the threads
        constexpr int fa = 3 * PH;                       // L0: pair (fa, fa + 1)
        const int Ea = PH == 0 ? E0 : PH == 1 ? E2 : E4;
        for (int i = threadIdx.x; i < zt * (M + 1); i += nt) {
            const int m = divz(i), z = i - m * zt;
            const size_t o = (size_t)m * Pz + z;
            constexpr int fx_ = PH == 1 ? 0 : 2, fy_ = PH == 0 ? 5 : PH == 1 ? 1 : 8;
            const cx A = h[fa * fs + o], C = h[(fa + 1) * fs + o], X = h[fx_ * fs + o], Y = h[fy_ * fs + o];
            const int ea = eh[fa * es + m].x, ec = eh[(fa + 1) * es + m].x, ex = eh[fx_ * es + m].x, ey = eh[fy_ * es + m].x;
            put_pair(buf + z * lp, P, m, shr2(A, Ea - ea), shr2(C, Ea - ec));
            cx* l1 = buf + (zt + z) * lp;
            if (PH == 0) put_real2(l1, P, m, shr2(X, E1x - ex), shr2(Y, E1y - ey));
            else if (PH == 1) put_pair(l1, P, m, imul(X, a.mm[m], a.emm, E3, ex), imul(Y, a.mm[m], a.emm, E3, ey));
            else put_real2(l1, P, m, imul(X, a.mm[m], a.emm, E5x, ex), shr2(Y, E5y - ey));
        }
    };
    auto products = [&](auto ph) {
        constexpr int PH = decltype(ph)::value;
        // shifts that bring the largest value of each kind to the top, exponents of the shifted
        // values, and from these the exponents of the products and of the sums: a sum of two
        // gets one bit, of three two bits of headroom
        const int nx = 30 - bits(s_mx[PH][0]), ny = 30 - bits(s_mx[PH][1]), nu = 30 - bits(s_mx[PH][2]), nv = 30 - bits(s_mx[PH][3]);
        const int ex = (PH == 0 ? E0 : PH == 1 ? E2 : E4) - nx, ey = (PH == 0 ? E0 : PH == 1 ? E2 : E4) - ny;
        const int eu = (PH == 0 ? E1x : PH == 1 ? E3 : E5x) - nu, ev = (PH == 0 ? E1y : PH == 1 ? E3 : E5y) - nv;
        Sum sr, st, sz;
        if (PH == 0) {
            Eu = ex;
            Eut = ey + eir;
            Euz = eu;
            ENr = ey + Eut;
            ENt = ex + Eut;
            ENz = ex + ev;
        } else if (PH == 1) {
            sr.set(ENr, Eu + ex, Eut + eu);
            st.set(ENt, Eu + ey, Eut + ev);
        } else {
            sr.set(ENr, Euz + ex, Euz + ex);
            st.set(ENt, Euz + ey, Euz + ey);
            sz.set(ENz, Eut + eu, Euz + ev);
        }
        unsigned long long th = 0, tz = 0;
        long long yh = 0, yl = 0;   // the sum of N_t, exactly: high and low words
        const int EN = max(ENr, ENt), dr = min(EN - ENr, 63), dt = min(EN - ENt, 63);
#pragma unroll 2
        for (int pt = threadIdx.x; pt < zt * P; pt += nt) {
            const int z = divp(pt), i = pd(pt - z * P);
            const cx p = buf[z * lp + i], q = buf[(zt + z) * lp + i];
            const long long pxx = shl(p.x, nx), quu = shl(q.x, nu);
            const lim px = split(pxx), py = split(shl(p.y, ny)), qx = split(quu), qy = split(shl(q.y, nv));
            if (PH == 0) {
                const long long utr = mulq(py, ir);
                const lim tl = split(utr);
                Ua[pt] = mk(pxx, utr);
                Nn[pt] = mk(-mulq(py, tl), mulq(px, tl));   // curvature terms
                Ub[pt] = mk(quu, mulq(px, qy));             // N_z = u_r d_r u_z
            } else if (PH == 1) {
                const cx w = Ua[pt];
                const lim wr = split(w.x), wt = split(w.y);
                const cx n = Nn[pt];
                Nn[pt] = mk(sr.old(n.x) + sr.first(wr, px) + sr.second(wt, qx), st.old(n.y) + st.first(wr, py) + st.second(wt, qy));
            } else {
                const cx b = Ub[pt], n = Nn[pt];
                const lim wz = split(b.x);
                const cx s = mk(sr.old(n.x) + sr.first(wz, px), st.old(n.y) + st.first(wz, py));
                const long long nz = sz.old(b.y) + sz.first(split(Ua[pt].y), qx) + sz.second(wz, qy);
                Nn[pt] = s;
                Ub[pt].y = nz;
                th += (((unsigned long long)llabs(s.x) >> 12) >> dr) + (((unsigned long long)llabs(s.y) >> 12) >> dt) + 2;
                tz += ((unsigned long long)llabs(nz) >> 12) + 1;
                yh += s.y >> 32;
                yl += (unsigned)s.y;
            }
        }
        if (PH == 2) {   // sums of the moduli of N over the block
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                th += __shfl_xor_sync(0xffffffffu, th, o);
                tz += __shfl_xor_sync(0xffffffffu, tz, o);
            }
            // over the warp in three chunks of 26 bits
            const unsigned lo = 0x3ffffffu;
            const long long hi = (yh << 6) + (yl >> 26);
            const unsigned c0 = __reduce_add_sync(0xffffffffu, (unsigned)yl & lo), c1 = __reduce_add_sync(0xffffffffu, (unsigned)hi & lo);
            const int c2 = (int)__reduce_add_sync(0xffffffffu, (unsigned)(hi >> 26));
            if (lane == 0) {
                s_sum[0][wid] = th;
                s_sum[1][wid] = tz;
                s_t[0][wid] = c2;
                s_t[1][wid] = ((long long)c1 << 26) + c0;
            }
        }
    };
    // forward transform: line z holds N_r + i N_t, line zt + z/2 holds N_z of two z values, real
    // and imaginary parts exchanged; both shifted so that the sum of the moduli over the block
    // stays below 2^62
    auto fill_forward = [&]() {
        unsigned long long th = 0, tz = 0;
        long long yh = 0, yl = 0;
        for (int w = 0; w < nw; ++w) {
            th += s_sum[0][w];
            tz += s_sum[1][w];
            yh += s_t[0][w];
            yl += s_t[1][w];
        }
        const int EN = max(ENr, ENt), fh = bits64(th) - 50, fz = bits64(tz) - 50;   // right shift (left if negative)
        const int fr = min(fh + EN - ENr, 62), ft = min(fh + EN - ENt, 62);
        if (threadIdx.x < 2) {
            const int E = threadIdx.x ? ENz + fz : EN + fh;
            a.e2[(r * tiles + tile) * 2 + threadIdx.x] = E;
            atomicMax(&a.e2max[r * 2 + threadIdx.x], E);
        }
        if (threadIdx.x == 2) a.s2[r * tiles + tile] = make_longlong2(yl, (yh << 32) | (unsigned)ENt);
        const long long hr = half_of(fr), ht = half_of(ft), hz = half_of(fz);
        auto sft = [](long long x, int s, long long h) { return s >= 0 ? (x + h) >> s : x << -s; };
#pragma unroll 2
        for (int pt = threadIdx.x; pt < zt * P; pt += nt) {
            const int z = divp(pt), i = pt - z * P;
            const cx n = Nn[pt];
            buf[z * lp + i] = mk(sft(n.y, ft, ht), sft(n.x, fr, hr));
            cx* l = buf + (zt + z / 2) * lp + i;
            const long long nz = sft(Ub[pt].y, fz, hz);
            if (z & 1) {
                l->x = nz;
            } else {
                l->y = nz;
                if (z + 1 == zt) l->x = 0;
            }
        }
    };
#pragma unroll 1
    for (int ph = 0; ph < 4; ++ph) {
        if (ph == 0) fill(std::integral_constant<int, 0>{});
        else if (ph == 1) fill(std::integral_constant<int, 1>{});
        else if (ph == 2) fill(std::integral_constant<int, 2>{});
        else fill_forward();
        if (ph < 3) zero_band(pl, buf, lp, nl, M + 1, P - M);
        __syncthreads();
        uint4 mx = transform(pl, buf, lp, ph < 3 ? nl : zt + (zt + 1) / 2, a.tw, ph < 3, true, zt);
        if (ph == 3) break;
        mx.x = __reduce_max_sync(0xffffffffu, mx.x);
        mx.y = __reduce_max_sync(0xffffffffu, mx.y);
        mx.z = __reduce_max_sync(0xffffffffu, mx.z);
        mx.w = __reduce_max_sync(0xffffffffu, mx.w);
        if (lane < 4) atomicMax(&s_mx[ph][lane], lane == 0 ? mx.x : lane == 1 ? mx.y : lane == 2 ? mx.z : mx.w);
        __syncthreads();
        if (ph == 0) products(std::integral_constant<int, 0>{});
        else if (ph == 1) products(std::integral_constant<int, 1>{});
        else products(std::integral_constant<int, 2>{});
        __syncthreads();   // the next fill overwrites the lines
    }
    for (int i = threadIdx.x; i < zt * (M + 1); i += nt) {
        const int m = divz(i), z = i - m * zt, ip = pd(m), in = pd(m ? P - m : 0);
        const cx Q = buf[z * lp + ip], Qn = buf[z * lp + in];   // (im, re)
        const cx* SL = buf + (zt + z / 2) * lp;
        const cx S = SL[ip], Sn = SL[in];
        const cx nz = (z & 1) ? mk((S.x + Sn.x) >> 1, (Sn.y - S.y) >> 1) : mk((S.y + Sn.y) >> 1, (S.x - Sn.x) >> 1);
        const size_t o = ((size_t)r * (M + 1) + m) * Pz + z0 + z;
        a.H2[o] = mk(Q.y, Q.x);
        a.H2[fs + o] = mk(Qn.y, -Qn.x);
        a.H2[2 * fs + o] = nz;
    }
}

template <class PL, int ZT, int NT, int MINB>
tc_status theta_pass(tc_plan* p, const ThetaArgs& a, cudaStream_t s) {
    const size_t sm = (size_t)(2 * a.zt * line_pitch(p->P_t) + 3 * a.zt * p->P_t) * sizeof(cx);
    auto k = k_fx_theta<PL, ZT, NT, MINB>;
    TC_CUDA(p, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int thr = PL::kStatic ? NT : round32(2 * a.zt * ((p->P_t + 7) / 8));
    k<<<a.nh * (p->P_z / a.zt), thr, sm, s>>>(a, p->fx_t);
    TC_LAUNCHED(p, "k_fx_theta");
    return TC_OK;
}

// z values of the blocks of the lengths with a compile-time plan (0: none)
int static_zt(int P) {
    switch (P) {
        case 12: return 2;
        case 24: return 8;
        case 36: case 48: case 72: case 96: case 144: return 4;
        case 192: case 288: case 384: case 576: return 2;
        case 768: case 1152: return 1;
    }
    return 0;
}

}  // namespace

// z values per theta block
int fx_zt(const tc_plan* p, int forced) {
    const int z = static_zt(p->P_t);
    if (forced == 0 && z > 0 && p->P_z % z == 0 && 3 * p->M <= p->P_t) return z;
    auto smem = [&](int t) { return (size_t)(2 * t * line_pitch(p->P_t) + 3 * t * p->P_t) * sizeof(cx); };
    auto threads = [&](int t) { return 2 * t * ((p->P_t + 7) / 8); };
    auto fits = [&](int t) { return p->P_z % t == 0 && threads(t) <= 320 && (t == 1 || smem(t) <= (size_t)(forced > 0 ? 200 : 100) * 1024); };
    if (forced > 0) {
        int zt = forced;
        while (zt > 1 && !fits(zt)) --zt;
        return zt;
    }
    // about 128 threads and whole warps: the best-filled block of up to 8 z values
    int best = 1;
    double fill = 0;
    for (int t = 1; t <= 8; ++t) {
        if (!fits(t) || (t > 1 && threads(t) > 160)) continue;
        const double q = (double)threads(t) / round32(threads(t)) + 0.002 * t;
        if (q > fill) {
            fill = q;
            best = t;
        }
    }
    return best;
}

tc_status fx::launch_fx_theta(tc_plan* p, ThetaArgs a, cudaStream_t s) {
    const int zs = static_zt(p->P_t);
    const bool st = p->theta_zt_forced == 0 && p->fx_zt == zs && 3 * p->M <= p->P_t;
    if (st) a.tw += p->fx_t.table;
    switch (st ? p->P_t : 0) {
        case 12: return theta_pass<Ct<12>, 2, 32, 12>(p, a, s);
        case 24: return theta_pass<Ct<24>, 8, 64, 8>(p, a, s);
        case 36: return theta_pass<Ct<36>, 4, 64, 8>(p, a, s);
        case 48: return theta_pass<Ct<48>, 4, 64, 8>(p, a, s);
        case 72: return theta_pass<Ct<72>, 4, 96, 6>(p, a, s);
        case 96: return theta_pass<Ct<96>, 4, 96, 6>(p, a, s);
        case 144: return theta_pass<Ct<144>, 4, 160, 4>(p, a, s);
        case 192: return theta_pass<Ct<192>, 2, 96, 5>(p, a, s);
        case 288: return theta_pass<Ct<288>, 2, 160, 4>(p, a, s);
        case 384: return theta_pass<Ct<384>, 2, 192, 3>(p, a, s);
        case 576: return theta_pass<Ct<576>, 2, 288, 2>(p, a, s);
        case 768: return theta_pass<Ct<768>, 1, 192, 3>(p, a, s);
        case 1152: return theta_pass<Ct<1152>, 1, 288, 2>(p, a, s);
        default: return 2 * p->fx_zt * ((p->P_t + 7) / 8) <= 128 ? theta_pass<Rt, 0, 128, 4>(p, a, s) : theta_pass<Rt, 0, 320, 2>(p, a, s);
    }
}

}  // namespace tc
