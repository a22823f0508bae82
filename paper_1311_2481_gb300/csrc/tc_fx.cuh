// 64-bit fixed-point arithmetic and transforms for the FP64 form of the nonlinear term.
//
// GB300 retires 2 FP64 lanes per SM and clock, so an FP64 instruction costs a warp 64 issue
// cycles of its sub-partition.  Measured on the integer and FMA pipes: a 64-bit add (two
// instructions) 59 lanes per SM and clock, a 32 x 32 + 64 -> 64 multiply-add 58.  A transform
// is additions and multiplications by numbers of modulus <= 1, so it runs in fixed point
// with one exponent per line: 2^62 holds the largest sum the line can reach, which leaves
// more bits than the 53 of a double for every value within 2^-9 of that sum, at 1/32 of the
// cost of an FP64 addition and about 1/10 of that of an FP64 complex multiplication.
//
// A value x is held as X = x 2^(62 - E), |X| < 2^62, E per line or block.  A factor c of
// modulus <= 1 is held as C = c 2^62 in two 32-bit limbs, C = ch 2^32 + cl with cl signed.
#pragma once

#include "tc_internal.cuh"

namespace tc {
namespace fx {

struct __align__(16) cx { long long x, y; };
struct lim { int h, l; };

constexpr int kExpNaN = 1 << 20;     // exponent of a line that holds a NaN or an Inf
constexpr int kExpZero = -(1 << 17);  // exponent of a line of zeros

__device__ __forceinline__ cx mk(long long x, long long y) { cx c; c.x = x; c.y = y; return c; }
__device__ __forceinline__ cx add(cx a, cx b) { return mk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ cx sub(cx a, cx b) { return mk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ cx neg(cx a) { return mk(-a.x, -a.y); }
__device__ __forceinline__ cx conj(cx a) { return mk(a.x, -a.y); }
template <bool INV> __device__ __forceinline__ cx rot(cx a) { return INV ? mk(-a.y, a.x) : mk(a.y, -a.x); }

// limbs with both halves signed: x = h 2^32 + l, l in [-2^31, 2^31)
__host__ __device__ __forceinline__ constexpr lim split(long long x) {
    lim r{(int)(x >> 32) + (int)((unsigned)x >> 31), (int)(unsigned)x};
    return r;
}
__device__ __forceinline__ long long mad(int a, int b, long long c) { return c + (long long)a * b; }
// (T 2^32 + low word of mid) >> s for 0 <= s < 32, with mid's high word already in T
__device__ __forceinline__ long long take(long long T, long long mid, int s) {
    const unsigned l = __funnelshift_r((unsigned)mid, (unsigned)T, s);
    const unsigned h = __funnelshift_r((unsigned)T, (unsigned)(T >> 32), s);
    return (long long)(((unsigned long long)h << 32) | l);
}
// (x C) / 2^62, rounded, up to a unit (the product of the low limbs is left out)
constexpr long long kHalf = 1ll << 29;
__device__ __forceinline__ long long mulq(lim x, lim c) {
    const long long mid = mad(x.h, c.l, mad(x.l, c.h, kHalf));
    return take(mad(x.h, c.h, mid >> 32), mid, 30);
}
__device__ __forceinline__ long long mulq(long long x, lim c) { return mulq(split(x), c); }
// x >> t for t >= 0 (PTX shifts clamp at 64: the sign remains)
__device__ __forceinline__ long long shr(long long x, int t) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(t));
    return r;
}
__device__ __forceinline__ long long shl(long long x, int t) {
    long long r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(t));
    return r;
}
// (x c) >> (32 + sh), sh >= 0
__device__ __forceinline__ long long mulsh(lim x, lim c, int sh) {
    const long long mid = mad(x.h, c.l, mad(x.l, c.h, 0));
    const long long T = mad(x.h, c.h, mid >> 32);
    if (sh < 32) return take(T, mid, sh);
    return shr(T, sh - 32);
}
// (x c + rnd) >> (64 + sh), sh >= 0; rnd = half_of(32 + sh), in units of 2^32, rounds to nearest.
// Sums over many points need the rounding: a truncated product is half a unit low on
// average, which would show in their mean.
__device__ __forceinline__ long long mulhi(lim x, lim c, int sh, long long rnd) {
    const long long mid = mad(x.h, c.l, mad(x.l, c.h, rnd));
    return shr(mad(x.h, c.h, mid >> 32), sh);
}
constexpr long long kHalf32 = 1ll << 31;   // half_of(32)
__device__ __forceinline__ long long half_of(int sh) { return sh > 0 && sh < 62 ? 1ll << (sh - 1) : 0ll; }

// v (c + i s) or its conjugate
template <bool INV> __device__ __forceinline__ cx cmul(cx v, lim c, lim s) {
    const lim a = split(v.x), b = split(v.y);
    const int sh = INV ? s.h : -s.h, sl = INV ? s.l : -s.l;
    const int nh = -sh, nl = -sl;
    const long long mr = mad(b.l, nh, mad(b.h, nl, mad(a.l, c.h, mad(a.h, c.l, kHalf))));
    const long long mi = mad(a.l, sh, mad(a.h, sl, mad(b.l, c.h, mad(b.h, c.l, kHalf))));
    const long long Tr = mad(b.h, nh, mad(a.h, c.h, mr >> 32));
    const long long Ti = mad(a.h, sh, mad(b.h, c.h, mi >> 32));
    return mk(take(Tr, mr, 30), take(Ti, mi, 30));
}
template <bool INV> __device__ __forceinline__ cx cmul(cx v, int4 w) { return cmul<INV>(v, lim{w.x, w.y}, lim{w.z, w.w}); }

// ---------------------------------------------------------------- in-register DFTs
// X_k = sum_n x_n exp(s 2 pi i n k / R), s = +1 (INV) or -1, natural order.  Every partial
// sum is bounded by the sum of the moduli of the inputs, so nothing overflows.
constexpr long long kSin60 = 3993837246235628775LL;   // sin(pi/3) 2^62
constexpr long long kH = 3260954456333195553LL;       // cos(pi/4) 2^62
constexpr long long kC16 = 4260642322793532497LL, kS16 = 1764815834521887442LL;   // pi/8
constexpr long long kC9a = 3532756447825785444LL, kS9a = 2964334632409774423LL;   // 2 pi/9
constexpr long long kC9b = 800810873071977681LL, kS9b = 4541624145405292212LL;    // 4 pi/9
constexpr long long kC9d = -4333567320897763126LL, kS9d = 1577289512995517789LL;  // 8 pi/9

template <bool INV> __device__ __forceinline__ void dft2(cx* v) {
    const cx a = v[0];
    v[0] = add(a, v[1]);
    v[1] = sub(a, v[1]);
}
template <bool INV> __device__ __forceinline__ void dft3(cx& a, cx& b, cx& c) {
    constexpr lim s = split(kSin60);
    const cx t1 = add(b, c), t2 = sub(b, c);
    const cx m1 = mk(a.x - (t1.x >> 1), a.y - (t1.y >> 1));
    const cx m2 = rot<INV>(mk(mulq(t2.x, s), mulq(t2.y, s)));
    a = add(a, t1);
    b = add(m1, m2);
    c = sub(m1, m2);
}
template <bool INV> __device__ __forceinline__ void dft4(cx& v0, cx& v1, cx& v2, cx& v3) {
    const cx a0 = add(v0, v2), a1 = sub(v0, v2), a2 = add(v1, v3), a3 = rot<INV>(sub(v1, v3));
    v0 = add(a0, a2);
    v2 = sub(a0, a2);
    v1 = add(a1, a3);
    v3 = sub(a1, a3);
}
// a exp(s 2 pi i / 8): (x - y, x + y) h for s = +1
template <bool INV> __device__ __forceinline__ cx w8(cx a) {
    constexpr lim h = split(kH);
    return INV ? mk(mulq(a.x - a.y, h), mulq(a.x + a.y, h)) : mk(mulq(a.x + a.y, h), mulq(a.y - a.x, h));
}
template <bool INV> __device__ __forceinline__ void dft8(cx* v) {
    dft4<INV>(v[0], v[2], v[4], v[6]);   // even samples: E0..E3 in v[0], v[2], v[4], v[6]
    dft4<INV>(v[1], v[3], v[5], v[7]);
    v[3] = w8<INV>(v[3]);
    v[5] = rot<INV>(v[5]);
    v[7] = rot<INV>(w8<INV>(v[7]));
    cx e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = add(e[k], o[k]);
        v[k + 4] = sub(e[k], o[k]);
    }
}
template <bool INV> __device__ __forceinline__ void dft16(cx* v) {
    constexpr lim c1 = split(kC16), s1 = split(kS16);
#pragma unroll
    for (int n = 0; n < 4; ++n) dft4<INV>(v[n], v[n + 4], v[n + 8], v[n + 12]);   // k1 in v[n + 4 k1]
    v[5] = cmul<INV>(v[5], c1, s1);
    v[9] = w8<INV>(v[9]);
    v[13] = cmul<INV>(v[13], s1, c1);
    v[6] = w8<INV>(v[6]);
    v[10] = rot<INV>(v[10]);
    v[14] = rot<INV>(w8<INV>(v[14]));
    v[7] = cmul<INV>(v[7], s1, c1);
    v[11] = rot<INV>(w8<INV>(v[11]));
    v[15] = neg(cmul<INV>(v[15], c1, s1));
    cx t[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        dft4<INV>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
#pragma unroll
        for (int q = 0; q < 4; ++q) t[k + 4 * q] = v[4 * k + q];
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = t[q];
}
template <bool INV> __device__ __forceinline__ void dft9(cx* v) {
    constexpr lim ca = split(kC9a), sa = split(kS9a), cb = split(kC9b), sb = split(kS9b), cd = split(kC9d), sd = split(kS9d);
#pragma unroll
    for (int n = 0; n < 3; ++n) dft3<INV>(v[n], v[n + 3], v[n + 6]);
    v[4] = cmul<INV>(v[4], ca, sa);
    v[7] = cmul<INV>(v[7], cb, sb);
    v[5] = cmul<INV>(v[5], cb, sb);
    v[8] = cmul<INV>(v[8], cd, sd);
    cx t[9];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dft3<INV>(v[3 * k], v[3 * k + 1], v[3 * k + 2]);
#pragma unroll
        for (int q = 0; q < 3; ++q) t[k + 3 * q] = v[3 * k + q];
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] = t[q];
}
// 6 = 2 x 3 and 12 = 3 x 4 by the prime-factor mapping (no inner twiddles)
template <bool INV> __device__ __forceinline__ void dft6(cx* v) {
    cx t[6];
#pragma unroll
    for (int a = 0; a < 2; ++a) dft3<INV>(v[(3 * a) % 6], v[(3 * a + 2) % 6], v[(3 * a + 4) % 6]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const cx p = v[(2 * b) % 6], q = v[(2 * b + 3) % 6];
        t[(4 * b) % 6] = add(p, q);
        t[(4 * b + 3) % 6] = sub(p, q);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = t[q];
}
template <bool INV> __device__ __forceinline__ void dft12(cx* v) {
    cx t[12];
#pragma unroll
    for (int b = 0; b < 4; ++b) dft3<INV>(v[(3 * b) % 12], v[(3 * b + 4) % 12], v[(3 * b + 8) % 12]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        dft4<INV>(v[(4 * a) % 12], v[(4 * a + 3) % 12], v[(4 * a + 6) % 12], v[(4 * a + 9) % 12]);
#pragma unroll
        for (int q = 0; q < 4; ++q) t[(4 * a + 9 * q) % 12] = v[(4 * a + 3 * q) % 12];
    }
#pragma unroll
    for (int q = 0; q < 12; ++q) v[q] = t[q];
}
template <int R, bool INV> __device__ __forceinline__ void dft(cx* v) {
    if constexpr (R == 2) dft2<INV>(v);
    else if constexpr (R == 3) dft3<INV>(v[0], v[1], v[2]);
    else if constexpr (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 6) dft6<INV>(v);
    else if constexpr (R == 8) dft8<INV>(v);
    else if constexpr (R == 9) dft9<INV>(v);
    else if constexpr (R == 12) dft12<INV>(v);
    else dft16<INV>(v);
}

// |x| up to one unit, without a carry: the bits below the sign
__device__ __forceinline__ unsigned mag_hi(long long x) { const int h = (int)(x >> 32); return (unsigned)(h ^ (h >> 31)); }
__device__ __forceinline__ int bits(unsigned v) { return 32 - __clz((int)v); }
__device__ __forceinline__ int bits64(unsigned long long v) { return 64 - __clzll((long long)v); }

// ---------------------------------------------------------------- plans
// Butterflies per thread of a pass: at least 8 points per thread, so a line of n points takes at
// most n / 8 threads whatever its radices.
__host__ __device__ constexpr int per_thread_of(int R) { return R == 2 ? 4 : R == 3 ? 3 : R <= 6 ? 2 : 1; }

// i / d for i < 2^16 with magic = ceil(2^32 / d) (0 for d = 1)
__device__ __forceinline__ int udiv(int i, unsigned magic) { return magic ? (int)__umulhi((unsigned)i, magic) : i; }

// Position of entry i of a line in shared memory: one 16-byte slot of padding per 8 entries, so
// that the stride-R stores of a pass spread over the banks (R = 8 without a conflict, the
// others at most two-way), and strides of a multiple of 8 entries stay constant offsets.
__host__ __device__ constexpr int pd(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int line_pitch(int n) { return n + (n + 7) / 8; }

// Compile-time plans of the lengths 3 2^a and 9 2^a (the 3/2 grids of M = 2^a and 3 2^a):
// two or three passes; every pass after the first has n / R a multiple of 8 where the length
// allows it, and the first radix is 8 or 16 where it can be (its butterflies have inputs that
// lie wholly in the zero band of a dealiased spectrum).
template <int N> struct Radix;
template <> struct Radix<12> { static constexpr int np = 2, r[3] = {4, 3, 1}; };
template <> struct Radix<24> { static constexpr int np = 2, r[3] = {8, 3, 1}; };
template <> struct Radix<36> { static constexpr int np = 2, r[3] = {6, 6, 1}; };
template <> struct Radix<48> { static constexpr int np = 2, r[3] = {8, 6, 1}; };
template <> struct Radix<72> { static constexpr int np = 2, r[3] = {8, 9, 1}; };
template <> struct Radix<96> { static constexpr int np = 2, r[3] = {8, 12, 1}; };
template <> struct Radix<144> { static constexpr int np = 2, r[3] = {12, 12, 1}; };
template <> struct Radix<192> { static constexpr int np = 2, r[3] = {16, 12, 1}; };
template <> struct Radix<288> { static constexpr int np = 3, r[3] = {8, 6, 6}; };
template <> struct Radix<384> { static constexpr int np = 3, r[3] = {8, 8, 6}; };
template <> struct Radix<576> { static constexpr int np = 3, r[3] = {8, 6, 12}; };
template <> struct Radix<768> { static constexpr int np = 3, r[3] = {8, 8, 12}; };
template <> struct Radix<1152> { static constexpr int np = 3, r[3] = {8, 12, 12}; };
template <> struct Radix<1536> { static constexpr int np = 3, r[3] = {16, 8, 12}; };
template <> struct Radix<2304> { static constexpr int np = 3, r[3] = {16, 12, 12}; };

// A plan with compile-time length (Ct) or with run-time radices (Rt, any 2^a 3^b): length, and
// for pass p its radix, ns (product of the earlier radices), nb (n / radix) and table offset.
template <int N> struct Ct {
    static constexpr bool kStatic = true;
    static constexpr int np = Radix<N>::np, n = N;
    __host__ __device__ static constexpr int r(int p) { return Radix<N>::r[p]; }
    __host__ __device__ static constexpr int ns(int p) { return p == 0 ? 1 : ns(p - 1) * r(p - 1); }
    __host__ __device__ static constexpr int nb(int p) { return N / r(p); }
    __host__ __device__ static constexpr int tw(int p) { return p <= 1 ? 0 : tw(p - 1) + (r(p - 1) - 1) * ns(p - 1); }
    // inputs q of the first pass with qlo() <= q < qhi() lie in [n/3 + 1, 2n/3) and are not read
    __host__ __device__ static constexpr int qlo() { return r(0) / 3 + 1; }
    __host__ __device__ static constexpr int qhi() { return r(0) * 2 / 3 > qlo() ? r(0) * 2 / 3 : qlo(); }
    __host__ __device__ Ct(const FxPlan&) {}
    __device__ static constexpr int size() { return N; }
};
struct Rt {
    static constexpr bool kStatic = false;
    const FxPlan& f;
    __device__ explicit Rt(const FxPlan& f_) : f(f_) {}
    __device__ int size() const { return f.n; }
};

// ---------------------------------------------------------------- passes
// A transform of nl lines of pitch lp in shared memory, inverse sign (exp(+i)); a forward one is
// the same on entries with real and imaginary part exchanged, before and after.  The input
// lies at entry positions i, all later states at pd(i).  With want_max the largest |part|
// that the thread has written goes to mx, in units of 2^32: (x, y) for lines < nl0, (z, w)
// for the others.
template <int R>
__device__ __forceinline__ void butterfly(cx (&v)[R], int ns, int k, const int4* __restrict__ t) {
    if (ns > 1) {
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = cmul<true>(v[q], __ldg(&t[(q - 1) * ns + k]));
    }
    dft<R, true>(v);
}

// right shifts of the input, taken in the first pass: lines < nl0 by (x0, y0), others by (x1, y1)
struct InShift {
    bool on = false;
    int x0 = 0, y0 = 0, x1 = 0, y1 = 0;
};

// [qlo, qhi): inputs known to be zero
template <int R, int QLO, int QHI>
__device__ __forceinline__ void pass(cx* buf, int lp, int nl, bool first, int ns, int nb, unsigned mnb, unsigned mns,
                                     const int4* __restrict__ tw, bool want_max, int nl0, uint4& mx, bool fold, const InShift& in) {
    constexpr int B = per_thread_of(R);
    cx v[B][R];
    int ln[B], jj[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int idx = threadIdx.x + b * blockDim.x;
        ln[b] = -1;
        if (idx < nl * nb) {
            const int line = fold ? idx / nb : udiv(idx, mnb), j = idx - line * nb;
            const cx* src = buf + line * lp;
            ln[b] = line;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (q >= QLO && q < QHI) v[b][q] = mk(0, 0);
                else if (first) v[b][q] = src[j + q * nb];
                else if (fold && nb % 8 == 0) v[b][q] = src[pd(j) + q * pd(nb)];
                else v[b][q] = src[pd(j + q * nb)];
            }
            if (first && in.on) {
                const int sx = line < nl0 ? in.x0 : in.x1, sy = line < nl0 ? in.y0 : in.y1;
#pragma unroll
                for (int q = 0; q < R; ++q) v[b][q] = mk(shr(v[b][q].x, sx), shr(v[b][q].y, sy));
            }
            const int k = first ? 0 : fold ? j % ns : j - udiv(j, mns) * ns;
            butterfly<R>(v[b], first ? 1 : ns, k, tw);
            jj[b] = (j - k) * R + k;
        } else {   // defined on every path: registers written on one path only stay live around the caller's loop
            jj[b] = 0;
#pragma unroll
            for (int q = 0; q < R; ++q) v[b][q] = mk(0, 0);
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; ++b)
        if (ln[b] >= 0) {
            cx* dst = buf + ln[b] * lp;
#pragma unroll
            for (int q = 0; q < R; ++q) {
                if (fold && ns % 8 == 0) dst[pd(jj[b]) + q * pd(ns)] = v[b][q];
                else dst[pd(jj[b] + q * ns)] = v[b][q];
            }
            if (want_max) {
                unsigned mx_ = 0, my_ = 0;
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    mx_ = max(mx_, mag_hi(v[b][q].x));
                    my_ = max(my_, mag_hi(v[b][q].y));
                }
                if (ln[b] < nl0) mx = make_uint4(max(mx.x, mx_), max(mx.y, my_), mx.z, mx.w);
                else mx = make_uint4(mx.x, mx.y, max(mx.z, mx_), max(mx.w, my_));
            }
        }
    __syncthreads();
}

template <int N, int P, bool BAND>
__device__ __forceinline__ void pass_of(cx* buf, int lp, int nl, const int4* __restrict__ tw, bool want_max, int nl0, uint4& mx,
                                        const InShift& in) {
    using C = Ct<N>;
    constexpr bool z = P == 0 && BAND;
    pass<C::r(P), z ? C::qlo() : 0, z ? C::qhi() : 0>(buf, lp, nl, P == 0, C::ns(P), C::nb(P), 0u, 0u, tw + C::tw(P),
                                                      want_max && P == C::np - 1, nl0, mx, true, in);
}
// band: the input is zero in [n/3 + 1, 2n/3), and entries the first pass skips are not read
template <int N>
__device__ __forceinline__ uint4 transform(const Ct<N>&, cx* buf, int lp, int nl, const int4* __restrict__ tw, bool band,
                                           bool want_max = false, int nl0 = 0, const InShift& in = InShift{}) {
    uint4 mx = make_uint4(0, 0, 0, 0);
    if (band) pass_of<N, 0, true>(buf, lp, nl, tw, false, nl0, mx, in);
    else pass_of<N, 0, false>(buf, lp, nl, tw, false, nl0, mx, in);
    pass_of<N, 1, false>(buf, lp, nl, tw, want_max, nl0, mx, in);
    if constexpr (Ct<N>::np > 2) pass_of<N, 2, false>(buf, lp, nl, tw, want_max, nl0, mx, in);
    return mx;
}
__device__ __forceinline__ uint4 transform(const Rt& pl, cx* buf, int lp, int nl, const int4* __restrict__ tw, bool,
                                           bool want_max = false, int nl0 = 0, const InShift& in = InShift{}) {
    uint4 mx = make_uint4(0, 0, 0, 0);
#pragma unroll 1
    for (int p = 0; p < pl.f.np; ++p) {
        const FxPass& s = pl.f.p[p];
        const bool wm = want_max && p == pl.f.np - 1;
        const int4* t = tw + s.tw;
#define TC_FX_PASS(R) \
    case R: pass<R, 0, 0>(buf, lp, nl, p == 0, s.ns, s.nb, s.mnb, s.mns, t, wm, nl0, mx, false, in); break;
        switch (s.r) {
            TC_FX_PASS(2) TC_FX_PASS(3) TC_FX_PASS(4) TC_FX_PASS(6) TC_FX_PASS(8) TC_FX_PASS(9) TC_FX_PASS(12)
        }
#undef TC_FX_PASS
    }
    return mx;
}
// zero the entries zlo <= p < zhi of the input of nl lines, as far as the first pass reads them
template <class PL>
__device__ __forceinline__ void zero_band(const PL& pl, cx* buf, int lp, int nl, int zlo, int zhi) {
    int a = zhi, b = zhi;   // [a, b) is skipped
    if constexpr (PL::kStatic) {
        a = PL::qlo() * PL::nb(0);
        b = PL::qhi() * PL::nb(0);
    }
    const int w1 = a - zlo, w = w1 + zhi - b;
    for (int l = 0; l < nl; ++l)
        for (int i = threadIdx.x; i < w; i += blockDim.x) buf[l * lp + (i < w1 ? zlo + i : b + i - w1)] = mk(0, 0);
}

// ---------------------------------------------------------------- conversions
// biased exponent of |d| (2047 for NaN and Inf, 0 for zeros and subnormals, which count as 0)
__device__ __forceinline__ int bexp(double d) { return (__double2hiint(d) >> 20) & 0x7ff; }
// d 2^(62 + 1022 - emax) truncated, for a biased exponent of d of at most emax: |result| < 2^62
__device__ __forceinline__ long long fix(double d, int emax) {
    const int h = __double2hiint(d);
    const int e = (h >> 20) & 0x7ff;
    const unsigned mh = ((unsigned)h & 0xfffffu) | 0x100000u, ml = (unsigned)__double2loint(d);
    // 53-bit mantissa moved up by 9, then down by the exponent difference
    const unsigned long long m = ((unsigned long long)((mh << 9) | (ml >> 23)) << 32) | (ml << 9);
    const int t = emax - e;
    long long v = (e == 0 || t > 62) ? 0 : (long long)(m >> t);
    return h < 0 ? -v : v;
}
// X 2^s rounded to a double (s outside the range of a double gives 0 or Inf)
__device__ __forceinline__ double to_double(long long X, int s) {
    const unsigned long long a = X < 0 ? 0ull - (unsigned long long)X : (unsigned long long)X;
    if (a == 0) return 0.0;
    const int z = __clzll((long long)a);
    const unsigned long long m = a << z;                       // top bit set
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1);  // 53 bits, rounded (up to 2^53)
    const int e = 1023 + 63 - z + s;                           // biased exponent of the top bit
    unsigned long long b;
    if (e <= 0) b = 0;
    else if (e >= 2047) b = 0x7ff0000000000000ull;
    else b = ((unsigned long long)(e - 1) << 52) + r;          // the leading bit adds one to the exponent
    return __longlong_as_double((long long)(b | (X < 0 ? 0x8000000000000000ull : 0ull)));
}
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }

// ---------------------------------------------------------------- radial stencils
// The window of R consecutive rows j0 .. j0 + R - 1 of a real column: rows j0 - 4 .. j0 + R + 3,
// converted once to the exponent e of the largest, |x| < 2^60: nine products of the limbs then add
// up to less than 9 2^59 + 2^61 < 2^63.  An output costs 27 32-bit multiply-adds instead of 9 FP64
// FMAs of 64 issue cycles per warp, plus (R + 8) / R conversions.
// Rounding: values are cut at 2^-60 of the window's largest, and the products of the low limbs, left
// out, are of that size as well (standard deviation 2^-60 2^(e + ew), ew the exponent of sum |w|;
// 9 times that at most).  An FP64 sum of the row is off by 0.3 to 2 times 2^-53 sum |w f| (9 times at
// most).  So a row is left to the FP64 sum (far) unless one of its four nearest neighbours has
// |w f| >= 2^-7 2^(e + ew), exponents taken: the error is then below 2^-53 sum |w f|.  Measured
// against rationals over columns that are smooth, wavy, vanish at the walls or go as r^+-32, r^+-192
// (N_r = 48 to 256): at most 0.9 in a row, 2.3 with FP64 sums; columns in norm as good or
// better.  The four rows next to each wall, whose stencils are shorter, and rows near a NaN, an Inf
// or the smallest numbers are FP64 sums too, but windows of zeros (modes that a flow does not have)
// are not.
constexpr int kFar = 6, kLowExp = 70;
// fix() for emax > kLowExp, where zeros and subnormals are shifted out like all that is small
__device__ __forceinline__ long long fix_tile(double d, int emax) {
    const int h = __double2hiint(d);
    const unsigned mh = ((unsigned)h & 0xfffffu) | 0x100000u, ml = (unsigned)__double2loint(d);
    unsigned long long m = ((unsigned long long)((mh << 9) | (ml >> 23)) << 32) | (ml << 9);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(emax - ((h >> 20) & 0x7ff)));
    return h < 0 ? -(long long)m : (long long)m;
}
template <int R> struct Tile {
    lim x[R + 8];
    int e;          // exponent of the window
    unsigned fp64;   // bit i: row i is left to the FP64 sum
    __device__ __forceinline__ bool far(int i) const { return (fp64 >> i) & 1; }
    // weights w[9] and their exponent ew of the row j0 + i
    __device__ __forceinline__ double row(int i, const int2* __restrict__ w, int ew) const {
        long long m = 0, s = 0;
#pragma unroll
        for (int t = 0; t < kStencil; ++t) {
            const int2 v = __ldg(&w[t]);
            m = mad(x[i + t].h, v.y, mad(x[i + t].l, v.x, m));
            s = mad(x[i + t].h, v.x, s);
        }
        return to_double(take(s + (m >> 32), m, 28), e + ew - 1084);
    }
    // b: exponents of the window's entries; limit: kFar, or more where less accuracy does; near(i): those of 2^ew / |w| of the entries i + 2, i + 3,
    // i + 5, i + 6 of row j0 + i, a byte each
    // zero: all entries are zero (not merely small): the rows are then 0 without an FP64 sum.  Returns the
    // exponent to convert the window to.
    template <class Near, class Zero>
    __device__ __forceinline__ int exponents(const int (&b)[R + 8], int limit, Near near, Zero zero) {
        e = 0;
#pragma unroll
        for (int i = 0; i < R + 8; ++i) e = max(e, b[i]);
        fp64 = e >= 2047 || e <= kLowExp ? ~0u : 0u;
        if (e <= 1 && zero()) {
            fp64 = 0;
            return 4096;   // shifts all out
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const unsigned q = near(i);
            const int c = min(min((int)(q & 255) - b[i + 2], (int)(q >> 8 & 255) - b[i + 3]),
                              min((int)(q >> 16 & 255) - b[i + 5], (int)(q >> 24) - b[i + 6]));
            if (e + c > limit) fp64 |= 1u << i;
        }
        return e + 2;
    }
    static __device__ __forceinline__ bool zeros(const double (&d)[R + 8]) {
        unsigned any = 0;
#pragma unroll
        for (int i = 0; i < R + 8; ++i) any |= (unsigned)__double2hiint(d[i]) << 1 | (unsigned)__double2loint(d[i]);
        return any == 0;
    }
    template <class Near> __device__ __forceinline__ void load(const double (&d)[R + 8], int limit, Near near) {
        int b[R + 8];
#pragma unroll
        for (int i = 0; i < R + 8; ++i) b[i] = bexp(d[i]);
        const int to = exponents(b, limit, near, [&] { return zeros(d); });
#pragma unroll
        for (int i = 0; i < R + 8; ++i) x[i] = split(fix_tile(d[i], to));
    }
    // the window of a + d, added after the conversion (one exponent more)
    template <class Near>
    __device__ __forceinline__ void load(const double (&a)[R + 8], const double (&d)[R + 8], int limit, Near near) {
        int b[R + 8];
#pragma unroll
        for (int i = 0; i < R + 8; ++i) b[i] = max(bexp(a[i]), bexp(d[i])) + 1;
        const int to = exponents(b, limit, near, [&] { return zeros(a) && zeros(d); });
#pragma unroll
        for (int i = 0; i < R + 8; ++i) x[i] = split(fix_tile(a[i], to) + fix_tile(d[i], to));
    }
};
}  // namespace fx
}  // namespace tc
