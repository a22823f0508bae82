// Declarations shared by the fixed-point passes of the FP64 nonlinear term (tc_fx_z.cu,
// tc_fx_theta.cu).
#pragma once

#include <algorithm>

#include "tc_fx.cuh"

namespace tc {
namespace fx {

inline unsigned magic(int d) { return d <= 1 ? 0u : (unsigned)((((unsigned long long)1 << 32) + d - 1) / d); }
inline int round32(int t) { return (t + 31) / 32 * 32; }

struct ThetaArgs {
    const cx* H1;
    cx* H2;
    const int2* e1;
    int* e2;
    int* e2max;
    longlong2* s2;     // sum of N_t over the points of each block [nh][tiles] (see block_sum)
    const int4* ir;    // 1 / r_j: limbs, exponent
    const int2* mm;    // m m_p: limbs of m m_p 2^(62 - emm)
    const int4* tw;
    int r0, nh, M, Pz, zt, emm;
    unsigned mzt, mP;   // magics of zt and P_theta
    long long mp;
};

// Exponents of a sum that takes one or two products: shifts of the old sum and of the
// products, with their rounding constants.
struct Sum {
    int so, s1, s2;
    long long ro, r1, r2;
    __device__ __forceinline__ void set(int& E, int e1, int e2) {
        const int En = max(E, max(e1, e2)) + 2;
        so = min(En - E, 63);
        s1 = En - e1 - 2;
        s2 = En - e2 - 2;
        ro = half_of(so);
        r1 = half_of(s1 + 32);
        r2 = half_of(s2 + 32);
        E = En;
    }
    __device__ __forceinline__ long long old(long long x) const { return (x + ro) >> so; }
    __device__ __forceinline__ long long first(lim a, lim b) const { return mulhi(a, b, s1, r1); }
    __device__ __forceinline__ long long second(lim a, lim b) const { return mulhi(a, b, s2, r2); }
};

// For each of NK line kinds the largest exponent er and the sum over m of its fields' largest
// values at that exponent, in units of 2^32, which bounds every sum of a theta line.  at(q, m)
// gives (exponent, largest value) of field q < NF; bound calls f(kind, field, weighted by
// m m_p) for each field of each kind; half: kinds that are one part of a pair of real fields
// (m and -m both count).  The sum is taken in a fixed order: the exponents decide rounding.  A
// weighted kind has no m = 0 entry: er does not cover that one, whose 2^(v.x - er) may overflow.
template <int NF, int NK, int NT, class AT, class BOUND>
__device__ __forceinline__ void line_bounds(AT at, BOUND bound, unsigned half, int M, long long mp, int nt, int* s_E, float (*s_bound)[NK],
                                            int (&er)[NK], float (&sum)[NK]) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int2 v[NF];
#pragma unroll
    for (int s = 0; s < NK; ++s) er[s] = 4 * kExpZero;
    for (int m = threadIdx.x; m <= M; m += nt) {
#pragma unroll
        for (int q = 0; q < NF; ++q) v[q] = at(q, m);
        bound([&](int s, int q, bool mul) {
            if (!mul || m > 0) er[s] = max(er[s], v[q].x);
        });
    }
    if (threadIdx.x < NK) s_E[threadIdx.x] = 4 * kExpZero;
    __syncthreads();
    int mine = 0;
#pragma unroll
    for (int s = 0; s < NK; ++s) {
        const int x = __reduce_max_sync(0xffffffffu, er[s]);
        if (lane == s) mine = x;
    }
    if (lane < NK) atomicMax(&s_E[lane], mine);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NK; ++s) {
        er[s] = s_E[s];
        sum[s] = 0.f;
    }
    for (int m = threadIdx.x; m <= M; m += nt) {
        const float mm = (float)(m * mp);
#pragma unroll
        for (int q = 0; q < NF; ++q) v[q] = at(q, m);
        bound([&](int s, int q, bool mul) {
            if (mul && m == 0) return;
            const int d = min(er[s] - v[q].x, 127);   // 2^-d, 0 below 2^-126
            const float x = (float)(unsigned)v[q].y * __int_as_float(max(127 - d, 0) << 23) * ((half >> s) & 1 ? 2.f : 1.f);
            sum[s] += mul ? x * mm : x;
        });
    }
#pragma unroll
    for (int s = 0; s < NK; ++s)
#pragma unroll
        for (int o = 16; o; o >>= 1) sum[s] += __shfl_xor_sync(0xffffffffu, sum[s], o);
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < NK; ++s) s_bound[wid][s] = sum[s];
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < NK; ++s) {
        sum[s] = 0.f;
        for (int w = 0; w < nt / 32; ++w) sum[s] += s_bound[w][s];
    }
}
// exponent that brings such a sum below 2^62, the parts of a real pair below 2^61 each
__device__ __forceinline__ int kind_exponent(int er, float sum, bool mul, bool half, int emm) {
    const int b = ((__float_as_int(sum * 1.001f) >> 23) & 0xff) - 126;   // sum < 2^b
    const int E = er + max(0, b - (half ? 29 : 30));
    return mul ? max(E, er + emm - 30) : E;   // keeps the shift of the products with m m_p positive
}

// Entries m and n - m of a theta line from two spectra.  pair: x = c_r + i c_t of (c_+, c_-) = (A, B);
// real2: x + i y of the real fields (X, Y).
__device__ __forceinline__ void put_pair(cx* l, int n, int m, cx A, cx B) {
    if (m == 0) {
        l[0] = mk((A.x + B.x) >> 1, (A.y - B.y) >> 1);
    } else {
        l[m] = A;
        l[n - m] = conj(B);
    }
}
__device__ __forceinline__ void put_real2(cx* l, int n, int m, cx X, cx Y) {
    if (m == 0) {
        l[0] = mk(X.x, Y.x);
    } else {
        l[m] = mk(X.x - Y.y, X.y + Y.x);
        l[n - m] = mk(X.x + Y.y, Y.x - X.y);
    }
}
__device__ __forceinline__ cx shr2(cx v, int t) { return mk(shr(v.x, t), shr(v.y, t)); }
// i m m_p v with the limbs F of m m_p 2^(62 - emm): exponents E of the result, e of v
__device__ __forceinline__ cx imul(cx v, int2 F, int emm, int E, int e) {
    const lim f = {F.x, F.y};
    const int sh = 30 - emm + E - e;
    return mk(-mulsh(split(v.y), f, sh), mulsh(split(v.x), f, sh));
}

struct ThetaAdjArgs {
    const cx* H1;      // lines of u, d_r u, d_z u; exponents e1
    const cx* Ha;      // lines of s_r, s_t, s_z; exponents e1a
    cx* H3;            // A, R, Z in the (+, -, z) basis
    const int2* e1;
    const int2* e1a;
    int* e2;           // [nh][tiles][6], e2max [nh][6]
    int* e2max;
    const int4* ir;
    const int2* mm;
    const int4* tw;
    int r0, nh, M, Pz, zt, emm;
    unsigned mzt, mP;
    long long mp;
};

// The sum of a block's N_t, h 2^52 + l in units of 2^(E - 62), is stored as (l, h and E)
__device__ __forceinline__ double block_sum(longlong2 v) {
    const int E = (int)(unsigned)v.y;
    return E > kExpNaN / 2 ? nan64() : to_double(v.y >> 32, E - 10) + to_double(v.x, E - 62);
}

tc_status launch_fx_theta_adj(tc_plan* p, ThetaAdjArgs a, cudaStream_t s);
tc_status launch_fx_theta(tc_plan* p, ThetaArgs a, cudaStream_t s);

}  // namespace fx
}  // namespace tc
