// Declarations shared by the fixed-point passes of the FP64 nonlinear term (tc_fx_z.cu,
// tc_fx_theta.cu).
#pragma once

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
    const int4* ir;    // 1 / r_j: limbs, exponent
    const int2* mm;    // m m_p: limbs of m m_p 2^(62 - emm)
    const int4* tw;
    int r0, nh, M, Pz, zt, emm;
    unsigned mzt, mP;   // magics of zt and P_theta
    long long mp;
};

tc_status launch_fx_theta(tc_plan* p, ThetaArgs a, cudaStream_t s);

}  // namespace fx
}  // namespace tc
