// Pseudospectral nonlinear term N(u) = u . grad u (Sec. 3.2 step 1, Eq. NS_cyl) on the
// P_theta x P_z dealiased grid (Sec. 3.1): the entry for both forms, and the theta pass of the
// mixed form for lengths without a specialised kernel (tc_theta_s.cu).  Three passes, one
// device-memory staging area between each (the single-GPU counterpart of the paper's global
// transposes, Sec. 4):
//
//   inverse z  per (r, m): 9 zero-padded inverse transforms along z of the u_+, u_-, u_z lines
//              and of their d_r and d_z lines                            -> H1[9][r][m][z]
//   theta      per (r, z tile): the 12 real physical fields as 6 complex inverse transforms
//              along theta (two real fields per complex line; d_theta = i m m_p applied here),
//              the pointwise products with the curvature terms, and the forward transform of
//              N_r + i N_theta (giving N_+ and N_- directly) and of N_z (two z per line).
//                                                                        -> H2[3][r][m][z]
//   forward z  per (r, m): forward transforms along z, truncation to |k| <= K, 1/(P_theta P_z).
//
// FP64 form: 64-bit fixed-point lines (tc_fx_z.cu, tc_fx_theta.cu).  Mixed form: FP32 lines
// (tc_mixed.cu); the transforms here are mixed-radix (4, 2, 3) Stockham passes in shared memory
// with twiddles from a long-double table.
#include "tc_internal.cuh"
#include "tc_fft_core.cuh"

namespace tc {

// ---------------------------------------------------------------- theta pass + products
// Line p of a z value (6 per z):  0 (u_r, u_t)  1 (d_r u_r, d_r u_t)  2 (d_t u_r, d_t u_t)
//                                 3 (d_z u_r, d_z u_t)  4 (u_z, d_r u_z)  5 (d_t u_z, d_z u_z)
template <typename V>
__global__ void __launch_bounds__(256) k_theta(const V* __restrict__ H1, V* __restrict__ H2,
                                               const double* __restrict__ irn, int r0, int nh, int M,
                                               int Pz, double mp, int zt,
                                               const V* __restrict__ tw, Radices rad,
                                               const float* __restrict__ dsc) {
    using T = typename Real<V>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Pt = rad.n;
    const int nl = 6 * zt;
    V* a = reinterpret_cast<V*>(smem_raw);
    V* b = a + (size_t)nl * Pt;
    const int tiles = Pz / zt;
    const int r = blockIdx.x / tiles;   // row within the staged rows r0 .. r0 + nh - 1
    const int z0 = (blockIdx.x % tiles) * zt;
    const size_t fstride = (size_t)nh * (M + 1) * Pz;
    const V* h = H1 + (size_t)r * (M + 1) * Pz + z0;
    // d_r u_z enters line 4 scaled by a power of two
    const T ds = (T)dsc[r0 + r], ids = (T)1 / ds;

    for (int idx = threadIdx.x; idx < nl * Pt; idx += blockDim.x) { a[idx].x = 0; a[idx].y = 0; }
    __syncthreads();
    // spectra of the 6 complex lines per z
    for (int idx = threadIdx.x; idx < 6 * zt * (M + 1); idx += blockDim.x) {
        // z fastest: neighbouring threads read neighbouring z of one (field, m) line
        const int zi = idx % zt;
        const int t = idx / zt;
        const int m = t % (M + 1);
        const int pr = t / (M + 1);
        V* line = a + (size_t)(zi * 6 + pr) * Pt;
        const size_t o = (size_t)m * Pz + zi;
        const T mm = (T)(mp * m);
        if (pr < 4) {  // (+,-) pair: x = c_r + i c_t has spectrum A_m (m>0), conj(B_m) at -m
            const int fa = pr == 0 ? 0 : pr == 1 ? 3 : pr == 2 ? 0 : 6;
            V A = h[fa * fstride + o], B = h[(fa + 1) * fstride + o];
            if (pr == 2) { A = cmuli(A); A.x *= mm; A.y *= mm; B = cmuli(B); B.x *= mm; B.y *= mm; }
            if (m == 0) {
                V c0; c0.x = (T)0.5 * (A.x + B.x); c0.y = (T)0.5 * (A.y - B.y);
                line[0] = c0;
            } else {
                line[m] = A;
                line[Pt - m] = cconj(B);
            }
        } else {       // two real fields x, y: spectrum X_m + i Y_m, conj(X_m) + i conj(Y_m) at -m
            V X, Y;
            if (pr == 4) { X = h[2 * fstride + o]; Y = h[5 * fstride + o]; Y.x *= ds; Y.y *= ds; }
            else { X = h[2 * fstride + o]; X = cmuli(X); X.x *= mm; X.y *= mm; Y = h[8 * fstride + o]; }
            if (m == 0) {
                V c0; c0.x = X.x; c0.y = Y.x;
                line[0] = c0;
            } else {
                V p1; p1.x = X.x - Y.y; p1.y = X.y + Y.x;
                V p2; p2.x = X.x + Y.y; p2.y = Y.x - X.y;
                line[m] = p1;
                line[Pt - m] = p2;
            }
        }
    }
    __syncthreads();
    V* phys = smem_fft(a, b, nl, tw, true, rad);
    V* fw = phys == a ? b : a;
    const int nzl = (zt + 1) / 2;
    const T ir = (T)irn[r0 + r];   // 1 / r_j from the plan
    for (int idx = threadIdx.x; idx < zt * Pt; idx += blockDim.x) {
        const int zi = idx / Pt;
        const int th = idx - zi * Pt;
        const V* L0 = phys + (size_t)(zi * 6) * Pt + th;
        const V p0 = L0[0], p1 = L0[Pt], p2 = L0[2 * Pt], p3 = L0[3 * Pt], p4 = L0[4 * Pt], p5 = L0[5 * Pt];
        const T ur = p0.x, ut = p0.y, uz = p4.x;
        const T utr = ut * ir;
        const T Nr = ur * p1.x + utr * p2.x + uz * p3.x - ut * utr;
        const T Nt = ur * p1.y + utr * p2.y + uz * p3.y + utr * ur;
        const T Nz = ur * (p4.y * ids) + utr * p5.x + uz * p5.y;
        V q; q.x = Nr; q.y = Nt;
        fw[(size_t)zi * Pt + th] = q;
        V* zl = fw + (size_t)(zt + zi / 2) * Pt + th;
        if (zi & 1) zl->y = Nz;
        else { zl->x = Nz; if (zi + 1 == zt) zl->y = 0; }
    }
    __syncthreads();
    V* other = fw == a ? b : a;
    V* spec = smem_fft(fw, other, zt + nzl, tw, false, rad);
    for (int idx = threadIdx.x; idx < zt * (M + 1); idx += blockDim.x) {
        const int m = idx / zt;
        const int zi = idx - m * zt;
        const V Q = spec[(size_t)zi * Pt + m];
        const V Qm = spec[(size_t)zi * Pt + (m ? Pt - m : 0)];
        const V* SL = spec + (size_t)(zt + zi / 2) * Pt;
        const V Sp = SL[m], Sm = cconj(SL[m ? Pt - m : 0]);
        V nz;
        if (zi & 1) { nz.x = (T)0.5 * (Sp.y - Sm.y); nz.y = (T)0.5 * (Sm.x - Sp.x); }  // (S - conj S-)/(2i)
        else        { nz.x = (T)0.5 * (Sp.x + Sm.x); nz.y = (T)0.5 * (Sp.y + Sm.y); }
        const size_t o = ((size_t)r * (M + 1) + m) * Pz + z0 + zi;
        H2[o] = Q;
        H2[fstride + o] = cconj(Qm);
        H2[2 * fstride + o] = nz;
    }
}

// theta pass of the mixed form with the generic kernel: FP32 lines (H1, H2 in float2), all rows
tc_status launch_theta32(tc_plan* p, const float2* H1, float2* H2, cudaStream_t s) {
    const int zt = p->zt32;
    const size_t sm2 = (size_t)2 * 6 * zt * p->P_t * sizeof(float2);
    TC_CUDA(p, cudaFuncSetAttribute(k_theta<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm2));
    const int slot = prof_begin(p, kKTheta32, s);
    k_theta<float2><<<p->N_r * (p->P_z / zt), 256, sm2, s>>>(H1, H2, p->d_ir, 0, p->N_r, p->M, p->P_z,
                                                             (double)p->m_p, zt, p->d_tw_t32, p->rad_t, p->d_dsc);
    prof_end(p, slot, s);
    TC_LAUNCHED(p, "k_theta");
    return TC_OK;
}

// The nonlinear term.  FP64: fixed-point lines of p->stage_rows radial rows at a time (tc_fx_z.cu).
// Mixed form: FP32 lines of all rows (tc_mixed.cu).
tc_status launch_nonlinear(tc_plan* p, const double2* u, double2* N, char* ws, cudaStream_t s) {
    if (p->precision == TC_MIXED && p->opt.mean_fp32) {
        TC_TRY_STATUS(launch_nl_pre32(p, u, ws, s, 0, p->M + 1));
        TC_TRY_STATUS(launch_nl_theta32(p, ws, s));
        return launch_nl_post32(p, u, N, ws, s, 0, p->M + 1);
    }
    if (p->precision == TC_MIXED) {
        // the mean mode reads only u: it runs on the plan's second stream beside the FP32
        // transforms, and its sums replace N's (0, 0) coefficients after the forward z pass
        TC_CUDA(p, cudaEventRecord(p->mean_ev[0], s));
        TC_CUDA(p, cudaStreamWaitEvent(p->mean_stream, p->mean_ev[0], 0));
        TC_TRY_STATUS(launch_mean00_part(p, u, ws, p->mean_stream));
        TC_CUDA(p, cudaEventRecord(p->mean_ev[1], p->mean_stream));
        TC_TRY_STATUS(launch_nl_pre32(p, u, ws, s, 0, p->M + 1));
        TC_TRY_STATUS(launch_nl_theta32(p, ws, s));
        TC_TRY_STATUS(launch_nl_post32(p, u, N, ws, s, 0, p->M + 1));
        TC_CUDA(p, cudaStreamWaitEvent(s, p->mean_ev[1], 0));
        return launch_mean00_fin(p, N, ws, s);
    }
    return launch_nonlinear_fx(p, u, N, ws, s);
}

}  // namespace tc
