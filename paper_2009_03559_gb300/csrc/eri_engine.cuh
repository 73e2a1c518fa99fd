// Table-driven engine for contracted shell quartets (ab|cd) with the erfc(omega r)/r
// kernel, fused with the exchange-matrix digest: the thread kernel, which runs on request
// (hfx_set_group_size(1)); the default for every class is the Hermite engine (hfx_md.cuh).  It runs in
// FP64; the recurrence and contraction steps are templated on the arithmetic type, and an FP32
// primitive set-up (prim_core_f32) feeds them, so the mixed-precision kernel runs set-up, recurrences
// and contraction in FP32 for the quartets that qualify (HRR, spherical step and digest in FP64).
//
// One thread evaluates one contracted quartet:
//   1. for every surviving primitive quartet: the Boys step (G_m = F_m(T) -
//      kappa^{m+1/2} F_m(kappa T), times the prefactor), then the Obara-Saika vertical
//      recurrence level by level, then the contraction into the accumulator block (e0|f0);
//   2. the post-contraction stages: Head-Gordon-Pople horizontal recurrence on the bra,
//      Cartesian -> spherical on a and b, HRR on the ket, spherical on c and d;
//   3. the digest into the half exchange matrix A (K = A + A^T afterwards):
//      A_ac += sum_bd v P_bd, A_ad += sum_bc v P_bc, A_bc += sum_ad v P_ad,
//      A_bd += sum_ac v P_ac, with v = deg (ab|cd), deg = 1/2^[a=b] 1/2^[c=d] 1/2^[ab=cd].
// The per-class op lists come from gen_eri_tables.py (eri_tables.inc).
#pragma once
#include <type_traits>
#include "eri_prim.cuh"

namespace hfx {

#define HFX_TABLE_QUAL __device__ __align__(16) const
#include "eri_tables.inc"
#undef HFX_TABLE_QUAL

__device__ __constant__ double kSphCoef[6] = {0.0, 1.0, -0.28867513459481287, 0.57735026918962573,
                                              0.5, -0.5};
__device__ __constant__ float kSphCoefF[6] = {0.0f, 1.0f, -0.28867513459481287f, 0.57735026918962573f,
                                              0.5f, -0.5f};

// fused multiply-add in the precision of the arguments (an unqualified fma() on floats
// would promote to FP64, which runs on the FP64 pipe together with the conversions)
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename R>
__device__ __forceinline__ R sph_coef(int i);
template <>
__device__ __forceinline__ float sph_coef<float>(int i) { return kSphCoefF[i]; }
template <>
__device__ __forceinline__ double sph_coef<double>(int i) { return kSphCoef[i]; }

// Coefficients held in registers (one quartet per thread); selects avoid indexed
// register arrays.
template <typename R>
struct CoefRgT {
  R PA[3], WP[3], QC[3], WQ[3];
  R ca1, ca2, ca3, RP, ck1, ck2, ck3, RQ, cb1, cb2, cb3, cb4;
  __device__ __forceinline__ R pa(int i) const { return i == 0 ? PA[0] : (i == 1 ? PA[1] : PA[2]); }
  __device__ __forceinline__ R wp(int i) const { return i == 0 ? WP[0] : (i == 1 ? WP[1] : WP[2]); }
  __device__ __forceinline__ R qc(int i) const { return i == 0 ? QC[0] : (i == 1 ? QC[1] : QC[2]); }
  __device__ __forceinline__ R wq(int i) const { return i == 0 ? WQ[0] : (i == 1 ? WQ[1] : WQ[2]); }
  __device__ __forceinline__ R ca(int n) const { return n == 1 ? ca1 : (n == 2 ? ca2 : ca3); }
  __device__ __forceinline__ R ck(int n) const { return n == 1 ? ck1 : (n == 2 ? ck2 : ck3); }
  __device__ __forceinline__ R cb(int n) const { return n == 1 ? cb1 : (n == 2 ? cb2 : (n == 3 ? cb3 : cb4)); }
  __device__ __forceinline__ R rp() const { return RP; }
  __device__ __forceinline__ R rq() const { return RQ; }
};
using CoefRg = CoefRgT<double>;

// FP32 copy of a coefficient set (conversions on the integer units, see to_f32)
__device__ __forceinline__ CoefRgT<float> coef_f32(const CoefRg& c, int E, int F) {
  CoefRgT<float> f;
  if (E > 0) {
    for (int i = 0; i < 3; ++i) {
      f.PA[i] = to_f32(c.PA[i]);
      f.WP[i] = to_f32(c.WP[i]);
    }
    f.ca1 = to_f32(c.ca1); f.ca2 = to_f32(c.ca2); f.ca3 = to_f32(c.ca3); f.RP = to_f32(c.RP);
  }
  if (F > 0) {
    for (int i = 0; i < 3; ++i) {
      f.QC[i] = to_f32(c.QC[i]);
      f.WQ[i] = to_f32(c.WQ[i]);
    }
    f.ck1 = to_f32(c.ck1); f.ck2 = to_f32(c.ck2); f.ck3 = to_f32(c.ck3); f.RQ = to_f32(c.RQ);
    f.cb1 = to_f32(c.cb1); f.cb2 = to_f32(c.cb2); f.cb3 = to_f32(c.cb3); f.cb4 = to_f32(c.cb4);
  }
  return f;
}

// Set-up into registers (one quartet per thread).
__device__ __forceinline__ bool prim_setup(const PrimPair& b, const PrimPair& k, int E, int F, int Lt, double omega,
                                           double omega2, const double* __restrict__ tabs, CoefRg& c, double* Gm,
                                           const Fp64& op) {
  PrimScalars ps;
  if (!prim_core(b, k, Lt, omega, omega2, tabs, Gm, ps, op)) return false;
  if (E > 0) {
    c.PA[0] = b.PA[0]; c.PA[1] = b.PA[1]; c.PA[2] = b.PA[2];
    c.WP[0] = -ps.RP * ps.PQ[0]; c.WP[1] = -ps.RP * ps.PQ[1]; c.WP[2] = -ps.RP * ps.PQ[2];   // W - P
    c.ca1 = b.inv2p; c.ca2 = scale2(b.inv2p, 1); c.ca3 = b.inv2p3;
    c.RP = ps.RP;
  }
  if (F > 0) {
    c.QC[0] = k.PA[0]; c.QC[1] = k.PA[1]; c.QC[2] = k.PA[2];
    c.WQ[0] = ps.RQ * ps.PQ[0]; c.WQ[1] = ps.RQ * ps.PQ[1]; c.WQ[2] = ps.RQ * ps.PQ[2];      // W - Q
    c.ck1 = k.inv2p; c.ck2 = scale2(k.inv2p, 1); c.ck3 = k.inv2p3;
    c.RQ = ps.RQ;
    c.cb1 = scale2(ps.inv_s, -1); c.cb2 = ps.inv_s; c.cb3 = 1.5 * ps.inv_s; c.cb4 = scale2(ps.inv_s, 1);
  }
  return true;
}

// Register coefficients from the FP32 set-up (one quartet per thread).
__device__ __forceinline__ int prim_setup_f32(const PrimPair& b, const PrimPair& k, int E, int F, int Lt,
                                              float omega_f, CoefRgT<float>& c, float* G, const Fp64& op) {
  PrimScalarsF ps;
  const int st = prim_core_f32(b, k, Lt, omega_f, G, ps, op);
  if (st != F32_OK) return st;
  if (E > 0) {
    c.PA[0] = b.PAf[0]; c.PA[1] = b.PAf[1]; c.PA[2] = b.PAf[2];
    c.WP[0] = -ps.RP * ps.PQ[0]; c.WP[1] = -ps.RP * ps.PQ[1]; c.WP[2] = -ps.RP * ps.PQ[2];
    c.ca1 = b.inv2pf; c.ca2 = 2.0f * b.inv2pf; c.ca3 = 3.0f * b.inv2pf;
    c.RP = ps.RP;
  }
  if (F > 0) {
    c.QC[0] = k.PAf[0]; c.QC[1] = k.PAf[1]; c.QC[2] = k.PAf[2];
    c.WQ[0] = ps.RQ * ps.PQ[0]; c.WQ[1] = ps.RQ * ps.PQ[1]; c.WQ[2] = ps.RQ * ps.PQ[2];
    c.ck1 = k.inv2pf; c.ck2 = 2.0f * k.inv2pf; c.ck3 = 3.0f * k.inv2pf;
    c.RQ = ps.RQ;
    c.cb1 = 0.5f * ps.inv_s; c.cb2 = ps.inv_s; c.cb3 = 1.5f * ps.inv_s; c.cb4 = 2.0f * ps.inv_s;
  }
  return F32_OK;
}

__device__ __forceinline__ uint4 ld_op(const uint32_t* base, int idx) {
  return __ldg(reinterpret_cast<const uint4*>(base) + idx);
}

// VRR ops.  bra:  v = PA_i V[s1] + WP_i V[s2] (+ n/(2p) (V[s3] - rho/p V[s4]))
//           ket:  v = QC_i V[s1] + WQ_i V[s2] (+ n/(2q) (V[s3] - rho/q V[s4]))
//                                             (+ e_i/(2(p+q)) V[s5])
// The result is stored to V[dst]; ops flagged "acc" (targets no op reads) instead add it
// to the accumulator S[dst], starting their FMA chain from the accumulator value.
// FOLD = false compiles the plain form (no accumulator branch) for classes without folding.
template <bool FOLD, typename R, class Coef>
__device__ __forceinline__ void vrr_bra(uint4 op, R* V, R* S, int st, const Coef& c) {
  const int dst = op.x & 0xFFFF, s1 = op.x >> 16, s2 = op.y & 0xFFFF, s3 = op.y >> 16, s4 = op.z & 0xFFFF;
  const int i = op.w & 3, nA = (op.w >> 2) & 7;
  const bool acc = FOLD && ((op.w >> 8) & 1);
  R v = acc ? fmar(c.pa(i), V[s1 * st], S[dst * st]) : c.pa(i) * V[s1 * st];
  v = fmar(c.wp(i), V[s2 * st], v);
  if (nA) v = fmar(c.ca(nA), fmar(-c.rp(), V[s4 * st], V[s3 * st]), v);
  if (acc)
    S[dst * st] = v;
  else
    V[dst * st] = v;
}

template <bool FOLD, typename R, class Coef>
__device__ __forceinline__ void vrr_ket(uint4 op, R* V, R* S, int st, const Coef& c) {
  const int dst = op.x & 0xFFFF, s1 = op.x >> 16, s2 = op.y & 0xFFFF, s3 = op.y >> 16;
  const int s4 = op.z & 0xFFFF, s5 = op.z >> 16;
  const int i = op.w & 3, nA = (op.w >> 2) & 7, nB = (op.w >> 5) & 7;
  const bool acc = FOLD && ((op.w >> 8) & 1);
  R v = acc ? fmar(c.qc(i), V[s1 * st], S[dst * st]) : c.qc(i) * V[s1 * st];
  v = fmar(c.wq(i), V[s2 * st], v);
  if (nA) v = fmar(c.ck(nA), fmar(-c.rq(), V[s4 * st], V[s3 * st]), v);
  if (nB) v = fmar(c.cb(nB), V[s5 * st], v);
  if (acc)
    S[dst * st] = v;
  else
    V[dst * st] = v;
}

// Post-contraction op on the group scratch S.
template <typename R>
__device__ __forceinline__ void post_op(uint4 op, int type, R* S, int st, const R* AB, const R* CD) {
  const int dst = op.x & 0xFFFF, s1 = op.x >> 16, s2 = op.y & 0xFFFF, s3 = op.y >> 16;
  R v;
  if (type == 2) {
    const int c0 = op.z & 15, c1 = (op.z >> 4) & 15, c2 = (op.z >> 8) & 15;
    v = sph_coef<R>(c0) * S[s1 * st];
    if (c1) v = fmar(sph_coef<R>(c1), S[s2 * st], v);
    if (c2) v = fmar(sph_coef<R>(c2), S[s3 * st], v);
  } else {
    const int i = (op.z >> 12) & 3;
    const R d = (type == 0) ? AB[i] : CD[i];
    v = fmar(d, S[s2 * st], S[s1 * st]);
  }
  S[dst * st] = v;
}

// Digest of the final spherical block v (stride st) into the half matrix A.
// Outputs o in [o0, nout) step ostep (lanes of the group).
template <typename R>
__device__ __forceinline__ void digest(const EriClassInfo& ci, const R* v, int st, int A, int B,
                                       int C, int D, double deg, const double* __restrict__ P,
                                       double* K, int ld, int o0, int ostep) {
  const int na = ci.dims[0], nb = ci.dims[1], nc = ci.dims[2], nd = ci.dims[3];
  const int nAC = na * nc, nAD = na * nd, nBC = nb * nc, nBD = nb * nd;
  const int nout = nAC + nAD + nBC + nBD;
  for (int o = o0; o < nout; o += ostep) {
    double acc = 0.0;
    int row, col;
    if (o < nAC) {
      const int a = o / nc, c = o - a * nc;
      for (int b = 0; b < nb; ++b)
        for (int d = 0; d < nd; ++d)
          acc = fma((double)v[(((a * nb + b) * nc + c) * nd + d) * st], __ldg(P + (size_t)(B + b) * ld + D + d), acc);
      row = A + a; col = C + c;
    } else if (o < nAC + nAD) {
      const int t = o - nAC, a = t / nd, d = t - a * nd;
      for (int b = 0; b < nb; ++b)
        for (int c = 0; c < nc; ++c)
          acc = fma((double)v[(((a * nb + b) * nc + c) * nd + d) * st], __ldg(P + (size_t)(B + b) * ld + C + c), acc);
      row = A + a; col = D + d;
    } else if (o < nAC + nAD + nBC) {
      const int t = o - nAC - nAD, b = t / nc, c = t - b * nc;
      for (int a = 0; a < na; ++a)
        for (int d = 0; d < nd; ++d)
          acc = fma((double)v[(((a * nb + b) * nc + c) * nd + d) * st], __ldg(P + (size_t)(A + a) * ld + D + d), acc);
      row = B + b; col = C + c;
    } else {
      const int t = o - nAC - nAD - nBC, b = t / nd, d = t - b * nd;
      for (int a = 0; a < na; ++a)
        for (int c = 0; c < nc; ++c)
          acc = fma((double)v[(((a * nb + b) * nc + c) * nd + d) * st], __ldg(P + (size_t)(A + a) * ld + C + c), acc);
      row = B + b; col = D + d;
    }
    atomicAdd(K + (size_t)row * ld + col, deg * acc);
  }
}

}  // namespace hfx
