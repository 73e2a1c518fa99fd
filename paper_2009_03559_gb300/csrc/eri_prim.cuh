// Primitive-quartet set-ups: the prefactor-scaled attenuated Boys values in FP64 and in FP32.
#pragma once
#include "hfx_internal.cuh"

namespace hfx {

// Scalars of one primitive quartet besides its Boys values.
struct PrimScalars {
  double RP, RQ, inv_s, PQ[3];
};

// Primitive-quartet set-up: the prefactor-scaled attenuated Boys values
//   G_m = C_ab C_cd / sqrt(p+q) * (F_m(T) - kappa^{m+1/2} F_m(kappa T)),  m = 0..Lt,
// kappa = omega^2 / (omega^2 + rho), T = rho |PQ|^2 (omega = 0: the Coulomb F_m(T)).  Both
// Boys functions are taken at the top order only; the lower orders come from one downward
// recursion on G itself: with A_m = pref F_m(T) and B_m = pref kappa^{m+1/2} F_m(kappa T),
// F_{m-1}(x) = (2x F_m(x) + e^{-x}) / (2m-1) gives
//   G_{m-1} = (2T G_m + pref e^{-T} - pref kappa^{m-1/2} e^{-kappa T}) / (2m-1).
// Returns false if the quartet is negligible (kappa T beyond the tables: G_m < e^{-60}).
__device__ __forceinline__ bool prim_core(const PrimPair& b, const PrimPair& k, int Lt, double omega, double omega2,
                                          const double* __restrict__ tabs, double* G, PrimScalars& ps,
                                          const Fp64& op) {
  const double p = b.p, q = k.p;
  const double s = op.add(p, q);
  const double y = rsqrt_nr(s, op);   // 1/sqrt(p+q)
  const double inv_s = op.mul(y, y);
  ps.inv_s = inv_s;
  ps.RP = op.mul(q, inv_s);       // rho / p
  ps.RQ = op.mul(p, inv_s);       // rho / q
  const double rho = op.mul(p, ps.RP);
  ps.PQ[0] = op.sub(b.P[0], k.P[0]);
  ps.PQ[1] = op.sub(b.P[1], k.P[1]);
  ps.PQ[2] = op.sub(b.P[2], k.P[2]);
  const double T = op.mul(rho, fma(ps.PQ[0], ps.PQ[0], fma(ps.PQ[1], ps.PQ[1], op.mul(ps.PQ[2], ps.PQ[2]))));
  const double pref = op.mul(op.mul(b.C, k.C), y);
  double F1, e1;
  boys_any(Lt, T, tabs, F1, e1, op);
  const double T2 = op.add(T, T);
  if (omega2 > 0.0) {
    const double sk = op.mul(omega, rsqrt_nr(op.add(rho, omega2), op));   // sqrt(kappa)
    const double kap = op.mul(sk, sk);
    const double kT = op.mul(kap, T);
    if (ge_hi(kT, kBoysXmaxHi)) return false;
    double F2, e2;
    boys_top(Lt, kT, tabs, F2, e2, op);
    // c[m] = pref kappa^{m-1/2}, m = 1..Lt+1
    double c[kMaxLt + 2];
    c[1] = op.mul(pref, sk);
#pragma unroll
    for (int m = 1; m <= kMaxLt; ++m)
      if (m <= Lt) c[m + 1] = op.mul(c[m], kap);
    const double pe1 = op.mul(pref, e1);
    double g = 0.0;
#pragma unroll
    for (int m = 0; m <= kMaxLt; ++m)
      if (m == Lt) g = fma(-c[m + 1], F2, op.mul(pref, F1));
    G[Lt] = g;
#pragma unroll
    for (int m = kMaxLt; m >= 1; --m) {
      if (m <= Lt) {
        g = fma(T2, g, fma(-c[m], e2, pe1)) * (1.0 / (2 * m - 1));
        G[m - 1] = g;
      }
    }
  } else {
    const double pe1 = op.mul(pref, e1);
    double g = op.mul(pref, F1);
    G[Lt] = g;
#pragma unroll
    for (int m = kMaxLt; m >= 1; --m) {
      if (m <= Lt) {
        g = fma(T2, g, pe1) * (1.0 / (2 * m - 1));
        G[m - 1] = g;
      }
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// FP32 set-up (FP32 passes of the mixed-precision build).  With a = m + 1/2,
//   F_m(T) - kappa^a F_m(kappa T) = 1/2 T^{-a} (Gamma(a, kappa T) - Gamma(a, T)),
// because F_m(x) = 1/2 x^{-a} gamma(a, x) and gamma(a, x) = Gamma(a) - Gamma(a, x).  So with
// A_m = 1/2 T^{-a} Gamma(a, kappa T) and B_m = 1/2 T^{-a} Gamma(a, T), from Gamma(1/2, x) =
// sqrt(pi) erfc(sqrt x) and Gamma(a + 1, x) = a Gamma(a, x) + x^a e^{-x}:
//   A_0 = 1/2 sqrt(pi/T) erfc(sqrt(kappa T)),  A_{m+1} = ((m + 1/2) A_m + 1/2 kappa^{m+1/2} e^{-kappa T}) / T,
//   B_0 = 1/2 sqrt(pi/T) erfc(sqrt(T)),        B_{m+1} = ((m + 1/2) B_m + 1/2 e^{-T}) / T.
// Every term is positive, so this upward recursion keeps FP32's relative accuracy at any T; the
// one subtraction, G_m = pref (A_m - B_m), loses at most a factor 1 / (1 - B_m / A_m).  Where
// B_m > A_m / 64 for some m (T (1 - kappa) small: close or diffuse pairs) the primitive quartet
// takes the FP64 set-up instead.  P - Q is formed in FP64 (3 instructions), so that T keeps
// FP32's relative accuracy for centres far from the origin; nothing else runs on the FP64 pipe.
// ---------------------------------------------------------------------------
struct PrimScalarsF {
  float RP, RQ, inv_s, PQ[3];
};

enum { F32_SKIP = 0, F32_OK = 1, F32_FP64 = 2 };

__device__ __forceinline__ int prim_core_f32(const PrimPair& b, const PrimPair& k, int Lt, float omega_f, float* G,
                                             PrimScalarsF& ps, const Fp64& op) {
  const float p = b.pf, q = k.pf;
  const float y = rsqrtf(p + q);  // 1/sqrt(p+q)
  const float inv_s = y * y;
  ps.inv_s = inv_s;
  ps.RP = q * inv_s;
  ps.RQ = p * inv_s;
  const float rho = p * ps.RP;
  ps.PQ[0] = to_f32(op.sub(b.P[0], k.P[0]));
  ps.PQ[1] = to_f32(op.sub(b.P[1], k.P[1]));
  ps.PQ[2] = to_f32(op.sub(b.P[2], k.P[2]));
  const float T = rho * fmaf(ps.PQ[0], ps.PQ[0], fmaf(ps.PQ[1], ps.PQ[1], ps.PQ[2] * ps.PQ[2]));
  const float sk = omega_f * rsqrtf(fmaf(omega_f, omega_f, rho));  // sqrt(kappa)
  const float kap = sk * sk;
  const float kT = kap * T;
  if (kT >= 60.0f) return F32_SKIP;  // as the FP64 set-up: G_m < e^{-60}
  const float pref = to_f32(b.C) * to_f32(k.C) * y;
  const float yT = rsqrtf(T);
  const float invT = yT * yT;
  const float c0 = 0.886226925f * yT;  // sqrt(pi) / 2 / sqrt(T)
  float A = c0 * erfcf(sqrtf(kT));
  float B = c0 * erfcf(sqrtf(T));
  const float hk = 0.5f * expf(-kT), h1 = 0.5f * expf(-T);
  // accepted only with B_m <= A_m / 64 and A_m finite at every order (on this path A_m stays far
  // below 1: T (1 - kappa) is not small); T near 0 overflows the recursion and is declined
  bool ok = (B <= A * (1.0f / 64.0f)) && (A <= 1e30f);
  G[0] = pref * (A - B);
  float kp = sk;  // kappa^{m+1/2}
#pragma unroll
  for (int m = 0; m < kMaxLt; ++m) {
    if (m < Lt) {
      const float a = (float)m + 0.5f;
      A = fmaf(a, A, kp * hk) * invT;
      B = fmaf(a, B, h1) * invT;
      kp *= kap;
      ok = ok && (B <= A * (1.0f / 64.0f)) && (A <= 1e30f);
      G[m + 1] = pref * (A - B);
    }
  }
  return ok ? F32_OK : F32_FP64;
}

}  // namespace hfx
