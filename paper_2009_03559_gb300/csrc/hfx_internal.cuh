// Internal device-side definitions of the HFX library (not part of the C ABI).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace hfx {

// ---------------------------------------------------------------------------
// Per-class recurrence description (generated tables, see gen_eri_tables.py)
// ---------------------------------------------------------------------------
struct EriClassInfo {
  int la, lb, lc, ld, E, F, Lt;
  int n_acc, work_base, scratch;       // group scratch (doubles): acc | VRR slots
  int n_bra_lv, n_ket_lv;
  int lv_off[8], lv_n[8];              // VRR levels: op offset (in uint4) and count
  int acc_off;                         // into kAccSrc: (acc index | slot << 16) entries
  int n_accl;                          // accumulators added after the levels (others are
                                       // accumulated by the op that makes them)
  int n_post;                          // post-contraction stages
  int post_type[8], post_off[8], post_n[8];  // 0 bra HRR, 1 ket HRR, 2 spherical
  int out_base;                        // final spherical block in group scratch
  int dims[4];                         // final block extents (a, b, c, d)
  int flops_prim, flops_quartet;       // flop model (VRR+acc per primitive quartet;
                                       // HRR+spherical+digest per contracted quartet)
  int flops_digest;                    // the digest part of flops_quartet (always FP64)
};

extern const EriClassInfo* class_info_host();

// Hermite engine (generated tables, see gen_md_tables.py): the steps of a class ...
struct MdClassInfo {
  int Lt;
  int kc, n_kc, bc, n_bc;              // contraction tables (first entry, entries)
  int n_row, nab, ncd;                 // rows of Y, function pairs of bra and ket
  int bra_coef0, bra_coef, bra_set;    // bra pair type: first coefficient, coefficients, sets
  int ket_coef, ket_set;
  int z1_round, z1_n, z1_dst, z2_round, z2_n, z2_dst;  // transformation passes
  int dig, dig_n;                      // digest (first round, rounds)
};
// ... and the sets and coefficients of a pair type (set: power of 1/2p | of u_b << 4 | of u_a << 8)
struct MdPairInfo {
  int coef0, n_coef, n_set;
  int set[14];
};
extern const MdClassInfo* md_class_host();
extern const MdPairInfo* md_pair_host();
// per class: flops per primitive quartet, per run of a bra primitive pair, per quartet, in its digest
extern const int (*md_flops_host())[4];

// ---------------------------------------------------------------------------
// Boys function tables, one per order L = 0..kMaxLt, with F_m(x) = int_0^1 u^{2m} exp(-x u^2) du.
// A row holds the Taylor coefficients about its grid point x_g in powers of d = x - x_g:
//   doubles [0] x_g, [1..3] f_0, f_1, f_2, [4] e_0 = exp(-x_g), [5] e_0 / 2, then floats
//   [12..14] f_3, f_4, f_5;  f_k = (-1)^k F_{L+k}(x_g) / k!,  exp(-x) = e_0 - e_0 d + e_0/2 d^2 - ...
// Rows 0..kBoysRows-1: x_g = g / 256 up to 60.  |d| <= 1/512, so the terms from the third on are
// below 1.3e-9 of the value and their FP32 rounding below 8e-17: they cost no FP64 instruction
// (with the former spacing of 1/32 both chains had six).  The rows after them hold the asymptote
// (2L-1)!!/2^{L+1} sqrt(pi) t^{-L-1/2} for t = 1 + g / 1024 in [1, 4], e_0 = 0: T >= 60 is looked
// up as t = T / 4^k and the value scaled by 2^{-k(2L+1)}, exponent arithmetic on the integer pipe
// (the neglected part of F_L is below exp(-60) relative).
// ---------------------------------------------------------------------------
constexpr int kBoysRowLen = 8;
constexpr int kBoysPerUnit = 256;
constexpr double kBoysXmax = 60.0;
constexpr int kBoysXmaxHi = 0x404E0000;   // high word of 60.0 (low word 0)
constexpr int kBoysRows = 60 * kBoysPerUnit + 2;
constexpr int kBoysTailPerUnit = 1024;
constexpr int kBoysTailRows = 3 * kBoysTailPerUnit + 1;
constexpr int kMaxLt = 8;
constexpr int kBoysTableLen = (kBoysRows + kBoysTailRows) * kBoysRowLen;   // doubles per order

// ---------------------------------------------------------------------------
// Primitive-pair record (one per surviving primitive pair of a shell pair).
// C = sqrt(2) pi^{5/4} w_a w_b exp(-ab/p |AB|^2) / p so that the primitive
// quartet prefactor 2 pi^{5/2} K_ab K_cd / (p q sqrt(p+q)) = C_ab C_cd / sqrt(p+q).
// For a basis whose Hermite integrals could leave FP64's range (hfx_ctx::hexp, 0 for any other) C is held
// times 2^{hexp/2}; the transformation coefficients T of a pair (PairArrays::md) carry the inverse.
// ---------------------------------------------------------------------------
struct __align__(16) PrimPair {
  double p, inv2p;     // exponent sum and 1/(2p)
  double P[3];         // Gaussian product centre
  double PA[3];        // P - A (A = centre of the pair's first shell)
  double C;            // prefactor (see above)
  double inv2p3;       // 3/(2p)
  double ua, ub;       // a/p and b/p, a and b the exponents of the pair's two shells
  // FP32 copies for the FP32 recurrences
  float pf, inv2pf, PAf[3], Pf[3];
};

// Device arrays describing shell pairs (indexed by candidate-pair id).
struct PairArrays {
  const int* sa;            // first shell (l_a >= l_b)
  const int* sb;            // second shell
  const int* prim_off;      // first PrimPair of the pair
  const int* prim_n;        // number of surviving primitive pairs
  const double* AB;         // 3 per pair: A - B
  const PrimPair* prim;     // primitive-pair records
  const long long* md_off;  // first double of the pair's Hermite data in md: the coefficients T of its
  const double* md;         // type, then the factors W of every surviving primitive pair
};

struct ShellArrays {
  const int* bf_off;        // first function of each shell
  const int* atom;          // atom of each shell
};

// ---------------------------------------------------------------------------
// Conversions and reciprocals that keep the FP64 pipe free.  On this part the FP64 pipe
// executes one warp instruction every 16 SM cycles whatever the number of active lanes,
// while integer, FP32 and special-function units are some 64 times wider, so the FP32 seeds
// of reciprocals are made from the bit patterns of the doubles.
// ---------------------------------------------------------------------------
// FP32 value of a double x in [2^-126, 2^128) by truncation of the mantissa (0 below).
__device__ __forceinline__ float approx_f32(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int fb = (int)(((unsigned)(hi - (896 << 20)) << 3) | (lo >> 29));
  return __int_as_float(hi < (897 << 20) ? 0 : fb);
}
// Double with the value 2^e2 * f of a positive normal float f (e2 = 0 or -1): exact.
__device__ __forceinline__ double widen_f32(float f, int e2 = 0) {
  const int fb = __float_as_int(f);
  return __hiloint2double((fb >> 3) + ((896 + e2) << 20), fb << 29);
}
// 2^e x for a positive normal double x (exact; e small).
__device__ __forceinline__ double scale2(double x, int e) {
  return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}
// 2^e x, e > 0, for any x but 0 and subnormals (at most 2^e 2^-1022 comes of those); what overflows and
// what is not finite stays not finite.
__device__ __forceinline__ double scale_up(double x, int e) {
  const int hi = __double2hiint(x);
  return __hiloint2double((hi & 0x7fffffff) >= ((0x7ff - e) << 20) ? hi | 0x7ff00000 : hi + (e << 20),
                          __double2loint(x));
}
// x >= 2^e... comparisons of non-negative doubles on the high word (integer units).
__device__ __forceinline__ bool ge_hi(double x, int hi) { return __double2hiint(x) >= hi; }

// FP32 value of any finite double by truncation of the mantissa (relative error below
// 2^-23): magnitudes below 2^-126 give 0, above 2^128 are not expected.
__device__ __forceinline__ float to_f32(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const int mag = hi & 0x7fffffff;
  const unsigned fb = ((unsigned)(mag - (896 << 20)) << 3) | (lo >> 29);
  return __int_as_float((int)((mag < (897 << 20) ? 0u : fb) | ((unsigned)hi & 0x80000000u)));
}
// FP32 value of a double by rounding to nearest (ties away from zero), on the integer units;
// magnitudes below 2^-126 give 0, above 2^128 are not expected.
__device__ __forceinline__ float to_f32_rn(double x) {
  return to_f32(__longlong_as_double(__double_as_longlong(x) + (1ll << 28)));
}
// Exact double of a float (subnormal floats give 0).
__device__ __forceinline__ double to_f64(float f) {
  const int fb = __float_as_int(f);
  const int mag = fb & 0x7fffffff;
  if (mag < 0x00800000) return 0.0;
  return __hiloint2double(((mag >> 3) + (896 << 20)) | (fb & (int)0x80000000), mag << 29);
}

// ---------------------------------------------------------------------------
// FP64 instructions with three vector-register operands.  A DFMA of three registers takes 16
// cycles of an SM; DADD, DMUL and a DFMA with a constant, immediate or zero-register operand take
// 19 (measured: chains of each form on 8 warps, 16.00 and 19.00 cycles per warp instruction).  So
// sums and products are written as a DFMA with 1 or -0 from a register that the compiler cannot
// see through; both are exact, so the results are those of the plain operations.
// ---------------------------------------------------------------------------
constexpr int kFp64Recip = 8;
static __device__ double kFp64Operands[kFp64Recip + kMaxLt + 1] = {
    1.0, -0.0, 3.0, 5.0, 7.0, 0.0, 0.0, 0.0,              // one, -0, multipliers
    -1.0, 1.0, 1.0 / 3, 1.0 / 5, 1.0 / 7, 1.0 / 9, 1.0 / 11, 1.0 / 13, 1.0 / 15};  // [kFp64Recip + m] 1 / (2m - 1)
// operand i, loaded where this stands (not hoisted: registers are scarce) ...
__device__ __forceinline__ double fp64_operand(int i) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(kFp64Operands + i));
  return v;
}
// ... and the two of all sums and products, held by a kernel from its start
struct Fp64 {
  double one, nzero;
  __device__ __forceinline__ void init() {
    one = fp64_operand(0);
    nzero = fp64_operand(1);
  }
  __device__ __forceinline__ double mul(double a, double b) const { return __fma_rn(a, b, nzero); }
  __device__ __forceinline__ double add(double a, double b) const { return __fma_rn(a, one, b); }
  __device__ __forceinline__ double sub(double a, double b) const { return __fma_rn(-b, one, a); }
};

// 1/sqrt(x) for x > 0 in FP32 range: FP32 hardware seed (relative error below 2^-22),
// one Newton-Raphson step (the error squares: below 1e-13 relative).  3 FP64 instructions.
__device__ __forceinline__ double rsqrt_nr(double x, const Fp64& op) {
  const float yf = rsqrtf(approx_f32(x));
  const double y = widen_f32(yf);
  const double hy = widen_f32(yf, -1);            // y / 2
  const double r = fma(-op.mul(x, y), y, op.one); // 1 - x y^2
  return fma(hy, r, y);
}

// F_L(x) and exp(-x) from row g of the table of order L: 7 FP64 instructions.
__device__ __forceinline__ void boys_row(double x, const double* __restrict__ tabL, int g, double& F, double& e,
                                         const Fp64& op) {
  // (no argument leads past the table: a NaN from coordinates that overflowed takes its last row)
  g = (int)min((unsigned)g, (unsigned)(kBoysRows + kBoysTailRows - 1));
  const double2* row = reinterpret_cast<const double2*>(tabL + g * kBoysRowLen);
  const double2 r0 = __ldg(row), r1 = __ldg(row + 1), r2 = __ldg(row + 2);
  const float4 r3 = __ldg(reinterpret_cast<const float4*>(row + 3));
  const double d = op.sub(x, r0.x);
  const float df = to_f32(d), ef = to_f32(r2.x);
  const double f3 = to_f64(fmaf(df, fmaf(df, r3.z, r3.y), r3.x));
  const double e3 = to_f64(ef * fmaf(df, fmaf(df, -1.0f / 120, 1.0f / 24), -1.0f / 6));
  F = fma(fma(fma(f3, d, r1.y), d, r1.x), d, r0.y);
  e = fma(fma(fma(e3, d, r2.y), d, -r2.x), d, r2.x);
}

// the same for 0 <= x < kBoysXmax
__device__ __forceinline__ void boys_top(double x, const double* __restrict__ tabL, double& F, double& e,
                                         const Fp64& op) {
  boys_row(x, tabL, __float2int_rn(approx_f32(x) * (float)kBoysPerUnit), F, e, op);
}

// F_L(x) and exp(-x) (0 from kBoysXmax on) for any x >= 0, by one sequence of instructions
__device__ __forceinline__ void boys_any(int L, double x, const double* __restrict__ tabL, double& F, double& e,
                                         const Fp64& op) {
  const bool tail = ge_hi(x, kBoysXmaxHi);
  const int k = tail ? ((__double2hiint(x) >> 20) - 1023) >> 1 : 0;
  const double t = scale2(x, -2 * k);
  const float f = approx_f32(t);
  const int g = tail ? kBoysRows + __float2int_rn((f - 1.0f) * (float)kBoysTailPerUnit)
                     : __float2int_rn(f * (float)kBoysPerUnit);
  boys_row(t, tabL, g, F, e, op);
  if (tail) {
    const int hi = __double2hiint(F), up = k * (2 * L + 1);
    F = (hi >> 20) > up ? scale2(F, -up) : 0.0;
  }
}

// Lattice images (periodic builds): the library holds the home cell's shells repeated in a
// box of cells (the image shells, cell-major, the home cell first); every pair of the pair
// list has one shell in the home cell (list-IJ anchored in the home cell, Sec. 3.1).
struct PerCell;
struct PeriodicInfo {
  const int* shell_cell;            // image shell -> cell index (0 = home cell)
  const int* shell_bf;              // image shell -> first function in the home-cell numbering
  const int* cell_xyz;              // cell index -> integer cell coordinates (3 each)
  const unsigned char* home_first;  // candidate pair -> 1 if its first shell is the home-cell one
  const int* rmap;                  // density block index of cell R (-1: absent), R in [-rb, rb]^3
  int rb;
  const double* P;                  // density blocks P^R, n_R x nbf x nbf
  int nbf;
  const double* pmax;               // max |P^R| per (R, home shell, home shell): n_R x nsh x nsh
  int nsh;                          // shells of the home cell
  const PerCell* cells;             // the launch's passes over the quartet list of the class
  long long n_list;                 // quartets of the list
};

// A pass over the list of a class: quartets (bra | ket + shift) of cell G; reverse = 0: the bra pair
// carries the row function of K^G, 1: the ket pair does (the pass then evaluates (q | p - G L) for
// the quartet (p | q + G L) of a lower bra class)
struct PerCell {
  double shift[3];
  double* KG;  // K^G, nbf x nbf
  int gcell[3];
  int reverse;
};

// Arguments of one class launch (passed by value).
struct EriLaunch {
  EriClassInfo ci;
  PairArrays pa;
  ShellArrays sh;
  const int* sorted;          // sorted pair index -> candidate-pair id
  const long long* qoff;      // exclusive scan of quartets per row (global), + total
  int row_begin, row_end;     // rows of this class pair
  int bra_bin_start, ket_bin_start;
  long long q_begin, q_count; // quartet range of this class pair
  int schedule;               // 0 quartet split, 1 bra-pair split, 2 dynamic chunks
  unsigned long long* work;   // schedule 2: next unclaimed quartet (relative to q_begin)
  int chunk;                  // schedule 2: quartets per claim
  const double* boys;         // kMaxLt + 1 tables of kBoysTableLen doubles
  double omega, omega2;
  double unscale;             // 2^-hexp (see PrimPair::C): the thread kernel's factor for its integrals
  MdClassInfo mc;              // Hermite engine: the steps of this class
  int prec;                    // precision pass (PREC_*)
  const double* P;
  double* K;
  int ld;
  // Schwarz-diagonal mode: quartet (p|p) for candidate pairs [diag_begin, diag_end)
  const int* diag_list;
  int diag_n;
  double* diag_Q;
  unsigned long long* busy;     // optional per-SM globaltimer busy ns (indexed by %smid)
  unsigned long long* counters; // optional: [0] primitive quartets evaluated, [1] quartets, [2] skipped
  const double* pmax;           // optional: max |P| of each shell-pair block (ns x ns)
  int ns;
  int skip_zero;                // skip quartets whose four density blocks are all zero
  int fp32_ok;                  // mixed precision allowed for this class
  double fp32_tau;              // FP32 iff Q_IJ Q_KL Pmax < fp32_tau, Pmax = max|P_blocks| ...
  const double* pglob;          // ... or, when non-NULL, *pglob = max |P| over the matrix
  double dens_tau;              // > 0: drop quartets with Q_IJ Q_KL max|P_blocks| < dens_tau
  double dist_tau;              // > 0: drop quartets with Q_IJ Q_KL exp(-kappa rho R^2) < dist_tau
  const double* dist;           // per sorted pair: most diffuse primitive-pair centre (3), spread,
                                // smallest exponent sum (5 doubles)
  const double* Qs;             // Schwarz factor of each sorted pair
  // batched launch (n_sys > 0): quartets of all systems' lists for this class, concatenated;
  // seg[s] = first index of system s (seg[n_sys] = total = q_count); batch[s] = that
  // system's record for this class (device memory)
  int n_sys;
  const long long* seg;
  const EriLaunch* batch;
  // periodic launch: the list of the class once for each of per.cells (q_count = all of them)
  PeriodicInfo per;
};


}  // namespace hfx
