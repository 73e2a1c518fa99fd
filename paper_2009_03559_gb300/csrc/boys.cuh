// Attenuated-kernel arithmetic that needs care: conversions beside the FP64 pipe, FP64 operands, the
// Boys function and its tables.  Only CUDA's bit casts, FMAs and read-only loads are used, so that the
// tables and look-ups can be compiled for the host and checked there.
#pragma once
#include <cmath>
#include <cstdint>

namespace hfx {

constexpr int kMaxLt = 8;

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

// ---------------------------------------------------------------------------
// Boys function tables: F_m(x) = int_0^1 u^{2m} exp(-x u^2) du and exp(-x) from Taylor rows about grid
// points x_g, in powers of d = x - x_g.
//   per order L = 0..kMaxLt rows of 6 doubles: f_0, f_1, f_2, f_3, then the floats f_4, f_5, f_6, 0 in units
//   of 2^8 ulp(f_2);  f_k = (-1)^k F_{L+k}(x_g) / k!;  rows 0..kBoysRows-1 at x_g = g / 75 (an FP32 product) up
//   to 60, then kBoysTailRows rows of the asymptote (2L-1)!!/2^{L+1} sqrt(pi) t^{-L-1/2} at 512 points an octave
//   of t in [1, 4]: T >= 60 is looked up as t = T / 4^k and the value scaled by 2^{-k(2L+1)}, exponent arithmetic
//   on the integer pipe (the neglected part of F_L is below exp(-60) relative; exp(-T) counts as 0);
//   then for all orders the rows (e_0, e_0 / 6), e_0 = exp(-x_g), up to 60.  2.5 MB in all.
// The terms up to the third order are held and summed in FP64.  The ones from the fourth on, at |d| <= 1/150
// (and 1/1024 of t) at most 8.3e-11 of exp(-x), 5.7e-11 of F_L and 3.7e-10 of the asymptote at L = 8, are summed in
// FP32 and added to the second-order coefficient as an integer, so that neither chain has a fourth FP64
// step (a fourth costs 4 % of a 16-atom s, p cluster's build and 2 % of an 8-atom diamond's, this 0.2 %); their
// rounding adds at most 3.8e-17, 2.1e-17 and 1.7e-16 of the value.  (With the third term in FP32 as well, at a
// spacing of 1/256, evaluation errors were 2.6e-16 for exp(-x) and 1.4e-16 for F_L, against 1.1e-16 for both now, and
// the tables took 10.6 MB.)  The sum is positive and may not lead f_2 or e_0 / 2 past a power
// of two, where an ulp doubles: with 75 points a unit no entry lies that close below one (by a factor of 19;
// with 64 two do; tests/test_boys_tables.py).
// ---------------------------------------------------------------------------
constexpr int kBoysRowLen = 6;
constexpr int kBoysPerUnit = 75;
constexpr double kBoysXmax = 60.0;
constexpr int kBoysXmaxHi = 0x404E0000;   // high word of 60.0 (low word 0)
constexpr int kBoysRows = 60 * kBoysPerUnit + 1;
constexpr int kBoysTailBits = 9;          // mantissa bits of the grid of t
constexpr int kBoysTailRows = (2 << kBoysTailBits) + 1;
constexpr int kBoysTableLen = (kBoysRows + kBoysTailRows) * kBoysRowLen;  // doubles per order
constexpr int kBoysExp = (kMaxLt + 1) * kBoysTableLen;                    // first of the exp rows
constexpr int kBoysDoubles = kBoysExp + 2 * kBoysRows;

// Table entries.  rcp[k] = 1 / (2 kBoysTop + 2 k + 1): the series multiplies by reciprocals made once.
constexpr int kBoysTop = 15, kBoysTerms = 512;
constexpr int kBoysUnit = 44;  // exponent of the unit of the FP32 terms below f_2's: 2^8 of its ulps
__host__ __device__ __forceinline__ void boys_put_row(double* row, const double* f) {
  for (int k = 0; k < 4; ++k) row[k] = f[k];
  float* r = reinterpret_cast<float*>(row + 4);
  for (int k = 0; k < 3; ++k) r[k] = (float)ldexp(f[4 + k], kBoysUnit - ilogb(f[2]));
  r[3] = 0.f;
}
__host__ __device__ __forceinline__ float boys_grid(float g) { return g * (1.0f / kBoysPerUnit); }
// an integer below 2^23 as FP32, on the FP32 pipe
__device__ __forceinline__ float small_int_f32(int g) { return __int_as_float(0x4b000000 | g) - 8388608.0f; }
// row g < kBoysRows of every order and of exp: F_15 from its series
// exp(-x) sum_k (2x)^k / ((31)(33)...(31+2k)), the lower orders by F_{m-1} = (2x F_m + e^{-x}) / (2m-1)
__host__ __device__ __forceinline__ void boys_make_rows(int g, const double* rcp, double* tabs) {
  const double x = boys_grid((float)g);
  double term = rcp[0], sum = term;
  for (int k = 1; k < kBoysTerms; ++k) {  // (some 250 terms at x = 60)
    term *= 2.0 * x * rcp[k];
    sum += term;
    if (term < 1e-18 * sum) break;
  }
  const double e = exp(-x);
  double F[kBoysTop + 1], f[7];
  F[kBoysTop] = e * sum;
  for (int m = kBoysTop; m >= 1; --m) F[m - 1] = (2.0 * x * F[m] + e) / (2 * m - 1);
  const double inv_fact[7] = {1.0, -1.0, 1.0 / 2, -1.0 / 6, 1.0 / 24, -1.0 / 120, 1.0 / 720};
  for (int L = 0; L <= kMaxLt; ++L) {
    for (int k = 0; k < 7; ++k) f[k] = inv_fact[k] * F[L + k];
    boys_put_row(tabs + L * kBoysTableLen + g * kBoysRowLen, f);
  }
  tabs[kBoysExp + 2 * g] = e;
  tabs[kBoysExp + 2 * g + 1] = e / 6;
}
// row kBoysRows + g of order L
__host__ __device__ __forceinline__ void boys_make_tail_row(int L, int g, double* tabs) {
  const int n = 1 << kBoysTailBits;
  const double t = g < n ? 1.0 + (double)g / n : 2.0 + 2.0 * (g - n) / n;
  double c = 0.886226925452758014, f[7];  // (2L-1)!!/2^{L+1} sqrt(pi)
  for (int m = 0; m < L; ++m) c *= m + 0.5;
  f[0] = c / sqrt(t);
  for (int m = 0; m < L; ++m) f[0] /= t;
  for (int k = 1; k < 7; ++k) f[k] = -f[k - 1] * (L + k - 0.5) / (k * t);
  boys_put_row(tabs + L * kBoysTableLen + (kBoysRows + g) * kBoysRowLen, f);
}

// x + n 2^8 ulp(x) for a positive x that this leads past no power of two
__device__ __forceinline__ double add_units(double x, int n) {
  return __longlong_as_double(__double_as_longlong(x) + ((long long)n << (52 - kBoysUnit)));
}
// mantissa in [1, 2] of a positive normal x, rounded to FP32
__device__ __forceinline__ float mantissa_f32(double x) {
  const long long b = __double_as_longlong(x) + (1ll << 28);
  const unsigned hi = (unsigned)(b >> 32) - ((unsigned)__double2hiint(x) & 0x7ff00000u);
  return __int_as_float((int)(0x3f800000u + ((hi << 3) | ((unsigned)b >> 29))));
}

// F and exp(-x) from a row of an order and a row of exp, d = x - x_g: 6 FP64 instructions.
__device__ __forceinline__ void boys_row(const double* __restrict__ f, const double* __restrict__ ex, double d,
                                         double& F, double& e) {
  const double2 r0 = __ldg(reinterpret_cast<const double2*>(f)), r1 = __ldg(reinterpret_cast<const double2*>(f) + 1);
  const float4 r2 = __ldg(reinterpret_cast<const float4*>(f) + 2);
  const double2 e0 = __ldg(reinterpret_cast<const double2*>(ex));
  constexpr float kU = (float)(2ll << kBoysUnit);  // e_0 / 2 of mantissa 1 in its units, times 2
  const float df = to_f32_rn(d), d2 = df * df;
  const int nf = __float2int_rn(d2 * __fmaf_rn(df, __fmaf_rn(df, r2.z, r2.y), r2.x));
  const int ne = __float2int_rn(d2 * mantissa_f32(e0.x) *
                                __fmaf_rn(df, __fmaf_rn(df, kU / 720, -kU / 120), kU / 24));
  F = fma(fma(fma(r1.y, d, add_units(r1.x, nf)), d, r0.y), d, r0.x);
  e = fma(fma(fma(-e0.y, d, add_units(scale2(e0.x, -1), ne)), d, -e0.x), d, e0.x);
}

// row of x < kBoysXmax (the FP32 sum rounds to an integer); no argument leads past the table, a NaN from
// coordinates that overflowed neither
__device__ __forceinline__ int boys_index(float x) {
  const float r = __fmaf_rn(x, (float)kBoysPerUnit, 8388608.0f);
  return (int)min((unsigned)(__float_as_int(r) - 0x4b000000), (unsigned)(kBoysRows - 1));
}

// F_L(x) and exp(-x) for 0 <= x < kBoysXmax
__device__ __forceinline__ void boys_top(int L, double x, const double* __restrict__ tabs, double& F, double& e,
                                         const Fp64& op) {
  const int g = boys_index(approx_f32(x));
  const double d = op.sub(x, to_f64(boys_grid(small_int_f32(g))));
  boys_row(tabs + L * kBoysTableLen + g * kBoysRowLen, tabs + kBoysExp + 2 * g, d, F, e);
}

// F_L(x) and exp(-x) (0 from kBoysXmax on) for any x >= 0, by one sequence of instructions
__device__ __forceinline__ void boys_any(int L, double x, const double* __restrict__ tabs, double& F, double& e,
                                         const Fp64& op) {
  constexpr int kShift = 23 - kBoysTailBits, kOne = 127 << kBoysTailBits;
  const bool tail = ge_hi(x, kBoysXmaxHi);
  const int k = tail ? ((__double2hiint(x) >> 20) - 1023) >> 1 : 0;
  const double t = scale2(x, -2 * k);
  const float f = approx_f32(t);
  const int g = boys_index(f);
  const int gt = ((__float_as_int(f) + (1 << (kShift - 1))) >> kShift) - kOne;  // t in [1, 4): at most kBoysTailRows - 1
  const float xg = tail ? __int_as_float((gt + kOne) << kShift) : boys_grid(small_int_f32(g));
  const double d = op.sub(t, to_f64(xg));
  boys_row(tabs + L * kBoysTableLen + (tail ? kBoysRows + gt : g) * kBoysRowLen, tabs + kBoysExp + (tail ? 0 : 2 * g), d,
           F, e);
  if (tail) {
    const int hi = __double2hiint(F), up = k * (2 * L + 1);
    F = (hi >> 20) > up ? scale2(F, -up) : 0.0;
    e = 0.0;
  }
}

}  // namespace hfx
