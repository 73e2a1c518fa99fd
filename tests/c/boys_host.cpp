// The Boys tables and look-ups of csrc/boys.cuh compiled for the host: CUDA's bit casts, FMAs and loads
// written out in C++ (a * b + c contracted nowhere else: build with -ffp-contract=off).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
struct double2 { double x, y; };
struct float4 { float x, y, z, w; };
template <class To, class From>
static To bits(From f) {
  To t;
  std::memcpy(&t, &f, sizeof(t));
  return t;
}
static int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)(uint32_t)bits<uint64_t>(x); }
static double __hiloint2double(int hi, int lo) { return bits<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static double __longlong_as_double(long long x) { return bits<double>(x); }
static int __float_as_int(float x) { return bits<int>(x); }
static float __int_as_float(int x) { return bits<float>(x); }
static int __float2int_rn(float x) { return (int)std::nearbyint(x); }
static double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
template <class T>
static T __ldg(const T* p) { return *p; }
using std::fma;
using std::min;

#include "boys.cuh"

static std::vector<double> tables;

extern "C" void boys_tables() {
  std::vector<double> rcp(hfx::kBoysTerms);
  for (int k = 0; k < hfx::kBoysTerms; ++k) rcp[k] = 1.0 / (2 * hfx::kBoysTop + 2 * k + 1);
  tables.assign(hfx::kBoysDoubles, NAN);
  for (int g = 0; g < hfx::kBoysRows; ++g) hfx::boys_make_rows(g, rcp.data(), tables.data());
  for (int L = 0; L <= hfx::kMaxLt; ++L)
    for (int g = 0; g < hfx::kBoysTailRows; ++g) hfx::boys_make_tail_row(L, g, tables.data());
}
extern "C" double* boys_table_data() { return tables.data(); }
extern "C" void boys_sizes(int* s) {
  const int v[6] = {hfx::kBoysRowLen,   hfx::kBoysPerUnit, hfx::kBoysRows, hfx::kBoysTableLen,
                    hfx::kBoysTailBits, hfx::kBoysDoubles};
  std::copy(v, v + 6, s);
}
extern "C" void boys_at(int L, double x, int any, double* F, double* e) {
  const hfx::Fp64 op{1.0, -0.0};
  if (any)
    hfx::boys_any(L, x, tables.data(), *F, *e, op);
  else
    hfx::boys_top(L, x, tables.data(), *F, *e, op);
}
