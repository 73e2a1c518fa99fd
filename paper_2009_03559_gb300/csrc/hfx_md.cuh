// Hermite engine: the kernel of every class launch, in FP64 and (R = float) for the FP32 pass of a
// mixed-precision build.  A warp, or a team of 2 or 4 for the largest classes, evaluates and digests a
// stream of quartets.
//
// What bounds it: the FP64 pipe, one warp instruction per 64 cycles and SM quarter whatever the
// number of active lanes, so the algorithm with the fewest FP64 warp instructions wins and a
// handful of resident warps hides everything else (an FMA chain on one warp per quarter already
// runs at the full rate).  The Hermite form (tables: gen_md_tables.py) contracts over the
// primitives before it transforms, which leaves (dp|dp) 320 + 225 lane operations per primitive
// quartet where the Obara-Saika schedule had 2053, and keeps the recursion on the lanes' own
// registers: no interpreted op, no idle lane.  64-atom diamond, FP64 build 4331 -> 1784 ms, mixed
// precision 2999 -> 1098 ms; the FP64 pipe is 94-97 % busy at L = 1-4, 86-94 % at L = 5-7, 74 % at L = 8.
//
// A warp runs a stream of primitive quartets that crosses quartet borders, 32 at a time:
//   set-up and Hermite recursion, a lane per primitive quartet (results to shared memory);
//   per run of lanes of one (quartet, bra primitive pair): ket contraction, a lane per H value;
//   at the end of a bra primitive pair: bra contraction; at the end of a quartet: the two
//   transformation passes and the digest.
#pragma once
#include <type_traits>
#include "eri_prim.cuh"
#include "eri_quartets.cuh"
#include "hfx_eri.h"

namespace hfx {

#define HFX_N_CLASSES 21
#define HFX_TABLE_QUAL __device__ __align__(16) const
#include "md_tables.inc"
#undef HFX_TABLE_QUAL

// n S for a small integer n: doubling and quadrupling are exponent increments (integer pipe).
// S = 0 or subnormal becomes at most 4 x 2^-1022: nothing next to any integral.
template <int N>
__device__ __forceinline__ double times(double x, const Fp64& op) {
  if constexpr (N == 1) return x;
  if constexpr (N == 2) return scale_up(x, 1);
  if constexpr (N == 3) return op.mul(x, fp64_operand(2));
  if constexpr (N == 4) return scale_up(x, 2);
  if constexpr (N == 5) return op.mul(x, fp64_operand(3));
  if constexpr (N == 6) return scale_up(op.mul(x, fp64_operand(2)), 1);
  if constexpr (N == 7) return op.mul(x, fp64_operand(4));
  return x;  // not reached: a chain of order L <= 8 raises with N <= 7
}
template <int N>
__device__ __forceinline__ float times(float x, const Fp64&) {
  return x * float(N);
}
__device__ __forceinline__ float mulr(float a, float b, const Fp64&) { return a * b; }
__device__ __forceinline__ double mulr(double a, double b, const Fp64& op) { return op.mul(a, b); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// compile-time loop: f(integral constant I), ..., f(integral constant N - 1)
template <int I, int N, class F>
__device__ __forceinline__ void unrolled(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>());
    unrolled<I + 1, N>(f);
  }
}

// f(integral constant n) for a run-time n of 1 .. N
template <int N, class F>
__device__ __forceinline__ void exact_rounds(int n, F&& f) {
  if constexpr (N > 1) {
    if (n < N) {
      exact_rounds<N - 1>(n, f);
      return;
    }
  }
  if (n >= N) f(std::integral_constant<int, N>());  // (n may be 0: a team's last warps)
}

// f(0) .. f(n - 1), U at a time and the rest one by one (a loop unrolled by the compiler ran its
// rest as a predicated copy, whose FP64 instructions cost the same when off)
template <int U, class F>
__device__ __forceinline__ void stepped(int n, F&& f) {
  int i = 0;
#pragma unroll 1
  for (; i + U <= n; i += U) {
#pragma unroll
    for (int k = 0; k < U; ++k) f(i + k);
  }
#pragma unroll 1
  for (; i < n; ++i) f(i);
}

__host__ __device__ constexpr int n_herm(int n) { return (n + 1) * (n + 2) * (n + 3) / 6; }
// position of Hermite index (x, y, z) in the list of all by order (x descending, then y)
__host__ __device__ constexpr int herm_index(int x, int y, int z) {
  const int n = x + y + z;
  return n * (n + 1) * (n + 2) / 6 + (n - x) * (n - x + 1) / 2 + (n - x - y);
}

// Share of the x chains (U, V) of the Hermite recursion that warp W of an NW-warp team runs: a
// contiguous part of the chains in V-major order with about 1 / NW of the operations.
template <int L, int NW>
__host__ __device__ constexpr int chain_owner(int u, int v) {
  int total = 0, before = 0;
  for (int vv = 0; vv <= L; ++vv)
    for (int uu = 0; uu <= L - vv; ++uu) {
      const int n = L - uu - vv, cost = n * (n + 1) / 2 + n + 1;
      if (vv < v || (vv == v && uu < u)) before += cost;
      if (vv == v && uu == u) before += cost / 2;
      total += cost;
    }
  return before * NW / total;
}
// the largest u of plane v (with v < 0: the largest v) that has a chain of warp W; -1: none
template <int L, int NW, int W>
__host__ __device__ constexpr int chain_last(int v) {
  int last = -1;
  for (int vv = 0; vv <= L; ++vv)
    for (int uu = 0; uu <= L - vv; ++uu)
      if (chain_owner<L, NW>(uu, vv) == W && (v < 0 || vv == v)) last = v < 0 ? vv : uu;
  return last;
}

// S_r, |r| <= L, from the base values B[m] = (2 rho)^m G_m:  rows in m, first along z, from each
// of them along y, from each of those along x; only the last two rows of a chain stay live.
// Warp W of NW writes its share.  In FP32 the recursion runs on s_r = S_r / lam^{|r|} with
// lam = sqrt(2 rho) (base values G_m, coordinates times lam), whose values stay in range for any
// exponents, and lp[n] = lam^n scales the results.
template <int L, int NW, int W, typename R>
__device__ __forceinline__ void hermite(const R (&B)[L + 1], R X, R Y, R Z, const R* lp, R* out,
                                        const Fp64& op) {
  constexpr int kLastV = chain_last<L, NW, W>(-1);
  R zr[L + 1], zp[L + 1];
#pragma unroll
  for (int m = 0; m <= L; ++m) zr[m] = B[m];
  unrolled<0, kLastV + 1>([&](auto cv) {
    constexpr int V = decltype(cv)::value;
    constexpr int kLastU = chain_last<L, NW, W>(V);
    R yr[L + 1 - V], yp[L + 1 - V];
#pragma unroll
    for (int m = 0; m <= L - V; ++m) yr[m] = zr[m];
    unrolled<0, kLastU + 1>([&](auto cu) {
      constexpr int U = decltype(cu)::value;
      constexpr int N = L - V - U;
      if constexpr (chain_owner<L, NW>(U, V) == W) {
        R xr[N + 1], xp[N + 1];
#pragma unroll
        for (int m = 0; m <= N; ++m) xr[m] = yr[m];
        unrolled<0, N + 1>([&](auto ct) {
          constexpr int T = decltype(ct)::value;
          if constexpr (sizeof(R) == 8 || T + U + V == 0)
            out[herm_index(T, U, V)] = xr[0];
          else
            out[herm_index(T, U, V)] = xr[0] * lp[T + U + V];
#pragma unroll
          for (int m = 0; m < N - T; ++m) {
            R v;
            if constexpr (T == 0)
              v = mulr(X, xr[m + 1], op);
            else
              v = fmar(X, xr[m + 1], -times<T>(xp[m + 1], op));
            xp[m] = xr[m];
            xr[m] = v;
          }
          if constexpr (N - T > 0) xp[N - T] = xr[N - T];
        });
      }
      if constexpr (U < kLastU) {
#pragma unroll
        for (int m = 0; m < N; ++m) {
          R v;
          if constexpr (U == 0)
            v = mulr(Y, yr[m + 1], op);
          else
            v = fmar(Y, yr[m + 1], -times<U>(yp[m + 1], op));
          yp[m] = yr[m];
          yr[m] = v;
        }
        if constexpr (N > 0) yp[N] = yr[N];
      }
    });
    if constexpr (V < kLastV) {
#pragma unroll
      for (int m = 0; m < L - V; ++m) {
        R v;
        if constexpr (V == 0)
          v = mulr(Z, zr[m + 1], op);
        else
          v = fmar(Z, zr[m + 1], -times<V>(zp[m + 1], op));
        zp[m] = zr[m];
        zr[m] = v;
      }
      if constexpr (L - V > 0) zp[L - V] = zr[L - V];
    }
  });
}

// Set-up of one primitive quartet: B[m] = (2 rho)^m G_m, the base values of the Hermite
// recursion, with G_m = pref (F_m(T) - kappa^{m+1/2} F_m(kappa T)) (see prim_core, whose downward
// recursion this is, multiplied through by (2 rho)^m):
//   B_{m-1} = (R^2 B_m + a_m - c_m e^{-kappa T}) / (2m-1),
//   a_m = pref (2 rho)^{m-1} e^{-T},  c_m = pref (2 rho)^{m-1} kappa^{m-1/2}.
// False if the quartet is negligible (kappa T beyond the tables: G_m < e^{-60}).
template <int L>
__device__ __forceinline__ bool md_setup(const PrimPair& b, const PrimPair& k, const double* qc, double omega,
                                         double omega2, const double* __restrict__ tabs, double (&B)[L + 1],
                                         double* PQ, const Fp64& op) {
  const double p = b.p, q = k.p;
  const double y = rsqrt_nr(op.add(p, q), op);  // 1/sqrt(p+q)
  const double rho = op.mul(op.mul(p, y), op.mul(q, y));
  PQ[0] = op.sub(b.P[0], qc[0]);
  PQ[1] = op.sub(b.P[1], qc[1]);
  PQ[2] = op.sub(b.P[2], qc[2]);
  const double R2 = fma(PQ[0], PQ[0], fma(PQ[1], PQ[1], op.mul(PQ[2], PQ[2])));
  const double T = op.mul(rho, R2);
  const double pref = op.mul(op.mul(b.C, k.C), y);
  double kap = 0.0, sk = 0.0, kT = 0.0;
  if (omega2 > 0.0) {
    sk = op.mul(omega, rsqrt_nr(op.add(rho, omega2), op));  // sqrt(kappa)
    kap = op.mul(sk, sk);
    kT = op.mul(kap, T);
    if (ge_hi(kT, kBoysXmaxHi)) return false;
  }
  double F1, e1;
  boys_any(L, T, tabs, F1, e1, op);
  const double r2 = scale2(rho, 1);
  double pL = pref;  // pref (2 rho)^L
  if constexpr (L > 0) {
    double w = r2;
    pL = (L & 1) ? op.mul(pref, r2) : pref;
#pragma unroll
    for (int i = 1; (L >> i) > 0; ++i) {
      w = op.mul(w, w);
      if ((L >> i) & 1) pL = op.mul(pL, w);
    }
  }
  double a[L + 1], g = op.mul(pL, F1);
  a[0] = op.mul(pref, e1);
#pragma unroll
  for (int m = 1; m < L; ++m) a[m] = op.mul(a[m - 1], r2);
  if (omega2 > 0.0) {
    double F2, e2;
    boys_top(L, kT, tabs, F2, e2, op);
    const double kr = op.mul(kap, r2);
    double c[L + 1];
    c[0] = op.mul(pref, sk);
#pragma unroll
    for (int m = 1; m <= L; ++m) c[m] = op.mul(c[m - 1], kr);
    g = fma(-c[L], F2, g);
#pragma unroll
    for (int m = 0; m < L; ++m) a[m] = fma(-c[m], e2, a[m]);
  }
  B[L] = g;
#pragma unroll
  for (int m = L; m >= 1; --m) {
    g = fma(R2, g, a[m - 1]);
    if (m > 1) g = op.mul(g, fp64_operand(kFp64Recip + m));
    B[m - 1] = g;
  }
  return true;
}

// Warps that work on one stream together (a team): they share its Hermite integrals and
// contraction buffers, each with an even share of every step's rounds.  The buffers of a lone warp
// leave 6, 4 and 2 resident warps per SM at L = 6, 7, 8 (FP64 pipe 73, 49 and 26 % busy); teams
// bring that to 10, 12 and 8.  Up to L = 5 a lone warp's buffers leave 9 to 16 and the pipe 87 to
// 97 % busy, and a team's barriers would only cost.
// (md_team: 1 up to L = 5, then 2, 4, 4)
// threads per block: two lone warps up to L = 4, one at L = 5 (whose 23 KB a warp fill the SM better
// in single pieces: (dp|pp) 199 -> 193 ms at 64 atoms), one team beyond
__host__ __device__ constexpr int md_block(int Lt) { return Lt <= 4 ? 64 : 32 * md_team(Lt); }

// The FP32 pass of a mixed-precision class runs the same steps with the set-up, the Hermite
// recursion and both contractions in FP32 (the transformations, which replace the horizontal
// recurrences and the spherical step, and the digest in FP64).  A team sets up kSub32 times 32
// primitive quartets before it contracts them (at least its warps' 32 each), so that those whose
// Boys step the FP32 set-up declines (a few per cent) are set up in FP64 together and not in every
// 32.  More of them save FP64 set-ups and cost shared memory, hence resident warps (64-atom mixed
// build: 2 times 1095 ms, 4 times 1104, 6 times 1185, 8 times 1221).
constexpr int kSub32 = 2;
// 32s of primitive quartets set up together; whether their set-up passes through shared memory;
// its values per primitive quartet: base values, P - Q (in FP32 times lam, lam, and where it belongs)
template <typename R>
__host__ __device__ constexpr int md_sub(int Lt) {
  return sizeof(R) == 4 && kSub32 > md_team(Lt) ? kSub32 : md_team(Lt);
}
template <typename R>
__host__ __device__ constexpr int md_xval(int Lt) { return sizeof(R) == 4 ? Lt + 6 : Lt + 4; }

// Row of a primitive quartet in shared memory: its Hermite integrals, then the factors of its ket
// primitive pair (at most as many as the classes of this L have sets); an odd length, so that the
// lanes' rows start in different banks, and known when compiling, so that the contraction's loads
// need no address arithmetic.
__host__ __device__ constexpr int md_row(int Lt) {
  return (n_herm(Lt) + md_ket_sets(Lt)) | 1;
}
// Up to L = 4, in FP32 up to L = 7, a lane's entries of the contraction tables and its A values stay
// in registers (at most this many rounds of a warp of the team); up to L = 2, where a ket
// contraction has at most 13 results, the warp runs 32 / md_group of them side by side.
template <typename R>
__host__ __device__ constexpr bool md_in_regs(int Lt) { return Lt <= (sizeof(R) == 4 ? 7 : 4); }
__host__ __device__ constexpr int md_group(int Lt) { return Lt == 0 ? 1 : (Lt == 1 ? 4 : 16); }

// Shared memory of one team, in doubles (offsets; every region starts on an even double).
struct MdLayout {
  int R, H, Y, A, Tb, Tk, Q;  // rows, H, transformed rows (in H's place from L = 3), A and the final block
  int X;                      // set-up results, where several 32s are set up together
  int size;
};
// quartets waiting in a team's queue: at most 31, and 32 more
constexpr int kMdQueue = 64;

template <typename R>
MdLayout md_layout(const MdClassInfo& c, const MdPairInfo& b, const MdPairInfo& k) {
  MdLayout l{};
  auto even = [](int n) { return (n + 1) & ~1; };
  auto mem = [&](int n) { return even(sizeof(R) == 8 ? n : (n + 1) / 2); };  // n values of type R
  l.R = 0;
  l.H = l.R + mem(32 * md_row(c.Lt));
  l.Y = c.Lt <= 2 ? l.H + mem(32) + 18 : l.H;  // 18: the runs' first rows
  l.A = l.Y + std::max(c.Lt <= 2 ? 0 : mem(c.n_kc), even(c.n_row * c.ncd));
  l.Tb = l.A + std::max(mem(c.n_bc), even(c.nab * c.ncd));
  l.Tk = l.Tb + even(b.n_coef);
  l.Q = l.Tk + even(k.n_coef);
  l.X = l.Q + 4 * kMdQueue;
  const int ns = md_sub<R>(c.Lt);
  // the values of 32 lanes; the accepted and declined masks; the team's claim
  l.size = even(l.X + (ns > 1 ? mem(ns * md_xval<R>(c.Lt) * 32) + ns + 2 : 0));  // 16-byte entries in Q
  return l;
}

// A sparse pass out[dst] = sum of T[c] in[i] (generated: rounds of 32 outputs of like length),
// rounds w, w + nw, ...
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) { return to_f64(x); }
template <typename R>
__device__ __forceinline__ void md_gather(int round0, int n_round, int dst0, const double* T, const R* in,
                                          double* out, int lane, int w, int nw) {
#pragma unroll 1
  for (int r = w; r < n_round; r += nw) {
    const uint32_t rd = __ldg(kMdZRound + round0 + r);
    const uint32_t* word = kMdZ + (rd & 0xFFFFFFu) + lane;
    const int n = rd >> 24;
    double v = 0.0;
#pragma unroll 4
    for (int t = 0; t < n; ++t) {
      const uint32_t e = __ldg(word + 32 * t);
      v = fma(T[e & 0xFFFFu], widen(in[e >> 16]), v);
    }
    const uint32_t d = __ldg(kMdZDst + dst0 + 32 * r + lane);
    if (d != 0xFFFFu) out[d] = v;
  }
}

// Digest of the final block into the half matrix A: rounds w, w + nw, ... of 32 generated tasks, a
// lane per (part of a) sum.  Every lane runs the same instructions with its own strides, so the
// sums of the four blocks share a round, and long sums (the 25 terms of A_bd in (ds|ds)) are cut so
// that a round's longest does not set the pace (64 atoms: FP64 build 1819 -> 1795 ms, mixed
// 1193 -> 1153 ms, whose FP32 pass the digest weighs on most).
__device__ __forceinline__ void md_digest(const MdClassInfo& mc, const int4& dim, const double* v, int A, int B,
                                          int C, int D, double deg, const double* __restrict__ P, double* K, int ld,
                                          int lane, int w0, int nw0, const Fp64& op) {
  const int sb = dim.z * dim.w, sa = dim.y * sb;
#pragma unroll 1
  for (int r = w0; r < mc.dig_n; r += nw0) {
    const uint32_t e = __ldg(kMdDigest + mc.dig + 32 * r + lane);
    const bool isB = e & 1, isD = e & 2;
    const int x = (e >> 2) & 7, y = (e >> 5) & 7, u = (e >> 8) & 7, n = (e >> 14) & 31;
    int w = (e >> 11) & 7;
    const int su = isB ? sa : sb, sw = isD ? dim.w : 1, nw = isD ? dim.z : dim.w;
    const double* vp = v + x * (isB ? sb : sa) + y * (isD ? 1 : dim.w) + u * su + w * sw;
    const double* pp = P + (size_t)((isB ? A : B) + u) * ld + (isD ? C : D) + w;
    double acc = op.nzero;
    // at the end of a row of w: v to the next u's first w, P to the next row's
    const int vskip = su - nw * sw, pskip = ld - nw;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      acc = fma(*vp, __ldg(pp), acc);
      vp += sw;
      ++pp;
      if (++w == nw) {
        w = 0;
        vp += vskip;
        pp += pskip;
      }
    }
    if (n) atomicAdd(K + (size_t)((isB ? B : A) + x) * ld + (isD ? D : C) + y, op.mul(deg, acc));
  }
}

// resident blocks per SM that the registers must allow: what shared memory allows
template <typename R>
__host__ __device__ constexpr int md_minb(int Lt) {
  const int f32[kMaxLt + 1] = {10, 10, 10, 10, 8, 12, 7, 4, 4}, f64[kMaxLt + 1] = {8, 8, 8, 8, 8, 10, 5, 3, 2};
  return sizeof(R) == 4 ? f32[Lt] : f64[Lt];
}

template <int LT, int KIND, typename R>
__global__ void __launch_bounds__(md_block(LT), md_minb<R>(LT))
    eri_md_kernel(const __grid_constant__ EriLaunch L, const __grid_constant__ MdLayout ly) {
  // the next class's launch may start (see md_launch): nothing it reads comes from this one
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(16) double smem[];
  constexpr bool F32 = sizeof(R) == 4;
  constexpr int NW = md_team(LT), kQ = kMdQueue, kTeams = md_block(LT) / (32 * NW);
  constexpr int NS = md_sub<R>(LT), NX = md_xval<R>(LT);
  constexpr int kRow = md_row(LT), kW = n_herm(LT);
  constexpr bool kRegs = md_in_regs<R>(LT);
  constexpr int KR = md_kc_rounds(LT), BR = md_bc_rounds(LT);
  const int lane = threadIdx.x & 31;
  const int wt = NW == 1 ? 0 : (int)(threadIdx.x >> 5);             // warp of the team
  const int team = NW == 1 ? (int)(threadIdx.x >> 5) : 0;           // team of the block
  double* S = smem + team * ly.size;
  R* const Rb = reinterpret_cast<R*>(S + ly.R);
  R* const H = reinterpret_cast<R*>(S + ly.H);
  R* const A = reinterpret_cast<R*>(S + ly.A);
  double* const Y = S + ly.Y;
  double* const F = S + ly.A;
  int4* const Q = reinterpret_cast<int4*>(S + ly.Q);  // system, bra position, ket position, nb | nk << 16
  // the bra's and the ket's first primitive pair, and where their Hermite data begin (in fours of
  // doubles): looked up once per quartet, not once per primitive quartet and run
  uint4* const Qo = reinterpret_cast<uint4*>(Q + kQ);
  R* const X = reinterpret_cast<R*>(S + ly.X);
  unsigned* const Xok = reinterpret_cast<unsigned*>(S + ly.size - NS - 2);  // masks [NS], [NS], then the claim
  const unsigned lt_mask = (1u << lane) - 1u;
  const MdClassInfo mc = L.mc;
  const EriLaunch* const Lp = &L;
  const int4 dims = make_int4(L.ci.dims[0], L.ci.dims[1], L.ci.dims[2], L.ci.dims[3]);
  unsigned long long t0 = 0;
  if (L.busy && threadIdx.x == 0) t0 = globaltimer_ns();

  int head = 0, head_off = 0, tail = 0, waiting = 0;  // queue: entries [head, tail), primitive quartets left
  bool h_valid = false, a_valid = false;              // the head quartet's H and A hold partial sums
  int n_eval = 0;                                     // its primitive quartets evaluated so far
  R carry = R(0);                                     // L <= 2: the partial sum of a lane's H value
  int tb_sys = -1, tb_bra = -1;                       // whose transformation is in Tb
  Tally tally;
  Fp64 op;
  op.init();
  const double omega = op.mul(L.omega, op.one), omega2 = op.mul(L.omega2, op.one);

  int kc_r[kRegs ? KR : 1], kc_w[kRegs ? KR : 1], bc_h[kRegs ? BR : 1], bc_w[kRegs ? BR : 1];
  R a_reg[kRegs ? BR : 1];
  if constexpr (kRegs) {
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      const int o = 32 * (wt + NW * u) + (LT <= 2 ? lane % md_group(LT) : lane);
      const int e = o < mc.n_kc ? __ldg(kMdKc + mc.kc + o) : 0;
      kc_r[u] = e & 0xFF;
      kc_w[u] = kW + (e >> 8);
    }
#pragma unroll
    for (int u = 0; u < BR; ++u) {
      const int o = 32 * (wt + NW * u) + lane, e = o < mc.n_bc ? __ldg(kMdBc + mc.bc + o) : 0;
      bc_h[u] = e & 0xFFF;
      bc_w[u] = e >> 12;
      a_reg[u] = R(0);
    }
  }

  auto sync = [&]() {
    if constexpr (NW == 1)
      __syncwarp();
    else
      __syncthreads();
  };
  auto rec = [&](int sys) -> const EriLaunch& {
    if constexpr (KIND == MD_BATCH)
      return L.batch[sys];
    else
      return *Lp;
  };
  auto pair_id = [&](const EriLaunch& Ls, int pos) -> int {
    if constexpr (KIND == MD_DIAG)
      return pos;
    else
      return __ldg(Ls.sorted + pos);
  };

  auto narrow = [](double x) -> R {
    if constexpr (F32)
      return to_f32_rn(x);
    else
      return x;
  };

  // this warp's rounds of n results: wt, wt + NW, ...
  auto team_rounds = [&](int n) { return (((n + 31) >> 5) - wt + NW - 1) / NW; };

  // H[s, r] (+)= sum over the primitive quartets in rows [p0, p1) of W_s S_r
  auto ket_contract = [&](int p0, int p1) {
    if constexpr (kRegs) {
      // the round count decides a branch: as a predicate inside the loop it was turned into
      // selects, with the FP64 instructions of all rounds executed
      exact_rounds<KR>(team_rounds(mc.n_kc), [&](auto nc) {
        constexpr int N = decltype(nc)::value;
        const R *r[N], *w[N];
        R v[N];
#pragma unroll
        for (int u = 0; u < N; ++u) {
          r[u] = Rb + p0 * kRow + kc_r[u];
          w[u] = Rb + p0 * kRow + kc_w[u];
          const int o = 32 * (wt + NW * u) + lane;
          v[u] = h_valid && o < mc.n_kc ? H[o] : R(0);
        }
        stepped<4>(p1 - p0, [&](int p) {
#pragma unroll
          for (int u = 0; u < N; ++u) v[u] = fmar(w[u][p * kRow], r[u][p * kRow], v[u]);
        });
#pragma unroll
        for (int u = 0; u < N; ++u) {
          const int o = 32 * (wt + NW * u) + lane;
          if (o < mc.n_kc) H[o] = v[u];
        }
      });
    } else {
      auto rounds = [&](int g, auto nc) {
        constexpr int N = decltype(nc)::value;
        const R *r[N], *w[N];
        R v[N];
#pragma unroll
        for (int u = 0; u < N; ++u) {
          const int e = __ldg(kMdKc + mc.kc + 32 * (g + NW * u) + lane);  // padded to whole rounds
          r[u] = Rb + p0 * kRow + (e & 0xFF);
          w[u] = Rb + p0 * kRow + kW + (e >> 8);
          const int o = 32 * (g + NW * u) + lane;
          v[u] = h_valid && o < mc.n_kc ? H[o] : R(0);
        }
          stepped<2>(p1 - p0, [&](int p) {
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = fmar(w[u][p * kRow], r[u][p * kRow], v[u]);
          });
#pragma unroll
        for (int u = 0; u < N; ++u) {
          const int o = 32 * (g + NW * u) + lane;
          if (o < mc.n_kc) H[o] = v[u];
        }
      };
      const int n = (mc.n_kc + 31) >> 5;
      int g = wt;  // this warp's rounds: wt, wt + NW, ...
#pragma unroll 1
      for (; g + 3 * NW < n; g += 4 * NW) rounds(g, std::integral_constant<int, 4>());
#pragma unroll 1
      for (; g < n; g += NW) rounds(g, std::integral_constant<int, 1>());
    }
    sync();
  };

  // A[s', s, r] (+)= W_s' H[s, r] for the bra primitive pair with factors w
  auto bra_contract = [&](const double* w, const R* H) {
    ++tally.run;
    if constexpr (kRegs) {
      const int n = team_rounds(mc.n_bc);
      if constexpr (F32) {  // spare rounds cost less than copies of the code
#pragma unroll
        for (int u = 0; u < BR; ++u)
          if (u < n) a_reg[u] = fmar(narrow(__ldg(w + bc_w[u])), H[bc_h[u]], a_reg[u]);
      } else {
        exact_rounds<BR>(n, [&](auto nc) {
#pragma unroll
          for (int u = 0; u < decltype(nc)::value; ++u) a_reg[u] = fmar(__ldg(w + bc_w[u]), H[bc_h[u]], a_reg[u]);
        });
      }
      if constexpr (LT > 2) sync();
      return;
    }
    auto rounds = [&](int o, auto nc) {
      constexpr int N = decltype(nc)::value;
      R x[N], h[N], a[N];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const int e = __ldg(kMdBc + mc.bc + o + 32 * NW * u);  // padded to whole rounds
        x[u] = narrow(__ldg(w + (e >> 12)));
        h[u] = H[e & 0xFFF];
        a[u] = a_valid && o + 32 * NW * u < mc.n_bc ? A[o + 32 * NW * u] : R(0);
      }
#pragma unroll
      for (int u = 0; u < N; ++u)
        if (o + 32 * NW * u < mc.n_bc) A[o + 32 * NW * u] = fmar(x[u], h[u], a[u]);
    };
    const int n = (mc.n_bc + 31) >> 5;
    int g = wt;
    for (; g + 3 * NW < n; g += 4 * NW) rounds(32 * g + lane, std::integral_constant<int, 4>());
    for (; g < n; g += NW) rounds(32 * g + lane, std::integral_constant<int, 1>());
    sync();
  };

  auto finish = [&](int slot) {
    const int4 e = Q[slot];
    const EriLaunch& Ls = rec(e.x);
    const int nb = e.w & 0xFFFF, nk = e.w >> 16;
    tally.prim += n_eval;
    tally.skip += nb * nk - n_eval;
    double* Tb = S + ly.Tb;
    double* Tk = S + ly.Tk;
    const int bra = pair_id(Ls, e.y), ket = pair_id(Ls, e.z);
    const uint4 eo = Qo[slot];
    if (a_valid) {
      if constexpr (kRegs) {
#pragma unroll
        for (int u = 0; u < BR; ++u) {
          const int o = 32 * (wt + NW * u) + lane;
          if (o < mc.n_bc) A[o] = a_reg[u];
          a_reg[u] = R(0);
        }
      }
      ++tally.quart;
      if (F32) {
        ++tally.q32;
        tally.p32 += n_eval;
      }
      const double* mk = Ls.pa.md + 4ull * eo.w;
      for (int i = 32 * wt + lane; i < mc.ket_coef; i += 32 * NW) Tk[i] = __ldg(mk + i);
      if (tb_bra != bra || tb_sys != e.x) {
        // the bra side carries (-1)^{|p|}: the sign of every second coefficient degree
        const double* mb = Ls.pa.md + 4ull * eo.z;
        for (int i = 32 * wt + lane; i < mc.bra_coef; i += 32 * NW) {
          const double x = __ldg(mb + i);
          Tb[i] = __hiloint2double(__double2hiint(x) ^ (__ldg(kMdCoefSign + mc.bra_coef0 + i) << 31),
                                   __double2loint(x));
        }
        tb_bra = bra;
        tb_sys = e.x;
      }
      sync();
      md_gather<R>(mc.z1_round, mc.z1_n, mc.z1_dst, Tk, A, Y, lane, wt, NW);
      sync();
      md_gather<double>(mc.z2_round, mc.z2_n, mc.z2_dst, Tb, Y, F, lane, wt, NW);
      sync();
    }
    if constexpr (KIND == MD_DIAG) {
      double mx = 0.0;
      if (a_valid) {
        for (int f = lane; f < mc.ncd; f += 32) mx = fmax(mx, fabs(F[f * mc.ncd + f]));
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      if (lane == 0 && wt == 0) Ls.diag_Q[bra] = sqrt(mx);
    } else if (a_valid) {
      if constexpr (KIND == MD_PER) {
        PerQuartet pq;
        if (per_quartet(Ls, e.x, bra, ket, pq))
          digest_per(L.ci, F, 1, pq, Ls.per.cells[e.x].KG, Ls.per.nbf, 32 * wt + lane, 32 * NW);
      } else {
        const int sa = __ldg(Ls.pa.sa + bra), sb = __ldg(Ls.pa.sb + bra);
        const int sc = __ldg(Ls.pa.sa + ket), sd = __ldg(Ls.pa.sb + ket);
        double deg = 1.0;
        if (sa == sb) deg *= 0.5;
        if (sc == sd) deg *= 0.5;
        if (e.y == e.z) deg *= 0.5;
        md_digest(mc, dims, F, __ldg(Ls.sh.bf_off + sa), __ldg(Ls.sh.bf_off + sb), __ldg(Ls.sh.bf_off + sc),
                  __ldg(Ls.sh.bf_off + sd), deg, Ls.P, Ls.K, Ls.ld, lane, wt, NW, op);
      }
    }
    sync();
    a_valid = h_valid = false;
    n_eval = 0;
  };

  // primitive quartet number pos of the stream: its queue entry, the quartet, the primitive pairs
  struct Prim {
    int e, nb, nk, ib, ik;
    int4 q;
  };
  auto locate = [&](int pos) {
    Prim s;
    s.e = head;
    int off = head_off + pos;
    s.q = Q[s.e & (kQ - 1)];
    int npq = (s.q.w & 0xFFFF) * (s.q.w >> 16);
    while (off >= npq) {
      off -= npq;
      s.q = Q[++s.e & (kQ - 1)];
      npq = (s.q.w & 0xFFFF) * (s.q.w >> 16);
    }
    s.nb = s.q.w & 0xFFFF;
    s.nk = s.q.w >> 16;
    s.ib = off / s.nk;
    s.ik = off - s.ib * s.nk;
    return s;
  };

  // the primitive pairs of s
  auto prims = [&](const Prim& s, const PrimPair*& pb, const PrimPair*& pk) -> const EriLaunch& {
    const EriLaunch& Ls = rec(s.q.x);
    const uint4 o = Qo[s.e & (kQ - 1)];
    pb = Ls.pa.prim + o.x + s.ib;
    pk = Ls.pa.prim + o.y + s.ik;
    return Ls;
  };
  // the factors of the bra primitive pair ib of the quartet in a slot
  auto bra_factors = [&](int slot, int ib) {
    return rec(Q[slot].x).pa.md + 4ull * Qo[slot].z + mc.bra_coef + ib * mc.bra_set;
  };

  // the next n (<= 32 NS, <= waiting) primitive quartets of the stream
  auto batch = [&](int n) {
    Prim s{};
    unsigned okm = 0;
    bool ok = false;
    R B[LT + 1], PQ[3], lam = R(1);
#pragma unroll 1
    for (int sub = wt; sub < NS; sub += NW) {  // set-up
      s = Prim{};
      s.nb = s.nk = 1;
      ok = false;
      bool declined = false;
      if (32 * sub + lane < n) {
        s = locate(32 * sub + lane);
        const PrimPair *pb, *pk;
        const EriLaunch& Ls = prims(s, pb, pk);
        if constexpr (F32) {
          PrimScalarsF ps;
          const int st = prim_core_f32(*pb, *pk, LT, to_f32(Ls.omega), B, ps, op);
          lam = sqrtf(2.0f * pb->pf * ps.RP);
          for (int i = 0; i < 3; ++i) PQ[i] = ps.PQ[i] * lam;
          ok = st == F32_OK;
          declined = st == F32_FP64;
        } else {
          double qc[3] = {pk->P[0], pk->P[1], pk->P[2]};
          if constexpr (KIND == MD_PER) {  // the ket pair's image in cell G
            const double* shift = L.per.cells[s.q.x].shift;
            qc[0] = op.add(qc[0], __ldg(shift));
            qc[1] = op.add(qc[1], __ldg(shift + 1));
            qc[2] = op.add(qc[2], __ldg(shift + 2));
          }
          // (a kernel parameter is a constant operand: one product makes it a register's)
          const double om = KIND == MD_BATCH ? Ls.omega : omega, om2 = KIND == MD_BATCH ? Ls.omega2 : omega2;
          ok = md_setup<LT>(*pb, *pk, qc, om, om2, L.boys, B, PQ, op);
        }
      }
      okm = __ballot_sync(0xffffffffu, ok);
      if constexpr (NS > 1) {
        R* x = X + sub * NX * 32 + lane;
#pragma unroll
        for (int m = 0; m <= LT; ++m) x[32 * m] = B[m];
#pragma unroll
        for (int i = 0; i < 3; ++i) x[32 * (LT + 1 + i)] = PQ[i];
        if constexpr (F32) {
          x[32 * (LT + 4)] = lam;
          x[32 * (LT + 5)] = __int_as_float((s.e & (kQ - 1)) | (s.ib << 6) | (s.ik << 12) |
                                            (s.ik == s.nk - 1 ? 1 << 18 : 0) | (s.ib == s.nb - 1 ? 1 << 19 : 0));
        }
        const unsigned dm = __ballot_sync(0xffffffffu, declined);
        if (lane == 0) {
          Xok[sub] = okm;
          Xok[NS + sub] = dm;
        }
      }
    }
    if constexpr (NS > 1) sync();
    if constexpr (F32) {
      // the declined ones in FP64, 32 at a time: their base values replace the FP32 ones
      int nd = 0;
      for (int sub = 0; sub < NS; ++sub) nd += __popc(Xok[NS + sub]);
      for (int d0 = 32 * wt; d0 < nd; d0 += 32 * NW) {
        int d = d0 + lane, sub = 0;
        if (d < nd) {
          unsigned m = Xok[NS];
          while (d >= __popc(m)) {
            d -= __popc(m);
            m = Xok[NS + ++sub];
          }
          for (; d > 0; --d) m &= m - 1;
          const int l = __ffs(m) - 1;
          const Prim t = locate(32 * sub + l);
          const PrimPair *pb, *pk;
          const EriLaunch& Ls = prims(t, pb, pk);
          double G[kMaxLt + 1];
          PrimScalars ps;
          if (prim_core(*pb, *pk, LT, Ls.omega, Ls.omega2, L.boys, G, ps, op)) {
#pragma unroll
            for (int k = 0; k <= LT; ++k) X[(sub * NX + k) * 32 + l] = to_f32_rn(G[k]);
            atomicOr(Xok + sub, 1u << l);
          }
        }
      }
      sync();
    }
#pragma unroll 1
    for (int sub = 0; sub < NS && 32 * sub < n; ++sub) {
      const int ns = min(32, n - 32 * sub);
      R lp[F32 ? LT + 1 : 1];
      lp[0] = R(1);
      if constexpr (NS > 1) {
        okm = Xok[sub];
        ok = (okm >> lane) & 1;
        s = Prim{};
        s.nb = s.nk = 1;
        const R* x = X + sub * NX * 32 + lane;
        if constexpr (F32) {
          const int p = lane < ns ? __float_as_int(x[32 * (LT + 5)]) : 0;
          s.e = head + (((p & (kQ - 1)) - head) & (kQ - 1));
          s.ib = (p >> 6) & 63;
          s.ik = (p >> 12) & 63;
          s.nk = s.ik + ((p >> 18) & 1 ? 1 : 2);  // only what tells the last ones
          s.nb = s.ib + ((p >> 19) & 1 ? 1 : 2);
        } else if (lane < ns) {
          s = locate(32 * sub + lane);
        }
#pragma unroll
        for (int m = 0; m <= LT; ++m) B[m] = x[32 * m];
#pragma unroll
        for (int i = 0; i < 3; ++i) PQ[i] = x[32 * (LT + 1 + i)];
        if constexpr (F32) {
          lam = x[32 * (LT + 4)];
#pragma unroll
          for (int m = 1; m <= LT; ++m) lp[m] = lp[m - 1] * lam;
        }
      }
      if (ok) {
        const int slot = s.e & (kQ - 1);
        const double* wk = rec(Q[slot].x).pa.md + 4ull * Qo[slot].w + mc.ket_coef + s.ik * mc.ket_set;
        const int pos = __popc(okm & lt_mask);
        R* r = Rb + pos * kRow;
        for (int i = wt; i < mc.ket_set; i += NW) r[kW + i] = narrow(__ldg(wk + i));
        if constexpr (NW == 1) hermite<LT, 1, 0>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
        if constexpr (NW == 2) {
          if (wt == 0)
            hermite<LT, 2, 0>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
          else
            hermite<LT, 2, 1>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
        }
        if constexpr (NW == 4) {
          if (wt == 0)
            hermite<LT, 4, 0>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
          else if (wt == 1)
            hermite<LT, 4, 1>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
          else if (wt == 2)
            hermite<LT, 4, 2>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
          else
            hermite<LT, 4, 3>(B, PQ[0], PQ[1], PQ[2], lp, r, op);
        }
      }
      sync();
      // runs of lanes of one (quartet, bra primitive pair)
      const int e_up = __shfl_up_sync(0xffffffffu, s.e, 1), ib_up = __shfl_up_sync(0xffffffffu, s.ib, 1);
      unsigned lead = __ballot_sync(0xffffffffu, lane < ns && (lane == 0 || s.e != e_up || s.ib != ib_up));
      const unsigned last_k = __ballot_sync(0xffffffffu, s.ik == s.nk - 1);
      const unsigned last_q = __ballot_sync(0xffffffffu, s.ik == s.nk - 1 && s.ib == s.nb - 1);
      if constexpr (LT <= 2) {
        // 32 / md_group runs side by side, then the bra contraction of each.  The sum of a run cut by the end of
        // the 32 goes on with the next ones: as two contractions the FP32 pass's roundings depended on where in
        // the stream a quartet came (K of repeated mixed builds of 32 atoms differed by 9e-13; now by 1e-14).
        constexpr int GL = md_group(LT), G = 32 / GL;
        int* const first_row = reinterpret_cast<int*>(S + ly.Y - 18);
        const int nr = __popc(lead);
        if ((lead >> lane) & 1) first_row[__popc(lead & lt_mask)] = __popc(okm & lt_mask);
        if (lane == 0) first_row[nr] = __popc(okm);
        __syncwarp();
#pragma unroll 1
        for (int t0 = 0; t0 < nr; t0 += G) {
          const int t = t0 + lane / GL;
          const int p0 = t < nr ? first_row[t] : 0, len = t < nr ? first_row[t + 1] - p0 : 0;
          const int most = __reduce_max_sync(0xffffffffu, len);
          const R* r = Rb + p0 * kRow + kc_r[0];
          const R* w = Rb + p0 * kRow + kc_w[0];
          R v = h_valid && t == 0 ? carry : R(0);
#pragma unroll 4
          for (int p = 0; p < most; ++p)
            if (p < len) v = fmar(w[p * kRow], r[p * kRow], v);
          H[lane] = v;
          __syncwarp();
#pragma unroll 1
          for (int u = t0; u < min(t0 + G, nr); ++u) {
            const int l0 = __ffs(lead) - 1;
            lead &= lead - 1;
            const int l1 = lead ? __ffs(lead) - 1 : ns;
            const int np = first_row[u + 1] - first_row[u];
            const int slot = __shfl_sync(0xffffffffu, s.e, l0) & (kQ - 1), ib = __shfl_sync(0xffffffffu, s.ib, l0);
            const bool sum = np > 0 || (u == 0 && h_valid);
            n_eval += np;
            if (!((last_k >> (l1 - 1)) & 1)) {  // cut: the last run
              carry = H[(u - t0) * GL + lane % GL];
              h_valid = sum;
              continue;
            }
            if (sum) {
              bra_contract(bra_factors(slot, ib), H + (u - t0) * GL);
              a_valid = true;
            }
            if (u == 0) h_valid = false;
            if ((last_q >> (l1 - 1)) & 1) finish(slot);
          }
          __syncwarp();
        }
      } else {
        while (lead) {
          const int l0 = __ffs(lead) - 1;
          lead &= lead - 1;
          const int l1 = lead ? __ffs(lead) - 1 : ns;
          const int p0 = __popc(okm & ((1u << l0) - 1u)), p1 = __popc(okm & (0xffffffffu >> (32 - l1)));
          if (p1 > p0) {
            ket_contract(p0, p1);
            h_valid = true;
            n_eval += p1 - p0;
          }
          if ((last_k >> (l1 - 1)) & 1) {
            const int slot = __shfl_sync(0xffffffffu, s.e, l0) & (kQ - 1), ib = __shfl_sync(0xffffffffu, s.ib, l0);
            if (h_valid) {
              bra_contract(bra_factors(slot, ib), H);
              a_valid = true;
              h_valid = false;
            }
            if ((last_q >> (l1 - 1)) & 1) finish(slot);
          }
        }
      }
      if (32 * (sub + 1) >= n) {  // the stream's new head: after the last lane
        const int l = ns - 1;
        const int e_last = __shfl_sync(0xffffffffu, s.e, l);
        const int ib_last = __shfl_sync(0xffffffffu, s.ib, l), ik_last = __shfl_sync(0xffffffffu, s.ik, l);
        const bool done = (last_q >> l) & 1;
        head = done ? e_last + 1 : e_last;
        head_off = done ? 0 : ib_last * (Q[e_last & (kQ - 1)].w >> 16) + ik_last + 1;
      }
    }
    waiting -= n;
    sync();
  };

  // The team's next candidates, up to 32 of them, a lane each (the same in every warp): quartets
  // [q0, q1) of the list of Ls (system sys), r the row of q0; or pairs of the diagonal.
  long long q0 = 0, q1 = 0, c0 = 0, c1 = 0;
  int r = 0, sys = 0;
  bool first = true;
  const long long wid = blockIdx.x * kTeams + team, nteam = (long long)gridDim.x * kTeams;
  auto next_range = [&]() -> bool {
    if constexpr (KIND == MD_DIAG) {
      q0 = first ? wid : q0 - 32 + nteam;  // one pair at a time: q0 has been advanced by 32
      q1 = q0 + 1;
      first = false;
      return q0 < L.diag_n;
    } else {
      while (true) {
        if (KIND != MD_BATCH && KIND != MD_PER && L.schedule != 2) {
          if (!first) return false;
          first = false;
          group_range(L, wid, nteam, q0, q1);
        } else {
          if (c0 >= c1) {  // claim a chunk
            unsigned long long c = 0;
            if (lane == 0 && wt == 0) c = atomicAdd(L.work, (unsigned long long)L.chunk);
            if constexpr (NW == 1) {
              c = __shfl_sync(0xffffffffu, c, 0);
            } else {
              volatile unsigned long long* xc = reinterpret_cast<unsigned long long*>(Xok + 2 * NS);
              if (threadIdx.x == 0) *xc = c;
              __syncthreads();
              c = *xc;
              __syncthreads();
            }
            c0 = (long long)c;
            if (c0 >= L.q_count) return false;
            c1 = min(c0 + L.chunk, L.q_count);
          }
          if constexpr (KIND == MD_BATCH) {  // the chunk's part in the next system's list
            int lo = 0, hi = L.n_sys - 1;    // last s with seg[s] <= c0
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (__ldg(L.seg + mid) <= c0) lo = mid; else hi = mid - 1;
            }
            const long long e = min(c1, __ldg(L.seg + lo + 1)), s0 = __ldg(L.seg + lo);
            sys = lo;
            q0 = L.batch[lo].q_begin + (c0 - s0);
            q1 = L.batch[lo].q_begin + (e - s0);
            c0 = e;
          } else if constexpr (KIND == MD_PER) {  // the chunk's part in the next pass over the list
            sys = (int)(c0 / L.per.n_list);
            const long long s0 = sys * L.per.n_list, e = min(c1, s0 + L.per.n_list);
            q0 = L.q_begin + (c0 - s0);
            q1 = L.q_begin + (e - s0);
            c0 = e;
          } else {
            q0 = L.q_begin + c0;
            q1 = L.q_begin + c1;
            c0 = c1;
          }
        }
        if (q0 < q1) {
          const EriLaunch& Ls = rec(sys);
          r = find_row(Ls.qoff, Ls.row_begin, Ls.row_end, q0);
          return true;
        }
      }
    }
  };

  // one loop and one place for the batches: the kernel's code is large, and a second copy of it
  // cost more in instruction fetches than anything else in the FP32 pass
  for (bool more = true; more;) {
    if (q0 >= q1) more = next_range();
    bool keep = false;
    int bra_s = 0, ket_s = 0, nb = 0, nk = 0;
    if (more) {
      const long long q = q0 + lane;
      q0 += 32;
      if (q < q1) {
        if constexpr (KIND == MD_DIAG) {
          const int p = __ldg(L.diag_list + q);
          bra_s = ket_s = p;
          nb = nk = __ldg(L.pa.prim_n + p);
          keep = nb > 0;
          if (!keep && wt == 0) L.diag_Q[p] = 0.0;
        } else {
          const EriLaunch& Ls = rec(sys);
          while (__ldg(Ls.qoff + r + 1) <= q) ++r;
          bra_s = Ls.bra_bin_start + (r - Ls.row_begin);
          ket_s = Ls.ket_bin_start + (int)(q - __ldg(Ls.qoff + r));
          const int bra = __ldg(Ls.sorted + bra_s), ket = __ldg(Ls.sorted + ket_s);
          if constexpr (KIND == MD_PER) {
            PerQuartet pq;
            keep = per_quartet(Ls, sys, bra, ket, pq);  // a density block exists for its cell offset
          } else {
            const double pm = pmax4(Ls, __ldg(Ls.pa.sa + bra), __ldg(Ls.pa.sb + bra), __ldg(Ls.pa.sa + ket),
                                    __ldg(Ls.pa.sb + ket));
            keep = !(Ls.skip_zero && pm == 0.0) &&
                   !(Ls.dens_tau > 0.0 && __ldg(Ls.Qs + bra_s) * __ldg(Ls.Qs + ket_s) * pm < Ls.dens_tau) &&
                   dist_keeps(Ls, bra_s, ket_s) &&
                   (L.prec == PREC_FP64 || fp32_eligible(Ls, bra_s, ket_s, pm) == F32);
          }
          if (keep) {
            nb = __ldg(Ls.pa.prim_n + bra);
            nk = __ldg(Ls.pa.prim_n + ket);
            keep = nb > 0 && nk > 0;
          }
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      if (keep && wt == 0) {
        const EriLaunch& Ls = rec(sys);
        const int slot = (tail + __popc(m & lt_mask)) & (kQ - 1), bra = pair_id(Ls, bra_s), ket = pair_id(Ls, ket_s);
        Q[slot] = make_int4(sys, bra_s, ket_s, nb | (nk << 16));
        Qo[slot] = make_uint4(__ldg(Ls.pa.prim_off + bra), __ldg(Ls.pa.prim_off + ket),
                              (unsigned)(__ldg(Ls.pa.md_off + bra) >> 2), (unsigned)(__ldg(Ls.pa.md_off + ket) >> 2));
      }
      tail += __popc(m);
      waiting += __reduce_add_sync(0xffffffffu, keep ? nb * nk : 0);
      sync();
    }
    // full batches; short of full where the queue could not take the next 32 quartets, and at the end
    while (waiting >= 32 * NS || tail - head >= 32 || (!more && waiting > 0)) batch(min(waiting, 32 * NS));
  }
  if (KIND != MD_DIAG && lane == 0 && wt == 0) flush_tally(L, tally);
  record_busy(L, t0);
  // a launch completes after the one before it, so that what follows the last waits for all
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace hfx
