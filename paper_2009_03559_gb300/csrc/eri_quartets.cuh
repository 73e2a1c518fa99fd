// What the ERI kernels share: the quartet list (rows, ranges, chunks), the screening tests,
// the precision passes, the periodic quartets and their digest, the counters.
#pragma once
#include "hfx_internal.cuh"

namespace hfx {

// Locate the row of quartet q (global index) in [rlo, rhi): qoff[r] <= q < qoff[r+1].
__device__ __forceinline__ int find_row(const long long* qoff, int rlo, int rhi, long long q) {
  int lo = rlo, hi = rhi - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(qoff + mid) <= q) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// The quartet range [q0, q1) handled by group gid of ngroups.
__device__ __forceinline__ void group_range(const EriLaunch& L, long long gid, long long ngroups,
                                            long long& q0, long long& q1) {
  if (L.schedule == 1) {
    // parallel-pair split (paper Algorithm 2): an even share of the bra pairs, whatever
    // the number of quartets they carry
    const long long nr = L.row_end - L.row_begin;
    const int r0 = L.row_begin + (int)(nr * gid / ngroups);
    const int r1 = L.row_begin + (int)(nr * (gid + 1) / ngroups);
    q0 = __ldg(L.qoff + r0);
    q1 = __ldg(L.qoff + r1);
  } else {
    // parallel-quartet split (paper Algorithm 3 without the replicated screening): an
    // even share of the screened quartet list
    q0 = L.q_begin + L.q_count * gid / ngroups;
    q1 = L.q_begin + L.q_count * (gid + 1) / ngroups;
  }
}

// Precision passes of a class launch: 0 every quartet in FP64; 1 (mixed precision, first
// pass) the quartets that must stay FP64; 2 (second pass) those whose recurrences run in FP32.
// PREC_PERIODIC: the FP64 periodic instance (quartets of the lattice sums, see per_quartet).
enum { PREC_FP64 = 0, PREC_MIXED64 = 1, PREC_MIXED32 = 2, PREC_PERIODIC = 3 };

// The digest reads P_bd, P_bc, P_ad, P_ac.  max of their max|P| (or 1 without the table):
// 0 means the quartet contributes exactly nothing; the mixed-precision and the
// density-weighted screening tests use it too.
__device__ __forceinline__ double pmax4(const EriLaunch& L, int sa, int sb, int sc, int sd) {
  if (!L.pmax) return 1.0;
  const double* pm = L.pmax;
  const size_t ns = L.ns;
  return fmax(fmax(__ldg(pm + sb * ns + sd), __ldg(pm + sb * ns + sc)),
              fmax(__ldg(pm + sa * ns + sd), __ldg(pm + sa * ns + sc)));
}

// Distance-aware test: Q_IJ Q_KL exp(-kappa rho R^2) >= dist_tau (see hfx_options.dist_tau).
__device__ __forceinline__ bool dist_keeps(const EriLaunch& Ls, int bra_s, int ket_s) {
  if (!(Ls.dist_tau > 0.0)) return true;
  const double* a = Ls.dist + 5 * (size_t)bra_s;
  const double* b = Ls.dist + 5 * (size_t)ket_s;
  const double dx = __ldg(a) - __ldg(b), dy = __ldg(a + 1) - __ldg(b + 1), dz = __ldg(a + 2) - __ldg(b + 2);
  double r = sqrt(dx * dx + dy * dy + dz * dz) - __ldg(a + 3) - __ldg(b + 3);
  if (r < 0.0) r = 0.0;
  const double p = __ldg(a + 4), q = __ldg(b + 4);
  const double rho = p * q / (p + q);
  const double lam = Ls.omega2 * rho / (Ls.omega2 + rho);
  return __ldg(Ls.Qs + bra_s) * __ldg(Ls.Qs + ket_s) * exp(-lam * r * r) >= Ls.dist_tau;
}

// Mixed precision: FP32 recurrences for the quartet when the class allows it and its
// Schwarz bound times the largest density element it touches (or the largest of all of P)
// is below fp32_tau.
__device__ __forceinline__ bool fp32_eligible(const EriLaunch& Ls, int bra_s, int ket_s, double pm) {
  if (!Ls.fp32_ok) return false;
  const double pf = Ls.pglob ? __ldg(Ls.pglob) : pm;
  return __ldg(Ls.Qs + bra_s) * __ldg(Ls.Qs + ket_s) * pf < Ls.fp32_tau;
}

// whether pass PREC takes the quartet
template <int PREC>
__device__ __forceinline__ bool pass_takes(const EriLaunch& Ls, int bra_s, int ket_s, double pm) {
  if constexpr (PREC == PREC_FP64) return true;
  const bool f32 = fp32_eligible(Ls, bra_s, ket_s, pm);
  return PREC == PREC_MIXED32 ? f32 : !f32;
}

__device__ __forceinline__ void record_busy(const EriLaunch& L, unsigned long long t0) {
  if (L.busy && threadIdx.x == 0) {
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    atomicAdd(L.busy + smid, globaltimer_ns() - t0);
  }
}

// ---------------------------------------------------------------------------
// Periodic quartets (Eq. vx with lattice images): the pass for cell G evaluates
// (X | Y + shift) for bra pair X and ket pair Y of the home-anchored pair list and adds
//   K^G_{ab} += sum_{c,d} (a c | b d) P^{R}_{cd},   R = cell(d) - cell(c),
// where a is the home-cell shell of the pair holding the row function (X for a forward
// pass, Y for a reverse one), c its partner, b the home-cell shell of the other pair
// (in cell G) and d its partner.  Every ordered pair of pairs is one quartet (no
// permutational symmetry is used across cells), so the degeneracy factor is 1.
// ---------------------------------------------------------------------------
struct PerQuartet {
  int pa, pb, pc, pd;        // positions of shells a, b, c, d in the quartet block (x1 x2 y1 y2)
  int bfa, bfb, bfc, bfd;    // their first functions (home-cell numbering)
  const double* PR;          // density block P^R
};

__device__ __forceinline__ bool per_quartet(const EriLaunch& L, int pass, int bra, int ket, PerQuartet& q) {
  const PeriodicInfo& pi = L.per;
  const PerCell& cell = pi.cells[pass];
  const bool reverse = __ldg(&cell.reverse);
  const int sax = __ldg(L.pa.sa + bra), sbx = __ldg(L.pa.sb + bra);
  const int say = __ldg(L.pa.sa + ket), sby = __ldg(L.pa.sb + ket);
  const bool hx = __ldg(pi.home_first + bra), hy = __ldg(pi.home_first + ket);
  const int hxs = hx ? sax : sbx, oxs = hx ? sbx : sax;
  const int hys = hy ? say : sby, oys = hy ? sby : say;
  const int* cx = pi.cell_xyz + 3 * __ldg(pi.shell_cell + oxs);
  const int* cy = pi.cell_xyz + 3 * __ldg(pi.shell_cell + oys);
  const int w = 2 * pi.rb + 1;
  int idx = 0;
  for (int i = 0; i < 3; ++i) {
    const int d = __ldg(cy + i) - __ldg(cx + i);
    const int R = __ldg(&cell.gcell[i]) + (reverse ? -d : d);
    if (R < -pi.rb || R > pi.rb) return false;
    idx = idx * w + (R + pi.rb);
  }
  const int blk = __ldg(pi.rmap + idx);
  if (blk < 0) return false;
  // an exactly zero density block P^R_{cd} makes the quartet's contribution exactly zero
  {
    const int c = reverse ? oys : oxs, d = reverse ? oxs : oys;
    if (__ldg(pi.pmax + ((size_t)blk * pi.nsh + c % pi.nsh) * pi.nsh + d % pi.nsh) == 0.0) return false;
  }
  q.PR = pi.P + (size_t)blk * pi.nbf * pi.nbf;
  const int phx = hx ? 0 : 1, pox = 1 - phx, phy = hy ? 2 : 3, poy = 5 - phy;
  if (!reverse) {
    q.pa = phx; q.pc = pox; q.pb = phy; q.pd = poy;
    q.bfa = __ldg(pi.shell_bf + hxs); q.bfc = __ldg(pi.shell_bf + oxs);
    q.bfb = __ldg(pi.shell_bf + hys); q.bfd = __ldg(pi.shell_bf + oys);
  } else {
    q.pa = phy; q.pc = poy; q.pb = phx; q.pd = pox;
    q.bfa = __ldg(pi.shell_bf + hys); q.bfc = __ldg(pi.shell_bf + oys);
    q.bfb = __ldg(pi.shell_bf + hxs); q.bfd = __ldg(pi.shell_bf + oxs);
  }
  return true;
}

// K^G_{ab} += sum_{cd} v P^R_{cd} for the final block v (stride st); outputs o0, o0 + ostep, ...
__device__ __forceinline__ void digest_per(const EriClassInfo& ci, const double* v, int st, const PerQuartet& q,
                                           double* KG, int nbf, int o0, int ostep) {
  int str[4];
  str[3] = 1;
  str[2] = ci.dims[3];
  str[1] = ci.dims[2] * str[2];
  str[0] = ci.dims[1] * str[1];
  const int na = ci.dims[q.pa], nb = ci.dims[q.pb], nc = ci.dims[q.pc], nd = ci.dims[q.pd];
  const int sa = str[q.pa], sb = str[q.pb], sc = str[q.pc], sd = str[q.pd];
  for (int o = o0; o < na * nb; o += ostep) {
    const int ia = o / nb, ib = o - ia * nb;
    double acc = 0.0;
    for (int ic = 0; ic < nc; ++ic)
      for (int id = 0; id < nd; ++id)
        acc = fma(v[(ia * sa + ib * sb + ic * sc + id * sd) * st], __ldg(q.PR + (size_t)(q.bfc + ic) * nbf + q.bfd + id),
                  acc);
    atomicAdd(KG + (size_t)(q.bfa + ia) * nbf + q.bfb + ib, acc);
  }
}

// Per-thread tallies of one kernel, added to the launch's counters once at the end.
struct Tally {
  unsigned long long prim = 0, quart = 0, skip = 0, q32 = 0, p32 = 0, run = 0;
};

// The quartet ranges a warp of the thread kernel works on.  Static schedules: one range (group_range).
// Dynamic: chunks claimed from the launch's device counter.
template <class F>
__device__ __forceinline__ void for_each_range(const EriLaunch& L, long long wid, long long nw, int lane, F&& f) {
  if (L.schedule != 2) {
    long long q0, q1;
    group_range(L, wid, nw, q0, q1);
    f(q0, q1);
    return;
  }
  while (true) {
    unsigned long long c = 0;
    if (lane == 0) c = atomicAdd(L.work, (unsigned long long)L.chunk);
    const long long c0 = (long long)__shfl_sync(0xffffffffu, c, 0);
    if (c0 >= L.q_count) break;
    f(L.q_begin + c0, L.q_begin + min(c0 + L.chunk, L.q_count));
  }
}

__device__ __forceinline__ void flush_tally(const EriLaunch& L, const Tally& t) {
  if (!L.counters) return;
  atomicAdd(L.counters + 0, t.prim);
  atomicAdd(L.counters + 1, t.quart);
  atomicAdd(L.counters + 2, t.skip);
  atomicAdd(L.counters + 3, t.q32);
  atomicAdd(L.counters + 4, t.p32);
  atomicAdd(L.counters + 5, t.run);
}

}  // namespace hfx
