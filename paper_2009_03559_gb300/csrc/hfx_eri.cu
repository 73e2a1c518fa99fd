// Class launches: one evaluates every screened quartet of one class pair (bra pair bin >= ket
// pair bin) -- of one system, or of all systems of a batch -- and digests it into the half
// exchange matrix, or, in diagonal mode, evaluates (p|p) for candidate pairs and stores the
// Schwarz factor.  Here: the thread kernel (one quartet per thread, on request), and which
// kernel, chunk and overlap a launch gets; the default kernel is the Hermite engine (hfx_md.cu).
#include <algorithm>
#include <cstdio>
#include <type_traits>
#include "eri_engine.cuh"
#include "eri_quartets.cuh"
#include "hfx_eri.h"

namespace hfx {

const EriClassInfo* class_info_host() { return kClassInfo; }

// ---------------------------------------------------------------------------
// Contracted quartet, G = 1: the thread owns the quartet.  Group scratch slots are
// interleaved over the block's threads (slot k of thread t at smem[k*st + t]).
// ---------------------------------------------------------------------------
// ci is the launch's class record (kernel parameter space); L supplies the system's data.
// R = float runs the recurrences and the contraction on FP32 slots, slot k in the first half
// of the thread's own FP64 slot k (so no other lane's slots are ever touched); the
// accumulated block is then widened in place into the FP64 slots Sd, where the horizontal
// recurrences and the spherical step run.  R = double: the FP64 slots themselves.
template <typename R>
__device__ __forceinline__ int contract_g1(const EriClassInfo& ci, const EriLaunch& L, int bra, int ket, double* Sd,
                                           int st) {
  R* S = reinterpret_cast<R*>(Sd);
  const int sts = st * (int)(sizeof(double) / sizeof(R));  // slot stride in units of R
  const PairArrays pa = L.pa;
  const double omega = L.omega, omega2 = L.omega2;
  const double* boys = L.boys;
  Fp64 op;
  op.init();
  R* V = S + ci.work_base * sts;
  const int nb = __ldg(pa.prim_n + bra), nk = __ldg(pa.prim_n + ket);
  const PrimPair* pb = pa.prim + __ldg(pa.prim_off + bra);
  const PrimPair* pk = pa.prim + __ldg(pa.prim_off + ket);
  for (int a = 0; a < ci.n_acc; ++a) S[a * sts] = R(0);
  int any = 0;
  // one flat loop over the primitive quartets: lanes whose quartets have the same count
  // (the queue groups them so) run the same number of iterations
  const int npq = nb * nk;
  if constexpr (sizeof(R) == 4) {
    // vertical recurrences and contraction on FP32 slots for one primitive quartet
    auto vrr = [&](const CoefRgT<float>& cf, const float* Gf) {
      for (int m = 0; m <= ci.Lt; ++m) V[m * sts] = Gf[m];
      for (int lv = 0; lv < ci.n_bra_lv; ++lv) {
        const int off = ci.lv_off[lv], n = ci.lv_n[lv];
        for (int o = 0; o < n; ++o) vrr_bra<true>(ld_op(kVrrOps, off + o), V, S, sts, cf);
      }
      for (int lv = ci.n_bra_lv; lv < ci.n_bra_lv + ci.n_ket_lv; ++lv) {
        const int off = ci.lv_off[lv], n = ci.lv_n[lv];
        for (int o = 0; o < n; ++o) vrr_ket<true>(ld_op(kVrrOps, off + o), V, S, sts, cf);
      }
      for (int a = 0; a < ci.n_accl; ++a) {
        const uint32_t w = __ldg(kAccSrc + ci.acc_off + a);
        S[(w & 0xFFFF) * sts] += V[(w >> 16) * sts];
      }
    };
    // the FP64 set-up of one primitive quartet, rounded to FP32 (false: negligible)
    auto setup64 = [&](int t, CoefRgT<float>& cf, float* Gf) {
      const int ib = t / nk, ik = t - ib * nk;
      CoefRg c;
      double Gm[kMaxLt + 1];
      if (!prim_setup(pb[ib], pk[ik], ci.E, ci.F, ci.Lt, omega, omega2, boys, c, Gm, op)) return false;
      cf = coef_f32(c, ci.E, ci.F);
      for (int m = 0; m <= ci.Lt; ++m) Gf[m] = to_f32(Gm[m]);
      return true;
    };
    // FP32 set-up first; the primitive quartets it declines (bit t - c0 of pend) take the FP64
    // set-up at the end of their chunk of 96, so that a lane's FP64 set-ups run together with
    // the other lanes' instead of once per iteration in which any lane needs one
    const float omega_f = to_f32(omega);
    for (int c0 = 0; c0 < npq; c0 += 96) {
      const int c1 = min(npq, c0 + 96);
      unsigned pend0 = 0, pend1 = 0, pend2 = 0;
      for (int t = c0; t < c1; ++t) {
        const int ib = t / nk, ik = t - ib * nk;
        CoefRgT<float> cf;
        float Gf[kMaxLt + 1];
        const int stt = prim_setup_f32(pb[ib], pk[ik], ci.E, ci.F, ci.Lt, omega_f, cf, Gf, op);
        if (stt == F32_SKIP) continue;
        if (stt == F32_FP64) {
          const int u = t - c0;
          if (u < 32) pend0 |= 1u << u;
          else if (u < 64) pend1 |= 1u << (u - 32);
          else pend2 |= 1u << (u - 64);
          continue;
        }
        ++any;
        vrr(cf, Gf);
      }
      while (pend0 | pend1 | pend2) {
        int t;
        if (pend0) {
          t = c0 + __ffs(pend0) - 1;
          pend0 &= pend0 - 1;
        } else if (pend1) {
          t = c0 + 32 + __ffs(pend1) - 1;
          pend1 &= pend1 - 1;
        } else {
          t = c0 + 64 + __ffs(pend2) - 1;
          pend2 &= pend2 - 1;
        }
        CoefRgT<float> cf;
        float Gf[kMaxLt + 1];
        if (!setup64(t, cf, Gf)) continue;
        ++any;
        vrr(cf, Gf);
      }
    }
  } else {
    auto vrr = [&](const CoefRg& c, const double* Gm) {
      for (int m = 0; m <= ci.Lt; ++m) V[m * sts] = Gm[m];
      for (int lv = 0; lv < ci.n_bra_lv; ++lv) {
        const int off = ci.lv_off[lv], n = ci.lv_n[lv];
        for (int o = 0; o < n; ++o) vrr_bra<true>(ld_op(kVrrOps, off + o), V, S, sts, c);
      }
      for (int lv = ci.n_bra_lv; lv < ci.n_bra_lv + ci.n_ket_lv; ++lv) {
        const int off = ci.lv_off[lv], n = ci.lv_n[lv];
        for (int o = 0; o < n; ++o) vrr_ket<true>(ld_op(kVrrOps, off + o), V, S, sts, c);
      }
      for (int a = 0; a < ci.n_accl; ++a) {
        const uint32_t w = __ldg(kAccSrc + ci.acc_off + a);
        S[(w & 0xFFFF) * sts] += V[(w >> 16) * sts];
      }
    };
    for (int t = 0; t < npq; ++t) {
      const int ib = t / nk, ik = t - ib * nk;
      CoefRg c;
      double Gm[kMaxLt + 1];
      if (!prim_setup(pb[ib], pk[ik], ci.E, ci.F, ci.Lt, omega, omega2, boys, c, Gm, op)) continue;
      ++any;
      vrr(c, Gm);
    }
  }
  if (!any) return 0;
  if constexpr (sizeof(R) == 4) {
    for (int a = 0; a < ci.n_acc; ++a) Sd[a * st] = to_f64(S[a * sts]);  // in place: read, then write
  }
  double AB[3], CD[3];
  for (int i = 0; i < 3; ++i) {
    AB[i] = __ldg(pa.AB + 3 * bra + i);
    CD[i] = __ldg(pa.AB + 3 * ket + i);
  }
  for (int s = 0; s < ci.n_post; ++s) {
    const int off = ci.post_off[s], n = ci.post_n[s], type = ci.post_type[s];
    for (int o = 0; o < n; ++o) post_op(ld_op(kPostOps, off + o), type, Sd, st, AB, CD);
  }
  return any;
}

// Register caps (blocks of 64 threads per SM): FP64 6 (at most 170 registers), measured fastest;
// the FP32 pass, which carries both set-ups, 4 to stay free of spills.
#ifndef HFX_G1_MINB
#define HFX_G1_MINB 6
#endif
#ifndef HFX_G1F_MINB
#define HFX_G1F_MINB 4
#endif

// One quartet evaluated and digested by one lane (one quartet per thread), recurrences in
// precision R; Sd: the thread's FP64 slots.
template <typename R>
__device__ __forceinline__ void g1_quartet(const EriClassInfo& ci, const EriLaunch& Ls, int bra_s, int ket_s,
                                           double* Sd, int st, Tally& t) {
  const int bra = __ldg(Ls.sorted + bra_s), ket = __ldg(Ls.sorted + ket_s);
  const int sa = __ldg(Ls.pa.sa + bra), sb = __ldg(Ls.pa.sb + bra);
  const int sc = __ldg(Ls.pa.sa + ket), sd = __ldg(Ls.pa.sb + ket);
  const int npq = __ldg(Ls.pa.prim_n + bra) * __ldg(Ls.pa.prim_n + ket);
  const int ne = contract_g1<R>(ci, Ls, bra, ket, Sd, st);
  t.prim += ne;
  t.skip += npq - ne;
  if (!ne) return;
  ++t.quart;
  if (sizeof(R) == 4) {
    ++t.q32;
    t.p32 += ne;
  }
  double deg = Ls.unscale;
  if (sa == sb) deg *= 0.5;
  if (sc == sd) deg *= 0.5;
  if (bra_s == ket_s) deg *= 0.5;
  digest(ci, Sd + ci.out_base * st, st, __ldg(Ls.sh.bf_off + sa), __ldg(Ls.sh.bf_off + sb), __ldg(Ls.sh.bf_off + sc),
         __ldg(Ls.sh.bf_off + sd), deg, Ls.P, Ls.K, Ls.ld, 0, 1);
}

// Per-warp queue of the quartets that pass the density tests (64 entries: bra position, ket
// position, primitive quartets, unused).  Lanes evaluate quartets 32 at a time, the
// 32 with the most primitive quartets first, so that few lanes idle while the others
// finish their primitive loops (the FP64 pipe charges a warp instruction in full whatever
// the number of active lanes).
struct G1Queue {
  int4* q;
  int n;
};

// Descending bitonic sort of 64 keys, two per lane (element i = lane + 32 h).
__device__ __forceinline__ void sort64_desc(int& k0, int& k1, int lane) {
#pragma unroll
  for (int size = 2; size <= 64; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      int o0, o1;
      if (stride == 32) {
        o0 = k1;
        o1 = k0;
      } else {
        o0 = __shfl_xor_sync(0xffffffffu, k0, stride);
        o1 = __shfl_xor_sync(0xffffffffu, k1, stride);
      }
      const int i0 = lane, i1 = lane + 32;
      const int j0 = i0 ^ stride, j1 = i1 ^ stride;
      const bool d0 = ((min(i0, j0) & size) == 0), d1 = ((min(i1, j1) & size) == 0);
      const bool m0 = (i0 < j0) == d0, m1 = (i1 < j1) == d1;
      k0 = m0 ? max(k0, o0) : min(k0, o0);
      k1 = m1 ? max(k1, o1) : min(k1, o1);
    }
  }
}

template <typename R>
__device__ __forceinline__ void g1_drain(const EriLaunch& L, G1Queue& Q, int lane, double* Sd, int st, Tally& t,
                                         bool all) {
  while (Q.n >= 32 || (all && Q.n > 0)) {
    int4 e;
    int take;
    if (Q.n >= 32) {
      // the 32 entries with the most primitive quartets; the rest move to the front
      int k0 = lane < Q.n ? ((Q.q[lane].z << 6) | lane) : -1;
      int k1 = lane + 32 < Q.n ? ((Q.q[lane + 32].z << 6) | (lane + 32)) : -1;
      sort64_desc(k0, k1, lane);
      e = Q.q[k0 & 63];
      int4 rest = make_int4(0, 0, 0, 0);
      if (k1 >= 0) rest = Q.q[k1 & 63];
      __syncwarp();
      if (k1 >= 0) Q.q[lane] = rest;
      take = 32;
    } else {
      e = Q.q[lane];
      take = Q.n;
    }
    __syncwarp();
    Q.n -= take;
    if (lane < take) g1_quartet<R>(L.ci, L, e.x, e.y, Sd, st, t);
  }
}

// Quartets [q0, q1) of the list, one quartet per thread: the warp tests 32 consecutive quartets
// at a time and queues the survivors.
template <int PREC, typename R>
__device__ __forceinline__ void g1_range(const EriLaunch& L, long long q0, long long q1, double* Sd, int st, int lane,
                                         G1Queue& Q, Tally& t) {
  const long long* qoff = L.qoff;
  const int row_begin = L.row_begin, bra0 = L.bra_bin_start, ket0 = L.ket_bin_start;
  const bool skip = L.skip_zero;
  const double dens = L.dens_tau;
  int r = -1;
  for (long long base = q0; base < q1; base += 32) {
    const long long q = base + lane;
    bool keep = false;
    int bra_s = 0, ket_s = 0, npq = 0;
    if (q < q1) {
      if (r < 0) r = find_row(qoff, row_begin, L.row_end, q);
      while (__ldg(qoff + r + 1) <= q) ++r;
      bra_s = bra0 + (r - row_begin);
      ket_s = ket0 + (int)(q - __ldg(qoff + r));
      const int bra = __ldg(L.sorted + bra_s), ket = __ldg(L.sorted + ket_s);
      const double pm = pmax4(L, __ldg(L.pa.sa + bra), __ldg(L.pa.sb + bra), __ldg(L.pa.sa + ket),
                              __ldg(L.pa.sb + ket));
      keep = !(skip && pm == 0.0) && !(dens > 0.0 && __ldg(L.Qs + bra_s) * __ldg(L.Qs + ket_s) * pm < dens) &&
             dist_keeps(L, bra_s, ket_s) && pass_takes<PREC>(L, bra_s, ket_s, pm);
      npq = __ldg(L.pa.prim_n + bra) * __ldg(L.pa.prim_n + ket);
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep) Q.q[Q.n + __popc(m & ((1u << lane) - 1u))] = make_int4(bra_s, ket_s, npq, 0);
    Q.n += __popc(m);
    __syncwarp();
    g1_drain<R>(L, Q, lane, Sd, st, t, false);
  }
}

template <int PREC>
__global__ void __launch_bounds__(64, PREC == PREC_MIXED32 ? HFX_G1F_MINB : HFX_G1_MINB)
    eri_g1_kernel(const EriLaunch L) {
  extern __shared__ double smem[];
  const int st = blockDim.x;
  double* Sd = smem + threadIdx.x;
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long ng = (long long)gridDim.x * blockDim.x;
  unsigned long long t0 = 0;
  if (L.busy && threadIdx.x == 0) t0 = globaltimer_ns();
  using R = typename std::conditional<PREC == PREC_MIXED32, float, double>::type;
  const int lane = threadIdx.x & 31;
  Tally t;
  G1Queue Q{reinterpret_cast<int4*>(smem + (size_t)L.ci.scratch * blockDim.x) + (threadIdx.x >> 5) * 64, 0};
  for_each_range(L, gid >> 5, ng >> 5, lane,
                 [&](long long q0, long long q1) { g1_range<PREC, R>(L, q0, q1, Sd, st, lane, Q, t); });
  g1_drain<R>(L, Q, lane, Sd, st, t, true);
  flush_tally(L, t);
  record_busy(L, t0);
}

// ---------------------------------------------------------------------------
// Host-side launch helpers
// ---------------------------------------------------------------------------
static const int kBlock = 64;

// Whole warps, but for long lists of uncontracted quartets in the nine classes of at most 100 slots a thread.
// The Hermite engine's steps after the contraction cost a warp the same for 1 primitive quartet as for 81: with
// 3 primitives a shell it is the faster in every class (64-atom diamond, (ss|ss) 17.0 -> 11.2 ms, (pp|ps)
// 219 -> 129 ms, (dd|ss) 44 -> 26 ms), with 2 too (24 atoms, 1.3 to 4.8 times), with 1 the thread kernel
// (64 atoms: (ss|ss) 0.92 -> 0.48 ms, (ps|ss) 3.63 -> 1.40, (pp|ps) 7.36 -> 5.81, (dd|ss) 3.87 -> 2.14; whole
// build 306 -> 291 ms; 300 s shells 4.18 -> 1.24 ms) where a list is long enough for four quartets a thread (24
// atoms, 260 000: (pp|ps) 0.61 -> 0.58 ms; 190 000: (ds|ps) 0.44 -> 0.47; 90 000: (ds|ss) 0.23 -> 0.27).  Groups of 8 or 16 lanes were slower than
// either in every class.
int eri_group_size(int cls, bool uncontracted, long long n_quartets, int n_sm) {
  if (!uncontracted || kClassInfo[cls].scratch > HFX_G1_MAX_SCRATCH) return 32;
  return n_quartets >= 4ll * n_sm * eri_blocks_per_sm(cls, 0, 1, PREC_FP64, false) * kBlock ? 1 : 32;
}

bool eri_group_size_valid(int gs) { return gs == 1 || gs == 32; }

// Streams (primitive quartets of one quartet run at a time by the schedules of the former warp
// kernel): the choice is still taken, checked and reported, and no kernel depends on it.  The
// values a class carries, the largest up to its default last chosen.
static const int kDefaultStreams[HFX_N_CLASSES] = {
    4, 4, 4, 4, 4, 4,   // ss|ss ps|ss ps|ps pp|ss pp|ps pp|pp
    4, 4, 4, 4,         // ds|ss ds|ps ds|pp ds|ds
    4, 4, 2, 4, 2,      // dp|ss dp|ps dp|pp dp|ds dp|dp
    4, 4, 2, 2, 1, 1};  // dd|ss dd|ps dd|pp dd|ds dd|dp dd|dd

static int variant_index(int cls, int streams) {
  const int* v = kStreams[cls];
  if (streams > 0) {
    for (int i = 0; i < 3; ++i)
      if (v[i] == streams) return i;
    return -1;
  }
  int best = 0;  // the largest variant carried up to the default
  for (int i = 1; i < 3; ++i)
    if (v[i] && v[i] <= kDefaultStreams[cls]) best = i;
  return best;
}

bool eri_streams_valid(int cls, int streams) {
  return cls >= 0 && cls < HFX_N_CLASSES && (streams == 0 || variant_index(cls, streams) >= 0);
}

int eri_streams(int cls, int streams) {
  const int i = variant_index(cls, streams);
  return i < 0 ? 0 : kStreams[cls][i];
}

// The kernel of a class launch: the Hermite engine (md_*) on whole warps, in FP32 for the FP32
// pass; the thread kernel for gs = 1.
static int md_kind(int mode, int prec, bool batch) {
  return mode == 1 ? MD_DIAG : prec == PREC_PERIODIC ? MD_PER : batch ? MD_BATCH : MD_PLAIN;
}

static const void* g1_kernel(int prec) {
  if (prec == PREC_MIXED64) return (const void*)eri_g1_kernel<PREC_MIXED64>;
  if (prec == PREC_MIXED32) return (const void*)eri_g1_kernel<PREC_MIXED32>;
  return (const void*)eri_g1_kernel<PREC_FP64>;
}

// one quartet per thread: interleaved scratch, then a 64-entry quartet queue per warp
static size_t g1_smem_bytes(int cls) {
  return sizeof(double) * (size_t)kClassInfo[cls].scratch * kBlock + sizeof(int4) * 64 * (kBlock / 32);
}

cudaError_t eri_prepare() {
  // allow the largest dynamic shared memory any class needs, for every instance
  size_t mx = 0;
  for (int c = 0; c < HFX_N_CLASSES; ++c) mx = std::max(mx, g1_smem_bytes(c));
  if (mx > 227 * 1024) mx = 227 * 1024;
  cudaError_t e = md_prepare();
  for (int prec : {PREC_FP64, PREC_MIXED64, PREC_MIXED32})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(g1_kernel(prec), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mx);
  return e;
}

int eri_blocks_per_sm(int cls, int mode, int gs, int prec, bool batch) {
  if (gs != 1) return md_blocks_per_sm(cls, md_kind(mode, prec, batch), prec == PREC_MIXED32);
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, g1_kernel(prec), kBlock, g1_smem_bytes(cls)) != cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

int eri_groups_per_block(int cls, int gs) {
  return gs == 1 ? kBlock : md_teams_per_block(cls);
}

// Quartets per claim of the dynamic schedule.  A thread-kernel warp takes 256.  A whole warp takes
// at most 32 (it tests a claim's quartets with a lane each) and at least 1: a 32nd of an even
// share of the list, so that the last claims of a launch, while the other warps are done, stay a
// few per cent of it also for the smallest systems, where a claim of 8 left most warps without one.
int eri_chunk(int gs, long long n_quartets, long long n_groups) {
  if (gs == 1) return 256;
  return (int)std::max(1LL, std::min(32LL, n_quartets / (32 * std::max(1LL, n_groups))));
}

// Whether the next class launch of a build is let start before a launch of n_quartets on n_groups
// warps has ended.  Below 32 quartets a warp the launch is mostly ramp and tail (3-atom diamond build
// 1.14 -> 0.52 ms, 8 atoms 8.6 -> 8.1 ms; then 0.41 and 7.9 with the longest classes first); above,
// two classes sharing the SMs cost more than the tail (64 atoms 1781 -> 1806 ms when all overlapped;
// 16 atoms 55.2 -> 55.4 with the line at 96).
bool eri_overlap(int gs, long long n_quartets, long long n_groups) { return gs != 1 && n_quartets < 32 * n_groups; }

cudaError_t eri_launch(const EriLaunch& L0, int cls, int mode, int grid, cudaStream_t stream, int gs, int prec,
                       bool batch, bool overlap) {
  if (gs != 1) return md_launch(L0, cls, md_kind(mode, prec, batch), prec, prec == PREC_MIXED32, grid, stream, overlap);
  // the thread kernel: builds of one system, classes whose slots fit
  const size_t smem = g1_smem_bytes(cls);
  if (mode != 0 || batch || prec == PREC_PERIODIC || smem > 227 * 1024) return cudaErrorInvalidValue;
  EriLaunch L = L0;
  void* args[] = {(void*)&L};
  return cudaLaunchKernel(g1_kernel(prec), dim3(grid), dim3(kBlock), args, smem, stream);
}

}  // namespace hfx
