// Host side of the Hermite engine: class descriptions, launches, and the pair data it reads.
#include <algorithm>
#include <cmath>
#include "hfx_md.cuh"
#include "hfx_eri.h"

namespace hfx {

const MdClassInfo* md_class_host() { return kMdClass; }
const MdPairInfo* md_pair_host() { return kMdPair; }
const int (*md_flops_host())[4] { return kMdFlops; }

const void* md_kernel_l0(int kind, bool f32);
const void* md_kernel_l1(int kind, bool f32);
const void* md_kernel_l2(int kind, bool f32);
const void* md_kernel_l3(int kind, bool f32);
const void* md_kernel_l4(int kind, bool f32);
const void* md_kernel_l5(int kind, bool f32);
const void* md_kernel_l6(int kind, bool f32);
const void* md_kernel_l7(int kind, bool f32);
const void* md_kernel_l8(int kind, bool f32);

static const void* md_kernel(int Lt, int kind, bool f32) {
  switch (Lt) {
    case 0: return md_kernel_l0(kind, f32);
    case 1: return md_kernel_l1(kind, f32);
    case 2: return md_kernel_l2(kind, f32);
    case 3: return md_kernel_l3(kind, f32);
    case 4: return md_kernel_l4(kind, f32);
    case 5: return md_kernel_l5(kind, f32);
    case 6: return md_kernel_l6(kind, f32);
    case 7: return md_kernel_l7(kind, f32);
    default: return md_kernel_l8(kind, f32);
  }
}

static MdLayout layout_of(int cls, bool f32) {
  int hi = 0;
  while ((hi + 1) * (hi + 2) / 2 <= cls) ++hi;
  const MdPairInfo &b = kMdPair[hi], &k = kMdPair[cls - hi * (hi + 1) / 2];
  return f32 ? md_layout<float>(kMdClass[cls], b, k) : md_layout<double>(kMdClass[cls], b, k);
}

int md_teams_per_block(int cls) {
  const int l = kMdClass[cls].Lt;
  return md_block(l) / (32 * md_team(l));
}

size_t md_smem_bytes(int cls, bool f32) {
  return sizeof(double) * (size_t)layout_of(cls, f32).size * md_teams_per_block(cls);
}

cudaError_t md_prepare() {
  for (bool f32 : {false, true}) {
    int mx[kMaxLt + 1] = {};
    for (int c = 0; c < HFX_N_CLASSES; ++c)
      mx[kMdClass[c].Lt] = std::max(mx[kMdClass[c].Lt], (int)md_smem_bytes(c, f32));
    for (int l = 0; l <= kMaxLt; ++l)
      for (int kind : {MD_PLAIN, MD_BATCH, MD_PER, MD_DIAG}) {
        const void* k = md_kernel(l, kind, f32);
        if (!k) continue;
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, mx[l]);
        if (e != cudaSuccess) return e;
      }
  }
  return cudaSuccess;
}

int md_blocks_per_sm(int cls, int kind, bool f32) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, md_kernel(kMdClass[cls].Lt, kind, f32), md_block(kMdClass[cls].Lt),
                                                    md_smem_bytes(cls, f32)) != cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

// overlap: the launch may start while the one before it on the stream (a class launch of the same
// build) still runs.  The launches of a build are independent (their K updates are atomic, their
// work counters apart), so the last quartets of one class, with most SMs idle, run beside the
// first of the next.  Each kernel lets its successor start at once and itself ends only after its
// predecessor has (griddepcontrol), so the build's last launch ends after all of them.
cudaError_t md_launch(const EriLaunch& L0, int cls, int kind, int prec, bool f32, int grid, cudaStream_t stream,
                      bool overlap) {
  EriLaunch L = L0;
  L.mc = kMdClass[cls];
  L.prec = prec == PREC_PERIODIC ? PREC_FP64 : prec;
  MdLayout ly = layout_of(cls, f32);
  void* args[] = {(void*)&L, (void*)&ly};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(md_block(L.mc.Lt));
  cfg.dynamicSmemBytes = md_smem_bytes(cls, f32);
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, md_kernel(L.mc.Lt, kind, f32), args);
}

// ---------------------------------------------------------------------------
// Pair data: per candidate pair the coefficients T of its type (polynomials in AB, times `scale`), then the
// factors W_s = u_b^i u_a^j (1/2p)^e of its surviving primitive pairs.
// ---------------------------------------------------------------------------
struct MdPairs {
  MdPairInfo t[6];
};

static MdPairs pair_infos() {
  MdPairs m;
  for (int i = 0; i < 6; ++i) m.t[i] = kMdPair[i];
  return m;
}

__global__ void k_md_size(int n, const int* __restrict__ pcls, const int* __restrict__ cap, const MdPairs info,
                          long long* __restrict__ size) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const MdPairInfo& t = info.t[pcls[c]];
  size[c] = (t.n_coef + (long long)t.n_set * cap[c] + 3) & ~3ll;  // the engine counts in fours
}

// one warp per pair
__global__ void k_md_fill(int n, const int* __restrict__ pcls, const double* __restrict__ AB,
                          const int* __restrict__ pp_off, const int* __restrict__ pp_n,
                          const PrimPair* __restrict__ pp, const long long* __restrict__ md_off, const MdPairs info,
                          double scale, double* __restrict__ md) {
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (c >= n) return;
  const MdPairInfo& t = info.t[pcls[c]];
  double* out = md + md_off[c];
  const double x[3] = {AB[3 * c], AB[3 * c + 1], AB[3 * c + 2]};
  for (int i = lane; i < t.n_coef; i += 32) {
    const uint32_t d = kMdCoef[t.coef0 + i];
    double v = 0.0;
    for (uint32_t k = d & 0xFFFF; k < (d & 0xFFFF) + (d >> 16); ++k) {
      // monomial number: degree, then x power, then y power descending
      int m = kMdTermMono[k], deg = 0, px, py;
      while (m >= (deg + 1) * (deg + 2) / 2) {
        m -= (deg + 1) * (deg + 2) / 2;
        ++deg;
      }
      for (px = deg; m > deg - px; --px) m -= deg - px + 1;
      py = deg - px - m;
      double w = kMdTermVal[k];
      for (int j = 0; j < px; ++j) w *= x[0];
      for (int j = 0; j < py; ++j) w *= x[1];
      for (int j = 0; j < deg - px - py; ++j) w *= x[2];
      v += w;
    }
    out[i] = v * scale;
  }
  out += t.n_coef;
  const PrimPair* p = pp + pp_off[c];
  for (int i = lane; i < pp_n[c] * t.n_set; i += 32) {
    const int k = i / t.n_set, s = t.set[i - k * t.n_set];
    double w = 1.0;
    for (int j = 0; j < ((s >> 4) & 15); ++j) w *= p[k].ub;
    for (int j = 0; j < (s >> 8); ++j) w *= p[k].ua;
    for (int j = 0; j < (s & 15); ++j) w *= p[k].inv2p;
    out[i] = w;
  }
}

cudaError_t launch_md_size(int n, const int* pcls, const int* cap, long long* size, cudaStream_t s) {
  k_md_size<<<(n + 255) / 256, 256, 0, s>>>(n, pcls, cap, pair_infos(), size);
  return cudaGetLastError();
}

cudaError_t launch_md_fill(int n, const int* pcls, const double* AB, const int* pp_off, const int* pp_n,
                           const PrimPair* pp, const long long* md_off, int hexp, double* md, cudaStream_t s) {
  k_md_fill<<<(n + 3) / 4, 128, 0, s>>>(n, pcls, AB, pp_off, pp_n, pp, md_off, pair_infos(),
                                              std::ldexp(1.0, -hexp / 2), md);
  return cudaGetLastError();
}

}  // namespace hfx
