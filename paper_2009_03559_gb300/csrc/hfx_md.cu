// Instances of the Hermite engine for one total angular momentum (HFX_MD_L, compiled once for
// each so that the instances build in parallel).
#include <algorithm>
#include "hfx_md.cuh"

#define HFX_CAT2(a, b) a##b
#define HFX_CAT(a, b) HFX_CAT2(a, b)

namespace hfx {
const void* HFX_CAT(md_kernel_l, HFX_MD_L)(int kind, bool f32) {
  constexpr int l = HFX_MD_L;
  if (f32)
    return kind == MD_PLAIN   ? (const void*)eri_md_kernel<l, MD_PLAIN, float>
           : kind == MD_BATCH ? (const void*)eri_md_kernel<l, MD_BATCH, float>
                              : nullptr;
  switch (kind) {
    case MD_PLAIN: return (const void*)eri_md_kernel<l, MD_PLAIN, double>;
    case MD_BATCH: return (const void*)eri_md_kernel<l, MD_BATCH, double>;
    case MD_PER: return (const void*)eri_md_kernel<l, MD_PER, double>;
  }
#if HFX_MD_L % 2 == 0  // the diagonal (p|p) has an even total angular momentum
  if (kind == MD_DIAG) return (const void*)eri_md_kernel<l, MD_DIAG, double>;
#endif
  return nullptr;
}
}  // namespace hfx
