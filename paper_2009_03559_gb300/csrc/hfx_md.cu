// Instances of the Hermite engine for one total angular momentum (HFX_MD_L, compiled once for
// each so that the instances build in parallel).
#include <algorithm>
#include "hfx_md.cuh"

#define HFX_CAT2(a, b) a##b
#define HFX_CAT(a, b) HFX_CAT2(a, b)

namespace hfx {
const void* HFX_CAT(md_kernel_l, HFX_MD_L)(int kind) {
  switch (kind) {
    case MD_PLAIN: return (const void*)eri_md_kernel<HFX_MD_L, MD_PLAIN>;
    case MD_BATCH: return (const void*)eri_md_kernel<HFX_MD_L, MD_BATCH>;
    case MD_PER: return (const void*)eri_md_kernel<HFX_MD_L, MD_PER>;
    // the diagonal (p|p) has an even total angular momentum
    case MD_DIAG: return HFX_MD_L % 2 ? nullptr : (const void*)eri_md_kernel<HFX_MD_L - HFX_MD_L % 2, MD_DIAG>;
  }
  return nullptr;
}
}  // namespace hfx
