// vd_resident_dir.cu -- instantiations of the resident eviction kernel
// (vd_resident.cuh) for one scoring rule.
#include "vd_resident.cuh"

namespace vd {

const void* resident_kernel_dir(bool decode, bool holefill, bool fused) {
  const void* k[2][2][2] = {
      {{reinterpret_cast<const void*>(&resident_evict_kernel<1, false, false, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<1, false, false, true>)},
       {reinterpret_cast<const void*>(&resident_evict_kernel<1, false, true, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<1, false, true, true>)}},
      {{reinterpret_cast<const void*>(&resident_evict_kernel<1, true, false, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<1, true, false, true>)},
       {reinterpret_cast<const void*>(&resident_evict_kernel<1, true, true, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<1, true, true, true>)}}};
  return k[decode][holefill][fused];
}

}  // namespace vd
