// vd_resident_l2.cu -- instantiations of the resident eviction kernel
// (vd_resident.cuh) for one scoring rule.
#include "vd_resident.cuh"

namespace vd {

const void* resident_kernel_l2(bool decode, bool holefill, bool fused) {
  const void* k[2][2][2] = {
      {{reinterpret_cast<const void*>(&resident_evict_kernel<0, false, false, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<0, false, false, true>)},
       {reinterpret_cast<const void*>(&resident_evict_kernel<0, false, true, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<0, false, true, true>)}},
      {{reinterpret_cast<const void*>(&resident_evict_kernel<0, true, false, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<0, true, false, true>)},
       {reinterpret_cast<const void*>(&resident_evict_kernel<0, true, true, false>),
        reinterpret_cast<const void*>(&resident_evict_kernel<0, true, true, true>)}}};
  return k[decode][holefill][fused];
}

}  // namespace vd
