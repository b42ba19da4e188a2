// vd_resident_l2.cu -- instantiations of the resident eviction kernel
// (vd_resident.cuh) for one scoring rule.
#include "vd_resident.cuh"

namespace vd {

const void* resident_kernel_l2(bool decode, bool fused) {
  if (decode)
    return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<0, true, true>)
                 : reinterpret_cast<const void*>(&resident_evict_kernel<0, true, false>);
  return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<0, false, true>)
               : reinterpret_cast<const void*>(&resident_evict_kernel<0, false, false>);
}

}  // namespace vd
