// vd_resident_norm.cu -- instantiations of the resident eviction kernel
// (vd_resident.cuh) for one scoring rule.
#include "vd_resident.cuh"

namespace vd {

const void* resident_kernel_norm(bool decode, bool fused) {
  if (decode)
    return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<2, true, true>)
                 : reinterpret_cast<const void*>(&resident_evict_kernel<2, true, false>);
  return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<2, false, true>)
               : reinterpret_cast<const void*>(&resident_evict_kernel<2, false, false>);
}

}  // namespace vd
