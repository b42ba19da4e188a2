// vd_resident_dir.cu -- instantiations of the resident eviction kernel
// (vd_resident.cuh) for one scoring rule.
#include "vd_resident.cuh"

namespace vd {

const void* resident_kernel_dir(bool decode, bool fused) {
  if (decode)
    return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<1, true, true>)
                 : reinterpret_cast<const void*>(&resident_evict_kernel<1, true, false>);
  return fused ? reinterpret_cast<const void*>(&resident_evict_kernel<1, false, true>)
               : reinterpret_cast<const void*>(&resident_evict_kernel<1, false, false>);
}

}  // namespace vd
