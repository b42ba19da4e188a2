// vd_evict_l2.cu -- instantiates the fused eviction kernel and the short-cache
// kernel for one scoring rule (compiled separately so the translation units
// build in parallel).
#include "vd_evict.cuh"
#include "vd_small.cuh"

namespace vd {
namespace {
template <bool GEN>
const void* pick(bool decode, bool holefill, bool fused) {
  const void* k[2][2][2] = {
      {{reinterpret_cast<const void*>(&evict_kernel<0, false, false, false, GEN>),
        reinterpret_cast<const void*>(&evict_kernel<0, false, false, true, GEN>)},
       {reinterpret_cast<const void*>(&evict_kernel<0, false, true, false, GEN>),
        reinterpret_cast<const void*>(&evict_kernel<0, false, true, true, GEN>)}},
      {{reinterpret_cast<const void*>(&evict_kernel<0, true, false, false, GEN>),
        reinterpret_cast<const void*>(&evict_kernel<0, true, false, true, GEN>)},
       {reinterpret_cast<const void*>(&evict_kernel<0, true, true, false, GEN>),
        reinterpret_cast<const void*>(&evict_kernel<0, true, true, true, GEN>)}}};
  return k[decode][holefill][fused];
}
}  // namespace

// general: the score pass for any head dim (else d is 64, 128 or 256)
const void* evict_kernel_l2(bool decode, bool holefill, bool fused, bool general) {
  return general ? pick<true>(decode, holefill, fused) : pick<false>(decode, holefill, fused);
}

const void* small_kernel_l2(bool decode, bool fused) {
  const void* k[2][2] = {
      {reinterpret_cast<const void*>(&small_evict_kernel<0, false, false>),
       reinterpret_cast<const void*>(&small_evict_kernel<0, false, true>)},
      {reinterpret_cast<const void*>(&small_evict_kernel<0, true, false>),
       reinterpret_cast<const void*>(&small_evict_kernel<0, true, true>)}};
  return k[decode][fused];
}

const void* score_kernel_l2(bool general) {
  return general ? reinterpret_cast<const void*>(&evict_kernel<0, true, false, false, true, true>)
                 : reinterpret_cast<const void*>(&evict_kernel<0, true, false, false, false, true>);
}
}  // namespace vd
