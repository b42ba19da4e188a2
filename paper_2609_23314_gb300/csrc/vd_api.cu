// vd_api.cu -- host side of libvd.so: the C ABI declared in include/vd.h.
//
// Validates arguments before any launch, sizes the thread-block cluster per
// unit, launches the fused eviction kernel with cudaLaunchKernelExC on the
// caller's stream, and owns the device status word (a static __device__
// variable: the library allocates no device memory).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <mutex>

#include "vd.h"
#include "vd_evict.cuh"
#include "vd_resident.cuh"
#include "vd_small.cuh"

namespace vd {
const void* evict_kernel_l2(bool decode, bool holefill, bool fused, bool general);
const void* evict_kernel_dir(bool decode, bool holefill, bool fused);
const void* evict_kernel_norm(bool decode, bool holefill, bool fused, bool general);
const void* small_kernel_l2(bool decode, bool fused);
const void* small_kernel_dir(bool decode, bool fused);
const void* small_kernel_norm(bool decode, bool fused);
const void* resident_kernel_l2(bool decode, bool holefill, bool fused);
const void* resident_kernel_dir(bool decode, bool holefill, bool fused);
const void* resident_kernel_norm(bool decode, bool holefill, bool fused);
const void* score_kernel_l2(bool general);
const void* score_kernel_dir();
const void* score_kernel_norm(bool general);
}  // namespace vd

using vd::kThreads;

// First device-side anomaly since the last vd_get_device_status (0 = none).
static __device__ unsigned g_vd_status;

// ---------------------------------------------------------------------------
// small kernels: append (Eq. block_processing's concatenation), length
// update after an eviction, and the from-scratch running sum.  The append and
// the length updates are programmatic dependents of the kernel before them
// (launch_dependent) and wait for it before they read anything.
// ---------------------------------------------------------------------------
__global__ void vd_append_kernel(uint16_t* __restrict__ k, uint16_t* __restrict__ v,
                                 const uint16_t* __restrict__ kn, const uint16_t* __restrict__ vn,
                                 const int32_t* len, int units_per_seq,
                                 long long n_units, int cap, int d, int B, unsigned* status) {
  vd::grid_dependency_wait();
  vd::grid_launch_dependents();
  const int d8 = d >> 3;
  const long long total = n_units * (long long)B * d8;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(idx % d8);
    const long long ub = idx / d8;
    const int b = (int)(ub % B);
    const long long u = ub / B;
    // from L2: the previous kernel may set it while this one is resident
    const int n = __ldcg(len + u / units_per_seq);
    if (n < 0 || n > cap - B) {
      if (b == 0 && c == 0 && u % units_per_seq == 0) vd::record_status(status, vd::kStDeviceLen);
      continue;
    }
    const size_t src = (size_t)ub * d + (size_t)c * 8;
    const size_t dst = ((size_t)u * cap + (size_t)(n + b)) * d + (size_t)c * 8;
    vd::st16(k + dst, vd::ld_cg16(kn + src));
    vd::st16(v + dst, vd::ld_cg16(vn + src));
  }
}

__global__ void vd_len_add_kernel(int32_t* len, int n_seq, int cap, int B) {
  vd::grid_dependency_wait();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_seq) return;
  const int n = len[s];
  if (n >= 0 && n <= cap - B) len[s] = n + B;
}

// Mirrors the eviction kernel's per-sequence decision exactly.  added: the
// rows a fused append adds to len (0 when they were appended beforehand).
// Launched as a programmatic dependent of the eviction (which lets its
// dependents be scheduled at once): it is resident before the eviction ends
// and waits for it to complete before reading or writing len.
__global__ void vd_len_clamp_kernel(int32_t* len, const int32_t* N_dev, int N, int n_seq,
                                    int cap, int B, int running, int decode, int added) {
  vd::grid_dependency_wait();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_seq) return;
  const int n0 = len[s];
  const int n = n0 + added;
  const int Nb = N_dev ? N_dev[s] : N;
  if (vd::len_marked(n0)) {  // a unit was not evicted: the length stays
    len[s] = vd::mark_len(0) - n0;
    return;
  }
  if (n0 < 0 || n > cap || (running && B > n)) return;
  if (Nb < 1 || Nb > N) return;
  if (n <= Nb) {
    if (added) len[s] = n;
    return;
  }
  if (decode && n > Nb + 1) return;
  len[s] = Nb;
}

__global__ void __launch_bounds__(kThreads) vd_rsum_init_kernel(const uint16_t* __restrict__ v,
                                                                const int32_t* __restrict__ len,
                                                                double* rs, int units_per_seq,
                                                                int cap, int d, int lpr,
                                                                unsigned* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  vd::Smem& S = *reinterpret_cast<vd::Smem*>(smem_raw);
  const uint32_t ring = vd::smem_addr(smem_raw + vd::smem_layout(cap, 1, vd::kKindDecode).ring);
  const int u = blockIdx.x;
  const int n = len[u / units_per_seq];
  if (n < 0 || n > cap) {
    if (threadIdx.x == 0 && u % units_per_seq == 0) vd::record_status(status, vd::kStDeviceLen);
    return;
  }
  const uint16_t* vb = v + (size_t)u * cap * d;
  vd::sum_rows<vd::DecodeRing>(0, d >> 3, lpr, n, [&](int i) { return vb + (size_t)i * d; },
                               [](int) { return 1.f; }, S, ring);
  if ((int)threadIdx.x < d)
    rs[(size_t)u * d + threadIdx.x] = (double)S.acc_hi[threadIdx.x] + (double)S.acc_lo[threadIdx.x];
}

// ---------------------------------------------------------------------------
// per-device state
// ---------------------------------------------------------------------------
namespace {

// How calls of one shape are launched.  The occupancy queries behind it, up to
// two dozen, take 2.3 us of host time (a call 8.3 us through the Python binding,
// 6.1 with its plan at hand), as much as a small eviction's phases take on the
// device: so the answers are kept.
struct PlanKey {
  const void* kern;           // the streaming kernel; fits plans: the short-cache kernel
  long long units, want_solo;
  int d, capacity, kind, running, want_cluster, want_resident;
  bool operator==(const PlanKey& o) const {
    return kern == o.kern && units == o.units && want_solo == o.want_solo && d == o.d &&
           capacity == o.capacity && kind == o.kind && running == o.running &&
           want_cluster == o.want_cluster && want_resident == o.want_resident;
  }
};
struct Plan {
  int cluster;          // fits plans: 0 if the cluster does not fit
  bool resident, both;  // the resident kernel; with a buffer for each tensor
  size_t smem;
  long long solo;       // split launch: units run one CTA each (split_plan)
};
// 1024 shapes per device, in sets of 4 picked by the key's hash: a program that
// serves a few hundred batch sizes with a few kinds of calls finds them all again.
constexpr int kPlanSets = 256, kPlanWays = 4;
struct PlanSet {
  PlanKey key[kPlanWays];
  Plan plan[kPlanWays];
  int used, next;  // entries in use; the one replaced next
};

struct DeviceState {
  bool ready = false;
  unsigned* status = nullptr;
  int sms = 0;
  int smem_optin = 0;
  int smem_sm = 0, smem_reserved = 0;  // per SM; what each CTA takes of it besides its own
  PlanSet plans[kPlanSets];            // guarded by g_mu
};

constexpr int kMaxDevices = 64;
std::mutex g_mu;
DeviceState g_dev[kMaxDevices];

PlanSet& plan_set(DeviceState& st, const PlanKey& k) {
  unsigned long long h = reinterpret_cast<uintptr_t>(k.kern);
  for (const long long x : {k.units, k.want_solo, (long long)k.d, (long long)k.capacity,
                            (long long)k.kind, (long long)k.running, (long long)k.want_cluster,
                            (long long)k.want_resident})
    h = (h ^ (unsigned long long)x) * 0x9e3779b97f4a7c15ull, h ^= h >> 29;
  return st.plans[h % kPlanSets];
}

bool find_plan(DeviceState& st, const PlanKey& k, Plan* out) {
  std::lock_guard<std::mutex> lk(g_mu);
  const PlanSet& s = plan_set(st, k);
  for (int i = 0; i < s.used; ++i)
    if (s.key[i] == k) {
      *out = s.plan[i];
      return true;
    }
  return false;
}

void keep_plan(DeviceState& st, const PlanKey& k, const Plan& p) {
  std::lock_guard<std::mutex> lk(g_mu);
  PlanSet& s = plan_set(st, k);
  const int i = s.next;
  s.key[i] = k;
  s.plan[i] = p;
  s.next = (i + 1) % kPlanWays;
  if (s.used < kPlanWays) ++s.used;
}

// general: the score pass for any rule and head dim, else the batched one
// (vd::batched_scores)
const void* evict_kernel(vd_variant var, bool decode, bool holefill, bool fused, bool general) {
  switch (var) {
    case VD_SCORE_L2: return vd::evict_kernel_l2(decode, holefill, fused, general);
    case VD_SCORE_DIR: return vd::evict_kernel_dir(decode, holefill, fused);
    default: return vd::evict_kernel_norm(decode, holefill, fused, general);
  }
}

const void* score_kernel(vd_variant var, bool general) {
  switch (var) {
    case VD_SCORE_L2: return vd::score_kernel_l2(general);
    case VD_SCORE_DIR: return vd::score_kernel_dir();
    default: return vd::score_kernel_norm(general);
  }
}

const void* small_kernel(vd_variant var, bool decode, bool fused) {
  switch (var) {
    case VD_SCORE_L2: return vd::small_kernel_l2(decode, fused);
    case VD_SCORE_DIR: return vd::small_kernel_dir(decode, fused);
    default: return vd::small_kernel_norm(decode, fused);
  }
}

const void* resident_kernel(vd_variant var, bool decode, bool holefill, bool fused) {
  switch (var) {
    case VD_SCORE_L2: return vd::resident_kernel_l2(decode, holefill, fused);
    case VD_SCORE_DIR: return vd::resident_kernel_dir(decode, holefill, fused);
    default: return vd::resident_kernel_norm(decode, holefill, fused);
  }
}

vd_status device_state(DeviceState** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return VD_ERR_NO_DEVICE;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  DeviceState& st = g_dev[dev];
  if (!st.ready) {
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) {
      cudaGetLastError();
      return VD_ERR_NO_DEVICE;
    }
    if (p.major != 10 || p.minor != 3) return VD_ERR_NO_DEVICE;  // built for sm_103a only
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_vd_status) != cudaSuccess) return VD_ERR_CUDA;
    st.status = static_cast<unsigned*>(ptr);
    st.sms = p.multiProcessorCount;
    st.smem_optin = (int)p.sharedMemPerBlockOptin;
    st.smem_sm = (int)p.sharedMemPerMultiprocessor;
    st.smem_reserved = (int)p.reservedSharedMemPerBlock;
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(&vd_rsum_init_kernel),
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             st.smem_optin) != cudaSuccess)
      return VD_ERR_CUDA;
    for (int var = 0; var < 3; ++var)
      for (int kind = 0; kind < 16; ++kind) {
        const void* kern = evict_kernel((vd_variant)var, (kind & 1) != 0, (kind & 2) != 0,
                                        (kind & 4) != 0, (kind & 8) != 0);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 st.smem_optin) != cudaSuccess ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                cudaSuccess)
          return VD_ERR_CUDA;
      }
    for (int var = 0; var < 3; ++var)
      for (int kind = 0; kind < 14; ++kind) {
        const bool dec = (kind & 1) != 0, fus = (kind & 2) != 0;
        const void* kern = kind >= 12 ? score_kernel((vd_variant)var, kind == 13)
                           : kind < 4 ? small_kernel((vd_variant)var, dec, fus)
                                      : resident_kernel((vd_variant)var, dec, kind >= 8, fus);
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 st.smem_optin) != cudaSuccess ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                cudaSuccess)
          return VD_ERR_CUDA;
      }
    st.ready = true;
  }
  *out = &st;
  return VD_OK;
}

vd_status validate_cache(const vd_cache* c) {
  if (!c || !c->k || !c->v || !c->len) return VD_ERR_INVALID_ARG;
  if (c->n_seq < 1 || c->n_layer < 1 || c->n_kv_head < 1 || c->capacity < 1 || c->head_dim < 1)
    return VD_ERR_INVALID_ARG;
  if (c->head_dim % 8 != 0) return VD_ERR_ALIGNMENT;
  if (c->head_dim > 256) return VD_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(c->k) | reinterpret_cast<uintptr_t>(c->v)) & 15u)
    return VD_ERR_ALIGNMENT;
  const long long units = (long long)c->n_seq * c->n_layer * c->n_kv_head;
  if (units * 16 > INT_MAX) return VD_ERR_UNSUPPORTED;  // grid of units x cluster CTAs
  return VD_OK;
}

int lanes_per_row(int d) {
  int p = 1;
  while (p < d / 8) p <<= 1;
  return p;
}

// How many clusters of c CTAs (of kThreads threads) run at once.
long long active_clusters(const void* kern, long long groups, int c, size_t smem,
                          const DeviceState& st) {
  int n = 0;
  if (c == 1) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kThreads, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return (long long)n * st.sms;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(groups * c));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)c;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

bool cluster_fits(const void* kern, long long groups, int c, size_t smem,
                  const DeviceState& st) {
  return c == 1 || active_clusters(kern, groups, c, smem, st) > 0;
}

bool cluster_allowed(int c, int d) {
  const int total_chunks = 2 * (d / 8);
  return c == 1 || (total_chunks % c == 0 && total_chunks / c >= 4);
}

// CTAs per unit: C in {1, 2, 4, 8}, keeping row segments of at least 64 bytes
// of [K | V].  Waves = CTAs / resident slots at that C's shared-memory size.
//
// Up to about 2.6 CTAs per SM, more CTAs per unit shorten the launch (each
// reads less, and all of them still run side by side); beyond, the CTAs of an
// SM only share its bandwidth while every cluster barrier still costs.
// `side` is the largest C with units * C <= 2.6 SMs that leaves a CTA at least
// kMinRowsPerCta rows.  It is taken by ordered block eviction unless its
// slices exceed 1.25 MB (where the mean is recomputed, `resum`, the lines of the
// next paragraph), by hole-fill decode and by score-only launches without the
// bulk ring.  d = 128, us: ordered block, n = 1152, 96 units C = 4 39.0
// (C = 2 42, 8 58), 192 units C = 2 55 (1 61, 4 73), 240 units C = 1 66.6
// (2 69.5, 8 115); n = 2176, 288 units C = 1 131 (2 136); where the score pass
// is bound by instruction issue (`heavy`: Dir, or a head dim off the batched
// path), up to 0.95 of a wave instead (Dir, 288 units C = 2 161, C = 1 189;
// hole-fill decode, d = 192, n = 2001, 240 units C = 2 129, C = 1 150);
// hole-fill decode,
// n = 4097, 192 units C = 2 50.6 (8 76), 384 units C = 1 79 (2 103); scores,
// d = 96, n = 2048, 288 units C = 1 84 (2 90, 4 96).
//
// Ordered block eviction with more units, or larger slices: several waves,
// whose tail shrinks with the slice.  The smallest C with slices of at most
// 300 KB: 164 KB units C = 1 (800 units 102 us; C = 2 111, 4 158), 557 KB
// units C = 2 (800 units 344; C = 1 361), prefill_wide's 2.2 MB C = 8 (568 us;
// C = 4 586, C = 1 612).  With a recomputed mean C = 2 only up to 185 KB (288
// units of 2176 rows C = 4 146.4 us, C = 2 149, C = 1 154; 800 units of 1828
// rows C = 4 309, C = 2 321; d = 64, 2828 rows, 181 KB, C = 2 253, C = 4 264);
// it is bound by more instructions per row, so a short last wave costs more.
// Where that C makes 1 to 1.5 waves, the largest C within one wave is taken (192
// units of 2176 rows, recomputed, C = 2 107, C = 4 109; Dir, 288 units, C = 1 179,
// C = 2 198), for a batched score pass with a recomputed mean only if its slices
// stay within 300 KB (160 units of 4224 rows C = 4 176, C = 2 198); if not even
// C = 1 is within one wave, the next C (Dir, 480 units of 1152 rows C = 2 142, C
// = 1 152; 640 units, L2, C = 2 151, C = 1 161).  Ordered decode, which has no select to synchronise
// on: the largest C within 0.85 of a wave, or the smallest (up to 4) with
// slices of at most 200 KB where that is larger (n = 4097, 128 units C = 4
// 79.7 us, C = 2 86; 16384 units C = 4 7.28 ms, C = 1 7.37; n = 3001, 800
// units C = 4 282 us, C = 1 313).  Hole-fill decode and score-only with more
// units: C = 1 up to one wave, else the smallest C with two waves.
//
// The lines are fitted at d = 128 where no other head dim is named.  Elsewhere,
// ordered block, the rule's C and the others: d = 64, 288 units, n = 1152 C = 1
// 42.9 (C = 2 40.8, C = 4 59), n = 2176 C = 1 72.2 (C = 2 73.7, C = 4 81); d = 256,
// 192 units, n = 1152 C = 2 97 (C = 1 107, C = 4 117).
//
// Hole-fill block eviction (moves few rows, so the select's cluster
// synchronisation dominates and grows with C): the smallest C with at least
// 0.4 of a wave (one short wave beats a long tail and more cluster barriers:
// prefill_wide C=1, 0.74 waves, 0.211-0.216 ms vs C=2, 1.47 waves,
// 0.216-0.221; prefill_gqa8b C=1, 0.47 waves, 0.064 ms vs C=2, 0.95 waves,
// 0.069).  Score-only launches on the bulk-copy ring: the smallest C with at
// least half a wave (fewer, longer contiguous slices: the prefill_wide sigma
// pass at C=1, 0.74 waves, 0.115 ms vs C=2 0.131, C=4 0.139; 2 ring stages at
// 3 CTAs per SM; 3 stages 0.141 ms, 4 stages 0.149).  With none such (few
// units), the largest C that leaves every CTA at least kMinRowsPerCta rows of
// the capacity, else the smallest allowed C.  Where no C with 64-byte segments
// fits the shared memory (a large capacity at a small head dim), the smallest
// C that fits.  want (VD_CLUSTER_SIZE: 1, 2, 4, 8 or 16) overrides the choice,
// for tuning.
constexpr int kMinRowsPerCta = 128;

int choose_cluster(const void* kern, long long units, int d, int capacity, int kind,
                   bool holefill, bool heavy, bool resum, int want, const DeviceState& st,
                   size_t* smem_out) {
  int roomy = 0, smallest = 0, narrow = 0;  // see above
  int side = 0, sliced = 0, filled = 0, waved = 0;
  int single = 0, next = 0;      // largest C in one wave; first C above `sliced`
  double sliced_waves = 0;
  auto slice_of = [&](int c) { return (long long)((capacity + c - 1) / c) * d * 2; };
  auto most_of = [&](int c) {  // the largest slice for C = c, see above
    return kind == vd::kKindDecode ? 200LL << 10 : resum && !heavy && c == 2 ? 185LL << 10 : 300LL << 10;
  };
  for (int c = 1; c <= 16; c *= 2) {
    if (want >= 1 && c != want) continue;
    if ((d / 8 * 2) % c) continue;
    const size_t smem = vd::smem_layout(capacity, c, kind).total;
    if (smem > (size_t)st.smem_optin) continue;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (occ < 1 || !cluster_fits(kern, units, c, smem, st)) continue;
    if (want >= 1 || !cluster_allowed(c, d)) {
      // forced, or narrower row segments than preferred: only when nothing
      // else fits (a large capacity at a small head dim)
      if (narrow == 0) narrow = c;
      continue;
    }
    if (smallest == 0) smallest = c;
    if (c > 8) continue;  // 16-CTA clusters leave SMs of a GPC idle: never the fastest
    const long long rows = (capacity + c - 1) / c;
    const double waves = (double)(units * c) / ((double)st.sms * occ);
    const bool room = c == 1 || rows >= kMinRowsPerCta;
    if (room) roomy = c;
    if (room && (heavy ? waves <= 0.95 : (double)(units * c) <= 2.6 * st.sms)) side = c;
    if (room && waves <= 0.85) filled = c;
    if (waves <= 1.0) single = c;
    if (sliced != 0 && next == 0 && room) next = c;
    if (sliced == 0 && slice_of(c) <= most_of(c)) {
      sliced = c;
      sliced_waves = waves;
    }
    const bool enough = kind == vd::kKindBlock       ? waves >= 0.4
                        : kind == vd::kKindScoreBulk ? waves >= 0.5
                                                     : waves <= 1.0 || waves >= 2.0;
    if (waved == 0 && enough) waved = c;
  }
  const int large = roomy ? roomy : smallest;
  int chosen;
  if (want >= 1 || smallest == 0) {
    chosen = narrow ? narrow : 1;
  } else if (kind == vd::kKindScoreBulk || (kind == vd::kKindBlock && holefill)) {
    chosen = waved ? waved : large;
  } else if (kind == vd::kKindBlock) {
    const bool fits_side = side && slice_of(side) <= (resum ? most_of(side) : (5LL << 20) / 4);
    if (sliced_waves > 1.0 && sliced_waves < 1.5) {
      if (single && (!resum || heavy || slice_of(single) <= 300 << 10)) sliced = single;
      else if (!single && next) sliced = next;
    }
    chosen = fits_side ? side : sliced ? sliced : large;
  } else if (kind == vd::kKindDecode && !holefill) {
    chosen = std::max(filled, std::min(sliced ? sliced : large, 4));
  } else {
    chosen = side ? side : waved ? waved : large;
  }
  *smem_out = vd::smem_layout(capacity, chosen, kind).total;
  return chosen;
}

// Split launch, for launches that fit one wave of one CTA per unit and
// carry more units than the GPU has SMs.  The block scheduler hands CTAs out
// breadth-first, so with U = k P + L units on P SMs (0 < L < P), L SMs run
// k + 1 whole units and the rest k, and the launch lasts as long as the
// busiest SMs (prefill_wide in the hole-fill layout, 336 units on 152 SMs:
// the CTAs of the 32 SMs that held three finished 28 us after the median).
// Instead, a first launch runs the first k P units (rounded down to a
// multiple of c) one CTA each, and a second launch, a programmatic dependent
// of the first, runs each remaining unit on a cluster of c CTAs: its CTAs
// take the slots the first leaves free, so an SM carries at most
// k + ceil(L c / P) / c units.  c in {2, 4, 8, 16} is the one with the
// smallest such load whose CTAs still form one wave; the split is taken when
// it lowers the load by at least a quarter of a unit.  Used by hole-fill
// block eviction and the score-only launches (each reads its units once and
// moves few rows, so a unit's time is its share of the read bandwidth);
// VD_SPLIT_LAUNCH=0 turns it off.  Returns the number of units of the first
// launch (0: no split) and sets *c_out and *smem_out for the second.
long long split_plan(const void* kern, long long units, int d, int capacity, int kind,
                     const DeviceState& st, int* c_out, size_t* smem_out) {
  const long long P = st.sms;
  if (P < 1 || units <= P) return 0;
  const size_t smem1 = vd::smem_layout(capacity, 1, kind).total;
  if (smem1 > (size_t)st.smem_optin) return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (occ < 1 || units > P * occ) return 0;  // more than one wave: CTAs balance themselves
  const long long k = units / P;
  if (units % P == 0) return 0;
  double best = (double)(k + 1) - 0.25;
  long long best_solo = 0;
  for (int c = 2; c <= 16; c *= 2) {
    if (!cluster_allowed(c, d)) continue;
    const long long solo = (k * P) / c * c;
    const long long joint = units - solo;
    if (solo + joint * c > P * occ) continue;  // one wave
    const double load = (double)((solo + P - 1) / P) + (double)((joint * c + P - 1) / P) / c;
    const size_t smem_c = vd::smem_layout(capacity, c, kind).total;
    if (load < best && cluster_fits(kern, joint, c, smem_c, st)) {
      best = load;
      best_solo = solo;
      *c_out = c;
      *smem_out = smem_c;
    }
  }
  return best_solo;
}

// choose_cluster and split_plan.  A forced cluster size (VD_CLUSTER_SIZE) turns
// the automatic split off; VD_SOLO_UNITS with it forces a split whose first
// launch runs that many units (at most all but one) one CTA each, for tests
// (want_solo: that, else 0 when VD_SPLIT_LAUNCH turns the split off, else -1).
Plan streaming_plan(const PlanKey& k, bool holefill, bool heavy, bool resum,
                    const DeviceState& st) {
  Plan p{};
  p.cluster = choose_cluster(k.kern, k.units, k.d, k.capacity, k.kind, holefill, heavy, resum,
                             k.want_cluster, st, &p.smem);
  if (k.want_cluster >= 1 && k.want_solo > 0) {
    p.solo = std::min(k.want_solo, k.units - 1);
  } else if (k.want_cluster < 1 && k.want_solo != 0 &&
             ((k.kind == vd::kKindBlock && holefill) || k.kind == vd::kKindScore ||
              k.kind == vd::kKindScoreBulk)) {
    int c = p.cluster;
    size_t smem = p.smem;
    p.solo = split_plan(k.kern, k.units, k.d, k.capacity, k.kind, st, &c, &smem);
    if (p.solo > 0) {
      p.cluster = c;
      p.smem = smem;
    }
  }
  return p;
}

// The short-cache kernel (vd_small.cuh) takes a block or decode event when
// the unit's K and V rows fit in shared memory with room to spare
// (capacity * head_dim * 4 bytes <= kSmallRowBytes, capacity <=
// vd::kSmallMaxRows) and no sigma, hole-fill layout or forced cluster size
// (VD_CLUSTER_SIZE) is asked for.  It sets the lengths itself where a
// sequence's units fit in one cluster (<= 16) and the launch is at most one CTA
// per SM (60 units of 160 rows 9.5 us; 200 units 13.2, and 12.9 without).
// VD_SMALL_PATH=0 turns it off.  The choice depends on the shape only, so the
// fused and two-call forms, block and decode, take the same kernel.
constexpr size_t kSmallRowBytes = 64 * 1024;

bool use_small(const vd_cache* c, bool score_only, bool holefill, const float* disp_out,
               const DeviceState& st) {
  if (score_only || holefill || disp_out) return false;
  const char* off = std::getenv("VD_SMALL_PATH");
  if ((off && std::atoi(off) == 0) || std::getenv("VD_CLUSTER_SIZE")) return false;
  if (c->capacity > vd::kSmallMaxRows) return false;
  if ((size_t)c->capacity * c->head_dim * 4 > kSmallRowBytes) return false;
  return vd::small_layout(c->capacity, c->head_dim).total <= (size_t)st.smem_optin;
}

// cluster_fits, kept like the plans (of kind kFitsKind).
constexpr int kFitsKind = -1;
bool cached_fits(const void* kern, long long groups, int c, size_t smem, DeviceState& st) {
  const PlanKey k{kern, groups, (long long)smem, 0, 0, kFitsKind, 0, c, 0};
  Plan p{};
  if (!find_plan(st, k, &p)) {
    p.cluster = cluster_fits(kern, groups, c, smem, st) ? c : 0;
    keep_plan(st, k, p);
  }
  return p.cluster != 0;
}

// A plain kernel of kThreads-thread blocks as a programmatic dependent launch
// (it waits in griddepcontrol.wait before its first access to memory).
template <class... Params, class... Args>
vd_status launch_dependent(unsigned blocks, cudaStream_t s, void (*kern)(Params...),
                           Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...) != cudaSuccess) {
    cudaGetLastError();
    return VD_ERR_CUDA;
  }
  return VD_OK;
}

// groups clusters of c CTAs: the streaming and resident kernels' grids are units x
// c CTAs (a cluster per unit), the short-cache kernel's n_seq x units_per_seq (a
// cluster per sequence, a CTA per unit) or units x 1.
// A programmatic dependent launch: the kernel waits in griddepcontrol.wait.
vd_status launch(const void* kern, long long groups, int c, size_t smem, const void* params,
                 cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(groups * c));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  void* args[] = {const_cast<void*>(params)};
  if (cudaLaunchKernelExC(&cfg, kern, args) != cudaSuccess) {
    cudaGetLastError();
    return VD_ERR_CUDA;
  }
  return VD_OK;
}

// The resident kernel (vd_resident.cuh) takes an eviction whose
// clusters all run at once: it is bound by the latency of its phases, so it
// wins where the streaming kernel has too few rows per SM to hide its own, and
// loses once several waves of clusters follow one another (288 units of 2176
// rows, d = 128: 176 us against 130).  C is the largest size, up to 12, that
// leaves a CTA at least 64 rows and the launch at most two CTAs per SM (decode,
// which has fewer phases: three), and whose clusters form one wave.  us,
// streaming / resident, d = 128, n = 2176: 8 units 25.1 / 18.7 (C = 12; C = 8
// 21.7), 16 units 27.8 / 22.2 (C = 10; C = 8 23.8), 32 units 31.2 / 29.1 (C = 8; C
// = 4 30.5); n = 1152, 96 units 34.8 / 33.6 (C = 3; C = 4, 2.5 CTAs per SM, 48.8);
// d = 64, n = 2176, 32 units 24.4 / 20.6, 64 units 28.6 / 27.8.  Both tensors get a
// buffer where that keeps the wave (8 units 19.2, else 19.8).  More units, or
// larger ones: C = 1 where three CTAs share an SM (decode:
// two), in any number of waves, since a small unit is only its phases in either
// kernel: d = 64, 340 rows, 320 units 26.8 / 22.4, 4800
// units 208 / 182; d = 96, 240 rows, 1600 units 105 / 86 (340 rows, two CTAs per
// SM, 110 / 127); decode, d = 128, 301 rows, 640 units 42.9 / 33.7, 4800 units
// 197 / 172 (451 rows, one CTA per SM, 249 / 328).  A hole-fill block event moves
// so few rows that the streaming kernel catches up at 12 MB of scored rows: n =
// 2176, d = 128, 16 units (8.9 MB) 22.7 / 21.4, 24 units (13.4 MB) 23.8 / 25.2; d =
// 64, 40 units (11 MB) 21.8 / 21.4, 48 units (13 MB) 22.1 / 23.3; n = 1128, d =
// 256, 16 units (9.2 MB) 23.6 / 23.4, 24 units (14 MB) 24.8 / 28.3.  Otherwise the
// same lines: hole-fill block, d = 128, 2176 rows, 8 units 20.6 / 17.9, 230 rows, 320
// units 39.1 / 20.1; hole-fill decode, 4097 rows, 8 units 19.2 / 11.0, 201 rows,
// 4800 units 138 / 86.  VD_RESIDENT=0 turns the kernel off, VD_RESIDENT=c forces
// clusters of c CTAs (100 + c: with both buffers), for tests; a size that cannot
// run falls back to the streaming kernel.  Returns C, or 0.
constexpr int kResidentMinRows = 64;

int resident_plan(const void* kern, const PlanKey& k, bool decode, bool holefill,
                  const DeviceState& st, size_t* smem_out, bool* both_out) {
  const int want = k.want_resident, capacity = k.capacity;
  const long long units = k.units;
  if (want == 0 || capacity > vd::kMaxMarkedLen) return 0;
  auto smem_of = [&](int c, bool both) {
    return vd::resident_layout(capacity, k.d, c, decode, holefill, k.running != 0, both).total;
  };
  // whether `need` units run at once on clusters of c CTAs (asked only where
  // their shared memory alone lets them)
  auto at_once = [&](int c, bool both, long long need) {
    const size_t smem = smem_of(c, both);
    if (smem > (size_t)st.smem_optin) return false;
    const long long ctas = (long long)st.sms * (st.smem_sm / ((int)smem + st.smem_reserved));
    return ctas / c >= need && active_clusters(kern, units, c, smem, st) >= need;
  };
  int c = 0;
  bool both = false;
  if (want > 0) {
    c = want % 100;
    both = want >= 100 && !holefill;
    if (c < 1 || c > vd::kResMaxCluster || !at_once(c, both, 1)) c = 0;
  } else {
    const long long room = (decode ? 3LL : 2LL) * st.sms;
    if (units <= room) {
      const long long most = std::min<long long>(room / units, capacity / kResidentMinRows);
      for (c = (int)std::max(1LL, std::min(12LL, most)); c >= 1; --c)
        if (at_once(c, false, units)) break;
      both = !holefill && c >= 1 && at_once(c, true, units);
    }
    if (holefill && !decode && c > 1 && units * capacity * k.d * 2 > 12LL << 20) c = 0;
    if (c < 1 && at_once(1, false, (decode ? 2LL : 3LL) * st.sms)) c = 1;
  }
  *smem_out = c >= 1 ? smem_of(c, both) : 0;
  *both_out = both;
  return c;
}

int env_int(const char* name, int unset) {
  const char* s = std::getenv(name);
  return s ? std::atoi(s) : unset;
}

// Polls after which a device wait gives up.  VD_WAIT_LIMIT=a or a:b lowers them,
// for tests (a for the scored rows' copies, b for the other tensor's; 0: at once).
void wait_limits(uint32_t* scored, uint32_t* other) {
  *scored = *other = vd::kWaitLimit;
  const char* s = std::getenv("VD_WAIT_LIMIT");
  if (!s) return;
  char* end = nullptr;
  *scored = (uint32_t)std::min<unsigned long>(std::strtoul(s, &end, 10), vd::kWaitLimit);
  if (*end == ':')
    *other = (uint32_t)std::min<unsigned long>(std::strtoul(end + 1, nullptr, 10), vd::kWaitLimit);
}

vd_status run(const vd_cache* c, int32_t N, const int32_t* N_dev, int32_t B, vd_variant var,
              vd_mu_mode mu, double* running_sum, int32_t* evicted_out, int32_t* kept_idx_out,
              float* scores_out, cudaStream_t s, bool decode, bool score_only,
              int32_t* pos = nullptr, const int32_t* pos_new = nullptr, int score_k = 0,
              const float* weights = nullptr, float* disp_out = nullptr,
              const void* k_new = nullptr, const void* v_new = nullptr) {
  vd_status r = validate_cache(c);
  if (r != VD_OK) return r;
  if (var != VD_SCORE_L2 && var != VD_SCORE_DIR && var != VD_SCORE_NORM) return VD_ERR_INVALID_ARG;
  if (mu != VD_MU_RECOMPUTE && mu != VD_MU_RUNNING) return VD_ERR_INVALID_ARG;
  if (!score_only) {
    if (N < 1 || N > c->capacity) return VD_ERR_INVALID_ARG;
    if (B < 0 || B > c->capacity) return VD_ERR_INVALID_ARG;
    if (mu == VD_MU_RUNNING && !running_sum) return VD_ERR_INVALID_ARG;
  } else if (!scores_out && !disp_out) {
    return VD_ERR_INVALID_ARG;
  }
  if (disp_out && (decode || var != VD_SCORE_L2)) return VD_ERR_INVALID_ARG;
  if (weights && (score_only || decode)) return VD_ERR_INVALID_ARG;
  const bool holefill = pos != nullptr || pos_new != nullptr;
  if (holefill && (!pos || !pos_new)) return VD_ERR_INVALID_ARG;
  const bool fused = k_new != nullptr || v_new != nullptr;
  if (fused) {
    if (!k_new || !v_new || B < 1 || score_only) return VD_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(k_new) | reinterpret_cast<uintptr_t>(v_new)) & 15u)
      return VD_ERR_ALIGNMENT;
  }
  DeviceState* st = nullptr;
  r = device_state(&st);
  if (r != VD_OK) return r;

  // score-only launches have their own instantiation (no per-token buffers)
  const bool general = !vd::batched_scores((int)var, c->head_dim);
  const int kind = score_only ? (general ? vd::kKindScore : vd::kKindScoreBulk)
                 : decode     ? vd::kKindDecode
                              : vd::kKindBlock;
  if (kind == vd::kKindBlock && c->capacity > 65536) return VD_ERR_UNSUPPORTED;  // 16-bit lists
  if (vd::smem_layout(c->capacity, 16, kind).total > (size_t)st->smem_optin)
    return VD_ERR_UNSUPPORTED;
  const void* kern = score_only ? score_kernel(var, general)
                                : evict_kernel(var, decode, holefill, fused, general);
  const void* rk = score_only ? nullptr : resident_kernel(var, decode, holefill, fused);
  const long long units = (long long)c->n_seq * c->n_layer * c->n_kv_head;

  vd::EvictArgs a;
  a.k = static_cast<uint16_t*>(c->k);
  a.v = static_cast<uint16_t*>(c->v);
  a.len = c->len;
  a.N_dev = score_only ? nullptr : N_dev;
  a.running_sum = running_sum;
  a.kept_out = score_only ? nullptr : kept_idx_out;
  a.evicted_out = decode ? evicted_out : nullptr;
  a.scores_out = scores_out;
  a.status = st->status;
  a.units_per_seq = c->n_layer * c->n_kv_head;
  a.d = c->head_dim;
  a.lpr = lanes_per_row(c->head_dim);
  a.capacity = c->capacity;
  a.N = score_only ? 1 : N;
  a.B = decode ? 1 : B;
  a.mu_running = mu == VD_MU_RUNNING ? 1 : 0;
  a.score_only = score_only ? 1 : 0;
  a.pos = pos;
  a.pos_new = pos_new;
  a.holefill = holefill ? 1 : 0;
  a.score_k = score_k ? 1 : 0;
  a.weights = weights;
  a.disp_out = disp_out;
  a.k_new = static_cast<const uint16_t*>(k_new);
  a.v_new = static_cast<const uint16_t*>(v_new);
  a.unit_base = 0;
  a.wait_first = 1;
  a.let_next = score_only ? 0 : 1;
  wait_limits(&a.wait_limit, &a.wait_limit_other);
  // the eviction's length update
  auto clamp_lengths = [&]() {
    return launch_dependent((unsigned)((c->n_seq + kThreads - 1) / kThreads), s,
                            vd_len_clamp_kernel, c->len, N_dev, N, c->n_seq, c->capacity, (int)a.B,
                            (int)a.mu_running, decode ? 1 : 0, fused ? (int)a.B : 0);
  };
  if (use_small(c, score_only, holefill, disp_out, *st)) {
    const void* sk = small_kernel(var, decode, fused);
    const size_t ssmem = vd::small_layout(c->capacity, c->head_dim).total;
    // few units: n_seq clusters of units_per_seq CTAs (one CTA per unit), which
    // also set the sequences' lengths: one launch
    a.cluster = a.units_per_seq;
    if (a.cluster <= 16 && units <= st->sms && cached_fits(sk, c->n_seq, a.cluster, ssmem, *st)) {
      const vd::SmallArgs sa{a, (int32_t)units, 1};
      return launch(sk, c->n_seq, a.cluster, ssmem, &sa, s);
    }
    a.cluster = 1;
    const vd::SmallArgs sa{a, (int32_t)units, 0};
    r = launch(sk, units, 1, ssmem, &sa, s);
    return r != VD_OK ? r : clamp_lengths();
  }
  const bool cluster_env = std::getenv("VD_CLUSTER_SIZE") != nullptr;
  const int want_cluster = env_int("VD_CLUSTER_SIZE", 0);
  long long want_solo = -1;  // see streaming_plan
  if (want_cluster >= 1)
    want_solo = env_int("VD_SOLO_UNITS", -1);
  else if (env_int("VD_SPLIT_LAUNCH", 1) == 0)
    want_solo = 0;
  // a forced cluster size is one of the streaming kernel's
  const int want_resident = score_only || cluster_env ? 0 : env_int("VD_RESIDENT", -1);
  const PlanKey key{kern, units, want_solo, c->head_dim, c->capacity, kind,
                    mu == VD_MU_RUNNING ? 1 : 0, want_cluster, want_resident};
  Plan plan{};
  if (!find_plan(*st, key, &plan)) {
    size_t rsmem = 0;
    bool both = false;
    const int rc = resident_plan(rk, key, decode, holefill, *st, &rsmem, &both);
    plan = rc > 0 ? Plan{rc, true, both, rsmem, 0}
                  : streaming_plan(key, holefill, general,
                                   mu == VD_MU_RECOMPUTE && var != VD_SCORE_NORM, *st);
    keep_plan(*st, key, plan);
  }
  a.cluster = plan.cluster;
  const size_t smem = plan.smem;
  if (plan.resident) {
    const vd::ResidentArgs ra{a, plan.both ? 1 : 0};
    r = launch(rk, units, a.cluster, smem, &ra, s);
    return r != VD_OK ? r : clamp_lengths();
  }
  const long long solo = plan.solo;
  if (smem > (size_t)st->smem_optin) return VD_ERR_UNSUPPORTED;

  if (solo > 0) {
    // split launch: units [0, solo) one CTA each, then the rest on clusters,
    // as a programmatic dependent of the first part
    vd::EvictArgs a1 = a;
    a1.cluster = 1;
    a1.let_next = 1;
    const size_t smem1 = vd::smem_layout(c->capacity, 1, kind).total;
    if (smem1 > (size_t)st->smem_optin) return VD_ERR_UNSUPPORTED;
    r = launch(kern, solo, 1, smem1, &a1, s);
    if (r != VD_OK) return r;
    // the second part's per-unit pointers start at unit `solo`
    const size_t rows = (size_t)solo * c->capacity, dd = (size_t)c->head_dim;
    a.unit_base = (int32_t)solo;
    a.wait_first = 0;  // it runs beside the first part
    a.k += rows * dd;
    a.v += rows * dd;
    if (a.running_sum) a.running_sum += (size_t)solo * dd;
    if (a.kept_out) a.kept_out += (size_t)solo * a.N;
    if (a.evicted_out) a.evicted_out += solo;
    if (a.scores_out) a.scores_out += rows;
    if (a.pos) a.pos += rows;
    if (a.weights) a.weights += rows;
    if (a.disp_out) a.disp_out += solo;
    if (a.k_new) a.k_new += (size_t)solo * a.B * dd;
    if (a.v_new) a.v_new += (size_t)solo * a.B * dd;
    r = launch(kern, units - solo, a.cluster, smem, &a, s);
  } else {
    r = launch(kern, units, a.cluster, smem, &a, s);
  }
  return r != VD_OK || score_only ? r : clamp_lengths();
}

}  // namespace

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" {

vd_status vd_score(const vd_cache* c, vd_variant var, float* scores_out, vd_stream_t stream) {
  return run(c, 1, nullptr, 0, var, VD_MU_RECOMPUTE, nullptr, nullptr, nullptr, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, true);
}

vd_status vd_append_evict_block(const vd_cache* c, const void* k_new, const void* v_new,
                                int32_t B, int32_t N, const int32_t* N_dev, vd_variant var,
                                vd_mu_mode mu, double* running_sum, int32_t* pos,
                                const int32_t* pos_first_new, int32_t* kept_idx_out,
                                float* scores_out, vd_stream_t stream) {
  return run(c, N, N_dev, B, var, mu, running_sum, nullptr, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, false, pos, pos_first_new, 0,
             nullptr, nullptr, k_new, v_new);
}

vd_status vd_append_evict_decode(const vd_cache* c, const void* k_new, const void* v_new,
                                 int32_t N, const int32_t* N_dev, vd_variant var, vd_mu_mode mu,
                                 double* running_sum, int32_t* pos, const int32_t* pos_first_new,
                                 int32_t* evicted_out, int32_t* kept_idx_out, float* scores_out,
                                 vd_stream_t stream) {
  return run(c, N, N_dev, 1, var, mu, running_sum, evicted_out, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), true, false, pos, pos_first_new, 0, nullptr,
             nullptr, k_new, v_new);
}

vd_status vd_evict_block(const vd_cache* c, int32_t N, const int32_t* N_dev, int32_t B,
                         vd_variant var, vd_mu_mode mu, double* running_sum,
                         int32_t* kept_idx_out, float* scores_out, vd_stream_t stream) {
  return run(c, N, N_dev, B, var, mu, running_sum, nullptr, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, false);
}

vd_status vd_evict_decode(const vd_cache* c, int32_t N, const int32_t* N_dev, vd_variant var,
                          vd_mu_mode mu, double* running_sum, int32_t* evicted_out,
                          int32_t* kept_idx_out, float* scores_out, vd_stream_t stream) {
  return run(c, N, N_dev, 1, var, mu, running_sum, evicted_out, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), true, false);
}

vd_status vd_score_ex(const vd_cache* c, vd_variant var, vd_mu_mode mu,
                      const double* running_sum, int32_t score_keys, float* scores_out,
                      float* dispersion_out, vd_stream_t stream) {
  if (mu == VD_MU_RUNNING && !running_sum) return VD_ERR_INVALID_ARG;
  // the score-only kernel reads the running sum and never writes it
  return run(c, 1, nullptr, 0, var, mu, const_cast<double*>(running_sum), nullptr, nullptr,
             scores_out, reinterpret_cast<cudaStream_t>(stream), false, true, nullptr, nullptr,
             score_keys, nullptr, dispersion_out);
}

vd_status vd_evict_block_ex(const vd_cache* c, int32_t N, const int32_t* N_dev, int32_t B,
                            vd_variant var, vd_mu_mode mu, double* running_sum,
                            int32_t score_keys, const float* attn, int32_t* kept_idx_out,
                            float* scores_out, float* dispersion_out, vd_stream_t stream) {
  return run(c, N, N_dev, B, var, mu, running_sum, nullptr, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, false, nullptr, nullptr, score_keys,
             attn, dispersion_out);
}

vd_status vd_append_evict_block_ex(const vd_cache* c, const void* k_new, const void* v_new,
                                   int32_t B, int32_t N, const int32_t* N_dev, vd_variant var,
                                   vd_mu_mode mu, double* running_sum, int32_t score_keys,
                                   const float* attn, int32_t* kept_idx_out, float* scores_out,
                                   float* dispersion_out, vd_stream_t stream) {
  return run(c, N, N_dev, B, var, mu, running_sum, nullptr, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, false, nullptr, nullptr, score_keys,
             attn, dispersion_out, k_new, v_new);
}

vd_status vd_evict_block_holefill(const vd_cache* c, int32_t N, const int32_t* N_dev, int32_t B,
                                  vd_variant var, vd_mu_mode mu, double* running_sum,
                                  int32_t* pos, const int32_t* pos_first_new,
                                  int32_t* kept_idx_out, float* scores_out, vd_stream_t stream) {
  if (!pos || !pos_first_new) return VD_ERR_INVALID_ARG;
  return run(c, N, N_dev, B, var, mu, running_sum, nullptr, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), false, false, pos, pos_first_new);
}

vd_status vd_evict_decode_holefill(const vd_cache* c, int32_t N, const int32_t* N_dev,
                                   vd_variant var, vd_mu_mode mu, double* running_sum,
                                   int32_t* pos, const int32_t* pos_first_new,
                                   int32_t* evicted_out, int32_t* kept_idx_out, float* scores_out,
                                   vd_stream_t stream) {
  if (!pos || !pos_first_new) return VD_ERR_INVALID_ARG;
  return run(c, N, N_dev, 1, var, mu, running_sum, evicted_out, kept_idx_out, scores_out,
             reinterpret_cast<cudaStream_t>(stream), true, false, pos, pos_first_new);
}

vd_status vd_append(const vd_cache* c, const void* k_new, const void* v_new, int32_t B,
                    vd_stream_t stream) {
  vd_status r = validate_cache(c);
  if (r != VD_OK) return r;
  if (!k_new || !v_new || B < 0 || B > c->capacity) return VD_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(k_new) | reinterpret_cast<uintptr_t>(v_new)) & 15u)
    return VD_ERR_ALIGNMENT;
  if (B == 0) return VD_OK;
  DeviceState* st = nullptr;
  r = device_state(&st);
  if (r != VD_OK) return r;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const long long units = (long long)c->n_seq * c->n_layer * c->n_kv_head;
  const long long work = units * B * (c->head_dim / 8);
  const long long want = (work + 255) / 256;
  const int blocks = (int)(want < (long long)st->sms * 32 ? want : (long long)st->sms * 32);
  r = launch_dependent((unsigned)blocks, s, vd_append_kernel, static_cast<uint16_t*>(c->k),
                       static_cast<uint16_t*>(c->v), static_cast<const uint16_t*>(k_new),
                       static_cast<const uint16_t*>(v_new), c->len, c->n_layer * c->n_kv_head,
                       units, c->capacity, c->head_dim, B, st->status);
  if (r != VD_OK) return r;
  return launch_dependent((unsigned)((c->n_seq + kThreads - 1) / kThreads), s, vd_len_add_kernel,
                          c->len, c->n_seq, c->capacity, B);
}

vd_status vd_running_sum_init(const vd_cache* c, double* running_sum, vd_stream_t stream) {
  return vd_running_sum_init_ex(c, 0, running_sum, stream);
}

vd_status vd_running_sum_init_ex(const vd_cache* c, int32_t of_keys, double* running_sum,
                                 vd_stream_t stream) {
  vd_status r = validate_cache(c);
  if (r != VD_OK) return r;
  if (!running_sum) return VD_ERR_INVALID_ARG;
  DeviceState* st = nullptr;
  r = device_state(&st);
  if (r != VD_OK) return r;
  const long long units = (long long)c->n_seq * c->n_layer * c->n_kv_head;
  const size_t smem = vd::smem_layout(c->capacity, 1, vd::kKindDecode).total;
  vd_rsum_init_kernel<<<(unsigned)units, kThreads, smem, reinterpret_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint16_t*>(of_keys ? c->k : c->v), c->len, running_sum,
      c->n_layer * c->n_kv_head,
      c->capacity, c->head_dim, lanes_per_row(c->head_dim), st->status);
  if (cudaGetLastError() != cudaSuccess) return VD_ERR_CUDA;
  return VD_OK;
}

size_t vd_workspace_size(const vd_cache* c) {
  (void)c;
  return 0;
}

const char* vd_status_string(vd_status st) {
  switch (st) {
    case VD_OK: return "ok";
    case VD_ERR_INVALID_ARG: return "invalid argument";
    case VD_ERR_ALIGNMENT: return "misaligned pointer or head_dim not a multiple of 8";
    case VD_ERR_UNSUPPORTED: return "unsupported shape";
    case VD_ERR_NONFINITE: return "non-finite score on the device";
    case VD_ERR_TIMEOUT: return "device wait timed out";
    case VD_ERR_CUDA: return "CUDA runtime error";
    case VD_ERR_DEVICE_LEN: return "device: sequence length out of range";
    case VD_ERR_DEVICE_BUDGET: return "device: budget out of range or decode over budget";
    case VD_ERR_NO_DEVICE: return "no sm_103 CUDA device";
    case VD_ERR_INTERNAL: return "device: inconsistent slot list (internal self-check)";
    default: return "unknown status";
  }
}

vd_status vd_get_device_status(vd_stream_t stream) {
  DeviceState* st = nullptr;
  vd_status r = device_state(&st);
  if (r != VD_OK) return r;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return VD_ERR_CUDA;
  }
  unsigned w = 0;
  const unsigned z = 0;
  if (cudaMemcpyFromSymbolAsync(&w, g_vd_status, sizeof w, 0, cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaMemcpyToSymbolAsync(g_vd_status, &z, sizeof z, 0, cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    cudaGetLastError();
    return VD_ERR_CUDA;
  }
  return static_cast<vd_status>(w);
}

}  // extern "C"
