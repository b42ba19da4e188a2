// vd_resident.cuh -- pi_N of Sec. 2.1 Eq. (eviction) with the scored rows of a
// unit kept in the shared memory of its thread-block cluster.
//
// For launches of few or small units, where the streaming kernel (vd_evict.cuh)
// waits for its own phases: a cluster of C CTAs (any C up to 16) loads a unit's
// scored rows once.  CTA r holds the rows [r * R, (r + 1) * R) and the mean,
// the scores, the retired part of the running sum and the compacted rows all
// come from that copy (the streaming kernel reads the scored tensor twice,
// three times with a recomputed mean).
//
//   1. load    the scored tensor's slice, in up to four bulk copies
//   2. mean    running mean: S plus the appended rows, which every CTA sums by
//              itself (no exchange) up to 64 KB of them; recomputed: column
//              sums of the slice, exchanged through distributed shared memory
//   3. score   chunk by chunk as the copies land, with the operations of the
//              streaming kernel in its order: the same bits for the same mean
//              (whose sums are added in another order; its remainder may differ)
//   4. select  every CTA gets every key (16-byte remote stores) and finds the
//              threshold by itself: one histogram of 1024 buckets over the
//              range the keys span, then a rank among the threshold's bucket
//              (repeated on that bucket while it holds more than 256 keys).
//              No cluster barrier after the keys'.  Decode exchanges one minimum.
//   5. sum     running mean: minus the evicted rows, added over the cluster
//   6. move    kept rows go from shared memory to their slots: every source
//              was loaded before the barrier of step 4, so the in-place
//              gather has no order to respect.  The other tensor's slice is
//              then loaded into the same buffer (it was brought to L2 during
//              steps 2 to 4), or was loaded with the first one where both
//              fit, and written after one more barrier.  Hole-fill layout:
//              only the movers are copied, from global memory into the holes.
//
// What bounds it: the latency of these steps, each of which runs once; ncu
// counts half of the warps' stalls as instruction fetch (no loop repeats often
// enough to stay cached).  us per fused call, calls back to back, streaming /
// this kernel: 8 units of 2176 rows, d = 128 (C = 12) 25.1 / 18.7 (19.5 with
// inputs that rotate), recomputed mean 26.0 / 17.4, Dir 29.1 / 20.8, d = 96 30.8 /
// 19.2; decode, 8 units of 4097 rows 22.8 / 13.4.  8 warps per CTA beat 16 (17.9
// us in the kernel against 19.6), and rolling the loops up lost 0.8 us: the loads
// that an unrolled loop keeps in flight count for more.  The barriers that
// only order execution are relaxed arrivals: the release form waited 2 to 5 us
// for the bulk copies in flight.
#pragma once

#include <climits>
#include <cstdint>

#include "vd_evict.cuh"

namespace vd {

constexpr int kResBuckets = 1024;
constexpr int kResMaxCluster = 16;
constexpr int kResChunks = 4;    // bulk copies (and barriers) of the scored slice
constexpr int kResSumRanks = 4;  // CTAs that share the sum of the appended rows

struct ResidentArgs {
  EvictArgs e;
  int32_t both;  // 1: the other tensor's slice has a buffer of its own
};

struct ResSmem {
  float mu[256];     // the mean rounded to fp32 ...
  float mulo[256];   // ... and its remainder, both in column order
  float acc_hi[256];  // this CTA's partial column sums (read by peer CTAs)
  float acc_lo[256];
  // the select's histogram lies over the four arrays above (hist_of): they
  // are dead between the scores and the retired rows' sum
  double snew[256];  // running mode: the running sum plus the appended rows
  unsigned long long bar[kResChunks + 1];  // scored tensor's chunks, other tensor
  // decode: every CTA's minimum (pushed by it); the last entry: kLostBest where a
  // wait in the cluster gave up
  unsigned long long best[kResMaxCluster + 1];
  int best_slot[kResMaxCluster];            // hole-fill decode: its slot (pushed)
  int wslot[kWarps];
  uint32_t kmin[kResMaxCluster];  // every CTA's smallest and largest key (pushed)
  uint32_t kmax[kResMaxCluster + 1];  // (the last entry: kLostKey, as for best)
  unsigned long long wbest[kWarps];
  uint32_t wmin[kWarps], wmax[kWarps];
  int scan[kWarps], pre[kWarps];
  uint32_t cand[kThreads];
  uint32_t sel_lo;
  int sel_above, sel_cnt, ncand;
  float dsc[4 * kWarps];
  float disp[4];  // dispersion partials (read by rank 0)
  float fsh[kWarps];
  float inv_mnorm;
  int mu_zero;
  int lost;  // a wait for this CTA's scored rows gave up
};
// Values that no minimum and no key has: they win the exchange's min and max, so
// that the outcome needs no load of its own.
constexpr unsigned long long kLostBest = 0ull;
constexpr uint32_t kLostKey = 0xffffffffu;
static_assert(kResBuckets * 4 == 4 * 256 * 4, "the histogram covers mu .. acc_lo");

__host__ __device__ inline int resident_rows(int n, int c) {
  return ((n + c - 1) / c + 3) & ~3;  // a multiple of 4: 16-byte stores of keys
}

struct ResLayout {
  size_t keys, list, pairs, buf, obuf, total;
};

// The keys' region also holds resident_sum's partials, before the keys are
// written.  Decode keeps no keys, and sums rows
// only where the mean is recomputed.
__host__ __device__ inline ResLayout resident_layout(int capacity, int d, int cluster, bool decode,
                                                     bool holefill, bool running, bool both) {
  const size_t rcap = (size_t)resident_rows(capacity, cluster);
  const size_t keys = decode ? 0 : rcap * (size_t)cluster * 4;
  const size_t scratch = decode && running ? 0 : (size_t)d * kWarps * 8;
  ResLayout l;
  l.keys = (sizeof(ResSmem) + 127) & ~(size_t)127;
  l.list = l.keys + (keys > scratch ? keys : scratch);
  l.pairs = (l.list + (decode ? 0 : rcap * 2) + 3) & ~(size_t)3;
  // hole-fill: at most half of the rows are holes, and as many movers
  l.buf = (l.pairs + (decode || !holefill ? 0 : (size_t)capacity * 2 + 4) + 127) & ~(size_t)127;
  const size_t bytes = (rcap * (size_t)d * 2 + 127) & ~(size_t)127;
  l.obuf = both ? l.buf + bytes : l.buf;
  l.total = l.obuf + bytes;
  return l;
}

__device__ __forceinline__ void st_cluster16(uint32_t addr, const uint4& v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

// Brings a contiguous block into L2 (both a multiple of 16 bytes).
__device__ __forceinline__ void bulk_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ void st_cluster_u64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// Sum over the items [0, count) of sign(i) * row i, double-float per element
// (TwoSum), added in a fixed order: within a thread, over a warp's groups, then
// over the warps (through `scratch`, 2 * kWarps * d floats).  ld(i, ci) loads
// 16-byte chunk ci of item i, U items at a time.  Thread t < d returns column
// t.  One block barrier, after which `scratch` is still being read.
template <int U, class Ld, class SignOf>
__device__ __forceinline__ ff resident_sum(int d, int lpr, int count, Ld ld, SignOf sign_of,
                                           float* scratch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ci = lane & (lpr - 1), g = tid / lpr, ng = kThreads / lpr;
  const bool active = ci < (d >> 3);
  unsigned long long hi2[4], lo2[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) hi2[k] = lo2[k] = 0ull;
  if (active)
    for (int i0 = g; i0 < count; i0 += U * ng) {
      uint4 q[U];
#pragma unroll
      for (int m = 0; m < U; ++m)
        if (i0 + m * ng < count) q[m] = ld(i0 + m * ng, ci);
#pragma unroll
      for (int m = 0; m < U; ++m) {
        if (i0 + m * ng >= count) break;
        const uint32_t flip = sign_of(i0 + m * ng) < 0.f ? 0x80008000u : 0u;
        const uint32_t w[4] = {q[m].x ^ flip, q[m].y ^ flip, q[m].z ^ flip, q[m].w ^ flip};
#pragma unroll
        for (int k = 0; k < 4; ++k) ff2_accumulate(hi2[k], lo2[k], bf16x2_to_f2(w[k]));
      }
    }
  ff p[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float h0, h1, l0, l1;
    f2_unpack(hi2[k], h0, h1);
    f2_unpack(lo2[k], l0, l1);
    p[2 * k] = ff_add(ff{h0, 0.f}, ff{0.f, l0});
    p[2 * k + 1] = ff_add(ff{h1, 0.f}, ff{0.f, l1});
  }
  for (int off = lpr; off < 32; off <<= 1) {
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = ff_add(p[k], ff_shfl_xor(p[k], off));
  }
  if (lane < lpr && active) {
    float4* h = reinterpret_cast<float4*>(scratch + warp * d + ci * 8);
    float4* l = reinterpret_cast<float4*>(scratch + (kWarps + warp) * d + ci * 8);
    h[0] = make_float4(p[0].hi, p[1].hi, p[2].hi, p[3].hi);
    h[1] = make_float4(p[4].hi, p[5].hi, p[6].hi, p[7].hi);
    l[0] = make_float4(p[0].lo, p[1].lo, p[2].lo, p[3].lo);
    l[1] = make_float4(p[4].lo, p[5].lo, p[6].lo, p[7].lo);
  }
  __syncthreads();
  ff t{0.f, 0.f};
  if (tid < d) {
    ff v[kWarps];
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
      v[w] = ff{scratch[w * d + tid], scratch[(kWarps + w) * d + tid]};
#pragma unroll
    for (int h = 1; h < kWarps; h <<= 1) {
#pragma unroll
      for (int w = 0; w < kWarps; w += 2 * h) v[w] = ff_add(v[w], v[w + h]);
    }
    t = v[0];
  }
  return t;
}

// The sum, in rank order, of column c of the partial sums S.acc of the first
// `ranks` CTAs of the cluster.  Four ranks' remote loads are in flight at a time.
__device__ __forceinline__ ff resident_gather(int c, int ranks, const ResSmem& S) {
  const uint32_t ah = smem_addr(&S.acc_hi[c]), al = smem_addr(&S.acc_lo[c]);
  ff t{0.f, 0.f};
  for (int rr = 0; rr < ranks; rr += 4) {
    float h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned r = (unsigned)min(rr + k, ranks - 1);
      h[k] = ld_cluster_f32(mapa(ah, r));
      l[k] = ld_cluster_f32(mapa(al, r));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (rr + k < ranks) t = ff_add(t, ff{h[k], l[k]});
  }
  return t;
}

// Scores of the local rows [ca, cb) in shared memory, head dims 64, 128, 256
// (LPR lanes per row, one 16-byte chunk each), L2 and Norm.  Eight rows per
// group of lanes at a time: per element and per row the arithmetic of
// score_rows_fast, reduced over the lanes in its order.
template <int VAR, int LPR, class Finish>
__device__ __forceinline__ void resident_score_fast(uint32_t buf, int ca, int cb,
                                                    const float* mu, const float* mulo,
                                                    Finish finish) {
  constexpr int kBatch = 8, kG = kThreads / LPR, kRowBytes = LPR * 16, kSpread = LPR / kBatch;
  const int ci = (threadIdx.x & 31) & (LPR - 1), g = threadIdx.x / LPR;
  unsigned long long m2[4], l2[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    m2[k] = VAR == 0 ? f2_pack(mu[ci * 8 + 2 * k], mu[ci * 8 + 2 * k + 1]) : 0ull;
    l2[k] = VAR == 0 ? f2_pack(mulo[ci * 8 + 2 * k], mulo[ci * 8 + 2 * k + 1]) : 0ull;
  }
  for (int base = ca; base < cb; base += kBatch * kG) {
    float part[kBatch];
    uint4 q[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int j = base + g + k * kG;
      q[k] = make_uint4(0u, 0u, 0u, 0u);
      if (j < cb) q[k] = ld_shared16(buf + (uint32_t)(j * kRowBytes + ci * 16));
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const uint32_t w[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
      unsigned long long acc = 0ull;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned long long x = bf16x2_to_f2(w[e]);
        if (VAR == 0) {
          const unsigned long long dv = f2_sub(f2_sub(x, m2[e]), l2[e]);
          acc = f2_fma(dv, dv, acc);
        } else {
          acc = f2_fma(x, x, acc);
        }
      }
      part[k] = f2_hsum(acc);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const int h = kBatch >> (s + 1), off = LPR >> (s + 1);
      const bool upper = (ci & off) != 0;
#pragma unroll
      for (int k = 0; k < h; ++k) {
        const float send = upper ? part[k] : part[k + h];
        const float keep = upper ? part[k + h] : part[k];
        part[k] = keep + __shfl_xor_sync(kFull, send, off);
      }
    }
#pragma unroll
    for (int off = kSpread / 2; off >= 1; off >>= 1)
      part[0] += __shfl_xor_sync(kFull, part[0], off);
    const int j = base + g + (ci / kSpread) * kG;
    if (ci % kSpread == 0 && j < cb) finish(j, sqrtf(part[0]));
  }
}

// The same for every other head dim, and for the Dir rule: four rows (Dir,
// whose second pass needs the first one's sum: two) per group of lpr lanes at
// a time, per row the arithmetic of the streaming kernel's general path (lanes
// added at distance 1, 2, 4, ...).  With at least as many lanes as rows the
// last reduction hands each of the first lanes one row.
// Sm: ResSmem or SmallSmem (the mean in column order, and Dir's factors).
template <int VAR, class Sm, class Finish>
__device__ __forceinline__ void resident_score_general(uint32_t buf, int ca, int cb, int d, int lpr,
                                                       const Sm& S, Finish finish) {
  constexpr int kBatch = VAR == 1 ? 2 : 4, kLog = VAR == 1 ? 1 : 2;
  const int ci = (threadIdx.x & 31) & (lpr - 1), g = threadIdx.x / lpr, ng = kThreads / lpr;
  const bool active = ci < (d >> 3);
  float m8[8], l8[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    m8[k] = (VAR != 2 && active) ? S.mu[ci * 8 + k] : 0.f;
    l8[k] = (VAR != 2 && active) ? S.mulo[ci * 8 + k] : 0.f;
  }
  const bool mu_zero = VAR == 1 && S.mu_zero;
  const float inv_mnorm = VAR == 1 ? S.inv_mnorm : 0.f;
  for (int base = ca; base < cb; base += kBatch * ng) {
    uint4 q[kBatch];
    float acc[kBatch], nv[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int j = base + g + k * ng;
      q[k] = make_uint4(0u, 0u, 0u, 0u);
      if (active && j < cb) q[k] = ld_shared16(buf + (uint32_t)(j * d * 2 + ci * 16));
      nv[k] = 0.f;
    }
    if (VAR == 1) {
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        float x[8];
        unpack8(q[k], x);
#pragma unroll
        for (int e = 0; e < 8; ++e) nv[k] = fmaf(x[e], x[e], nv[k]);
      }
      for (int off = 1; off < lpr; off <<= 1) {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) nv[k] += __shfl_xor_sync(kFull, nv[k], off);
      }
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      float x[8];
      unpack8(q[k], x);
      acc[k] = 0.f;
      const float lam = VAR == 1 ? sqrtf(nv[k]) * inv_mnorm : 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float w = x[e];
        if (VAR == 0) w = (x[e] - m8[e]) - l8[e];
        if (VAR == 1) w = fmaf(-lam, l8[e], fmaf(-lam, m8[e], x[e]));
        acc[k] = fmaf(w, w, acc[k]);
      }
    }
    auto value = [&](float t, float v2) {
      return VAR == 1 ? ((v2 > 0.f && !mu_zero) ? (0.5f * t) / v2 : 1.f) : sqrtf(t);
    };
    if (lpr >= kBatch) {
      const float nk = VAR == 1 && (ci & 1) ? nv[1] : nv[0];  // of the row this lane ends up with
#pragma unroll
      for (int s = 0; s < kLog; ++s) {
        const int h = kBatch >> (s + 1), off = 1 << s;
        const bool upper = (ci & off) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
          const float send = upper ? acc[k] : acc[k + h];
          const float keep = upper ? acc[k + h] : acc[k];
          acc[k] = keep + __shfl_xor_sync(kFull, send, off);
        }
      }
      for (int off = kBatch; off < lpr; off <<= 1) acc[0] += __shfl_xor_sync(kFull, acc[0], off);
      const int r = VAR == 1 ? ci : 2 * (ci & 1) + ((ci >> 1) & 1);
      const int j = base + g + r * ng;
      if (ci < kBatch && j < cb) finish(j, value(acc[0], nk));
    } else {
      for (int off = 1; off < lpr; off <<= 1) {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) acc[k] += __shfl_xor_sync(kFull, acc[k], off);
      }
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        const int j = base + g + k * ng;
        if (ci == 0 && j < cb) finish(j, value(acc[k], nv[k]));
      }
    }
  }
}

// The N-th largest of a unit's keys (all in this CTA's reach), how many
// keys equal to it are kept, and how many there are.  [kmin, kmax] spans the
// keys.  A pass spreads the keys of the current range over 1024 buckets of
// equal width and keeps the bucket that holds the threshold; at most 256 keys
// in it are ranked directly.  The range shrinks 1024-fold per pass, so there
// are at most four (fp32 keys of one unit differ in a few high bits: one pass
// resolves all but heavily tied caches).
// for_keys(use) calls use(key) for every key, spread over the threads.
template <class ForKeys>
__device__ __forceinline__ Selection resident_select(ForKeys for_keys, int N, uint32_t kmin,
                                                     uint32_t kmax, ResSmem& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* hist = reinterpret_cast<uint32_t*>(S.mu);
  int need = N;
  for (;;) {
    const uint32_t range = kmax - kmin;
    const int sh = max(0, 22 - __clz(range));  // (range >> sh) < 1024
    reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) S.ncand = 0;
    __syncthreads();
    for_keys([&](uint32_t key) {
      const uint32_t off = key - kmin;
      if (off <= range) atomicAdd(&hist[off >> sh], 1u);
    });
    __syncthreads();
    // thread t holds buckets 1023 - 4 t .. 1020 - 4 t: prefix sums from the top
    const uint4 h = reinterpret_cast<const uint4*>(hist)[kThreads - 1 - tid];
    const int c[4] = {(int)h.w, (int)h.z, (int)h.y, (int)h.x};
    const int sum = c[0] + c[1] + c[2] + c[3];
    int cum = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(kFull, cum, off);
      if (lane >= off) cum += y;
    }
    if (lane == 31) S.scan[warp] = cum;
    __syncthreads();
    cum -= sum;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) cum += w < warp ? S.scan[w] : 0;
    if (cum < need && need <= cum + sum) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (cum < need && need <= cum + c[i]) {
          S.sel_lo = kmin + ((uint32_t)(kResBuckets - 1 - (tid * 4 + i)) << sh);
          S.sel_above = cum;
          S.sel_cnt = c[i];
        }
        cum += c[i];
      }
    }
    __syncthreads();
    const uint32_t lo = S.sel_lo;
    const int cnt = S.sel_cnt;
    need -= S.sel_above;
    if (sh == 0) return {lo, need, cnt};  // one key value per bucket
    const uint32_t width = (1u << sh) - 1u;
    if (cnt > kThreads) {
      kmin = lo;
      kmax = lo + width;
      __syncthreads();  // sel_* is read before the next pass writes it
      continue;
    }
    for_keys([&](uint32_t key) {
      if (key - lo <= width) {
        const int at = atomicAdd(&S.ncand, 1);
        if (at < kThreads) S.cand[at] = key;
      }
    });
    __syncthreads();
    if (tid < cnt) {
      const uint32_t mine = S.cand[tid];
      int g = 0, e = 0;
      for (int i = 0; i < cnt; i += 8) {
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const uint32_t o = S.cand[min(i + m, cnt - 1)];
          g += i + m < cnt && o > mine;
          e += i + m < cnt && o == mine;
        }
      }
      if (g < need && need <= g + e) {  // every candidate equal to it writes the same
        S.sel_lo = mine;
        S.sel_above = need - g;
        S.sel_cnt = e;
      }
    }
    __syncthreads();
    return {S.sel_lo, S.sel_above, S.sel_cnt};
  }
}

// VAR: 0 L2, 1 Dir, 2 Norm.  DECODE: one token is evicted (arg-min).  HF: the
// hole-fill layout (ties by token position; only the kept rows at or above the
// budget move, from where they are in global memory: the other tensor is not
// loaded).  FUSED: rows at or above len come from the caller's staging buffers.
// Same arguments, validation, outputs and status codes as evict_kernel.
template <int VAR, bool DECODE, bool HF, bool FUSED>
__global__ void __launch_bounds__(kThreads, 3) resident_evict_kernel(const ResidentArgs ra) {
  const EvictArgs& a = ra.e;
  // launched as a programmatic dependent: lets the next kernel be scheduled,
  // sets up its barriers and waits for the previous kernel on the stream
  // before it touches global memory
  grid_launch_dependents();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ResSmem& S = *reinterpret_cast<ResSmem*>(smem_raw);
  const uint32_t bar_s = smem_addr(&S.bar[0]), bar_o = smem_addr(&S.bar[kResChunks]);
  if (threadIdx.x == 0) {
    for (int i = 0; i <= kResChunks; ++i) mbar_init(bar_s + 8u * (uint32_t)i, 1);
    fence_mbar_init();
    S.lost = 0;
    S.best[kResMaxCluster] = ~0ull;
    S.kmax[kResMaxCluster] = 0u;
  }
  __syncthreads();
  grid_dependency_wait();
  const int C = a.cluster, d = a.d, d8 = d >> 3, lpr = a.lpr, cap = a.capacity;
  const ResLayout L = resident_layout(cap, d, C, DECODE, HF, a.mu_running != 0, ra.both != 0);
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw + L.keys);
  float* scratch = reinterpret_cast<float*>(smem_raw + L.keys);
  uint16_t* list = reinterpret_cast<uint16_t*>(smem_raw + L.list);
  uint16_t* holes = reinterpret_cast<uint16_t*>(smem_raw + L.pairs);
  uint16_t* movers = holes + (cap >> 1);
  const uint32_t sbuf = smem_addr(smem_raw + L.buf), obuf = smem_addr(smem_raw + L.obuf);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned rank = C > 1 ? cluster_ctarank() : 0u;
  const int u = C > 1 ? (int)cluster_id_x() : (int)blockIdx.x;
  const int seq = u / a.units_per_seq;
  // from L2: the previous launch may have set it while this one was resident
  const int len0 = __ldcg(a.len + seq);
  const int n = len0 + (FUSED ? a.B : 0);
  const int Nb = a.N_dev ? a.N_dev[seq] : a.N;
  uint16_t* kb = a.k + (size_t)u * cap * d;
  uint16_t* vb = a.v + (size_t)u * cap * d;
  const uint16_t* knu = FUSED ? a.k_new + (size_t)u * a.B * d : nullptr;
  const uint16_t* vnu = FUSED ? a.v_new + (size_t)u * a.B * d : nullptr;

  // ---- validation: uniform across the cluster (per-sequence values only) ---
  if (len0 < 0 || n > cap || (a.mu_running && a.B > n)) {
    if (rank == 0 && tid == 0) record_status(a.status, kStDeviceLen);
    return;
  }
  if (Nb < 1 || Nb > a.N || (DECODE && n > Nb + 1)) {
    if (rank == 0 && tid == 0) record_status(a.status, kStDeviceBudget);
    return;
  }
  const int first_new = n - a.B;
  const int first_stage = FUSED ? len0 : INT_MAX;
  double* rsu = a.mu_running ? a.running_sum + (size_t)u * d : nullptr;
  uint16_t* sb = a.score_k ? kb : vb;  // the scored tensor, and the other one
  uint16_t* ob = a.score_k ? vb : kb;
  const uint16_t* snu = a.score_k ? knu : vnu;
  const uint16_t* onu = a.score_k ? vnu : knu;
  // hole-fill layout: token positions (rows at or above first_new are the
  // appended ones, numbered from pos_new)
  int32_t* posu = HF ? a.pos + (size_t)u * cap : nullptr;
  const int pnew = HF ? a.pos_new[seq] : 0;
  auto pos_of = [&](int r) -> int { return r < first_new ? posu[r] : pnew + (r - first_new); };

  if (n <= Nb) {
    // ---- nothing to evict: append (fused), identity outputs, running sum ---
    if (FUSED) {
      const int i0 = (int)((long long)a.B * rank / C), i1 = (int)((long long)a.B * (rank + 1) / C);
      copy_new_rows(kb, vb, knu + (size_t)i0 * d, vnu + (size_t)i0 * d, d, 0, 2 * d8, len0 + i0,
                    i1 - i0);
    }
    if (HF && rank == 0)
      for (int r = max(first_new, 0) + tid; r < n; r += kThreads) posu[r] = pnew + (r - first_new);
    if (a.kept_out)
      for (int i = (int)rank * kThreads + tid; i < a.N; i += C * kThreads)
        a.kept_out[(size_t)u * a.N + i] = i < n ? i : -1;
    if (DECODE && a.evicted_out && rank == 0 && tid == 0) a.evicted_out[u] = -1;
    if (rsu && a.B > 0 && rank == 0) {
      const uint16_t* nb = FUSED ? snu : sb + (size_t)first_new * d;
      if (DECODE) {
        if (tid < d) rsu[tid] += (double)__uint_as_float((uint32_t)nb[tid] << 16);
      } else {
        const ff t = resident_sum<4>(
            d, lpr, a.B, [&](int i, int c) { return ld_cg16(nb + (size_t)i * d + c * 8); },
            [](int) { return 1.f; }, scratch);
        if (tid < d) rsu[tid] = rsu[tid] + (double)t.hi + (double)t.lo;
      }
    }
    return;
  }

  // ---- 1. this CTA's slice of the scored tensor into shared memory --------
  const int rows_per = resident_rows(n, C);
  const int r0 = min(n, (int)rank * rows_per), r1 = min(n, r0 + rows_per), R = r1 - r0;
  const int row_bytes = d * 2;
  // thread 0: local rows [lo, hi) of a tensor into buf, in one bulk copy (two
  // where they go on into the staged rows)
  const int fs = FUSED ? min(R, max(0, first_stage - r0)) : R;  // the first staged local row
  auto load_rows = [&](uint32_t buf, const uint16_t* base, const uint16_t* stage, int lo, int hi,
                       uint32_t bar) {
    mbar_expect_tx(bar, (uint32_t)(max(0, hi - lo) * row_bytes));
    const int m = min(hi, max(lo, fs));  // [lo, m) cache, [m, hi) staged
    if (lo < m)
      bulk_g2s(buf + (uint32_t)(lo * row_bytes), base + (size_t)(r0 + lo) * d,
               (uint32_t)((m - lo) * row_bytes), bar);
    if (FUSED && m < hi)
      bulk_g2s(buf + (uint32_t)(m * row_bytes), stage + (size_t)(r0 + m - first_stage) * d,
               (uint32_t)((hi - m) * row_bytes), bar);
  };
  // the scored slice in chunks of whole score steps, scored as they land
  const int step = (VAR == 1 ? 2 : lpr * 8 == d && lpr >= 8 ? 8 : 4) * (kThreads / lpr);
  const int rch = ((rows_per + kResChunks * step - 1) / (kResChunks * step)) * step;
  const int nch = (R + rch - 1) / rch;
  if (tid == 0) {
    for (int i = 0; i < nch; ++i)
      load_rows(sbuf, sb, snu, i * rch, min(R, (i + 1) * rch), bar_s + 8u * (uint32_t)i);
    if (!HF && ra.both)
      load_rows(obuf, ob, onu, 0, R, bar_o);
    else if (!HF && !DECODE && fs > 0)  // on its way to L2 while the scores and the select run
      bulk_prefetch_l2(ob + (size_t)r0 * d, (uint32_t)(fs * row_bytes));
  }
  // A wait that gives up goes on with whatever the buffer holds (shared memory
  // only, every index clamped) up to the exchange of step 4, before the first
  // store to the cache.  There the cluster agrees, waits for its copies in flight
  // and leaves the unit as it is.
  auto tell_lost = [&](unsigned cc) {  // to CTA cc of the cluster
    if (DECODE) {
      if (C > 1) st_cluster_u64(mapa(smem_addr(&S.best[kResMaxCluster]), cc), kLostBest);
      else S.best[kResMaxCluster] = kLostBest;
    } else {
      if (C > 1) st_cluster_u32(mapa(smem_addr(&S.kmax[kResMaxCluster]), cc), kLostKey);
      else S.kmax[kResMaxCluster] = kLostKey;
    }
  };
  auto leave_unit = [&]() {
    if (tid != 0) return;
    for (int i = 0; i < nch; ++i) mbar_wait(bar_s + 8u * (uint32_t)i, 0u, a.status, kWaitLimit);
    if (!HF && ra.both) mbar_wait(bar_o, 0u, a.status, kWaitLimit);
    if (rank == 0) {
      __threadfence();  // the status first
      a.len[seq] = mark_len(len0);
    }
  };
  auto ld_row = [&](int j, int ci) {
    return *reinterpret_cast<const uint4*>(smem_raw + L.buf + (size_t)(j * row_bytes + ci * 16));
  };

  // ---- 2. mean -------------------------------------------------------------
  bool met = C == 1;  // the cluster has been through a barrier
  if (VAR != 2) {
    const bool run = rsu != nullptr;
    double sum = run && tid < d ? rsu[tid] : 0.0;
    // the division by n as a product with its reciprocal and one correction
    // (both computed off the critical path: fp64 issues at 1/64 of fp32's rate)
    const double dn = (double)n, rn = tid < d ? 1.0 / dn : 0.0;
    const uint16_t* nb = FUSED ? snu : sb + (size_t)first_new * d;  // the appended rows
    if (DECODE && run) {  // one row, read by every CTA
      if (tid < d) sum += (double)__uint_as_float((uint32_t)nb[tid] << 16);
    } else {
      // The appended rows are read from where they are, so that the mean does
      // not wait for the slice.  Up to 64 KB of them every CTA sums by itself
      // (no exchange); more are shared among kResSumRanks CTAs.
      const int ranks = !run ? C : a.B * row_bytes <= 65536 ? 1 : min(C, kResSumRanks);
      const bool alone = run && ranks == 1;
      ff t{0.f, 0.f};
      if (run) {
        const int per = (a.B + ranks - 1) / ranks;
        const int i0 = alone ? 0 : min(a.B, (int)rank * per), i1 = min(a.B, i0 + per);
        if (alone || (int)rank < ranks)
          t = resident_sum<4>(
              d, lpr, i1 - i0,
              [&](int i, int c) {
                return __ldcg(reinterpret_cast<const uint4*>(nb + (size_t)(i0 + i) * d + c * 8));
              },
              [](int) { return 1.f; }, scratch);
      } else {
        for (int i = 0; i < nch; ++i)
          if (!mbar_wait(bar_s + 8u * (uint32_t)i, 0u, a.status, a.wait_limit)) S.lost = 1;
        t = resident_sum<4>(d, lpr, R, ld_row, [](int) { return 1.f; }, scratch);
      }
      if (C > 1 && !alone) {
        met = true;
        if (tid < d) {
          S.acc_hi[tid] = t.hi;
          S.acc_lo[tid] = t.lo;
        }
        cluster_sync();
        if (tid < d) t = resident_gather(tid, ranks, S);
      }
      if (tid < d) sum = (double)t.hi + (double)t.lo + sum;
    }
    if (tid < d) {
      S.snew[tid] = sum;
      const double m0 = sum * rn, m = fma(fma(-m0, dn, sum), rn, m0);
      const float mh = (float)m;
      S.mu[tid] = mh;
      S.mulo[tid] = (float)(m - (double)mh);
    }
    __syncthreads();
    if (VAR == 1) {
      const float m = tid < d ? S.mu[tid] : 0.f;
      const float nrm2 = block_sum_f32(m * m, S.fsh);
      if (tid == 0) {
        S.mu_zero = !(nrm2 > 0.f);
        S.inv_mnorm = nrm2 > 0.f ? 1.f / sqrtf(nrm2) : 0.f;
      }
      __syncthreads();
    }
  } else {
    if (DECODE && rsu && tid < d) {
      const uint16_t* nb = FUSED ? snu : sb + (size_t)first_new * d;
      S.snew[tid] = rsu[tid] + (double)__uint_as_float((uint32_t)nb[tid] << 16);
    }
  }
  // Peers write into this CTA's keys only once it is past the mean, whose sum
  // used their memory: without an exchange above, they wait for this.
  if (!met) cluster_arrive_relaxed();

  // ---- 3. scores -----------------------------------------------------------
  const bool disp = VAR == 0 && !DECODE && a.disp_out != nullptr;
  float ds_hi = 0.f, ds_lo = 0.f, dq_hi = 0.f, dq_lo = 0.f;
  unsigned long long best = ~0ull;
  uint32_t kmin = 0xffffffffu, kmax = 0u;  // (hole-fill decode: kmin is the minimum's key)
  int best_slot = -1;
  {
    float* sc_out = a.scores_out ? a.scores_out + (size_t)u * cap + r0 : nullptr;
    const float* wu = !DECODE && a.weights ? a.weights + (size_t)u * cap + r0 : nullptr;
    auto finish = [&](int j, float s) {
      if (VAR == 0 && disp) {  // sum s and s^2 (the square split exactly by an FMA)
        ff_accumulate(ds_hi, ds_lo, s);
        const float q2 = s * s;
        ff_accumulate(dq_hi, dq_lo, q2);
        dq_lo += fmaf(s, s, -q2);
      }
      bool bad;
      uint32_t key = score_key(s, bad);
      if (bad) record_status(a.status, kStNonfinite);
      if (!DECODE && wu) {
        // attention-weighted score (the FastCAOTE form of App. A):
        // s'_j = a_j / (1 - a_j) * s_j, for weights a_j in [0, 1)
        const float w = wu[j];
        s = key_score(key) * ((w >= 0.f && w < 1.f) ? w / (1.f - w) : __int_as_float(0x7fc00000));
        key = score_key(s, bad);
        if (bad) record_status(a.status, kStNonfinite);
      }
      if (sc_out) sc_out[j] = s;
      if (DECODE && !HF) {
        const unsigned long long pk = ((unsigned long long)key << 32) |
                                      (unsigned long long)(0xffffffffu - (unsigned)(r0 + j));
        best = pk < best ? pk : best;
      } else if (DECODE) {  // positions are read only to settle an exact tie
        if (key < kmin || best_slot < 0 || (key == kmin && pos_of(r0 + j) > pos_of(best_slot))) {
          kmin = key;
          best_slot = r0 + j;
        }
      } else {
        keys[r0 + j] = key;
        kmin = min(kmin, key);
        kmax = max(kmax, key);
      }
    };
    for (int i = 0; i < nch; ++i) {
      if (!mbar_wait(bar_s + 8u * (uint32_t)i, 0u, a.status, a.wait_limit)) S.lost = 1;
      const int x = i * rch, y = min(R, x + rch);
      if (VAR != 1 && d == 128)
        resident_score_fast<VAR, 16>(sbuf, x, y, S.mu, S.mulo, finish);
      else if (VAR != 1 && d == 64)
        resident_score_fast<VAR, 8>(sbuf, x, y, S.mu, S.mulo, finish);
      else if (VAR != 1 && d == 256)
        resident_score_fast<VAR, 32>(sbuf, x, y, S.mu, S.mulo, finish);
      else
        resident_score_general<VAR>(sbuf, x, y, d, lpr, S, finish);
    }
  }

  // ---- 4. exchange, select, kept list --------------------------------------
  int kept_off = 0, nk = 0, e_first = n;  // block: this slice's kept rows; decode: the evicted slot
  int nhole = 0;                          // hole-fill block: rows that move
  uint32_t tkey = 0u;                     // hole-fill block: a row with key > tkey is kept
  if (DECODE) {
    if (HF) {
      if (best_slot >= 0)
        best = ((unsigned long long)kmin << 32) |
               (unsigned long long)(0xffffffffu - (unsigned)pos_of(best_slot));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(kFull, best, off);
        const int os = __shfl_xor_sync(kFull, best_slot, off);
        if (o < best) {
          best = o;
          best_slot = os;
        }
      }
      if (lane == 0) S.wslot[warp] = best_slot;
    } else {
      best = warp_min_u64(best);
    }
    if (lane == 0) S.wbest[warp] = best;
    __syncthreads();
    if (!met) cluster_wait();
    if (tid < C) {
      unsigned long long b = ~0ull;
      int bs = -1;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        if (HF && S.wbest[w] < b) bs = S.wslot[w];
        b = S.wbest[w] < b ? S.wbest[w] : b;
      }
      if (C > 1) {
        st_cluster_u64(mapa(smem_addr(&S.best[rank]), (unsigned)tid), b);
        if (HF) st_cluster_u32(mapa(smem_addr(&S.best_slot[rank]), (unsigned)tid), (uint32_t)bs);
      } else {
        S.best[0] = b;
        S.best_slot[0] = bs;
      }
      if (S.lost) tell_lost((unsigned)tid);
    }
    if (!HF && ra.both && !mbar_wait(bar_o, 0u, a.status, a.wait_limit_other))
      for (int cc = 0; cc < C; ++cc) tell_lost((unsigned)cc);
    if (C > 1) cluster_sync(); else __syncthreads();
    const unsigned long long mine = lane < C || lane == kResMaxCluster ? S.best[lane] : ~0ull;
    const unsigned long long b = warp_min_u64(mine);
    if (b == kLostBest) return leave_unit();
    if (HF) {  // positions are distinct: one CTA has it
      const unsigned who = __ballot_sync(kFull, mine == b && lane < C);
      e_first = max(0, min(S.best_slot[__ffs(who) - 1], n - 1));
    } else {
      e_first = (int)(0xffffffffu - (unsigned)(b & 0xffffffffull));
    }
    if (a.evicted_out && rank == 0 && tid == 0) a.evicted_out[u] = e_first;
    if (a.kept_out)
      for (int i = (int)rank * kThreads + tid; i < a.N; i += C * kThreads)
        a.kept_out[(size_t)u * a.N + i] =
            i >= Nb ? -1 : HF ? (i == e_first ? n - 1 : i) : i < e_first ? i : i + 1;
  } else {
    kmin = __reduce_min_sync(kFull, kmin);
    kmax = __reduce_max_sync(kFull, kmax);
    if (lane == 0) {
      S.wmin[warp] = kmin;
      S.wmax[warp] = kmax;
    }
    if (VAR == 0 && disp) {
      ff a1 = ff_add(ff{ds_hi, 0.f}, ff{0.f, ds_lo});
      ff a2 = ff_add(ff{dq_hi, 0.f}, ff{0.f, dq_lo});
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        a1 = ff_add(a1, ff_shfl_xor(a1, off));
        a2 = ff_add(a2, ff_shfl_xor(a2, off));
      }
      if (lane == 0) {
        S.dsc[warp] = a1.hi;
        S.dsc[kWarps + warp] = a1.lo;
        S.dsc[2 * kWarps + warp] = a2.hi;
        S.dsc[3 * kWarps + warp] = a2.lo;
      }
    }
    __syncthreads();  // own keys and the warps' results
    if (!met) cluster_wait();
    if (VAR == 0 && disp && tid == 0) {
      ff t1{0.f, 0.f}, t2{0.f, 0.f};
      for (int w = 0; w < kWarps; ++w) {
        t1 = ff_add(t1, ff{S.dsc[w], S.dsc[kWarps + w]});
        t2 = ff_add(t2, ff{S.dsc[2 * kWarps + w], S.dsc[3 * kWarps + w]});
      }
      S.disp[0] = t1.hi;
      S.disp[1] = t1.lo;
      S.disp[2] = t2.hi;
      S.disp[3] = t2.lo;
    }
    if (tid < C) {
      uint32_t mn = S.wmin[0], mx = S.wmax[0];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) {
        mn = min(mn, S.wmin[w]);
        mx = max(mx, S.wmax[w]);
      }
      if (C > 1) {
        st_cluster_u32(mapa(smem_addr(&S.kmin[rank]), (unsigned)tid), mn);
        st_cluster_u32(mapa(smem_addr(&S.kmax[rank]), (unsigned)tid), mx);
      } else {
        S.kmin[0] = mn;
        S.kmax[0] = mx;
      }
      if (S.lost) tell_lost((unsigned)tid);
    }
    if (C > 1) {  // this slice's keys to every peer (the tail of the last slice carries padding)
      const int q4 = (R + 3) >> 2;
      const uint32_t at = smem_addr(keys + r0);
      // warp w serves the peers w, w + 8: a lane's vector goes to each of them
      for (int q = lane; q < q4; q += 32) {
        const uint4 v = reinterpret_cast<const uint4*>(keys + r0)[q];
#pragma unroll
        for (int m = 0; m < kResMaxCluster / kWarps; ++m) {
          const int cc = warp + m * kWarps;
          if (cc < C && cc != (int)rank) st_cluster16(mapa(at + 16u * (uint32_t)q, (unsigned)cc), v);
        }
      }
    }
    if (!HF && ra.both && !mbar_wait(bar_o, 0u, a.status, a.wait_limit_other))
      for (int cc = 0; cc < C; ++cc) tell_lost((unsigned)cc);
    if (C > 1) cluster_sync(); else __syncthreads();
    kmin = __reduce_min_sync(kFull, lane < C ? S.kmin[lane] : 0xffffffffu);
    kmax = __reduce_max_sync(kFull, lane < C || lane == kResMaxCluster ? S.kmax[lane] : 0u);
    if (kmax == kLostKey) return leave_unit();
    Selection sel = resident_select(
        [&](auto use) {  // four keys per load
          const int nv = n >> 2;
#pragma unroll 2
          for (int i = tid; i < nv; i += kThreads) {
            const uint4 k = reinterpret_cast<const uint4*>(keys)[i];
            use(k.x);
            use(k.y);
            use(k.z);
            use(k.w);
          }
          if (tid < (n & 3)) use(keys[4 * nv + tid]);
        },
        Nb, kmin, kmax, S);
    if (HF) {
      // a kept row is one with key > t from here on: the surviving ties are
      // the lowest positions, found by a second select over the complemented
      // positions of the tied rows, whose keys this CTA's copy then raises
      // (t >= 1 where every tie survives: a row with a lower key goes)
      if (sel.cnt_eq > sel.keep_eq) {
        const uint32_t t = sel.t;
        const Selection s2 = resident_select(
            [&](auto use) {
              for (int j = tid; j < n; j += kThreads)
                if (keys[j] == t) use(~(uint32_t)pos_of(j));
            },
            sel.keep_eq, 0u, 0xffffffffu, S);
        for (int j = tid; j < n; j += kThreads)
          if (keys[j] == t && ~(uint32_t)pos_of(j) >= s2.t) keys[j] = t + 1u;
        __syncthreads();
      } else {
        sel.t -= 1u;
      }
      sel.keep_eq = 0;
    }
    if (VAR == 0 && disp && rank == 0 && tid == 0) {
      double s1 = 0.0, s2 = 0.0;
      const uint32_t base = smem_addr(&S.disp[0]);
      for (int rr = 0; rr < C; ++rr) {
        float v[4];
        for (int k = 0; k < 4; ++k)
          v[k] = C > 1 ? ld_cluster_f32(mapa(base + 4u * (unsigned)k, (unsigned)rr)) : S.disp[k];
        s1 += (double)v[0] + (double)v[1];
        s2 += (double)v[2] + (double)v[3];
      }
      const double m = s1 / (double)n;
      const double var = s2 / (double)n - m * m;
      a.disp_out[u] = (float)sqrt(var > 0.0 ? var : 0.0);
    }
    // kept list: counts of keys > t (low half) and == t (high half) before
    // this slice, and before this thread's rows of it; ties go to the lower slot
    const uint32_t t = sel.t;
    tkey = t;
    const int q = sel.keep_eq;
    auto count = [&](uint32_t key) { return (key > t ? 1u : 0u) + (key == t ? 0x10000u : 0u); };
    uint32_t before = 0u, mine = 0u;
    for (int i = tid; i < (r0 >> 2); i += kThreads) {  // whole vectors: r0 is n or a multiple of 4
      const uint4 k = reinterpret_cast<const uint4*>(keys)[i];
      before += count(k.x) + count(k.y) + count(k.z) + count(k.w);
    }
    const int ch = (R + kThreads - 1) / kThreads;
    const int c0 = min(R, tid * ch), c1 = min(R, c0 + ch);
    for (int j = c0; j < c1; ++j) mine += count(keys[r0 + j]);
    before = __reduce_add_sync(kFull, before);
    uint32_t incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += y;
    }
    if (lane == 31) S.scan[warp] = (int)incl;
    if (lane == 0) S.pre[warp] = (int)before;
    __syncthreads();
    uint32_t pre = 0u, ex = incl - mine, tot = 0u;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      pre += (uint32_t)S.pre[w];
      tot += (uint32_t)S.scan[w];
      if (w < warp) ex += (uint32_t)S.scan[w];
    }
    auto kept = [&](uint32_t cnt) { return (int)(cnt & 0xffffu) + min(q, (int)(cnt >> 16)); };
    kept_off = kept(pre);
    nk = kept(pre + tot) - kept_off;
    uint32_t at = pre + ex;
    for (int j = c0; j < c1; ++j) {
      const uint32_t key = keys[r0 + j];
      const bool keep = key > t || (key == t && (int)(at >> 16) < q);
      const int ki = kept(at) - kept_off;          // kept rows of this slice before row j
      const int pos = keep ? ki : nk + (j - ki);
      at += count(key);
      if ((unsigned)pos < (unsigned)R) list[pos] = (uint16_t)j;
      else record_status(a.status, kStInternal);  // never for a consistent selection
    }
    if (HF) {
      // the evicted slots below the budget and the kept ones at or above it,
      // ascending (every CTA lists them all), by contiguous runs of slots
      auto kind = [&](int r) {  // hole: low half, mover: high half
        const bool kp = keys[r] > t;
        return r < Nb ? (kp ? 0u : 1u) : (kp ? 0x10000u : 0u);
      };
      const int run = (n + kThreads - 1) / kThreads;
      const int x = min(n, tid * run), y = min(n, x + run);
      uint32_t own = 0u;
      for (int r = x; r < y; ++r) own += kind(r);
      uint32_t sum = own;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(kFull, sum, off);
        if (lane >= off) sum += z;
      }
      if (lane == 31) S.wslot[warp] = (int)sum;
      __syncthreads();
      uint32_t at2 = sum - own, all = 0u;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        all += (uint32_t)S.wslot[w];
        if (w < warp) at2 += (uint32_t)S.wslot[w];
      }
      nhole = min((int)(all & 0xffffu), cap >> 1);
      if ((all & 0xffffu) != (all >> 16) && tid == 0) record_status(a.status, kStInternal);
      for (int r = x; r < y; ++r) {
        const uint32_t kd = kind(r);
        if ((kd & 1u) && (int)(at2 & 0xffffu) < nhole) holes[at2 & 0xffffu] = (uint16_t)r;
        if ((kd >> 16) && (int)(at2 >> 16) < nhole) movers[at2 >> 16] = (uint16_t)r;
        at2 += kd;
      }
    }
    __syncthreads();
  }

  // ---- 5. running sum: this slice's evicted rows leave it (Norm, which had no
  // mean to compute, adds the appended ones here).  Before any row is written,
  // so that the cluster barrier has no stores to wait for.
  const bool exchange = !DECODE && rsu != nullptr;
  if (exchange) {
    const int j0 = VAR == 2 ? min(R, max(0, first_new - r0)) : R;
    const int nnew = R - j0;
    // one column per thread, kThreads / d threads per column: a short loop (the
    // kernel runs once through its code, so instruction fetch bounds it)
    const int parts = kThreads / d, part = tid / d, c = tid - part * d;
    float hi = 0.f, lo = 0.f;
    if (part < parts) {
#pragma unroll 2
      for (int i = part; i < nnew + R - nk; i += parts) {
        const int j = i < nnew ? j0 + i : min((int)list[nk + i - nnew], R - 1);
        const float x = __uint_as_float(
            (uint32_t)reinterpret_cast<const uint16_t*>(smem_raw + L.buf)[j * d + c] << 16);
        ff_accumulate(hi, lo, i < nnew ? x : -x);
      }
      S.mu[part * d + c] = hi;  // the histogram's memory is free again
      S.mulo[part * d + c] = lo;
    }
    __syncthreads();
    if (tid < d) {
      ff t{0.f, 0.f};
#pragma unroll 1
      for (int m = 0; m < parts; ++m)
        t = ff_add(t, ff{S.mu[m * d + tid], S.mulo[m * d + tid]});
      S.acc_hi[tid] = t.hi;
      S.acc_lo[tid] = t.lo;
    }
    if (C > 1) cluster_arrive(); else __syncthreads();
  }
  if (!DECODE && !HF && a.kept_out) {
    int32_t* ko = a.kept_out + (size_t)u * a.N;
    for (int i = tid; i < nk; i += kThreads)
      if (kept_off + i < a.N) ko[kept_off + i] = r0 + (int)list[i];
    if (rank == 0)
      for (int i = Nb + tid; i < a.N; i += kThreads) ko[i] = -1;
  }

  if constexpr (HF) {
    // ---- 6. hole-fill: movers into holes, from where they are -------------
    // Every source lies at or above the budget and every destination below it;
    // the holes' old rows are in shared memory since before the exchange.
    const int ci = lane & (lpr - 1), g = tid / lpr, ng = kThreads / lpr;
    auto copy_row = [&](int item, int src, int dst) {  // item & 1: K or V
      const uint16_t* from = src >= first_stage
                                 ? ((item & 1) ? vnu : knu) + (size_t)(src - first_stage) * d
                                 : ((item & 1) ? vb : kb) + (size_t)src * d;
      st16(((item & 1) ? vb : kb) + (size_t)dst * d + ci * 8, ld_cg16(from + ci * 8));
    };
    if (DECODE) {
      if (rsu && e_first >= r0 && e_first < r1 && tid < d) {
        const uint16_t* row =
            reinterpret_cast<const uint16_t*>(smem_raw + L.buf) + (size_t)(e_first - r0) * d;
        rsu[tid] = S.snew[tid] - (double)__uint_as_float((uint32_t)row[tid] << 16);
      }
      if (rank == 0 && e_first < Nb) {
        for (int it = g; it < 2 && ci < d8; it += ng) copy_row(it, n - 1, e_first);
        if (tid == 0) posu[e_first] = pos_of(n - 1);
      }
      return;
    }
    if (C > 1 && !exchange) cluster_arrive_relaxed();
    const int mine = nhole > (int)rank ? (nhole - (int)rank + C - 1) / C : 0;
    if (ci < d8) {
      for (int it = g; it < 2 * mine; it += ng) {  // pairs rank, rank + C, ...
        const int i = (int)rank + (it >> 1) * C;
        copy_row(it, movers[i], holes[i]);
      }
      // fused append: kept new rows below the budget into their own slots
      if (FUSED)
        for (int it = g;; it += ng) {
          const int r = first_stage + (int)rank + (it >> 1) * C;
          if (r >= Nb) break;
          if (keys[r] > tkey) copy_row(it, r, r);
        }
    }
    if (a.kept_out) {
      int32_t* ko = a.kept_out + (size_t)u * a.N;
      for (int r = (int)rank * kThreads + tid; r < a.N; r += C * kThreads)
        if (r >= Nb || keys[r] > tkey) ko[r] = r < Nb ? r : -1;
      for (int i = tid; i < mine; i += kThreads) ko[holes[rank + i * C]] = movers[rank + i * C];
    }
    if (C > 1) cluster_wait();  // every CTA is done with the positions, and with its partial sums
    for (int r = max(first_new, 0) + (int)rank * kThreads + tid; r < Nb; r += C * kThreads)
      if (keys[r] > tkey) posu[r] = pnew + (r - first_new);
    for (int i = tid; i < mine; i += kThreads)
      posu[holes[rank + i * C]] = pos_of(movers[rank + i * C]);
    if (exchange) {
      const int c = (int)((unsigned)d * rank / (unsigned)C) + tid;
      if (c < (int)((unsigned)d * (rank + 1) / (unsigned)C)) {
        const ff t = C > 1 ? resident_gather(c, C, S) : ff{S.acc_hi[c], S.acc_lo[c]};
        const double base = VAR != 2 ? S.snew[c] : rsu[c];
        rsu[c] = base + (double)t.hi + (double)t.lo;
      }
      if (C > 1) {  // peers have read this CTA's partial results
        cluster_arrive_relaxed();
        cluster_wait();
      }
    }
    return;
  }

  // ---- 6. kept rows to their slots -----------------------------------------
  // Rows that stay in place (those before the first evicted slot) are not
  // written; staged rows always are.
  const int ci = lane & (lpr - 1), g = tid / lpr, ng = kThreads / lpr;
  auto write_rows = [&](uint16_t* base, size_t buf) {
    if (ci >= d8) return;
    const unsigned char* src = smem_raw + buf + ci * 16;
    uint16_t* out = base + ci * 8;
    constexpr int U = 4;  // rows per thread in flight
    if (DECODE) {  // slots above the evicted one move down by one
      for (int j0 = max(0, e_first + 1 - r0) + g; j0 < R; j0 += U * ng) {
        uint4 q[U];
#pragma unroll
        for (int m = 0; m < U; ++m)
          q[m] = *reinterpret_cast<const uint4*>(src + (size_t)min(j0 + m * ng, R - 1) * row_bytes);
#pragma unroll
        for (int m = 0; m < U; ++m)
          if (j0 + m * ng < R) st16(out + (size_t)(r0 + j0 + m * ng - 1) * d, q[m]);
      }
    } else {
      for (int i0 = g; i0 < nk; i0 += U * ng) {
        uint4 q[U];
        int j[U];
#pragma unroll
        for (int m = 0; m < U; ++m) j[m] = min((int)list[min(i0 + m * ng, nk - 1)], R - 1);
#pragma unroll
        for (int m = 0; m < U; ++m)
          q[m] = *reinterpret_cast<const uint4*>(src + (size_t)j[m] * row_bytes);
#pragma unroll
        for (int m = 0; m < U; ++m) {
          const int i = i0 + m * ng, dst = kept_off + i;
          if (i < nk && (dst != r0 + j[m] || r0 + j[m] >= first_stage) && dst < Nb)
            st16(out + (size_t)dst * d, q[m]);
        }
      }
    }
  };
  write_rows(sb, L.buf);
  if (DECODE && rsu && e_first >= r0 && e_first < r1 && tid < d) {
    // the evicted row leaves the running sum: its owner holds it
    const uint16_t* row =
        reinterpret_cast<const uint16_t*>(smem_raw + L.buf) + (size_t)(e_first - r0) * d;
    rsu[tid] = S.snew[tid] - (double)__uint_as_float((uint32_t)row[tid] << 16);
  }
  if (!ra.both) {
    __syncthreads();  // the slice is no longer read
    if (tid == 0) {
      int lo = 0;  // the first row of the slice that is written again
      if (DECODE) {
        lo = min(R, max(0, e_first + 1 - r0));
      } else if (kept_off == r0) {  // nothing evicted before this slice
        lo = min(nk < R ? (int)list[nk] : R, fs);
      }
      fence_proxy_async_smem();  // generic reads above, bulk writes below
      load_rows(obuf, ob, onu, lo, R, bar_o);
    }
  }
  if (exchange) {
    if (C > 1) cluster_wait();
    // columns [d r / C, d (r + 1) / C) are CTA r's
    const int c = (int)((unsigned)d * rank / (unsigned)C) + tid;
    if (c < (int)((unsigned)d * (rank + 1) / (unsigned)C)) {
      const ff t = C > 1 ? resident_gather(c, C, S) : ff{S.acc_hi[c], S.acc_lo[c]};
      const double base = VAR != 2 ? S.snew[c] : rsu[c];
      rsu[c] = base + (double)t.hi + (double)t.lo;
    }
  }
  if (!ra.both) {
    // The scored tensor is compacted: a wait that gives up here leaves the other
    // one's rows as they are, and the unit's contents are unspecified.  Its copy
    // lands before the barrier, after which peers write what it reads.
    const bool landed = mbar_wait(bar_o, 0u, a.status, a.wait_limit_other);
    if (!landed) {
      mbar_wait(bar_o, 0u, a.status, kWaitLimit);
      __threadfence();  // the status first
      a.len[seq] = mark_len(len0);
    }
    // every CTA holds its rows of the other tensor, and has read its peers'
    // partial results
    if (C > 1) {
      cluster_arrive_relaxed();
      cluster_wait();
    }
    if (landed) write_rows(ob, L.obuf);
  } else {
    const bool late = C > 1 && (exchange || disp);
    if (late) cluster_arrive_relaxed();
    write_rows(ob, L.obuf);
    if (late) cluster_wait();  // peers have read this CTA's partial results
  }
}

}  // namespace vd
