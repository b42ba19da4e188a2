// vd_small.cuh -- pi_N of Sec. 2.1 Eq. (eviction) for short caches, where the
// streaming kernel's machinery (multi-pass radix select, streaming rings, the
// separate length update) costs more than the work itself.
//
// One CTA per (sequence, layer, KV head) unit.  In a launch of few units the
// CTAs of one sequence form one thread-block cluster (units_per_seq <= 16), so
// that after a cluster barrier the sequence's length can be written by the
// kernel itself: one launch per event.  With more units the length update is a
// launch of its own.  The unit's n rows of K and V are copied into shared
// memory once; everything after that reads shared memory:
//
//   1. mean    double-float column sums (running mode: the caller's fp64 sum
//              S plus the appended rows), kept as an fp32 part and remainder
//   2. score   L2 ((v - hi) - lo)^2, Dir |w|^2 / (2 |v|^2) with
//              w = v - (|v|/|m|) m, Norm |v|^2, as in the streaming kernel
//   3. select  decode: an arg-min over (key, -slot); block:
//              rank_j = #{i : key_i > key_j} + #{i < j : key_i == key_j}, row
//              j survives iff rank_j < N (Eq. eviction, ties to the lower
//              slot), n comparisons per thread, four keys per load
//   4. list    kept slots ascending (a block prefix sum), then the evicted
//   5. sum     running mode: S + sum(appended rows) - sum(evicted rows)
//   6. move    rows [first moved, N) written from the shared-memory copy,
//              so the in-place gather has no read-after-write hazard
//
// Bound by the latency of these steps.  The rows arrive by bulk copies (K while
// V is scored), the running sum is read before they land, rows are scored four
// at a time and compacted two at a time: 2 units of 160 rows, d = 64, 9.2 ->
// 7.8 us a call.  Up to 256 rows: beyond, the comparisons cost more than the
// resident kernel's histogram and second launch (d = 64, 256 rows 9.9 us against
// 11.8; d = 32, 384 rows 14.4 against 12.0; d = 16, 1000 rows 45.7 against 13.0).
// With many units three CTAs share an SM; us, streaming kernel / this one: d =
// 128, 128 rows, 320 units 23.7 / 15.7, 1600 units 64 / 42, 4800 units 179 / 108;
// decode, 101 rows, 1600 units 50 / 29.
//
// Same validation, outputs and status codes as the streaming kernel; no hole-fill
// layout and no sigma (those calls take the other kernels).
#pragma once

#include <cstdint>

#include "vd_resident.cuh"

namespace vd {

constexpr int kSmallMaxRows = kThreads;  // one row per thread in the rank select

struct SmallSmem {
  float mu[256];
  float mulo[256];     // mean = mu + mulo (natural column order)
  float part_hi[256];  // column-sum partials, [part][column]
  float part_lo[256];
  unsigned long long bar[2];  // V rows, K rows
  unsigned long long best[kWarps];
  int scan[kWarps];
  float fsh[kWarps];
  float inv_mnorm;
  int mu_zero;
  int lost;               // a wait for this unit's rows gave up
  uint32_t any_lost;      // rank 0: a unit of the sequence did (set by its CTA)
};

struct SmallLayout {
  size_t v, k, keys, perm, total;
};

// rows: the capacity (every row the unit may hold); d: head_dim
__host__ __device__ inline SmallLayout small_layout(int capacity, int d) {
  SmallLayout l;
  l.v = (sizeof(SmallSmem) + 127) & ~(size_t)127;
  l.k = l.v + align16((size_t)capacity * d * 2);
  l.keys = l.k + align16((size_t)capacity * d * 2);
  l.perm = l.keys + align16((size_t)capacity * 4);
  l.total = l.perm + align16((size_t)capacity * 2);
  return l;
}

// acc (S.mu as hi, S.mulo as lo, natural columns) <- sum over list items
// [0, count) of sign(i) * row(i), exact per element (TwoSum); P = 256 / d
// threads per column, each summing items p, p + P, ...; the P partials are
// added in a fixed order.  Returns through hi/lo of threads t < d.
template <class RowOf, class SignOf>
__device__ __forceinline__ ff small_column_sum(int d, int count, RowOf row_of, SignOf sign_of,
                                               SmallSmem& S) {
  const int tid = threadIdx.x;
  const int P = kThreads / d;
  const int col = tid % d, part = tid / d;
  float hi = 0.f, lo = 0.f;
  if (part < P)
#pragma unroll 4
    for (int i = part; i < count; i += P)
      ff_accumulate(hi, lo, sign_of(i) * __uint_as_float((uint32_t)row_of(i)[col] << 16));
  if (part < P) {
    S.part_hi[part * d + col] = hi;
    S.part_lo[part * d + col] = lo;
  }
  __syncthreads();
  ff t{0.f, 0.f};
  if (tid < d)
    for (int p = 0; p < P; ++p) t = ff_add(t, ff{S.part_hi[p * d + tid], S.part_lo[p * d + tid]});
  __syncthreads();
  return t;
}

// The kernel's parameters: the streaming kernel's, plus the number of units.
struct SmallArgs {
  EvictArgs e;
  int32_t n_units;  // n_seq * units_per_seq: the grid's CTAs
  int32_t set_len;  // 1: clusters of a sequence's units, which set its length here
};

// VAR: 0 L2, 1 Dir, 2 Norm.  DECODE: the decode entry points (n <= N + 1);
// the selection is the same.  FUSED: rows at or above len come from the
// caller's staging buffers (the append of Eq. block_processing).
// a.cluster: the cluster size, with set_len the units per sequence, else 1.
// a.capacity <= kSmallMaxRows.
template <int VAR, bool DECODE, bool FUSED>
__global__ void __launch_bounds__(kThreads, 1) small_evict_kernel(const SmallArgs sa) {
  const EvictArgs& a = sa.e;
  // launched as a programmatic dependent: set up the barriers, wait for the
  // previous kernel on the stream before reading anything, and let the next one
  // be scheduled
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmallSmem& S = *reinterpret_cast<SmallSmem*>(smem_raw);
  const uint32_t bar_v = smem_addr(&S.bar[0]), bar_k = smem_addr(&S.bar[1]);
  if (threadIdx.x == 0) {
    mbar_init(bar_v, 1);
    mbar_init(bar_k, 1);
    fence_mbar_init();
    S.lost = 0;
    S.any_lost = 0u;
  }
  const int C = a.cluster;
  if (sa.set_len && C > 1) cluster_arrive();  // waited for before peers set any_lost
  grid_dependency_wait();
  grid_launch_dependents();
  const int d = a.d, d8 = d >> 3, cap = a.capacity;
  const SmallLayout L = small_layout(cap, d);
  uint16_t* Vs = reinterpret_cast<uint16_t*>(smem_raw + L.v);
  uint16_t* Ks = reinterpret_cast<uint16_t*>(smem_raw + L.k);
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw + L.keys);
  uint16_t* perm = reinterpret_cast<uint16_t*>(smem_raw + L.perm);
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned rank = C > 1 ? cluster_ctarank() : 0u;
  const int u = (int)blockIdx.x;
  // a CTA past the last unit (impossible for the host's grid) reads and
  // writes nothing but still reaches the cluster barrier
  const bool unit_ok = u < sa.n_units;
  const int seq = unit_ok ? u / a.units_per_seq : 0;
  // from L2: the previous launch may have set it while this one was resident
  const int len0 = unit_ok ? __ldcg(a.len + seq) : -1;
  const int n = len0 + (FUSED ? a.B : 0);
  const int Nb = unit_ok ? (a.N_dev ? a.N_dev[seq] : a.N) : 0;
  const size_t ubase = (size_t)u * cap * d;
  // "V" is the scored tensor below: K for the key-side rule (the two are
  // otherwise treated alike)
  uint16_t* kb = (a.score_k ? a.v : a.k) + ubase;
  uint16_t* vb = (a.score_k ? a.k : a.v) + ubase;
  const uint16_t* knu = FUSED ? (a.score_k ? a.v_new : a.k_new) + (size_t)u * a.B * d : nullptr;
  const uint16_t* vnu = FUSED ? (a.score_k ? a.k_new : a.v_new) + (size_t)u * a.B * d : nullptr;

  // ---- validation: the same per-sequence checks as the streaming kernel -------
  bool ok = unit_ok;
  if (!unit_ok) {
    if (tid == 0) record_status(a.status, kStInternal);
  } else if (len0 < 0 || n > cap || (a.mu_running && a.B > n)) {
    if (rank == 0 && tid == 0 && u % a.units_per_seq == 0) record_status(a.status, kStDeviceLen);
    ok = false;
  } else if (Nb < 1 || Nb > a.N || (DECODE && n > Nb + 1)) {
    if (rank == 0 && tid == 0 && u % a.units_per_seq == 0)
      record_status(a.status, kStDeviceBudget);
    ok = false;
  }
  const bool evict = ok && n > Nb;
  const int first_new = n - a.B;

  if (ok) {
    // ---- the unit's rows into shared memory: one bulk copy per tensor of the
    // cache rows, one of the staged ones; K, which only the compaction reads,
    // lands while V is scored ---------------------------------------------
    const uint32_t vs_a = smem_addr(Vs), ks_a = smem_addr(Ks);
    double* rsu = a.mu_running ? a.running_sum + (size_t)u * d : nullptr;
    if (tid == 0) {
      const uint32_t row = (uint32_t)d * 2u, old = (uint32_t)len0 * row, all = (uint32_t)n * row;
      for (int t = 0; t < 2; ++t) {
        const uint32_t bar = t ? bar_k : bar_v, dst = t ? ks_a : vs_a;
        mbar_expect_tx(bar, all);
        if (old > 0) bulk_g2s(dst, t ? kb : vb, old, bar);
        if (FUSED) bulk_g2s(dst + old, t ? knu : vnu, all - old, bar);
      }
    }
    // the running sum and 1 / n do not wait for the rows
    const double rs_old = rsu && tid < d ? rsu[tid] : 0.0;
    const double dn = (double)n, rn = tid < d ? 1.0 / dn : 0.0;
    __syncthreads();
    // a wait that gives up leaves the unit as it is: what follows computes on
    // whatever the buffers hold (every index is clamped) and stores none of it
    if (!mbar_wait(bar_v, 0u, a.status, a.wait_limit)) S.lost = 1;
    auto vrow = [&](int r) { return Vs + (size_t)r * d; };

    if (!evict) {
      // ---- nothing to evict: append (fused), running sum += appended rows --
      if (!mbar_wait(bar_k, 0u, a.status, a.wait_limit_other)) S.lost = 1;
      __syncthreads();
      const bool landed = S.lost == 0;
      if (FUSED && landed)
        for (int c = tid; c < a.B * d8; c += kThreads) {
          const int r = len0 + c / d8, col = (c % d8) * 8;
          st16(kb + (size_t)r * d + col, ld_shared16(ks_a + (uint32_t)(r * d + col) * 2u));
          st16(vb + (size_t)r * d + col, ld_shared16(vs_a + (uint32_t)(r * d + col) * 2u));
        }
      if (a.kept_out && landed)
        for (int i = tid; i < a.N; i += kThreads) a.kept_out[(size_t)u * a.N + i] = i < n ? i : -1;
      if (DECODE && a.evicted_out && landed && tid == 0) a.evicted_out[u] = -1;
      if (rsu && a.B > 0 && landed) {
        const ff t = small_column_sum(d, a.B, [&](int i) { return vrow(first_new + i); },
                                      [](int) { return 1.f; }, S);
        if (tid < d) rsu[tid] = rs_old + (double)t.hi + (double)t.lo;
      }
    } else {
      // ---- 1. mean ----------------------------------------------------
      double s_app = 0.0;  // running mode: the caller's sum plus the appended rows
      if (VAR != 2 || rsu) {
        const bool run = rsu != nullptr;
        const int cnt = run ? a.B : n;
        const int r0 = run ? first_new : 0;
        const ff t = small_column_sum(d, cnt, [&](int i) { return vrow(r0 + i); },
                                      [](int) { return 1.f; }, S);
        if (tid < d) {
          double sum = (double)t.hi + (double)t.lo;
          if (run) sum += rs_old;
          s_app = sum;
          // sum / n as a product with the reciprocal and one correction
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
      }
      // ---- 2. scores: lpr lanes per row, one 16-byte chunk each ----------
      float* sc_out = a.scores_out ? a.scores_out + (size_t)u * cap : nullptr;
      const float* wu = !DECODE && a.weights ? a.weights + (size_t)u * cap : nullptr;
      resident_score_general<VAR>(vs_a, 0, n, d, a.lpr, S, [&](int j, float sc) {
        bool bad;
        uint32_t key = score_key(sc, bad);
        if (bad) record_status(a.status, kStNonfinite);
        if (!DECODE && wu) {  // a_j / (1 - a_j) * s_j (the FastCAOTE form of App. A)
          const float w = wu[j];
          sc = key_score(key) * ((w >= 0.f && w < 1.f) ? w / (1.f - w) : __int_as_float(0x7fc00000));
          key = score_key(sc, bad);
          if (bad) record_status(a.status, kStNonfinite);
        }
        keys[j] = key;
        if (sc_out) sc_out[j] = sc;
      });
      __syncthreads();

      // ---- 3./4. rank select and the kept list -------------------------
      // perm entries index the shared-memory copy: clamped to [0, n) so that
      // even after a failed self-check no access leaves it
      int e_first;  // the lowest evicted slot
      if (DECODE) {
        // one row goes: the lowest key, the highest slot among equal ones
        unsigned long long best = ~0ull;
        if (tid < n)
          best = ((unsigned long long)keys[tid] << 32) | (unsigned long long)(0xffffffffu - (unsigned)tid);
        best = warp_min_u64(best);
        if (lane == 0) S.best[tid >> 5] = best;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kWarps; ++w) best = S.best[w] < best ? S.best[w] : best;
        e_first = min((int)(0xffffffffu - (unsigned)(best & 0xffffffffull)), n - 1);
      } else {
        // thread t owns row t, so prefix sums follow slot order (ties go to the
        // lower slot)
        bool keep = false;
        if (tid < n) {
          const uint32_t kj = keys[tid];
          int rank_j = 0;
          auto rank_against = [&](uint32_t ki, int i) {
            rank_j += (ki > kj) | ((ki == kj) & (i < tid));
          };
          const uint4* k4 = reinterpret_cast<const uint4*>(keys);  // four keys per load
#pragma unroll 4
          for (int i = 0; i < (n >> 2); ++i) {
            const uint4 k = k4[i];
            rank_against(k.x, 4 * i);
            rank_against(k.y, 4 * i + 1);
            rank_against(k.z, 4 * i + 2);
            rank_against(k.w, 4 * i + 3);
          }
          for (int i = n & ~3; i < n; ++i) rank_against(keys[i], i);
          keep = rank_j < Nb;
        }
        int total_kept;
        const int kept_at = block_exclusive_scan(keep ? 1 : 0, S.scan, total_kept);
        if (tid < n) {
          const int pos = keep ? kept_at : Nb + (tid - kept_at);
          if ((unsigned)pos >= (unsigned)n || total_kept != Nb)  // self-check
            record_status(a.status, kStInternal);
          else
            perm[pos] = (uint16_t)tid;
        }
        __syncthreads();
        e_first = min((int)perm[Nb], n - 1);
      }
      auto slot = [&](int i) {
        if (DECODE) return min(i < Nb ? i + (i >= e_first) : e_first, n - 1);
        return min((int)perm[i], n - 1);
      };

      // ---- 5. running sum: (S + appended) - evicted rows ------------------
      double s_left = s_app;
      if (rsu) {
        const ff t = small_column_sum(d, n - Nb, [&](int i) { return vrow(slot(Nb + i)); },
                                      [](int) { return -1.f; }, S);
        if (tid < d) s_left = s_app + (double)t.hi + (double)t.lo;
      }

      // ---- outputs, once K has landed too --------------------------------
      if (!mbar_wait(bar_k, 0u, a.status, a.wait_limit_other)) S.lost = 1;
      __syncthreads();
      const bool landed = S.lost == 0;
      if (rsu && landed && tid < d) rsu[tid] = s_left;
      if (a.kept_out && landed)
        for (int i = tid; i < a.N; i += kThreads)
          a.kept_out[(size_t)u * a.N + i] = i < Nb ? slot(i) : -1;
      if (DECODE && a.evicted_out && landed && tid == 0) a.evicted_out[u] = e_first;

      // ---- 6. compaction from the shared-memory copy ---------------------
      // (fused: the kept new rows below the budget are written too)
      const int r_begin = FUSED ? min(e_first, len0) : e_first;
      const int ci = lane & (a.lpr - 1), g = tid / a.lpr, ng = kThreads / a.lpr;
      const unsigned char* vp = reinterpret_cast<const unsigned char*>(Vs) + ci * 16;
      const unsigned char* kp = reinterpret_cast<const unsigned char*>(Ks) + ci * 16;
      if (ci < d8 && landed)
        for (int r0 = r_begin + g; r0 < Nb; r0 += 2 * ng) {
          uint4 qk[2], qv[2];  // two rows of each tensor in flight
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const size_t src = (size_t)slot(min(r0 + m * ng, Nb - 1)) * d * 2;
            qk[m] = *reinterpret_cast<const uint4*>(kp + src);
            qv[m] = *reinterpret_cast<const uint4*>(vp + src);
          }
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            if (r0 + m * ng >= Nb) break;
            const size_t dst = (size_t)(r0 + m * ng) * d + ci * 8;
            st16(kb + dst, qk[m]);
            st16(vb + dst, qv[m]);
          }
        }
    }
    if (tid == 0 && S.lost) {
      mbar_wait(bar_v, 0u, a.status, kWaitLimit);
      mbar_wait(bar_k, 0u, a.status, kWaitLimit);
      if (!sa.set_len) {
        __threadfence();  // the status first
        a.len[seq] = mark_len(len0);
      }
    }
  }

  // ---- the sequence's new length, once every unit of it has read len -----
  if (!sa.set_len) return;  // a launch of its own does it
  if (C > 1) {
    cluster_wait();  // every CTA has set up its shared memory (long ago)
    if (ok && tid == 0 && S.lost) st_cluster_u32(mapa(smem_addr(&S.any_lost), 0u), 1u);
    cluster_sync();
  } else {
    if (tid == 0 && S.lost) S.any_lost = 1u;
    __syncthreads();
  }
  if (ok && (evict || FUSED) && rank == 0 && tid == 0 && u + C <= sa.n_units && !S.any_lost)
    a.len[seq] = evict ? Nb : n;
}

}  // namespace vd
