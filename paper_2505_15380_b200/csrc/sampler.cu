// Fused logits -> sampling transform -> acceptance test -> residual resample / bonus draw
// (Algorithm 1's inner loop, Eq. 5 and Eq. 6), plus the KV commit.  Probability rows q_i never
// reach global memory: each (stream, row) CTA keeps its row in shared memory, tests its draft token
// and draws the token that would follow if this were the first rejected row; it leaves one word.  The CTA
// that finishes last for a stream picks the accepted length k and row k's token.
//
// What bounds it: the chain of trips to memory and block barriers of ONE row (6564 logits are seven per
// thread), not bytes.  So every row draws ahead of the decision (rereading row k afterwards cost three
// more trips to L2), block reductions take two warp steps, and the cuts below one histogram pass.
//
// p = DRAFT distribution, q = TARGET distribution, as in the paper.
#include <math_constants.h>

#include <mutex>

#include "kernels.h"
#include "tc.h"
#include "tc_ptx.cuh"

namespace ssd {

constexpr int SAMP_THREADS = 1024;  // a row of a few thousand logits: short per-thread loops

struct RowStats {
  float zmax;        // max of z = logit / T over the row
  float sum;         // sum of exp(z - zmax) over the kept set
  uint32_t thr_key;  // order-preserving key of the smallest kept value (0 when top-k is off)
  int tie_id_max;    // among values equal to the threshold, ids <= this are kept
};

// Monotone map float -> uint32 (larger float <=> larger key).
__device__ __forceinline__ uint32_t order_key(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) { return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k); }
__device__ __forceinline__ bool is_kept(float z, int t, const RowStats& s) {
  uint32_t k = order_key(z);
  return k > s.thr_key || (k == s.thr_key && t <= s.tie_id_max);
}

// Sums of two values over the block, in every thread: lanes, then warps (fixed order).
__device__ __forceinline__ double2 block_sum_d(double a, double b, bool two, double2* red) {
  a = warp_sum_d(a);
  if (two) b = warp_sum_d(b);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(a, b);
  __syncthreads();
  const double2 v = red[threadIdx.x & 31];
  return make_double2(warp_sum_d(v.x), two ? warp_sum_d(v.y) : 0.0);
}

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long r = 0;
  for (int i = 0; i < SAMP_THREADS / 32; ++i) r += red[i];
  __syncthreads();
  return r;
}
// Mass exp(x), x <= 0, in units of 2^-32: integer sums of these do not depend on the order of
// the additions, so the nucleus cut is the same in every run.
__device__ __forceinline__ unsigned long long mass_fx(float x) { return __float2ull_rn(expf(x) * 4294967296.f); }

// Repetition-aware sampling: a nucleus draw that repeats one of the last `win` tokens at least
// win * tau times is thrown away and redrawn from the full softmax.  As one distribution:
//   q(x) = q_nuc(x) [x not repeated] + R q_full(x),  R = mass of q_nuc on the repeated ids.
constexpr int RAS_MAX_WIN = 32;
struct Ras {
  int win;               // 0: off
  float thresh;          // win * tau
  const int32_t* recent; // [B, win]: last tokens of T_in, oldest first, pending token last, -1 = none
};
struct RasRow {
  float sum_full;  // sum of exp(z - zmax) over all ids
  float R;
};

constexpr int SEL_BINS = 512;  // bins of a row's range of values, for the cuts
constexpr int SEL_CAND = 512;  // most ids of the bin in which a cut falls that are ranked one by one

struct SampSmem {
  int rep_ids[RAS_MAX_WIN];  // repeated ids of this row's window (-1: none)
  uint32_t cnt[SEL_BINS];                 // ids per bin
  uint32_t mass_lo[SEL_BINS], mass_hi[SEL_BINS];  // their mass, low 16 bits and the rest (32-bit atomics, no carries)
  union {  // the cuts' candidates; later the draw's running sums
    struct {
      unsigned long long cand_mass[SEL_CAND];
      uint32_t cand_key[SEL_CAND];
      int cand_id[SEL_CAND];
    };
    double scan[SAMP_THREADS];
  };
  unsigned long long hist_fx[256];
  unsigned long long red_u[SAMP_THREADS / 32];
  unsigned long long mass_above, target;
  double2 red_d2[SAMP_THREADS / 32];
  double red_d[SAMP_THREADS / 32];
  uint32_t red_max[SAMP_THREADS / 32], red_min[SAMP_THREADS / 32];
  int hist[256];
  uint32_t prefix, cut;
  int k_rem, eq_count, tie_id, cut_id, sel_bin, n_cand, y;
};

// A row's values by size in bins of equal width, bin 0 the largest: monotone, so a cut falls in one bin.
struct BinMap {
  float zmax, scale;
  bool ok;  // a finite range (else the cuts use the bits of the values)
  __device__ __forceinline__ int operator()(float z) const {
    return min((int)__fmul_rn(__fsub_rn(zmax, z), scale), SEL_BINS - 1);
  }
};

// Before the row arrives: nothing is counted yet.  The load's barrier publishes it.
__device__ __forceinline__ void clear_bins(SampSmem& sm) {
  for (int i = threadIdx.x; i < SEL_BINS; i += SAMP_THREADS) sm.cnt[i] = sm.mass_lo[i] = sm.mass_hi[i] = 0u;
}

// A row of logits to z / T in shared memory; its range.  Block-collective.
__device__ __forceinline__ BinMap load_row(const float* __restrict__ lrow, int V, float inv_t, float* z, SampSmem& sm,
                                           int32_t* status) {
  float mx = -CUDART_INF_F, mn = CUDART_INF_F;
  int bad = 0;
#pragma unroll 8
  for (int t = threadIdx.x; t < V; t += SAMP_THREADS) {
    const float v = lrow[t];
    if (!isfinite(v)) bad = 1;
    const float x = v * inv_t;
    z[t] = x;
    mx = fmaxf(mx, x);
    mn = fminf(mn, x);
  }
  const uint32_t kmx = __reduce_max_sync(0xffffffffu, order_key(mx)), kmn = __reduce_min_sync(0xffffffffu, order_key(mn));
  if ((threadIdx.x & 31) == 0) {
    sm.red_max[threadIdx.x >> 5] = kmx;
    sm.red_min[threadIdx.x >> 5] = kmn;
  }
  bad = __syncthreads_or(bad);
  if (bad && threadIdx.x == 0) atomicOr(status, SSD_STATUS_NONFINITE);
  BinMap m;
  m.zmax = key_value(__reduce_max_sync(0xffffffffu, sm.red_max[threadIdx.x & 31]));
  const float range = m.zmax - key_value(__reduce_min_sync(0xffffffffu, sm.red_min[threadIdx.x & 31]));
  m.ok = !bad && range > 1e-20f && range < 1e30f;
  m.scale = (float)SEL_BINS / range;
  return m;
}

// Both cuts: one pass counts ids (or adds up masses) per bin, one warp finds the bin in which the cut
// falls, a second pass lists that bin's ids, and each of those finds its own place among them.  A radix select
// over the bits of the values took four passes and, since the top eight bits of a row take a handful of values,
// serialised its shared-memory atomics.  Rows that do not spread over the bins (more than SEL_CAND ids
// in that one, e.g. many equal values) still take it.

// The top_k-th largest id (lower id first among equals).  False: not found this way.
__device__ bool cut_by_count(const float* z, int V, int top_k, const BinMap& map, SampSmem& sm, RowStats& st) {
  const int tid = threadIdx.x;
  for (int t = tid; t < V; t += SAMP_THREADS) atomicAdd(&sm.cnt[map(z[t])], 1u);
  __syncthreads();
  if (tid < 32) {
    constexpr int PER = SEL_BINS / 32;
    uint32_t h[PER], tot = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) tot += h[i] = sm.cnt[PER * tid + i];
    uint32_t run = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, run, o);
      if (tid >= o) run += v;
    }
    run -= tot;
    if (run < (uint32_t)top_k && run + tot >= (uint32_t)top_k) {
      bool found = false;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (!found && run + h[i] >= (uint32_t)top_k) {
          found = true;
          sm.sel_bin = PER * tid + i;
          sm.k_rem = top_k - (int)run;
        }
        run += h[i];
      }
    }
    if (tid == 0) sm.n_cand = 0;
  }
  __syncthreads();
  const int sel = sm.sel_bin;
  for (int t = tid; t < V; t += SAMP_THREADS) {
    const float x = z[t];
    if (map(x) == sel) {
      const int i = atomicAdd(&sm.n_cand, 1);
      if (i < SEL_CAND) {
        sm.cand_key[i] = order_key(x);
        sm.cand_id[i] = t;
      }
    }
  }
  __syncthreads();
  const int n = sm.n_cand;
  if (n > SEL_CAND) return false;
  if (tid < n) {
    const uint32_t key = sm.cand_key[tid];
    const int id = sm.cand_id[tid];
    int before = 0;
    for (int i = 0; i < n; ++i) before += sm.cand_key[i] > key || (sm.cand_key[i] == key && sm.cand_id[i] < id);
    if (before == sm.k_rem - 1) {
      sm.cut = key;
      sm.cut_id = id;
    }
  }
  __syncthreads();
  st.thr_key = sm.cut;
  st.tie_id_max = sm.cut_id;
  return true;
}

// The id at which the running mass of the kept ids first reaches top_p of their mass.
__device__ bool cut_by_mass(const float* z, int V, float top_p, const BinMap& map, SampSmem& sm, RowStats& st) {
  const int tid = threadIdx.x;
  for (int t = tid; t < V; t += SAMP_THREADS) {
    const float x = z[t];
    if (is_kept(x, t, st)) {
      const unsigned long long m = mass_fx(x - st.zmax);
      const int b = map(x);
      if (m) {  // (V is below 2^16: neither word overflows)
        atomicAdd(&sm.mass_lo[b], (uint32_t)m & 0xffffu);
        atomicAdd(&sm.mass_hi[b], (uint32_t)(m >> 16));
      }
    }
  }
  __syncthreads();
  if (tid < 32) {
    constexpr int PER = SEL_BINS / 32;
    auto mass = [&](int i) { return (unsigned long long)sm.mass_lo[PER * tid + i] + ((unsigned long long)sm.mass_hi[PER * tid + i] << 16); };
    unsigned long long tot = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) tot += mass(i);
    unsigned long long run = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long v = __shfl_up_sync(0xffffffffu, run, o);
      if (tid >= o) run += v;
    }
    const unsigned long long total = __shfl_sync(0xffffffffu, run, 31);
    run -= tot;
    const double td = (double)top_p * (double)total;
    unsigned long long target = (unsigned long long)td;
    if ((double)target < td) ++target;  // an id stays iff (mass before it) < target
    if (target < 1) target = 1;
    if (run < target && run + tot >= target) {
      bool found = false;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const unsigned long long h = mass(i);
        if (!found && run + h >= target) {
          found = true;
          sm.sel_bin = PER * tid + i;
          sm.mass_above = run;
        }
        run += h;
      }
    }
    if (tid == 0) {
      sm.target = target;
      sm.n_cand = 0;
    }
  }
  __syncthreads();
  const int sel = sm.sel_bin;
  for (int t = tid; t < V; t += SAMP_THREADS) {
    const float x = z[t];
    if (map(x) == sel && is_kept(x, t, st)) {
      const int i = atomicAdd(&sm.n_cand, 1);
      if (i < SEL_CAND) {
        sm.cand_key[i] = order_key(x);
        sm.cand_id[i] = t;
        sm.cand_mass[i] = mass_fx(x - st.zmax);
      }
    }
  }
  __syncthreads();
  const int n = sm.n_cand;
  if (n > SEL_CAND) return false;
  if (tid < n) {
    const uint32_t key = sm.cand_key[tid];
    const int id = sm.cand_id[tid];
    unsigned long long before = sm.mass_above;
    for (int i = 0; i < n; ++i)
      if (sm.cand_key[i] > key || (sm.cand_key[i] == key && sm.cand_id[i] < id)) before += sm.cand_mass[i];
    if (before < sm.target && before + sm.cand_mass[tid] >= sm.target) {
      sm.cut = key;
      sm.cut_id = id;
    }
  }
  __syncthreads();
  st.thr_key = sm.cut;
  st.tie_id_max = sm.cut_id;
  return true;
}

// The same cuts by a radix select over the bits of the values.
__device__ __noinline__ void radix_cut_by_count(const float* z, int V, int top_k, SampSmem& sm, RowStats& st) {
  {
    __syncthreads();
    // radix select (4 passes of 8 bits, most significant first) of the top_k-th largest key
    if (threadIdx.x == 0) { sm.prefix = 0u; sm.k_rem = top_k; }
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = threadIdx.x; i < 256; i += SAMP_THREADS) sm.hist[i] = 0;
      __syncthreads();
      const uint32_t prefix = sm.prefix;
      const uint32_t mask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
      for (int t = threadIdx.x; t < V; t += SAMP_THREADS) {
        uint32_t k = order_key(z[t]);
        if ((k & mask) == prefix) atomicAdd(&sm.hist[(k >> shift) & 0xFF], 1);
      }
      __syncthreads();
      if (threadIdx.x < 32) {
        // the highest bin at which the count from the top reaches k_rem (bin 0 if none does), found
        // by the first warp: 8 bins per lane, a suffix sum over the lanes, then a walk of 8 bins
        const int lane = threadIdx.x, rem0 = sm.k_rem;
        int h[8], tot = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) { h[i] = sm.hist[8 * lane + i]; tot += h[i]; }
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_down_sync(0xffffffffu, incl, o);
          if (lane + o < 32) incl += v;
        }
        const int above = incl - tot;  // in the bins of the higher lanes
        const bool mine = above < rem0 && above + tot >= rem0;
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        if (bal == 0u ? lane == 0 : mine) {
          int run = above, bin = 8 * lane;  // no crossing: bin 0, everything above it counted
          if (bal == 0u) {
            run = incl - h[0];
          } else {
#pragma unroll
            for (int i = 7; i >= 0; --i) {
              if (run + h[i] >= rem0) { bin = 8 * lane + i; break; }
              run += h[i];
            }
          }
          sm.prefix = prefix | ((uint32_t)bin << shift);
          sm.k_rem = rem0 - run;
          sm.eq_count = sm.hist[bin];
        }
      }
      __syncthreads();
    }
    st.thr_key = sm.prefix;
    if (sm.eq_count > sm.k_rem) {  // equal values straddle the cut: keep the k_rem lowest ids
      if (threadIdx.x == 0) {
        int need = sm.k_rem, t = 0;
        for (; t < V; ++t)
          if (order_key(z[t]) == st.thr_key && --need == 0) break;
        sm.tie_id = t;
      }
      __syncthreads();
      st.tie_id_max = sm.tie_id;
    }
    __syncthreads();
  }
}
__device__ __noinline__ void radix_cut_by_mass(const float* z, int V, float top_p, SampSmem& sm, RowStats& st) {
  {
    __syncthreads();
    // Nucleus: walking the kept ids from the most to the least probable (lower id first among
    // equals), an id stays while the mass before it is below top_p of the kept mass.  The id at
    // which the running mass first reaches that target is found by a radix select over the
    // ordered keys with histograms of mass instead of counts.
    unsigned long long mine = 0;
    for (int t = threadIdx.x; t < V; t += SAMP_THREADS)
      if (is_kept(z[t], t, st)) mine += mass_fx(z[t] - st.zmax);
    const unsigned long long total = block_sum_u64(mine, sm.red_u);
    const double td = (double)top_p * (double)total;
    unsigned long long target = (unsigned long long)td;
    if ((double)target < td) ++target;  // an id stays iff (mass before it) < target
    if (target < 1) target = 1;
    if (threadIdx.x == 0) { sm.prefix = 0u; sm.mass_above = 0; }
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = threadIdx.x; i < 256; i += SAMP_THREADS) { sm.hist_fx[i] = 0; sm.hist[i] = 0; }
      __syncthreads();
      const uint32_t prefix = sm.prefix;
      const uint32_t mask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
      for (int t = threadIdx.x; t < V; t += SAMP_THREADS) {
        const uint32_t k = order_key(z[t]);
        if ((k & mask) == prefix && is_kept(z[t], t, st)) {
          atomicAdd(&sm.hist_fx[(k >> shift) & 0xFF], mass_fx(z[t] - st.zmax));
          atomicAdd(&sm.hist[(k >> shift) & 0xFF], 1);
        }
      }
      __syncthreads();
      if (threadIdx.x < 32) {
        // the highest bin at which the mass from the top reaches the target (bin 0 if none does):
        // the same walk as for the counts, on the mass histogram
        const int lane = threadIdx.x;
        const unsigned long long base = sm.mass_above;
        unsigned long long h[8], tot = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) { h[i] = sm.hist_fx[8 * lane + i]; tot += h[i]; }
        unsigned long long incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned long long v = __shfl_down_sync(0xffffffffu, incl, o);
          if (lane + o < 32) incl += v;
        }
        const unsigned long long above = base + (incl - tot);
        const bool mine = above < target && above + tot >= target;
        const unsigned bal = __ballot_sync(0xffffffffu, mine);
        if (bal == 0u ? lane == 0 : mine) {
          unsigned long long run = above;
          int bin = 8 * lane;
          if (bal == 0u) {
            run = base + (incl - h[0]);
          } else {
#pragma unroll
            for (int i = 7; i >= 0; --i) {
              if (run + h[i] >= target) { bin = 8 * lane + i; break; }
              run += h[i];
            }
          }
          sm.prefix = prefix | ((uint32_t)bin << shift);
          sm.mass_above = run;
          sm.eq_count = sm.hist[bin];
        }
      }
      __syncthreads();
    }
    const uint32_t cut = sm.prefix;
    int tie_id = st.thr_key == cut ? st.tie_id_max : V;  // ties already trimmed by the top-k cut
    if (threadIdx.x == 0) {
      // ids with the cut's value have equal mass: as many of them as it takes to reach the target
      sm.tie_id = tie_id;
      if (sm.eq_count > 1) {
        unsigned long long each = 0;
        int first = -1;
        for (int t = 0; t < V && first < 0; ++t)
          if (order_key(z[t]) == cut && is_kept(z[t], t, st)) first = t;
        each = first >= 0 ? mass_fx(z[first] - st.zmax) : 1;
        if (each < 1) each = 1;
        unsigned long long need = (target - sm.mass_above + each - 1) / each;
        if (need < 1) need = 1;
        if (need < (unsigned long long)sm.eq_count) {
          int t = first;
          for (; t < V; ++t)
            if (order_key(z[t]) == cut && is_kept(z[t], t, st) && --need == 0) break;
          sm.tie_id = t;
        }
      }
    }
    __syncthreads();
    st.thr_key = cut;
    st.tie_id_max = sm.tie_id;
    __syncthreads();
  }
}

// exp(z - zmax) of an id, negative where the id is cut off (zero there unless `full`).
__device__ __forceinline__ float signed_exp(float z, int t, const RowStats& st, bool full) {
  const bool kept = is_kept(z, t, st);
  if (!kept && !full) return 0.f;
  const float e = expf(z - st.zmax);
  return kept ? e : -e;
}

// Row statistics of the sampling transform of a loaded row, and the sum over all ids where `full` asks for it;
// z becomes signed_exp.  Block-collective.
__device__ __forceinline__ RowStats compute_row_stats(float* z, int V, int top_k, float top_p, const BinMap& map,
                                                      bool full, float* sum_full, SampSmem& sm) {
  RowStats st;
  st.zmax = map.zmax;
  st.thr_key = 0u;
  st.tie_id_max = V;
  if (top_k > 0 && top_k < V && !(map.ok && cut_by_count(z, V, top_k, map, sm, st))) radix_cut_by_count(z, V, top_k, sm, st);
  if (top_p > 0.f && top_p < 1.f && !(map.ok && cut_by_mass(z, V, top_p, map, sm, st))) radix_cut_by_mass(z, V, top_p, sm, st);
  double s = 0.0, f = 0.0;
#pragma unroll 4
  for (int t = threadIdx.x; t < V; t += SAMP_THREADS) {
    const float v = signed_exp(z[t], t, st, full);
    z[t] = v;
    if (v > 0.f) s += (double)v;
    if (full) f += (double)fabsf(v);
  }
  const double2 sums = block_sum_d(s, f, full, sm.red_d2);
  st.sum = (float)sums.x;
  *sum_full = (float)sums.y;
  return st;
}

// Inverse-CDF draw in ascending id over weights w[0..V) (shared): smallest t whose inclusive
// cumulative sum exceeds u * total.  Returns -1 through *total_out <= 0.  Block-collective.
__device__ int block_inverse_cdf(const float* w, int V, float u, SampSmem& sm, double* total_out) {
  const int seg = (V + SAMP_THREADS - 1) / SAMP_THREADS;
  const int t0 = min(threadIdx.x * seg, V), t1 = min(t0 + seg, V);
  double s = 0.0;
  for (int t = t0; t < t1; ++t) s += (double)w[t];
  if (threadIdx.x == 0) sm.y = -1;
  {  // inclusive scan of the threads' sums in a fixed order: inside each warp, then over the warps
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double n = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += n;
    }
    if (lane == 31) sm.red_d[wp] = s;
    __syncthreads();
    if (wp == 0) {
      double v = lane < SAMP_THREADS / 32 ? sm.red_d[lane] : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += n;
      }
      if (lane < SAMP_THREADS / 32) sm.red_d[lane] = v;
    }
    __syncthreads();
    if (wp > 0) s += sm.red_d[wp - 1];
    sm.scan[threadIdx.x] = s;
  }
  __syncthreads();
  const double total = sm.scan[SAMP_THREADS - 1];
  *total_out = total;
  if (!(total > 0.0)) {
    __syncthreads();
    return -1;
  }
  const double target = (double)u * total;
  const double incl = sm.scan[threadIdx.x];
  const double excl = threadIdx.x == 0 ? 0.0 : sm.scan[threadIdx.x - 1];
  if (excl <= target && target < incl) {
    double run = excl;
    int y = -1;
    for (int t = t0; t < t1; ++t) {
      run += (double)w[t];
      if (w[t] > 0.f) {
        y = t;
        if (run > target) break;
      }
    }
    sm.y = y;
  }
  __syncthreads();
  if (sm.y < 0 && threadIdx.x == 0) {  // u * total rounded up to total: last id with mass
    int t = V - 1;
    while (t > 0 && !(w[t] > 0.f)) --t;
    sm.y = t;
  }
  __syncthreads();
  int y = sm.y;
  __syncthreads();
  return y;
}

// The repeated ids of row r's window: the last `win` tokens of recent[b] ++ x_1..x_r (row r's
// own token x_{r+1} is not part of it).  One warp; leaves them in sm.rep_ids.
__device__ __forceinline__ void ras_window(const Ras& ras, const int32_t* __restrict__ draft_tokens, int gamma, int b, int r,
                                           int V, SampSmem& sm) {
  const int j = threadIdx.x & 31, c = r + j;  // lane j: j-th token of the window
  int t = -1;
  if (j < ras.win) t = c < ras.win ? ras.recent[(size_t)b * ras.win + c] : draft_tokens[b * gamma + c - ras.win];
  int cnt = 0;
  bool first = true;
  for (int i = 0; i < ras.win; ++i) {
    const bool same = __shfl_sync(0xffffffffu, t, i) == t;
    cnt += same;
    if (same && i < j) first = false;
  }
  sm.rep_ids[j] = j < ras.win && t >= 0 && t < V && first && (float)cnt >= ras.thresh ? t : -1;
}
__device__ __forceinline__ bool ras_is_rep(const SampSmem& sm, int win, int t) {
  bool rep = false;
  for (int j = 0; j < win; ++j) rep |= sm.rep_ids[j] == t;
  return rep;
}
// R of a row of signed_exp.
__device__ __forceinline__ float ras_mass(const float* v, const RowStats& st, int win, const SampSmem& sm) {
  float R = 0.f;
  for (int j = 0; j < win; ++j) {  // fixed order
    const int t = sm.rep_ids[j];
    if (t >= 0 && v[t] > 0.f) R += v[t] / st.sum;
  }
  return R;
}
// Its share of `sum`, 0 where it is cut off.  (A zero numerator would take the division's slow path, on most of a
// row under a top-k cut.)
__device__ __forceinline__ float kept_share(float v, float sum) {
  const float q = (v > 0.f ? v : 1.f) / sum;
  return v > 0.f ? q : 0.f;
}

// q(t) of the target's sampler from signed_exp: the (top-k, top-p) softmax, or the repetition-aware mixture.
__device__ __forceinline__ float q_value(float v, int t, const RowStats& st, int win, const RasRow& rr,
                                         const SampSmem& sm) {
  float q = kept_share(v, st.sum);
  if (win > 0) {
    if (q > 0.f && ras_is_rep(sm, win, t)) q = 0.f;
    q += rr.R * (fabsf(v) / rr.sum_full);
  }
  return q;
}

// A row's token and flag; the last row of a stream to arrive finds the first rejection and that row's token.
// One warp; lane 0's y and flag count.
__device__ __forceinline__ void finish_row(int y, bool flag, int b, int r, int R, int32_t* row_words, int32_t* counters,
                                           int32_t* accepted_len, int32_t* next_token) {
  const int lane = threadIdx.x & 31;
  int prev = 0;
  if (lane == 0) {
    row_words[b * R + r] = y * 2 + (int)flag;
    __threadfence();
    prev = atomicAdd(&counters[b], 1);
  }
  if (__shfl_sync(0xffffffffu, prev, 0) != R - 1) return;
  __threadfence();
  const int w = lane < R ? __ldcg(&row_words[b * R + lane]) : 1;  // R is at most 16
  const uint32_t rejected = __ballot_sync(0xffffffffu, lane < R - 1 && !(w & 1));
  const int k = rejected ? __ffs(rejected) - 1 : R - 1;
  if (lane == k) {
    counters[b] = 0;
    accepted_len[b] = k;
    next_token[b] = w >> 1;
  }
}

// Grid (R, B), R = gamma + 1.
__global__ void __launch_bounds__(SAMP_THREADS)
verify_sampler_kernel(const float* __restrict__ logits, int V,
                      const int32_t* __restrict__ draft_tokens,
                      const float* __restrict__ draft_probs, const float* __restrict__ uniforms,
                      int gamma, float inv_t, int top_k, float top_p, float beta, Ras ras,
                      int32_t* row_words, int32_t* counters, int32_t* __restrict__ accepted_len,
                      int32_t* __restrict__ next_token, int32_t* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SampSmem& sm = *reinterpret_cast<SampSmem*>(smem_raw);
  float* z = reinterpret_cast<float*>(smem_raw + sizeof(SampSmem));
  const int tid = threadIdx.x, r = blockIdx.x, b = blockIdx.y, R = gamma + 1;
  const float* prow = r < gamma ? draft_probs + ((size_t)b * gamma + r) * V : nullptr;
  clear_bins(sm);
  if (prow)  // (a hint: whoever writes the row may still be at it)
    for (int t = tid * 32; t < V; t += SAMP_THREADS * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(prow + t));
  tc_pdl_enter();
  int x = 0;
  if (tid == 0 && prow) x = draft_tokens[b * gamma + r];
  const float2 u = make_float2(uniforms[((size_t)b * R + r) * 2], uniforms[((size_t)b * R + r) * 2 + 1]);
  if (ras.win > 0 && tid >= SAMP_THREADS - 32) ras_window(ras, draft_tokens, gamma, b, r, V, sm);
  const BinMap map = load_row(logits + ((size_t)b * R + r) * V, V, inv_t, z, sm, status);
  float px = 0.f;
  const bool x_ok = x >= 0 && x < V;
  if (tid == 0 && prow && x_ok) px = prow[x];
  RasRow rr{1.f, 0.f};
  const RowStats st = compute_row_stats(z, V, top_k, top_p, map, ras.win > 0, &rr.sum_full, sm);
  if (ras.win > 0) rr.R = ras_mass(z, st, ras.win, sm);
  int flag = 0;
  if (tid == 0 && prow) {  // Eq. 5: accept x_i iff r_i < min(1, q_i(x_i) / p_i(x_i)) + beta
    float qx = 0.f;
    bool valid = x_ok;  // a draft token or probability that cannot be one is rejected, never accepted
    if (!x_ok) {
      atomicOr(status, SSD_STATUS_BAD_TOKEN);
    } else {
      qx = q_value(z[x], x, st, ras.win, rr, sm);
      if (!(px >= 0.f) || !isfinite(px)) {
        atomicOr(status, SSD_STATUS_BAD_PROB);
        valid = false;
      }
    }
    const float ratio = px <= qx ? 1.f : qx / px;
    flag = valid && u.x < ratio + beta;
  }
  __syncthreads();  // the values above are read: z becomes the weights of the draw
  // Eq. 6: w = max(0, q_r - p_r), for the case that row r is the first to be rejected; the bonus row q_{gamma+1} otherwise
#pragma unroll 4
  for (int t = tid; t < V; t += SAMP_THREADS) {
    const float q = q_value(z[t], t, st, ras.win, rr, sm);
    z[t] = prow ? fmaxf(0.f, q - prow[t]) : q;
  }
  __syncthreads();
  double total;
  int y = block_inverse_cdf(z, V, u.y, sm, &total);
  if (y < 0) {  // residual has no mass (numerical corner): draw from q_r itself
    for (int t = tid; t < V; t += SAMP_THREADS)
      z[t] = q_value(signed_exp(logits[((size_t)b * R + r) * V + t] * inv_t, t, st, ras.win > 0), t, st, ras.win, rr, sm);
    __syncthreads();
    y = block_inverse_cdf(z, V, u.y, sm, &total);
    if (y < 0) y = 0;
  }
  if (tid < 32) finish_row(y, flag, b, r, R, row_words, counters, accepted_len, next_token);
}

// ---- plain rows (softmax over the whole vocabulary: no cut, no repetition window), split over a cluster
//
// One CTA per row is bound by that SM's instructions (6564 ids take 18 thousand cycles in all) while the
// rest of the chip is idle.  Eight CTAs take an eighth each and exchange three numbers - largest value, sum,
// mass of the draw - as remote stores that complete on the receivers' barriers; a cluster barrier with
// its fence would cost a thousand cycles each time.  Every CTA adds the contributions in rank order.
constexpr int PL_CLUSTER = 8, PL_THREADS = 256, PL_WARPS = PL_THREADS / 32;
enum { PL_MAX, PL_SUM, PL_MASS, PL_FLAG, PL_MASS2, PL_SLOTS };

struct PlainSmem {
  double slot[PL_SLOTS][PL_CLUSTER];  // what the CTAs of the cluster sent
  unsigned long long bar[3 + 1];      // of max; sum; mass and flag; mass of the second draw
  double red[PL_WARPS];
  double scan[PL_THREADS];
  float red_f[PL_WARPS];
  int y, abort;
};

__device__ __forceinline__ void plain_send(PlainSmem& sm, int what, int bar, double v) {  // lanes 0 .. PL_CLUSTER - 1 of warp 0
  const uint32_t to = threadIdx.x, me = tcx::cluster_rank();
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
               ::"r"(tcx::map_rank(tcx::smem_u32(&sm.slot[what][me]), to)), "l"(__double_as_longlong(v)),
                 "r"(tcx::map_rank(tcx::smem_u32(&sm.bar[bar]), to))
               : "memory");
}
// Sum over the CTA, valid in warp 0.
__device__ __forceinline__ double plain_block_sum(double v, PlainSmem& sm) {
  v = warp_sum_d(v);
  if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = v;
  __syncthreads();
  return warp_sum_d(threadIdx.x < PL_WARPS ? sm.red[threadIdx.x] : 0.0);
}

// The draw over the weights w[0..n) of the cluster's CTAs: each CTA's running sums, the masses exchanged, and the
// CTA in which u * total falls finds the id.  Returns its place in this CTA's slice, -1 in the other CTAs, -2
// in all of them where there is no mass.
__device__ int plain_draw(const float* w, int n, float u, int what, int bar, double flag, PlainSmem& sm) {
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, me = (int)tcx::cluster_rank();
  const int seg = (n + PL_THREADS - 1) / PL_THREADS, i0 = min(tid * seg, n), i1 = min(i0 + seg, n);
  double s = 0.0;
  for (int i = i0; i < i1; ++i) s += (double)w[i];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += v;
  }
  if (lane == 31) sm.red[wp] = s;
  if (tid == 0) sm.y = -1;
  __syncthreads();
  double ahead = 0.0, mass = 0.0;
#pragma unroll
  for (int i = 0; i < PL_WARPS; ++i) {
    if (i == wp) ahead = mass;
    mass += sm.red[i];
  }
  if (tid < PL_CLUSTER) {
    plain_send(sm, what, bar, mass);
    if (what == PL_MASS) plain_send(sm, PL_FLAG, bar, flag);
  }
  sm.scan[tid] = ahead + s;
  __syncthreads();
  tcx::mbar_wait(tcx::smem_u32(&sm.bar[bar]), 0u, &sm.abort);
  double total = 0.0, before = 0.0;
  int last = -1;  // last CTA with mass
  for (int i = 0; i < PL_CLUSTER; ++i) {
    if (i == me) before = total;
    if (sm.slot[what][i] > 0.0) last = i;
    total += sm.slot[what][i];
  }
  if (!(total > 0.0)) return -2;
  const double target = (double)u * total;
  int owner = -1;
  double run = 0.0;
  for (int i = 0; i < PL_CLUSTER; ++i) {
    run += sm.slot[what][i];
    if (owner < 0 && target < run) owner = i;
  }
  if (me != (owner < 0 ? last : owner)) return -1;
  const double excl = before + (tid == 0 ? 0.0 : sm.scan[tid - 1]), incl = before + sm.scan[tid];
  if (owner >= 0 && excl <= target && target < incl) {
    double r = excl;
    int y = -1;
    for (int i = i0; i < i1; ++i) {
      r += (double)w[i];
      if (w[i] > 0.f) {
        y = i;
        if (r > target) break;
      }
    }
    sm.y = y;
  }
  __syncthreads();
  if (sm.y < 0 && tid == 0) {  // u * total rounded up to this CTA's end: its last id with mass
    int i = n - 1;
    while (i > 0 && !(w[i] > 0.f)) --i;
    sm.y = i;
  }
  __syncthreads();
  return sm.y;
}

struct PlainArgs {
  const float* logits;
  size_t ld;  // from one row's logits to the next one's
  int V, R;   // rows per stream (drafting: 1)
  float inv_t;
  const float* uniforms;  // verify: [B, R, 2]; drafting: [B]
  // verify
  const int32_t* draft_tokens;
  const float* draft_probs;
  float beta;
  int32_t *row_words, *counters, *accepted_len, *next_token;
  // drafting
  int32_t* out_token;
  int tok_stride;
  float* out_prob;
  size_t prob_stride;
  int32_t *pending, *len;
  int add, cap;
  int32_t* status;
};

// Grid (R * PL_CLUSTER, B), clusters along x.
template <bool DRAFT>
__global__ void __launch_bounds__(PL_THREADS) plain_sampler_kernel(const __grid_constant__ PlainArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PlainSmem& sm = *reinterpret_cast<PlainSmem*>(smem_raw);
  float* z = reinterpret_cast<float*>(smem_raw + sizeof(PlainSmem));
  const int tid = threadIdx.x, lane = tid & 31, me = (int)tcx::cluster_rank();
  const int r = blockIdx.x / PL_CLUSTER, b = blockIdx.y, R = A.R, gamma = R - 1, V = A.V;
  const int per = (V + PL_CLUSTER - 1) / PL_CLUSTER, t0 = min(me * per, V), n = min(per, V - t0);
  const float* prow = !DRAFT && r < gamma ? A.draft_probs + ((size_t)b * gamma + r) * V : nullptr;
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) tcx::mbar_init(tcx::smem_u32(&sm.bar[i]), 1);
    sm.abort = 0;
    tcx::mbar_init_fence();
    for (int i = 0; i < 4; ++i) tcx::mbar_expect_tx(tcx::smem_u32(&sm.bar[i]), (i == 2 ? 16u : 8u) * PL_CLUSTER);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (prow)  // (a hint: whoever writes the row may still be at it)
    for (int i = tid * 32; i < n; i += PL_THREADS * 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(prow + t0 + i));
  tc_pdl_enter();
  int x = -1;
  if (!DRAFT && tid == 0 && prow) x = A.draft_tokens[b * gamma + r];
  const float u = DRAFT ? A.uniforms[b] : A.uniforms[((size_t)b * R + r) * 2 + 1];
  const float ur = DRAFT ? 0.f : A.uniforms[((size_t)b * R + r) * 2];
  const float* lrow = A.logits + (size_t)(b * R + r) * A.ld + t0;
  float mx = -CUDART_INF_F;
  int bad = 0;
#pragma unroll 4
  for (int i = tid; i < n; i += PL_THREADS) {
    const float v = lrow[i];
    if (!isfinite(v)) bad = 1;
    z[i] = v * A.inv_t;
    mx = fmaxf(mx, z[i]);
  }
  float px = 0.f;
  if (!DRAFT && prow && x >= t0 && x < t0 + n) px = prow[x];
  mx = warp_max(mx);
  if (lane == 0) sm.red_f[tid >> 5] = mx;
  bad = __syncthreads_or(bad);
  if (bad && tid == 0) atomicOr(A.status, SSD_STATUS_NONFINITE);
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // the other CTAs' barriers exist
  if (tid < 32) {
    mx = warp_max(lane < PL_WARPS ? sm.red_f[lane] : -CUDART_INF_F);
    if (lane < PL_CLUSTER) plain_send(sm, PL_MAX, 0, (double)mx);
  }
  tcx::mbar_wait(tcx::smem_u32(&sm.bar[0]), 0u, &sm.abort);
  float zmax = (float)sm.slot[PL_MAX][0];
#pragma unroll
  for (int i = 1; i < PL_CLUSTER; ++i) zmax = fmaxf(zmax, (float)sm.slot[PL_MAX][i]);
  double s = 0.0;
#pragma unroll 2
  for (int i = tid; i < n; i += PL_THREADS) {
    const float e = expf(z[i] - zmax);
    z[i] = e;
    s += (double)e;
  }
  s = plain_block_sum(s, sm);
  if (tid < PL_CLUSTER) plain_send(sm, PL_SUM, 1, s);
  tcx::mbar_wait(tcx::smem_u32(&sm.bar[1]), 0u, &sm.abort);
  s = 0.0;
#pragma unroll
  for (int i = 0; i < PL_CLUSTER; ++i) s += sm.slot[PL_SUM][i];
  const float sum = (float)s;
  int flag = 0;
  if (!DRAFT && prow && tid == 0) {  // Eq. 5: accept x_i iff r_i < min(1, q_i(x_i) / p_i(x_i)) + beta
    // a draft token or probability that cannot be one is rejected, never accepted
    if (x < 0 || x >= V) {
      if (me == 0) atomicOr(A.status, SSD_STATUS_BAD_TOKEN);
    } else if (x >= t0 && x < t0 + n) {
      if (!(px >= 0.f) || !isfinite(px)) {
        atomicOr(A.status, SSD_STATUS_BAD_PROB);
      } else {
        const float qx = z[x - t0] / sum, ratio = px <= qx ? 1.f : qx / px;
        flag = ur < ratio + A.beta;
      }
    }
  }
  flag = __syncthreads_or(flag);  // and the value above is read: z becomes the weights of the draw
#pragma unroll 4
  for (int i = tid; i < n; i += PL_THREADS) {
    const float q = z[i] / sum;
    if (DRAFT) A.out_prob[(size_t)b * A.prob_stride + t0 + i] = q;
    z[i] = prow ? fmaxf(0.f, q - prow[t0 + i]) : q;
  }
  __syncthreads();
  int y = plain_draw(z, n, u, PL_MASS, 2, (double)flag, sm);
  if (!DRAFT && y == -2) {  // residual has no mass (numerical corner): draw from q_r itself
    __syncthreads();
    for (int i = tid; i < n; i += PL_THREADS) z[i] = expf(lrow[i] * A.inv_t - zmax) / sum;
    __syncthreads();
    y = plain_draw(z, n, u, PL_MASS2, 3, 0.0, sm);
  }
  if (y == -2 && me == 0) y = 0;
  if (tid == 0 && sm.abort) atomicOr(A.status, SSD_STATUS_TIMEOUT);
  if (y < 0 || tid >= 32) return;
  y += t0;
  if (DRAFT) {
    if (tid == 0) {
      A.out_token[(size_t)b * A.tok_stride] = y;
      A.pending[b] = y;
      const int nl = A.len[b] + A.add;  // the rows of the forward are committed
      if (nl > A.cap) atomicOr(A.status, SSD_STATUS_KV_OVERFLOW);
      A.len[b] = min(nl, A.cap);
    }
    return;
  }
  double f = 0.0;
  for (int i = 0; i < PL_CLUSTER; ++i) f += sm.slot[PL_FLAG][i];
  finish_row(y, f > 0.0, b, r, R, A.row_words, A.counters, A.accepted_len, A.next_token);
}

// Plain rows take the cluster kernel while its CTAs leave most of an SM to each other: 5 rows 14.3 -> 11.7 us,
// 24 rows 14.4 -> 12.3, 96 rows the same.
bool plain_rows(int rows, int V, int top_k, float top_p, int ras_window) {
  return !(top_k > 0 && top_k < V) && !(top_p > 0.f && top_p < 1.f) && ras_window <= 0 && rows <= 64;
}
template <bool DRAFT>
cudaError_t launch_plain(const PlainArgs& a, int B, cudaStream_t st) {
  const size_t smem = sizeof(PlainSmem) + (size_t)((a.V + PL_CLUSTER - 1) / PL_CLUSTER) * sizeof(float);
  const cudaError_t e = tc_launch_pdl_cluster(plain_sampler_kernel<DRAFT>, dim3(a.R * PL_CLUSTER, B), dim3(PL_THREADS),
                                              PL_CLUSTER, smem, st, a);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_verify_sampler(const float* logits, int V, const int32_t* draft_tokens,
                                  const float* draft_probs, const float* uniforms, int B,
                                  int gamma, float inv_temperature, int top_k, float top_p, float beta,
                                  int ras_window, float ras_tau, const int32_t* recent_tokens,
                                  int32_t* row_words, int32_t* counters,
                                  int32_t* accepted_len, int32_t* next_token, int32_t* status,
                                  cudaStream_t st) {
  Ras ras{0, 0.f, nullptr};
  if (ras_window > 0) {
    if (ras_window > RAS_MAX_WIN || !recent_tokens) return cudaErrorInvalidValue;
    ras = Ras{ras_window, (float)ras_window * ras_tau, recent_tokens};
  }
  if (plain_rows(B * (gamma + 1), V, top_k, top_p, ras_window)) {
    PlainArgs a{};
    a.logits = logits;
    a.ld = (size_t)V;
    a.V = V;
    a.R = gamma + 1;
    a.inv_t = inv_temperature;
    a.uniforms = uniforms;
    a.draft_tokens = draft_tokens;
    a.draft_probs = draft_probs;
    a.beta = beta;
    a.row_words = row_words;
    a.counters = counters;
    a.accepted_len = accepted_len;
    a.next_token = next_token;
    a.status = status;
    return launch_plain<false>(a, B, st);
  }
  size_t smem = sizeof(SampSmem) + (size_t)V * sizeof(float);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(verify_sampler_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  dim3 grid(gamma + 1, B);
  tc_launch_pdl(verify_sampler_kernel, grid, dim3(SAMP_THREADS), smem, st, logits, V, draft_tokens, draft_probs,
                uniforms, gamma, inv_temperature, top_k, top_p, beta, ras, row_words, counters,
                accepted_len, next_token, status);
  count_launch();
  return cudaGetLastError();
}

// Draft side (Eq. 2-3): p = transform(logits row), x ~ p by inverse CDF; p is written out in full
// because the verifier needs the whole row (Eq. 6).  One CTA per stream.
__global__ void __launch_bounds__(SAMP_THREADS)
draft_sampler_kernel(const float* __restrict__ logits, int ld_logits, int V,
                     const float* __restrict__ uniform, float inv_t, int top_k, float top_p,
                     int32_t* __restrict__ out_token, int tok_stride, float* __restrict__ out_prob,
                     size_t prob_stride, int32_t* pending, int32_t* len, int add, int cap, int32_t* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SampSmem& sm = *reinterpret_cast<SampSmem*>(smem_raw);
  float* z = reinterpret_cast<float*>(smem_raw + sizeof(SampSmem));
  const int b = blockIdx.x;
  clear_bins(sm);
  tc_pdl_enter();
  const float u = uniform[b];
  const BinMap map = load_row(logits + (size_t)b * ld_logits, V, inv_t, z, sm, status);
  float sum_full;
  const RowStats st = compute_row_stats(z, V, top_k, top_p, map, false, &sum_full, sm);
#pragma unroll 4
  for (int t = threadIdx.x; t < V; t += SAMP_THREADS) {  // each thread's own elements of z: no barrier before
    const float p = kept_share(z[t], st.sum);
    z[t] = p;
    out_prob[(size_t)b * prob_stride + t] = p;
  }
  __syncthreads();
  double total;
  int y = block_inverse_cdf(z, V, u, sm, &total);
  if (y < 0) y = 0;
  if (threadIdx.x == 0) {
    out_token[(size_t)b * tok_stride] = y;
    pending[b] = y;
    const int nl = len[b] + add;  // the rows of the forward are committed
    if (nl > cap) atomicOr(status, SSD_STATUS_KV_OVERFLOW);
    len[b] = min(nl, cap);
  }
}

cudaError_t launch_draft_sampler(const float* logits, int ld_logits, int V, const float* uniform,
                                 int B, float inv_temperature, int top_k, float top_p,
                                 int32_t* out_token, int tok_stride, float* out_prob_row,
                                 size_t prob_stride, int32_t* pending, int32_t* len, int add, int cap,
                                 int32_t* status, cudaStream_t st) {
  if (plain_rows(B, V, top_k, top_p, 0)) {
    PlainArgs a{};
    a.logits = logits;
    a.ld = (size_t)ld_logits;
    a.V = V;
    a.R = 1;
    a.inv_t = inv_temperature;
    a.uniforms = uniform;
    a.out_token = out_token;
    a.tok_stride = tok_stride;
    a.out_prob = out_prob_row;
    a.prob_stride = prob_stride;
    a.pending = pending;
    a.len = len;
    a.add = add;
    a.cap = cap;
    a.status = status;
    return launch_plain<true>(a, B, st);
  }
  size_t smem = sizeof(SampSmem) + (size_t)V * sizeof(float);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(draft_sampler_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  tc_launch_pdl(draft_sampler_kernel, dim3(B), dim3(SAMP_THREADS), smem, st, logits, ld_logits, V, uniform,
                inv_temperature, top_k, top_p, out_token, tok_stride, out_prob_row, prob_stride, pending, len, add,
                cap, status);
  count_launch();
  return cudaGetLastError();
}

// "Append to T_in" (Algorithm 1): the prefix grows by the k accepted tokens plus the new one.
__global__ void kv_commit_kernel(int32_t* len, int32_t* pending, const int32_t* accepted_len,
                                 const int32_t* next_token, int B, int cap, int max_gamma,
                                 int32_t* status, int32_t* host_out) {
  tc_pdl_enter();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int k = accepted_len[b], y = next_token[b];
  if (host_out) {
    host_out[b] = k;
    host_out[B + b] = y;
  }
  if (k < 0 || k > max_gamma) {  // not an accepted length: the stream stays as it is
    atomicOr(status, SSD_STATUS_BAD_TOKEN);
    return;
  }
  int nl = max(len[b], 0) + 1 + k;
  if (nl > cap) {
    atomicOr(status, SSD_STATUS_KV_OVERFLOW);
    nl = cap;
  }
  len[b] = nl;
  pending[b] = y;
}

void launch_kv_commit(int32_t* len, int32_t* pending, const int32_t* accepted_len, const int32_t* next_token, int B, int cap,
                      int max_gamma, int32_t* status, cudaStream_t st, int32_t* host_out) {
  tc_launch_pdl(kv_commit_kernel, dim3((B + 127) / 128), dim3(128), 0, st, len, pending, accepted_len, next_token, B,
                cap, max_gamma, status, host_out);
  count_launch();
}

}  // namespace ssd

// ------------------------------------------------------------------------------------------------
// Acceptance step for callers that cannot allocate device memory.
//
// Some hosts of this library may not call cudaMalloc at all: code that runs inside a serving loop
// whose memory pool is fixed at start-up, or a plug-in that is handed device pointers by its host
// process and owns none.  ssd_verify needs a workspace such callers cannot provide.  This entry
// point runs the same fused acceptance kernel on logits the caller already has, and keeps the
// kernel's scratch (one word per row, one counter per stream, one status word) in the fixed device array below instead.
namespace {

constexpr int NOALLOC_MAX_STREAMS = 256;  // streams per call
constexpr int NOALLOC_MAX_ROWS = ssd::R_MAX;  // gamma + 1 <= 16

struct NoAllocScratch {
  int32_t row_words[NOALLOC_MAX_STREAMS * NOALLOC_MAX_ROWS];
  int32_t counters[NOALLOC_MAX_STREAMS];
  int32_t status;
};

// About 17 KB, resident on every GPU that loads the library until the process exits.  In host
// code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
NoAllocScratch* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of the scratch array on the current device (looked up once per device).
cudaError_t noalloc_scratch(NoAllocScratch** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = static_cast<NoAllocScratch*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" int ssd_accept_noalloc(const float* dev_logits, const int32_t* dev_draft_tokens,
                                  const float* dev_draft_probs, const float* dev_uniforms,
                                  const ssd_verify_params* params, int32_t batch, int32_t vocab,
                                  int32_t* dev_accepted_len, int32_t* dev_next_token,
                                  void* stream) {
  if (!dev_logits || !dev_draft_tokens || !dev_draft_probs || !dev_uniforms || !params ||
      !dev_accepted_len || !dev_next_token)
    return SSD_ERR_NULL;
  if (params->gamma < 1 || params->gamma + 1 > NOALLOC_MAX_ROWS) return SSD_ERR_BAD_GAMMA;
  if (batch < 1 || batch > NOALLOC_MAX_STREAMS) return SSD_ERR_TOO_SMALL;  // beyond the fixed scratch
  if (vocab < 2 || (size_t)vocab * 4 > 180 * 1024) return SSD_ERR_BAD_CONFIG;
  if (!(params->temperature > 0.f) || !isfinite(params->temperature) || !(params->beta >= 0.f) ||
      !isfinite(params->beta))
    return SSD_ERR_BAD_PARAM;
  NoAllocScratch* sc = nullptr;
  cudaError_t e = noalloc_scratch(&sc);
  if (e != cudaSuccess) return ssd::report_cuda_error(e, "ssd_accept_noalloc: cudaGetSymbolAddress");
  cudaStream_t st = (cudaStream_t)stream;
  // the per-stream counters must start at zero; everything else is overwritten before it is read
  e = cudaMemsetAsync(sc->counters, 0, sizeof(int32_t) * (NOALLOC_MAX_STREAMS + 1), st);
  if (e != cudaSuccess) return ssd::report_cuda_error(e, "ssd_accept_noalloc: cudaMemsetAsync");
  e = ssd::launch_verify_sampler(dev_logits, vocab, dev_draft_tokens, dev_draft_probs, dev_uniforms,
                                 batch, params->gamma, 1.0f / params->temperature, params->top_k,
                                 params->top_p, params->beta, params->ras_window, params->ras_tau,
                                 params->dev_recent_tokens, sc->row_words, sc->counters,
                                 dev_accepted_len, dev_next_token, &sc->status, st);
  if (e != cudaSuccess) return ssd::report_cuda_error(e, "ssd_accept_noalloc: launch");
  return SSD_OK;
}
