// Verify attention of a forward of at most TC_CHAIN_ROWS rows (tc_chain.cu), one launch: the key splits
// of a stream's kv head are the CTAs of a cluster, and merge through distributed shared memory.
//
// Grid (split, kv head x row group, stream), clusters of S <= 8 along the splits.  A CTA takes up to 64
// of the G * R query rows that share the kv head and every tile of 64 keys of its range; the ranges
// follow the stream's own length.  Eight warps: four slabs of 16 rows x two halves of a tile's keys, so
// that a tile costs a warp 64 instructions instead of 128 (the warp-level tensor instruction is what a
// tile waits for).  Arithmetic as in tc_attn_kernel (tc_attention.cu): q and the softmax weights as bf16
// leading part + remainder, running max and sum in registers.
//
// What bounds it: latency.  So the tiles of the cached prefix, which the projection before this kernel
// does not touch, are requested before the dependency wait, three stages deep; and the partial
// results (two halves per CTA) go to the CTA that owns their rows by bulk copies that complete on its
// barrier, instead of through memory to a merge kernel (one launch, one round trip and 6 us less).
#include <math_constants.h>

#include <algorithm>

#include "kernels.h"
#include "tc.h"
#include "tc_ptx.cuh"

namespace ssd {

namespace {

using namespace tcx;

constexpr int AC_THREADS = 256;
constexpr int AC_TILE = 64;
static_assert(AC_TILE == TC_PAGE_TOKENS, "a key tile is one page of a paged cache");

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

template <int HD>
struct AcLay {
  static constexpr int ROWB = HD * 2 + 16;             // padded K / V row: conflict-free matrix loads
  static constexpr int STAGE = 2 * AC_TILE * ROWB;     // K tile, V tile
  static constexpr int STAGES = HD == 128 ? 2 : 3;
  static constexpr int Q_BYTES = 4 * (HD / 16) * 32 * 32;
  static constexpr int PW = HD + 4;                    // floats of a row's partial: output, max, sum, padding
  static constexpr int PART = 2 * 70 * PW * 4;         // two halves x 64 rows, rounded up to the owners' shares
  static constexpr int OFF_Q = STAGES * STAGE > PART ? STAGES * STAGE : PART;  // the outgoing partials take the tiles' place
  static constexpr int OFF_G = OFF_Q + Q_BYTES;
  static constexpr int OFF_B = OFF_G + PART, TOTAL = OFF_B + 32;
};

template <int HD>
__global__ void __launch_bounds__(AC_THREADS, HD == 128 ? 1 : 2)
tc_attn_chain_kernel(const float* __restrict__ qrot, const bf16* __restrict__ kv_layer, const int32_t* __restrict__ len,
                     RowMap rm, int cap, int Hq, int Hkv, int n_rowgroups, const int32_t* __restrict__ page_table,
                     int max_pages, uint8_t* __restrict__ apack, ActLay lay, int32_t* status) {
  using Lay = AcLay<HD>;
  constexpr int ROWB = Lay::ROWB, KSTEPS = HD / 16, DT = HD / 8, CH = HD / 8, PW = Lay::PW;
  extern __shared__ __align__(128) uint8_t smem[];
  uint4* q_s = reinterpret_cast<uint4*>(smem + Lay::OFF_Q);   // [slab][kstep][lane][hi 4 words | lo 4 words]
  float* push = reinterpret_cast<float*>(smem);               // [owner][half][row of the owner][PW]
  float* gath = reinterpret_cast<float*>(smem + Lay::OFF_G);  // [source][half][row of this CTA][PW]
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem + Lay::OFF_B);
  int* abort_word = reinterpret_cast<int*>(bar + 1);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int S = (int)gridDim.x, rank = (int)blockIdx.x;  // a cluster is one row of the grid
  const int gk = blockIdx.y / n_rowgroups, rg = blockIdx.y % n_rowgroups, bi = blockIdx.z;
  const int b = rm.b0 + bi, R = rm.R, G = Hq / Hkv, NQ = G * R;
  if (tid == 0) {
    mbar_init(smem_u32(bar), 1);
    *abort_word = 0;
    mbar_init_fence();
  }
  __syncthreads();
  if (S > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  tc_pdl_trigger();

  // Lengths and the cached prefix were complete before the chain of dependent launches began.
  const int L = __ldcg(len + b), total = min(L + R, cap);
  const int tiles = (total + AC_TILE - 1) / AC_TILE, per = (tiles + S - 1) / S;
  const int k_begin = rank * per * AC_TILE, k_end = min(k_begin + per * AC_TILE, total);
  const int n_tiles = k_end > k_begin ? (k_end - k_begin + AC_TILE - 1) / AC_TILE : 0;
  const bf16* kbase = kv_layer + (((size_t)b * 2 + 0) * Hkv + gk) * (size_t)cap * HD;
  const bf16* vbase = kv_layer + (((size_t)b * 2 + 1) * Hkv + gk) * (size_t)cap * HD;
  bool waited = false;
  auto stage_tile = [&](int it) {
    const int key0 = k_begin + it * AC_TILE;
    if (!waited && key0 + AC_TILE > L) {  // rows that the projection before this kernel appends
      tc_pdl_wait();
      waited = true;
    }
    uint8_t* ks = smem + (size_t)(it % Lay::STAGES) * Lay::STAGE;
    const bf16 *kt = kbase, *vt = vbase;
    int first = 0;
    if (page_table) {  // a tile is one page
      const int pg = max(__ldcg(page_table + (size_t)b * max_pages + key0 / TC_PAGE_TOKENS), 0);
      kt = kv_layer + (((size_t)pg * 2 + 0) * Hkv + gk) * (size_t)TC_PAGE_TOKENS * HD;
      vt = kv_layer + (((size_t)pg * 2 + 1) * Hkv + gk) * (size_t)TC_PAGE_TOKENS * HD;
      first = key0;
    }
#pragma unroll
    for (int i = 0; i < AC_TILE * CH / AC_THREADS; ++i) {
      const int idx = tid + i * AC_THREADS, key = idx / CH, c = idx % CH;
      // keys past the range repeat the last valid one: finite data, masked out below
      const size_t src = (size_t)(min(key0 + key, k_end - 1) - first) * HD + c * 8;
      cp_async16(smem_u32(ks + key * ROWB + c * 16), kt + src);
      cp_async16(smem_u32(ks + AC_TILE * ROWB + key * ROWB + c * 16), vt + src);
    }
  };
#pragma unroll
  for (int it = 0; it < Lay::STAGES - 1; ++it) {
    if (it < n_tiles) stage_tile(it);
    cp_async_commit();
  }
  if (!waited) tc_pdl_wait();
  waited = true;

  const int slab = warp & 3, kh = warp >> 2;
  const int i0 = rg * 64 + slab * 16 + g, i1 = i0 + 8;
  const bool active = rg * 64 + slab * 16 < NQ, ok0 = i0 < NQ, ok1 = i1 < NQ;
  const int r0 = ok0 ? i0 % R : 0, r1 = ok1 ? i1 % R : 0;
  // q as A fragments: the warps of a slab share the work
  for (int s = kh; s < KSTEPS; s += 2) {
    const float* q0 = qrot + ((size_t)(bi * R + r0) * Hq + gk * G + (ok0 ? i0 / R : 0)) * HD + s * 16 + 2 * t;
    const float* q1 = qrot + ((size_t)(bi * R + r1) * Hq + gk * G + (ok1 ? i1 / R : 0)) * HD + s * 16 + 2 * t;
    float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0, a3 = a0;
    if (ok0) {
      a0 = __ldcg(reinterpret_cast<const float2*>(q0));
      a2 = __ldcg(reinterpret_cast<const float2*>(q0 + 8));
    }
    if (ok1) {
      a1 = __ldcg(reinterpret_cast<const float2*>(q1));
      a3 = __ldcg(reinterpret_cast<const float2*>(q1 + 8));
    }
    uint4 hi, lo;
    split2(a0.x, a0.y, hi.x, lo.x);
    split2(a1.x, a1.y, hi.y, lo.y);
    split2(a2.x, a2.y, hi.z, lo.z);
    split2(a3.x, a3.y, hi.w, lo.w);
    uint4* dst = q_s + ((size_t)(slab * KSTEPS + s) * 32 + lane) * 2;
    dst[0] = hi;
    dst[1] = lo;
  }

  float m_run[2] = {-CUDART_INF_F, -CUDART_INF_F}, l_run[2] = {0.f, 0.f};
  float o[DT][4];
#pragma unroll
  for (int dt = 0; dt < DT; ++dt) o[dt][0] = o[dt][1] = o[dt][2] = o[dt][3] = 0.f;
  const int lim0 = L + r0, lim1 = L + r1;  // last visible key of the two rows

  for (int it = 0; it < n_tiles; ++it) {
    const int key0 = k_begin + it * AC_TILE + kh * 32;
    cp_async_wait<Lay::STAGES - 2>();
    __syncthreads();  // this tile has landed for everybody, and nobody reads the one before it any more
    if (it + Lay::STAGES - 1 < n_tiles) stage_tile(it + Lay::STAGES - 1);
    cp_async_commit();
    if (active) {
      const uint8_t* ks = smem + (size_t)(it % Lay::STAGES) * Lay::STAGE + kh * 32 * ROWB;
      const uint32_t k_addr = smem_u32(ks) + ((lane >> 4) * 8 + (lane & 7)) * ROWB + ((lane >> 3) & 1) * 16;
      const uint32_t v_addr = smem_u32(ks + AC_TILE * ROWB) + (((lane >> 3) & 1) * 8 + (lane & 7)) * ROWB + (lane >> 4) * 16;
      float sc[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
      for (int s = 0; s < KSTEPS; ++s) {
        const uint4* qa = q_s + ((size_t)(slab * KSTEPS + s) * 32 + lane) * 2;
        const uint4 hi = qa[0], lo = qa[1];
        const uint32_t ahi[4] = {hi.x, hi.y, hi.z, hi.w}, alo[4] = {lo.x, lo.y, lo.z, lo.w};
        uint32_t b0[4], b1[4];
        ldmatrix_x4(k_addr + s * 32, b0[0], b0[1], b0[2], b0[3]);
        ldmatrix_x4(k_addr + 16 * ROWB + s * 32, b1[0], b1[1], b1[2], b1[3]);
        mma_bf16(sc[0], ahi, b0[0], b0[1]);  // four accumulators in turn
        mma_bf16(sc[1], ahi, b0[2], b0[3]);
        mma_bf16(sc[2], ahi, b1[0], b1[1]);
        mma_bf16(sc[3], ahi, b1[2], b1[3]);
        mma_bf16(sc[0], alo, b0[0], b0[1]);
        mma_bf16(sc[1], alo, b0[2], b0[3]);
        mma_bf16(sc[2], alo, b1[0], b1[1]);
        mma_bf16(sc[3], alo, b1[2], b1[3]);
      }
      const bool whole = __all_sync(0xffffffffu, key0 + 31 < k_end && (!ok0 || key0 + 31 <= lim0) && (!ok1 || key0 + 31 <= lim1));
      if (!whole) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int key = key0 + nt * 8 + 2 * t + e;
            if (!(ok0 && key < k_end && key <= lim0)) sc[nt][e] = -CUDART_INF_F;
            if (!(ok1 && key < k_end && key <= lim1)) sc[nt][2 + e] = -CUDART_INF_F;
          }
        }
      }
      float corr[2], mn[2];
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        float mt = -CUDART_INF_F;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mt = fmaxf(mt, fmaxf(sc[nt][2 * hh], sc[nt][2 * hh + 1]));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 1));
        mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, 2));
        mn[hh] = fmaxf(m_run[hh], mt);
        corr[hh] = mn[hh] == -CUDART_INF_F ? 1.f : __expf(m_run[hh] - mn[hh]);
        m_run[hh] = mn[hh];
        l_run[hh] *= corr[hh];
        if (mn[hh] == -CUDART_INF_F) mn[hh] = 0.f;  // nothing visible yet: exp(-inf - 0) = 0
      }
#pragma unroll
      for (int dt = 0; dt < DT; ++dt) {
        o[dt][0] *= corr[0];
        o[dt][1] *= corr[0];
        o[dt][2] *= corr[1];
        o[dt][3] *= corr[1];
      }
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sc[nt][e] = __expf(sc[nt][e] - mn[e >> 1]);
          l_run[e >> 1] += sc[nt][e];
        }
      }
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        uint32_t phi[4], plo[4];
        split2(sc[2 * kk][0], sc[2 * kk][1], phi[0], plo[0]);
        split2(sc[2 * kk][2], sc[2 * kk][3], phi[1], plo[1]);
        split2(sc[2 * kk + 1][0], sc[2 * kk + 1][1], phi[2], plo[2]);
        split2(sc[2 * kk + 1][2], sc[2 * kk + 1][3], phi[3], plo[3]);
#pragma unroll
        for (int dt = 0; dt < DT; dt += 2) {
          uint32_t b0, b1, b2, b3;
          ldmatrix_x4_trans(v_addr + kk * 16 * ROWB + dt * 16, b0, b1, b2, b3);
          mma_bf16(o[dt], phi, b0, b1);
          mma_bf16(o[dt + 1], phi, b2, b3);
          mma_bf16(o[dt], plo, b0, b1);
          mma_bf16(o[dt + 1], plo, b2, b3);
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();  // the tiles are dead: their place takes the outgoing partials

  // ---- partials to the CTAs that own their rows (RPO rows each)
  const int RPO = (64 + S - 1) / S, block = 2 * RPO * PW;
  if (active) {
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      float l = l_run[hh];
      l += __shfl_xor_sync(0xffffffffu, l, 1);
      l += __shfl_xor_sync(0xffffffffu, l, 2);
      const int i = slab * 16 + g + 8 * hh, own = i / RPO;
      float* dst = (S > 1 ? push : gath) + (size_t)own * block + (size_t)(kh * RPO + i - own * RPO) * PW;
#pragma unroll
      for (int dt = 0; dt < DT; ++dt) *reinterpret_cast<float2*>(dst + dt * 8 + 2 * t) = make_float2(o[dt][2 * hh], o[dt][2 * hh + 1]);
      if (t == 0) *reinterpret_cast<float2*>(dst + HD) = make_float2(m_run[hh], l);
    }
  }
  if (S > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (S > 1) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every CTA has started: its barrier exists
    if (warp == 0 && elect_one()) {
      mbar_expect_tx(smem_u32(bar), (uint32_t)(S * block) * 4u);
      for (int i = 0; i < S; ++i) {
        const uint32_t to = (uint32_t)(rank + i < S ? rank + i : rank + i - S);
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(map_rank(smem_u32(gath) + (uint32_t)(rank * block) * 4u, to)),
                     "r"(smem_u32(push) + to * (uint32_t)block * 4u), "r"((uint32_t)block * 4u), "r"(map_rank(smem_u32(bar), to))
                     : "memory");
      }
    }
    __syncwarp();
    mbar_wait(smem_u32(bar), 0u, abort_word);
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }

  // ---- merge, one warp per row: lane p holds the statistics of partial p (source p / 2, half p % 2)
  const int np = 2 * S;
  for (int rl = warp; rl < RPO; rl += AC_THREADS / 32) {
    const int i = rg * 64 + rank * RPO + rl;
    if (rank * RPO + rl >= 64 || i >= NQ) break;
    const float* base = gath + (size_t)rl * PW;
    float pm = -CUDART_INF_F, pl = 0.f;
    if (lane < np) {
      const float2 ml = *reinterpret_cast<const float2*>(base + (size_t)lane * RPO * PW + HD);
      pm = ml.x;
      pl = ml.y;
    }
    const float m_tot = warp_max(pm), e = pm == -CUDART_INF_F ? 0.f : __expf(pm - m_tot), inv = 1.f / warp_sum(e * pl);
    const int hl = i / R, row = bi * R + (i - hl * R), k0 = (gk * G + hl) * HD;
    uint8_t* arow = lay.row(apack, row);
#pragma unroll
    for (int c = 0; c < (HD + 63) / 64; ++c) {
      const int d = c * 64 + lane * 2;
      float2 acc = make_float2(0.f, 0.f), v[16];
#pragma unroll
      for (int p = 0; p < 16; ++p)  // all loads in flight
        v[p] = p < np && d < HD ? *reinterpret_cast<const float2*>(base + (size_t)p * RPO * PW + d) : make_float2(0.f, 0.f);
#pragma unroll
      for (int p = 0; p < 16; ++p) {  // fixed order; absent partials weigh nothing
        const float w = __shfl_sync(0xffffffffu, e, p);
        acc.x = fmaf(w, v[p].x, acc.x);
        acc.y = fmaf(w, v[p].y, acc.y);
      }
      if (d < HD) {
        uint32_t hi, lo;
        split2(acc.x * inv, acc.y * inv, hi, lo);
        uint8_t* dst = arow + lay.col(k0 + d);
        *reinterpret_cast<uint32_t*>(dst) = hi;
        *reinterpret_cast<uint32_t*>(dst + lay.part_off) = lo;
      }
    }
  }
  if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // nobody reads this CTA's memory any more
  if (tid == 0 && *abort_word) atomicOr(status, SSD_STATUS_TIMEOUT);
}

template <int HD>
cudaError_t launch_t(const float* qrot, const bf16* kv_layer, const int32_t* len, RowMap rm, int cap, int Hq, int Hkv,
                     int n_sm, const int32_t* page_table, int max_pages, uint8_t* apack, ActLay lay, int32_t* status,
                     cudaStream_t st) {
  const int rowgroups = ((Hq / Hkv) * rm.R + 63) / 64, items = rm.nb * Hkv * rowgroups;
  // splits: no more than there are tiles, and as many CTAs as fit the SMs at once with a margin - the CTAs of
  // a cluster need SMs of one GPC, and 32 clusters of 8 at two CTAs per SM left one for a second wave
  // (17.6 us; 32 clusters of 7 do not)
  const int room = (HD == 128 ? 3 : 6) * n_sm / 4 / items;
  const int S = std::max(1, std::min(std::min(8, room), (cap + AC_TILE - 1) / AC_TILE));
  cudaError_t e = cudaFuncSetAttribute(tc_attn_chain_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, AcLay<HD>::TOTAL);
  if (e != cudaSuccess) return e;
  e = tc_launch_pdl_cluster(tc_attn_chain_kernel<HD>, dim3(S, Hkv * rowgroups, rm.nb), dim3(AC_THREADS), S,
                            (size_t)AcLay<HD>::TOTAL, st, qrot, kv_layer, len, rm, cap, Hq, Hkv, rowgroups, page_table,
                            max_pages, apack, lay, status);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tc_attention_chain(const float* qrot, const bf16* kv_layer, const int32_t* len, RowMap rm, int cap,
                                      int Hq, int Hkv, int hd, int n_sm, const int32_t* page_table, int max_pages,
                                      uint8_t* apack, ActLay lay, int32_t* status, cudaStream_t st) {
  switch (hd) {
    case 32: return launch_t<32>(qrot, kv_layer, len, rm, cap, Hq, Hkv, n_sm, page_table, max_pages, apack, lay, status, st);
    case 64: return launch_t<64>(qrot, kv_layer, len, rm, cap, Hq, Hkv, n_sm, page_table, max_pages, apack, lay, status, st);
    case 128: return launch_t<128>(qrot, kv_layer, len, rm, cap, Hq, Hkv, n_sm, page_table, max_pages, apack, lay, status, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ssd
