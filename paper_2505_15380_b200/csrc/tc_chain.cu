// Projections of a verify forward of at most TC_CHAIN_ROWS rows on tcgen05 tensor cores, with
// everything that sits between them in their epilogues: one launch per projection, no partial sums in
// global memory.
//
// A CTA owns a slab of up to 16 groups of 8 weight rows (the 128 lanes of the instruction's M; missing
// groups are lanes nobody reads).  Where K is short it takes all of K, and all token rows or half of
// them; where K is long (the down projection) the CTAs of a cluster split K, and each hands its sums
// of a token row to the CTA that owns the row by bulk copies through distributed shared memory.  Slabs are
// cut so that every SM streams the same number of weight bytes.  Both bf16 parts of the activations ride
// in one instruction (128 x 2 Mc x 16).  The epilogue adds the contributions in rank order
// (bit-reproducible) and finishes the rows:
//   QKV       x 1/rms of the row, + bias, rotary embedding, q to memory, K and V to the cache
//   residual  + h; the operand of the next projection (x times the next norm's gain, as bf16 leading
//             parts and remainders) and the slab's share of the row's sum of squares, from which the
//             consumer forms 1/rms: no norm kernel
//   SwiGLU    x 1/rms; SiLU(gate) up as the operand of the down projection
//   logits    x 1/rms
//
// What bounds it: latency - the dependency wait, one trip to L2, the instructions (97 cycles each at 96
// rows, 40 at 16), the exchange and the epilogue.  So weights, which depend on nothing, are requested
// before the dependency wait, what the epilogue reads from memory while the instructions run, and
// shared memory is held below half of an SM where that holds a CTA's operands, so that the next
// projection's CTAs come in while this one's finish.
//
// Every wait but the cluster barrier (all CTAs of a cluster always arrive) is bounded; when one runs
// out the CTA raises SSD_STATUS_TIMEOUT, drains its copies, frees its tensor memory and returns.
#include <algorithm>

#include "kernels.h"
#include "tc.h"
#include "tc_ptx.cuh"

namespace ssd {

namespace {

using namespace tcx;

constexpr int CH_THREADS = 256;   // copy warp, issuing warp, six more; all eight run the epilogue
constexpr int CH_MAX_STAGES = 8;
constexpr int CH_SK = 8;          // most k-steps per stage

struct ChParams {
  ChainGemm g;
  int n_groups, n_clusters;
  int KS, Mpad, Mc, tsplit, sk, stages, ng_max, rows_max, Tc, Tcp;
  uint32_t tmem_cols, off_red, off_push;
};

struct ChShared {
  unsigned long long full[CH_MAX_STAGES], empty[CH_MAX_STAGES], accum, gathered;
  uint32_t tmem_base;
  int abort;
  alignas(16) float inv_rms[TC_CHAIN_ROWS * 16];  // of this CTA's token rows; residual epilogue: its blocks' sums of squares
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Shared memory of this CTA to shared memory of another one of the cluster; completes on the
// receiver's barrier.
__device__ __forceinline__ void bulk_s2cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}

// Columns k .. k + 3 of a token's row of a packed operand.
__device__ __forceinline__ void store_quad(uint8_t* row, const ActLay& lay, int k, float4 x) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(x.x, x.y), h1 = __floats2bfloat162_rn(x.z, x.w);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(x.x - __low2float(h0), x.y - __high2float(h0));
  const __nv_bfloat162 l1 = __floats2bfloat162_rn(x.z - __low2float(h1), x.w - __high2float(h1));
  uint8_t* e = row + lay.col(k);
  *reinterpret_cast<uint2*>(e) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
  *reinterpret_cast<uint2*>(e + lay.part_off) =
      make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
}
// Column k of a token's row, in lanes whose neighbour (lane ^ 4) holds column k ^ 1: the even lane of the
// pair stores both leading parts, the odd one both remainders, a word each.  All lanes take part.
__device__ __forceinline__ void store_shared(uint8_t* row, const ActLay& lay, int k, float x, bool valid) {
  const bf16 h = __float2bfloat16_rn(x), l = __float2bfloat16_rn(x - __bfloat162float(h));
  const uint32_t hb = __bfloat16_as_ushort(h), lb = __bfloat16_as_ushort(l), odd = (uint32_t)k & 1u;
  const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? hb : lb, 4);
  if (valid)
    *reinterpret_cast<uint32_t*>(row + lay.col(k & ~1) + (odd ? lay.part_off : 0u)) = odd ? got | (lb << 16) : hb | (got << 16);
}
// Token rows t .. t + 3 (t a multiple of 4, so all of one chunk) of columns k (even lanes) and k + 1 (odd
// lanes): the lanes of a pair exchange two rows each, so that every store is a whole word.
__device__ __forceinline__ void store_pair4(const ActLay& lay, uint8_t* base, int t, int k, int lane, const float (&x)[4],
                                            int valid) {
  uint8_t* dst = lay.row(base, t) + lay.col(k);
  const int odd = lane & 1;
  const float s0 = odd ? x[0] : x[2], s1 = odd ? x[1] : x[3];
  const float r0 = __shfl_xor_sync(0xffffffffu, s0, 1), r1 = __shfl_xor_sync(0xffffffffu, s1, 1);
  const float a0 = odd ? r0 : x[0], b0 = odd ? x[2] : r0, a1 = odd ? r1 : x[1], b1 = odd ? x[3] : r1;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float a = q ? a1 : a0, b = q ? b1 : b0;
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
    if (odd * 2 + q < valid) {
      uint8_t* e = dst + (odd * 2 + q) * 16;
      *reinterpret_cast<__nv_bfloat162*>(e) = h;
      *reinterpret_cast<__nv_bfloat162*>(e + lay.part_off) = l;
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(CH_THREADS) tc_chain_kernel(const __grid_constant__ ChParams P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const ChainGemm& G = P.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, C = G.cluster;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int cl = (int)blockIdx.x / (C * P.tsplit), chunk = C > 1 ? 0 : (int)blockIdx.x - cl * P.tsplit;
  const int tbase = chunk * P.Mc, M = min(G.M - tbase, P.Mc);  // this CTA's token rows
  const int g0 = cl * P.n_groups / P.n_clusters, g1 = (cl + 1) * P.n_groups / P.n_clusters;
  const int ng = g1 - g0, rows = ng * 8, n0 = g0 * 8;  // this slab's groups and weight rows
  const int k0 = rank * P.KS / C, k1 = (rank + 1) * P.KS / C, n_iter = (k1 - k0 + P.sk - 1) / P.sk;
  const uint32_t gstride = (uint32_t)P.sk * 256u, act_block = (uint32_t)P.Mc * 64u;
  const uint32_t stage_w = (uint32_t)P.ng_max * gstride, stage_bytes = stage_w + (uint32_t)P.sk * act_block;
  float* red = reinterpret_cast<float*>(smem + P.off_red);    // [C][weight row][token row of this CTA, padded to Tcp]
  float* push = reinterpret_cast<float*>(smem + P.off_push);  // C > 1: this CTA's sums [owner][weight row][token row]
  ChShared& S = *reinterpret_cast<ChShared*>(red + (size_t)C * P.Tcp * P.rows_max * (C > 1 ? 2 : 1));
  volatile int* abort = &S.abort;

  if (tid == 0) {
    for (int s = 0; s < P.stages; ++s) {
      mbar_init(smem_u32(&S.full[s]), 1);
      mbar_init(smem_u32(&S.empty[s]), 1);
    }
    mbar_init(smem_u32(&S.accum), 1);
    mbar_init(smem_u32(&S.gathered), 1);
    S.abort = 0;
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(smem_u32(&S.tmem_base), P.tmem_cols);
  fence_before();
  __syncthreads();
  fence_after();
  if (C > 1) cluster_arrive();  // waited for before the first access to another CTA's memory
  // Tensor memory is held by now: a successor that is launched from here on cannot take it first.
  tc_pdl_trigger();
  const uint32_t tmem = S.tmem_base;

  if (warp == 0) {
    if (elect_one()) {  // ---- operand copies
      const uint64_t pol = policy_evict_first();
      const uint8_t* wsrc = G.w + ((size_t)g0 * P.KS + k0) * 256;
      const size_t wgroup = (size_t)P.KS * 256;
      const uint8_t* asrc = G.a + ((size_t)chunk * P.KS + k0) * act_block;
      const uint32_t smem0 = smem_u32(smem), nk_last = (uint32_t)(k1 - k0 - (n_iter - 1) * P.sk);
      auto weights = [&](int it, uint32_t s) {
        const uint32_t nk = it + 1 < n_iter ? (uint32_t)P.sk : nk_last, bar = smem_u32(&S.full[s]);
        mbar_expect_tx(bar, nk * ((uint32_t)ng * 256u + act_block));
        uint32_t dst = smem0 + s * stage_bytes;
        const uint8_t* src = wsrc + (size_t)it * gstride;
#pragma unroll 4
        for (int g = 0; g < ng; ++g) {
          bulk_g2s_hint(dst, src, nk * 256u, bar, pol);
          dst += gstride;
          src += wgroup;
        }
      };
      auto acts = [&](int it, uint32_t s) {
        const uint32_t nk = it + 1 < n_iter ? (uint32_t)P.sk : nk_last;
        bulk_g2s(smem0 + s * stage_bytes + stage_w, asrc + (size_t)it * P.sk * act_block, nk * act_block, smem_u32(&S.full[s]));
      };
      const int first = min(n_iter, P.stages);
      for (int it = 0; it < first; ++it) weights(it, (uint32_t)it);
      if (C > 1) mbar_expect_tx(smem_u32(&S.gathered), (uint32_t)(C * rows * P.Tcp) * 4u);
      tc_pdl_wait();
      for (int it = 0; it < first; ++it) acts(it, (uint32_t)it);
      uint32_t s = 0, par = 0;
      int it = first;
      for (; it < n_iter; ++it) {
        if (!mbar_wait(smem_u32(&S.empty[s]), par, abort)) break;
        acts(it, s);
        weights(it, s);
        if (++s == (uint32_t)P.stages) {
          s = 0;
          par ^= 1u;
        }
      }
      if (*abort)  // never leave with copies in flight into this CTA's shared memory
        for (int j = max(0, it - P.stages); j < it; ++j)
          mbar_wait(smem_u32(&S.full[j % P.stages]), (uint32_t)(j / P.stages) & 1u, abort);
    }
    __syncwarp();
    tc_pdl_wait();
  } else if (warp == 1) {
    if (elect_one()) {  // ---- MMA issue
      const uint32_t idesc = umma_idesc(2 * P.Mc);
      const uint64_t da = umma_desc(smem_u32(smem), 128u, gstride);
      const uint64_t db = umma_desc(smem_u32(smem) + stage_w, (uint32_t)P.Mc * 32u, 128u);
      const uint32_t ahi = (uint32_t)(da >> 32), bhi = (uint32_t)(db >> 32), alo = (uint32_t)da, blo = (uint32_t)db;
      uint32_t s = 0, par = 0;
      for (int it = 0; it < n_iter; ++it) {
        if (!mbar_wait(smem_u32(&S.full[s]), par, abort)) break;
        fence_after();
        const int nk = min(P.sk, k1 - k0 - it * P.sk);
        const uint32_t off = (s * stage_bytes) >> 4, a = alo + off, b = blo + off, bstep = act_block >> 4;
        if (nk == CH_SK) {  // straight-line: what the issuing thread executes is what these short instructions cost
          umma_bf16_lo(tmem, a, ahi, b, bhi, idesc, it > 0 ? 1u : 0u);
#pragma unroll
          for (int j = 1; j < CH_SK; ++j) umma_bf16_lo(tmem, a + j * 16, ahi, b + j * bstep, bhi, idesc, 1u);
        } else {
          for (int j = 0; j < nk; ++j) umma_bf16_lo(tmem, a + j * 16, ahi, b + j * bstep, bhi, idesc, it > 0 || j > 0 ? 1u : 0u);
        }
        umma_commit(smem_u32(&S.empty[s]));
        if (++s == (uint32_t)P.stages) {
          s = 0;
          par ^= 1u;
        }
      }
      umma_commit(smem_u32(&S.accum));
    }
    __syncwarp();
    tc_pdl_wait();
  } else {
    // ---- 1/rms of the token rows this CTA will finish, from the producers' shares of their sums of squares
    tc_pdl_wait();
    if (G.ssq_in) {
      const int t = rank * P.Tc + tid - 64;
      if (tid - 64 < P.Tc && t < M) {
        float v = 0.f;
#pragma unroll 8
        for (int i = 0; i < G.n_ssq_in; ++i) v += __ldcg(G.ssq_in + (size_t)i * P.Mpad + tbase + t);
        S.inv_rms[tid - 64] = rsqrtf(v * G.inv_d + G.eps);
      }
    }
  }

  // ---- the epilogue's tasks: a warp takes a quad of token rows x a block of 8 weight rows (QKV: of 8 rotary
  // pairs; SwiGLU: of 8 columns of its output), one element per lane: token lane % 4, row lane / 4.  So
  // shared memory is read without conflicts, operands are stored in contiguous 16-byte rows, and the
  // code is short: it runs once or twice per launch, and what it costs is mostly its instruction
  // fetches (four token rows per thread, unrolled, took 2200 cycles).  What the first task reads from memory
  // is requested while the instructions run; warps 2..7 come first, the copying and the issuing warp
  // have other work until now.
  const int tr = rank * P.Tc, t0 = tbase + tr, nt = min(P.Tc, M - tr), n_quads = (nt + 3) >> 2;
  const int n_elems = EPI == CHAIN_QKV || EPI == CHAIN_SWIGLU ? rows >> 1 : rows, n_blocks = (n_elems + 7) >> 3;
  const int n_tasks = n_quads * n_blocks, task0 = (warp + 6) & 7;
  const int hl2 = G.hd_log2, half = 1 << (hl2 - 1);
  struct Task {
    int tl, t, e, blk;      // token row of this CTA, of the forward; element; its block
    bool ok;
    int hh, j, owner, slot; // QKV: head, rotary pair, where K or V goes
    float2 cs, bias;
    float h, gain;          // residual
  } T;
  auto load_task = [&](int i) {
    const int quad = i / n_blocks;
    T.blk = i - quad * n_blocks;
    T.tl = quad * 4 + (lane & 3);
    T.e = T.blk * 8 + (lane >> 2);
    T.ok = T.tl < nt && T.e < n_elems;
    T.t = t0 + min(T.tl, nt - 1);
    if (EPI == CHAIN_QKV && T.ok) {
      const int pr = (n0 >> 1) + T.e;  // weight rows 2 e and 2 e + 1 of the slab are a rotary pair (chain_qkv_row)
      T.hh = pr >> (hl2 - 1);
      T.j = pr & (half - 1);
      const bf16* bias = G.bias + ((size_t)T.hh << hl2) + T.j;
      T.bias = make_float2(__bfloat162float(bias[0]), __bfloat162float(bias[half]));
      T.cs = make_float2(1.f, 0.f);
      if (T.hh < G.Hq + G.Hkv) T.cs = __ldcg(reinterpret_cast<const float2*>(G.rope_cs + ((size_t)T.t << hl2) + 2 * T.j));
      if (T.hh >= G.Hq) {  // the stream's slice of a contiguous cache, or its page
        const int2 br = row_at(G.rm, T.t);
        const int pos = __ldcg(G.len + br.x) + br.y;
        T.owner = br.x;
        T.slot = pos;
        if (pos < 0 || pos >= G.cap) {  // never write outside the stream's slice of the cache
          atomicOr(G.status, SSD_STATUS_KV_OVERFLOW);
          T.slot = -1;
        } else if (G.page_table) {  // no page granted (pool exhausted): flagged by the page kernel
          T.owner = __ldcg(G.page_table + (size_t)br.x * G.max_pages + pos / TC_PAGE_TOKENS);
          T.slot = T.owner < 0 ? -1 : pos % TC_PAGE_TOKENS;
        }
      }
    }
    if (EPI == CHAIN_RESIDUAL) {
      T.h = T.gain = 0.f;
      if (T.ok) {
        T.gain = __bfloat162float(G.gain[n0 + T.e]);
        T.h = __ldcg(G.h + (size_t)T.t * G.n_rows + n0 + T.e);
      }
    }
  };
  if (EPI != CHAIN_SWIGLU && EPI != CHAIN_LOGITS && task0 < n_tasks) load_task(task0);

  // ---- the accumulator's columns to the owners of their token rows
  {
    const int q = warp & 3, sub = warp >> 2, row = q * 32 + lane;
    const bool ok = mbar_wait(smem_u32(&S.accum), 0u, abort);
    fence_after();
    if (ok && q * 32 < rows) {  // uniform per warp
      const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
      float* mine = (C > 1 ? push : red) + (size_t)row * P.Tcp;
      for (int c0 = sub * 32; c0 < M; c0 += 64) {
        uint32_t v[32], w[32];
        tmem_ld32_async(lane_addr + (uint32_t)c0, v);
        tmem_ld32_async(lane_addr + (uint32_t)(P.Mc + c0), w);
        tmem_wait_ld();
        tmem_ready(v);
        tmem_ready(w);
        if (row < rows) {
          const int o = C > 1 ? c0 / P.Tc : 0;
          int tl = c0 - o * P.Tc;
          float* dst = mine + (size_t)o * P.rows_max * P.Tcp + tl;
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            // four token rows, all of one owner (C = 1: room for whole ranges of 32)
            if (C > 1 && c0 + i >= M) break;
            *reinterpret_cast<float4*>(dst) =
                make_float4(__uint_as_float(v[i]) + __uint_as_float(w[i]), __uint_as_float(v[i + 1]) + __uint_as_float(w[i + 1]),
                            __uint_as_float(v[i + 2]) + __uint_as_float(w[i + 2]), __uint_as_float(v[i + 3]) + __uint_as_float(w[i + 3]));
            dst += 4;
            if (C > 1 && (tl += 4) >= P.Tc) {
              tl = 0;
              dst += (size_t)P.rows_max * P.Tcp - P.Tc;
            }
          }
        }
      }
    }
  }
  fence_before();
  if (C > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // ordinary stores, read by the copies
  __syncthreads();
  if (C > 1) {
    cluster_wait();  // every CTA of the cluster has started: its barriers exist
    if (warp == 0 && elect_one()) {
      const uint32_t bytes = (uint32_t)(rows * P.Tcp) * 4u, block = (uint32_t)(P.rows_max * P.Tcp) * 4u;
      for (int i = 0; i < C; ++i) {
        const uint32_t o = (uint32_t)((rank + i) & (C - 1));  // not all to the same CTA at once (C is a power of two)
        bulk_s2cluster(map_rank(smem_u32(red) + (uint32_t)rank * block, o), smem_u32(push) + o * block, bytes,
                       map_rank(smem_u32(&S.gathered), o));
      }
    }
    __syncwarp();
    mbar_wait(smem_u32(&S.gathered), 0u, abort);
    cluster_arrive();  // this CTA has what it needs of the others' memory
  }
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tmem, P.tmem_cols);
  }

  // ---- the C contributions of this CTA's token rows, in rank order, and what becomes of them
  const int src = P.rows_max * P.Tcp;  // floats from one CTA's contributions to the next one's
  auto sum = [&](int row, int tl) {
    const float* r = red + row * P.Tcp + tl;
    float a = r[0];
    if (C == 8) {  // all loads in flight
      float b[7];
#pragma unroll
      for (int s = 0; s < 7; ++s) b[s] = r[(s + 1) * src];
#pragma unroll
      for (int s = 0; s < 7; ++s) a += b[s];
    }
    return a;
  };
  auto sum4 = [&](int row, int quad) {  // of four token rows
    const float* r = red + row * P.Tcp + quad * 4;
    float4 a = *reinterpret_cast<const float4*>(r);
    for (int s = 1; s < C; ++s) {
      const float4 b = *reinterpret_cast<const float4*>(r + s * src);
      a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    return a;
  };
  if (!*abort) {
    float* sq = &S.inv_rms[0];  // residual: [token][block] sums of squares (1/rms is not in use by that epilogue)
    if (EPI == CHAIN_SWIGLU) {
      // every CTA has hundreds of elements here: four token rows per thread (one per thread: 10.5 instead of
      // 8.9 us at 96 rows); lanes are neighbouring columns
      const int per = rows >> 1, n_all = n_quads * per;  // rows interleaved: gate, up; per is a multiple of 4
      for (int i0 = warp * 32; i0 < n_all; i0 += CH_THREADS) {
        const int i = min(i0 + lane, n_all - 1), quad = i / per, e = i - quad * per, k = (n0 >> 1) + e;
        const float4 g = sum4(2 * e, quad), u = sum4(2 * e + 1, quad);
        const float4 inv = *reinterpret_cast<const float4*>(&S.inv_rms[quad * 4]);
        const float g4[4] = {g.x * inv.x, g.y * inv.y, g.z * inv.z, g.w * inv.w};
        const float u4[4] = {u.x * inv.x, u.y * inv.y, u.z * inv.z, u.w * inv.w};
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = __fdividef(g4[q], 1.f + __expf(-g4[q])) * u4[q];
        store_pair4(G.lay_out, G.act_out, t0 + quad * 4, k & ~1, lane, x, i0 + lane < n_all ? min(4, nt - quad * 4) : 0);
      }
    } else if (EPI == CHAIN_LOGITS) {
      for (int i = tid; i < n_quads * rows; i += CH_THREADS) {
        const int quad = i / rows, e = i - quad * rows;
        const float4 a = sum4(e, quad);
        const float a4[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int tl = quad * 4 + q;
          if (tl < nt && n0 + e < G.n_rows) G.out[(size_t)(t0 + tl) * G.n_rows + n0 + e] = a4[q] * S.inv_rms[tl];
        }
      }
    } else {
#pragma unroll 1
    for (int i = task0; i < n_tasks; i += CH_THREADS / 32) {
      if (i != task0) load_task(i);
      if (EPI == CHAIN_QKV) {
        if (T.ok) {
          const float inv = S.inv_rms[T.tl];
          const float x = fmaf(sum(2 * T.e, T.tl), inv, T.bias.x), y = fmaf(sum(2 * T.e + 1, T.tl), inv, T.bias.y);
          const float u = x * T.cs.x - y * T.cs.y, v = y * T.cs.x + x * T.cs.y;  // values: (1, 0), unchanged
          if (T.hh < G.Hq) {
            float* dst = G.qrot + (((size_t)T.t * G.Hq + T.hh) << hl2) + T.j;
            dst[0] = u * G.qscale;
            dst[half] = v * G.qscale;
          } else if (T.slot >= 0) {
            const int which = T.hh >= G.Hq + G.Hkv, g = T.hh - G.Hq - which * G.Hkv;
            const size_t rows_per = G.page_table ? (size_t)TC_PAGE_TOKENS : (size_t)G.cap;
            bf16* dst = G.kv_layer + (((((size_t)T.owner * 2 + which) * G.Hkv + g) * rows_per + T.slot) << hl2) + T.j;
            dst[0] = __float2bfloat16_rn(u);
            dst[half] = __float2bfloat16_rn(v);
          }
        }
      } else if (EPI == CHAIN_RESIDUAL) {
        const int n = n0 + T.e;
        float x = 0.f;
        if (T.ok) {
          x = T.h + sum(T.e, T.tl);
          G.h[(size_t)T.t * G.n_rows + n] = x;
        }
        store_shared(G.lay_out.row(G.act_out, T.t), G.lay_out, n, x * T.gain, T.ok);
        float ss = x * x;
        ss += __shfl_xor_sync(0xffffffffu, ss, 4);
        ss += __shfl_xor_sync(0xffffffffu, ss, 8);
        ss += __shfl_xor_sync(0xffffffffu, ss, 16);
        if (lane < 4 && T.ok) sq[T.tl * n_blocks + T.blk] = ss;
      }
    }
    }
    if (EPI == CHAIN_RESIDUAL) {
      __syncthreads();  // (every thread of the CTA is here)
      if (tid < nt) {
        float v = 0.f;
        for (int e = 0; e < n_blocks; ++e) v += sq[tid * n_blocks + e];
        G.ssq_out[(size_t)cl * P.Mpad + t0 + tid] = v;
      }
    }
  }
  if (C > 1) cluster_wait();  // the others have gathered: this CTA's memory is no longer read
  if (tid == 0 && *abort) atomicOr(G.status, SSD_STATUS_TIMEOUT);
}

// ---- the rows that enter the chain: ids, embedding, the first projection's operand, rotary table --

__global__ void __launch_bounds__(256)
chain_embed_kernel(const bf16* __restrict__ table, int vocab_in, int d, const int32_t* __restrict__ row_ids,
                   const int32_t* __restrict__ pending, const int32_t* __restrict__ draft,
                   const int32_t* __restrict__ len, RowMap rm, const bf16* __restrict__ gain,
                   const double* __restrict__ inv_freq, int half, float* __restrict__ h, uint8_t* __restrict__ apack,
                   ActLay lay, float* __restrict__ ssq, float* __restrict__ cs, int32_t* status) {
  __shared__ float red[8];
  const int m = blockIdx.x, tid = threadIdx.x;
  tc_pdl_enter();  // not before the wait: the attention of the first layer relies on older kernels being complete
  const int2 br = row_at(rm, m);
  int id = row_ids ? row_ids[m] : br.y == 0 ? pending[br.x] : draft[(size_t)br.x * (rm.R - 1) + br.y - 1];
  if (id < 0 || id >= vocab_in) {
    if (tid == 0) atomicOr(status, SSD_STATUS_BAD_TOKEN);
    id = min(max(id, 0), vocab_in - 1);
  }
  const double pos = (double)(len[br.x] + br.y);
  for (int j = tid; j < half; j += 256) {
    double s, c;
    sincos(pos * inv_freq[j], &s, &c);
    *reinterpret_cast<float2*>(cs + ((size_t)m * half + j) * 2) = make_float2((float)c, (float)s);
  }
  const bf16* src = table + (size_t)id * d;
  uint8_t* arow = lay.row(apack, m);
  float ss = 0.f;
  for (int j = tid * 4; j < d; j += 1024) {  // d is a multiple of 8
    const uint2 v = *reinterpret_cast<const uint2*>(src + j), g = *reinterpret_cast<const uint2*>(gain + j);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    const float2 ga = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g.x));
    const float2 gb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g.y));
    *reinterpret_cast<float4*>(h + (size_t)m * d + j) = make_float4(a.x, a.y, b.x, b.y);
    store_quad(arow, lay, j, make_float4(a.x * ga.x, a.y * ga.y, b.x * gb.x, b.y * gb.y));
    ss += a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y;
  }
  ss = warp_sum(ss);
  if ((tid & 31) == 0) red[tid >> 5] = ss;
  __syncthreads();
  if (tid == 0) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += red[w];
    ssq[m] = t;
  }
}

// ---- weight packing (once per model): group of 8 rows, k-step: 256 bytes (two core matrices) ------

// Weight row of a packed row of the QKV projection: the rotary partners (j, j + hd / 2) of a head are
// neighbours (value heads likewise: only the order of their rows changes), so that a slab of any
// number of groups holds whole pairs.
__device__ __forceinline__ int chain_qkv_row(int r, int hd_log2) {
  const int head = r >> hd_log2, i = r & ((1 << hd_log2) - 1);
  return (head << hd_log2) + (i >> 1) + ((i & 1) << (hd_log2 - 1));
}

__global__ void chain_pack_kernel(const bf16* __restrict__ w, int n_rows, int K, int KS, int hd_log2, size_t n,
                                  uint4* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // ((group * KS + kstep) * 2 + half) * 8 + row
  if (i >= n) return;
  const int r = (int)(i & 7), half = (int)((i >> 3) & 1);
  const size_t blk = i >> 4;
  const int prow = (int)(blk / KS) * 8 + r, row = hd_log2 ? chain_qkv_row(prow, hd_log2) : prow;
  const int k = (int)(blk % KS) * 16 + half * 8;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (row < n_rows && k < K) v = *reinterpret_cast<const uint4*>(w + (size_t)row * K + k);  // K is a multiple of 8
  out[i] = v;
}

template <int EPI>
cudaError_t launch_chain(const ChParams& p, size_t smem, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(tc_chain_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  e = tc_launch_pdl_cluster(tc_chain_kernel<EPI>, dim3(p.n_clusters * p.g.cluster * p.tsplit), dim3(CH_THREADS), p.g.cluster,
                            smem, st, p);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t chain_pack_weights(const bf16* w, int n_rows, int K, int hd_log2, uint8_t* packed, cudaStream_t st) {
  const int KS = (K + 15) / 16;
  const size_t n = chain_weight_bytes(n_rows, K) / 16;
  chain_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w, n_rows, K, KS, hd_log2, n, reinterpret_cast<uint4*>(packed));
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_chain_embed(const bf16* table, int vocab_in, int d, const int32_t* row_ids, const int32_t* pending,
                               const int32_t* draft, const int32_t* len, RowMap rm, const bf16* gain,
                               const double* inv_freq, int half, float* h, uint8_t* apack, float* ssq, float* cs,
                               int32_t* status, cudaStream_t st) {
  const int M = row_count(rm);
  const cudaError_t e = tc_launch_pdl(chain_embed_kernel, dim3(M), dim3(256), 0, st, table, vocab_in, d, row_ids, pending, draft,
                                      len, rm, gain, inv_freq, half, h, apack, tc_act_lay(chain_chunk_rows(M, d, false), d), ssq,
                                      cs, status);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

// How a projection is cut.  Where K is short every CTA takes all of it: the instructions of 56 k-steps
// cost less than exchanging partial sums (~5000 cycles), and reading all activations in every CTA
// runs at L2's 70 to 100 bytes per cycle and SM; with more than 48 rows a slab's token rows are halved
// between two CTAs, which halves both.  A long K (the down projection) is split over a cluster of 8, of which
// 15 fit at once when each CTA takes an SM (cudaOccupancyMaxActiveClusters; the GPCs are not all of
// one size, and a cluster too many makes a second wave: 20 instead of 9 us).
// There are as many slabs as fill the SMs once, and no fewer than 16 groups each need.
ChainSplit chain_split(int n_rows, int K, int M, int n_sm, bool whole) {
  const int groups = (n_rows + 7) / 8;
  ChainSplit s;
  s.cluster = chain_long(K) ? 8 : 1;
  s.tsplit = s.cluster == 1 && !whole && M > 48 ? 2 : 1;
  const int room = s.cluster > 1 ? std::max(1, std::min(14, n_sm / s.cluster)) : n_sm / s.tsplit;
  s.clusters = std::max((groups + 15) / 16, std::min(groups, room));
  return s;
}

cudaError_t launch_tc_chain(const ChainGemm& g, int epi, int K, bool whole, int n_sm, cudaStream_t st) {
  if (g.M < 1 || g.M > TC_CHAIN_ROWS || (K & 7) || (g.n_rows & 7 && epi != CHAIN_LOGITS)) return cudaErrorInvalidValue;
  ChParams p{};
  p.g = g;
  const ChainSplit cs = chain_split(g.n_rows, K, g.M, n_sm, whole);
  p.g.cluster = cs.cluster;
  p.n_groups = (g.n_rows + 7) / 8;
  p.n_clusters = cs.clusters;
  p.KS = (K + 15) / 16;
  p.Mpad = tc_round16(g.M);
  p.tsplit = cs.tsplit;
  p.Mc = cs.tsplit > 1 ? chain_chunk_rows(g.M, K, whole) : p.Mpad;
  const int Mcta = cs.tsplit > 1 ? p.Mc : g.M;
  p.Tc = ((Mcta + cs.cluster - 1) / cs.cluster + 3) / 4 * 4;  // quads of token rows have one owner
  p.Tcp = cs.cluster > 1 ? p.Tc : (p.Tc + 31) / 32 * 32;
  if (p.Tcp % 8 == 0) p.Tcp += 4;                            // 16-byte stores of 8 lanes to 32 banks
  p.ng_max = (p.n_groups + cs.clusters - 1) / cs.clusters;
  p.rows_max = p.ng_max * 8;
  const size_t red = (size_t)cs.cluster * p.Tcp * p.rows_max * 4 * (cs.cluster > 1 ? 2 : 1);  // gathered, and pushed
  const int ks_cta = (p.KS + cs.cluster - 1) / cs.cluster;
  const size_t per_ks = (size_t)p.ng_max * 256 + (size_t)p.Mc * 64;
  // half an SM (the next kernel's CTAs then come in while this one's finish) where that holds all of a
  // CTA's operands or three stages of at least 16 KB, else the whole of it: with two stages in flight a
  // CTA took in 26 bytes per cycle (measured), with five 70
  size_t budget = 111 * 1024 - sizeof(ChShared) - 128;
  p.sk = std::min(CH_SK, ks_cta);
  if (ks_cta * per_ks + red > budget && (3 * p.sk * per_ks + red > budget || p.sk * per_ks < 16384)) {
    budget = 226 * 1024 - sizeof(ChShared) - 128;
    while (p.sk > 2 && 4 * p.sk * per_ks + red > budget && p.sk * per_ks > 32768) p.sk = (p.sk + 1) / 2;
  }
  if (2 * p.sk * per_ks + red > budget) return cudaErrorInvalidValue;
  p.stages = (int)std::min((budget - red) / (p.sk * per_ks), (size_t)CH_MAX_STAGES);
  p.stages = std::min(p.stages, (ks_cta + p.sk - 1) / p.sk);
  // the instruction reads 16 groups whatever the slab holds: the last stage's must lie in shared memory
  const size_t stage = p.sk * per_ks;
  p.off_red = (uint32_t)std::max(p.stages * stage, (p.stages - 1) * stage + (size_t)p.sk * 4096);
  p.off_push = p.off_red + (uint32_t)(cs.cluster * p.Tcp * p.rows_max * 4);
  p.tmem_cols = 32;
  while (p.tmem_cols < (uint32_t)(p.Mc + (Mcta + 31) / 32 * 32)) p.tmem_cols <<= 1;
  const size_t smem = p.off_red + red + sizeof(ChShared) + 64;
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  switch (epi) {
    case CHAIN_QKV: return launch_chain<CHAIN_QKV>(p, smem, st);
    case CHAIN_RESIDUAL: return launch_chain<CHAIN_RESIDUAL>(p, smem, st);
    case CHAIN_SWIGLU: return launch_chain<CHAIN_SWIGLU>(p, smem, st);
    case CHAIN_LOGITS: return launch_chain<CHAIN_LOGITS>(p, smem, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ssd
