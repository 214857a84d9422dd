// Projections of a prefill chunk (hundreds to TC_MAX_ROWS rows) on tcgen05 tensor cores.
//
// A work item is a pair of tiles of 128 weight rows x two chunks of at most 64 token rows x the whole
// K, worked on by a pair of CTAs (cta_group::2): CTA r holds the weights of tile r and the bf16
// leading parts (r = 0) or remainders (r = 1) of the activations; one 256 x 128 x 16 instruction,
// issued by the leader, multiplies both tiles with both parts.  A persistent grid of pairs takes
// items in turn.  A row is summed in exactly the order in which a forward of up to 128 rows sums it
// (tc_gemm.cu): K in the same slices; within a slice even and odd k-steps, and the two parts, in
// accumulators of their own; the slices added one after the other to the bias, the residual stream
// or zero.  A prompt's keys and values therefore do not depend on the chunk it travelled in.  Two
// chunks of four accumulators of 64 columns fill tensor memory; four warps per chunk move a slice's
// accumulators to registers (64 columns per thread) and add them there while the other chunk's
// instructions run.  SwiGLU and the stores overlap the next item.  Chunks of few rows have too few
// items for the chip: their slices are shared out, and each slice's sums go to memory for the row
// kernels to add (tc_rows.cu).
//
// What bounds it: shared-memory bandwidth (128 bytes per cycle).  Per k-step of 16 columns a CTA
// writes 4 KB of weights and 4 KB of activations and the two instructions read 12 KB: 156 cycles,
// against 130 of tensor-core work.  (The same kernel on single CTAs moved 28 KB per k-step and took
// 290 cycles; one chunk of 128 rows, 24 KB, 228 cycles and 1300 cycles more per slice, in which
// nothing ran.)  The operands of a stage of four k-steps are contiguous, so one elected thread moves
// them with three bulk copies: a single thread spends ~250 cycles on a stage's barrier and ~30 per
// copy (measured), which small stages do not hide.
//
// Every wait is bounded; when one runs out the CTA raises SSD_STATUS_TIMEOUT, waits (bounded) for
// its copies in flight, frees its tensor memory and returns.
#include <algorithm>

#include "kernels.h"
#include "tc.h"
#include "tc_ptx.cuh"

namespace ssd {

namespace {

using namespace tcx;

constexpr int PF_EPI_WARPS = 8;
constexpr int PF_THREADS = PF_EPI_WARPS * 32 + 64;  // + copy warp, + issuing (leader) or relaying warp
constexpr int PF_SK = 8;                            // k-steps per stage
constexpr int PF_MAX_STAGES = 8;
constexpr uint32_t PF_STG_STRIDE = 528;             // SwiGLU staging: 32 rows of 16 bytes, padded
constexpr uint32_t PF_STG_BYTES = PF_EPI_WARPS * 4 * PF_STG_STRIDE;

struct PfParams {
  const uint8_t* w;
  const uint8_t* a;
  int n_rows, KS, M, Mpad, Mc, tiles, pairs, nchunk, groups, n_items, nslice, slice_q, slice_r, stages, dual, ldo;
  const bf16* bias;
  float* out;      // QKV: q/k/v rows [M][ldo]; residual: the stream h [M][ldo], read and written
  uint8_t* act_out;
  ActLay lay_out;
  int32_t* status;
};

// The K slices [s KS / n, (s + 1) KS / n) one after the other, without dividing: a 64-bit division per
// slice in each role cost 1100 cycles of a slice's 2200.
struct SliceWalk {
  int s, k0 = 0, k1, left, acc, q, r, n;
  __device__ __forceinline__ SliceWalk(const PfParams& P, int s0, int s1)
      : s(s0 - 1), k1(s0 * P.KS / P.nslice), left(s1 - s0), acc(s0 * P.slice_r % P.nslice), q(P.slice_q), r(P.slice_r), n(P.nslice) {}
  __device__ __forceinline__ bool next() {
    if (left-- == 0) return false;
    ++s;
    k0 = k1;
    acc += r;
    k1 += q;
    if (acc >= n) {
      acc -= n;
      ++k1;
    }
    return true;
  }
};
// A work item: a pair of weight tiles, a pair of row chunks, and - where the slices are shared out over
// several items - a range of them.
struct PfItem {
  int tile, chunk, s0, s1;
  __device__ __forceinline__ PfItem(const PfParams& P, int item, uint32_t rank) {
    const int g = item % P.groups, tc = item / P.groups, c = tc / P.pairs;
    tile = (tc - c * P.pairs) * 2 + (int)rank;
    chunk = c * 2;
    s0 = g * P.nslice / P.groups;
    s1 = (g + 1) * P.nslice / P.groups;
  }
};

struct PfShared {
  unsigned long long full[PF_MAX_STAGES];  // this CTA's copies of the stage have landed; leader: the other CTA's too
  unsigned long long empty[PF_MAX_STAGES], accum[2];
  unsigned long long drained[2];                // leader: both CTAs' warps have emptied the chunk's accumulators
  uint32_t tmem_base;
  int abort;
};

template <int EPI>
__global__ void __launch_bounds__(PF_THREADS, 1) tc_prefill_gemm_kernel(const __grid_constant__ PfParams P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  const int pair0 = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const uint32_t act_block = (uint32_t)P.Mc * 32u;  // one part of a k-step
  const uint32_t stage_w = PF_SK * TC_WBLOCK, stage_a = PF_SK * act_block, stage_bytes = stage_w + 2 * stage_a;
  uint8_t* staging = smem + (size_t)P.stages * stage_bytes;
  PfShared& S = *reinterpret_cast<PfShared*>(staging + PF_STG_BYTES);
  volatile int* abort = &S.abort;
  if (tid == 0) {
    for (int s = 0; s < P.stages; ++s) {
      mbar_init(smem_u32(&S.full[s]), rank == 0 ? 2 : 1);
      mbar_init(smem_u32(&S.empty[s]), 1);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(smem_u32(&S.accum[u]), 1);
      mbar_init(smem_u32(&S.drained[u]), PF_EPI_WARPS);  // four warps of each CTA
    }
    S.abort = 0;
    mbar_init_fence();
  }
  tc_pdl_trigger();
  if (warp != PF_EPI_WARPS) tc_pdl_wait();
  if (warp == PF_EPI_WARPS + 1) tmem_alloc_pair(smem_u32(&S.tmem_base), 512);
  fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist
  fence_after();
  const uint32_t tmem = S.tmem_base, bar_accum = smem_u32(&S.accum[0]), bar_drained = smem_u32(&S.drained[0]);

  if (warp == PF_EPI_WARPS) {
    // ---- operand copies.  The first fill's weights go out before the predecessor has finished.
    if (elect_one()) {
      uint32_t s = 0, par = 1, n_issued = 0;
      bool waited = false;
      const size_t part_bytes = (size_t)P.KS * act_block, chunk_bytes = 2 * part_bytes;
      uint32_t pend_bytes[PF_MAX_STAGES], pend_two = 0;  // first fill: activations still to request
      const uint8_t* pend_src[PF_MAX_STAGES];
      auto acts = [&](uint32_t stage, const uint8_t* src, uint32_t bytes, bool two) {
        const uint32_t dst = smem_u32(smem) + stage * stage_bytes + stage_w, bar = smem_u32(&S.full[stage]);
        bulk_g2s(dst, src, bytes, bar);
        if (two) bulk_g2s(dst + stage_a, src + chunk_bytes, bytes, bar);
      };
      auto flush = [&]() {
        tc_pdl_wait();
        waited = true;
        for (uint32_t i = 0; i < n_issued; ++i) acts(i, pend_src[i], pend_bytes[i], (pend_two >> i) & 1u);
      };
      for (int item = pair0; item < P.n_items && !*abort; item += n_pairs) {
        const PfItem it(P, item, rank);
        const int tile = it.tile, chunk = it.chunk;
        const bool two = chunk + 1 < P.nchunk;
        const uint32_t wblock = tile < P.tiles ? TC_WBLOCK : 0u;  // an odd last tile: the other half computes nothing of use
        const uint8_t* w = P.w + (size_t)tile * P.KS * TC_WBLOCK;
        const uint8_t* a = P.a + (size_t)chunk * chunk_bytes + rank * part_bytes;
        for (SliceWalk walk(P, it.s0, it.s1); walk.next();) {
          const int k0 = walk.k0, k1 = walk.k1;
          for (int k = k0; k < k1; k += PF_SK) {
            const uint32_t nk = (uint32_t)min(PF_SK, k1 - k);
            const uint32_t bar = smem_u32(&S.full[s]), dst = smem_u32(smem) + s * stage_bytes;
            if (n_issued >= (uint32_t)P.stages && !mbar_wait(smem_u32(&S.empty[s]), par, abort)) break;
            mbar_expect_tx(bar, nk * (wblock + (two ? 2u : 1u) * act_block));
            if (wblock) bulk_g2s(dst, w + (size_t)k * TC_WBLOCK, nk * TC_WBLOCK, bar);
            if (waited) {
              acts(s, a + (size_t)k * act_block, nk * act_block, two);
            } else {
              pend_src[n_issued] = a + (size_t)k * act_block;
              pend_bytes[n_issued] = nk * act_block;
              pend_two |= two ? 1u << n_issued : 0u;
            }
            ++n_issued;
            if (!waited && n_issued == (uint32_t)P.stages) flush();
            if (++s == (uint32_t)P.stages) {
              s = 0;
              par ^= 1u;
            }
          }
        }
      }
      if (!waited) flush();
      // never leave with copies in flight: wait for the last use of every stage
      const uint32_t last = n_issued < (uint32_t)P.stages ? n_issued : (uint32_t)P.stages;
      for (uint32_t j = 0; j < last; ++j) {
        const uint32_t n = n_issued - last + j;
        mbar_wait(smem_u32(&S.full[n % P.stages]), (n / P.stages) & 1u, abort);
      }
    }
    __syncwarp();
  } else if (warp == PF_EPI_WARPS + 1) {
    if (rank != 0) {
      // ---- tell the leader which stages have landed here
      if (elect_one()) {
        uint32_t s = 0, par = 0;
        for (int item = pair0; item < P.n_items && !*abort; item += n_pairs) {
          const PfItem it(P, item, rank);
          for (SliceWalk walk(P, it.s0, it.s1); walk.next();) {
            const int k0 = walk.k0, k1 = walk.k1;
            for (int k = k0; k < k1; k += PF_SK) {
              if (!mbar_wait(smem_u32(&S.full[s]), par, abort)) break;
              mbar_arrive_cluster(map_rank(smem_u32(&S.full[s]), 0));
              if (++s == (uint32_t)P.stages) {
                s = 0;
                par ^= 1u;
              }
            }
          }
        }
      }
    } else if (elect_one()) {
      // ---- MMA issue
      // One wait per stage of eight instructions: the tensor core's queue covers it (measured: with
      // a wait, or a second one, per four instructions of this size they ran at 350 to 400 cycles
      // instead of 258; so the other CTA's arrival counts on the same barrier).
      const uint32_t idesc = umma_idesc_pair(2 * P.Mc), set = 2u * (uint32_t)P.Mc;
      const uint64_t da = umma_desc(smem_u32(smem), 2048u, 128u), db = umma_desc(smem_u32(smem) + stage_w, act_block >> 1, 128u);
      const uint32_t ahi = (uint32_t)(da >> 32), bhi = (uint32_t)(db >> 32), stage16 = stage_bytes >> 4;
      const uint32_t astep = TC_WBLOCK >> 4, bstep = act_block >> 4, bchunk = stage_a >> 4;
      uint32_t s = 0, par = 0, alo = (uint32_t)da, blo = (uint32_t)db, n_acc0 = 0, n_acc1 = 0;
      for (int item = pair0; item < P.n_items && !*abort; item += n_pairs) {
        const PfItem it(P, item, rank);
        const bool two = it.chunk + 1 < P.nchunk;
        for (SliceWalk walk(P, it.s0, it.s1); walk.next();) {
          const int k0 = walk.k0, k1 = walk.k1;
          const uint32_t dual = P.dual && k1 - k0 >= 2 ? 1u : 0u;
          for (int k = k0; k < k1; k += PF_SK) {
            if (!mbar_wait_cluster(smem_u32(&S.full[s]), par, abort)) break;
            const int nk = min(PF_SK, k1 - k);
            // even k-steps: columns [0, 2 Mc) of the chunk's, odd ones [2 Mc, 4 Mc)
            auto chunk = [&](uint32_t acc, uint32_t b0) {
              fence_after();
#pragma unroll
              for (int j = 0; j < PF_SK; ++j) {
                const uint32_t kk = (uint32_t)(k - k0 + j);
                if (j < nk)
                  umma_bf16_pair_lo(acc + (kk & dual) * set, alo + j * astep, ahi, b0 + j * bstep, bhi, idesc,
                                    kk > dual ? 1u : 0u);
              }
            };
            // a slice begins: the chunk's previous accumulators are in registers
            if (k == k0 && n_acc0 > 0 && !mbar_wait_cluster(bar_drained, (n_acc0 - 1) & 1u, abort)) break;
            chunk(tmem, blo);
            if (k + PF_SK >= k1) {
              umma_commit_pair(bar_accum);
              ++n_acc0;
            }
            if (two) {
              if (k == k0 && n_acc1 > 0 && !mbar_wait_cluster(bar_drained + 8, (n_acc1 - 1) & 1u, abort)) break;
              chunk(tmem + 2 * set, blo + bchunk);
              if (k + PF_SK >= k1) {
                umma_commit_pair(bar_accum + 8);
                ++n_acc1;
              }
            }
            umma_commit_pair(smem_u32(&S.empty[s]));
            alo += stage16;
            blo += stage16;
            if (++s == (uint32_t)P.stages) {
              s = 0;
              par ^= 1u;
              alo = (uint32_t)da;
              blo = (uint32_t)db;
            }
          }
        }
      }
    }
    __syncwarp();
  } else {
    // ---- accumulators to registers, slices added, results out
    const int q = warp & 3, sub = warp >> 2, row = q * 32 + lane;
    const uint32_t Mc = (uint32_t)P.Mc, t_lane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)sub * 4u * Mc;
    const uint32_t drained0 = map_rank(bar_drained + sub * 8, 0);
    uint32_t n_acc = 0;
    for (int item = pair0; item < P.n_items; item += n_pairs) {
      const PfItem it(P, item, rank);
      const int tile = it.tile, chunk = it.chunk + sub, n = tile * TC_TILE_ROWS + row;
      if (chunk >= P.nchunk) break;  // the last row chunk stands alone (items of a CTA have rising chunks)
      const int t0 = chunk * P.Mc, rows_here = min(P.M - t0, P.Mc);
      float acc[2][32];
      {
        float b = 0.f;
        if (EPI == PF_EPI_BIAS && P.bias && n < P.n_rows) b = __bfloat162float(P.bias[n]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            acc[h][i] = b;
            if (EPI == PF_EPI_RESIDUAL) {
              const int c = h * 32 + i;
              if (c < rows_here && n < P.n_rows) acc[h][i] = __ldcg(P.out + (size_t)(t0 + c) * P.ldo + n);
            }
          }
        }
      }
      for (SliceWalk walk(P, it.s0, it.s1); walk.next();) {
        const int k0 = walk.k0, k1 = walk.k1;
        const bool dual = P.dual && k1 - k0 >= 2;
        if (!mbar_wait(bar_accum + sub * 8, n_acc & 1u, abort)) break;
        ++n_acc;
        fence_after();
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint32_t c0 = (uint32_t)(h * 16);
          if ((int)c0 < rows_here) {  // uniform
            uint32_t a[16], b[16], c[16], d[16];
            tmem_ld16_async(t_lane + c0, a);
            tmem_ld16_async(t_lane + Mc + c0, b);
            if (dual) {
              tmem_ld16_async(t_lane + 2 * Mc + c0, c);
              tmem_ld16_async(t_lane + 3 * Mc + c0, d);
            }
            tmem_wait_ld();
            tmem_ready(a);
            tmem_ready(b);
            if (dual) {
              tmem_ready(c);
              tmem_ready(d);
            }
            if (h == 3) {
              fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive_cluster(drained0);  // the next slice's instructions may overwrite them
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              float v = __uint_as_float(a[i]) + __uint_as_float(b[i]);
              if (dual) v += __uint_as_float(c[i]) + __uint_as_float(d[i]);
              float& x = acc[h >> 1][(h & 1) * 16 + i];
              x = EPI == PF_EPI_PARTIAL ? v : x + v;
            }
          } else if (h == 3) {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(drained0);
          }
        }
        if (EPI == PF_EPI_PARTIAL && tile < P.tiles) {  // out[slice][row][tiles * 128]
          float* dst = P.out + ((size_t)walk.s * P.Mpad + t0) * P.ldo + n;
#pragma unroll
          for (int c = 0; c < 64; ++c)
            if (c < rows_here) dst[(size_t)c * P.ldo] = acc[c >> 5][c & 31];
        }
      }
      if (*abort) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c0 = h * 32;
        if (EPI == PF_EPI_PARTIAL || c0 >= rows_here) continue;  // uniform
        if (EPI != PF_EPI_SWIGLU) {
          if (n < P.n_rows) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c0 + i < rows_here) P.out[(size_t)(t0 + c0 + i) * P.ldo + n] = acc[h][i];
          }
        } else {
          // Even lanes hold gate_j, odd lanes up_j, j = n / 2; the warp's 16 columns j are one k-step
          // block of the output operand.  The lanes of a pair share the tokens; the bf16 parts go
          // through shared memory so that global memory sees whole 16-byte rows.
          const int j0 = (tile * TC_TILE_ROWS + q * 32) >> 1, jl = lane >> 1, odd = lane & 1;
          uint8_t* stg = staging + (size_t)warp * (4 * PF_STG_STRIDE);
          const uint32_t my = (uint32_t)((jl >> 3) * 2) * PF_STG_STRIDE + (uint32_t)(jl & 7) * 2u;
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const float a = acc[h][i], b = acc[h][i + 1];
            const float got = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
            const float gate = odd ? got : a, up = odd ? b : got;
            const float x = __fdividef(gate, 1.f + __expf(-gate)) * up;
            const bf16 hi = __float2bfloat16_rn(x);
            const bf16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
            uint8_t* e = stg + my + (uint32_t)(i + odd) * 16u;
            *reinterpret_cast<bf16*>(e) = hi;
            *reinterpret_cast<bf16*>(e + PF_STG_STRIDE) = lo;
          }
          __syncwarp();
          if (j0 < ((P.n_rows / 2 + 15) & ~15) && c0 + lane < rows_here) {
            uint8_t* blk = P.lay_out.row(P.act_out, t0 + c0 + lane) + (size_t)(j0 >> 4) * P.lay_out.kstep;
#pragma unroll
            for (int hp = 0; hp < 4; ++hp)  // hp = half * 2 + part
              *reinterpret_cast<uint4*>(blk + (hp >> 1) * P.lay_out.half + (hp & 1) * P.lay_out.part_off) =
                  *reinterpret_cast<const uint4*>(stg + (uint32_t)hp * PF_STG_STRIDE + (uint32_t)lane * 16u);
          }
          __syncwarp();
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  cluster_sync();  // the other CTA's memory and barriers are in use up to here
  if (warp == PF_EPI_WARPS + 1) {
    fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
  if (tid == 0 && *abort) atomicOr(P.status, SSD_STATUS_TIMEOUT);
}

template <int EPI>
cudaError_t launch_pf(const PfParams& p, int n_sm, size_t smem, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(tc_prefill_gemm_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return e;
  e = tc_launch_pdl_cluster(tc_prefill_gemm_kernel<EPI>, dim3(2 * std::min(p.n_items, n_sm / 2)), dim3(PF_THREADS), 2,
                            smem, st, p);
  if (e != cudaSuccess) return e;
  count_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tc_prefill_gemm(const TcGemm& g, int epi, const bf16* bias, float* out, int n_sm, cudaStream_t st,
                                   ActLay act_out_lay) {
  if (g.M < 1 || g.M > TC_MAX_ROWS || g.mc < 16 || g.mc > TC_PREFILL_CHUNK || g.ksplit < 1 || (g.K & 7))
    return cudaErrorInvalidValue;
  PfParams p{};
  p.w = g.w;
  p.a = g.a;
  p.n_rows = g.n_rows;
  p.KS = (g.K + 15) / 16;
  p.M = g.M;
  p.Mc = g.mc;
  p.tiles = (g.n_rows + TC_TILE_ROWS - 1) / TC_TILE_ROWS;
  p.nchunk = (g.M + g.mc - 1) / g.mc;
  p.pairs = (p.tiles + 1) / 2;
  p.groups = epi == PF_EPI_PARTIAL ? tc_prefill_groups(g.n_rows, g.M, g.ksplit, n_sm) : 1;
  p.n_items = p.pairs * ((p.nchunk + 1) / 2) * p.groups;
  p.Mpad = tc_round16(g.M);
  p.nslice = g.ksplit;
  p.slice_q = p.KS / g.ksplit;
  p.slice_r = p.KS % g.ksplit;
  p.dual = tc_dual_sets(p.tiles * g.ksplit, n_sm);
  p.bias = bias;
  p.out = out;
  p.ldo = epi == PF_EPI_PARTIAL ? p.tiles * TC_TILE_ROWS : g.n_rows;
  p.act_out = g.act_out;
  p.lay_out = act_out_lay;
  p.status = g.status;
  const size_t stage = (size_t)PF_SK * (TC_WBLOCK + (size_t)p.Mc * 64);
  p.stages = (int)((227 * 1024 - 1024 - PF_STG_BYTES - sizeof(PfShared)) / stage);
  if (p.stages > PF_MAX_STAGES) p.stages = PF_MAX_STAGES;
  const size_t smem = p.stages * stage + PF_STG_BYTES + sizeof(PfShared) + 64;
  switch (epi) {
    case PF_EPI_BIAS: return launch_pf<PF_EPI_BIAS>(p, n_sm, smem, st);
    case PF_EPI_RESIDUAL: return launch_pf<PF_EPI_RESIDUAL>(p, n_sm, smem, st);
    case PF_EPI_PARTIAL: return launch_pf<PF_EPI_PARTIAL>(p, n_sm, smem, st);
    case PF_EPI_SWIGLU: return launch_pf<PF_EPI_SWIGLU>(p, n_sm, smem, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ssd
