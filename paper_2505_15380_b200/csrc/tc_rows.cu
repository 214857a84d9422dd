// Row-wise kernels of the batched verify forward (Eq. 4's decoder pass for more than 16 rows):
// what sits between the tensor-core projections.  Each consumes a projection's partial sums
// (one slab per K slice, added here in a fixed order, so results are bit-reproducible) and
// produces the next projection's input already packed as a tensor-core operand (tc.h).
#include "kernels.h"
#include "tc.h"

namespace ssd {

namespace {

// Columns (k, k + 1), k even, of the token whose row term is `row` (ActLay): bf16 leading parts and
// remainders.
__device__ __forceinline__ void store_pair(uint8_t* row, const ActLay& lay, int k, float x0, float x1) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __low2float(h), x1 - __high2float(h));
  uint8_t* e = row + lay.col(k);
  *reinterpret_cast<__nv_bfloat162*>(e) = h;
  *reinterpret_cast<__nv_bfloat162*>(e + lay.part_off) = l;
}

// Sum over the K slices of a projection's partial sums for two adjacent columns, in slice order
// (bit-reproducible).  The loads of up to 24 slices are in flight together: the kernels that call
// this are one dependent round trip to L2 after another, so every slice waited for separately is
// a microsecond (measured: rounds of eight cost 1.5 us more on 21 slices).  With many rows the
// kernels are built with eight in flight instead, which keeps them at four CTAs per SM: 448 rows
// then still run as one wave.
template <int NF>
__device__ __forceinline__ float2 sum_slices(float2 v, const float* __restrict__ p, size_t slice_stride, int nsplit) {
  for (int s = 0; s < nsplit; s += NF) {
    float2 t[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i)
      t[i] = s + i < nsplit ? __ldcg(reinterpret_cast<const float2*>(p + (size_t)(s + i) * slice_stride))
                            : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      if (s + i < nsplit) {
        v.x += t[i].x;
        v.y += t[i].y;
      }
    }
  }
  return v;
}

constexpr int TC_ROWS_DEEP = 256;  // up to this many rows (CTAs) the deep variant still is one wave

// One CTA per row.  h[m, :] += sum_s part[s][m][:]; out = h / rms(h) * gain, packed.
template <int NF, int MINB>
__global__ void __launch_bounds__(256, MINB)
tc_norm_pack_kernel(float* __restrict__ h, const float* __restrict__ part, int nsplit, int ld_part, int Mpad,
                    ActLay lay, int d, const bf16* __restrict__ gain, float eps, uint8_t* __restrict__ apack) {
  extern __shared__ float row[];
  __shared__ float red[8];
  const int m = blockIdx.x, tid = threadIdx.x;
  tc_pdl_trigger();
  tc_pdl_wait();
  float ss = 0.f;
  for (int j = tid * 2; j < d; j += 512) {
    float2 v = *reinterpret_cast<const float2*>(h + (size_t)m * d + j);
    if (nsplit > 0) {
      v = sum_slices<NF>(v, part + (size_t)m * ld_part + j, (size_t)Mpad * ld_part, nsplit);
      *reinterpret_cast<float2*>(h + (size_t)m * d + j) = v;
    }
    row[j] = v.x;
    row[j + 1] = v.y;
    ss += v.x * v.x + v.y * v.y;
  }
  ss = warp_sum(ss);
  if ((tid & 31) == 0) red[tid >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += red[w];
  const float inv = rsqrtf(tot / (float)d + eps);
  uint8_t* arow = lay.row(apack, m);
  for (int j = tid * 2; j < d; j += 512) {
    const float2 g = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(gain + j));
    store_pair(arow, lay, j, row[j] * inv * g.x, row[j + 1] * inv * g.y);
  }
}

__global__ void tc_pack_rows_kernel(const float* __restrict__ x, int K, ActLay lay, uint8_t* __restrict__ apack) {
  const int m = blockIdx.x;
  uint8_t* arow = lay.row(apack, m);
  for (int j = threadIdx.x * 2; j < K; j += blockDim.x * 2)
    store_pair(arow, lay, j, x[(size_t)m * K + j], x[(size_t)m * K + j + 1]);
}

// One CTA per row: q/k/v = sum of the K slices + bias; rotate q and k by the row's position
// (rotate-half pairs (j, j + hd/2)); q scaled by 1/sqrt(hd) to qrot; K (rotated) and V to the
// cache at slot len + r.  A thread takes two adjacent pairs, so the row needs no shared memory and
// no barrier (hd is a power of two: 1936 rows 17 -> 7 us against staging the row and dividing).
template <int NF, int MINB>
__global__ void __launch_bounds__(256, MINB)
tc_qkv_post_kernel(const float* __restrict__ part, int nsplit, int ld_part, int Mpad,
                   const bf16* __restrict__ bias, const float* __restrict__ cs, float* __restrict__ qrot,
                   bf16* __restrict__ kv_layer, const int32_t* __restrict__ len, RowMap rm, int cap, int Hq,
                   int Hkv, int hd_log2, float scale, const int32_t* __restrict__ page_table, int max_pages,
                   int32_t* status) {
  const int m = blockIdx.x, tid = threadIdx.x;
  tc_pdl_trigger();
  tc_pdl_wait();
  const int2 br = row_at(rm, m);
  const int b = br.x, pos = len[b] + br.y, hd = 1 << hd_log2, half = hd >> 1;
  // where this row's K and V live: the stream's slice of a contiguous cache, or its page
  size_t owner = (size_t)b, rows_per = (size_t)cap, slot = (size_t)pos;
  bool store = pos >= 0 && pos < cap;  // never write outside the stream's slice of the cache
  if (!store && tid == 0) atomicOr(status, SSD_STATUS_KV_OVERFLOW);
  if (page_table && store) {
    const int pg = page_table[(size_t)b * max_pages + pos / TC_PAGE_TOKENS];
    store = pg >= 0;  // no page was granted (pool exhausted): flagged by the page kernel
    owner = (size_t)max(pg, 0);
    rows_per = TC_PAGE_TOKENS;
    slot = (size_t)(pos % TC_PAGE_TOKENS);
  }
  const float* c = cs + (size_t)m * hd;
  const float* prow = part + (size_t)m * ld_part;
  const int n_tasks = (Hq + 2 * Hkv) << (hd_log2 - 2);  // a quarter of the row
  for (int i = tid; i < n_tasks; i += 256) {
    const int hh = i >> (hd_log2 - 2), j = (i & ((half >> 1) - 1)) * 2, col = (hh << hd_log2) + j;
    float2 x = make_float2(0.f, 0.f), y = x;
    if (bias) {
      x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(bias + col));
      y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(bias + col + half));
    }
    x = sum_slices<NF>(x, prow + col, (size_t)Mpad * ld_part, nsplit);
    y = sum_slices<NF>(y, prow + col + half, (size_t)Mpad * ld_part, nsplit);
    if (hh < Hq + Hkv) {
      const float4 r = *reinterpret_cast<const float4*>(c + 2 * j);  // cos, sin of dims j and j + 1
      const float2 u = make_float2(x.x * r.x - y.x * r.y, x.y * r.z - y.y * r.w);
      const float2 v = make_float2(y.x * r.x + x.x * r.y, y.y * r.z + x.y * r.w);
      x = u;
      y = v;
    }
    if (hh < Hq) {
      float* q = qrot + ((size_t)m * Hq << hd_log2) + col;
      *reinterpret_cast<float2*>(q) = make_float2(x.x * scale, x.y * scale);
      *reinterpret_cast<float2*>(q + half) = make_float2(y.x * scale, y.y * scale);
    } else if (store) {
      const int which = hh >= Hq + Hkv, g = hh - Hq - which * Hkv;
      bf16* dst = kv_layer + (((owner * 2 + which) * Hkv + g) * rows_per + slot) * hd + j;
      *reinterpret_cast<__nv_bfloat162*>(dst) = __floats2bfloat162_rn(x.x, x.y);
      *reinterpret_cast<__nv_bfloat162*>(dst + half) = __floats2bfloat162_rn(y.x, y.y);
    }
  }
}

}  // namespace

void launch_tc_norm_pack(float* h, const float* part, int nsplit, int ld_part, int M, ActLay lay, int d,
                         const bf16* gain, float eps, uint8_t* apack, cudaStream_t st) {
  if (!part)
    tc_launch_pdl(tc_norm_pack_kernel<1, 8>, dim3(M), dim3(256), (size_t)d * 4, st, h, part, 0, ld_part,
                  tc_round16(M), lay, d, gain, eps, apack);
  else if (M <= TC_ROWS_DEEP)
    tc_launch_pdl(tc_norm_pack_kernel<24, 1>, dim3(M), dim3(256), (size_t)d * 4, st, h, part, part ? nsplit : 0,
                  ld_part, tc_round16(M), lay, d, gain, eps, apack);
  else
    tc_launch_pdl(tc_norm_pack_kernel<8, 4>, dim3(M), dim3(256), (size_t)d * 4, st, h, part, part ? nsplit : 0,
                  ld_part, tc_round16(M), lay, d, gain, eps, apack);
  count_launch();
}

void launch_tc_pack_rows(const float* x, int M, int K, uint8_t* apack, cudaStream_t st) {
  tc_pack_rows_kernel<<<M, 128, 0, st>>>(x, K, tc_act_lay(tc_chunks(M).rows, K), apack);
  count_launch();
}

void launch_tc_qkv_post(const float* part, int nsplit, int ld_part, int Mpad, const bf16* bias,
                        const float* cs, float* qrot, bf16* kv_layer, const int32_t* len, RowMap rm,
                        int cap, int Hq, int Hkv, int hd, const int32_t* page_table, int max_pages,
                        int32_t* status, cudaStream_t st) {
  const int M = row_count(rm);
  const int hl = hd == 32 ? 5 : hd == 64 ? 6 : 7;
  if (nsplit == 1)
    tc_launch_pdl(tc_qkv_post_kernel<1, 6>, dim3(M), dim3(256), 0, st, part, nsplit, ld_part, Mpad, bias, cs, qrot,
                  kv_layer, len, rm, cap, Hq, Hkv, hl, 1.0f / sqrtf((float)hd), page_table, max_pages, status);
  else if (M <= TC_ROWS_DEEP)
    tc_launch_pdl(tc_qkv_post_kernel<24, 1>, dim3(M), dim3(256), 0, st, part, nsplit, ld_part, Mpad, bias, cs, qrot,
                  kv_layer, len, rm, cap, Hq, Hkv, hl, 1.0f / sqrtf((float)hd), page_table, max_pages, status);
  else
    tc_launch_pdl(tc_qkv_post_kernel<8, 4>, dim3(M), dim3(256), 0, st, part, nsplit, ld_part, Mpad, bias, cs, qrot,
                  kv_layer, len, rm, cap, Hq, Hkv, hl, 1.0f / sqrtf((float)hd), page_table, max_pages, status);
  count_launch();
}

namespace {

__device__ __forceinline__ void page_ensure_stream(const int32_t* __restrict__ len, int b, int rows, int32_t* page_table,
                                                   int32_t* pages_used, const int32_t* __restrict__ free_stack,
                                                   int32_t* free_top, int max_pages, int32_t* status) {
  int need = (len[b] + rows + TC_PAGE_TOKENS - 1) / TC_PAGE_TOKENS;
  if (need > max_pages) {  // rows beyond the block table are not written (flagged as an overflow)
    atomicOr(status, SSD_STATUS_KV_OVERFLOW);
    need = max_pages;
  }
  int used = pages_used[b];
  while (used < need) {
    const int idx = atomicSub(free_top, 1) - 1;  // pops from different streams race only on this counter
    if (idx < 0) {
      atomicAdd(free_top, 1);
      atomicOr(status, SSD_STATUS_KV_OVERFLOW);  // the pool is exhausted: the rows of this page are dropped
      break;
    }
    page_table[(size_t)b * max_pages + used] = free_stack[idx];
    ++used;
  }
  pages_used[b] = used;
}

__global__ void page_ensure_kernel(const int32_t* __restrict__ len, RowMap rm, int32_t* page_table,
                                   int32_t* pages_used, const int32_t* __restrict__ free_stack, int32_t* free_top,
                                   int max_pages, int32_t* status) {
  tc_pdl_enter();
  const int bi = blockIdx.x * blockDim.x + threadIdx.x;
  if (bi < rm.nb)
    page_ensure_stream(len, rm.b0 + bi, rm.R, page_table, pages_used, free_stack, free_top, max_pages, status);
}

// The streams of a prefill chunk, one after the other: the pages a prompt gets do not depend on
// which thread was first.
__global__ void page_ensure_segs_kernel(const int32_t* __restrict__ len, const __grid_constant__ PrefillSegs P,
                                        int32_t* page_table, int32_t* pages_used,
                                        const int32_t* __restrict__ free_stack, int32_t* free_top, int max_pages,
                                        int32_t* status) {
  tc_pdl_enter();
  for (int q = 0; q < P.n; ++q)
    page_ensure_stream(len, P.s[q].stream, P.s[q].count, page_table, pages_used, free_stack, free_top, max_pages, status);
}

__global__ void page_release_kernel(const int32_t* __restrict__ len, int B, int32_t* page_table, int32_t* pages_used,
                                    int32_t* free_stack, int32_t* free_top, int max_pages) {
  tc_pdl_enter();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int keep = (max(len[b], 0) + TC_PAGE_TOKENS - 1) / TC_PAGE_TOKENS;
  int used = pages_used[b];
  while (used > keep) {
    --used;
    const int idx = atomicAdd(free_top, 1);
    free_stack[idx] = page_table[(size_t)b * max_pages + used];
    page_table[(size_t)b * max_pages + used] = -1;
  }
  pages_used[b] = used;
}

}  // namespace

void launch_page_ensure(const int32_t* len, RowMap rm, int32_t* page_table, int32_t* pages_used,
                        int32_t* free_stack, int32_t* free_top, int max_pages, int32_t* status,
                        cudaStream_t st) {
  tc_launch_pdl(page_ensure_kernel, dim3((rm.nb + 127) / 128), dim3(128), 0, st, len, rm, page_table, pages_used, free_stack, free_top,
                                                         max_pages, status);
  count_launch();
}

void launch_page_ensure_segs(const int32_t* len, const PrefillSegs& segs, int32_t* page_table, int32_t* pages_used,
                             int32_t* free_stack, int32_t* free_top, int max_pages, int32_t* status, cudaStream_t st) {
  tc_launch_pdl(page_ensure_segs_kernel, dim3(1), dim3(1), 0, st, len, segs, page_table, pages_used, free_stack, free_top, max_pages, status);
  count_launch();
}

void launch_page_release(const int32_t* len, int B, int32_t* page_table, int32_t* pages_used,
                         int32_t* free_stack, int32_t* free_top, int max_pages, cudaStream_t st) {
  tc_launch_pdl(page_release_kernel, dim3((B + 127) / 128), dim3(128), 0, st, len, B, page_table, pages_used, free_stack, free_top,
                                                      max_pages);
  count_launch();
}

}  // namespace ssd
