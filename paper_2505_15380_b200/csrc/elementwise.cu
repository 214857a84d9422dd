// Small memory-bound pieces of the verify forward: the rows that enter it (ids, embedding, rotary
// table), RMSNorm of wide models, and the bookkeeping of lengths
// (the decoder is the Qwen2.5-style Transformer of Sec. 3.1).
#include <atomic>

#include "kernels.h"
#include "tc.h"

namespace ssd {

static std::atomic<uint64_t> g_launches{0};
void count_launch(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }
uint64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

// The rows that enter a forward: ids (given, or of a verify step: row 0 of a stream is its pending token,
// the others its draft), embedding, and cos/sin of position * inv_freq in double, rounded once.  One launch:
// as three it was 8 us of launches in front of a model of two layers.
template <typename T>
__global__ void embed_kernel(const T* __restrict__ table, int vocab_in, int d, const int32_t* __restrict__ row_ids,
                             const int32_t* __restrict__ pending, const int32_t* __restrict__ draft,
                             const int32_t* __restrict__ len, RowMap rm, const double* __restrict__ inv_freq, int half,
                             float* __restrict__ h, float* __restrict__ cs, int32_t* status) {
  tc_pdl_enter();
  const int m = blockIdx.x;
  const int2 br = row_at(rm, m);
  int id = row_ids ? row_ids[m] : br.y == 0 ? pending[br.x] : draft[(size_t)br.x * (rm.R - 1) + br.y - 1];
  const double pos = (double)(len[br.x] + br.y);
  if (id < 0 || id >= vocab_in) {
    if (threadIdx.x == 0) atomicOr(status, SSD_STATUS_BAD_TOKEN);
    id = min(max(id, 0), vocab_in - 1);
  }
  const T* src = table + (size_t)id * d;
  for (int j = threadIdx.x; j < d; j += blockDim.x) h[(size_t)m * d + j] = to_f32<T>(src[j]);
  for (int j = threadIdx.x; j < half; j += blockDim.x) {
    double s, c;
    sincos(pos * inv_freq[j], &s, &c);
    cs[((size_t)m * half + j) * 2 + 0] = (float)c;
    cs[((size_t)m * half + j) * 2 + 1] = (float)s;
  }
}

void launch_embed(int dtype, const void* table, int vocab_in, int d, const int32_t* row_ids, const int32_t* pending,
                  const int32_t* draft, const int32_t* len, RowMap rm, const double* inv_freq, int half, float* h,
                  float* cs, int32_t* status, cudaStream_t st) {
  if (dtype == 0)
    tc_launch_pdl(embed_kernel<float>, dim3(row_count(rm)), dim3(128), 0, st, (const float*)table, vocab_in, d, row_ids,
                  pending, draft, len, rm, inv_freq, half, h, cs, status);
  else
    tc_launch_pdl(embed_kernel<bf16>, dim3(row_count(rm)), dim3(128), 0, st, (const bf16*)table, vocab_in, d, row_ids,
                  pending, draft, len, rm, inv_freq, half, h, cs, status);
  count_launch();
}

template <typename T>
__global__ void rmsnorm_kernel(const float* __restrict__ h, const T* __restrict__ gain,
                               float* __restrict__ out, int d, float eps) {
  tc_pdl_enter();
  __shared__ float red[32];
  int m = blockIdx.x;
  const float* x = h + (size_t)m * d;
  float ss = 0.f;
  for (int j = threadIdx.x; j < d; j += blockDim.x) ss += x[j] * x[j];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) red[0] = rsqrtf(v / (float)d + eps);
  }
  __syncthreads();
  float inv = red[0];
  for (int j = threadIdx.x; j < d; j += blockDim.x)
    out[(size_t)m * d + j] = x[j] * inv * to_f32<T>(gain[j]);
}

void launch_rmsnorm(int dtype, const float* h, const void* gain, float* out, int M, int d, float eps,
                    cudaStream_t st) {
  if (dtype == 0)
    tc_launch_pdl(rmsnorm_kernel<float>, dim3(M), dim3(256), 0, st, h, (const float*)gain, out, d, eps);
  else
    tc_launch_pdl(rmsnorm_kernel<bf16>, dim3(M), dim3(256), 0, st, h, (const bf16*)gain, out, d, eps);
  count_launch();
}

// Prefill bookkeeping: len[b] += add; optionally pending[b] = ids[pending_index].
__global__ void advance_len_kernel(int32_t* len, int32_t* pending, int b, int add,
                                   const int32_t* ids, int pending_index) {
  len[b] += add;
  if (pending_index >= 0) pending[b] = ids[pending_index];
}

void launch_advance_len(int32_t* len, int32_t* pending, int b, int add, const int32_t* ids,
                        int pending_index, cudaStream_t st) {
  advance_len_kernel<<<1, 1, 0, st>>>(len, pending, b, add, ids, pending_index);
  count_launch();
}

// Rows of a prefill chunk: ids, (stream, r) of every row, the attention's tiles.
__global__ void prefill_stage_kernel(const __grid_constant__ PrefillSegs P, const int32_t* __restrict__ ids,
                                     int32_t* __restrict__ row_ids, int2* __restrict__ rows,
                                     int4* __restrict__ tiles) {
  tc_pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < P.n_rows) {
    int q = 0;
    while (q + 1 < P.n && i >= P.s[q + 1].m0) ++q;  // segments without rows share their m0: the last one wins,
    while (P.s[q].count == 0) --q;                  // so step back to the one that has the row
    const int r = i - P.s[q].m0;
    row_ids[i] = ids[P.s[q].src + r];
    rows[i] = make_int2(P.s[q].stream, r);
  }
  if (i < P.n_tiles) {
    int q = 0;
    while (q + 1 < P.n && i >= P.s[q + 1].tile0) ++q;
    while (P.s[q].count == 0) --q;
    const int r = (i - P.s[q].tile0) * P.tile_rows;
    tiles[i] = make_int4(P.s[q].stream, P.s[q].m0 + r, r, min(P.tile_rows, P.s[q].count - r));
  }
}

void launch_prefill_stage(const PrefillSegs& segs, const int32_t* ids, int32_t* row_ids, int2* rows, int4* tiles,
                          cudaStream_t st) {
  tc_launch_pdl(prefill_stage_kernel, dim3((segs.n_rows + 127) / 128), dim3(128), 0, st, segs, ids, row_ids, rows,
                tiles);
  count_launch();
}

// The chunk's rows are in the cache: lengths grow, prompts that end here leave their last id pending.
__global__ void prefill_advance_kernel(const __grid_constant__ PrefillSegs P, const int32_t* __restrict__ ids,
                                       int32_t* len, int32_t* pending) {
  tc_pdl_enter();
  const int q = threadIdx.x;
  if (q >= P.n) return;
  len[P.s[q].stream] += P.s[q].count;
  if (P.s[q].pend_src >= 0) pending[P.s[q].stream] = ids[P.s[q].pend_src];
}

void launch_prefill_advance(const PrefillSegs& segs, const int32_t* ids, int32_t* len, int32_t* pending,
                            cudaStream_t st) {
  tc_launch_pdl(prefill_advance_kernel, dim3(1), dim3(PREFILL_SEGS), 0, st, segs, ids, len, pending);
  count_launch();
}

__global__ void fetch_words_kernel(const uint32_t* __restrict__ host, uint32_t* __restrict__ dst, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t v = i < n ? host[i] : 0u;  // ahead of the wait: nothing on the device writes it
  tc_pdl_enter();
  if (i < n) dst[i] = v;
}

void launch_fetch_words(const uint32_t* host, uint32_t* dst, int n, cudaStream_t st) {
  tc_launch_pdl(fetch_words_kernel, dim3((n + 127) / 128), dim3(128), 0, st, host, dst, n);
  count_launch();
}

// O(1) rollback from device arrays: len[b] = src_len[b] (clamped to the capacity).
__global__ void kv_restore_kernel(int32_t* len, int32_t* pending, const int32_t* src_len,
                                  const int32_t* src_pending, int B, int cap) {
  tc_pdl_enter();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  len[b] = min(max(src_len[b], 0), cap);
  pending[b] = src_pending[b];
}

void launch_kv_restore(int32_t* len, int32_t* pending, const int32_t* src_len,
                       const int32_t* src_pending, int B, int cap, cudaStream_t st) {
  tc_launch_pdl(kv_restore_kernel, dim3((B + 127) / 128), dim3(128), 0, st, len, pending, src_len, src_pending, B,
                cap);
  count_launch();
}

}  // namespace ssd
