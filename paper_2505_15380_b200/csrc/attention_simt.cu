// Generic verify attention (Eq. 4: the gamma+1 new rows of a stream attend to the cached prefix
// and, causally, to each other), grouped-query, any storage type, split over the key axis.
//
// Grid (split, kv head, stream).  A CTA stages its chunk of ATTN_CHUNK keys/values (fp32) and all
// G*R query rows of the kv head in shared memory; each warp then walks its rows with an online
// softmax (lane = key for the scores, lane = channel for the weighted sum) and writes an
// un-normalised partial (acc[hd], running max, running sum) per (row, head, split).  The O projection
// merges the partials of a row by log-sum-exp weights as it stages them (gemm_simt.cu), or, where
// they are many, a second kernel does.
//
// q comes straight from the projection and is rotated while it is staged; the chunk that holds a new
// position rotates its key, appends key and value to the cache and stages what it stored.  (As a
// launch of its own that cost 3.5 us per layer.)
#include <math_constants.h>

#include "kernels.h"
#include "tc.h"

namespace ssd {

// A warp per query row of the kv head, as far as that goes: a row is a chain of shuffles and sums, and three
// rows one after the other took 12 us of a 68 us forward (4 warps; 10 rows).
constexpr int ATTN_MIN_WARPS = 4, ATTN_MAX_WARPS = 16;

template <typename T, int HD>
__global__ void __launch_bounds__(ATTN_MAX_WARPS * 32)
attn_split_kernel(const float* __restrict__ qkv, const float* __restrict__ cs, T* __restrict__ kv_layer,
                  const int32_t* __restrict__ len, RowMap rm, int cap, int Hq, int Hkv, float scale,
                  float* __restrict__ part, int nsplit_max, int32_t* status) {
  tc_pdl_enter();
  constexpr int NI = HD / 32;
  constexpr int KP = HD + 1;  // padded key row: lane = key reads are conflict-free
  extern __shared__ __align__(16) float smem[];
  const int s = blockIdx.x, g = blockIdx.y, bi = blockIdx.z, b = rm.b0 + bi;
  const int R = rm.R, G = Hq / Hkv, NQ = G * R;
  const int L = len[b];
  const int total = min(L + R, cap);
  const int k_begin = s * ATTN_CHUNK;
  if (s == 0 && g == 0 && threadIdx.x == 0 && (L < 0 || L + R > cap))  // never write outside the stream's slice of the cache
    atomicOr(status, SSD_STATUS_KV_OVERFLOW);
  if (k_begin >= total) return;
  const int k_end = min(k_begin + ATTN_CHUNK, total);
  const int nk = k_end - k_begin;
  float* Ks = smem;                      // [ATTN_CHUNK][KP]
  float* Vs = Ks + ATTN_CHUNK * KP;      // [ATTN_CHUNK][HD]
  float* Qs = Vs + ATTN_CHUNK * HD;      // [NQ][HD]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* kbase = kv_layer + (((size_t)b * 2 + 0) * Hkv + g) * (size_t)cap * HD + (size_t)k_begin * HD;
  T* vbase = kv_layer + (((size_t)b * 2 + 1) * Hkv + g) * (size_t)cap * HD + (size_t)k_begin * HD;
  const int ld = (Hq + 2 * Hkv) * HD, n_old = max(0, min(nk, L - k_begin));
  for (int i = tid; i < n_old * (HD / 8); i += blockDim.x) {
    int key = i / (HD / 8), c = i % (HD / 8);
    float kx[8], vx[8];
    load8(kbase + (size_t)key * HD + c * 8, kx);
    load8(vbase + (size_t)key * HD + c * 8, vx);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      Ks[key * KP + c * 8 + e] = kx[e];
      Vs[key * HD + c * 8 + e] = vx[e];
    }
  }
  for (int i = tid; i < (nk - n_old) * (HD / 2); i += blockDim.x) {  // the new positions: rotary pairs
    const int key = n_old + i / (HD / 2), j = i % (HD / 2), m = bi * R + k_begin + key - L;
    const float* kr = qkv + (size_t)m * ld + (Hq + g) * HD + j;
    const float x1 = kr[0], x2 = kr[HD / 2], v1 = kr[Hkv * HD], v2 = kr[Hkv * HD + HD / 2];
    const float2 c = *reinterpret_cast<const float2*>(cs + ((size_t)m * (HD / 2) + j) * 2);
    const T k1 = from_f32<T>(x1 * c.x - x2 * c.y), k2 = from_f32<T>(x2 * c.x + x1 * c.y);
    const T w1 = from_f32<T>(v1), w2 = from_f32<T>(v2);
    T *kd = kbase + (size_t)key * HD + j, *vd = vbase + (size_t)key * HD + j;
    kd[0] = k1;
    kd[HD / 2] = k2;
    vd[0] = w1;
    vd[HD / 2] = w2;
    Ks[key * KP + j] = to_f32<T>(k1);
    Ks[key * KP + j + HD / 2] = to_f32<T>(k2);
    Vs[key * HD + j] = to_f32<T>(w1);
    Vs[key * HD + j + HD / 2] = to_f32<T>(w2);
  }
  for (int i = tid; i < NQ * (HD / 2); i += blockDim.x) {
    const int row = i / (HD / 2), j = i % (HD / 2);  // row = r * G + hl
    const int r = row / G, hl = row % G, m = bi * R + r;
    const float* q = qkv + (size_t)m * ld + (g * G + hl) * HD + j;
    const float x1 = q[0], x2 = q[HD / 2];
    const float2 c = *reinterpret_cast<const float2*>(cs + ((size_t)m * (HD / 2) + j) * 2);
    Qs[row * HD + j] = (x1 * c.x - x2 * c.y) * scale;
    Qs[row * HD + j + HD / 2] = (x2 * c.x + x1 * c.y) * scale;
  }
  __syncthreads();
  for (int row = warp; row < NQ; row += (int)blockDim.x >> 5) {
    const int r = row / G, hl = row % G;
    const int last_visible = L + r;      // row r sees keys 0..len+r
    float m_run = -CUDART_INF_F, l_run = 0.f, acc[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) acc[i] = 0.f;
    const float* q = Qs + row * HD;
    for (int t0 = 0; t0 < nk; t0 += 32) {
      const int kl = t0 + lane;
      const bool valid = kl < nk && (k_begin + kl) <= last_visible;
      float sc = 0.f;
      if (valid) {
        const float* kr = Ks + kl * KP;
#pragma unroll 8
        for (int d = 0; d < HD; ++d) sc = fmaf(q[d], kr[d], sc);
      }
      float tmax = warp_max(valid ? sc : -CUDART_INF_F);
      if (tmax == -CUDART_INF_F) continue;  // nothing visible in this tile (uniform per warp)
      float m_new = fmaxf(m_run, tmax);
      float p = valid ? expf(sc - m_new) : 0.f;
      float corr = expf(m_run - m_new);     // m_run = -inf gives 0
      l_run = l_run * corr + warp_sum(p);
#pragma unroll
      for (int i = 0; i < NI; ++i) acc[i] *= corr;
      const int lim = min(32, nk - t0);
#pragma unroll 8
      for (int kk = 0; kk < lim; ++kk) {
        float pk = __shfl_sync(0xffffffffu, p, kk);
        const float* vr = Vs + (t0 + kk) * HD;
#pragma unroll
        for (int i = 0; i < NI; ++i) acc[i] = fmaf(pk, vr[lane + 32 * i], acc[i]);
      }
      m_run = m_new;
    }
    const int m = bi * R + r, h = g * G + hl;
    float* dst = part + (((size_t)m * Hq + h) * nsplit_max + s) * (HD + 2);
#pragma unroll
    for (int i = 0; i < NI; ++i) dst[lane + 32 * i] = acc[i];
    if (lane == 0) {
      dst[HD] = m_run;
      dst[HD + 1] = l_run;
    }
  }
}

template <int HD>
__global__ void attn_merge_kernel(const float* __restrict__ part, const int32_t* __restrict__ len,
                                  RowMap rm, int cap, int Hq, int nsplit_max, float* __restrict__ out) {
  tc_pdl_enter();
  const int h = blockIdx.x, m = blockIdx.y;
  const int bi = m / rm.R, b = rm.b0 + bi;
  const int total = min(len[b] + rm.R, cap);
  const int ns = (total + ATTN_CHUNK - 1) / ATTN_CHUNK;
  const float* src = part + ((size_t)m * Hq + h) * nsplit_max * (HD + 2);
  float m_tot = -CUDART_INF_F;
  for (int s = 0; s < ns; ++s) m_tot = fmaxf(m_tot, src[s * (HD + 2) + HD]);
  float denom = 0.f;
  for (int s = 0; s < ns; ++s) {
    float ms = src[s * (HD + 2) + HD];
    if (ms != -CUDART_INF_F) denom += expf(ms - m_tot) * src[s * (HD + 2) + HD + 1];
  }
  for (int d = threadIdx.x; d < HD; d += blockDim.x) {
    float o = 0.f;
    for (int s = 0; s < ns; ++s) {
      float ms = src[s * (HD + 2) + HD];
      if (ms != -CUDART_INF_F) o += expf(ms - m_tot) * src[s * (HD + 2) + d];
    }
    out[((size_t)m * Hq + h) * HD + d] = o / denom;
  }
}

template <typename T, int HD>
static cudaError_t launch_t(const float* qkv, const float* cs, void* kv_layer, const int32_t* len, RowMap rm,
                            int cap, int Hq, int Hkv, float* part, int nsplit_max, int32_t* status, cudaStream_t st) {
  const int NQ = (Hq / Hkv) * rm.R;
  size_t smem = sizeof(float) * ((size_t)ATTN_CHUNK * (HD + 1) + (size_t)ATTN_CHUNK * HD + (size_t)NQ * HD);
  auto kern = attn_split_kernel<T, HD>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  dim3 grid(nsplit_max, Hkv, rm.nb);
  const int warps = NQ < ATTN_MIN_WARPS ? ATTN_MIN_WARPS : NQ > ATTN_MAX_WARPS ? ATTN_MAX_WARPS : NQ;
  tc_launch_pdl(kern, grid, dim3(warps * 32), smem, st, qkv, cs, (T*)kv_layer, len, rm, cap, Hq, Hkv,
                1.0f / sqrtf((float)HD), part, nsplit_max, status);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_attention_simt(int dtype, const float* qkv, const float* cs, void* kv_layer, const int32_t* len,
                                  RowMap rm, int cap, int Hq, int Hkv, int hd, float* part, int nsplit_max,
                                  int32_t* status, cudaStream_t st) {
#define SSD_ATTN_CASE(T)                                                                          \
  switch (hd) {                                                                                   \
    case 32: return launch_t<T, 32>(qkv, cs, kv_layer, len, rm, cap, Hq, Hkv, part, nsplit_max, status, st);  \
    case 64: return launch_t<T, 64>(qkv, cs, kv_layer, len, rm, cap, Hq, Hkv, part, nsplit_max, status, st);  \
    case 128: return launch_t<T, 128>(qkv, cs, kv_layer, len, rm, cap, Hq, Hkv, part, nsplit_max, status, st); \
  }
  if (dtype == 0) {
    SSD_ATTN_CASE(float)
  } else {
    SSD_ATTN_CASE(bf16)
  }
#undef SSD_ATTN_CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_attention_merge(const float* part, const int32_t* len, RowMap rm, int cap, int Hq, int hd,
                                   int nsplit_max, float* out, cudaStream_t st) {
  const dim3 grid(Hq, rm.nb * rm.R), block(hd < 64 ? 32 : 64);
  switch (hd) {
    case 32: tc_launch_pdl(attn_merge_kernel<32>, grid, block, 0, st, part, len, rm, cap, Hq, nsplit_max, out); break;
    case 64: tc_launch_pdl(attn_merge_kernel<64>, grid, block, 0, st, part, len, rm, cap, Hq, nsplit_max, out); break;
    case 128: tc_launch_pdl(attn_merge_kernel<128>, grid, block, 0, st, part, len, rm, cap, Hq, nsplit_max, out); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

}  // namespace ssd
