// Generic weight-streaming projection kernel (any shape; fp32 or bf16 weights; fp32 activations
// and accumulation): C[M,N] = A[M,K] * W[N,K]^T.  One warp owns two adjacent weight rows (output
// columns) and streams them once with 16-byte loads while MT activation rows sit in shared memory
// (staged K_CHUNK columns at a time); the K dimension is split over the lanes and reduced with
// shuffles.  The projections of the verify forward (Sec. 3.1 decoder) are skinny
// (M = B * (gamma+1) rows), so the weights dominate the bytes.
//
// Small models are bound by the number of launches (3.4 us each) and their dependent trips to L2: so the
// norm in front of a projection and the merge of the attention's key splits happen while the
// rows are staged (every CTA does it for its 8 rows), and a CTA's first weights are requested before it
// waits for its predecessor.  fp32 model of two layers: 23 launches, 79 us -> 15.
#include <math_constants.h>

#include "kernels.h"
#include "tc.h"

namespace ssd {

constexpr int GEMM_MT = 8;        // activation rows per CTA pass
constexpr int GEMM_WARPS = 8;     // warps per CTA, two columns each
constexpr int GEMM_KC = 2048;     // activation columns staged per pass (8 * 2048 * 4 B = 64 KB)
static_assert(GEMM_FUSED_K <= GEMM_KC, "a fused source is staged in one pass");
static_assert(GEMM_MT == GEMM_WARPS, "a warp normalises a row");
enum Source { SRC_PLAIN = 0, SRC_NORM = 1, SRC_MERGE = 2 };

// Columns k .. k + 3 of a row's attention output, from its partials (fixed order).
__device__ __forceinline__ float4 merged4(const SimtSrc& S, int m, int k) {
  const int h = k / S.hd, d = k - h * S.hd, ld = S.hd + 2;
  const int ns = (min(S.len[S.rm.b0 + m / S.rm.R] + S.rm.R, S.cap) + ATTN_CHUNK - 1) / ATTN_CHUNK;
  const float* p = S.part + ((size_t)m * S.Hq + h) * S.nsplit_max * ld;
  float mt = -CUDART_INF_F, den = 0.f;
  for (int s = 0; s < ns; ++s) mt = fmaxf(mt, p[s * ld + S.hd]);
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
  for (int s = 0; s < ns; ++s) {
    const float2 ml = *reinterpret_cast<const float2*>(p + s * ld + S.hd);
    const float2 a = *reinterpret_cast<const float2*>(p + s * ld + d), b = *reinterpret_cast<const float2*>(p + s * ld + d + 2);
    const bool seen = ml.x != -CUDART_INF_F;  // a split of which this row sees nothing leaves no output
    const float e = seen ? expf(ml.x - mt) : 0.f;
    den += e * (seen ? ml.y : 0.f);
    o.x += e * (seen ? a.x : 0.f);
    o.y += e * (seen ? a.y : 0.f);
    o.z += e * (seen ? b.x : 0.f);
    o.w += e * (seen ? b.y : 0.f);
  }
  return make_float4(o.x / den, o.y / den, o.z / den, o.w / den);
}

template <typename T, int EPI, int KS, int SRC>
__global__ void __launch_bounds__(GEMM_WARPS * 32)
gemm_simt_kernel(const SimtSrc S, const T* __restrict__ W,
                 const T* __restrict__ bias, float* __restrict__ C, int ldc, int M, int N, int K) {
  // KS warps share one pair of columns, each taking every KS-th 256-element slice of K; the
  // CTA covers NG = GEMM_WARPS / KS column pairs.
  constexpr int NG = GEMM_WARPS / KS;
  extern __shared__ __align__(16) float As[];  // [GEMM_MT][kc]
  __shared__ float red[GEMM_WARPS][GEMM_MT][2];
  const int m0 = blockIdx.y * GEMM_MT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = warp / KS, ks = warp % KS;
  const int n0 = (blockIdx.x * NG + grp) * 2;
  const bool active = n0 < N;
  const bool has1 = n0 + 1 < N;
  // bf16 weights lie in groups of 8 rows: a lane's 16 bytes of two neighbouring rows are one sector
  constexpr bool GROUPS = sizeof(T) == 2;
  constexpr int STEP = GROUPS ? 64 : 8;  // elements from 8 columns of a row to the next 8
  const int r0 = active ? n0 : 0, r1 = has1 ? n0 + 1 : r0, steps = (K + 15) / 16;
  const T* w0 = W + (GROUPS ? chain_elem(r0, 0, steps, S.w_hd_log2) : (size_t)r0 * K);
  const T* w1 = W + (GROUPS ? chain_elem(r1, 0, steps, S.w_hd_log2) : (size_t)r1 * K);
  const int kc_max = K < GEMM_KC ? K : GEMM_KC;
  float acc0[GEMM_MT], acc1[GEMM_MT];
#pragma unroll
  for (int r = 0; r < GEMM_MT; ++r) acc0[r] = acc1[r] = 0.f;
  // two 16-byte chunks per column in flight before any arithmetic
  float x0[8], x1[8], y0[8], y1[8];
  auto load_weights = [&](int k0, int c, int nch) {
    const int c2 = c + 32 * KS < nch ? c + 32 * KS : c;
    const size_t at = (size_t)(k0 / 8 + c) * STEP, at2 = (size_t)(k0 / 8 + c2) * STEP;
    load8_stream(w0 + at, x0);
    load8_stream(w1 + at, x1);
    load8_stream(w0 + at2, y0);
    load8_stream(w1 + at2, y1);
  };
  const int c_first = lane + 32 * ks;
  if (active && c_first < kc_max >> 3) load_weights(0, c_first, kc_max >> 3);
  // what the epilogue reads, requested now
  const bool mine = active && ks == 0 && lane < GEMM_MT && m0 + lane < M;
  const size_t at = (size_t)(m0 + lane) * ldc + n0;
  float b0 = 0.f, b1 = 0.f, c0 = 0.f, c1 = 0.f;
  if (EPI == EPI_STORE_F32 && mine && bias) {
    b0 = to_f32<T>(bias[n0]);
    b1 = has1 ? to_f32<T>(bias[n0 + 1]) : 0.f;
  }
  tc_pdl_enter();
  if (EPI == EPI_RESIDUAL && mine) {
    c0 = C[at];
    c1 = has1 ? C[at + 1] : 0.f;
  }
  for (int k0 = 0; k0 < K; k0 += GEMM_KC) {
    const int kc = min(GEMM_KC, K - k0);  // multiple of 8
    __syncthreads();
    if (SRC == SRC_NORM) {
      float* row = As + (size_t)warp * kc_max;
      const float* src = S.a + (size_t)min(m0 + warp, M - 1) * S.lda;
      float ss = 0.f;
      for (int c = lane; c < kc >> 2; c += 32) {
        const float4 v = *reinterpret_cast<const float4*>(src + c * 4);
        *reinterpret_cast<float4*>(row + c * 4) = v;
        ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
      }
      const float inv = rsqrtf(warp_sum(ss) / (float)K + S.eps);
      const T* gain = static_cast<const T*>(S.gain);
      for (int c = lane; c < kc >> 2; c += 32) {  // each lane's own columns
        float4 v = *reinterpret_cast<const float4*>(row + c * 4);
        v.x = v.x * inv * to_f32<T>(gain[c * 4]);
        v.y = v.y * inv * to_f32<T>(gain[c * 4 + 1]);
        v.z = v.z * inv * to_f32<T>(gain[c * 4 + 2]);
        v.w = v.w * inv * to_f32<T>(gain[c * 4 + 3]);
        *reinterpret_cast<float4*>(row + c * 4) = v;
      }
    } else {
      for (int i = tid; i < GEMM_MT * (kc >> 2); i += blockDim.x) {
        int r = i / (kc >> 2), c = i % (kc >> 2);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m0 + r < M)
          v = SRC == SRC_MERGE ? merged4(S, m0 + r, c * 4)
                               : *reinterpret_cast<const float4*>(S.a + (size_t)(m0 + r) * S.lda + k0 + c * 4);
        *reinterpret_cast<float4*>(As + (size_t)r * kc_max + c * 4) = v;
      }
    }
    __syncthreads();
    if (active) {
      const int nch = kc >> 3;
      for (int c = c_first; c < nch; c += 64 * KS) {
        const int c2 = c + 32 * KS;
        const bool two = c2 < nch;
        float a[8];
        if (k0 > 0 || c != c_first) load_weights(k0, c, nch);
#pragma unroll
        for (int r = 0; r < GEMM_MT; ++r) {
          load8(As + (size_t)r * kc_max + c * 8, a);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            acc0[r] = fmaf(a[e], x0[e], acc0[r]);
            acc1[r] = fmaf(a[e], x1[e], acc1[r]);
          }
        }
        if (two) {
#pragma unroll
          for (int r = 0; r < GEMM_MT; ++r) {
            load8(As + (size_t)r * kc_max + c2 * 8, a);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              acc0[r] = fmaf(a[e], y0[e], acc0[r]);
              acc1[r] = fmaf(a[e], y1[e], acc1[r]);
            }
          }
        }
      }
    }
  }
  // lane r finishes row r (one lane after the other, the residual's loads and stores were a chain)
  float v0 = 0.f, v1 = 0.f;
#pragma unroll
  for (int r = 0; r < GEMM_MT; ++r) {
    const float s0 = warp_sum(acc0[r]), s1 = warp_sum(acc1[r]);
    if (lane == r) {
      v0 = s0;
      v1 = s1;
    }
  }
  if (KS > 1) {
    if (lane < GEMM_MT) {
      red[warp][lane][0] = v0;
      red[warp][lane][1] = v1;
    }
    __syncthreads();
    if (ks == 0 && lane < GEMM_MT) {
      v0 = v1 = 0.f;
      for (int j = 0; j < KS; ++j) {  // fixed order: bit-reproducible
        v0 += red[warp + j][lane][0];
        v1 += red[warp + j][lane][1];
      }
    }
  }
  if (!mine) return;
  if (EPI == EPI_STORE_F32) {
    C[at] = v0 + b0;
    if (has1) C[at + 1] = v1 + b1;
  } else if (EPI == EPI_RESIDUAL) {
    C[at] = c0 + v0;
    if (has1) C[at + 1] = c1 + v1;
  } else {  // EPI_SWIGLU: row 2j = gate_j, row 2j+1 = up_j
    C[(size_t)(m0 + lane) * ldc + (n0 >> 1)] = v0 / (1.f + expf(-v0)) * v1;
  }
}

template <typename T, int EPI, int KS, int SRC>
static cudaError_t launch_ks(const SimtSrc& src, const void* W, const void* bias, float* C, int ldc, int M, int N, int K,
                             cudaStream_t st) {
  size_t smem = (size_t)GEMM_MT * (K < GEMM_KC ? K : GEMM_KC) * sizeof(float);
  auto kern = gemm_simt_kernel<T, EPI, KS, SRC>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  constexpr int cols = (GEMM_WARPS / KS) * 2;
  dim3 grid((N + cols - 1) / cols, (M + GEMM_MT - 1) / GEMM_MT);
  tc_launch_pdl(kern, grid, dim3(GEMM_WARPS * 32), smem, st, src, (const T*)W, (const T*)bias, C, ldc, M, N, K);
  count_launch();
  return cudaGetLastError();
}

template <typename T, int EPI, int SRC>
static cudaError_t launch_t(const SimtSrc& src, const void* W, const void* bias, float* C, int ldc, int M, int N, int K,
                            cudaStream_t st) {
  if ((K & 7) || (src.lda & 3) || (EPI == EPI_SWIGLU && (N & 1)) || (SRC != SRC_PLAIN && K > GEMM_FUSED_K))
    return cudaErrorInvalidValue;
  // split K over more warps when there are too few columns to fill the GPU
  const int row_tiles = (M + GEMM_MT - 1) / GEMM_MT;
  int ks = 1;
  // (each CTA stages the activations once, so more CTAs also means more L2 reads: stop at one wave)
  while (ks < 8 && (long)((N + 16 / ks - 1) / (16 / ks)) * row_tiles < 148) ks *= 2;
  switch (ks) {
    case 1: return launch_ks<T, EPI, 1, SRC>(src, W, bias, C, ldc, M, N, K, st);
    case 2: return launch_ks<T, EPI, 2, SRC>(src, W, bias, C, ldc, M, N, K, st);
    case 4: return launch_ks<T, EPI, 4, SRC>(src, W, bias, C, ldc, M, N, K, st);
    default: return launch_ks<T, EPI, 8, SRC>(src, W, bias, C, ldc, M, N, K, st);
  }
}

template <typename T>
static cudaError_t launch_epi(int epi, const SimtSrc& src, const void* W, const void* bias, float* C, int ldc, int M, int N,
                              int K, cudaStream_t st) {
  switch (epi) {  // (the sources that occur: norm in front of QKV, gate/up and head; merge in front of O)
    case EPI_STORE_F32:
      return src.gain ? launch_t<T, EPI_STORE_F32, SRC_NORM>(src, W, bias, C, ldc, M, N, K, st)
                      : launch_t<T, EPI_STORE_F32, SRC_PLAIN>(src, W, bias, C, ldc, M, N, K, st);
    case EPI_RESIDUAL:
      return src.part ? launch_t<T, EPI_RESIDUAL, SRC_MERGE>(src, W, bias, C, ldc, M, N, K, st)
                      : launch_t<T, EPI_RESIDUAL, SRC_PLAIN>(src, W, bias, C, ldc, M, N, K, st);
    case EPI_SWIGLU:
      return src.gain ? launch_t<T, EPI_SWIGLU, SRC_NORM>(src, W, bias, C, ldc, M, N, K, st)
                      : launch_t<T, EPI_SWIGLU, SRC_PLAIN>(src, W, bias, C, ldc, M, N, K, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm_simt(int dtype, int epi, const SimtSrc& src, const void* W, const void* bias, float* C, int ldc,
                             int M, int N, int K, cudaStream_t st) {
  return dtype == 0 ? launch_epi<float>(epi, src, W, bias, C, ldc, M, N, K, st)
                    : launch_epi<bf16>(epi, src, W, bias, C, ldc, M, N, K, st);
}

}  // namespace ssd
