// Candidate precompute support (Sec. 3.2, the pointer decoder's per-candidate
// rows): the set-up fold of the decoder matrices, and the fp32 operand split
// that lets the bf16 tensor-core GEMM compute the fp32 precompute products.
//
// The selection loop compares pointer logits to 1e-4, so the rows it reads
// (decoder tokens, folded keys / queries / values of every candidate) need
// fp32 accuracy.  A row times a power of two s (its largest element in
// [2^14, 2^15), so no element overflows and the small ones keep the row's
// absolute precision) splits into two fp16 parts, x s = a1 + a2 + r with
// |r| <= 2^-23 |x s|, and
//   a . b ~= (a2.b1 + a1.b2 + a1.b1) / (s_a s_b)
// (the dropped a2.b2 is below 2^-22 of the product).  As one GEMM over a K
// three times longer:
//   A segments [a2 a1 a1]  x  B segments [b1 b2 b1],
// with fp32 accumulation in TMEM, the two small segments first: a tensor-core
// accumulation rounds towards zero at every step, so what bounds the result's
// error is the number of steps at its full magnitude, K / 16 here.  (Three bf16
// parts, six segments, took twice the tensor time; all six ran at full
// magnitude.)  A is stored once as [a1 a2] (2K wide) and the GEMM producer maps
// each K segment to its part (GemmASplit); the weight side is expanded to 3K
// once, at selector creation; the epilogue multiplies the inverse scales.
//
// Grouped rounds (g > 1) and memories wider than kSplit2MaxD keep the first
// product in three bf16 parts (x = x0 + x1 + x2, |r| <= 2^-24 |x|) as six
// segments,
//   A segments [a0 a0 a1 a0 a1 a2]  x  B segments [b0 b1 b0 b2 b1 b0].
// No limit of the hardware stands behind this: that form is the slower one and
// its own rounding the larger (1.1e-5 of a logit at D = 1,024, 3.8e-5 at 3,584,
// against 1.2e-6 and 3.9e-6 for two parts; 9,218 rows of D = 1,024 in the two
// products 140 us against 78).  It keeps results comparable: the margins of
// grouped rounds are differences of neighbouring logits, and under two parts
// they differ by up to 5e-4 of themselves from those of earlier versions, where
// the measured cases allow 1.5e-4; with g = 1 the two forms' margins agree to
// 2e-5.  So the same image with g = 1 and with g = 5 has logits that differ by
// 1e-5, and a selector holds the weights in both forms.  Whoever can do without
// the comparison replaces the three parts by two everywhere.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sp {

namespace {

// A block per weight row: out[n] = [b1 b2 b1].
__global__ void __launch_bounds__(256)
split_weights_kernel(const float* __restrict__ w, int K4, uint2* __restrict__ out, float* __restrict__ inv) {
  __shared__ float red[8];
  const float4* x = reinterpret_cast<const float4*>(w) + (size_t)blockIdx.x * K4;
  float m = 0.f;
  for (int i = threadIdx.x; i < K4; i += 256) m = fmaxf(m, max_abs4(x[i]));
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int k = 0; k < 8; ++k) m = fmaxf(m, red[k]);
  float iv;
  const float sc = split_scale(m, &iv);
  if (threadIdx.x == 0) inv[blockIdx.x] = iv;
  uint2* o = out + (size_t)blockIdx.x * 3 * K4;
  for (int i = threadIdx.x; i < K4; i += 256) {
    uint2 a, b;
    split2_f16(x[i], sc, a, b);
    o[i] = a;
    o[K4 + i] = b;
    o[2 * K4 + i] = a;
  }
}

// out[n, s*K + k] = part pat[s] of w[n, k] for the six segments of three bf16 parts.
__global__ void split_weights3_kernel(const float* __restrict__ w, int N, int K, __nv_bfloat16* __restrict__ out) {
  const long long n = (long long)N * K;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / K), k = (int)(i - (long long)r * K);
    __nv_bfloat16 p[3];
    float x = w[i];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      p[s] = __float2bfloat16_rn(x);
      x -= __bfloat162float(p[s]);
    }
    const int pat[6] = {0, 1, 0, 2, 1, 0};
    __nv_bfloat16* o = out + (size_t)r * 6 * K + k;
#pragma unroll
    for (int s = 0; s < 6; ++s) o[(size_t)s * K] = p[pat[s]];
  }
}

__global__ void fold_kernel(const float* __restrict__ A, long sai, long sak, const float* __restrict__ B,
                            long sbk, long sbj, float* __restrict__ C, int ldc, int I, int J, int K,
                            float scale) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (i >= I || j >= J) return;
  double s = 0.0;
  for (int k = 0; k < K; ++k) s += (double)A[i * sai + k * sak] * (double)B[k * sbk + j * sbj];
  C[(size_t)i * ldc + j] = (float)(s * (double)scale);
}

}  // namespace

// A-side segment maps of the split products: a2 a1 a1, or a0 a0 a1 a0 a1 a2.
GemmASplit split_a_map(int K, int parts) {
  GemmASplit s;
  s.seg = K;
  s.map = parts == 2 ? 0x001u : 0x210100u;
  return s;
}

cudaError_t split_weights(const float* w, int N, int K, int parts, void* out, float* inv, cudaStream_t st) {
  if (N <= 0 || K <= 0) return cudaSuccess;
  if (K % 4) return cudaErrorInvalidValue;
  if (parts == 2) {
    split_weights_kernel<<<N, 256, 0, st>>>(w, K / 4, static_cast<uint2*>(out), inv);
  } else {
    const int grid = (int)std::min<long long>(((long long)N * K + 255) / 256, 4096);
    split_weights3_kernel<<<grid, 256, 0, st>>>(w, N, K, static_cast<__nv_bfloat16*>(out));
  }
  return cudaGetLastError();
}

cudaError_t fold_matmul(const float* A, long sai, long sak, const float* B, long sbk, long sbj,
                        float* C, int ldc, int I, int J, int K, float scale, cudaStream_t st) {
  dim3 grid((J + 127) / 128, I);
  fold_kernel<<<grid, 128, 0, st>>>(A, sai, sak, B, sbk, sbj, C, ldc, I, J, K, scale);
  return cudaGetLastError();
}

}  // namespace sp
