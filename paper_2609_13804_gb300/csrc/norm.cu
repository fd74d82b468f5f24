// Row-wise kernels: RMSNorm (LM), LayerNorm (selector), dtype conversion and the
// small layout kernels that build the encoder input and the candidate memory.
// All are HBM-bound: one block per row, the row held in registers/shared
// memory, one read and one write of it.
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace sp {

namespace {

constexpr int NT = 256;

SP_DEVINL float block_sum(float v, float* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float t = (l < (int)(blockDim.x >> 5)) ? red[l] : 0.f;
  t = warp_sum(t);
  return t;
}

SP_DEVINL int rows_from(int rows_cap, const int* row_count) {
  int r = rows_cap;
  if (row_count) r = min(r, __ldg(row_count));
  return r;
}

// d multiple of 4
template <bool OUT_BF16>
__global__ void __launch_bounds__(NT)
rmsnorm_kernel(const float* __restrict__ x, const float* __restrict__ gain, void* __restrict__ out,
               int rows_cap, const int* __restrict__ row_count, int d, float eps) {
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const int row = blockIdx.x;
  if (row >= rows_from(rows_cap, row_count)) return;
  const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * d);
  const int n4 = d >> 2;
  float ss = 0.f;
  for (int i = threadIdx.x; i < n4; i += NT) {
    const float4 v = xr[i];
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  ss = block_sum(ss, red);
  const float r = rsqrtf(ss / (float)d + eps);
  for (int i = threadIdx.x; i < n4; i += NT) {
    float4 v = xr[i];
    float4 g = gain ? reinterpret_cast<const float4*>(gain)[i] : make_float4(1.f, 1.f, 1.f, 1.f);
    v.x *= r * g.x; v.y *= r * g.y; v.z *= r * g.z; v.w *= r * g.w;
    if (OUT_BF16) {
      uint2 u;
      u.x = pack_bf16x2(v.x, v.y);
      u.y = pack_bf16x2(v.z, v.w);
      reinterpret_cast<uint2*>(out)[(size_t)row * n4 + i] = u;
    } else {
      reinterpret_cast<float4*>(out)[(size_t)row * n4 + i] = v;
    }
  }
}

// ---- LayerNorm rows held in registers
// A warp holds a row of d <= 4,096 floats (d a multiple of 4), NV float4 per
// lane (float4 i at lane i % 32): one read of the row, two reductions without a
// block barrier, one write, all of a row's loads in flight.  HBM-bound: 144 MB
// on the encoder's 23,552 rows of 1,024.
//
// The sums run in one fixed order, that of 256 partial sums (partial t: the
// elements t, t + 256, .. in turn) added pairwise over the bits 4, 3, 2, 1, 0
// and then 7, 6, 5 of t: a 16-bit encoder amplifies any change of rounding, so
// every row form keeps the same bits.  A lane holds the partials t = 128 p +
// 4 lane + c (p < 2, c < 4): bits 4, 3, 2 of t are lane bits 2, 1, 0, bits 1, 0
// are c, bit 7 is p, bits 6, 5 are lane bits 4, 3.
SP_DEVINL float sum_partials(const float (&s)[2][4]) {
  float y[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    float x[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      x[c] = s[p][c];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) x[c] += __shfl_xor_sync(0xffffffffu, x[c], o);
    }
    y[p] = (x[0] + x[2]) + (x[1] + x[3]);
  }
  float t = y[0] + y[1];
  t += __shfl_xor_sync(0xffffffffu, t, 16);
  t += __shfl_xor_sync(0xffffffffu, t, 8);
  return t;
}

SP_DEVINL float4 ld4(const float* p, int i, bool vec) {
  if (vec) return __ldg(reinterpret_cast<const float4*>(p) + i);
  return make_float4(__ldg(p + 4 * i), __ldg(p + 4 * i + 1), __ldg(p + 4 * i + 2), __ldg(p + 4 * i + 3));
}

// v <- LN(v) with gain / bias (may be NULL; vec: both 16-byte aligned), entries past n4 ignored.
template <int NV>
SP_DEVINL void row_layernorm(float4 (&v)[NV], int lane, int n4, const float* gain, const float* bias, bool vec,
                             float eps) {
  const float d = (float)(4 * n4);
  float s[2][4] = {};
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) {
      s[k & 1][0] += v[k].x; s[k & 1][1] += v[k].y; s[k & 1][2] += v[k].z; s[k & 1][3] += v[k].w;
    }
  const float mean = sum_partials(s) / d;
  float q[2][4] = {};
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) {
      v[k].x -= mean; v[k].y -= mean; v[k].z -= mean; v[k].w -= mean;
      q[k & 1][0] = fmaf(v[k].x, v[k].x, q[k & 1][0]);
      q[k & 1][1] = fmaf(v[k].y, v[k].y, q[k & 1][1]);
      q[k & 1][2] = fmaf(v[k].z, v[k].z, q[k & 1][2]);
      q[k & 1][3] = fmaf(v[k].w, v[k].w, q[k & 1][3]);
    }
  const float rstd = rsqrtf(sum_partials(q) / d + eps);
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int i = lane + 32 * k;
    if (i >= n4) continue;
    const float4 g = gain ? ld4(gain, i, vec) : make_float4(1.f, 1.f, 1.f, 1.f);
    const float4 b = bias ? ld4(bias, i, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[k].x = fmaf(__fmul_rn(v[k].x, rstd), g.x, b.x);
    v[k].y = fmaf(__fmul_rn(v[k].y, rstd), g.y, b.y);
    v[k].z = fmaf(__fmul_rn(v[k].z, rstd), g.z, b.z);
    v[k].w = fmaf(__fmul_rn(v[k].w, rstd), g.w, b.w);
  }
}

SP_DEVINL uint2 pack4(const float4& v) { return make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w)); }

// out [rows, d] bf16 = LN(x [rows, d] fp32); x and out rows contiguous and 16-byte aligned.
template <int NV>
__global__ void __launch_bounds__(NT)
layernorm_kernel(const float* x, const float* __restrict__ gain, const float* __restrict__ bias, int vec, uint2* out,
                 int rows, int n4, float eps) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const float4* xr = reinterpret_cast<const float4*>(x) + (size_t)row * n4;
  float4 v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) v[k] = xr[lane + 32 * k];
  row_layernorm<NV>(v, lane, n4, gain, bias, vec != 0, eps);
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) out[(size_t)row * n4 + lane + 32 * k] = pack4(v[k]);
}

// The same for rows wider than the register form holds (d > 4,096): the row in shared memory.
__global__ void __launch_bounds__(NT)
layernorm_wide_kernel(const float* x, const float* __restrict__ gain, const float* __restrict__ bias,
                      __nv_bfloat16* out, int rows, int d, float eps) {
  extern __shared__ float buf[];
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  const int row = blockIdx.x;
  if (row >= rows) return;
  const float* xr = x + (size_t)row * d;
  float s = 0.f;
  for (int i = threadIdx.x; i < d; i += NT) {
    const float v = xr[i];
    buf[i] = v;
    s += v;
  }
  const float mean = block_sum(s, red) / (float)d;
  float q = 0.f;
  for (int i = threadIdx.x; i < d; i += NT) {
    const float c = buf[i] - mean;
    q += c * c;
  }
  const float rstd = rsqrtf(block_sum(q, red) / (float)d + eps);
  for (int i = threadIdx.x; i < d; i += NT) {
    float v = (buf[i] - mean) * rstd;
    if (gain) v *= gain[i];
    if (bias) v += bias[i];
    out[(size_t)row * d + i] = __float2bfloat16_rn(v);
  }
}

__global__ void bf16_to_f32_kernel(const uint2* __restrict__ x, float4* __restrict__ out, int rows_cap,
                                   const int* __restrict__ row_count, int d) {
  pdl_wait();
  pdl_trigger();
  const int row = blockIdx.x;
  if (row >= rows_from(rows_cap, row_count)) return;
  const int n4 = d >> 2;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) {
    const uint2 u = x[(size_t)row * n4 + i];
    const float2 a = unpack_bf16x2(u.x), b = unpack_bf16x2(u.y);
    out[(size_t)row * n4 + i] = make_float4(a.x, a.y, b.x, b.y);
  }
}

// Rows [T, T + gridDim.x) of a row-major buffer, T = *row_count, below rows_cap, set to zero.
__global__ void zero_rows_after_kernel(uint4* __restrict__ buf, int row_u4, const int* __restrict__ row_count,
                                       int rows_cap) {
  pdl_wait();
  pdl_trigger();
  const int row = __ldg(row_count) + blockIdx.x;
  if (row < 0 || row >= rows_cap) return;
  for (int i = threadIdx.x; i < row_u4; i += blockDim.x) buf[(size_t)row * row_u4 + i] = make_uint4(0, 0, 0, 0);
}

SP_DEVINL int find_image(const int* off, int B, int r) {
  // largest b with off[b] <= r
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Image of packed encoder row r (image b's rows: its visual rows, then its text rows).
SP_DEVINL int find_encoder_image(const BatchDesc& bd, int r) {
  int lo = 0, hi = bd.B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (bd.vis_off[mid] + bd.txt_off[mid] <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Encoder input rows of image b: [X_b (bf16 -> fp32); g_text * LN(P_b)] (Eq. 3)
// into R, and the first block's LN1 of each row into A (bf16), while the row is
// in registers; block 0 also writes the sequences' offsets.
template <int NV>
__global__ void __launch_bounds__(NT)
assemble_kernel(const BatchDesc bd, const uint2* X, const float* P, int n4,
                const float* __restrict__ g, const float* __restrict__ bb, const float* __restrict__ g1,
                const float* __restrict__ b1, int vec, int vec1, float eps, float g_text, float4* R,
                uint2* A, int rows, int* cu) {
  pdl_wait();
  pdl_trigger();
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b <= bd.B; b += NT) cu[b] = bd.vis_off[b] + bd.txt_off[b];
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
  if (r >= rows) return;
  const int b = find_encoder_image(bd, r);
  const int local = r - (bd.vis_off[b] + bd.txt_off[b]);
  const int nv = bd.vis_off[b + 1] - bd.vis_off[b];
  float4 v[NV];
  if (local < nv) {
    const uint2* xr = X + (size_t)(bd.vis_off[b] + local) * n4;
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (lane + 32 * k < n4) {
        const uint2 u = xr[lane + 32 * k];
        const float2 lo = unpack_bf16x2(u.x), hi = unpack_bf16x2(u.y);
        v[k] = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
  } else {
    const float4* pr = reinterpret_cast<const float4*>(P) + (size_t)(bd.txt_off[b] + local - nv) * n4;
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (lane + 32 * k < n4) v[k] = pr[lane + 32 * k];
    row_layernorm<NV>(v, lane, n4, g, bb, vec != 0, eps);
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (lane + 32 * k < n4) { v[k].x *= g_text; v[k].y *= g_text; v[k].z *= g_text; v[k].w *= g_text; }
  }
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) R[(size_t)r * n4 + lane + 32 * k] = v[k];
  row_layernorm<NV>(v, lane, n4, g1, b1, vec1 != 0, eps);
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) A[(size_t)r * n4 + lane + 32 * k] = pack4(v[k]);
}

// The same rows and offsets for d > 4,096 (no LN1: a pass of its own follows).
__global__ void __launch_bounds__(NT)
assemble_wide_kernel(const BatchDesc bd, const __nv_bfloat16* X, const float* P, int D,
                     const float* __restrict__ g, const float* __restrict__ bb, float eps, float g_text,
                     float* R, int rows, int* cu) {
  extern __shared__ float buf[];
  __shared__ float red[32];
  pdl_wait();
  pdl_trigger();
  if (blockIdx.x == 0)
    for (int b = threadIdx.x; b <= bd.B; b += NT) cu[b] = bd.vis_off[b] + bd.txt_off[b];
  const int r = blockIdx.x;
  if (r >= rows) return;
  const int b = find_encoder_image(bd, r);
  const int local = r - (bd.vis_off[b] + bd.txt_off[b]);
  const int nv = bd.vis_off[b + 1] - bd.vis_off[b];
  float* out = R + (size_t)r * D;
  if (local < nv) {
    const __nv_bfloat16* xr = X + (size_t)(bd.vis_off[b] + local) * D;
    for (int i = threadIdx.x; i < D; i += NT) out[i] = __bfloat162float(xr[i]);
    return;
  }
  const float* pr = P + (size_t)(bd.txt_off[b] + local - nv) * D;
  float s = 0.f;
  for (int i = threadIdx.x; i < D; i += NT) {
    const float v = pr[i];
    buf[i] = v;
    s += v;
  }
  const float mean = block_sum(s, red) / (float)D;
  float q = 0.f;
  for (int i = threadIdx.x; i < D; i += NT) {
    const float c = buf[i] - mean;
    q += c * c;
  }
  const float rstd = rsqrtf(block_sum(q, red) / (float)D + eps);
  for (int i = threadIdx.x; i < D; i += NT) {
    float v = (buf[i] - mean) * rstd;
    if (g) v *= g[i];
    if (bb) v += bb[i];
    out[i] = g_text * v;
  }
}

// Candidate memory rows [every image's visual rows; s_stop; s_start] (row
// sources: the encoder's residual R, the given memory H, or the visual tokens X
// themselves) as the split operand of the precompute GEMM: [rows, 2D] fp16
// (parts a1 | a2 of the scaled row) with the inverse scales, or [rows, 3D] bf16
// (PARTS = 3, always where D > kSplit2MaxD); optionally the visual rows go to
// `memory` (fp32).  HBM-bound, a warp per row.  NV > 0: all of the row's 16-byte
// loads in flight, the row held in registers (NV float4 per lane), for PARTS = 2
// between the search for its largest element and the split; NV = 0: rows wider
// than that.
template <int NV, int PARTS>
__global__ void __launch_bounds__(NT)
memory_split_kernel(const BatchDesc bd, const float* R, const float* H, const uint2* X, const float* s_stop,
                    const float* s_start, uint2* out, float* inv, float* memory, int n4, int rows, int vec_ends,
                    int vec_mem) {
  pdl_wait();
  pdl_trigger();
  const int r = blockIdx.x * (NT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int nvis = bd.vis_off[bd.B];
  const float* src = nullptr;
  const uint2* xs = nullptr;
  bool vec = true;
  if (r >= nvis) {
    src = r == nvis ? s_stop : s_start;
    vec = vec_ends != 0;
  } else if (H) {
    src = H + (size_t)r * 4 * n4;
  } else if (X) {
    xs = X + (size_t)r * n4;
  } else {
    const int b = find_image(bd.vis_off, bd.B, r);
    src = R + (size_t)(r + bd.txt_off[b]) * 4 * n4;
  }
  uint2* o = out + (size_t)r * PARTS * n4;
  float* mem = memory && r < nvis ? memory + (size_t)r * 4 * n4 : nullptr;
  auto load = [&](int i) {
    if (xs) {
      const uint2 w = xs[i];
      const float2 lo = unpack_bf16x2(w.x), hi = unpack_bf16x2(w.y);
      return make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    if (vec) return reinterpret_cast<const float4*>(src)[i];
    return make_float4(src[4 * i], src[4 * i + 1], src[4 * i + 2], src[4 * i + 3]);
  };
  auto put = [&](int i, const float4& v, float sc) {
    if constexpr (PARTS == 2) {
      split2_f16(v, sc, o[i], o[n4 + i]);
    } else {
      float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const uint2 u = make_uint2(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]));
        const float2 lo = unpack_bf16x2(u.x), hi = unpack_bf16x2(u.y);
        x[0] -= lo.x; x[1] -= lo.y; x[2] -= hi.x; x[3] -= hi.y;
        o[s * n4 + i] = u;
      }
    }
    if (mem) {
      if (vec_mem) {
        reinterpret_cast<float4*>(mem)[i] = v;
      } else {
        mem[4 * i] = v.x; mem[4 * i + 1] = v.y; mem[4 * i + 2] = v.z; mem[4 * i + 3] = v.w;
      }
    }
  };
  if constexpr (NV > 0) {
    float4 v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (lane + 32 * k < n4) v[k] = load(lane + 32 * k);
    float sc = 1.f;
    if constexpr (PARTS == 2) {
      float m = 0.f, iv;
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (lane + 32 * k < n4) m = fmaxf(m, max_abs4(v[k]));
      sc = split_scale(warp_max(m), &iv);
      if (lane == 0) inv[r] = iv;
    }
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (lane + 32 * k < n4) put(lane + 32 * k, v[k], sc);
  } else {
#pragma unroll 4
    for (int i = lane; i < n4; i += 32) put(i, load(i), 1.f);
  }
}

// LN1 of the decoder tokens (rows of h floats, ldx apart) as the split operand of
// the second precompute GEMM, [rows, 2h] fp16, and its inverse scales; a warp per
// row (h <= 1,024).
template <int NV>
__global__ void __launch_bounds__(NT)
layernorm_split_kernel(const float* x, int ldx, const float* __restrict__ gain,
                       const float* __restrict__ bias, int vec, uint2* out, float* inv, int rows, int n4, float eps) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const float4* xr = reinterpret_cast<const float4*>(x + (size_t)row * ldx);
  float4 v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) v[k] = xr[lane + 32 * k];
  row_layernorm<NV>(v, lane, n4, gain, bias, vec != 0, eps);
  float m = 0.f, iv;
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4) m = fmaxf(m, max_abs4(v[k]));
  const float sc = split_scale(warp_max(m), &iv);
  if (lane == 0) inv[row] = iv;
#pragma unroll
  for (int k = 0; k < NV; ++k)
    if (lane + 32 * k < n4)
      split2_f16(v[k], sc, out[(size_t)row * 2 * n4 + lane + 32 * k], out[((size_t)row * 2 + 1) * n4 + lane + 32 * k]);
}

}  // namespace

cudaError_t rmsnorm_f32_to_bf16(const float* x, const float* gain, void* out, int rows_cap,
                                const int* row_count, int d, float eps, cudaStream_t st) {
  if (rows_cap <= 0) return cudaSuccess;
  prof_begin_launch(st);
  const cudaError_t r = launch_pdl(rmsnorm_kernel<true>, dim3(rows_cap), dim3(NT), 0, st, x, gain, out, rows_cap,
                                   row_count, d, eps);
  prof_end_launch(st, SP_K_NORM, 0.0, 6.0 * rows_cap * (double)d);
  return r;
}

cudaError_t rmsnorm_f32_to_f32(const float* x, const float* gain, float* out, int rows_cap,
                               const int* row_count, int d, float eps, cudaStream_t st) {
  if (rows_cap <= 0) return cudaSuccess;
  prof_begin_launch(st);
  const cudaError_t r = launch_pdl(rmsnorm_kernel<false>, dim3(rows_cap), dim3(NT), 0, st, x, gain,
                                   static_cast<void*>(out), rows_cap, row_count, d, eps);
  prof_end_launch(st, SP_K_NORM, 0.0, 8.0 * rows_cap * (double)d);
  return r;
}

static bool aligned16(const void* a, const void* b) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}

constexpr int kRowFormMax = 4096;  // widest row of the register form (32 float4 per lane)

// Calls f(float4 per lane) with the register form of a row of d <= MAX floats.
template <int MAX = kRowFormMax, class F>
static cudaError_t with_row_form(int d, F f) {
  if (d > MAX) return cudaErrorInvalidValue;
  if (d <= 256) return f(std::integral_constant<int, 2>{});
  if (d <= 512) return f(std::integral_constant<int, 4>{});
  if (MAX <= 1024 || d <= 1024) return f(std::integral_constant<int, 8>{});
  if constexpr (MAX > 1024) {
    if (MAX <= 2048 || d <= 2048) return f(std::integral_constant<int, 16>{});
    if constexpr (MAX > 2048) return f(std::integral_constant<int, 32>{});
  }
}

static int row_blocks(int rows) { return (rows + NT / 32 - 1) / (NT / 32); }

cudaError_t layernorm_bf16(const float* x, const float* gain, const float* bias, void* out, int rows, int d, float eps,
                           cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  prof_begin_launch(st);
  cudaError_t r;
  if (d <= kRowFormMax) {
    r = with_row_form(d, [&](auto nv) {
      return launch_pdl(layernorm_kernel<decltype(nv)::value>, dim3(row_blocks(rows)), dim3(NT), 0, st, x, gain, bias,
                        aligned16(gain, bias) ? 1 : 0, static_cast<uint2*>(out), rows, d / 4, eps);
    });
  } else {
    r = launch_pdl(layernorm_wide_kernel, dim3(rows), dim3(NT), d * sizeof(float), st, x, gain, bias,
                   static_cast<__nv_bfloat16*>(out), rows, d, eps);
  }
  prof_end_launch(st, SP_K_NORM, 0.0, 6.0 * rows * (double)d);
  return r;
}

cudaError_t layernorm_split(const float* x, int ldx, const float* gain, const float* bias, void* out, float* inv,
                            int rows, int d, float eps, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  if (d % 4 != 0 || ldx % 4 != 0) return cudaErrorInvalidValue;
  prof_begin_launch(st);
  const cudaError_t r = with_row_form<1024>(d, [&](auto nv) {
    return launch_pdl(layernorm_split_kernel<decltype(nv)::value>, dim3(row_blocks(rows)), dim3(NT), 0, st, x, ldx,
                      gain, bias, aligned16(gain, bias) ? 1 : 0, static_cast<uint2*>(out), inv, rows, d / 4, eps);
  });
  prof_end_launch(st, SP_K_NORM, 0.0, 8.0 * rows * (double)d);
  return r;
}

cudaError_t zero_rows_after(void* buf, size_t row_bytes, const int* row_count, int rows_cap, int nrows,
                            cudaStream_t st) {
  if (rows_cap <= 0 || nrows <= 0) return cudaSuccess;
  if (row_bytes % 16 != 0) return cudaErrorInvalidValue;
  prof_begin_launch(st);
  const cudaError_t r = launch_pdl(zero_rows_after_kernel, dim3(nrows), dim3(256), 0, st,
                                   reinterpret_cast<uint4*>(buf), (int)(row_bytes / 16), row_count, rows_cap);
  prof_end_launch(st, SP_K_MISC, 0.0, (double)nrows * row_bytes);
  return r;
}

cudaError_t bf16_to_f32(const void* x, float* out, int rows_cap, const int* row_count, int d,
                        cudaStream_t st) {
  if (rows_cap <= 0) return cudaSuccess;
  prof_begin_launch(st);
  const cudaError_t r = launch_pdl(bf16_to_f32_kernel, dim3(rows_cap), dim3(256), 0, st,
                                   reinterpret_cast<const uint2*>(x), reinterpret_cast<float4*>(out), rows_cap,
                                   row_count, d);
  prof_end_launch(st, SP_K_MISC, 0.0, 6.0 * rows_cap * (double)d);
  return r;
}

cudaError_t assemble_encoder_input(const BatchDesc& bd, const void* X, const float* P, int D,
                                   const float* ln_g, const float* ln_b, const float* ln1_g, const float* ln1_b,
                                   float eps, float g_text, float* R, void* A, int rows, int* cu, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  prof_begin_launch(st);
  cudaError_t r;
  if (D <= kRowFormMax) {
    r = with_row_form(D, [&](auto nv) {
      return launch_pdl(assemble_kernel<decltype(nv)::value>, dim3(row_blocks(rows)), dim3(NT), 0, st, bd,
                        static_cast<const uint2*>(X), P, D / 4, ln_g, ln_b, ln1_g, ln1_b,
                        aligned16(ln_g, ln_b) ? 1 : 0, aligned16(ln1_g, ln1_b) ? 1 : 0, eps, g_text,
                        reinterpret_cast<float4*>(R), static_cast<uint2*>(A), rows, cu);
    });
  } else {
    r = launch_pdl(assemble_wide_kernel, dim3(rows), dim3(NT), D * sizeof(float), st, bd,
                   static_cast<const __nv_bfloat16*>(X), P, D, ln_g, ln_b, eps, g_text, R, rows, cu);
  }
  prof_end_launch(st, SP_K_MISC, 0.0, 8.0 * rows * (double)D);
  if (r == cudaSuccess && D > kRowFormMax) r = layernorm_bf16(R, ln1_g, ln1_b, A, rows, D, eps, st);
  return r;
}

cudaError_t memory_split(const BatchDesc& bd, const float* R, const float* H, const void* X, const float* s_stop,
                         const float* s_start, void* out, float* inv, float* memory, int D, cudaStream_t st) {
  const int rows = bd.vis_off[bd.B] + 2;
  prof_begin_launch(st);
  auto go = [&](auto kern) {
    return launch_pdl(kern, dim3(row_blocks(rows)), dim3(NT), 0, st, bd, R, H, static_cast<const uint2*>(X), s_stop,
                      s_start, static_cast<uint2*>(out), inv, memory, D / 4, rows, aligned16(s_stop, s_start) ? 1 : 0,
                      aligned16(memory, nullptr) ? 1 : 0);
  };
  cudaError_t r;
  if (inv)
    r = with_row_form<2048>(D, [&](auto nv) { return go(memory_split_kernel<decltype(nv)::value, 2>); });
  else if (D <= kRowFormMax)
    r = with_row_form(D, [&](auto nv) { return go(memory_split_kernel<decltype(nv)::value, 3>); });
  else
    r = go(memory_split_kernel<0, 3>);
  prof_end_launch(st, SP_K_SGEMM, 0.0, (memory ? 12.0 : 8.0) * rows * (double)D);
  return r;
}

}  // namespace sp
