// Per-episode inner-product tables of the pointer decoder's precomputed rows.
//
// Everything a selection round evaluates is linear in the softmax weights p of
// the last history position over the history, apart from LN2's one variance:
//   u      = z_last + sum_k p_k vt_k,       p = softmax_k <qs_last, ks_k>
//   l(j)   = <LN2(u), kt_j>
//          = rstd (<kt_j o gain, zc_last> + sum_k p_k <kt_j o gain, vc_k>) + <kt_j, bias>
//   h var  = |zc_last|^2 + 2 sum_k p_k <zc_last, vc_k> + sum_km p_k p_m <vc_k, vc_m>
// with zc / vc the rows minus their own mean (LN2 removes the mean of u).  All
// history rows are candidates of the same episode (or START), so five tables
// per episode hold every inner product a rollout can ask for:
//   G = vc KTg^T | Gz = zc KTg^T | S = QS KS^T | VV = vc vc^T | ZV = zc vc^T
// and a round becomes a few gathers and (history x candidates) multiply-adds,
// with no h-wide vector left in it (select_gram.cu).
//
// The tables are fp32-accurate products on the fp16 tensor cores: a row is
// scaled by a power of two to a largest element in [2^14, 2^15) and split into
// two fp16 parts (22 bits and more), and a.b ~= a1.b1 + a1.b2 + a2.b1 (the
// dropped a2.b2 is below 2^-22 of the product) accumulates in fp32 in TMEM, the
// two small products apart from the large one (tensor-core accumulation rounds
// towards zero at every step: fewer steps at the full magnitude).
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace sp {

namespace {

constexpr int NT = 256;

struct Episode {
  int n;       // candidates
  int vis;     // first visual row
  int base;    // first operand row (every episode: its candidates, STOP, START)
};

SP_DEVINL Episode episode_of(const BatchDesc& bd, int b, int le) {
  const int n_img = bd.vis_off[b + 1] - bd.vis_off[b];
  const int gs = bd.group_size > 0 ? bd.group_size : n_img;
  const int c0 = le * gs;
  Episode ep;
  ep.n = min(gs, n_img - c0);
  ep.vis = bd.vis_off[b] + c0;
  ep.base = ep.vis + 2 * (bd.ep_off[b] + le);
  return ep;
}

SP_DEVINL Episode find_episode(const BatchDesc& bd, int e) {
  int lo = 0, hi = bd.B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (bd.ep_off[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return episode_of(bd, lo, e - bd.ep_off[lo]);
}

// ---- operand rows
// A row of h = 128 HV floats as HV float4 per lane -> its two fp16 parts
// (o[lane + 32 k]: part 1, o[h/4 + ..]: part 2); returns what undoes the scale.
template <int HV>
SP_DEVINL float put_split2(const float4 (&v)[HV], int lane, uint2* o) {
  float m = 0.f, inv;
#pragma unroll
  for (int k = 0; k < HV; ++k) m = fmaxf(m, max_abs4(v[k]));
  const float sc = split_scale(warp_max(m), &inv);
#pragma unroll
  for (int k = 0; k < HV; ++k) split2_f16(v[k], sc, o[lane + 32 * k], o[32 * HV + lane + 32 * k]);
  return inv;
}

template <int HV>
SP_DEVINL void load_row(const float* p, int lane, float4 (&v)[HV]) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int k = 0; k < HV; ++k) v[k] = q[lane + 32 * k];
}

template <int HV>
SP_DEVINL void center_row(float4 (&v)[HV]) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < HV; ++k) s += (v[k].x + v[k].y) + (v[k].z + v[k].w);
  const float mean = warp_sum(s) / (float)(128 * HV);
#pragma unroll
  for (int k = 0; k < HV; ++k) { v[k].x -= mean; v[k].y -= mean; v[k].z -= mean; v[k].w -= mean; }
}

// A warp per operand row: the five vectors of its source row (20 h bytes read,
// 20 h written; HBM-bound), the row's <kt, bias> and |zc|^2.
template <int HV>
__global__ void __launch_bounds__(NT)
gram_operands_kernel(const BatchDesc bd, const GramArgs g) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
  if (r >= g.rows) return;
  int lo = 0, hi = bd.B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (bd.vis_off[mid] + 2 * bd.ep_off[mid] <= r) lo = mid; else hi = mid - 1;
  }
  const int n_img = bd.vis_off[lo + 1] - bd.vis_off[lo];
  const int gs = bd.group_size > 0 ? min(bd.group_size, n_img) : n_img;
  const Episode ep = episode_of(bd, lo, (r - bd.vis_off[lo] - 2 * bd.ep_off[lo]) / (gs + 2));
  const int i = r - ep.base;
  const int src = i < ep.n ? ep.vis + i : (i == ep.n ? g.stop_row : g.start_row);

  constexpr int H4 = 32 * HV;
  uint2* op = static_cast<uint2*>(g.op);
  auto row_of = [&](int m) { return op + ((size_t)m * g.rows + r) * (2 * H4); };
  float4 v[HV];
  float inv[5];
  load_row<HV>(g.KT + (size_t)src * g.ldkt, lane, v);
  float d = 0.f;
  if (g.ln2_b) {
#pragma unroll
    for (int k = 0; k < HV; ++k) {
      const float* b = g.ln2_b + 4 * (lane + 32 * k);
      d += v[k].x * b[0] + v[k].y * b[1] + v[k].z * b[2] + v[k].w * b[3];
    }
    d = warp_sum(d);
  }
  if (g.ln2_g) {
#pragma unroll
    for (int k = 0; k < HV; ++k) {
      const float* w = g.ln2_g + 4 * (lane + 32 * k);
      v[k].x *= w[0]; v[k].y *= w[1]; v[k].z *= w[2]; v[k].w *= w[3];
    }
  }
  inv[0] = put_split2<HV>(v, lane, row_of(0));
  load_row<HV>(g.KS + (size_t)src * g.ldks, lane, v);
  inv[1] = put_split2<HV>(v, lane, row_of(1));
  load_row<HV>(g.VT + (size_t)src * g.ldvt, lane, v);
  center_row<HV>(v);
  inv[2] = put_split2<HV>(v, lane, row_of(2));
  load_row<HV>(g.Z + (size_t)src * g.ldz, lane, v);
  center_row<HV>(v);
  float q = 0.f;
#pragma unroll
  for (int k = 0; k < HV; ++k) q += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  q = warp_sum(q);
  inv[3] = put_split2<HV>(v, lane, row_of(3));
  load_row<HV>(g.QS + (size_t)src * g.ldqs, lane, v);
  inv[4] = put_split2<HV>(v, lane, row_of(4));
  if (lane == 0) {
#pragma unroll
    for (int m = 0; m < 5; ++m) g.inv[(size_t)m * g.rows + r] = inv[m];
    g.dj[r] = d;
    g.zz[r] = q;
  }
}

// ---- tables
// Persistent kernel, one CTA per SM, 10 warps: TMA producer, MMA issuer, eight
// epilogue warps (two per TMEM lane quadrant, every other 32 columns); two fp32 accumulators (large and small products)
// fill TMEM, so a tile's epilogue runs between its MMAs and the next tile's.  A
// work item is one 128 x n_tile tile of one table of one episode.  A stage
// holds both parts of 64 columns of both operands and feeds all three products
// (12 MMAs of K = 16): 85 KB for 1,250 tensor cycles at n_tile 208, 68 B/cycle,
// where staging the products one by one as a GEMM over 3h would take 101.  The
// large parts have a barrier of their own and their product starts first.
// 16 episodes of 576, h = 512 (82 useful GFLOP of three products, 107 MB of
// tables): 110 us (126 with four epilogue warps and one barrier), bound by the loads' latency at
// two stages and by the epilogue that nothing overlaps.
constexpr int BM = 128;
constexpr int BK = 64;
constexpr int STAGES = 2;
constexpr int NMAX = 256;
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t B_BYTES = NMAX * BK * 2;
constexpr uint32_t STAGE_BYTES = 2 * (A_BYTES + B_BYTES);
constexpr int EPI_WARPS = 8;
constexpr int GT = 64 + 32 * EPI_WARPS;
constexpr uint32_t EPI_BYTES = EPI_WARPS * 32 * 33 * 4;
constexpr size_t GRAM_SMEM = 1024 + STAGES * STAGE_BYTES + EPI_BYTES + 256;

struct Tile {
  Episode ep;
  int p, m0, n0, e;
};

// Work item t (episode slowest, then table, column tile, row tile); false where
// a smaller episode of the batch has no such tile.
SP_DEVINL bool tile_of(const BatchDesc& bd, const GramArgs& g, int t, Tile& o) {
  const int per_ep = 5 * g.mt * g.nt;
  o.e = t / per_ep;
  int u = t - o.e * per_ep;
  o.p = u / (g.mt * g.nt);
  u -= o.p * g.mt * g.nt;
  o.n0 = (u / g.mt) * g.n_tile;
  o.m0 = (u % g.mt) * BM;
  o.ep = find_episode(bd, o.e);
  return o.m0 < o.ep.n + 2 && o.n0 < o.ep.n + 2;
}

// operand matrices (KTg, KS, vc, zc, QS) of table p: rows A_MAT, columns B_MAT
SP_DEVINL int a_mat(int p) { return (0x32432 >> (4 * p)) & 15; }  // vc zc QS vc zc
SP_DEVINL int b_mat(int p) { return (0x22100 >> (4 * p)) & 15; }  // KTg KTg KS vc vc

__global__ void __launch_bounds__(GT, 1)
gram_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const BatchDesc bd,
            const GramArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* stg = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES + EPI_BYTES);
  uint64_t* empty = full + 2 * STAGES;  // (full: the large parts, then the small ones)
  uint64_t* tfull = empty + STAGES;
  uint64_t* tempty = tfull + 1;
  uint64_t* done = tempty + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* err = g.err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&full[STAGES + s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, EPI_WARPS);
    mbar_init(done, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tslot;
  pdl_wait();
  pdl_trigger();

  const int total = g.E * 5 * g.mt * g.nt;
  const int KB = g.h / BK;
  if (warp == 0) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        Tile w;
        if (!tile_of(bd, g, t, w)) continue;
        const int ar = a_mat(w.p) * g.rows + w.ep.base + w.m0;
        const int br = b_mat(w.p) * g.rows + w.ep.base + w.n0;
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(&empty[s], ph ^ 1u, err)) { ok = false; break; }
          const uint32_t half = A_BYTES + (uint32_t)g.n_tile * BK * 2;
          mbar_arrive_expect_tx(&full[s], half);
          uint8_t* st = smem + s * STAGE_BYTES;
          tma_load_2d(st, &tmA, &full[s], kb * BK, ar);
          tma_load_2d(st + 2 * A_BYTES, &tmB, &full[s], kb * BK, br);
          mbar_arrive_expect_tx(&full[STAGES + s], half);
          tma_load_2d(st + A_BYTES, &tmA, &full[STAGES + s], g.h + kb * BK, ar);
          tma_load_2d(st + 2 * A_BYTES + B_BYTES, &tmB, &full[STAGES + s], g.h + kb * BK, br);
          if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_f16_f32(BM, g.n_tile);
      int s = 0, it = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < total; t += gridDim.x) {
        Tile w;
        if (!tile_of(bd, g, t, w)) continue;
        if (!mbar_wait(tempty, (it & 1) ^ 1u, err)) break;
        tc_fence_after();
        for (int kb = 0; kb < KB; ++kb) {
          if (!mbar_wait(&full[s], ph, err)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a1 = smem_u32(smem + s * STAGE_BYTES), a2 = a1 + A_BYTES;
          const uint32_t b1 = a1 + 2 * A_BYTES, b2 = b1 + B_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma_bf16(tmem_base, umma_desc_sw128(a1 + k * 32), umma_desc_sw128(b1 + k * 32), idesc, (kb | k) ? 1u : 0u);
          if (!mbar_wait(&full[STAGES + s], ph, err)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            umma_bf16(tmem_base + NMAX, umma_desc_sw128(a1 + k * 32), umma_desc_sw128(b2 + k * 32), idesc,
                      (kb | k) ? 1u : 0u);
            umma_bf16(tmem_base + NMAX, umma_desc_sw128(a2 + k * 32), umma_desc_sw128(b1 + k * 32), idesc, 1u);
          }
          umma_commit(&empty[s]);
          if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        if (!ok) break;
        umma_commit(tfull);
        ++it;
      }
      umma_commit(done);
      mbar_wait(done, 0, err);
    }
    __syncwarp();
  } else {
    const int quad = warp & 3;
    float* st = stg + (warp - 2) * 32 * 33;
    int it = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
      Tile w;
      if (!tile_of(bd, g, t, w)) continue;
      if (!mbar_wait_warp(tfull, it & 1, err)) break;
      tc_fence_after();
      ++it;
      const int np = w.ep.n + 2;
      const int i0 = w.m0 + quad * 32;
      const int cols = min(g.n_tile, np - w.n0);
      const float* inv_a = g.inv + (size_t)a_mat(w.p) * g.rows + w.ep.base;
      const float* inv_b = g.inv + (size_t)b_mat(w.p) * g.rows + w.ep.base + w.n0;
      const float ia = i0 + lane < np ? inv_a[i0 + lane] : 0.f;
      float* out = g.table + (size_t)w.e * g.ep_stride + (size_t)i0 * (5 * g.ld) + (size_t)w.p * g.ld + w.n0;
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16);
      const int rows = min(32, np - i0);
      if (rows > 0) {
        for (int c = ((warp - 2) >> 2) * 32; c < cols; c += EPI_WARPS * 8) {
          float v[32], u[32];
          tmem_ld_32x32b_x32(taddr + c, v);
          tmem_ld_32x32b_x32(taddr + NMAX + c, u);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 32; ++k) st[lane * 33 + k] = (v[k] + u[k]) * ia;
          __syncwarp();
          const bool live = c + lane < cols;
          const float ib = live ? inv_b[c + lane] : 0.f;
          float* o = out + c + lane;
          if (rows == 32) {
#pragma unroll 16
            for (int r = 0; r < 32; ++r, o += 5 * g.ld) {
              const float x = st[r * 33 + lane] * ib;
              if (live) *o = x;
            }
          } else {
            for (int r = 0; r < rows; ++r, o += 5 * g.ld)
              if (live) *o = st[r * 33 + lane] * ib;
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

// Sizes of the tables and operands for episodes of at most n_max candidates.
void gram_layout(int E, int nvis, int n_max, int h, GramArgs* g) {
  g->E = E;
  g->h = h;
  g->rows = nvis + 2 * E;
  const int np = n_max + 2;
  g->ld = (np + 3) & ~3;
  g->ep_stride = (size_t)np * 5 * g->ld;
  g->mt = (np + BM - 1) / BM;
  g->nt = (np + NMAX - 1) / NMAX;
  g->n_tile = ((np + g->nt - 1) / g->nt + 15) & ~15;
}

cudaError_t gram_launch(const BatchDesc& bd, const GramArgs& g, cudaStream_t st) {
  CUtensorMap ta, tb;
  std::string msg;
  if (!encode_tmap_bf16(&ta, g.op, (uint64_t)5 * g.rows, 2 * g.h, BM, &msg) ||
      !encode_tmap_bf16(&tb, g.op, (uint64_t)5 * g.rows, 2 * g.h, g.n_tile, &msg))
    return cudaErrorInvalidValue;
  const dim3 grid((g.rows + NT / 32 - 1) / (NT / 32));
  cudaError_t r;
  prof_begin_launch(st);
  switch (g.h / 128) {
    case 1: r = launch_pdl(gram_operands_kernel<1>, grid, dim3(NT), 0, st, bd, g); break;
    case 2: r = launch_pdl(gram_operands_kernel<2>, grid, dim3(NT), 0, st, bd, g); break;
    case 4: r = launch_pdl(gram_operands_kernel<4>, grid, dim3(NT), 0, st, bd, g); break;
    case 8: r = launch_pdl(gram_operands_kernel<8>, grid, dim3(NT), 0, st, bd, g); break;
    default: r = cudaErrorInvalidValue;
  }
  prof_end_launch(st, SP_K_SGEMM, 0.0, 40.0 * g.rows * (double)g.h);
  if (r != cudaSuccess) return r;
  r = cudaFuncSetAttribute(gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GRAM_SMEM);
  if (r != cudaSuccess) return r;
  const int tiles = g.E * 5 * g.mt * g.nt;
  double flops = 0.0;
  for (int b = 0; b < bd.B; ++b) {
    const int n_img = bd.vis_off[b + 1] - bd.vis_off[b];
    const int gs = bd.group_size > 0 ? bd.group_size : n_img;
    for (int c = 0; c < n_img; c += gs) {
      const double np = std::min(gs, n_img - c) + 2;
      flops += 30.0 * np * np * g.h;
    }
  }
  prof_begin_launch(st);
  r = launch_pdl(gram_kernel, dim3(std::min(tiles, device_sm_count())), dim3(GT), GRAM_SMEM, st, ta, tb, bd, g);
  prof_end_launch(st, SP_K_SGEMM, flops, 0.0);
  return r;
}

}  // namespace sp
