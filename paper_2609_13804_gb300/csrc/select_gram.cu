// Sequential pointer selection (Sec. 3.2, Eq. 4; grouped rounds Sec. 3.5) from
// the per-episode inner-product tables of gram.cu: the same rounds as
// select.cu's kernel, for episodes whose tables cost less than the time their
// rounds save.
//
// One cluster of C CTAs runs one episode; CTA c owns a contiguous slice of the
// candidates.  A round, with last history position `last` and t positions:
//   1. loads, all issued at once, a thread per position or column: the scores
//      S[last][hist], ZV[last][hist], the newest positions' VV rows and slices
//      of their G rows, Gz[last]; what later rounds need too (G, VV) stays in
//      shared memory.  (One gather for the block: with every warp gathering the
//      scores for itself, a tag lookup per scattered address, steps 1 and 2 took
//      2,050 cycles at up to 192 positions, 1,780 so.)
//   2. every warp takes the softmax weights of the t scores into registers (four
//      consecutive positions per lane);
//   3. warp w multiplies the positions k = w mod 8, into its partial logits and
//      its part of the variance: one 16-byte load per position and lane covers
//      128 columns of a G slice or of a VV row (the loop is bound by its
//      instructions, not by shared memory);
//   4. block barrier; a thread per candidate sums the partials (warp order) and
//      applies rstd and the LN2 bias term.  g = 1: the logit goes to every CTA of
//      the cluster; grouped rounds: each warp's top g+1 does;
//   5. the CTA waits for all n logits (they count their bytes on its mbarrier; no
//      cluster barrier and no fence; a CTA without candidates sends one word, so
//      that nobody runs ahead of it) and finds the best, or, grouped, every warp
//      merges the lists after a cluster barrier; it takes the decision itself:
//      nothing else is exchanged.
// Three block barriers, one exchange and one trip to L2 per round, where the
// general kernel has six, two and two and reads its whole key slice from
// shared memory.  Latency-bound: the steps form one serial chain.  The margin
// trace (the second best logit) is worked out in the shadow of the next loads.
// Per round on GB300, general kernel -> here (rounds 97 to 192): 14 episodes of
// 576 with h = 512 5.9 -> 2.9 us, 4 of them 5.7 -> 2.4; 8 with the training
// aggregates 7.0 -> 3.4; one with h = 256 5.2 -> 2.5; one with g = 5 10.2 -> 5.2.
// (16 run in two waves of clusters on a card with room for 15: 12.1 -> 5.3.)
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "select_common.cuh"
#include "select_slices.h"

namespace cg = cooperative_groups;

namespace sp {

namespace {

constexpr int NT = 256;
constexpr int NW = NT / 32;
constexpr int kMaxCluster = 8;
constexpr int kMaxSlice = 127; // a slice and STOP: four columns per lane
constexpr int kMaxHist = 224; // history positions (START and the selected), eight per lane
constexpr size_t kSmemBudget = 225 * 1024;

struct GramSmem {
  size_t G, vv, lgp, qp, sc, zv, key, tv, ti, misc, total;
};

__host__ __device__ inline size_t al16g(size_t x) { return (x + 15) & ~size_t(15); }
__host__ __device__ inline int up4(int x) { return (x + 3) & ~3; }

// first float of VV row k: rows of up4(k + 1) floats, one after the other
__host__ __device__ inline int vv_row(int k) { return 4 * ((k >> 2) + 1) * (2 * (k >> 2) + (k & 3)); }

// T: history positions; n_loc: largest slice; g = 1: keys of all candidates, else lists
__host__ __device__ inline GramSmem gram_smem(int T, int n_loc, int C, int per) {
  GramSmem L;
  const int lc = up4(n_loc + 1);
  size_t o = 0;
  L.G = o;    o += (size_t)T * lc * 4;
  L.vv = o;   o += (size_t)vv_row(T) * 4;
  L.lgp = o;  o += (size_t)NW * lc * 4;
  L.qp = o;   o += NW * 16;
  L.sc = o;   o += (size_t)up4(T) * 4;
  L.zv = o;   o += (size_t)up4(T) * 4;
  const int lists = C * ((n_loc + 31) / 32);
  L.key = o;  o += per == 2 ? al16g((size_t)2 * C * n_loc * 4) : 0;
  L.tv = o;   o += per == 2 ? 0 : al16g((size_t)2 * lists * per * 4);
  L.ti = o;   o += per == 2 ? 0 : al16g((size_t)2 * lists * per * 4);
  // raw STOP logit and barrier by round parity; the warps' best keys and softmax sums
  L.misc = o; o += 32 + NW * 16;
  L.total = o;
  return L;
}

// Bounded wait by polling (test_wait): the exchange is a few hundred cycles away, and a thread that try_wait
// suspends wakes later than it completes.  Warp-uniform, lane 0 polls.
SP_DEVINL bool mbar_poll_cluster_warp(uint64_t* bar, uint32_t parity, int* err) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) {
    uint64_t t0 = 0;
    for (uint32_t i = 1;; ++i) {
      uint32_t done;
      asm volatile(
          "{\n"
          ".reg .pred p;\n"
          "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
          "selp.u32 %0, 1, 0, p;\n"
          "}\n"
          : "=r"(done)
          : "r"(smem_u32(bar)), "r"(parity)
          : "memory");
      if (done) break;
      if ((i & 1023u) == 0) {
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) {
          t0 = now;
        } else if (now - t0 > kWaitLimitNs) {
          set_error(err, SP_DEVERR_TIMEOUT);
          ok = false;
          break;
        }
      }
    }
  }
  __syncwarp();  // (orders the other lanes' reads behind lane 0's acquire: a shuffle does not)
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// LN2's variance from the tables is a sum of products of either sign. Where the
// residual and the attention output, or the values among themselves, cancel, its
// rounding grows with the square of the cancellation, that of the formed vector
// only with its first power. In the careful form of the rounds the vector is
// formed where the variance is below 1 / kCancel of what its terms come to
// without the cross terms (rows independent of one another: near 1; at 1 / 8 the
// tables' variance is still good to 3e-6). The usual form is for episodes where
// that cannot happen: no value longer than half of any residual (the ratio stays
// above 0.2), and START by itself no cancellation. Each form is a kernel, and
// both are launched: the usual one asks the question as it starts and leaves its
// answer in the table for the other. (Asked in every round it costs 2 to 5 % of
// the rounds, and with both forms in one kernel the usual one was 15 % slower;
// the question and the second launch are 2 to 5 us a call.)
constexpr float kCancel = 8.f;

// |zc_last + sum_k p_k vc_k|^2 from the operand rows of the tables (their fp16
// parts sum to the fp32 row up to 2^-23), all threads of the block: t rows of
// 4 h bytes from L2 by every CTA, in place of a few adds.  p_k = exp(sc_s[k] -
// mx) inv_sum; hist_s: the positions' rows, not yet synchronised; red: NW floats.
__device__ __noinline__ float direct_variance(const __half2* op, const float* inv, int rows, int base, int h, int last,
                                              int t, const float* sc_s, float mx, float inv_sum, const int* hist_s,
                                              float* red) {
  __syncthreads();
  const int h2 = h >> 1;
  auto row_of = [&](int m, int i) { return op + ((size_t)m * rows + base + i) * h; };
  auto at = [&](const __half2* r, int c) {
    const float2 a = __half22float2(r[c]), b = __half22float2(r[h2 + c]);
    return make_float2(a.x + b.x, a.y + b.y);
  };
  float s = 0.f;
  for (int c = threadIdx.x; c < h2; c += NT) {
    float2 o = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < t; ++k) {
      const int i = hist_s[k];
      const float p = __expf(sc_s[k] - mx) * inv[2 * rows + base + i];
      const float2 v = at(row_of(2, i), c);
      o.x = fmaf(p, v.x, o.x);
      o.y = fmaf(p, v.y, o.y);
    }
    const float iz = inv[3 * rows + base + last];
    const float2 z = at(row_of(3, last), c);
    const float x = fmaf(z.x, iz, o.x * inv_sum), y = fmaf(z.y, iz, o.y * inv_sum);
    s = fmaf(x, x, fmaf(y, y, s));
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  s = 0.f;
#pragma unroll
  for (int w = 0; w < NW; ++w) s += red[w];
  __syncthreads();
  return s;
}

// GL: capacity of the top lists (g + 1 <= GL).
template <int GL, bool TRAIN, bool CAREFUL>
__global__ void __launch_bounds__(NT, 1)
select_gram_kernel(const BatchDesc bd, const SelectArgs a, const GramArgs gr, int n_loc_max, int T_max) {
  constexpr int NG = GL - 1;  // new positions per round at most
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int e = blockIdx.x / C;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k_max = a.k_max, g = a.g, per = g + 1;
  pdl_wait();
  pdl_trigger();

  int lo = 0, hi = bd.B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (bd.ep_off[mid] <= e) lo = mid; else hi = mid - 1;
  }
  const int n_img = bd.vis_off[lo + 1] - bd.vis_off[lo];
  const int gs = bd.group_size > 0 ? bd.group_size : n_img;
  const int c0 = (e - bd.ep_off[lo]) * gs;
  const int n = min(gs, n_img - c0);
  const int row0 = bd.vis_off[lo] + c0;
  const int base = row0 + 2 * e;  // operand row of candidate 0
  const Slice slice = slice_of(n, C, rank);
  const int j0 = slice.j0, nl = slice.nl;
  const int round_bytes = 4 * words_of_round(n, C);
  const int lc = up4(n_loc_max + 1);
  const int wl = (n_loc_max + 31) >> 5;  // warps (lists) per CTA
  const int lists = C * wl;

  float* tab = gr.table + (size_t)e * gr.ep_stride;
  const int ld = gr.ld;
  float* flag = tab + (size_t)n * (5 * ld);  // (STOP is never in the history: its row is free)
  if (CAREFUL && *flag == 0.f) return;

  extern __shared__ __align__(16) uint8_t sm[];
  const GramSmem L = gram_smem(T_max, n_loc_max, C, per);
  float* Gs = reinterpret_cast<float*>(sm + L.G);
  float* vvs = reinterpret_cast<float*>(sm + L.vv);  // rows vv_row(k), off the diagonal doubled, padded with zeros
  float* lgp = reinterpret_cast<float*>(sm + L.lgp);
  float4* qp = reinterpret_cast<float4*>(sm + L.qp);
  float* sc_s = reinterpret_cast<float*>(sm + L.sc);
  float* zv_s = reinterpret_cast<float*>(sm + L.zv);
  uint32_t* all_key = reinterpret_cast<uint32_t*>(sm + L.key);  // [parity][C * n_loc_max]: candidates' keys, 0: taken
  float* all_tv = reinterpret_cast<float*>(sm + L.tv);
  int* all_ti = reinterpret_cast<int*>(sm + L.ti);
  float* stop_s = reinterpret_cast<float*>(sm + L.misc);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + L.misc + 16);
  uint4* best_s = reinterpret_cast<uint4*>(sm + L.misc + 32);  // per warp: key, index, softmax sum

  const float bias = __ldg(a.stop_bias + e);
  const size_t trace = (size_t)e * (k_max + 1);
  const bool tracer = rank == 0 && tid == NT - 32;    // writes the traces, in a warp without a candidate list
  const bool is_col = tid <= nl;                      // candidate of this CTA, or (tid == nl) STOP
  const int col = tid < nl ? j0 + tid : n;            // its column of G and Gz
  const float dj = is_col ? gr.dj[base + col] : 0.f;
  const float inv_h = 1.f / (float)a.h;
  bool avail = tid < nl;
  float score = 0.f;                                  // Eq. 6 of this thread's candidate (TRAIN)
  float alive = 1.f, disc = a.beta, kbar_acc = 0.f;   // A_t, beta^t, Eq. 7 (TRAIN)

  const int n_keys = C * n_loc_max;
  // margin and gap of a round whose keys are still in buffer kbuf (warp NW - 1 of rank 0, g = 1): the second
  // best logit is the best one without candidate jbest
  auto trace_round = [&](int rnd, int kbuf, int jbest, float vbest, float raw, int navail) {
    if (a.margin) {
      uint32_t k2 = 0u;
      for (int j = lane; j < n; j += 32) {
        const uint32_t k = all_key[kbuf * n_keys + j];
        k2 = j != jbest && k > k2 ? k : k2;
      }
      k2 = __reduce_max_sync(0xffffffffu, k2);
      if (lane == 0) {  // the best two of {best, second, STOP}
        const float stop = raw + bias, v2 = fkey_inv(k2);
        const float hi = fmaxf(vbest, stop), lo = fminf(vbest, stop);
        a.margin[trace + rnd] = hi - (navail > 1 ? fmaxf(lo, v2) : lo);
      }
    }
    if (a.gap && lane == 0) a.gap[trace + rnd] = vbest - raw;
  };
  const bool trace_warp = GL == 2 && rank == 0 && warp == NW - 1;
  float tr_best = 0.f, tr_raw = 0.f;
  int tr_j = -1, tr_round = 0, tr_nsel = 0;  // (-1: no round to trace)

  float vmax = 0.f, zmin = INFINITY, z2 = 0.f, zv2 = 0.f, v2 = 0.f;  // squared lengths; START's products
  if (!CAREFUL) {
    const float* start = tab + (size_t)(n + 1) * (5 * ld) + n + 1;
    z2 = gr.zz[base + n + 1];
    v2 = start[3 * ld];
    zv2 = start[4 * ld];
    for (int i = tid; i < n; i += NT) {
      vmax = fmaxf(vmax, tab[(size_t)i * (5 * ld) + 3 * ld + i]);
      zmin = fminf(zmin, gr.zz[base + i]);
    }
    vmax = warp_max(vmax);
    zmin = -warp_max(-zmin);
    if (lane == 0) qp[warp] = make_float4(vmax, zmin, 0.f, 0.f);
  }
  if (GL == 2) {
    if (tid == 0) {
      mbar_init(&mbar[0], 1);
      mbar_init(&mbar[1], 1);
      fence_mbar_init();
    }
  }
  cluster.sync();  // every CTA has started, and its barriers are ready, before the first push

  if (!CAREFUL) {
    vmax = v2;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      vmax = fmaxf(vmax, qp[w].x);
      zmin = fminf(zmin, qp[w].y);
    }
    const bool careful = 4.f * vmax > zmin || kCancel * (z2 + 2.f * zv2 + v2) < z2 + v2;  // (the same in every CTA)
    if (rank == 0 && tid == 0) *flag = careful ? 1.f : 0.f;
    if (careful) return;
  }

  int hist = n + 1;  // index of history position tid (START at 0)
  int hnew[NG];      // positions that joined last
#pragma unroll
  for (int q = 0; q < NG; ++q) hnew[q] = n + 1;
  int nnew = 1, last = n + 1;
  int nsel = 0, round = 0;

  while (nsel < k_max) {
    const int n_avail = n - nsel;
    if (n_avail == 0) {  // only STOP remains: it wins this round
      if (tracer) {
        if (a.margin) a.margin[trace + round] = INFINITY;
        if (a.gap) a.gap[trace + round] = -INFINITY;
      }
      ++round;
      break;
    }
    const int buf = round & 1;
    const int t = nsel + 1, t0 = t - nnew;

    // ---- 1. loads
    const float* lrow = tab + last * (5 * ld);
    const bool is_pos = tid < t;
    float sc = 0.f, zv = 0.f, gz = 0.f;
    float vn[NG], gn[NG];
    if (is_pos) sc = lrow[2 * ld + hist];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const float* nrow = tab + hnew[q] * (5 * ld);
      vn[q] = gn[q] = 0.f;
      if (q < nnew && tid <= t0 + q) vn[q] = nrow[3 * ld + hist];
      if (q < nnew && is_col) gn[q] = nrow[col];
    }
    if (is_pos) zv = lrow[4 * ld + hist];
    if (is_col) gz = lrow[ld + col];
    const float zz = gr.zz[base + last];
    if (trace_warp && tr_j >= 0) trace_round(round - 1, buf ^ 1, tr_j, tr_best, tr_raw, n - tr_nsel);
    if (tid < up4(t)) {  // (padded for 16-byte reads)
      sc_s[tid] = is_pos ? sc : -INFINITY;
      zv_s[tid] = zv;
    }
    // the words of every CTA, the keys of all n candidates among them, arrive on this round's barrier
    if (GL == 2 && tid == 0) mbar_arrive_expect_tx(&mbar[buf], (uint32_t)round_bytes);
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      const int k = t0 + q;
      if (q < nnew && is_col) Gs[k * lc + tid] = gn[q];
      if (q < nnew && tid < up4(k + 1)) vvs[vv_row(k) + tid] = tid < k ? 2.f * vn[q] : vn[q];
    }
    __syncthreads();

    // ---- 2. softmax weights relative to the largest score (their sum is applied at the end)
    float4 p0 = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), p1 = p0;
    const int i0 = 4 * lane, i1 = 128 + 4 * lane;
    if (i0 < t) p0 = reinterpret_cast<const float4*>(sc_s)[lane];
    if (i1 < t) p1 = reinterpret_cast<const float4*>(sc_s)[32 + lane];
    const float mx = warp_max(fmaxf(fmaxf(fmaxf(p0.x, p0.y), fmaxf(p0.z, p0.w)),
                                    fmaxf(fmaxf(p1.x, p1.y), fmaxf(p1.z, p1.w))));
    auto expo = [&](float4& x) {
      x = make_float4(__expf(x.x - mx), __expf(x.y - mx), __expf(x.z - mx), __expf(x.w - mx));
    };
    expo(p0);
    if (t > 128) expo(p1); else p1 = make_float4(0.f, 0.f, 0.f, 0.f);
    float lin = 0.f;
    if (warp == 0) {
      auto dot = [&](const float4& x, int i) {
        const float4 z = reinterpret_cast<const float4*>(zv_s)[i];
        lin += fmaf(x.x, z.x, x.y * z.y) + fmaf(x.z, z.z, x.w * z.w);
      };
      if (i0 < t) dot(p0, lane);
      if (i1 < t) dot(p1, 32 + lane);
    }

    float own = 0.f;  // this thread's position by itself
    if (CAREFUL && is_pos) {
      const float p = __expf(sc - mx);
      own = p * p * vvs[vv_row(tid) + tid];
    }

    // ---- 3. this warp's positions
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float quad = 0.f, sum = 0.f;
    // (no lane branches: columns past nl and entries past k are read where other rows lie and not used)
    const float* gk = Gs + warp * lc + i0;
#pragma unroll 4
    for (int k = warp; k < t; k += NW, gk += NW * lc) {
      const float pk = __expf(sc_s[k] - mx);
      const float4 x = *reinterpret_cast<const float4*>(gk);
      const float* vk = vvs + vv_row(k) + i0;
      const float4 y = *reinterpret_cast<const float4*>(vk);
      acc.x = fmaf(pk, x.x, acc.x);
      acc.y = fmaf(pk, x.y, acc.y);
      acc.z = fmaf(pk, x.z, acc.z);
      acc.w = fmaf(pk, x.w, acc.w);
      const float s = fmaf(p0.x, y.x, p0.y * y.y) + fmaf(p0.z, y.z, p0.w * y.w);
      quad = fmaf(pk, i0 <= k ? s : 0.f, quad);
      sum += pk;
    }
    for (int k = 128 + warp; k < t; k += NW) {  // the rows' entries from 128 on
      const float4 y = *reinterpret_cast<const float4*>(vvs + vv_row(k) + min(i1, k & ~3));
      const float s = fmaf(p1.x, y.x, p1.y * y.y) + fmaf(p1.z, y.z, p1.w * y.w);
      quad = fmaf(__expf(sc_s[k] - mx), i1 <= k ? s : 0.f, quad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      quad += __shfl_xor_sync(0xffffffffu, quad, o);
      lin += __shfl_xor_sync(0xffffffffu, lin, o);
      if (CAREFUL) own += __shfl_xor_sync(0xffffffffu, own, o);
    }
    if (lane == 0) qp[warp] = make_float4(sum, lin, quad, own);
    if (i0 <= nl) *reinterpret_cast<float4*>(lgp + warp * lc + i0) = acc;
    __syncthreads();

    // ---- 4. logits, exchange
    float v = -INFINITY;
    float formed = -1.f;
    if (CAREFUL) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float4 y = qp[w];
        x.x += y.x;
        x.y += y.y;
        x.z += y.z;
        x.w += y.w;
      }
      const float inv = 1.f / x.x;
      if (kCancel * (zz + inv * (2.f * x.y + inv * x.z)) < zz + inv * inv * x.w) {  // (the same in every CTA)
        int* hist_s = reinterpret_cast<int*>(zv_s);
        if (is_pos) hist_s[tid] = hist;
        formed = direct_variance(static_cast<const __half2*>(gr.op), gr.inv, gr.rows, base, a.h, last, t, sc_s, mx, inv,
                                 hist_s, reinterpret_cast<float*>(best_s));
      }
    }
    if (warp <= (n_loc_max >> 5)) {  // (threads 0 .. nl)
      float ps = 0.f, pl = 0.f, pq = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float4 x = qp[w];
        ps += x.x;
        pl += x.y;
        pq += x.z;
      }
      const float inv = 1.f / ps;
      const float var = CAREFUL && formed >= 0.f ? formed : zz + inv * (2.f * pl + inv * pq);
      const float rstd = rsqrtf(fmaxf(var * inv_h, 0.f) + a.ln_eps);
      if (is_col) {
        float x = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) x += lgp[w * lc + tid];
        v = fmaf(fmaf(x, inv, gz), rstd, dj);
        if (tid == nl) stop_s[buf] = v;
      }
      if (GL == 2) {
        if (tid < slice.words) {
          const uint32_t key = avail ? logit_key(v, gr.pass_nan) : 0u;
          const uint32_t d = smem_u32(all_key + buf * n_keys + j0 + tid), mb = smem_u32(&mbar[buf]);
#pragma unroll
          for (int r = 0; r < kMaxCluster; ++r)
            if (r < C) st_async_u32(mapa_shared(d, r), key, mapa_shared(mb, r));
        }
      } else if (warp < wl) {
        int id = avail ? col : INT_MAX;
        uint32_t key = avail ? logit_key(v, gr.pass_nan) : 0u;
        float* dv = all_tv + (size_t)(buf * lists + rank * wl + warp) * per;
        int* di = all_ti + (size_t)(buf * lists + rank * wl + warp) * per;
        if (lane < C) {
          dv = cluster.map_shared_rank(dv, lane);
          di = cluster.map_shared_rank(di, lane);
        }
#pragma unroll
        for (int r = 0; r < GL; ++r) {
          if (r < per) {
            const uint32_t mk = __reduce_max_sync(0xffffffffu, key);
            const int mi = (int)__reduce_min_sync(0xffffffffu, key == mk ? (uint32_t)id : 0x7fffffffu);
            if (lane < C) {
              dv[r] = fkey_inv(mk);
              di[r] = mk ? mi : INT_MAX;
            }
            if (id == mi) { key = 0u; id = INT_MAX; }
          }
        }
      }
    }
    bool ok = true;
    if (GL == 2)
      ok = mbar_poll_cluster_warp(&mbar[buf], (round >> 1) & 1, a.err);
    else
      cluster.sync();

    // ---- 5. the best of all and the decision, identically in every warp
    float tv[GL];
    int ti[GL];
    float stop_raw, stop_logit;
    if (GL == 2) {
      // candidates tid + 256 i: this warp's best (largest key, lowest index), then the block's
      const uint32_t* keys = all_key + buf * n_keys;
      uint32_t k[4], kw = 0u, jw = 0x7fffffffu;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        k[i] = tid + NT * i < n ? keys[tid + NT * i] : 0u;
        kw = max(kw, k[i]);
      }
      kw = __reduce_max_sync(0xffffffffu, kw);
#pragma unroll
      for (int i = 3; i >= 0; --i)
        if (k[i] == kw) jw = tid + NT * i;
      jw = __reduce_min_sync(0xffffffffu, jw);
      float z = 0.f;
      if (TRAIN) {  // the warp's softmax partial relative to its best logit
        const float m = fkey_inv(kw);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float ex = expf((fkey_inv(k[i]) - m) * a.inv_tau);
          z += k[i] ? ex : 0.f;
        }
        z = warp_sum(z);
      }
      if (lane == 0) best_s[warp] = make_uint4(kw, jw, __float_as_uint(z), 0u);
      if (__syncthreads_or(!ok)) break;  // a wait ran out: the error word says so, the cluster unwinds
      stop_raw = stop_s[buf];
      stop_logit = stop_raw + bias;
      uint32_t kb = 0u, jb = 0x7fffffffu;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const uint2 x = *reinterpret_cast<const uint2*>(&best_s[w]);
        const bool up = x.x > kb || (x.x == kb && x.y < jb);
        kb = up ? x.x : kb;
        jb = up ? x.y : jb;
      }
      tv[0] = fkey_inv(kb);
      ti[0] = kb ? (int)jb : INT_MAX;
      tr_best = tv[0];
      tr_raw = stop_raw;
      tr_j = ti[0];
      tr_round = round;
      tr_nsel = nsel;
      if (TRAIN && (warp < wl || warp == NW - 1)) {  // p_t = softmax(l_t / tau) over the available candidates and STOP
        const float top = fmaxf(tv[0], stop_logit);
        const uint4 x = best_s[lane & (NW - 1)];
        const float ex = expf((fkey_inv(x.x) - top) * a.inv_tau);
        float zs = x.x ? __uint_as_float(x.z) * ex : 0.f;
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) zs += __shfl_xor_sync(0xffffffffu, zs, o);
        const float es = expf((stop_logit - top) * a.inv_tau);
        const float iz = 1.f / (zs + es);
        const float ps = es / (zs + es);
        // Eqs. 5-7
        const float ev = expf((v - top) * a.inv_tau);
        score += avail ? alive * disc * (ev * iz) : 0.f;
        kbar_acc += alive * (1.f - ps);
        alive *= 1.f - ps;
        disc *= a.beta;
      }
    } else {
      stop_raw = stop_s[buf];
      stop_logit = stop_raw + bias;
      warp_merge_lists<GL, GL>(all_tv + (size_t)buf * lists * per, all_ti + (size_t)buf * lists * per, lists * per,
                               per, tv, ti);
    }
    const float best = tv[0];
    if (GL > 2 && tracer) {
      if (a.gap) a.gap[trace + round] = best - stop_raw;
      if (a.margin) {
        // smallest gap between consecutive values among the top g+1 of
        // {available visual logits} U {STOP}: STOP bubbles down the list
        const int nv = min(per, n_avail);
        const int use = min(nv + 1, per);
        float mg = INFINITY, c = stop_logit, prev = 0.f;
#pragma unroll
        for (int k = 0; k <= GL; ++k) {
          float x = c;
          if (k < GL && k < nv) {
            const float tk = tv[k < GL ? k : 0];
            x = fmaxf(tk, c);
            c = fminf(tk, c);
          }
          if (k > 0 && k < use) mg = fminf(mg, prev - x);
          prev = x;
        }
        a.margin[trace + round] = mg;
      }
    }
    ++round;
    if (stop_logit > best) break;  // STOP
    const int take = min(min(g, k_max - nsel), n_avail);
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      if (q < take) {
        int j = ti[q];
        if (j < 0 || j >= n) {
          if (tid == 0) set_error(a.err, SP_DEVERR_INDEX);
          j = n + 1;
        } else if (tracer && a.order) {
          a.order[(size_t)e * k_max + nsel + q] = j;
        }
        if (tid < nl && j == col) avail = false;
        hnew[q] = j;
        last = j;
        if (tid == t + q) hist = j;
      }
    }
    nnew = take;
    nsel += take;
  }
  if (trace_warp && tr_j >= 0) trace_round(tr_round, tr_round & 1, tr_j, tr_best, tr_raw, n - tr_nsel);
  if (tracer) {
    if (a.ep_count) a.ep_count[e] = nsel;
    if (a.rounds) a.rounds[e] = round;
    if (TRAIN) a.kbar[e] = kbar_acc;
  }
  if (TRAIN && tid < nl) a.score[row0 + j0 + tid] = score;
  cluster.sync();  // no CTA leaves while a peer may still write into it
}

}  // namespace

// START and every selected candidate but the last
static int gram_history(int k_max, int n_max) { return std::min(k_max, n_max); }

int select_gram_cluster(int n_max, int k_max, int g) {
  const int T = gram_history(k_max, n_max);
  if (T > kMaxHist) return 0;
  const int n_loc = (n_max + kMaxCluster - 1) / kMaxCluster;
  return n_loc <= kMaxSlice && gram_smem(T, n_loc, kMaxCluster, g + 1).total <= kSmemBudget ? kMaxCluster : 0;
}

template <bool CAREFUL>
static cudaError_t launch_form(const BatchDesc& bd, int n_episodes, const SelectArgs& a, const GramArgs& g, int n_loc,
                               int T, int C, cudaStream_t st) {
  const int per = a.g + 1;
  void (*kern)(const BatchDesc, const SelectArgs, const GramArgs, int, int) =
      a.score ? select_gram_kernel<2, true, CAREFUL>
              : (per <= 2 ? select_gram_kernel<2, false, CAREFUL>
                          : (per <= 6 ? select_gram_kernel<6, false, CAREFUL> : select_gram_kernel<17, false, CAREFUL>));
  // (one limit whatever the size: another thread may set it between this call and the launch)
  cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
  if (r != cudaSuccess) return r;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_episodes * C, 1, 1);
  cfg.blockDim = dim3(NT, 1, 1);
  cfg.dynamicSmemBytes = gram_smem(T, n_loc, C, per).total;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  prof_begin_launch(st);
  r = cudaLaunchKernelEx(&cfg, kern, bd, a, g, n_loc, T);
  prof_end_launch(st, SP_K_SELECT, 0.0, 0.0);
  return r;
}

cudaError_t select_gram_launch(const BatchDesc& bd, int n_episodes, const SelectArgs& a, const GramArgs& g, int n_max,
                               int C, cudaStream_t st) {
  if (n_episodes <= 0) return cudaSuccess;
  const int n_loc = (n_max + C - 1) / C;
  const int T = gram_history(a.k_max, n_max);
  const bool train = a.score != nullptr;
  if (train && (a.g != 1 || !a.kbar)) return cudaErrorInvalidValue;
  if (T > kMaxHist || C > kMaxCluster) return cudaErrorInvalidValue;
  const cudaError_t r = launch_form<false>(bd, n_episodes, a, g, n_loc, T, C, st);
  return r == cudaSuccess ? launch_form<true>(bd, n_episodes, a, g, n_loc, T, C, st) : r;
}

}  // namespace sp
