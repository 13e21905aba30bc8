// Merge of the unselected tokens into contextual tokens on sm_103a (Section 2.3, Stage 2: Rift
// uses VisionZip's mechanism to keep the dominant tokens and merge the remainder).
//
// For kept slot j with m_j = budgets[j] - s_j contextual tokens (s_j selected tokens):
//   merge_plan_kernel     m_j (capped at the R_j unselected tokens) and their offsets ctx_off
//   merge_targets_kernel  the unselected tokens in ascending index, the targets (every
//                         floor(R_j / m_j)-th of them from the first) and the targets' norms
//   merge_assign_kernel   (fp32 tokens) per 64 unselected tokens x 64 targets: fp32 dot products in
//                         32-term chunks, a running top 2 per token; the two are recomputed as
//                         float-float sums (good to ~2^-44) and compared as x.t1 / ||t1|| vs
//                         x.t2 / ||t2|| in fp64, so the decision is the cosine argmax of the exact
//                         arithmetic (ties to the lower target); where a third is within the fp32 sums' error
//                         of the best, all are compared
//   (bf16 tokens) merge_screen_kernel (gemm_tc.cu) lists the targets whose tcgen05 product is
//                         within its error bound of the best one's, for each 128 tokens of a slot, and
//                         merge_decide_kernel makes the same float-float decision among them
//   merge_mean_kernel     per contextual token: its members in ascending token index, the fp32 sum
//                         of their rows in that order, divided by the group size, stored as bf16
#include <type_traits>

#include "rift_internal.h"

namespace rift {

__device__ unsigned int g_err_merge;

unsigned int read_clear_err_merge() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_err_merge, sizeof(v));
  cudaMemcpyToSymbol(g_err_merge, &z, sizeof(z));
  return v;
}

namespace mg {

constexpr int TB = 64;     // tokens and targets per block of the similarity pass
constexpr int KC = 32;     // d-chunk staged per step (summed in 32-term sub-chunks)

// Eight consecutive elements of a row (16-byte aligned) as floats.
template <typename XT>
__device__ __forceinline__ void load8(const XT* p, float (&v)[8]) {
  if constexpr (sizeof(XT) == 2) {
    unpack_bf16x8(*reinterpret_cast<const uint4*>(p), v);
  } else {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
}

// a.b += into the float-float pair (hi, lo): TwoProduct with an FMA, then TwoSum.
__device__ __forceinline__ void ff_step(float x, float y, float& hi, float& lo) {
  const float p = __fmul_rn(x, y);
  const float pe = fmaf(x, y, -p);
  const float s = __fadd_rn(hi, p);
  const float bb = __fsub_rn(s, hi);
  const float er = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(er, pe));
}

// The sum of the lanes' float-float pairs in fp64, in every lane.
__device__ __forceinline__ double ff_warp_sum(float hi, float lo) {
  double acc = (double)hi + (double)lo;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// Two such sums at once (both in every lane): the halves of the warp take one each after the first step, so that
// the pair costs as many fp64 additions a lane as one sum does (an SM retires about two a cycle).
__device__ __forceinline__ double2 ff_warp_sum2(float h1, float l1, float h2, float l2) {
  const double a = (double)h1 + (double)l1, b = (double)h2 + (double)l2;
  const bool upper = (threadIdx.x & 16) != 0;
  double acc = upper ? b : a;
  acc += __shfl_xor_sync(0xffffffffu, upper ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return make_double2(__shfl_sync(0xffffffffu, acc, 0), __shfl_sync(0xffffffffu, acc, 16));
}

// Float-float accumulation of a.b over d terms by one warp, eight elements per lane and step, U steps' loads ahead of
// the serial chain, then the lanes' pairs summed (~2^-44 relative).
template <int U, typename XT>
__device__ double ff_dot(const XT* a, const XT* b, int d, int lane) {
  float hi = 0.f, lo = 0.f;
  for (int k0 = lane * 8; k0 < d; k0 += U * 256) {
    float x[U][8], y[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * 256 < d) {
        load8(a + k0 + u * 256, x[u]);
        load8(b + k0 + u * 256, y[u]);
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * 256 < d) {
#pragma unroll
        for (int e = 0; e < 8; ++e) ff_step(x[u][e], y[u][e], hi, lo);
      }
  }
  return ff_warp_sum(hi, lo);
}

// m_j = min(budgets[j] - s_j, n_v - s_j) and its exclusive prefix sum over the kept slots.  If
// the total exceeds max_ctx, RIFT_EBIT_CAPACITY is set and every m_j is taken as 0 (no contextual
// row is then written or read).
__global__ void __launch_bounds__(1024) merge_plan_kernel(const int* __restrict__ n_kept,
                                                          const int* __restrict__ budgets,
                                                          const int* __restrict__ sel_off, int N, int n_v,
                                                          int max_ctx, int* __restrict__ ctx_off) {
  __shared__ int sh[33];
  pdl_trigger();
  pdl_wait();
  const int n = *n_kept;
  auto count = [&](int j) {
    const int s = sel_off[j + 1] - sel_off[j];
    return max(0, min(budgets[j] - s, n_v - s));
  };
  int total_all = 0;
  for (int c0 = 0; c0 < n; c0 += blockDim.x) {
    const int j = c0 + threadIdx.x;
    int total;
    block_excl_scan(j < n ? count(j) : 0, sh, &total);
    total_all += total;
  }
  const bool fits = total_all <= max_ctx;
  if (threadIdx.x == 0 && !fits) atomicOr(&g_err_merge, RIFT_EBIT_CAPACITY);
  int base = 0;
  for (int c0 = 0; c0 < n; c0 += blockDim.x) {
    const int j = c0 + threadIdx.x;
    const int m = (j < n && fits) ? count(j) : 0;
    int total;
    const int pos = block_excl_scan(m, sh, &total);
    if (j < n) ctx_off[j] = base + pos;
    base += total;
  }
  for (int j = n + threadIdx.x; j <= N; j += blockDim.x) ctx_off[j] = base;
}

// Grid (kept slot, y): rest[j][0 .. R) = the unselected tokens in ascending index (written by y = 0),
// the targets (written to ctx_target) and their norms (tnorm, fp64 from a float-float sum of
// squares), one target per warp: the warps of the TY CTAs take targets y * 8 + warp, + TY * 8, ...
// The norm is a serial float-float chain, so the targets are spread over many warps, and a row is read
// once for its norm and its copy (400 tiles, about 95 kept, 45 targets a slot: 17 us; 20 with the copy
// in a loop of its own, 73 with one CTA per slot).
constexpr int TY = 8;
template <typename XT>
__global__ void __launch_bounds__(256) merge_targets_kernel(const XT* __restrict__ X, int n_v, int d,
                                                            const int* __restrict__ kept,
                                                            const int* __restrict__ n_kept,
                                                            const int* __restrict__ sel,
                                                            const int* __restrict__ sel_off,
                                                            const int* __restrict__ ctx_off, int max_ctx,
                                                            int* __restrict__ rest, int* __restrict__ ctx_target,
                                                            double* __restrict__ tnorm, float* __restrict__ tinv,
                                                            uint16_t* __restrict__ trow) {
  __shared__ unsigned char chosen[RIFT_MAX_NV];
  __shared__ int rj[RIFT_MAX_NV];
  __shared__ int sh[33];
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.x, y = blockIdx.y;
  if (j >= *n_kept) return;
  const int so = sel_off[j], s = sel_off[j + 1] - so;
  const int co = ctx_off[j], m = ctx_off[j + 1] - co;
  if (y > 0 && y * 8 >= m) return;
  for (int k = threadIdx.x; k < n_v; k += blockDim.x) chosen[k] = 0;
  __syncthreads();
  for (int q = threadIdx.x; q < s; q += blockDim.x) {
    const int k = sel[so + q];
    if (k >= 0 && k < n_v) chosen[k] = 1;
  }
  __syncthreads();
  int base = 0;
  for (int c0 = 0; c0 < n_v; c0 += blockDim.x) {
    const int k = c0 + threadIdx.x;
    const int f = (k < n_v && !chosen[k]) ? 1 : 0;
    int total;
    const int at = block_excl_scan(f, sh, &total);
    if (f) {
      rj[base + at] = k;
      if (y == 0) rest[(size_t)j * n_v + base + at] = k;
    }
    base += total;
  }
  __syncthreads();
  const int R = base;
  if (m == 0 || R == 0) return;
  const int step = R / m;
  const XT* Xt = X + (size_t)kept[j] * n_v * d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = y * 8 + warp; q < m; q += TY * 8) {
    const int t = rj[q * step];
    const XT* tr = Xt + (size_t)t * d;
    // the row's norm and, for the tensor-core screening (bf16 tokens), its copy, in one pass of eight
    // 16-byte loads ahead
    constexpr int U = sizeof(XT) == 2 ? 8 : 4;
    uint16_t* copy = trow && co + q < max_ctx ? trow + (size_t)(co + q) * d : nullptr;
    float hi = 0.f, lo = 0.f;
    for (int k0 = lane * 8; k0 < d; k0 += U * 256) {
      uint4 raw[U][sizeof(XT) / 2];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k0 + u * 256 < d)
#pragma unroll
          for (int r = 0; r < (int)sizeof(XT) / 2; ++r)
            raw[u][r] = reinterpret_cast<const uint4*>(tr + k0 + u * 256)[r];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k0 + u * 256 < d) {
          float x[8];
          if constexpr (sizeof(XT) == 2) {
            if (copy) *reinterpret_cast<uint4*>(copy + k0 + u * 256) = raw[u][0];
            unpack_bf16x8(raw[u][0], x);
          } else {
            const uint4 a = raw[u][0], b = raw[u][sizeof(XT) / 2 - 1];
            const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(w[e]);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) ff_step(x[e], x[e], hi, lo);
        }
    }
    const double nn = ff_warp_sum(hi, lo);
    if (co + q >= max_ctx) continue;
    if (lane == 0) {
      ctx_target[co + q] = t;
      tnorm[co + q] = sqrt(nn);
      if (tinv) tinv[co + q] = nn > 0.0 ? (float)(1.0 / sqrt(nn)) : 0.f;  // a zero target has similarity 0
    }
  }
}

// Grid (blocks of 64 unselected positions, kept slot), 8 warps: assign[j][a] = the screened target where no other is
// within the screening's error of it; the other tokens are listed and the warps take them in turn: the
// best of the candidates at ~fp64 accuracy, x.t / ||t|| from float-float dot products with the lanes' pairs
// summed in fp64 (ties to the lower target).  Candidates: the screening's list, or, where it is longer than that
// (near-duplicate targets, tokens next to zero), all targets of the slot but those whose row is
// a copy of an earlier target's (blank parts of a tile), which a tie never chooses; the warps share these.  34 us
// at 400 tiles (about 12% of the tokens have a list, most of two), against 111 with a second look at every token.
// Targets keep their own group.
constexpr int DT = 256;

// x.t1 and x.t2 by one warp, four steps' loads ahead of the serial chains.
__device__ __forceinline__ double2 ff_dots(const uint16_t* x, const uint16_t* t1, const uint16_t* t2, int d, int lane) {
  float h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f;
  for (int k0 = lane * 8; k0 < d; k0 += 4 * 256) {
    uint4 xr[4], r1[4], r2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k0 + u * 256 < d) {
        xr[u] = *reinterpret_cast<const uint4*>(x + k0 + u * 256);
        r1[u] = *reinterpret_cast<const uint4*>(t1 + k0 + u * 256);
        r2[u] = *reinterpret_cast<const uint4*>(t2 + k0 + u * 256);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k0 + u * 256 < d) {
        float xv[8], y1[8], y2[8];
        unpack_bf16x8(xr[u], xv);
        unpack_bf16x8(r1[u], y1);
        unpack_bf16x8(r2[u], y2);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          ff_step(xv[e], y1[e], h1, l1);
          ff_step(xv[e], y2[e], h2, l2);
        }
      }
  }
  return ff_warp_sum2(h1, l1, h2, l2);
}

__global__ void __launch_bounds__(DT, 2) merge_decide_kernel(const uint16_t* __restrict__ X, int n_v, int d,
                                                           const int* __restrict__ kept,
                                                           const int* __restrict__ n_kept,
                                                           const int* __restrict__ sel_off,
                                                           const int* __restrict__ ctx_off, int max_ctx,
                                                           const int* __restrict__ rest,
                                                           const int* __restrict__ ctx_target,
                                                           const double* __restrict__ tnorm,
                                                           const MergeCand* __restrict__ cand, int* __restrict__ assign) {
  __shared__ int open[64];        // the block's undecided tokens: those with a list from the front, those with all
  __shared__ MergeCand list[64];  // targets for candidates from the back, and their lists
  __shared__ int n_open, n_all;
  __shared__ unsigned char dup[RIFT_MAX_NV];  // target q's row is an earlier target's
  __shared__ double part_e[DT / 32], part_n[DT / 32];  // the warps' best among their share of all targets
  __shared__ int part_q[DT / 32];
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.y, a0 = blockIdx.x * 64;
  if (j >= *n_kept) return;
  const int R = n_v - (sel_off[j + 1] - sel_off[j]);
  const int co = ctx_off[j], m = ctx_off[j + 1] - co;
  if (m == 0 || co + m > max_ctx || a0 >= R) return;
  const int step = R / m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) n_open = n_all = 0;
  __syncthreads();
  const int al = a0 + threadIdx.x;
  if (threadIdx.x < 64 && al < R && !(al % step == 0 && al / step < m)) {
    const MergeCand c = cand[(size_t)j * n_v + al];
    if (c.c[0] >= m) {  // no finite similarity (a NaN token): the first target
      atomicOr(&g_err_merge, RIFT_EBIT_NONFINITE);
      assign[(size_t)j * n_v + al] = 0;
    } else if (c.c[1] >= m && !c.all) {
      assign[(size_t)j * n_v + al] = c.c[0];
    } else {
      const int at = c.all ? 63 - atomicAdd(&n_all, 1) : atomicAdd(&n_open, 1);
      open[at] = al;
      list[at] = c;
    }
  }
  __syncthreads();
  const uint16_t* Xt = X + (size_t)kept[j] * n_v * d;
  const int* target = ctx_target + co;
  const double* norm = tnorm + co;
  auto row = [&](int q) { return Xt + (size_t)target[q] * d; };
  // s1 = e1 / n1 vs s2 = e2 / n2 as e1 n2 vs e2 n1 (norms are positive; a zero target has similarity 0)
  struct Best {
    int q;
    double e, n;
    __device__ void offer(double e2, double norm2, int q2) {
      const double e0 = norm2 > 0.0 ? e2 : 0.0, n0 = norm2 > 0.0 ? norm2 : 1.0;
      const double s = e0 * n, s_best = e * n0;
      if (e0 == e0 && (q < 0 || s > s_best || (s == s_best && q2 < q))) {
        q = q2;
        e = e0;
        n = n0;
      }
    }
  };
  for (int i = warp; i < n_open; i += DT / 32) {
    const uint16_t* x = Xt + (size_t)rest[(size_t)j * n_v + open[i]] * d;
    Best best = {-1, 0.0, 1.0};
    for (int k = 0; k < MergeCand::MAX; k += 2) {
      const int t1 = list[i].c[k], t2 = k + 1 < MergeCand::MAX && list[i].c[k + 1] < m ? list[i].c[k + 1] : t1;
      if (t1 >= m) break;
      const double2 e = ff_dots(x, row(t1), row(t2), d, lane);
      best.offer(e.x, norm[t1], t1);
      best.offer(e.y, norm[t2], t2);
    }
    if (lane == 0) assign[(size_t)j * n_v + open[i]] = best.q < 0 ? list[i].c[0] : best.q;
  }
  if (n_all == 0) return;
  for (int q = warp; q < m; q += DT / 32) {  // a copy has its original's norm, bit for bit
    bool copy = false;
    const long long nq = __double_as_longlong(norm[q]);
    for (int p0 = 0; p0 < q && !copy; p0 += 32) {
      const int p = p0 + lane;
      unsigned eq = __ballot_sync(0xffffffffu, p < q && __double_as_longlong(norm[p < q ? p : q]) == nq);
      for (; eq && !copy; eq &= eq - 1) copy = same_row(row(p0 + __ffs(eq) - 1), row(q), d, lane);
    }
    if (lane == 0) dup[q] = copy;
  }
  __syncthreads();
  for (int i = 0; i < n_all; ++i) {  // the warps share the targets, two at a time
    const uint16_t* x = Xt + (size_t)rest[(size_t)j * n_v + open[63 - i]] * d;
    const bool zero = same_row<uint16_t>(x, nullptr, d, lane);  // all similarities are 0: the first target
    Best best = {-1, 0.0, 1.0};
    for (int q = 2 * warp; q < m && !zero; q += 2 * (DT / 32)) {
      const bool u1 = !dup[q], u2 = q + 1 < m && !dup[q + 1];
      if (!u1 && !u2) continue;
      const int t1 = u1 ? q : q + 1, t2 = u2 ? q + 1 : q;
      const double2 e = ff_dots(x, row(t1), row(t2), d, lane);
      best.offer(e.x, norm[t1], t1);
      best.offer(e.y, norm[t2], t2);
    }
    if (lane == 0) {
      part_q[warp] = best.q;
      part_e[warp] = best.e;
      part_n[warp] = best.n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < DT / 32; ++w)
        if (part_q[w] >= 0) best.offer(part_e[w], part_n[w], part_q[w]);
      assign[(size_t)j * n_v + open[63 - i]] = best.q < 0 ? list[63 - i].c[0] : best.q;
    }
    __syncthreads();
  }
}

// The best target for token k of a tile among `choice` and every `step`-th of the m from `first` on, by one warp:
// copies of the best so far are passed over, and a zero token (all similarities are 0) keeps its choice.
template <typename XT>
__device__ __noinline__ int best_of_all(const XT* Xt, int k, const int* target, const double* norm, int m, int d, int lane,
                                        int choice, int first, int step, double& best) {
  const XT* x = Xt + (size_t)k * d;
  best = 0.0;
  if (same_row<XT>(x, nullptr, d, lane)) return choice;
  auto row = [&](int q) { return Xt + (size_t)target[q] * d; };
  const int given = choice;
  for (int i = first - step; i < m; i += step) {  // the given choice first
    const int q = i < first ? given : i;
    if (i == given || (i > choice && __double_as_longlong(norm[q]) == __double_as_longlong(norm[choice]) &&
                       same_row(row(q), row(choice), d, lane)))
      continue;
    const double dt = ff_dot<1>(x, row(q), d, lane), s = norm[q] > 0.0 ? dt / norm[q] : 0.0;
    if (i < first || s > best || (s == best && q < choice)) {
      choice = q;
      best = s;
    }
  }
  return choice;
}

// Grid (block of TB unselected tokens, kept slot).  assign[j][a] = target index of rest[a].
// U: steps of loads ahead in the float-float dot products.  Four hide their latency where a CTA has an SM to itself, but
// take the registers of two more CTAs (164 against 80).  Launched without overlap: as a programmatic dependent its few
// CTAs with work land on the SMs that the kernel before it leaves first, several to one.  us of an fp32 scene with
// the merge at d = 4096, U = 4 : 1 (dependent launch, 1): 20 tiles of 100 tokens 378 : 429 (674), 64 of 576 722 : 726
// (883), 250 of 200 569 : 744 (893), 150 of 576 925 : 1015 (1037), 300 of 576 1481 : 1306 (1331); 700 of 576 at d = 1024
// 1101 : 1007 (1005).
template <typename XT, int U>
__global__ void __launch_bounds__(256) merge_assign_kernel(const XT* __restrict__ X, int n_v, int d,
                                                           const int* __restrict__ kept,
                                                           const int* __restrict__ n_kept,
                                                           const int* __restrict__ sel_off,
                                                           const int* __restrict__ ctx_off, int max_ctx,
                                                           const int* __restrict__ rest,
                                                           const int* __restrict__ ctx_target,
                                                           const double* __restrict__ tnorm,
                                                           int* __restrict__ assign) {
  extern __shared__ float ab_sm[];  // As[KC][TB + 4], Bs[KC][TB + 4]
  float (*As)[TB + 4] = reinterpret_cast<float (*)[TB + 4]>(ab_sm);
  float (*Bs)[TB + 4] = reinterpret_cast<float (*)[TB + 4]>(ab_sm + KC * (TB + 4));
  __shared__ float best_v[TB][3];  // the three highest similarities, the first two targets
  __shared__ int best_j[TB][2];
  __shared__ float inv_n[TB], row_ss[TB];
  __shared__ int far;              // a target's norm is below 2^-40
  __shared__ int twin[TB], any_twin;  // an earlier target of the same norm, or -1
  __shared__ int n_all, all[TB];   // rows with all targets for candidates
  __shared__ double part_s[8];
  __shared__ int part_q[8];
  pdl_wait();
  const int j = blockIdx.y;  // the token blocks of one slot are adjacent: its target rows stay in L2
  if (j >= *n_kept) return;
  const int s = sel_off[j + 1] - sel_off[j];
  const int R = n_v - s;
  const int co = ctx_off[j], m = ctx_off[j + 1] - co;
  const int a0 = blockIdx.x * TB;
  if (m == 0 || a0 >= R || co + m > max_ctx) return;
  const int* rj = rest + (size_t)j * n_v;
  const XT* Xt = X + (size_t)kept[j] * n_v * d;
  const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
  if (tid < TB) {
    best_v[tid][0] = best_v[tid][1] = best_v[tid][2] = -INFINITY;
    best_j[tid][0] = best_j[tid][1] = -1;
  }
  if (tid == 0) far = n_all = 0;
  __syncthreads();
  float ss = 0.f;  // of this thread's part of its token row
  for (int b0 = 0; b0 < m; b0 += TB) {
    if (tid < TB) {
      const double nn = b0 + tid < m ? tnorm[co + b0 + tid] : 0.0;
      inv_n[tid] = nn > 0.0 ? (float)(1.0 / nn) : 0.f;  // a zero target has similarity 0
      if (inv_n[tid] > 0x1p40f) far = 1;
    }
    // targets whose row is a copy of an earlier one's (blank parts of a tile): a tie never chooses them
    if (tid == 0) any_twin = 0;
    __syncthreads();
    if (tid < TB) {
      twin[tid] = -1;
      const int q = b0 + tid;
      for (int p = 0; q < m && p < q && twin[tid] < 0; ++p)
        if (__double_as_longlong(tnorm[co + p]) == __double_as_longlong(tnorm[co + q])) twin[tid] = p;
      if (twin[tid] >= 0) any_twin = 1;
    }
    __syncthreads();
    if (any_twin) {
      for (int q = tid >> 5; q < TB; q += 8)
        if (twin[q] >= 0 && same_row(Xt + (size_t)ctx_target[co + twin[q]] * d, Xt + (size_t)ctx_target[co + b0 + q] * d, d,
                                     tid & 31) &&
            (tid & 31) == 0)
          inv_n[q] = __int_as_float(0x7fffffff);  // NaN: no candidate
    }
    float acc[4][4] = {};
    // 64 rows x KC columns per operand and chunk: four 8-column groups per thread and operand,
    // kept packed while the next chunk's loads are in flight
    const int srow = tid >> 2, scol = (tid & 3) * 8;
    const XT* pa = a0 + srow < R ? Xt + (size_t)rj[a0 + srow] * d + scol : nullptr;
    const XT* pb = b0 + srow < m ? Xt + (size_t)ctx_target[co + b0 + srow] * d + scol : nullptr;
    constexpr int NG = KC / 32;  // 8-column groups per thread and operand
    float va[NG][8], vb[NG][8];
    auto fetch = [&](int k0) {
#pragma unroll
      for (int g = 0; g < NG; ++g) {
#pragma unroll
        for (int e = 0; e < 8; ++e) va[g][e] = vb[g][e] = 0.f;
        if (k0 + 32 * g >= d) continue;  // d % 32 == 0: a group is wholly inside the row or past it
        if (pa) load8(pa + k0 + 32 * g, va[g]);
        if (pb) load8(pb + k0 + 32 * g, vb[g]);
      }
    };
    fetch(0);
    for (int k0 = 0; k0 < d; k0 += KC) {
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          As[32 * g + scol + e][srow] = va[g][e];
          Bs[32 * g + scol + e][srow] = vb[g][e];
          if (b0 == 0) ss = fmaf(va[g][e], va[g][e], ss);
        }
      __syncthreads();
      if (k0 + KC < d) fetch(k0 + KC);
#pragma unroll 1
      for (int kc = 0; kc < KC; kc += 32) {
        float part[4][4] = {};
#pragma unroll 8
        for (int k = kc; k < kc + 32; ++k) {
          const float4 av = *reinterpret_cast<const float4*>(&As[k][ti * 4]);
          const float4 bv = *reinterpret_cast<const float4*>(&Bs[k][tj * 4]);
          const float aa[4] = {av.x, av.y, av.z, av.w}, bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) part[r][c] = fmaf(aa[r], bb[c], part[r][c]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] += part[r][c];
      }
      __syncthreads();
    }
    if (b0 == 0) {  // a row's four threads
      ss += __shfl_xor_sync(0xffffffffu, ss, 1);
      ss += __shfl_xor_sync(0xffffffffu, ss, 2);
      if ((tid & 3) == 0) row_ss[tid >> 2] = ss;
    }
    // running top 2, and the third value, per token: thread (ti, tj) offers its 4 x 4 candidates row by row
    for (int w = 0; w < 16; ++w) {
      if (tj == w) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int row = ti * 4 + r;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int b = b0 + tj * 4 + c;
            if (b >= m) continue;
            const float v = acc[r][c] * inv_n[tj * 4 + c];
            if (v > best_v[row][0] || (v == best_v[row][0] && b < best_j[row][0])) {
              best_v[row][2] = best_v[row][1];
              best_v[row][1] = best_v[row][0];
              best_j[row][1] = best_j[row][0];
              best_v[row][0] = v;
              best_j[row][0] = b;
            } else if (v > best_v[row][1] || (v == best_v[row][1] && b < best_j[row][1])) {
              best_v[row][2] = best_v[row][1];
              best_v[row][1] = v;
              best_j[row][1] = b;
            } else {
              best_v[row][2] = fmaxf(best_v[row][2], v);
            }
          }
        }
      }
      __syncthreads();
    }
  }
  // Decide between the top two at ~fp64 accuracy: x.t1 / ||t1|| vs x.t2 / ||t2||; where a third target is within the
  // product's error of the best, among all of them.  An fp32 similarity errs by at most
  // (32 + d / 32) 2^-24 ||x|| (chains of 32 products, then d / 32 sums, each rounded) and 2^-23 ||x|| from 1 / ||t|| and its
  // product; the difference of two by twice that.
  const int warp = tid >> 5, lane = tid & 31;
  for (int row = warp; row < TB; row += 8) {
    const int a = a0 + row;
    if (a >= R) break;
    const int k = rj[a];
    int choice = best_j[row][0];
    const int j2 = best_j[row][1];
    if (j2 >= 0) {
      const int t1 = ctx_target[co + choice], t2 = ctx_target[co + j2];
      const double d1 = ff_dot<U>(Xt + (size_t)k * d, Xt + (size_t)t1 * d, d, lane);
      const double d2 = ff_dot<U>(Xt + (size_t)k * d, Xt + (size_t)t2 * d, d, lane);
      const double n1 = tnorm[co + choice], n2 = tnorm[co + j2];
      const double s1 = n1 > 0.0 ? d1 / n1 : 0.0, s2 = n2 > 0.0 ? d2 / n2 : 0.0;
      if (s2 > s1 || (s2 == s1 && j2 < choice)) choice = j2;
      const float bound =
          row_ss[row] > 0x1p-60f && !far ? (48.f + (float)d / 32.f) * 0x1p-23f * sqrtf(row_ss[row]) : INFINITY;
      if (m > 2 && !(best_v[row][0] - best_v[row][2] > bound) && lane == 0) {
        best_j[row][0] = choice;
        all[atomicAdd(&n_all, 1)] = row;
      }
    }
    if (lane == 0) assign[(size_t)j * n_v + a] = choice;
  }
  __syncthreads();
  for (int i = 0; i < n_all; ++i) {  // the warps share the targets
    const int row = all[i], choice = best_j[row][0];
    double s;
    const int q = best_of_all(Xt, rj[a0 + row], ctx_target + co, tnorm + co, m, d, lane, choice, warp, 8, s);
    if (lane == 0) {
      part_q[warp] = q;
      part_s[warp] = s;
    }
    __syncthreads();
    if (tid == 0) {
      int w = 0;
      for (int o = 1; o < 8; ++o)
        if (part_s[o] > part_s[w] || (part_s[o] == part_s[w] && part_q[o] < part_q[w])) w = o;
      assign[(size_t)j * n_v + a0 + row] = part_q[w];
    }
    __syncthreads();
  }
}

// Grid (kept slot, 4096 columns, part), 256 threads of two groups of eight columns: the contextual tokens'
// means over the slot's unselected rows, read once, group after group, in ascending token index within a
// group (the target's own row and the tokens assigned to it): summed in fp32, divided by the group size
// and stored as bf16.  Each CTA takes its part (1 / MP) of the groups and sorts their tokens itself, a warp
// per group over the slot's groups in shared memory, so the rows' loads, MU rows ahead, do not wait for
// group boundaries.  A CTA reads whole 8 KB rows.  400 tiles, about 95 kept: 46 us; 61 with the slot's whole
// order placed by one warp and eight parts, which left a tile of few selected tokens to long CTAs (56 with the
// order alone, 48 in 16 parts); 73 in 1 KB pieces; 60 + 16 as two launches with a member at a time.
constexpr int MT = 256, MCOLS = 16 * MT, MU = 4, MP = 12;
template <typename XT>
__global__ void __launch_bounds__(MT) merge_mean_kernel(const XT* __restrict__ X, int n_v, int d,
                                                        const int* __restrict__ kept, const int* __restrict__ n_kept,
                                                        const int* __restrict__ sel_off,
                                                        const int* __restrict__ ctx_off, int max_ctx,
                                                        const int* __restrict__ rest, const int* __restrict__ assign,
                                                        uint16_t* __restrict__ ctx) {
  __shared__ uint16_t grp[RIFT_MAX_NV], tok[RIFT_MAX_NV];  // group and token index of unselected token a
  __shared__ uint32_t memb[RIFT_MAX_NV + MU];  // this part's members, sorted: group << 16 | token index
  __shared__ int cnt[RIFT_MAX_NV + 1], at[RIFT_MAX_NV + 1];  // group sizes; each group's first place
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.x, c0 = blockIdx.y * MCOLS + threadIdx.x * 8, lane = threadIdx.x & 31;
  if (j >= *n_kept) return;
  const int co = ctx_off[j], m = ctx_off[j + 1] - co;
  const int q_lo = m * (int)blockIdx.z / MP, q_hi = m * ((int)blockIdx.z + 1) / MP;
  if (q_lo == q_hi || co + m > max_ctx) return;
  const int R = n_v - (sel_off[j + 1] - sel_off[j]), step = R / m;
  const int* rj = rest + (size_t)j * n_v;
  for (int q = threadIdx.x; q < m; q += MT) cnt[q] = 0;
  __syncthreads();
  for (int a = threadIdx.x; a < R; a += MT) {
    int g = a / step;
    if (a % step != 0 || g >= m) {
      g = assign[(size_t)j * n_v + a];
      if (g < 0 || g >= m) g = 0;  // an unassigned token (no finite similarity) joins the first group
    }
    grp[a] = (uint16_t)g;
    tok[a] = (uint16_t)rj[a];
    atomicAdd(&cnt[g], 1);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int base = 0;
    for (int q0 = q_lo; q0 < q_hi; q0 += 32) {  // exclusive prefix sum of this part's group sizes
      const int v = q0 + lane < q_hi ? cnt[q0 + lane] : 0, inc = warp_incl_scan(v);
      if (q0 + lane < q_hi) at[q0 + lane] = base + inc - v;
      base += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) at[q_hi] = base;
  }
  __syncthreads();
  // placement in token order, a warp per group, 32 tokens at a time
  for (int q = q_lo + (int)(threadIdx.x >> 5); q < q_hi; q += MT / 32) {
    int base = at[q];
    for (int a0 = 0; a0 < R; a0 += 32) {
      const bool in = a0 + lane < R && grp[a0 + lane] == q;
      const unsigned b = __ballot_sync(0xffffffffu, in);
      if (in) memb[base + __popc(b & ((1u << lane) - 1u))] = ((uint32_t)q << 16) | tok[a0 + lane];
      base += __popc(b);
    }
  }
  if (threadIdx.x < MU) memb[at[q_hi] + threadIdx.x] = tok[0];  // a step past the end loads a row all the same
  __syncthreads();
  if (c0 >= d) return;
  const int i1 = at[q_hi];
  const XT* Xc = X + (size_t)kept[j] * n_v * d + c0;
  constexpr int GAP = 8 * MT;  // columns between a thread's two groups
  const bool two = c0 + GAP < d;
  float acc[2][8] = {};
  int cur = q_lo;
  auto flush = [&]() {
    const float inv = 1.f / (float)cnt[cur];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = pack_bf16x2(acc[v][2 * e] * inv, acc[v][2 * e + 1] * inv);
      if (v == 0 || two)
        *reinterpret_cast<uint4*>(ctx + (size_t)(co + cur) * d + c0 + v * GAP) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  };
  constexpr int NR = sizeof(XT) == 2 ? 1 : 2;  // 16-byte loads per group of a row
  for (int i = 0; i < i1; i += MU) {
    uint4 raw[MU][2][NR];
#pragma unroll
    for (int u = 0; u < MU; ++u) {
      const XT* row = Xc + (size_t)(memb[i + u] & 0xffffu) * d;
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (v == 0 || two) raw[u][v][r] = reinterpret_cast<const uint4*>(row + v * GAP)[r];
    }
#pragma unroll
    for (int u = 0; u < MU; ++u) {
      if (i + u >= i1) break;
      const int g = (int)(memb[i + u] >> 16);
      if (g != cur) {  // every group has its target: no group is empty
        flush();
        cur = g;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[0][e] = acc[1][e] = 0.f;
      }
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float x[8];
        if constexpr (NR == 1) {
          unpack_bf16x8(raw[u][v][0], x);
        } else {
          const uint4 a = raw[u][v][0], b = raw[u][v][NR - 1];
          const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(w[e]);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[v][e] += x[e];
      }
    }
  }
  flush();
}

}  // namespace mg

static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

MergeLayout merge_layout(int N, int n_v) {
  MergeLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
  L.rest_off = take((size_t)N * n_v * sizeof(int));
  L.assign_off = take((size_t)N * n_v * sizeof(int));
  L.tnorm_off = take((size_t)N * n_v * sizeof(double));
  L.tinv_off = take((size_t)N * n_v * sizeof(float));  // at most n_v - 1 targets per slot
  L.cand_off = take((size_t)N * n_v * sizeof(MergeCand));
  L.total = off;
  return L;
}

int launch_merge(const void* X, rift_dtype xdt, int N, int n_v, int d, const int* kept, const int* n_kept,
                 const int* budgets, const int* sel, const int* sel_off, uint16_t* ctx, int max_ctx, int* ctx_off,
                 int* ctx_target, char* ws, cudaStream_t st) {
  using namespace mg;
  const MergeLayout L = merge_layout(N, n_v);
  int* rest = reinterpret_cast<int*>(ws + L.rest_off);
  int* assign = reinterpret_cast<int*>(ws + L.assign_off);
  double* tnorm = reinterpret_cast<double*>(ws + L.tnorm_off);
  float* tinv = reinterpret_cast<float*>(ws + L.tinv_off);
  MergeCand* cand = reinterpret_cast<MergeCand*>(ws + L.cand_off);
  // every kernel but the fp32 tokens' assignment a programmatic dependent of the one before it
  bool ok = launch_ex(merge_plan_kernel, dim3(1), dim3(1024), 0, st, true, n_kept, budgets, sel_off, N, n_v, max_ctx,
                      ctx_off) == cudaSuccess;
  auto go = [&](auto* x) {
    using XT = std::remove_const_t<std::remove_pointer_t<decltype(x)>>;
    constexpr bool bf16 = sizeof(XT) == 2;
    ok = ok && launch_ex(merge_targets_kernel<XT>, dim3(N, TY), dim3(256), 0, st, true, x, n_v, d, kept, n_kept, sel,
                         sel_off, (const int*)ctx_off, max_ctx, rest, ctx_target, tnorm,
                         bf16 ? tinv : (float*)nullptr, bf16 ? ctx : (uint16_t*)nullptr) == cudaSuccess;
    if constexpr (bf16) {
      // the target rows go to ctx (overwritten by the means at the end), the top two of every token
      // come from the tensor cores, the choice between them where they are close from float-float sums
      if (max_ctx > 0)
        ok = ok && launch_merge_screen(x, N, n_v, d, kept, n_kept, sel_off, ctx_off, max_ctx, ctx, tinv, rest, cand, st) == 0;
      ok = ok && launch_ex(merge_decide_kernel, dim3((n_v + 63) / 64, N), dim3(DT), 0, st, true, x, n_v, d, kept,
                           n_kept, sel_off, (const int*)ctx_off, max_ctx, (const int*)rest, (const int*)ctx_target,
                           (const double*)tnorm, (const MergeCand*)cand, assign) == cudaSuccess;
    } else {
      const size_t ab_bytes = 2 * (size_t)KC * (TB + 4) * sizeof(float);
      const int blocks = (n_v + TB - 1) / TB;
      auto assign_by = [&](auto kern, std::atomic<unsigned long long>& smem_raised) {
        return raise_smem_limit(smem_raised, kern, (int)ab_bytes) == cudaSuccess &&
               launch_ex(kern, dim3(blocks, N), dim3(256), ab_bytes, st, false, x, n_v, d, kept, n_kept, sel_off,
                         (const int*)ctx_off, max_ctx, (const int*)rest, (const int*)ctx_target, (const double*)tnorm,
                         assign) == cudaSuccess;
      };
      static std::atomic<unsigned long long> raised4{0}, raised1{0};
      // (about a fifth of the tiles are kept: up to two CTAs with work an SM, or so)
      if (blocks * N <= 12 * sm_count()) ok = ok && assign_by(merge_assign_kernel<XT, 4>, raised4);
      else ok = ok && assign_by(merge_assign_kernel<XT, 1>, raised1);
    }
    ok = ok && launch_ex(merge_mean_kernel<XT>, dim3(N, (d + MCOLS - 1) / MCOLS, MP), dim3(MT), 0, st, true, x,
                         n_v, d, kept, n_kept, sel_off, (const int*)ctx_off, max_ctx, (const int*)rest, (const int*)assign, ctx) == cudaSuccess;
  };
  if (xdt == RIFT_BF16) go(static_cast<const uint16_t*>(X));
  else go(static_cast<const float*>(X));
  if (!ok) return -1;
  return xdt == RIFT_BF16 && max_ctx > 0 ? 5 : 4;
}

}  // namespace rift
