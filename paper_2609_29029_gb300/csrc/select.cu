// Stage 1 pruning and Stage 2 budgets and token selection on sm_103a.
//
//   select_kernel        (up to 512 tiles, one CTA per tile) both steps below: every CTA normalises all
//                        scores, takes the budgets and scans them for its own tile's place, and selects
//                        its tile's tokens
//   prune_budget_kernel  (more tiles; one CTA) per-scene min-max of the smoothed scores, u_i >= tau,
//                        the kept list (a block scan), the budget argmax of Eq. 2 and the
//                        exclusive scan of the budgets (the varlen offsets of the selection)
//   topb_kernel          (one CTA per kept tile) radix select of the b-th largest token
//                        score over order-preserving integer keys, ties to the lower index,
//                        and an ordered scan that writes the chosen indices ascending
//
// Every fp32 operation that decides an integer is a correctly rounded intrinsic written in
// the order the header documents, so the decisions are fixed by IEEE arithmetic.
#include "rift_internal.h"

namespace rift {

__device__ unsigned int g_err_select;

unsigned int read_clear_err_select() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_err_select, sizeof(v));
  cudaMemcpyToSymbol(g_err_select, &z, sizeof(z));
  return v;
}

// Budget: argmax_c U(c), U = ((p a+) + ((1 - p) a-)) - (lambda E), ties to the lower c.
__device__ __forceinline__ int budget_of(float p, const rift_policy& pol) {
  const float q = __fsub_rn(1.f, p);
  int best = 0;
  float bestU = 0.f;
  for (int c = 0; c < pol.n_c; ++c) {
    float acc = __fadd_rn(__fmul_rn(p, pol.alpha_pos[c]), __fmul_rn(q, pol.alpha_neg[c]));
    float Uc = __fsub_rn(acc, __fmul_rn(pol.lambda, pol.energy[c]));
    if (c == 0 || Uc > bestU) { best = c; bestU = Uc; }
  }
  return pol.C[best];
}

// With the merge on, c - floor(ctx_num c / ctx_den) of the c tokens are selected (the rest of the budget
// is contextual tokens); the full budget selects every token.
__device__ __forceinline__ int dominant_of(int b, int n_v, const rift_policy& pol) {
  return pol.ctx_num > 0 && b < n_v ? b - (pol.ctx_num * b) / pol.ctx_den : b;
}

constexpr int PB_THREADS = 1024;

// s_range (nullable): the min and max of the whole scene's smoothed scores, when these N tiles are
// one shard of it (the local scores are still checked for non-finite values).
__global__ void __launch_bounds__(PB_THREADS) prune_budget_kernel(
    const float* __restrict__ s, int N, int n_v, const float* __restrict__ p_ext, rift_policy pol,
    const float* __restrict__ s_range, float* __restrict__ u, int* __restrict__ kept, int* __restrict__ n_kept,
    int* __restrict__ budgets, int* __restrict__ sel_off) {
  pdl_trigger();
  pdl_wait();
  __shared__ float rmin[32], rmax[32];
  __shared__ int sh[33];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) s_bad = 0;
  float lo = INFINITY, hi = -INFINITY;
  bool bad = false;
  for (int i = tid; i < N; i += PB_THREADS) {
    float v = s[i];
    if (!isfinite(v)) bad = true;
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
  }
  lo = warp_min(lo);
  hi = warp_max(hi);
  if (lane == 0) { rmin[wid] = lo; rmax[wid] = hi; }
  __syncthreads();
  if (bad) s_bad = 1;
  if (tid < 32) {
    lo = warp_min(tid < PB_THREADS / 32 ? rmin[tid] : INFINITY);
    hi = warp_max(tid < PB_THREADS / 32 ? rmax[tid] : -INFINITY);
    if (tid == 0) { rmin[0] = lo; rmax[0] = hi; }
  }
  __syncthreads();
  lo = rmin[0];
  hi = rmax[0];
  if (s_range) {
    lo = s_range[0];
    hi = s_range[1];
    if (!isfinite(lo) || !isfinite(hi)) s_bad = 1;  // every thread read s_bad after the barrier above
  }
  __syncthreads();
  if (s_bad) {
    if (tid == 0) { atomicOr(&g_err_select, RIFT_EBIT_NONFINITE); *n_kept = 0; }
    for (int j = tid; j <= N; j += PB_THREADS) sel_off[j] = 0;
    return;
  }
  const float range = __fsub_rn(hi, lo);
  // u, keep flags, compaction in ascending tile order
  int base = 0;
  for (int c0 = 0; c0 < N; c0 += PB_THREADS) {
    const int i = c0 + tid;
    int keep = 0;
    if (i < N) {
      float ui = (hi == lo) ? 1.f : __fdiv_rn(__fsub_rn(s[i], lo), range);
      u[i] = ui;
      keep = ui >= pol.tau ? 1 : 0;
    }
    int total;
    int pos = block_excl_scan(keep, sh, &total);
    if (keep) kept[base + pos] = i;
    base += total;
  }
  const int n = base;
  if (tid == 0) *n_kept = n;
  __syncthreads();
  int off = 0;
  for (int c0 = 0; c0 < n; c0 += PB_THREADS) {
    const int j = c0 + tid;
    int b = 0;
    if (j < n) {
      const int i = kept[j];
      const float p = p_ext ? p_ext[i] : u[i];
      if (!isfinite(p)) atomicOr(&g_err_select, RIFT_EBIT_NONFINITE);
      b = budget_of(p, pol);
      budgets[j] = b;
      b = dominant_of(b, n_v, pol);
    }
    int total;
    int pos = block_excl_scan(b, sh, &total);
    if (j < n) sel_off[j] = off + pos;
    off += total;
  }
  for (int j = n + tid; j <= N; j += PB_THREADS) sel_off[j] = off;
}

// Order-preserving map of fp32 to uint32 (larger float -> larger key); -0 maps like +0.
__device__ __forceinline__ uint32_t float_key(float f) {
  uint32_t b = __float_as_uint(f);
  if (b == 0x80000000u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

constexpr int TB_THREADS = 256;
constexpr int TB_KPT = RIFT_MAX_NV / TB_THREADS;  // keys per thread (4)

// The token scores of a row in this thread's places: thread-major, so index order = (thread, e).
__device__ __forceinline__ void load_keys(const float* __restrict__ row, int n_v, float (&f)[TB_KPT]) {
#pragma unroll
  for (int e = 0; e < TB_KPT; ++e) {
    const int k = (int)threadIdx.x * TB_KPT + e;
    f[e] = k < n_v ? row[k] : 0.f;
  }
}

// The b highest of a row's n_v scores (load_keys), ties to the lower index: their indices, ascending, to out.
__device__ void top_b(const float (&f)[TB_KPT], int n_v, int b, int* __restrict__ out) {
  __shared__ int hist[256];
  __shared__ int sh[33];
  __shared__ uint32_t s_digit;
  __shared__ int s_rem;
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t key[TB_KPT];
  bool valid[TB_KPT];
  bool bad = false;
#pragma unroll
  for (int e = 0; e < TB_KPT; ++e) {
    valid[e] = tid * TB_KPT + e < n_v;
    if (valid[e] && !isfinite(f[e])) bad = true;
    key[e] = float_key(f[e]);
  }
  if (bad) atomicOr(&g_err_select, RIFT_EBIT_NONFINITE);

  // Radix select, 8 bits per pass from the top: the b-th largest key and how many of the
  // keys equal to it are taken (the lowest-index ones).
  uint32_t prefix = 0, mask = 0;
  int rem = b;
  for (int shift = 24; shift >= 0; shift -= 8) {
    hist[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < TB_KPT; ++e)
      if (valid[e] && (key[e] & mask) == prefix) atomicAdd(&hist[(key[e] >> shift) & 255u], 1);
    __syncthreads();
    if (tid < 32) {
      // lane l covers digits 255 - 8l down to 248 - 8l
      int c[8], loc = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) { c[q] = hist[255 - 8 * lane - q]; loc += c[q]; }
      const int inc = warp_incl_scan(loc);
      const int exc = inc - loc;
      if (exc < rem && rem <= inc) {
        int cum = exc;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (cum + c[q] >= rem) {
            s_digit = 255u - 8u * lane - q;
            s_rem = rem - cum;
            break;
          }
          cum += c[q];
        }
      }
    }
    __syncthreads();
    prefix |= s_digit << shift;
    mask |= 255u << shift;
    rem = s_rem;
    __syncthreads();
  }
  const uint32_t kth = prefix;
  const int need = rem;  // keys equal to kth that are selected

  int eq_loc = 0;
#pragma unroll
  for (int e = 0; e < TB_KPT; ++e) eq_loc += (valid[e] && key[e] == kth) ? 1 : 0;
  int tot;
  int eq_rank = block_excl_scan(eq_loc, sh, &tot);
  bool take[TB_KPT];
  int sel_loc = 0;
#pragma unroll
  for (int e = 0; e < TB_KPT; ++e) {
    bool eq = valid[e] && key[e] == kth;
    take[e] = valid[e] && (key[e] > kth || (eq && eq_rank < need));
    if (eq) ++eq_rank;
    sel_loc += take[e] ? 1 : 0;
  }
  int pos = block_excl_scan(sel_loc, sh, &tot);
#pragma unroll
  for (int e = 0; e < TB_KPT; ++e)
    if (take[e]) out[pos++] = tid * TB_KPT + e;
}

__global__ void __launch_bounds__(TB_THREADS) topb_kernel(const float* __restrict__ r, int n_v,
                                                          const int* __restrict__ kept,
                                                          const int* __restrict__ n_kept,
                                                          const int* __restrict__ sel_off,
                                                          int* __restrict__ sel) {
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.x;
  if (j >= *n_kept) return;
  float f[TB_KPT];
  load_keys(r + (size_t)kept[j] * n_v, n_v, f);
  // tokens to select: the budget less its contextual tokens
  top_b(f, n_v, sel_off[j + 1] - sel_off[j], sel + sel_off[j]);
}

// Both steps in one launch, CTA i = tile i: bound by latency, and a launch in the chain costs more than
// every CTA's own pass over the scores, TPT tiles a thread, while that is short: us alone, one launch against two,
// 64 tiles 8.3 : 12.3, 400 10.2 : 12.3, 512 12.3 : 14, 700 14-16 : 14, 1024 18.4 : 14-16; a scene's whole selection with
// small tokens, 512 tiles 160 : 161, 640 197 : 196, 1024 279 : 277.  The scene of 64 tiles went from 134 to 132 us (136
// with four tiles a thread: their budgets are a serial loop), 400 434 -> 430, four small tiles 47 -> 45.5.
// No early trigger: the next kernel's CTAs would take their SMs while these still wait for the smoothing, and those
// with work to do (the kept tiles' rows) then share few of them: a scene of 300 fp32 tiles at d = 4096 596 us with it,
// 562 without, 64 at 4096 215 : 200, 150 bf16 at 256 157 : 133.
// The results are those of prune_budget_kernel and topb_kernel, the same operations for every tile.
constexpr int SELECT_TPT = 2, SELECT_ONE = SELECT_TPT * TB_THREADS;  // tiles at most
// (unsigned, so that a sum past bit 31 would still be defined)
static_assert(SELECT_ONE <= 1024 && RIFT_MAX_NV <= 1024, "the scan packs the kept tiles above 21 bits of tokens");
template <int TPT>
__global__ void __launch_bounds__(TB_THREADS) select_kernel(
    const float* __restrict__ r, const float* __restrict__ s, int N, int n_v, const float* __restrict__ p_ext,
    rift_policy pol, const float* __restrict__ s_range, float* __restrict__ u, int* __restrict__ kept,
    int* __restrict__ n_kept, int* __restrict__ budgets, int* __restrict__ sel, int* __restrict__ sel_off) {
  pdl_wait();
  constexpr int NW = TB_THREADS / 32;
  __shared__ float rmin[NW], rmax[NW];
  __shared__ unsigned sh[33];
  __shared__ int own[4];  // this CTA's tile: kept, its place, its tokens' place, its tokens
  const int tid = threadIdx.x, tile = blockIdx.x, i0 = tid * TPT;
  float f[TB_KPT], v[TPT], p[TPT];
  load_keys(r + (size_t)tile * n_v, n_v, f);
  float lo = INFINITY, hi = -INFINITY;
  bool bad = false;
#pragma unroll
  for (int e = 0; e < TPT; ++e) {
    v[e] = i0 + e < N ? s[i0 + e] : 0.f;
    p[e] = p_ext && i0 + e < N ? p_ext[i0 + e] : 0.f;
  }
#pragma unroll
  for (int e = 0; e < TPT; ++e)
    if (i0 + e < N) {
      if (!isfinite(v[e])) bad = true;
      lo = fminf(lo, v[e]);
      hi = fmaxf(hi, v[e]);
    }
  lo = warp_min(lo);
  hi = warp_max(hi);
  if ((tid & 31) == 0) { rmin[tid >> 5] = lo; rmax[tid >> 5] = hi; }
  if (s_range && (!isfinite(s_range[0]) || !isfinite(s_range[1]))) bad = true;
  if (__syncthreads_or(bad)) {
    if (tile == 0) {
      if (tid == 0) { atomicOr(&g_err_select, RIFT_EBIT_NONFINITE); *n_kept = 0; }
      for (int j = tid; j <= N; j += TB_THREADS) sel_off[j] = 0;
    }
    return;
  }
  lo = rmin[0];
  hi = rmax[0];
#pragma unroll
  for (int w = 1; w < NW; ++w) {
    lo = fminf(lo, rmin[w]);
    hi = fmaxf(hi, rmax[w]);
  }
  if (s_range) { lo = s_range[0]; hi = s_range[1]; }
  const float range = __fsub_rn(hi, lo);
  int bud[TPT], tok[TPT];
  unsigned loc = 0;
  float ui[TPT];
#pragma unroll
  for (int e = 0; e < TPT; ++e) {
    ui[e] = hi == lo ? 1.f : __fdiv_rn(__fsub_rn(v[e], lo), range);
    bud[e] = tok[e] = 0;
    if (i0 + e < N && ui[e] >= pol.tau) {
      if (!p_ext) p[e] = ui[e];
      bud[e] = budget_of(p[e], pol);
      tok[e] = dominant_of(bud[e], n_v, pol);
      loc += (1u << 21) + (unsigned)tok[e];
    }
  }
  unsigned all;
  const unsigned at = block_excl_scan(loc, sh, &all);
  const int n = (int)(all >> 21), total = (int)(all & ((1u << 21) - 1u));
  int place = (int)(at >> 21), off = (int)(at & ((1u << 21) - 1));
#pragma unroll
  for (int e = 0; e < TPT; ++e) {
    if (i0 + e == tile) {
      u[tile] = ui[e];
      own[0] = bud[e] > 0;
      own[1] = place;
      own[2] = off;
      own[3] = tok[e];
      if (bud[e] > 0) {
        if (!isfinite(p[e])) atomicOr(&g_err_select, RIFT_EBIT_NONFINITE);
        kept[place] = tile;
        budgets[place] = bud[e];
        sel_off[place] = off;
      }
    }
    place += bud[e] > 0 ? 1 : 0;
    off += tok[e];
  }
  if (tile == 0) {
    if (tid == 0) *n_kept = n;
    for (int j = n + tid; j <= N; j += TB_THREADS) sel_off[j] = total;
  }
  __syncthreads();
  if (own[0]) top_b(f, n_v, own[3], sel + own[2]);
}

int launch_select(const float* token_scores, const float* tile_s, int N, int n_v, const float* p,
                  const rift_policy& pol, float* u, int* kept, int* n_kept, int* budgets, int* sel,
                  int* sel_off, cudaStream_t st, const float* s_range) {
  // (scores normalised in place are left to the one CTA that reads them before it writes)
  if (N <= SELECT_ONE && tile_s != u && p != u) {
    auto go = [&](auto kern) {
      launch_ex(kern, dim3(N), dim3(TB_THREADS), 0, st, true, token_scores, tile_s, N, n_v, p, pol, s_range, u, kept,
                n_kept, budgets, sel, sel_off);
    };
    if (N <= TB_THREADS) go(select_kernel<1>);
    else go(select_kernel<SELECT_TPT>);
    return 1;
  }
  launch_ex(prune_budget_kernel, dim3(1), dim3(PB_THREADS), 0, st, true, tile_s, N, n_v, p, pol, s_range, u, kept,
            n_kept, budgets, sel_off);
  launch_ex(topb_kernel, dim3(N), dim3(TB_THREADS), 0, st, true, token_scores, n_v, (const int*)kept,
            (const int*)n_kept, (const int*)sel_off, sel);
  return 2;
}

}  // namespace rift
