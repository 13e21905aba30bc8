// The per-tile features of the p_i predictor (Section 2.3, Stage 2: the tile embedding, its
// Stage-1 relevance, the vision-token scores and the relevance of its four quadrants) for a list of
// tiles, on sm_103a.
//
//   features_fold_kernel   w = t - (1/M) sum_j B_j (Eq. 1's background mean folded into one vector)
//   quad_sum_kernel        per (listed tile, quadrant, 2048 columns): the sum of the quadrant's
//                          g/2 x g/2 tokens (fp32, 16-byte loads, token rows in grid order)
//   features_final_kernel  per listed tile: each quadrant's Eq. 1 score l2norm(sum) . w, the tile
//                          embedding l2norm(sum of the four), and max / mean / population std of
//                          the tile's token scores (two passes)
#include "rift_internal.h"

namespace rift {

namespace ft {

constexpr int QT = 256;        // threads of the quadrant sum
constexpr int QCOLS = QT * 8;  // columns per CTA

__global__ void features_fold_kernel(const float* __restrict__ t, const float* __restrict__ B, int M, int d,
                                     float* __restrict__ w) {
  pdl_trigger();
  pdl_wait();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= d) return;
  float s = 0.f;
  for (int j = 0; j < M; ++j) s += B[(size_t)j * d + c];
  w[c] = M > 0 ? t[c] - s / (float)M : t[c];
}

template <typename XT>
__device__ __forceinline__ void load8(const XT* p, float (&v)[8]) {
  if constexpr (sizeof(XT) == 2) {
    unpack_bf16x8(*reinterpret_cast<const uint4*>(p), v);
  } else {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
}

// Grid (list slot, quadrant 0..3, column block).  Qsum[slot][q][c] = sum over the quadrant's tokens.
template <typename XT>
__global__ void __launch_bounds__(QT) quad_sum_kernel(const XT* __restrict__ X, int N, int n_v, int d, int g,
                                                      const int* __restrict__ tiles, const int* __restrict__ n_tiles,
                                                      float* __restrict__ Qsum) {
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.x;
  const int n = tiles ? *n_tiles : N;
  if (j >= n) return;
  const int tile = tiles ? tiles[j] : j;
  if (tile < 0 || tile >= N) return;
  const int q = blockIdx.y, h = g / 2;
  const int r0 = (q >> 1) * h, c0 = (q & 1) * h;
  const int col = blockIdx.z * QCOLS + threadIdx.x * 8;
  if (col >= d) return;
  const XT* Xt = X + (size_t)tile * n_v * d;
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int r = r0; r < r0 + h; ++r) {
#pragma unroll 4
    for (int c = c0; c < c0 + h; ++c) {
      float x[8];
      load8(Xt + (size_t)(r * g + c) * d + col, x);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] += x[e];
    }
  }
  float* out = Qsum + ((size_t)j * 4 + q) * d + col;
  reinterpret_cast<float4*>(out)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  reinterpret_cast<float4*>(out)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
}

// One CTA per listed tile.  Latency-bound (0.1 MB of sums per tile): all of a thread's columns of the
// four quadrants are loaded at once, and the ten sums and the maximum share one reduction (one
// quadrant after another with a reduction per sum took 39 us at 400 tiles, this 8).
__global__ void __launch_bounds__(256) features_final_kernel(const float* __restrict__ Qsum, const float* __restrict__ w,
                                                             const float* __restrict__ token_scores, int N, int n_v,
                                                             int d, const int* __restrict__ tiles,
                                                             const int* __restrict__ n_tiles,
                                                             float* __restrict__ features, float* __restrict__ V) {
  constexpr int NS = 11;  // per quadrant: sum of squares and dot with w; the tile's sum of squares; scores: max, sum
  __shared__ float red[8][NS];
  __shared__ float red2[32];
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.x;
  const int n = tiles ? *n_tiles : N;
  if (j >= n) return;
  const int tile = tiles ? tiles[j] : j;
  if (tile < 0 || tile >= N) return;
  const float4* Q = reinterpret_cast<const float4*>(Qsum + (size_t)j * 4 * d);
  const float4* w4 = reinterpret_cast<const float4*>(w);
  float* f = features + (size_t)j * RIFT_N_FEATURES;
  const int nv = d / 4, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float* r = token_scores + (size_t)tile * n_v;
  float s[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) s[k] = 0.f;
  s[9] = -INFINITY;
  float rv[RIFT_MAX_NV / 256];
#pragma unroll
  for (int k = 0; k < RIFT_MAX_NV / 256; ++k) {
    const int t = threadIdx.x + k * 256;
    rv[k] = t < n_v ? r[t] : 0.f;
    if (t < n_v) s[9] = fmaxf(s[9], rv[k]);
    s[10] += rv[k];
  }
  auto tile_sum = [](const float4& a, const float4& b, const float4& c, const float4& e) {
    return make_float4((a.x + b.x) + (c.x + e.x), (a.y + b.y) + (c.y + e.y), (a.z + b.z) + (c.z + e.z),
                       (a.w + b.w) + (c.w + e.w));
  };
#pragma unroll 4
  for (int c = threadIdx.x; c < nv; c += 256) {
    const float4 wc = w4[c];
    float4 q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = Q[(size_t)k * nv + c];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[2 * k] += (q[k].x * q[k].x + q[k].y * q[k].y) + (q[k].z * q[k].z + q[k].w * q[k].w);
      s[2 * k + 1] += (q[k].x * wc.x + q[k].y * wc.y) + (q[k].z * wc.z + q[k].w * wc.w);
    }
    const float4 t = tile_sum(q[0], q[1], q[2], q[3]);
    s[8] += (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) s[k] = k == 9 ? warp_max(s[k]) : warp_sum(s[k]);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) red[wid][k] = s[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    float v = red[0][k];
#pragma unroll
    for (int x = 1; x < 8; ++x) v = k == 9 ? fmaxf(v, red[x][k]) : v + red[x][k];
    s[k] = v;
  }
  if (threadIdx.x < 4) {
    const float ss = threadIdx.x == 0 ? s[0] : threadIdx.x == 1 ? s[2] : threadIdx.x == 2 ? s[4] : s[6];
    const float dt = threadIdx.x == 0 ? s[1] : threadIdx.x == 1 ? s[3] : threadIdx.x == 2 ? s[5] : s[7];
    f[threadIdx.x] = ss > 0.f ? dt / sqrtf(ss) : 0.f;
  }
  if (V) {
    const float inv = s[8] > 0.f ? 1.f / sqrtf(s[8]) : 0.f;
#pragma unroll 4
    for (int c = threadIdx.x; c < nv; c += 256) {
      const float4 t = tile_sum(Q[c], Q[(size_t)nv + c], Q[(size_t)2 * nv + c], Q[(size_t)3 * nv + c]);
      reinterpret_cast<float4*>(V + (size_t)j * d)[c] = make_float4(t.x * inv, t.y * inv, t.z * inv, t.w * inv);
    }
  }
  const float mean = s[10] / (float)n_v;
  float var = 0.f;
#pragma unroll
  for (int k = 0; k < RIFT_MAX_NV / 256; ++k)
    if ((int)threadIdx.x + k * 256 < n_v) var += (rv[k] - mean) * (rv[k] - mean);
  var = block_sum(var, red2) / (float)n_v;
  if (threadIdx.x == 0) {
    f[4] = s[9];
    f[5] = mean;
    f[6] = sqrtf(var);
  }
}

}  // namespace ft

FeaturesLayout features_layout(int N, int d) {
  FeaturesLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
  L.w_off = take((size_t)d * sizeof(float));
  L.qsum_off = take((size_t)N * 4 * d * sizeof(float));
  L.total = off;
  return L;
}

int launch_features(const void* X, rift_dtype xdt, int N, int n_v, int d, int g, const float* t, const float* B, int M,
                    const float* token_scores, const int* tiles, const int* n_tiles, float* features, float* V,
                    char* ws, cudaStream_t st) {
  using namespace ft;
  const FeaturesLayout L = features_layout(N, d);
  float* w = reinterpret_cast<float*>(ws + L.w_off);
  float* Qsum = reinterpret_cast<float*>(ws + L.qsum_off);
  launch_ex(features_fold_kernel, dim3((d + 255) / 256), dim3(256), 0, st, true, t, B, M, d, w);
  const dim3 gq(N, 4, (d + QCOLS - 1) / QCOLS);
  if (xdt == RIFT_BF16)
    launch_ex(quad_sum_kernel<uint16_t>, gq, dim3(QT), 0, st, true, static_cast<const uint16_t*>(X), N, n_v, d, g, tiles,
              n_tiles, Qsum);
  else
    launch_ex(quad_sum_kernel<float>, gq, dim3(QT), 0, st, true, static_cast<const float*>(X), N, n_v, d, g, tiles,
              n_tiles, Qsum);
  launch_ex(features_final_kernel, dim3(N), dim3(256), 0, st, true, (const float*)Qsum, (const float*)w, token_scores, N,
            n_v, d, tiles, n_tiles, features, V);
  return 3;
}

}  // namespace rift
