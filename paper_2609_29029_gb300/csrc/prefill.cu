// Decoder prefill over the packed batch (Section 2.1): the per-layer kernel sequence, the
// fused RMSNorm kernels and RoPE.
//
// Per layer, with the residual stream h kept in fp32 and every GEMM operand in fp16:
//   xn  = RMSNorm(h) g_attn                      rmsnorm_kernel            (fp16 out)
//   qkv = xn W_qkv^T, RoPE on q and k            GEMM, RoPE epilogue on the fp32 accumulators
//   a   = causal varlen attention(q, k, v)       attention
//   h  += a W_o^T                                GEMM, fp32 residual epilogue
//   xn  = RMSNorm(h) g_ffn
//   act = SiLU(xn W_g^T) * (xn W_u^T)            GEMM, SwiGLU epilogue (interleaved gate/up)
//   h  += act W_down^T                           GEMM, fp32 residual epilogue
// and finally hidden = RMSNorm(h) g_final in bf16.  Optional outputs: each layer's keys (after
// RoPE) and values (the KV cache, stored by the QKV product's epilogue), and the logits of every
// sequence's last token, RMSNorm(h_last) g_final times the output matrix.
//
// The decode step runs the same layer sequence for one new token per sequence, at position L_i,
// with the attention replaced by decode_attn_kernel over the sequence's cached keys and values
// plus the token's own.
// fp16 rather than bf16 operands: after 32 layers the bf16 rounding of the GEMM inputs alone
// moves the final hidden states by about 3% of their largest magnitude; fp16 (3 more mantissa
// bits, same tensor-core rate, LLaVA-1.5-7B's checkpoint dtype) keeps the whole path near 0.5%.
#include <atomic>
#include <cmath>
#include <type_traits>

#include "rift_internal.h"

namespace rift {

__device__ unsigned int g_err_prefill;

unsigned int read_clear_err_prefill() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_err_prefill, sizeof(v));
  cudaMemcpyToSymbol(g_err_prefill, &z, sizeof(z));
  return v;
}

constexpr int NORM_THREADS = 256;

// One row of the RMSNorm below: row `row` of out (and h32) from row `in_row` of in (negative: zeros).
template <bool IN_BF16, bool OUT_F16, int VPT>
__device__ __forceinline__ void rmsnorm_row(const void* __restrict__ in, float* __restrict__ h32,
                                            const uint16_t* __restrict__ gain, uint16_t* __restrict__ out, int d,
                                            float eps, size_t row, long long in_row, float* red) {
  const int nv = d / 4;
  float4 v[VPT];
  float ss = 0.f;
#pragma unroll
  for (int q = 0; q < VPT; ++q) {
    const int c = threadIdx.x + q * NORM_THREADS;
    if (c < nv) {
      if constexpr (IN_BF16) {
        const uint2 raw = in_row >= 0 ? reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(in) + in_row * d)[c]
                                      : make_uint2(0u, 0u);
        v[q] = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                           __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
        reinterpret_cast<float4*>(h32 + row * d)[c] = v[q];
      } else {
        v[q] = reinterpret_cast<const float4*>(static_cast<const float*>(in) + in_row * d)[c];
      }
      ss += v[q].x * v[q].x + v[q].y * v[q].y + v[q].z * v[q].z + v[q].w * v[q].w;
    }
  }
  const float inv = rsqrtf(block_sum(ss, red) / (float)d + eps);
#pragma unroll
  for (int q = 0; q < VPT; ++q) {
    const int c = threadIdx.x + q * NORM_THREADS;
    if (c < nv) {
      uint2 gr = reinterpret_cast<const uint2*>(gain)[c];
      const float g0 = __uint_as_float(gr.x << 16), g1 = __uint_as_float(gr.x & 0xffff0000u);
      const float g2 = __uint_as_float(gr.y << 16), g3 = __uint_as_float(gr.y & 0xffff0000u);
      uint2 o;
      if constexpr (OUT_F16) {
        o.x = pack_half2(v[q].x * inv * g0, v[q].y * inv * g1);
        o.y = pack_half2(v[q].z * inv * g2, v[q].w * inv * g3);
      } else {
        o.x = pack_bf16x2(v[q].x * inv * g0, v[q].y * inv * g1);
        o.y = pack_bf16x2(v[q].z * inv * g2, v[q].w * inv * g3);
      }
      reinterpret_cast<uint2*>(out + row * d)[c] = o;
    }
  }
}

// y = h / sqrt(mean(h^2) + eps) * g, one row per CTA at a time: rows blockIdx.x, + gridDim.x,
// ... below the row count (rows_dev: a device count clamped to max_rows, or max_rows itself).
// IN_BF16: h is the bf16 packed input, which is also widened into the fp32 residual stream h32.
// OUT_F16: y in fp16 (the GEMM operand); otherwise bf16 (the final hidden states).  VPT: float4
// per thread, the fewest that cover d (4 at d = 4096, 8 at the widest d = 8192), so the row held
// in registers is no larger than the row: fewer registers, more CTAs per SM and more bytes in
// flight.
template <bool IN_BF16, bool OUT_F16, int VPT>
__global__ void __launch_bounds__(NORM_THREADS, VPT <= 4 ? 8 : 4) rmsnorm_kernel(const void* __restrict__ in,
                                                               float* __restrict__ h32,
                                                               const uint16_t* __restrict__ gain,
                                                               uint16_t* __restrict__ out, int d,
                                                               float eps, const int* __restrict__ rows_dev,
                                                               int max_rows) {
  __shared__ float red[32];
  pdl_trigger();
  pdl_wait();
  const int n_rows = rows_dev ? max(0, min(max_rows, *rows_dev)) : max_rows;
  for (size_t row = blockIdx.x; row < (size_t)n_rows; row += gridDim.x)
    rmsnorm_row<IN_BF16, OUT_F16, VPT>(in, h32, gain, out, d, eps, row, (long long)row, red);
}

static RopeFreq rope_freq(const rift_model& m) {
  RopeFreq f;
  const int half = m.head_dim / 2;
  for (int j = 0; j < 64; ++j) f.inv[j] = j < half ? std::pow((double)m.rope_theta, -2.0 * j / m.head_dim) : 0.0;
  return f;
}

// out[i] = h32[cu[i + 1] - 1]: the residual stream of each sequence's last row (zeros for an
// empty sequence, or one that ends past the row_cap rows the buffers hold), for the sequences
// below the device count n_seq_dev (all gridDim.x of them without one).
__global__ void last_rows_kernel(const float* __restrict__ h32, const int* __restrict__ cu,
                                 const int* __restrict__ n_seq_dev, int row_cap, int d, float* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x;
  if (n_seq_dev && i >= *n_seq_dev) return;
  const bool empty = cu[i + 1] <= cu[i] || cu[i + 1] > row_cap;
  const float4* src = reinterpret_cast<const float4*>(h32 + (size_t)(empty ? 0 : cu[i + 1] - 1) * d);
  float4* dst = reinterpret_cast<float4*>(out + (size_t)i * d);
  for (int c = threadIdx.x; c < d / 4; c += blockDim.x) dst[c] = empty ? make_float4(0.f, 0.f, 0.f, 0.f) : src[c];
}

PrefillLayout prefill_layout(const rift_model& m, int max_T, int max_seqs, int max_len) {
  PrefillLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
  const size_t T = (size_t)max_T;
  L.h32_off = take(T * m.d * 4);
  L.xn_off = take(T * m.d * 2);
  L.qkv_off = take(T * 3 * m.d * 2);
  L.attn_off = take(T * m.d * 2);
  L.act_off = take(T * m.ffn * 2);
  L.rope_off = take((size_t)max_len * (m.head_dim / 2) * sizeof(float2));
  L.max_qblocks = attention_max_qblocks(max_T, max_seqs);
  L.sched_off = take((size_t)(L.max_qblocks + 1) * sizeof(int4));  // + the entry count
  L.last32_off = take((size_t)max_seqs * m.d * 4);
  L.last16_off = take((size_t)max_seqs * m.d * 2);
  L.total = off;
  return L;
}

int launch_gemm(const void* A, const void* B, int M, int N, int K, int epi, void* C, cudaStream_t st,
                const EpiParams& ep, bool pdl) {
  prof_begin(RIFT_PROF_GEMM, st);
  const int r = launch_gemm_tc(A, B, M, N, K, epi, C, ep, st, pdl);
  prof_end(RIFT_PROF_GEMM, st, 1);
  return r;
}

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

// CTAs of rmsnorm_kernel<IN_BF16, OUT_F16, VPT> resident per SM at once (asked once per
// instantiation; 1 if the query fails).
template <bool IN_BF16, bool OUT_F16, int VPT>
static int norm_resident_ctas() {
  static std::atomic<int> n{0};
  int v = n.load(std::memory_order_relaxed);
  if (v == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, rmsnorm_kernel<IN_BF16, OUT_F16, VPT>, NORM_THREADS, 0) !=
            cudaSuccess ||
        v < 1) {
      cudaGetLastError();
      v = 1;
    }
    n.store(v, std::memory_order_relaxed);
  }
  return v;
}

// kind 0: packed bf16 input -> h32 + fp16 xn; 1: h32 -> fp16 xn; 2: h32 -> bf16 final output.
// Rows: min(*rows_dev, T) with a device count, else T.  The grid is four times the CTAs that fit
// on the GPU at once (8 per SM at d <= 4096), each looping over rows: a CTA that finishes early
// frees its slot for another, so the last rows spread over the SMs as with one CTA per row.
static void norm_launch(int kind, int T, const void* in, float* h32, const void* gain, uint16_t* out, int d,
                        float eps, cudaStream_t st, const int* rows_dev = nullptr, bool pdl = false) {
  prof_begin(RIFT_PROF_NORM, st);
  const uint16_t* g = static_cast<const uint16_t*>(gain);
  const int per_thread = (d / 4 + NORM_THREADS - 1) / NORM_THREADS;  // d <= 8192: at most 8
  auto go = [&](auto vpt) {
    constexpr int V = decltype(vpt)::value;
    auto grid = [&](int per_sm) { return T < 4 * per_sm * sm_count() ? T : 4 * per_sm * sm_count(); };
    if (kind == 0)
      launch_ex(rmsnorm_kernel<true, true, V>, dim3(grid(norm_resident_ctas<true, true, V>())), dim3(NORM_THREADS), 0,
                st, pdl, in, h32, g, out, d, eps, rows_dev, T);
    else if (kind == 1)
      launch_ex(rmsnorm_kernel<false, true, V>, dim3(grid(norm_resident_ctas<false, true, V>())), dim3(NORM_THREADS), 0,
                st, pdl, in, (float*)nullptr, g, out, d, eps, rows_dev, T);
    else
      launch_ex(rmsnorm_kernel<false, false, V>, dim3(grid(norm_resident_ctas<false, false, V>())), dim3(NORM_THREADS),
                0, st, pdl, in, (float*)nullptr, g, out, d, eps, rows_dev, T);
  };
  if (per_thread <= 1) go(std::integral_constant<int, 1>{});
  else if (per_thread <= 2) go(std::integral_constant<int, 2>{});
  else if (per_thread <= 4) go(std::integral_constant<int, 4>{});
  else go(std::integral_constant<int, 8>{});
  prof_end(RIFT_PROF_NORM, st, 1);
}

int launch_prefill(const rift_model& m, void* hidden, int T, const int* T_dev, const int* cu_seqlens, int n_seq,
                   const int* n_seq_dev, int max_len, const int* positions, void* kv_out, float* last_logits,
                   char* ws, cudaStream_t st, const void* prefix_kv, int S_pre) {
  if (T == 0 || n_seq == 0) return 0;
  const PrefillLayout L = prefill_layout(m, T, n_seq, max_len);
  float* h32 = reinterpret_cast<float*>(ws + L.h32_off);
  uint16_t* xn = reinterpret_cast<uint16_t*>(ws + L.xn_off);
  uint16_t* qkv = reinterpret_cast<uint16_t*>(ws + L.qkv_off);
  uint16_t* att = reinterpret_cast<uint16_t*>(ws + L.attn_off);
  uint16_t* act = reinterpret_cast<uint16_t*>(ws + L.act_off);
  float2* rope = reinterpret_cast<float2*>(ws + L.rope_off);
  int4* sched = reinterpret_cast<int4*>(ws + L.sched_off);
  const int d = m.d, half = m.head_dim / 2;

  // With few rows the kernels after the first are launched as programmatic dependents of the kernel before
  // them: launch latencies are a good part of the time (two layers over one 131-row tile 373 -> 316 us
  // with the setup in one launch).  With many, the early launches cost more than they hide.  Time with them
  // over time without, two 7B layers: 1,938 rows 0.970, 3,660 0.992, 5,395 0.996, 7,333 0.998, 8,374 0.994,
  // 9,618 0.998, 12,728 1.018, 19,020 1.009, 27,047 1.015 (at d = 1024, where a kernel is shorter, 0.83 at 347
  // rows to 0.98 at 27,047).
  const bool pdl = T <= 8192;
  prof_begin(RIFT_PROF_ROPE, st);
  PrefillSetup ps = {rope, max_len, half, rope_freq(m), qkv, 3 * d, T_dev};
  launch_attention_schedule(cu_seqlens, n_seq, n_seq_dev, T, sched, L.max_qblocks, st, &ps);
  prof_end(RIFT_PROF_ROPE, st, 1);
  // every product covers the rows the device count holds (T rows of capacity)
  EpiParams rows_ep;
  rows_ep.m_dev = T_dev;
  EpiParams rope_ep = rows_ep;
  rope_ep.positions = positions;
  rope_ep.rope = rope;
  rope_ep.rope_cols = 2 * d;
  rope_ep.head_dim = m.head_dim;
  rope_ep.max_len = max_len;
  rope_ep.pos_offset = S_pre;
  for (int l = 0; l < m.n_layers; ++l) {
    if (l == 0)
      norm_launch(0, T, hidden, h32, m.g_attn[0], xn, d, m.eps, st, T_dev, pdl);
    else
      norm_launch(1, T, h32, nullptr, m.g_attn[l], xn, d, m.eps, st, T_dev, pdl);
    if (kv_out) {
      rope_ep.k_out = static_cast<uint16_t*>(kv_out) + (size_t)l * 2 * T * d;
      rope_ep.v_out = rope_ep.k_out + (size_t)T * d;
    }
    if (launch_gemm(xn, m.w_qkv[l], T, 3 * d, d, EPI_QKV_ROPE, qkv, st, rope_ep, pdl)) return 1;
    prof_begin(RIFT_PROF_ATTN, st);
    const uint16_t* pk = prefix_kv ? static_cast<const uint16_t*>(prefix_kv) + (size_t)l * 2 * S_pre * d : nullptr;
    if (launch_attention(qkv, T, cu_seqlens, n_seq, m.n_heads, m.head_dim, sched, L.max_qblocks, att, st, pk,
                         pk ? pk + (size_t)S_pre * d : nullptr, prefix_kv ? S_pre : 0, pdl))
      return 1;
    prof_end(RIFT_PROF_ATTN, st, 1);
    if (launch_gemm(att, m.w_o[l], T, d, d, EPI_RESID_F32, h32, st, rows_ep, pdl)) return 1;
    norm_launch(1, T, h32, nullptr, m.g_ffn[l], xn, d, m.eps, st, T_dev, pdl);
    if (launch_gemm(xn, m.w_gate_up[l], T, 2 * m.ffn, d, EPI_SWIGLU, act, st, rows_ep, pdl)) return 1;
    if (launch_gemm(act, m.w_down[l], T, d, m.ffn, EPI_RESID_F32, h32, st, rows_ep, pdl)) return 1;
  }
  norm_launch(2, T, h32, nullptr, m.g_final, static_cast<uint16_t*>(hidden), d, m.eps, st, T_dev, pdl);
  if (last_logits) {
    float* last32 = reinterpret_cast<float*>(ws + L.last32_off);
    uint16_t* last16 = reinterpret_cast<uint16_t*>(ws + L.last16_off);
    if (launch_ex(last_rows_kernel, dim3(n_seq), dim3(256), 0, st, pdl, (const float*)h32, cu_seqlens, n_seq_dev, T, d,
                  last32) != cudaSuccess)
      return 1;
    norm_launch(1, n_seq, last32, nullptr, m.g_final, last16, d, m.eps, st, n_seq_dev, pdl);
    EpiParams seq_ep;
    seq_ep.m_dev = n_seq_dev;
    if (launch_gemm(last16, m.lm_head, n_seq, m.vocab, d, EPI_STORE_F32, last_logits, st, seq_ep, pdl)) return 1;
  }
  return 0;
}

// ------------------------------------------------------------------------------------------
// Shared-prefix prefill: the system prompt once, then every sequence's suffix over its cache
// ------------------------------------------------------------------------------------------

// prefix rows = embed[sys_ids] (bf16), cu = {0, S}, positions 0 .. S-1; a bad id sets
// RIFT_EBIT_BADID and gives a zero row.
__global__ void prefix_rows_kernel(const int* __restrict__ sys_ids, int S, const uint16_t* __restrict__ embed,
                                   int vocab, int d, uint16_t* __restrict__ rows, int* __restrict__ cu,
                                   int* __restrict__ pos) {
  const int r = blockIdx.x;
  const int id = sys_ids[r];
  const bool ok = id >= 0 && id < vocab;
  if (threadIdx.x == 0) {
    pos[r] = r;
    if (!ok) atomicOr(&g_err_prefill, RIFT_EBIT_BADID);
    if (r == 0) {
      cu[0] = 0;
      cu[1] = S;
    }
  }
  const uint4* src = reinterpret_cast<const uint4*>(embed + (size_t)(ok ? id : 0) * d);
  uint4* dst = reinterpret_cast<uint4*>(rows + (size_t)r * d);
  for (int c = threadIdx.x; c < d / 8; c += blockDim.x) dst[c] = ok ? src[c] : make_uint4(0, 0, 0, 0);
}

SharedPrefixLayout shared_prefix_layout(const rift_model& m, int max_T, int max_seqs, int max_len, int S) {
  SharedPrefixLayout L{};
  const PrefillLayout P = prefill_layout(m, max_T > S ? max_T : S, max_seqs > 1 ? max_seqs : 1, max_len);
  size_t off = (P.total + 255) & ~size_t(255);
  L.prefill_bytes = P.total;
  L.cu_off = off;
  off += 256;
  L.pos_off = off;
  off += ((size_t)S * sizeof(int) + 255) & ~size_t(255);
  L.total = off;
  return L;
}

int launch_prefill_shared_prefix(const rift_model& m, const int* sys_ids, int S, const void* embed, int vocab,
                                 void* prefix_hidden, void* prefix_kv, void* hidden, int T, const int* T_dev,
                                 const int* cu_seqlens, int n_seq, const int* n_seq_dev, int max_len,
                                 const int* positions, float* last_logits, char* ws, cudaStream_t st) {
  const SharedPrefixLayout L = shared_prefix_layout(m, T, n_seq, max_len, S);
  int* cu_pre = reinterpret_cast<int*>(ws + L.cu_off);
  int* pos_pre = reinterpret_cast<int*>(ws + L.pos_off);
  prefix_rows_kernel<<<S, 128, 0, st>>>(sys_ids, S, static_cast<const uint16_t*>(embed), vocab, m.d,
                                        static_cast<uint16_t*>(prefix_hidden), cu_pre, pos_pre);
  // the prefix as one sequence, keeping its cache; then the suffixes over it (the two share the
  // prefill workspace: they run in order on the stream)
  if (launch_prefill(m, prefix_hidden, S, nullptr, cu_pre, 1, nullptr, max_len, pos_pre, prefix_kv, nullptr, ws, st))
    return 1;
  if (T > 0 && launch_prefill(m, hidden, T, T_dev, cu_seqlens, n_seq, n_seq_dev, max_len, positions, nullptr,
                              last_logits, ws, st, prefix_kv, S))
    return 1;
  return 0;
}

// ------------------------------------------------------------------------------------------
// Decode step: one new token per sequence
// ------------------------------------------------------------------------------------------

DecodeLayout decode_layout(const rift_model& m, int n_seq, int max_len) {
  DecodeLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
  const size_t n = (size_t)(n_seq > 0 ? n_seq : 1);
  L.h32_off = take(n * m.d * 4);
  L.xn_off = take(n * m.d * 2);
  L.qkv_off = take(n * 3 * m.d * 2);
  L.attn_off = take(n * m.d * 2);
  L.act_off = take(n * m.ffn * 2);
  L.rope_off = take(n * (m.head_dim / 2) * sizeof(float2));  // a row per sequence
  L.pos_off = take(n * sizeof(int));
  L.total = off;
  return L;
}

// The start of a decode step, one CTA per sequence i: h32[i] = embed[ids[i]], xn[i] = RMSNorm(h32[i]) gain
// (fp16), row i of the RoPE table = (cos, sin) at the new token's position L_i = cu[i + 1] - cu[i], and
// pos[i] = i, its row of the table (-1 if L_i is not below max_len: the QKV epilogue reports it).  An
// id outside [0, vocab) sets RIFT_EBIT_BADID and gives a zero row.
template <int VPT>
__global__ void __launch_bounds__(NORM_THREADS) decode_start_kernel(const int* __restrict__ ids,
                                                                   const int* __restrict__ cu,
                                                                   const uint16_t* __restrict__ embed, int vocab, int d,
                                                                   int max_len, int half,
                                                                   const __grid_constant__ RopeFreq freq,
                                                                   const uint16_t* __restrict__ gain, float eps,
                                                                   float* __restrict__ h32, uint16_t* __restrict__ xn,
                                                                   float2* __restrict__ rope, int* __restrict__ pos) {
  __shared__ float red[32];
  pdl_trigger();
  const int i = blockIdx.x;
  const int id = ids[i];
  const bool ok = id >= 0 && id < vocab;
  const int L = cu[i + 1] - cu[i];
  if (threadIdx.x == 0) {
    pos[i] = L >= 0 && L < max_len ? i : -1;
    if (!ok) atomicOr(&g_err_prefill, RIFT_EBIT_BADID);
  }
  if ((int)threadIdx.x < half)
    rope[(size_t)i * half + threadIdx.x] = rope_cos_sin((double)max(L, 0) * freq.inv[threadIdx.x]);
  rmsnorm_row<true, true, VPT>(embed, h32, gain, xn, d, eps, (size_t)i, ok ? (long long)id : -1, red);
}

int launch_decode(const rift_model& m, const void* kv_cache, int T, const int* cu_seqlens, int n_seq, int max_len,
                  const int* token_ids, const void* embed, int vocab_embed, void* hidden_out, void* kv_new,
                  float* logits, char* ws, cudaStream_t st) {
  if (n_seq == 0) return 0;
  const DecodeLayout L = decode_layout(m, n_seq, max_len);
  float* h32 = reinterpret_cast<float*>(ws + L.h32_off);
  uint16_t* xn = reinterpret_cast<uint16_t*>(ws + L.xn_off);
  uint16_t* qkv = reinterpret_cast<uint16_t*>(ws + L.qkv_off);
  uint16_t* att = reinterpret_cast<uint16_t*>(ws + L.attn_off);
  uint16_t* act = reinterpret_cast<uint16_t*>(ws + L.act_off);
  float2* rope = reinterpret_cast<float2*>(ws + L.rope_off);
  int* pos = reinterpret_cast<int*>(ws + L.pos_off);
  const int d = m.d, half = m.head_dim / 2, n = n_seq;

  prof_begin(RIFT_PROF_NORM, st);
  auto start = [&](auto kern) {
    kern<<<n, NORM_THREADS, 0, st>>>(token_ids, cu_seqlens, static_cast<const uint16_t*>(embed), vocab_embed, d, max_len,
                                     half, rope_freq(m), static_cast<const uint16_t*>(m.g_attn[0]), m.eps, h32, xn, rope,
                                     pos);
  };
  const int per_thread = (d / 4 + NORM_THREADS - 1) / NORM_THREADS;  // d <= 8192: at most 8
  if (per_thread <= 1) start(decode_start_kernel<1>);
  else if (per_thread <= 2) start(decode_start_kernel<2>);
  else if (per_thread <= 4) start(decode_start_kernel<4>);
  else start(decode_start_kernel<8>);
  prof_end(RIFT_PROF_NORM, st, 1);
  EpiParams rope_ep;
  rope_ep.positions = pos;
  rope_ep.rope = rope;
  rope_ep.rope_cols = 2 * d;
  rope_ep.head_dim = m.head_dim;
  rope_ep.max_len = n;  // the rows of the table
  const uint16_t* kv = static_cast<const uint16_t*>(kv_cache);
  // The layer's kernels are launched as programmatic dependents of the kernel before them: each
  // starts while its predecessor drains (the GEMMs already requesting their first weight tiles)
  // and waits for it before touching activations.
  const bool pdl = true;
  for (int l = 0; l < m.n_layers; ++l) {
    if (kv_new) {
      rope_ep.k_out = static_cast<uint16_t*>(kv_new) + (size_t)l * 2 * n * d;
      rope_ep.v_out = rope_ep.k_out + (size_t)n * d;
    }
    if (launch_gemm(xn, m.w_qkv[l], n, 3 * d, d, EPI_QKV_ROPE, qkv, st, rope_ep, pdl)) return 1;
    const uint16_t* Kc = kv + (size_t)l * 2 * T * d;
    const uint16_t* Vc = Kc + (size_t)T * d;
    prof_begin(RIFT_PROF_ATTN, st);
    const int nk = launch_decode_attention(qkv, Kc, Vc, T, cu_seqlens, n, m.n_heads, m.head_dim, max_len, att, st, pdl);
    if (nk < 0) return 1;
    prof_end(RIFT_PROF_ATTN, st, nk);
    if (launch_gemm(att, m.w_o[l], n, d, d, EPI_RESID_F32, h32, st, EpiParams(), pdl)) return 1;
    norm_launch(1, n, h32, nullptr, m.g_ffn[l], xn, d, m.eps, st, nullptr, pdl);
    if (launch_gemm(xn, m.w_gate_up[l], n, 2 * m.ffn, d, EPI_SWIGLU, act, st, EpiParams(), pdl)) return 1;
    if (launch_gemm(act, m.w_down[l], n, d, m.ffn, EPI_RESID_F32, h32, st, EpiParams(), pdl)) return 1;
    const void* next_gain = l + 1 < m.n_layers ? m.g_attn[l + 1] : m.g_final;
    norm_launch(1, n, h32, nullptr, next_gain, xn, d, m.eps, st, nullptr, pdl);
  }
  // xn now holds RMSNorm(h) g_final in fp16 (the logits operand)
  if (hidden_out)
    norm_launch(2, n, h32, nullptr, m.g_final, static_cast<uint16_t*>(hidden_out), d, m.eps, st, nullptr, pdl);
  if (logits) {
    if (launch_gemm(xn, m.lm_head, n, m.vocab, d, EPI_STORE_F32, logits, st, EpiParams(), pdl)) return 1;
  }
  return 0;
}

}  // namespace rift
