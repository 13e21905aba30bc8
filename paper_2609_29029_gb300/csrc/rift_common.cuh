// Shared device helpers of the Rift CUDA library (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cmath>

#include "rift.h"

// Device error bits, OR-ed into a per-translation-unit flag and collected by rift_sync_status.
#define RIFT_EBIT_NONFINITE 1u
#define RIFT_EBIT_CAPACITY 2u
#define RIFT_EBIT_TIMEOUT 4u
#define RIFT_EBIT_BADID 8u

// Upper bound on the spin iterations of any device-side wait (mbarrier, flag).  Waits that
// reach it set RIFT_EBIT_TIMEOUT and give up instead of hanging the GPU.
#define RIFT_SPIN_LIMIT (1u << 26)

#define RIFT_CUDA_TRY(expr)                          \
  do {                                               \
    cudaError_t _e = (expr);                         \
    if (_e != cudaSuccess) return RIFT_ERR_CUDA;     \
  } while (0)

#define RIFT_LAUNCH_CHECK() RIFT_CUDA_TRY(cudaGetLastError())

namespace rift {

// The unique id of the calling thread's current CUDA context (cuCtxGetId: ids are never reused
// within a process, unlike context handles), or 0 if it cannot be read.  (rift_abi.cu)
unsigned long long current_context_id();

// Raises `kernel`'s dynamic shared-memory limit to `bytes` in the current CUDA context.  A
// function's attributes belong to a context (every device's primary context, and any context a
// host creates with the driver API has its own), so `done`, the call site's record, holds the id
// of the context last raised; a call from another context (or with an unreadable id) raises again.
template <typename K>
inline cudaError_t raise_smem_limit(std::atomic<unsigned long long>& done, K* kernel, int bytes) {
  const unsigned long long ctx = current_context_id();
  if (ctx != 0 && done.load(std::memory_order_acquire) == ctx) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && ctx != 0) done.store(ctx, std::memory_order_release);
  return e;
}

// Allows `kernel` clusters of more than 8 CTAs (up to 16) in the current CUDA context; `done` as above.
template <typename K>
inline cudaError_t raise_cluster_limit(std::atomic<unsigned long long>& done, K* kernel) {
  const unsigned long long ctx = current_context_id();
  if (ctx != 0 && done.load(std::memory_order_acquire) == ctx) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && ctx != 0) done.store(ctx, std::memory_order_release);
  return e;
}

// A warp's value known to be the same in all lanes: it can be held in uniform registers.
template <typename T>
__device__ __forceinline__ T warp_uniform(T v) {
  return __shfl_sync(0xffffffffu, v, 0);
}

// True in one lane of a converged warp, the same one each time.  A warp whose lanes all run a loop of
// tcgen05 instructions and issue them under elect_one() pays ~15 cycles per instruction; one lane of its
// own branch pays ~70, because its operands (descriptors, addresses) have to be moved into uniform registers
// for each instruction.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.b32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// Programmatic dependent launch.  A kernel launched with `pdl` set (launch_ex) may begin while
// the kernel before it in the stream is still running: each of its threads calls pdl_wait()
// before its first access to memory that earlier kernels write or read (constant weights
// excepted), and pdl_trigger() lets the kernel after it begin launching.  Both are no-ops in a
// kernel launched without the attribute.  launch_cluster_ex
// also groups `cluster` consecutive CTAs along x into a thread-block cluster.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <typename... KArgs, typename... Args>
static inline cudaError_t launch_cluster_ex(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                            cudaStream_t st, bool pdl, int cluster, Args... args) {
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... KArgs, typename... Args>
static inline cudaError_t launch_ex(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                    bool pdl, Args... args) {
  return launch_cluster_ex(kernel, grid, block, smem, st, pdl, 1, args...);
}

// RoPE angular frequencies theta^(-2j / head_dim), j < head_dim / 2 <= 64, evaluated on the host in
// double.
struct RopeFreq {
  double inv[64];
};

// (cos, sin) of x >= 0 in double, good to ~2e-16 for x up to 2^31 and beyond: x reduced
// by the nearest multiple k of pi/2 (Cody and Waite's two-part reduction, its constants the leading
// bits of pi/2 and the rest), then the Taylor polynomials on |r| <= pi/4 (the first terms left out,
// r^17 / 17! and r^18 / 18!, are below 5e-17).
__host__ __device__ __forceinline__ double2 rope_cos_sin_f64(double x) {
  const double two_over_pi = 0.63661977236758134308, pio2 = 1.57079632679489661923, pio2_rest = 6.123233995736766e-17;
  const double k = rint(x * two_over_pi);
  const double r = fma(-k, pio2_rest, fma(-k, pio2, x));
  const double z = r * r;
  double s = fma(z, -1.0 / 1307674368000.0, 1.0 / 6227020800.0);
  s = fma(z, s, -1.0 / 39916800.0);
  s = fma(z, s, 1.0 / 362880.0);
  s = fma(z, s, -1.0 / 5040.0);
  s = fma(z, s, 1.0 / 120.0);
  s = fma(z, s, -1.0 / 6.0);
  s = fma(z * r, s, r);
  double c = fma(z, 1.0 / 20922789888000.0, -1.0 / 87178291200.0);
  c = fma(z, c, 1.0 / 479001600.0);
  c = fma(z, c, -1.0 / 3628800.0);
  c = fma(z, c, 1.0 / 40320.0);
  c = fma(z, c, -1.0 / 720.0);
  c = fma(z, c, 1.0 / 24.0);
  c = fma(z, c, -0.5);
  c = fma(z, c, 1.0);
  const int q = (int)((long long)k & 3);  // x = r + q pi/2 (mod 2 pi)
  return make_double2(q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s, q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c);
}
// The same, each rounded once to fp32.  A GB300 SM retires about two double operations a cycle,
// so they are what a RoPE table costs: this takes about 23 a value, the library's pow and sincos
// per value about 160 (a 131 x 64 table 11.6 us; now 4.3 us together with the attention schedule, whose own
// launch took 3.7; a decode step's start, which needs one row per sequence, 29.6 -> 8.0 us for one
// sequence of 635 rows).
__device__ __forceinline__ float2 rope_cos_sin(double x) {
  const double2 v = rope_cos_sin_f64(x);
  return make_float2((float)v.x, (float)v.y);
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Inclusive prefix sum over the 32 lanes of a warp.
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  return v;
}

// Block-wide sum; every thread gets the result.  `red` holds >= 32 floats.
__device__ __forceinline__ float block_sum(float v, float* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  float r = 0.f;
  for (int w = 0; w < nw; ++w) r += red[w];  // fixed order: same result in every thread
  return r;
}

// Block-wide exclusive prefix sum of one integer per thread (in thread order); *total gets the
// sum.  `sh` holds >= 33 ints.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* sh, T* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  const T inc = warp_incl_scan(v);
  __syncthreads();
  if (lane == 31) sh[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const T x = (lane < nw) ? sh[lane] : T(0);
    const T xi = warp_incl_scan(x);
    if (lane < nw) sh[lane] = xi - x;
    if (lane == nw - 1) sh[32] = xi;
  }
  __syncthreads();
  const T res = sh[wid] + inc - v;
  *total = sh[32];
  return res;
}

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) {
  return __uint_as_float(static_cast<uint32_t>(b) << 16);
}

// Unpack 8 bf16 values held in a uint4.
__device__ __forceinline__ void unpack_bf16x8(const uint4& v, float* f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Whether two rows hold the same bits (b null: whether the row is all zeros, of either sign), by one warp.
template <typename XT>
__device__ __forceinline__ bool same_row(const XT* a, const XT* b, int d, int lane) {
  constexpr int W = 16 / sizeof(XT);  // elements of a 16-byte load
  constexpr uint32_t ABS = sizeof(XT) == 2 ? 0x7fff7fffu : 0x7fffffffu;
  for (int k = lane * W; k < (d + 32 * W - 1) / (32 * W) * (32 * W); k += 32 * W) {
    uint32_t differ = 0u;
    if (k < d) {
      const uint4 x = *reinterpret_cast<const uint4*>(a + k);
      const uint4 y = b ? *reinterpret_cast<const uint4*>(b + k) : make_uint4(0u, 0u, 0u, 0u);
      differ = ((x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w)) & (b ? 0xffffffffu : ABS);
    }
    if (__any_sync(0xffffffffu, differ != 0u)) return false;
  }
  return true;
}

}  // namespace rift
