// The GEMMs on Blackwell's fifth-generation tensor cores (tcgen05, sm_103a).
//
// C[M, N] = A[M, K] . B[N, K]^T with fp16 operands (both K-major) and fp32 accumulation in
// tensor memory, plus the fused epilogues of the decoder layer (fp16 store with RoPE on q and
// k, fp32 residual add, SwiGLU over 16-column gate/up groups).  Two kernels:
//
// gemm_tc_kernel (many rows: the prefill of a scene): persistent and warp-specialised on SM pairs
// (2-CTA clusters, 256 x 256 tiles, or 256 x 192: tile_width), or on single SMs where 128 x 256 tiles take
// fewer waves (one_sm_tiles), 192 threads per CTA:
//   warp 0      one thread issues TMA tile loads (128B-swizzled) into a 6-stage shared-memory ring (4 on one SM)
//   warp 1      allocates 512 TMEM columns; the even CTA's issues tcgen05.mma (cta_group::2, M = 256,
//               N = 256, K = 16; a CTA alone cta_group::1, M = 128) into one of two 256-column fp32 accumulators and commits to
//               mbarriers
//   warps 2..5  epilogue: tcgen05.ld of their 32 TMEM lanes (one row per thread), fused op, store
// Warp 1 runs its loop with all lanes and issues under elect_one(): a K-block takes 514 cycles
// (the tensor pipe's own time is 512), against 551 with one lane issuing from a branch of its own.  The
// large products are limited by power all the same: their clock falls from 1650 to 1550 MHz with it, and the
// whole 400-tile query, a 5,900-row prefill and one of 2,448 rows over a prefix gained 1.2-1.9%, little more
// than two runs of one build differ by.
// Two accumulators let the epilogue of one tile overlap the main loop of the next.  Tiles are
// visited in bands whose rows of the larger operand fit in L2 (48 MB), so each tile of the other
// operand is read from DRAM once per band.
//
// gemm_ck_kernel (few rows: a decode step, one tile's prefill, a shared prompt, a small scene's
// Gram matrix): the operands swapped, K split over a thread-block cluster and the partial
// products summed through distributed shared memory (below).
//
// Every mbarrier wait is bounded (RIFT_SPIN_LIMIT iterations, ~4 s of globaltimer): on timeout
// the kernel sets RIFT_EBIT_TIMEOUT, lets every role fall through, waits for its issued copies
// and frees its tensor memory.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "rift_internal.h"

namespace rift {

__device__ unsigned int g_err_gemm;

unsigned int read_clear_err_gemm() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_err_gemm, sizeof(v));
  cudaMemcpyToSymbol(g_err_gemm, &z, sizeof(z));
  return v;
}

namespace tc {

constexpr int BM = 128, BN = 256, NARROW_BN = 192, BK = 64;
constexpr int A_BYTES = BM * BK * 2;  // 16 KB
constexpr int THREADS = 192;
// Depth of the ring of K-blocks: as deep as shared memory allows, 32 KB a CTA of a pair (cg = 2), 48 KB a CTA alone.
__host__ __device__ constexpr int ring_stages(int cg) { return cg == 2 ? 6 : 4; }
// Instruction descriptor, kind::f16: D fp32 (bits 4-5 = 1), A fp16 (bits
// 7-9 = 0), B fp16 (bits 10-12 = 0), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4
// at bits 24-28.

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor for a K-major tile written by TMA with 128-byte swizzling:
// start address >> 4 (bits 0-13), leading byte offset 16 B (unused for this layout), stride
// byte offset 1024 B between 8-row groups (bits 32-45), descriptor version 1 (bit 46),
// swizzle mode 2 = 128B (bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for the phase of parity `parity` (CL: acquire at cluster scope, for a barrier the
// other CTA of the pair arrives on).  Returns false if the kernel is aborting or the wait ran out
// (which starts the abort).
template <bool CL = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  auto tw = [&]() { return CL ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (tw()) return true;
  const uint64_t t0 = globaltimer();
  for (uint32_t i = 0; i < RIFT_SPIN_LIMIT; ++i) {
    if (tw()) return true;
    if ((i & 255u) == 255u) {
      if (*abort_flag) return false;
      if (globaltimer() - t0 > 4000000000ull) break;
    }
  }
  atomicOr(&g_err_gemm, RIFT_EBIT_TIMEOUT);
  *abort_flag = 1;
  return false;
}

// The same wait by a whole warp, one answer for all its lanes.
template <bool CL = false>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait<CL>(bar, parity, abort_flag));
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
               : "memory");
}
// The SM-pair forms (cta_group::2): the two CTAs of a 2-CTA cluster share one M = 256 product.
// The even CTA issues the MMA; each CTA holds its own 128 rows of A and 128 of the 256 B rows
// in shared memory at the same offsets, and its own 128 accumulator rows in tensor memory.
__device__ __forceinline__ void umma_f16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                              uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum));
}
// Arrive on the mbarrier at this offset in both CTAs of the pair once the pair's MMAs are done.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n" ::"r"(
          bar),
      "h"((uint16_t)3)
      : "memory");
}
// TMA load into this CTA's shared memory whose completion is counted on an mbarrier of either
// CTA of the pair (bar: a shared::cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// The shared::cluster address of this CTA's shared variable at `addr` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(d) : "r"(addr), "r"(rank));
  return d;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// 32 consecutive fp32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// Tile order.  group > 0: bands of `group` M-tiles, M fastest within a band, so the band's A rows
// stay in L2 while every B tile streams past them once per band.  group < 0: bands of -group
// N-tiles, N fastest, so the band's B rows stay in L2 and A streams once per band (the better
// order when B is the smaller operand: traffic A + B x bands vs B + A x bands).
__device__ __forceinline__ void tile_coords(int tile, int mt, int nt, int group, int& m_blk, int& n_blk) {
  const bool n_major = group < 0;
  const int g = n_major ? -group : group;
  const int inner = n_major ? nt : mt, outer = n_major ? mt : nt;
  const int per_group = g * outer;
  const int grp = tile / per_group;
  const int first = grp * g;
  const int gsz = min(inner - first, g);
  const int r = tile - grp * per_group;
  const int a = first + r % gsz, b = r / gsz;
  m_blk = n_major ? b : a;
  n_blk = n_major ? a : b;
}

// Tile t of the upper triangle (bi <= bj) of an mt x mt tile grid, row by row.
__device__ __forceinline__ void tri_coords(int t, int mt, int& bi, int& bj) {
  int b = 0;
  while (b < mt - 1 && t >= mt - b) {
    t -= mt - b;
    ++b;
  }
  bi = b;
  bj = b + t;
}

__device__ __forceinline__ float silu(float g) { return g / (1.f + expf(-g)); }

// Epilogue for one row of one 32-column chunk (columns n0 .. n0 + 31 of the tile).
template <int EPI>
__device__ __forceinline__ void epilogue_chunk(const uint32_t (&r)[32], int row, int col, int N, void* C,
                                               float out_scale = 1.f) {
  if constexpr (EPI == EPI_STORE_F32) {
    float* out = static_cast<float*>(C) + (size_t)row * N + col;
    if (col + 32 <= N) {
      float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        o4[q] = make_float4(__uint_as_float(r[4 * q]) * out_scale, __uint_as_float(r[4 * q + 1]) * out_scale,
                            __uint_as_float(r[4 * q + 2]) * out_scale, __uint_as_float(r[4 * q + 3]) * out_scale);
    } else {
      for (int j = 0; j < 32 && col + j < N; ++j) out[j] = __uint_as_float(r[j]) * out_scale;
    }
  } else if constexpr (EPI == EPI_STORE_BF16) {
    uint16_t* out = static_cast<uint16_t*>(C) + (size_t)row * N + col;
    if (col + 32 <= N) {
      uint4* o4 = reinterpret_cast<uint4*>(out);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        o4[q] = make_uint4(pack_half2(__uint_as_float(r[8 * q + 0]), __uint_as_float(r[8 * q + 1])),
                           pack_half2(__uint_as_float(r[8 * q + 2]), __uint_as_float(r[8 * q + 3])),
                           pack_half2(__uint_as_float(r[8 * q + 4]), __uint_as_float(r[8 * q + 5])),
                           pack_half2(__uint_as_float(r[8 * q + 6]), __uint_as_float(r[8 * q + 7])));
    } else {
#pragma unroll
      for (int j = 0; j < 32; j += 2)
        if (col + j < N)
          *reinterpret_cast<uint32_t*>(out + j) = pack_half2(__uint_as_float(r[j]), __uint_as_float(r[j + 1]));
    }
  } else if constexpr (EPI == EPI_RESID_F32) {
    float* out = static_cast<float*>(C) + (size_t)row * N + col;
    if (col + 32 <= N) {
      float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float4 v = o4[q];
        v.x += __uint_as_float(r[4 * q + 0]);
        v.y += __uint_as_float(r[4 * q + 1]);
        v.z += __uint_as_float(r[4 * q + 2]);
        v.w += __uint_as_float(r[4 * q + 3]);
        o4[q] = v;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (col + j < N) out[j] += __uint_as_float(r[j]);
    }
  } else if constexpr (EPI == EPI_SWIGLU) {  // columns col..col+15 gate, col+16..col+31 the matching up
    if (col >= N) return;
    const int F = N / 2;
    uint16_t* out = static_cast<uint16_t*>(C) + (size_t)row * F + col / 2;
    uint32_t p[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float g0 = __uint_as_float(r[2 * j]), g1 = __uint_as_float(r[2 * j + 1]);
      const float u0 = __uint_as_float(r[16 + 2 * j]), u1 = __uint_as_float(r[16 + 2 * j + 1]);
      p[j] = pack_half2(silu(g0) * u0, silu(g1) * u1);
    }
    uint4* o4 = reinterpret_cast<uint4*>(out);
    o4[0] = make_uint4(p[0], p[1], p[2], p[3]);
    o4[1] = make_uint4(p[4], p[5], p[6], p[7]);
  }
}

// x cos + partner sin, one rounding each for the product and the sum: written out, so that every
// kernel's RoPE gives the same bits.
__device__ __forceinline__ float rope_mul(float x, float partner, float c, float s) {
  return fmaf(x, c, __fmul_rn(partner, s));
}

// Rotate-half RoPE on fp32 accumulators: r1 holds dims j0..j0+31 of a head, r2 the partner
// dims j0+half..; y1 = x1 cos - x2 sin, y2 = x2 cos + x1 sin, rounded once to fp16.
// `out`: the row's element of r1[0]; `copy` (nullable): a second place to store to (the KV cache).
__device__ __forceinline__ void rope_chunk(const uint32_t (&r1)[32], const uint32_t (&r2)[32], int col, int half,
                                           int pos, const float2* __restrict__ tab, uint16_t* out, uint16_t* copy) {
  const int head_dim = 2 * half;
  const int j0 = col % head_dim;
  const float2* cs = tab + (size_t)pos * half + j0;
  uint32_t p1[16], p2[16];
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    const float2 c0 = cs[e], c1 = cs[e + 1];
    const float a0 = __uint_as_float(r1[e]), a1 = __uint_as_float(r1[e + 1]);
    const float b0 = __uint_as_float(r2[e]), b1 = __uint_as_float(r2[e + 1]);
    p1[e / 2] = pack_half2(rope_mul(a0, b0, c0.x, -c0.y), rope_mul(a1, b1, c1.x, -c1.y));
    p2[e / 2] = pack_half2(rope_mul(b0, a0, c0.x, c0.y), rope_mul(b1, a1, c1.x, c1.y));
  }
  auto store = [&](uint16_t* dst) {
    uint4* o1 = reinterpret_cast<uint4*>(dst);
    uint4* o2 = reinterpret_cast<uint4*>(dst + half);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      o1[q] = make_uint4(p1[4 * q], p1[4 * q + 1], p1[4 * q + 2], p1[4 * q + 3]);
      o2[q] = make_uint4(p2[4 * q], p2[4 * q + 1], p2[4 * q + 2], p2[4 * q + 3]);
    }
  };
  store(out);
  if (copy) store(copy);
}

// K-block k of an operand read through EpiParams' remap (mode 1: [hi | hi | lo], 2: [hi | lo | hi]
// over a stored [hi | lo] row of D blocks each; 0: k).
__device__ __forceinline__ int kblock(int mode, int D, int k) {
  return mode == 1 ? (k < D ? k : k - D) : mode == 2 ? (k < 2 * D ? k : k - 2 * D) : k;
}

// Width of the SM pairs' tiles: NARROW_BN where that takes no more waves of tiles than BN and there is
// more than one.  The narrower tiles' K-blocks take 0.89-0.92 of the time (not 0.75: they are bound by the
// supply from L2, ~14 TB/s), so the width pays where the last wave would leave SMs idle and nowhere else.
// us, 256 against 192: W_o at 1,500 rows (2 waves each) 57 : 53, at 2,448 (3) 78 : 70, W_down 119 : 107 and
// 179 : 160, gate/up at 203 (2) 70 : 60; at 3,000 rows (3 waves, 4) W_o 78 : 88, W_down 182 : 213.  In one wave
// W_o at 600 rows takes 35 both ways.
__device__ __forceinline__ int tile_width(int mt, int N, int pairs) {
  const int wide = (mt * ((N + BN - 1) / BN) + pairs - 1) / pairs;
  const int narrow = (mt * ((N + NARROW_BN - 1) / NARROW_BN) + pairs - 1) / pairs;
  return wide > 1 && narrow <= wide ? NARROW_BN : BN;
}

// 2-CTA clusters on an SM pair, 256 x 256 tiles (cta_group::2; 256 x 192 by tile_width): each SM stages 128
// rows of A and half of the tile's B rows per k-block, half the B traffic of one SM per tile row, and
// the even CTA issues the M = 256 MMAs into both SMs' tensor memory.  tmN: the B map with boxes of the
// narrower tile's half.
// CG = 1 (one_sm_tiles): one SM a tile, 128 x 256, all of the tile's B rows staged by its CTA; no clusters, no
// narrower tiles, tmB with boxes of a whole tile.
template <int EPI, int CG>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmN, int M_cap, int N, int K, void* C, const EpiParams ep,
                   int group_m) {
  constexpr int TM = CG * BM;      // rows of a tile (both CTAs of the pair)
  constexpr int B_ROWS = BN / CG;  // B rows staged by this CTA
  constexpr int STAGES = ring_stages(CG);
  constexpr int B_BYTES = B_ROWS * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr int ACC_COLS = BN, TMEM_COLS = 2 * ACC_COLS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull_bar(b), 1);
      mbar_init(tempty_bar(b), 128 * CG);  // the epilogue threads of the tile's CTAs
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
  if constexpr (CG == 2) cluster_sync();  // both CTAs' barriers initialised before any remote arrival
  if (warp == 1) {
    if constexpr (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem_base = warp_uniform(*tmem_slot);
  pdl_trigger();
  pdl_wait();
  // Rows: M_cap (host), or the device count ep.m_dev clamped to it (the rows the TMA map covers).
  const int M = ep.m_dev ? max(0, min(M_cap, *ep.m_dev)) : M_cap;

  // The first K-block, as a value the compiler does not know: with a constant it peels the K loops and the
  // products of 23,800 rows take 0.5% longer.
  int kb0;
  asm volatile("mov.s32 %0, 0;" : "=r"(kb0));
  const int mt = (M + TM - 1) / TM, kt = (K + BK - 1) / BK;
  int bn = BN;  // the RoPE epilogue wants whole heads in a tile, the symmetric product square tiles
  if constexpr (EPI != EPI_QKV_ROPE && CG == 2)
    if (!ep.symmetric) bn = tile_width(mt, N, (int)(gridDim.x >> 1));
  const int nt = (N + bn - 1) / bn;
  const int n_tiles = ep.symmetric ? mt * (mt + 1) / 2 : mt * nt;
  auto coords = [&](int tile, int& m_blk, int& n_blk) {
    if (ep.symmetric) tri_coords(tile, mt, m_blk, n_blk);
    else tile_coords(tile, mt, nt, group_m, m_blk, n_blk);
  };
  // the pair walks the tiles together, one tile per cluster
  const int u_first = (int)blockIdx.x / CG, u_step = (int)gridDim.x / CG;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer: both CTAs load their halves; the even CTA's full barrier
      // counts the bytes of both
      int it = 0;
      bool ok = true;
      for (int u = u_first; u < n_tiles && ok; u += u_step) {
        int m_blk, n_blk;
        coords(u, m_blk, n_blk);
        for (int k = kb0; k < kt; ++k, ++it) {
          const int s = it % STAGES;
          const uint32_t round = it / STAGES;
          if (!mbar_wait(empty_bar(s), (round & 1u) ^ 1u, abort_flag)) { ok = false; break; }
          const int ka = kblock(ep.kmap_a, ep.kmap_d, k) * BK, kb = kblock(ep.kmap_b, ep.kmap_d, k) * BK;
          if (rank == 0) mbar_expect_tx(full_bar(s), CG * A_BYTES + bn * BK * 2);
          if constexpr (CG == 2) {
            const uint32_t fb = mapa_shared(full_bar(s), 0);
            tma_load_2d_pair(smem_u32(sA + s * A_BYTES), &tmA, ka, m_blk * TM + (int)rank * BM, fb);
            tma_load_2d_pair(smem_u32(sB + s * B_BYTES), EPI == EPI_QKV_ROPE || bn == BN ? &tmB : &tmN, kb,
                             n_blk * bn + (int)rank * (bn >> 1), fb);
          } else {
            tma_load_2d(smem_u32(sA + s * A_BYTES), &tmA, ka, m_blk * TM, full_bar(s));
            tma_load_2d(smem_u32(sB + s * B_BYTES), &tmB, kb, n_blk * BN, full_bar(s));
          }
        }
      }
      // Before leaving, make sure no copy this thread issued is still in flight (bounded): the
      // copies are counted on the even CTA's barrier, so wait instead for the MMAs' releases of
      // the last stages, which also keeps this CTA alive until they have all arrived.
      for (int j = 1; j <= STAGES && it - j >= 0; ++j) {
        const int i2 = it - j;
        for (uint32_t w = 0; w < (1u << 22) && !mbar_try_wait(empty_bar(i2 % STAGES), (i2 / STAGES) & 1u); ++w) {
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------- MMA issuer (the even CTA only)
      int it = 0, tl = 0;
      bool ok = true;
      const uint32_t idesc = (1u << 4) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
      for (int u = u_first; u < n_tiles && ok; u += u_step, ++tl) {
        const int b = tl & 1;
        const uint32_t use = tl >> 1;
        if (!mbar_wait_warp<true>(tempty_bar(b), (use & 1u) ^ 1u, abort_flag)) break;
        fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(b * ACC_COLS);
        for (int k = kb0; k < kt; ++k, ++it) {
          const int s = it % STAGES;
          const uint32_t round = it / STAGES;
          if (!mbar_wait_warp(full_bar(s), round & 1u, abort_flag)) { ok = false; break; }
          fence_after();
          const uint64_t ad = smem_desc(smem_u32(sA + s * A_BYTES));
          const uint64_t bd = smem_desc(smem_u32(sB + s * B_BYTES));
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)  // +32 bytes along K per step (encoded >> 4)
              if constexpr (CG == 2) umma_f16_pair(tmem_d, ad + 2 * kk, bd + 2 * kk, idesc, (k != kb0 || kk != 0) ? 1u : 0u);
              else umma_f16(tmem_d, ad + 2 * kk, bd + 2 * kk, idesc, (k != kb0 || kk != 0) ? 1u : 0u);
            if constexpr (CG == 2) umma_commit_pair(empty_bar(s));
            else umma_commit(empty_bar(s));
          }
          __syncwarp();
        }
        if (ok && elect_one()) {
          if constexpr (CG == 2) umma_commit_pair(tfull_bar(b));
          else umma_commit(tfull_bar(b));
        }
        __syncwarp();
      }
      // the last two accumulators' releases (the odd CTA's arrivals among them) have landed
      for (int t = tl - 1; t >= 0 && t >= tl - 2; --t)
        for (uint32_t w = 0; w < (1u << 22) && !mbar_try_wait_cluster(tempty_bar(t & 1), (t >> 1) & 1u); ++w) {
        }
    }
  } else {
    // ---------------- epilogue (warps 2..5 -> TMEM lane quarters 2, 3, 0, 1)
    const int quarter = warp & 3;
    const uint32_t tempty_even0 = CG == 2 ? mapa_shared(tempty_bar(0), 0) : tempty_bar(0);
    const uint32_t tempty_even1 = CG == 2 ? mapa_shared(tempty_bar(1), 0) : tempty_bar(1);
    int tl = 0;
    for (int u = u_first; u < n_tiles; u += u_step, ++tl) {
      int m_blk, n_blk;
      coords(u, m_blk, n_blk);
      const int b = tl & 1;
      const uint32_t use = tl >> 1;
      if (!mbar_wait(tfull_bar(b), use & 1u, abort_flag)) break;
      fence_after();
      const int row = m_blk * TM + (int)rank * BM + quarter * 32 + lane;
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * ACC_COLS);
      if constexpr (EPI == EPI_QKV_ROPE) {
        const int half = ep.head_dim >> 1, kv_d = ep.rope_cols >> 1;
        const int pos = (row < M) ? ep.positions[row] + ep.pos_offset : 0;
        const bool pos_ok = pos >= 0 && pos < ep.max_len;
        if (row < M && !pos_ok) atomicOr(&g_err_gemm, RIFT_EBIT_BADID);
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          const int col = n_blk * BN + c;
          if (col >= N) break;
          if (col < ep.rope_cols) {
            if ((c % ep.head_dim) >= half) continue;  // done with its partner c - half
            uint32_t r1[32], r2[32];
            tmem_ld32(taddr + c, r1);
            tmem_ld32(taddr + c + half, r2);
            if (row < M && pos_ok)
              rope_chunk(r1, r2, col, half, pos, ep.rope, static_cast<uint16_t*>(C) + (size_t)row * N + col,
                         ep.k_out && col >= kv_d ? ep.k_out + (size_t)row * kv_d + col - kv_d : nullptr);
          } else {
            uint32_t r[32];
            tmem_ld32(taddr + c, r);
            if (row < M) {
              epilogue_chunk<EPI_STORE_BF16>(r, row, col, N, C);
              if (ep.v_out) epilogue_chunk<EPI_STORE_BF16>(r, row, col - ep.rope_cols, kv_d, ep.v_out);
            }
          }
        }
      } else {
#pragma unroll 1
        for (int c = 0; c < bn; c += 32) {
          uint32_t r[32];
          tmem_ld32(taddr + c, r);
          if (row < M) epilogue_chunk<EPI>(r, row, n_blk * bn + c, N, C, ep.out_scale);
          if constexpr (EPI == EPI_STORE_F32) {
            // symmetric product: the off-diagonal tile also fills its mirror (a warp's lanes hold
            // consecutive rows, so each transposed store is 32 consecutive floats)
            if (ep.symmetric && m_blk != n_blk && row < M) {
              float* out = static_cast<float*>(C);
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                const int col = n_blk * BN + c + e;
                if (col < M) out[(size_t)col * N + row] = __uint_as_float(r[e]) * ep.out_scale;
              }
            }
          }
        }
      }
      fence_before();
      if constexpr (CG == 2) mbar_arrive_cluster(b ? tempty_even1 : tempty_even0);
      else mbar_arrive(b ? tempty_even1 : tempty_even0);
    }
  }
  fence_before();
  __syncthreads();
  if constexpr (CG == 2) cluster_sync();  // neither CTA frees its tensor memory or exits before the other is done
  if (warp == 1) {
    fence_after();
    if constexpr (CG == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(TMEM_COLS)
                   : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(TMEM_COLS)
                   : "memory");
  }
}

// ---------------------------------------------------------------- few rows: split K over a cluster
// C[M, N] = A[M, K] . W[N, K]^T for products with few rows (M < 1024: a decode step, one tile's
// prefill, a shared prompt, a small scene's Gram matrix), which stream the weights once.  The
// operands are swapped: a CTA holds 128 weight rows as the MMA's M side and bn activation rows
// (16 .. 160, a multiple of 16) as its N side, so a few rows cost no
// more shared memory or tensor work than they need.  A cluster of S CTAs (1 .. 16) shares a tile:
// rank r multiplies the K-blocks [kt r / S, kt (r + 1) / S), every CTA leaves its fp32 partial
// product in its own shared memory, and after a cluster barrier rank r adds the S partials of
// the rows r, r + S, ... in rank order (through distributed shared memory) and applies the
// epilogue.  No partial product goes through HBM and no reduction kernel follows.  The ring is
// sized for two CTAs per SM, so that uneven unit counts share the memory bandwidth evenly and a
// programmatic dependent launch finds room next to the kernel before it: its CTAs request their
// first weight tiles (w_const) before they wait for that kernel.
// Bound by HBM (the weights) for one row tile; measured on one GB300, weights rotating through more
// than L2, us per launch, against one SM per 128 x 256 tile without a split (in brackets), 7B shapes:
//   rows   QKV           W_o           gate/up       W_down
//      1   22.8 (32.8)   12.3 (32.1)   35.8 (53.5)   21.6 (71.4)
//    131   27.0 (35.0)   17.6 (39.0)   46.8 (64.6)   27.7 (78.2)
// and 19.3 / 9.2 / 32.1 / 18.2 for one row as programmatic dependents, 1.2 - 1.9 times the time the
// weights take at the HBM rate; what is left is each launch's fill and drain.  The split-K it
// replaces in the decode step wrote its partial products to HBM and read them back in a
// reduction launch: one 7B layer's products at one row 113 us then, 79 us now.
namespace ck {
constexpr int THREADS = 192, PORTABLE_S = 8, MAX_S = 16, MAX_BN = 160;
constexpr int W_BYTES = BM * BK * 2;
constexpr int SMEM = 232448 / 2 - 1024;  // two CTAs per SM
constexpr int RING = SMEM - 1024 - 512;  // after alignment; the barriers at the end
__host__ __device__ constexpr int stage_bytes(int bn) { return W_BYTES + bn * BK * 2; }
__host__ __device__ constexpr int stages(int bn) {
  return RING / stage_bytes(bn) < 8 ? RING / stage_bytes(bn) : 8;
}
static_assert(MAX_BN * BM * 4 <= RING, "the partial product reuses the ring");

// Row tiles: as few as MAX_BN allows, of equal height.  S: as many CTAs per tile as the GPU holds
// at once, each with at least 8 K-blocks (a shorter slice is all fill and drain; a Gram
// matrix, on its own in a chain of small kernels, takes slices of 3).  More than 8 CTAs (a
// non-portable cluster) where one tile would leave the rest idle: 16 for the Gram matrix of up to 128 tiles, K = 3 d (64 tiles at d = 4096: 11 us with 16, 15 with 8).
// A Gram matrix of more than 32 tiles takes 4 at most: it starts while the kernel before it drains, and larger
// clusters then wait for a GPC.  Whole smoothing, us, S = 4 : 5: 1,024 scene tiles at d = 1024 59 : 69, 4096 93 : 101,
// 8192 150 : 162; 832 at 4096 79 : 84 (6: 84), 8192 123 : 122 (6: 121); up to 32 tiles 8 wins (700 at 8192 108, with 4 118).
// More CTAs than fit at once cost a second round: gate/up at one row 35.8 us with 172 CTAs, 43.6
// with 344; W_o 12.3 us with 256 (S = 8), 13.7 with 128, 28.9 with 32.  Two CTAs fit on an SM, but a cluster has to
// fit in one GPC: resident[S] clusters at once (asked from the driver), fewer than 2 SMs / S for most S.  100 rows,
// us, by the count of CTAs alone against resident[S]: N = 5120 x K = 4096 28.7 (S = 7) : 20.7 (6), 6144 x 4096
// 30.7 (6) : 22.5 (5).  A programmatic dependent launch (pdl) is placed around the CTAs of the kernel before it, and
// where all clusters of 3 or more would only just fit, some wait for a second round: a sixteenth is left free then
// (two layers over 347 rows, whose W_o takes 96 tiles, 507 us with S = 3, of which 97 fit, 466 with S = 2; 20 decoded
// tokens 472 : 459).  A quarter free is too much (524 rows 536 : 575), pairs need none (2,970 rows at d = 1024, 152 of
// 152 pairs, 298 : 321), nor does a launch of its own (W_o at 384 rows 26.6 : 32.8), nor do fewer than 8 rows, whose
// norm before it takes as many CTAs (decode steps over 4 layers, without : with: 1 row 418 : 420, 3 418 : 424, 6 420 : 422,
// 8 431 : 429, 16 453 : 441).
// K too short to split (fewer than 16 K-blocks): row tiles of at most SHORT_BN instead, as long as they fit at
// once; what a CTA takes is then its epilogue, a serial chain over its rows.  us, tiles of 160 rows, 48, and the
// SM pairs, 300 rows: 256 x 256 + residual 22.5 : 12.3 : 20.5, 768 x 256 10.2 : 8.2 : 14.3, SwiGLU 1376 x 256
// 14.3 : 10.2 : 16.4; 1,500 rows of the last (too many to fit) 14.3 : 14.3 : 16.4.
constexpr int SHORT_BN = 48;
struct Plan {
  int bn, S;
  bool one_round;  // all its CTAs are resident at once, or the K slices are
};
inline Plan plan(int M, int N, int K, int sms, const int* resident, bool gram, bool pdl) {
  const long long n_tiles = (N + BM - 1) / BM;
  const int kt = (K + BK - 1) / BK;
  const int min_blocks = gram ? 3 : 8;
  auto height = [&](int m_tiles) { return ((M + m_tiles - 1) / m_tiles + 15) / 16 * 16; };
  if (!gram && kt < 2 * min_blocks) {
    const int m_tiles = (M + SHORT_BN - 1) / SHORT_BN;
    if (m_tiles * n_tiles <= 2LL * sms) return {height(m_tiles), 1, true};
  }
  const int m_tiles = (M + MAX_BN - 1) / MAX_BN;
  const long long tiles = m_tiles * n_tiles;
  if (gram && tiles <= 2 && kt / MAX_S >= min_blocks) return {height(m_tiles), MAX_S, true};
  int S = gram && tiles > 32 ? 4 : PORTABLE_S;
  auto fit = [&](int s) { return pdl && M >= 8 && s > 2 ? resident[s] * 15 / 16 : resident[s]; };
  while (S > 1 && (tiles > fit(S) || kt / S < min_blocks)) --S;
  return {height(m_tiles), S, S >= 2};
}
}  // namespace ck

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// MAXS: the largest cluster this instance sums over (1, 4, 8 or 16; the partial sums' loads are unrolled
// over it, so that they are all in flight: with one instance for 16, 3 us more a launch).
template <int EPI, int MAXS>
__global__ void __launch_bounds__(ck::THREADS, 2)
    gemm_ck_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, int M_cap, int N,
                   int K, void* C, const EpiParams ep, int bn, int m_tiles, int S, int w_const) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + ck::RING);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 18);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int stage_bytes = ck::stage_bytes(bn), stages = ck::stages(bn);
  const uint32_t smem0 = smem_u32(smem), bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (8 + s); };
  const uint32_t done_bar = bar0 + 8u * 16;
  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  uint32_t cols = 32;  // tensor memory columns: the power of two that holds bn
  while (cols < (uint32_t)bn) cols *= 2;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = warp_uniform(*tmem_slot);
  pdl_trigger();
  if (warp != 0 || ep.m_dev) pdl_wait();
  const int M = ep.m_dev ? max(0, min(M_cap, *ep.m_dev)) : M_cap;
  const int rank = (int)cluster_ctarank();  // blockIdx.x % S
  const int tile = (int)blockIdx.x / S;
  const int m0 = (tile % m_tiles) * bn, n0 = (tile / m_tiles) * BM;
  const int mv = min(bn, M - m0);  // rows of this tile (<= 0: past the device count, nothing to do)
  const int kt = (K + BK - 1) / BK;
  const int k0 = kt * rank / S, k1 = kt * (rank + 1) / S;

  if (warp == 0) {
    if (mv > 0) {
      // ---------------- TMA producer: a weight tile and the activation tile per K-block
      auto load_w = [&](int s, int k) {
        tma_load_2d(smem0 + s * stage_bytes, &tmW, kblock(ep.kmap_b, ep.kmap_d, k) * BK, n0, full_bar(s));
      };
      auto load_x = [&](int s, int k) {
        tma_load_2d(smem0 + s * stage_bytes + ck::W_BYTES, &tmX, kblock(ep.kmap_a, ep.kmap_d, k) * BK, m0, full_bar(s));
      };
      const int n_pre = w_const && !ep.m_dev ? min(stages, k1 - k0) : 0;
      if (elect_one()) {
        for (int j = 0; j < n_pre; ++j) {
          mbar_expect_tx(full_bar(j), stage_bytes);
          load_w(j, k0 + j);
        }
      }
      __syncwarp();
      pdl_wait();
      int it = 0;
      for (int k = k0; k < k1; ++k, ++it) {
        const int s = it % stages;
        // (it < n_pre: the weight tile is on its way, and in the first round the stage is free)
        if (it >= n_pre && !mbar_wait_warp(empty_bar(s), ((it / stages) & 1u) ^ 1u, abort_flag)) break;
        if (elect_one()) {
          if (it >= n_pre) {
            mbar_expect_tx(full_bar(s), stage_bytes);
            load_w(s, k);
          }
          load_x(s, k);
        }
        __syncwarp();
      }
      for (int j = 1; j <= stages && it - j >= 0; ++j) {  // no copy left in flight (bounded)
        const int i2 = it - j;
        for (uint32_t w = 0; w < (1u << 22) && !mbar_try_wait(full_bar(i2 % stages), (i2 / stages) & 1u); ++w) {
        }
      }
    }
  } else if (warp == 1) {
    if (mv > 0) {
      // ---------------- MMA issuer
      const uint32_t idesc = (1u << 4) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      bool ok = true;
      for (int k = k0, it = 0; k < k1; ++k, ++it) {
        const int s = it % stages;
        if (!mbar_wait_warp(full_bar(s), (it / stages) & 1u, abort_flag)) { ok = false; break; }
        fence_after();
        const uint64_t wd = smem_desc(smem0 + s * stage_bytes), xd = smem_desc(smem0 + s * stage_bytes + ck::W_BYTES);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            umma_f16(tmem, wd + 2 * kk, xd + 2 * kk, idesc, (it != 0 || kk != 0) ? 1u : 0u);
          umma_commit(empty_bar(s));
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(done_bar);
      __syncwarp();
    }
  } else if (mv > 0) {
    // ---------------- the partial product to shared memory: P[row m][weight row], over the ring
    // (every copy has been consumed by a completed MMA)
    const int quarter = warp & 3;
    if (__all_sync(0xffffffffu, mbar_wait(done_bar, 0, abort_flag))) {
      fence_after();
      float* P = reinterpret_cast<float*>(smem) + quarter * 32 + lane;
      const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
      for (int c = 0; c < mv; c += 16) {
        uint32_t r[16];
        tmem_ld16(taddr + c, r);
#pragma unroll
        for (int e = 0; e < 16; ++e) P[(c + e) * BM] = __uint_as_float(r[e]);
      }
      fence_before();
    }
  }
  __syncwarp();
  if constexpr (MAXS == 1) __syncthreads();
  else cluster_sync();  // every CTA's partial product is in place
  if (mv > 0 && !*abort_flag) {
    uint32_t base[MAXS];
#pragma unroll
    for (int r = 0; r < MAXS; ++r) base[r] = MAXS == 1 ? smem0 : r < S ? mapa_shared(smem0, r) : 0u;
    // the sum over the ranks of four weight rows' partials (columns q .. q + 3) of row m
    auto acc4 = [&](int m, int q) {
      if constexpr (MAXS == 1) {
        return *reinterpret_cast<const float4*>(smem + (m * BM + q) * 4);
      } else {
        const uint32_t off = (uint32_t)(m * BM + q) * 4u;
        float4 f[MAXS];
#pragma unroll
        for (int r = 0; r < MAXS; ++r)
          if (r < S) f[r] = ld_cluster4(base[r] + off);
        float4 v = f[0];
#pragma unroll
        for (int r = 1; r < MAXS; ++r)
          if (r < S) {
            v.x += f[r].x;
            v.y += f[r].y;
            v.z += f[r].z;
            v.w += f[r].w;
          }
        return v;
      }
    };
    auto store_h4 = [](void* dst, float a, float b, float c, float d) {
      *reinterpret_cast<uint2*>(dst) = make_uint2(pack_half2(a, b), pack_half2(c, d));
    };
    constexpr int QUADS = EPI == EPI_SWIGLU ? 16 : 32;  // outputs of a row / 4
    const int rows = (mv - rank + S - 1) / S;           // rows rank, rank + S, ... of the tile
    for (int i = threadIdx.x; i < rows * QUADS; i += ck::THREADS) {
      const int m = rank + (i / QUADS) * S, q = (i % QUADS) * 4;
      const size_t row = (size_t)(m0 + m);
      if constexpr (EPI == EPI_SWIGLU) {  // outputs q .. q + 3 of the tile's 64: gate 32 (q / 16) + q % 16, up 16 on
        const int gq = 32 * (q / 16) + q % 16;
        if (n0 + gq >= N) continue;
        const float4 g = acc4(m, gq), u = acc4(m, gq + 16);
        store_h4(static_cast<uint16_t*>(C) + row * (N / 2) + n0 / 2 + q, silu(g.x) * u.x, silu(g.y) * u.y,
                 silu(g.z) * u.z, silu(g.w) * u.w);
      } else {
        const int col = n0 + q;
        if (col >= N) continue;
        float4 v = acc4(m, q);
        if constexpr (EPI == EPI_STORE_F32) {
          *reinterpret_cast<float4*>(static_cast<float*>(C) + row * N + col) =
              make_float4(v.x * ep.out_scale, v.y * ep.out_scale, v.z * ep.out_scale, v.w * ep.out_scale);
        } else if constexpr (EPI == EPI_RESID_F32) {
          float4* o = reinterpret_cast<float4*>(static_cast<float*>(C) + row * N + col);
          float4 h = *o;
          h.x += v.x;
          h.y += v.y;
          h.z += v.z;
          h.w += v.w;
          *o = h;
        } else {
          if constexpr (EPI == EPI_QKV_ROPE) {
            if (col < ep.rope_cols) {
              const int half = ep.head_dim >> 1, j = q % ep.head_dim;
              const int pos = ep.positions[row] + ep.pos_offset;
              if (pos < 0 || pos >= ep.max_len) {
                if (j == 0) atomicOr(&g_err_gemm, RIFT_EBIT_BADID);
                continue;  // q and k of a row without a valid position stay unwritten
              }
              const bool lo = j < half;
              const float4* cs4 = reinterpret_cast<const float4*>(ep.rope + (size_t)pos * half + (lo ? j : j - half));
              const float4 c01 = cs4[0], c23 = cs4[1];  // (cos, sin) of four dims
              const float4 x = acc4(m, lo ? q + half : q - half);
              const float sg = lo ? -1.f : 1.f;
              v = make_float4(rope_mul(v.x, x.x, c01.x, sg * c01.y), rope_mul(v.y, x.y, c01.z, sg * c01.w),
                              rope_mul(v.z, x.z, c23.x, sg * c23.y), rope_mul(v.w, x.w, c23.z, sg * c23.w));
            }
          }
          store_h4(static_cast<uint16_t*>(C) + row * N + col, v.x, v.y, v.z, v.w);
          if constexpr (EPI == EPI_QKV_ROPE) {
            const int kv_d = ep.rope_cols >> 1;
            if (ep.k_out && col >= kv_d)
              store_h4(col < ep.rope_cols ? ep.k_out + row * kv_d + col - kv_d : ep.v_out + row * kv_d + col - ep.rope_cols,
                       v.x, v.y, v.z, v.w);
          }
        }
      }
    }
  }
  __syncwarp();
  if constexpr (MAXS > 1) cluster_sync();  // no CTA leaves while another may still read its partial product
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols) : "memory");
  }
}

// ---------------------------------------------------------------- merge screening (Stage 2)
// Similarity of the unselected tokens of a kept tile to the tile's merge targets on the tensor cores:
// per (kept slot j, 128 of its unselected tokens) a 128 x m x d bf16 product against up to COLS target
// rows at a time, one token row per epilogue thread, which keeps the two best targets by
// x.t / ||t|| (fp32, ties to the lower target) for each token that is not itself a target.  Bound by
// HBM (the unselected tokens, read once): the four epilogue warps gather the token rows with
// cp.async into the swizzled tiles, so the selected tokens are neither read nor multiplied (three
// blocks a slot instead of five at 333 of 576 tokens), 48 KB a CTA in flight; TMA's gather4 form
// took 11 cycles per 128-byte row: 65 us at 400 tiles (about 95 kept), 102 with gather4, 87 reading
// every token.  A target is within the screening's error if x.t / ||t|| is less than the bound below the best one's;
// where others than the best are, the choice among them is made at ~fp64 accuracy outside (merge.cu).  The bound
// scales with ||x||, which the gathering threads sum from their own chunks.
// Bound.  An accumulator update adds 16 exact products to the accumulator: the 17 addends aligned to the largest and cut,
// the result cut to fp32.  Measured on this unit (a test holds it to that) an addend loses less than 2^-25 of the
// largest one's power of two, the result less than 2^-23 of its own, and no addend or result is larger than ||x|| ||t||:
// (16 / 4 + 1) 2^-23 an update, d / 16 of them (5 / 16) d 2^-23 ||x|| in x.t / ||t||, plus 2^-23 for the roundings of
// 1 / ||t|| and of the product with it; the difference of two twice that, (0.625 d + 2) 2^-23 ||x||.  Twice this is taken,
// (1.25 d + 8) 2^-23 ||x|| rounded up, which leaves room for the norm's own rounding and would cover a cut at 2^-24.  About
// 12% of the tokens of a random tile have a second target within it, 0.6% a third.  Where squares or products
// could underflow (||x|| < 2^-30, a target's norm < 2^-40) every target counts as within it.  Up to seven targets are
// listed for a token, from a second look at its products where more than two are within; more than seven, or more
// than two beyond one block of COLS targets, and all are candidates.
namespace ms {
constexpr int STAGES = 4, THREADS = 192, COLS = 80, TMEM_COLS = 128;
constexpr int BROWS = 16;  // target rows per TMA box: a product is as wide as its targets need
constexpr int A_BYTES = 128 * BK * 2, B_BYTES = COLS * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024 + 256;
// kind::f16 with bf16 A and B (bits 7-9 and 10-12 = 1), fp32 D, K-major, M = 128; N >> 3 added at bit 17
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);
}  // namespace ms

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}

__global__ void __launch_bounds__(ms::THREADS, 2)
    merge_screen_kernel(const __grid_constant__ CUtensorMap tmT, const uint16_t* __restrict__ X, int n_v, int d,
                        const int* __restrict__ kept, const int* __restrict__ n_kept,
                        const int* __restrict__ sel_off, const int* __restrict__ ctx_off, int max_ctx,
                        const uint16_t* __restrict__ targets, const float* __restrict__ tinv,
                        const int* __restrict__ rest, MergeCand* __restrict__ cand) {
  constexpr int STAGES = ms::STAGES, COLS = ms::COLS, A_BYTES = ms::A_BYTES, B_BYTES = ms::B_BYTES;
  pdl_trigger();
  pdl_wait();
  const int j = blockIdx.y, mb = blockIdx.x;
  if (j >= *n_kept) return;
  const int co = ctx_off[j], m = ctx_off[j + 1] - co;
  if (m == 0 || co + m > max_ctx) return;  // uniform over the CTA, before any setup (as the next)
  const int R = n_v - (sel_off[j + 1] - sel_off[j]);
  if (mb * 128 >= R) return;
  const int step = R / m;
  extern __shared__ uint8_t smem_raw[];
  __shared__ float nrm_s[128], inv_s[RIFT_MAX_NV];  // the tokens' ||x||^2; the targets' 1 / ||t||
  __shared__ uint16_t twin[RIFT_MAX_NV];            // an earlier target of the same norm, or NONE
  __shared__ int any_twin;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * ms::STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  const uint32_t tfull = bar0 + 8u * (2 * STAGES), tempty = bar0 + 8u * (2 * STAGES + 1);
  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s2 = 0; s2 < STAGES; ++s2) {
      mbar_init(full_bar(s2), 129);  // the gathering threads and the TMA thread
      mbar_init(empty_bar(s2), 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 128);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(ms::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem_base = warp_uniform(*tmem_slot);
  const int kt = d / BK, nblk = (m + COLS - 1) / COLS, n_it = nblk * kt;
  auto width = [&](int nb) { return min(COLS, (m - nb * COLS + ms::BROWS - 1) / ms::BROWS * ms::BROWS); };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA: the target rows
      int it = 0;
      bool ok = true;
      for (int nb = 0; nb < nblk && ok; ++nb) {
        const int w = width(nb);
        for (int k = 0; k < kt; ++k, ++it) {
          const int s2 = it % STAGES;
          if (!mbar_wait(empty_bar(s2), ((it / STAGES) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
          mbar_expect_tx(full_bar(s2), w * BK * 2);
          for (int b = 0; b < w; b += ms::BROWS)
            tma_load_2d(smem_u32(sB + s2 * B_BYTES + b * BK * 2), &tmT, k * BK, co + nb * COLS + b, full_bar(s2));
        }
      }
      for (int q = 1; q <= STAGES && it - q >= 0; ++q) {  // no copy left in flight (bounded)
        const int i2 = it - q;
        for (uint32_t w = 0; w < (1u << 22) && !mbar_try_wait(full_bar(i2 % STAGES), (i2 / STAGES) & 1u); ++w) {
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    int it = 0;
    bool ok = true;
    for (int nb = 0; nb < nblk && ok; ++nb) {
      if (!mbar_wait_warp(tempty, (nb & 1) ^ 1, abort_flag)) break;
      fence_after();
      const uint32_t idesc = ms::IDESC | ((uint32_t)(width(nb) >> 3) << 17);
      for (int k = 0; k < kt; ++k, ++it) {
        const int s2 = it % STAGES;
        if (!mbar_wait_warp(full_bar(s2), (it / STAGES) & 1u, abort_flag)) { ok = false; break; }
        fence_after();
        const uint64_t ad = smem_desc(smem_u32(sA + s2 * A_BYTES));
        const uint64_t bd = smem_desc(smem_u32(sB + s2 * B_BYTES));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            umma_f16(tmem_base, ad + 2 * kk, bd + 2 * kk, idesc, (k != 0 || kk != 0) ? 1u : 0u);
          umma_commit(empty_bar(s2));
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(tfull);
      __syncwarp();
    }
  } else {
    // ---------------- gather and epilogue (warps 2..5)
    // Gather: thread g takes 16-byte chunk g % 8 of rows g / 8 + 16 i (past the last unselected token: that
    // token again), at the chunk's place in the 128-byte swizzle.
    const int g = threadIdx.x - 64, c = g & 7;
    const uint16_t* src[8];
    uint32_t off[8];
    float ss[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int row = (g >> 3) + 16 * i;
      const int tok = rest[(size_t)j * n_v + min(mb * 128 + row, R - 1)];
      src[i] = X + ((size_t)kept[j] * n_v + tok) * d + c * 8;
      off[i] = (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4));
      ss[i] = 0.f;
    }
    // Epilogue: TMEM lane quarters 2, 3, 0, 1; thread = token row
    const int quarter = warp & 3, r = quarter * 32 + lane;
    const int a = mb * 128 + r;
    const bool want = a < R && !(a % step == 0 && a / step < m);
    float v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY, tinv_max = 0.f;
    int b1 = -1, b2 = -1;
    constexpr int LAG = STAGES - 1;  // tiles in flight behind the one being requested
    bool ok = true;
    // tile `it` has landed in this thread's chunks: norms (first pass over the tokens), then hand it over
    auto finish = [&](int it) {
      const uint8_t* tile = sA + (it % STAGES) * A_BYTES;
      if (it < kt) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float x[8];
          unpack_bf16x8(*reinterpret_cast<const uint4*>(tile + off[i]), x);
#pragma unroll
          for (int e = 0; e < 8; ++e) ss[i] = fmaf(x[e], x[e], ss[i]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_arrive(full_bar(it % STAGES));
    };
    for (int nb = 0; nb < nblk && ok; ++nb) {
      // request tiles up to LAG ahead of the end of this pass; hand over those that have landed
      const int it0 = nb == 0 ? 0 : nb * kt + LAG, it1 = min(n_it, (nb + 1) * kt + LAG);
      for (int it = it0; it < it1 || it - LAG < (nb + 1) * kt; ++it) {
        if (it < n_it) {
          if (!__all_sync(0xffffffffu, mbar_wait(empty_bar(it % STAGES), ((it / STAGES) & 1u) ^ 1u, abort_flag))) {
            ok = false;
            break;
          }
          const uint32_t dst = smem_u32(sA + (it % STAGES) * A_BYTES);
          const int k = (it % kt) * BK;
#pragma unroll
          for (int i = 0; i < 8; ++i) cp_async16(dst + off[i], src[i] + k);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (it >= LAG) {
          asm volatile("cp.async.wait_group %0;\n" ::"n"(LAG) : "memory");
          finish(it - LAG);
        }
      }
      if (nb == 0) {  // (also on an abort, so that no warp waits here for another)
        // row norms: the eight threads of a row hold its chunks' sums
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float v = ss[i];
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          v += __shfl_xor_sync(0xffffffffu, v, 4);
          if (c == 0) nrm_s[(g >> 3) + 16 * i] = v;
        }
        // 1 / ||t|| (0 for a zero target: similarity 0); NaN, which is no candidate, for a target whose row is a copy of an
        // earlier one's (blank parts of a tile): a tie never chooses it
        for (int q = g; q < m; q += 128) inv_s[q] = tinv[co + q];
        if (g == 0) any_twin = 0;
        asm volatile("bar.sync 1, 128;\n" ::: "memory");
        for (int q = g; q < m; q += 128) {
          int p = 0;
          while (p < q && inv_s[p] != inv_s[q]) ++p;
          twin[q] = p < q ? (uint16_t)p : MergeCand::NONE;
          if (p < q) any_twin = 1;
        }
        asm volatile("bar.sync 1, 128;\n" ::: "memory");
        if (any_twin) {
          for (int q = quarter; q < m; q += 4) {
            const int p = twin[q];
            if (p != MergeCand::NONE && same_row(targets + (size_t)(co + p) * d, targets + (size_t)(co + q) * d, d, lane) &&
                lane == 0)
              inv_s[q] = __int_as_float(0x7fffffff);
          }
          asm volatile("bar.sync 1, 128;\n" ::: "memory");
        }
      }
      if (!ok) break;
      const int c0 = nb * COLS, nc = min(COLS, m - c0);
      const float* inv_n = inv_s + c0;
      if (!__all_sync(0xffffffffu, mbar_wait(tfull, nb & 1, abort_flag))) { ok = false; break; }
      fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
      for (int cc = 0; cc < nc; cc += 16) {
        uint32_t acc[16];
        tmem_ld16(taddr + cc, acc);
        if (want) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            if (cc + e < nc) {
              // the three highest and the lower indices of the first two (ties keep the lower), without branches: the
              // lanes of a warp hardly ever agree on them; a NaN counts as -inf
              const float ti = inv_n[cc + e], v = fmaxf(__uint_as_float(acc[e]) * ti, -INFINITY);
              const int b = c0 + cc + e;
              tinv_max = fmaxf(tinv_max, ti);
              b2 = v > v1 ? b1 : v > v2 ? b : b2;
              b1 = v > v1 ? b : b1;
              v3 = fmaxf(v3, fminf(v, v2));
              v2 = fmaxf(v2, fminf(v, v1));
              v1 = fmaxf(v1, v);
            }
          }
        }
      }
      if (nb == nblk - 1) {
        // the best, and the targets within the product's error of it
        const float x2 = nrm_s[r];
        const float bound =
            x2 > 0x1p-60f && tinv_max <= 0x1p40f ? (1.25f * (float)d + 8.f) * 0x1p-23f * sqrtf(x2) : INFINITY;
        auto within = [&](float v) { return !(v1 - v > bound); };  // true with a NaN or an infinite norm
        const bool more = want && within(v3);
        MergeCand mc;
        mc.c[0] = (uint16_t)b1;
        mc.c[1] = (uint16_t)(within(v2) ? b2 : -1);
#pragma unroll
        for (int k = 2; k < MergeCand::MAX; ++k) mc.c[k] = MergeCand::NONE;
        mc.all = more ? 1 : 0;
        if (nblk == 1 && __any_sync(0xffffffffu, more)) {  // the products are still there: list the rest
          int n = 1;
          uint64_t lo = mc.c[0] | 0xffffffffffff0000ull, hi = ~0ull;
          for (int cc = 0; cc < nc; cc += 16) {
            uint32_t acc[16];
            tmem_ld16(taddr + cc, acc);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const int b = cc + e;
              if (b < nc && b != b1 && within(fmaxf(__uint_as_float(acc[e]) * inv_n[b], -INFINITY))) {
                const uint64_t keep = ~(0xffffull << (16 * (n & 3))), put = (uint64_t)b << (16 * (n & 3));
                if (n < 4) lo = (lo & keep) | put;
                else if (n < MergeCand::MAX) hi = (hi & keep) | put;
                ++n;
              }
            }
          }
          if (more && n <= MergeCand::MAX) {
#pragma unroll
            for (int k = 0; k < MergeCand::MAX; ++k) mc.c[k] = (uint16_t)((k < 4 ? lo : hi) >> (16 * (k & 3)));
            mc.all = 0;
          }
        }
        if (want) cand[(size_t)j * n_v + a] = mc;
      }
      fence_before();
      mbar_arrive(tempty);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(ms::TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------ host

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 2-D fp16 tensor [rows, inner] (row-major, inner contiguous), box [box_rows, 64], 128B swizzle,
// out-of-bounds elements read as zero.
static bool make_map(CUtensorMap* map, const void* base, uint64_t inner, uint64_t rows, uint32_t box_rows,
                     CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT16) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
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

// L2 band of the tile order (tile_coords): as many tiles of the resident operand as keep its rows
// within kBandBytes of L2 (lo..hi tiles).  The resident operand is the larger one when
// kOrientBands (the smaller one is then streamed once per band), else always A.
constexpr size_t kBandBytes = (size_t)48 << 20;
constexpr bool kOrientBands = true;
static int band_group(int M, int N, int K, int tm, int tn, int lo, int hi) {
  const bool n_major = kOrientBands && (size_t)N < (size_t)M;
  int g = (int)(kBandBytes / ((size_t)(n_major ? tn : tm) * K * 2));
  g = g < lo ? lo : (g > hi ? hi : g);
  return n_major ? -g : g;
}

// The paired kernel (2-CTA clusters), persistent over as many clusters as can be resident at once.
// b, bn: the B map with boxes of half a wide and half a narrow tile.  Returns -1 if no cluster can be
// resident (the caller then takes the cluster split-K kernel).
template <int EPI>
static int launch_pair(const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& bn, int M, int N, int K, void* C,
                       const EpiParams& ep, cudaStream_t st, bool pdl) {
  constexpr size_t smem = (size_t)ring_stages(2) * (A_BYTES + (BN / 2) * BK * 2) + 1024 + 256;
  auto kern = gemm_tc_kernel<EPI, 2>;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // per device: the raised shared-memory limit, and how many 2-CTA clusters fit at once (+1; 0 = not
  // asked yet)
  static std::atomic<unsigned long long> smem_raised{0};
  static std::atomic<int> clusters_plus1[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  int known = (dev >= 0 && dev < 64) ? clusters_plus1[dev].load(std::memory_order_acquire) : 0;
  if (known == 0) {
    int n = 0;
    cfg.gridDim = dim3(2, 1, 1);
    if (raise_smem_limit(smem_raised, kern, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    known = n + 1;
    if (dev >= 0 && dev < 64) clusters_plus1[dev].store(known, std::memory_order_release);
  } else if (raise_smem_limit(smem_raised, kern, (int)smem) != cudaSuccess) {
    return 1;
  }
  const int max_clusters = known - 1;
  if (max_clusters <= 0) return -1;
  const int units = ((M + 2 * BM - 1) / (2 * BM)) * ((N + BN - 1) / BN);
  const int clusters = units < max_clusters ? units : max_clusters;
  const int group_m = band_group(M, N, K, 2 * BM, BN, 4, 32);
  return launch_cluster_ex(kern, dim3(2 * clusters), dim3(THREADS), smem, st, pdl, 2, a, b, bn, M, N, K, C, ep, group_m) ==
                 cudaSuccess
             ? 0
             : 1;
}

// Whether 128 x 256 tiles on one SM each are the faster ones for fewer than 1024 rows: where they take fewer waves than the
// pairs' tiles by more than their waves are slower, a third (a pair shares its B tile).  257 .. 384 rows fill one and a
// half of the pairs' row tiles, 769 .. 896 three and a half.  us, pairs against one SM: 300 rows QKV (2 waves, 1) 49.2 : 45.1,
// gate/up (3, 2) 78.2 : 71.7, 24576 x 8192 (3, 2) 135 : 125; 777 x 5120 x 4096 (2, 1) 45.1 : 38.9; 600 rows of gate/up (4, 3)
// 94.2 : 94.2, which stays with the pairs.
static bool one_sm_tiles(int M, int N, int sms) {
  if (M >= 1024) return false;
  const long long nt = (N + BN - 1) / BN;
  const long long one = ((M + BM - 1) / BM * nt + sms - 1) / sms;
  const long long pair = ((M + 2 * BM - 1) / (2 * BM) * nt + sms / 2 - 1) / (sms / 2);
  return 4 * one < 3 * pair;
}

// One SM a tile, persistent.  b: the B map with boxes of a whole tile.
template <int EPI>
static int launch_single(const CUtensorMap& a, const CUtensorMap& b, int M, int N, int K, void* C, const EpiParams& ep,
                         cudaStream_t st, bool pdl) {
  constexpr size_t smem = (size_t)ring_stages(1) * (A_BYTES + BN * BK * 2) + 1024 + 256;
  static std::atomic<unsigned long long> smem_raised{0};
  if (raise_smem_limit(smem_raised, gemm_tc_kernel<EPI, 1>, (int)smem) != cudaSuccess) return 1;
  const int units = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
  return launch_ex(gemm_tc_kernel<EPI, 1>, dim3(std::min(units, sm_count())), dim3(THREADS), smem, st, pdl, a, b, b, M, N, K, C,
                   ep, band_group(M, N, K, BM, BN, 4, 32)) != cudaSuccess;
}

// Stands for gemm_ck_kernel in the question below: the driver counts a kernel with tcgen05.alloc as one CTA an SM,
// whatever it allocates.
__global__ void __launch_bounds__(ck::THREADS, 2) ck_shape_kernel() {}

// resident[S], S = 1 .. 8: the clusters of S CTAs of the cluster split-K kernel that the current device holds at once
// (asked once per device; 2 SMs / S where the query fails).
static const int* ck_resident() {
  struct Table {
    std::once_flag once;
    int n[ck::PORTABLE_S + 1];
  };
  static Table tables[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  Table& t = tables[dev];
  std::call_once(t.once, [&] {
    const bool raised = cudaFuncSetAttribute(ck_shape_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ck::SMEM) ==
                        cudaSuccess;
    for (int S = 1; S <= ck::PORTABLE_S; ++S) {
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = S;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(S);
      cfg.blockDim = dim3(ck::THREADS);
      cfg.dynamicSmemBytes = ck::SMEM;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (!raised || cudaOccupancyMaxActiveClusters(&n, ck_shape_kernel, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 2 * sm_count() / S;
      }
      t.n[S] = n;
    }
  });
  return t.n;
}

// The cluster split-K kernel: S CTAs per (128 weight rows, bn rows) tile.
template <int EPI, int MAXS>
static int launch_ck_instance(const void* A, const void* W, uint64_t Ks, int M, int N, int K, void* C, const EpiParams& ep,
                     cudaStream_t st, int bn, int S, bool pdl, int w_const) {
  CUtensorMap mw, mx;
  if (!make_map(&mw, W, Ks, (uint64_t)N, BM) || !make_map(&mx, A, Ks, (uint64_t)M, bn)) return 1;
  static std::atomic<unsigned long long> smem_raised{0}, cluster_raised{0};
  if (raise_smem_limit(smem_raised, gemm_ck_kernel<EPI, MAXS>, ck::SMEM) != cudaSuccess ||
      (MAXS > ck::PORTABLE_S && raise_cluster_limit(cluster_raised, gemm_ck_kernel<EPI, MAXS>) != cudaSuccess))
    return 1;
  const int m_tiles = (M + bn - 1) / bn, n_tiles = (N + BM - 1) / BM;
  return launch_cluster_ex(gemm_ck_kernel<EPI, MAXS>, dim3(m_tiles * n_tiles * S), dim3(ck::THREADS), ck::SMEM, st, pdl, S,
                           mw, mx, M, N, K, C, ep, bn, m_tiles, S, w_const) != cudaSuccess;
}

template <int EPI>
static int launch_ck(const void* A, const void* W, uint64_t Ks, int M, int N, int K, void* C, const EpiParams& ep,
                     cudaStream_t st, const ck::Plan& p, bool pdl, int w_const) {
  if (p.S == 1) return launch_ck_instance<EPI, 1>(A, W, Ks, M, N, K, C, ep, st, p.bn, p.S, pdl, w_const);
  if (p.S <= 4) return launch_ck_instance<EPI, 4>(A, W, Ks, M, N, K, C, ep, st, p.bn, p.S, pdl, w_const);
  if constexpr (EPI == EPI_STORE_F32)  // the Gram matrix of few tiles
    if (p.S > ck::PORTABLE_S)
      return launch_ck_instance<EPI, ck::MAX_S>(A, W, Ks, M, N, K, C, ep, st, p.bn, p.S, pdl, w_const);
  return launch_ck_instance<EPI, ck::PORTABLE_S>(A, W, Ks, M, N, K, C, ep, st, p.bn, p.S, pdl, w_const);
}

static int launch_ck_epi(const void* A, const void* W, uint64_t Ks, int M, int N, int K, int epi, void* C,
                         const EpiParams& ep, cudaStream_t st, const ck::Plan& p, bool pdl, int w_const) {
  switch (epi) {
    case EPI_STORE_BF16: return launch_ck<EPI_STORE_BF16>(A, W, Ks, M, N, K, C, ep, st, p, pdl, w_const);
    case EPI_RESID_F32: return launch_ck<EPI_RESID_F32>(A, W, Ks, M, N, K, C, ep, st, p, pdl, w_const);
    case EPI_SWIGLU: return launch_ck<EPI_SWIGLU>(A, W, Ks, M, N, K, C, ep, st, p, pdl, w_const);
    case EPI_QKV_ROPE: return launch_ck<EPI_QKV_ROPE>(A, W, Ks, M, N, K, C, ep, st, p, pdl, w_const);
    case EPI_STORE_F32: return launch_ck<EPI_STORE_F32>(A, W, Ks, M, N, K, C, ep, st, p, pdl, w_const);
    default: return 1;
  }
}

// A wait that can never complete (an mbarrier nobody arrives at), through the same bounded
// mbar_wait as the GEMM's pipeline: it gives up after ~4 s of globaltimer, sets
// RIFT_EBIT_TIMEOUT and returns, leaving the context usable.
__global__ void wait_timeout_check_kernel() {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  abort_flag = 0;
  mbar_init(smem_u32(&bar), 1);
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  mbar_wait(smem_u32(&bar), 0, reinterpret_cast<volatile int*>(&abort_flag));
}

}  // namespace tc

int launch_merge_screen(const uint16_t* X, int N, int n_v, int d, const int* kept, const int* n_kept,
                        const int* sel_off, const int* ctx_off, int max_ctx, const uint16_t* targets,
                        const float* tinv, const int* rest, MergeCand* cand, cudaStream_t st) {
  using namespace tc;
  CUtensorMap mt;
  if (!make_map(&mt, targets, (uint64_t)d, (uint64_t)max_ctx, ms::BROWS, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16)) return 1;
  static std::atomic<unsigned long long> smem_raised{0};
  if (raise_smem_limit(smem_raised, merge_screen_kernel, (int)ms::SMEM) != cudaSuccess) return 1;
  return launch_ex(merge_screen_kernel, dim3((n_v + 127) / 128, N), dim3(ms::THREADS), ms::SMEM, st, true, mt, X, n_v, d,
                   kept, n_kept, sel_off, ctx_off, max_ctx, targets, tinv, rest, cand) != cudaSuccess;
}

int launch_wait_timeout_check(cudaStream_t st) {
  tc::wait_timeout_check_kernel<<<1, 32, 0, st>>>();
  return 0;
}

// Requirements: K % 8 == 0 (16-byte row pitch), N % 8 == 0 (N % 32 == 0 for SwiGLU, N % 64 == 0 for
// the RoPE epilogue), A, B and C 16-byte aligned.
int launch_gemm_tc(const void* A, const void* B, int M, int N, int K, int epi, void* C, const EpiParams& ep,
                   cudaStream_t st, bool pdl, bool b_const) {
  using namespace tc;
  if (M <= 0 || N <= 0 || K <= 0) return 0;
  if (K % 8 != 0 || N % 8 != 0 || (epi == EPI_SWIGLU && N % 32 != 0)) return 1;
  if (epi == EPI_QKV_ROPE && (N % 64 != 0 || (ep.head_dim != 64 && ep.head_dim != 128) || !ep.positions || !ep.rope))
    return 1;
  // The operands' stored row width: K, or 2 kmap_d blocks when read through the K-block remap.
  if (ep.kmap_d && K != 3 * ep.kmap_d * BK) return 1;
  const uint64_t Ks = ep.kmap_d ? (uint64_t)2 * ep.kmap_d * BK : (uint64_t)K;
  const ck::Plan plan = ck::plan(M, N, K, sm_count(), ck_resident(), ep.kmap_d > 0, pdl);
  // The cluster split-K kernel for one row tile, or while its tiles fit on the GPU at once, split or, where K is
  // short, low: beyond that its 128-row tiles are bound by the L2 traffic of their operands and the SM pairs'
  // 256 x 256 tiles win.  us, cluster against pairs: W_o at 512 rows (S = 2) 27.4 : 35.0, at 777
  // (S = 1) 42.0 : 35.4; W_down 53.9 : 63.7 and 78.1 : 65.8; QKV at 131 rows 27.0 : 31.1, at 256
  // (S = 1) 40.8 : 31.1; gate/up 46.8 : 57.8 and 75.6 : 57.8 (wide tiles; the pairs' narrow ones, 14%
  // less, leave the order as it is).
  // A device count of the logits' rows (sequences) is usually a fraction of its capacity, and
  // row tiles past the count cost nothing there.
  if (M <= ck::MAX_BN || plan.one_round || (epi == EPI_STORE_F32 && ep.m_dev && M < 1024))
    return launch_ck_epi(A, B, Ks, M, N, K, epi, C, ep, st, plan, pdl, b_const ? 1 : 0);
  CUtensorMap ma, mb, mn;
  if (!make_map(&ma, A, Ks, (uint64_t)M, BM)) return 1;
  if (!ep.symmetric && one_sm_tiles(M, N, sm_count())) {
    if (!make_map(&mb, B, Ks, (uint64_t)N, BN)) return 1;
    switch (epi) {
      case EPI_STORE_BF16: return launch_single<EPI_STORE_BF16>(ma, mb, M, N, K, C, ep, st, pdl);
      case EPI_RESID_F32: return launch_single<EPI_RESID_F32>(ma, mb, M, N, K, C, ep, st, pdl);
      case EPI_SWIGLU: return launch_single<EPI_SWIGLU>(ma, mb, M, N, K, C, ep, st, pdl);
      case EPI_QKV_ROPE: return launch_single<EPI_QKV_ROPE>(ma, mb, M, N, K, C, ep, st, pdl);
      case EPI_STORE_F32: return launch_single<EPI_STORE_F32>(ma, mb, M, N, K, C, ep, st, pdl);
      default: return 1;
    }
  }
  if (!make_map(&mb, B, Ks, (uint64_t)N, BN / 2) || !make_map(&mn, B, Ks, (uint64_t)N, NARROW_BN / 2)) return 1;
  int r = -1;
  switch (epi) {
    case EPI_STORE_BF16: r = launch_pair<EPI_STORE_BF16>(ma, mb, mn, M, N, K, C, ep, st, pdl); break;
    case EPI_RESID_F32: r = launch_pair<EPI_RESID_F32>(ma, mb, mn, M, N, K, C, ep, st, pdl); break;
    case EPI_SWIGLU: r = launch_pair<EPI_SWIGLU>(ma, mb, mn, M, N, K, C, ep, st, pdl); break;
    case EPI_QKV_ROPE: r = launch_pair<EPI_QKV_ROPE>(ma, mb, mn, M, N, K, C, ep, st, pdl); break;
    case EPI_STORE_F32: r = launch_pair<EPI_STORE_F32>(ma, mb, mn, M, N, K, C, ep, st, pdl); break;
    default: return 1;
  }
  if (r >= 0) return r;
  return launch_ck_epi(A, B, Ks, M, N, K, epi, C, ep, st, plan, pdl, b_const ? 1 : 0);
}

}  // namespace rift
