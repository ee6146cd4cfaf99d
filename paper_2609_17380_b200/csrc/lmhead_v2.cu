// LM head, arithmetic version 2 (optional mode): an order-free, exactly defined contraction on the int8 tensor cores.
//
// Version 1 defines every logit as an ordered chain of binary32 roundings, which only the FP32 ALUs can replay.  Version 2
// uses the paper's own two devices instead (Sec. 3.2: int8 products accumulated exactly in int32; a wide exact integer
// total "for bitwise reproducibility"): every row of H and of W is aligned to its largest exponent and cut into two signed
// 7-bit slices (T = 128 hi + lo, a 14-bit magnitude: values within 2^-6 of the row's largest are kept exactly, smaller
// ones truncated toward zero), the four slice products are exact int32 sums on tcgen05.mma.kind::i8 in whatever order the
// hardware takes them, and the epilogue forms I = 2^14 hh + 2^7 (hl + lh) + ll in 64 bits and rounds I 2^(Ea + Eb - 280)
// to binary32 ONCE.  Nothing about the result depends on tiling, order or hardware.
//
//   k_slice_rows   one warp (or CTA) per row: row exponent (integer maximum), then the two int8 slices
//   k_igemm_sl     persistent, one CTA per SM, 128 x 128 output tile; warp 0 streams the FOUR operand tiles of a 128-deep
//                  step (H hi, H lo, W hi, W lo: 64 KiB) through a three-stage TMA ring, warp 1 issues the sixteen MMAs of
//                  the step into three TMEM accumulators (hh | hl + lh | ll, 128 columns each), sixteen more combine and round.
//                  Clusters of two or four share a tile with a long contraction
//   k_igemm_sl_pair  the same by CTA pairs, 256 x 128 output tile, where a problem takes every step of every tile, its rows
//                  come to whole pairs and the steps are not few
// Every mbarrier wait is bounded (DET_DEV_TIMEOUT), as in igemm.cu.
#include "tc05.cuh"
#include "internal.h"
#include "v2_slice.cuh"

namespace det {

// ---- slicing (bf_bits, slice1: v2_slice.cuh) ------------------------------------------------------------------------------
// eight values of a row as four words of packed bf16 patterns: bf16 source as stored, f32 source rounded to bf16
template <bool F32>
__device__ __forceinline__ void load8_bits(const void* X, size_t idx, uint32_t (&w)[4]) {
  if (F32) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X) + idx));
    const float4 b = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X) + idx) + 1);
    w[0] = bf_bits(a.x) | (bf_bits(a.y) << 16); w[1] = bf_bits(a.z) | (bf_bits(a.w) << 16);
    w[2] = bf_bits(b.x) | (bf_bits(b.y) << 16); w[3] = bf_bits(b.z) | (bf_bits(b.w) << 16);
  } else {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + idx));
    w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
  }
}
// WPR warps per row: one, or the eight of a CTA where a row is long and the rows are few (one warp walks 32768 values twice at
// the latency of its loads: 1024 rows of 32768 f32 values 0.163 ms, 0.059 with eight).
// Neither this kernel nor the sliced contraction lets the next one in before it is complete: with that, logits of 384 tokens x 8064 x 640
// took 39.0 us and 31.4 without (36.9 as plain launches), 1024 tokens 58.2, 52.7 and 53.3; both gradients of 1664 x 512 x 256 80.4 and 65.0.
template <bool F32, int WPR>
__global__ void __launch_bounds__(256) k_slice_rows(const void* __restrict__ X, int R, int K, int8_t* __restrict__ hi,
                                                    int8_t* __restrict__ lo, int32_t* __restrict__ E) {
  grid_wait();
  __shared__ int key_s[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = WPR == 1 ? (int)blockIdx.x * 8 + warp : (int)blockIdx.x;
  if (row >= R) return;
  const int first = WPR == 1 ? lane : (int)threadIdx.x, n8 = K / 8;
  int key = 0;                                       // exponent, bit 30: an infinity or a NaN
#pragma unroll 4
  for (int i = first; i < n8; i += 32 * WPR) {
    uint32_t w[4];
    load8_bits<F32>(X, (size_t)row * K + 8 * (size_t)i, w);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e0 = (w[j] >> 7) & 0xFF, e1 = (w[j] >> 23) & 0xFF, e = max(e0, e1);
      key = max(key, e == 255 ? (255 | (1 << 30)) : e);
    }
  }
  key = __reduce_max_sync(0xffffffffu, key);
  if (WPR > 1) {
    if (lane == 0) key_s[warp] = key;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) key = max(key, key_s[w]);
  }
  if (first == 0) E[row] = key;
  const int e = key & 0xFF;
#pragma unroll 2
  for (int i = first; i < n8; i += 32 * WPR) {
    uint32_t w[4];
    load8_bits<F32>(X, (size_t)row * K + 8 * (size_t)i, w);
    uint32_t h8[2] = {0u, 0u}, l8[2] = {0u, 0u};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t b = (j & 1) ? (w[j >> 1] >> 16) : (w[j >> 1] & 0xFFFFu);
      int h, l;
      slice1(b, e, h, l);
      h8[j >> 2] |= (uint32_t)(uint8_t)(int8_t)h << (8 * (j & 3));
      l8[j >> 2] |= (uint32_t)(uint8_t)(int8_t)l << (8 * (j & 3));
    }
    *reinterpret_cast<uint2*>(hi + (size_t)row * K + 8 * i) = make_uint2(h8[0], h8[1]);
    *reinterpret_cast<uint2*>(lo + (size_t)row * K + 8 * i) = make_uint2(l8[0], l8[1]);
  }
}
template <bool F32>
static void slice_rows_launch(const void* X, int R, int K, int8_t* hi, int8_t* lo, int32_t* E, cudaStream_t st) {
  // eight warps per row once a row holds a few rounds for each of them, unless a warp per row fills the GPU anyway
  if (K >= 4096 && R < 64 * 4 * dev_sm_count()) launch_after(k_slice_rows<F32, 8>, R, 256, 0, st, X, R, K, hi, lo, E);
  else launch_after(k_slice_rows<F32, 1>, (R + 7) / 8, 256, 0, st, X, R, K, hi, lo, E);
}

// Slicing along the OTHER index, for the gradient contractions: the exponent of column c is taken over the rows r, and the
// slices are written transposed ([C, R], so that the contracted index r is contiguous for the tensor core).
//   k_col_exp     E[c] = max over r (integer maximum through atomicMax: order-free); E must be zero before.  A thread takes 16
//                 bytes of a row and every V-th row of the tile
//   k_slice_cols  a CTA takes a 128 x 128 tile, copied into shared memory by 16-byte asynchronous copies: thread = column, 128
//                 rows in registers as packed bytes, out through the same buffer, swizzled, as whole 128-byte lines.
// With a value per lane and load both were bound by the latency of their loads (slices of 32768 x 1024 bf16 0.144 -> 0.044 ms, 1024
// x 1024 0.037 -> 0.008, 1024 x 32768 f32 0.101 -> 0.056).
template <bool F32>
__global__ void __launch_bounds__(128) k_col_exp(const void* __restrict__ X, int R, int C, int32_t* __restrict__ E) {
  constexpr int V = F32 ? 4 : 8, G = 128 / V;          // values per load, threads per row
  __shared__ int red[V][128];
  const int t = threadIdx.x, c0 = blockIdx.x * 128 + grid_dep(), r0 = blockIdx.y * 128;
  const int cg = t % G, rl = t / G;
  int key[V];
#pragma unroll
  for (int j = 0; j < V; ++j) key[j] = 0;
#pragma unroll 8
  for (int i = 0; i < 128 / V; ++i) {
    const size_t idx = (size_t)(r0 + i * V + rl) * C + c0 + cg * V;
    uint32_t b[V];
    if constexpr (F32) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X) + idx));
      b[0] = bf_bits(a.x); b[1] = bf_bits(a.y); b[2] = bf_bits(a.z); b[3] = bf_bits(a.w);
    } else {
      const uint4 u = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + idx));
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) { b[2 * j] = w[j] & 0xFFFFu; b[2 * j + 1] = w[j] >> 16; }
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const int e = (b[j] >> 7) & 0xFF;
      key[j] = max(key[j], e | (e == 255 ? (1 << 30) : 0));
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) red[rl][cg * V + j] = key[j];
  __syncthreads();
  int k = 0;
#pragma unroll
  for (int j = 0; j < V; ++j) k = max(k, red[j][t]);
  if (k > *reinterpret_cast<volatile int32_t*>(E + c0 + t)) atomicMax(E + c0 + t, k);
}
template <bool F32> constexpr size_t SC_SMEM = 128 * 128 * (F32 ? 4 : 2);
template <bool F32>
__global__ void __launch_bounds__(128) k_slice_cols(const void* __restrict__ X, int R, int C, const int32_t* __restrict__ E,
                                                    int8_t* __restrict__ hiT, int8_t* __restrict__ loT) {
  extern __shared__ __align__(16) uint8_t sc_buf[];
  constexpr int SZ = F32 ? 4 : 2, LPR = 128 * SZ / 16;   // bytes per value, copies per row
  const int t = threadIdx.x, c0 = blockIdx.x * 128 + grid_dep(), r0 = blockIdx.y * 128;
  const uint8_t* src = reinterpret_cast<const uint8_t*>(X) + ((size_t)(r0 + t / LPR) * C + c0) * SZ + (t % LPR) * 16;
#pragma unroll
  for (int i = 0; i < LPR; ++i)                          // 128 / LPR rows per step
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sc_buf + (i * 128 + t) * 16)),
                 "l"(src + (size_t)i * (128 / LPR) * C * SZ) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int e = E[c0 + t] & 0xFF;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  uint32_t hw[32], lw[32];
#pragma unroll
  for (int i = 0; i < 128; ++i) {
    const uint32_t b = F32 ? bf_bits(*reinterpret_cast<const float*>(sc_buf + i * 512 + t * 4))
                           : (uint32_t)*reinterpret_cast<const uint16_t*>(sc_buf + i * 256 + t * 2);
    int h, l;
    slice1(b, e, h, l);
    if ((i & 3) == 0) { hw[i >> 2] = 0u; lw[i >> 2] = 0u; }
    hw[i >> 2] |= (uint32_t)(uint8_t)(int8_t)h << (8 * (i & 3));
    lw[i >> 2] |= (uint32_t)(uint8_t)(int8_t)l << (8 * (i & 3));
  }
  __syncthreads();
#pragma unroll
  for (int g = 0; g < 8; ++g) {   // row t of the transposed tiles, sixteen-byte pieces XOR-swizzled by row
    const int off = t * 128 + ((g ^ (t & 7)) << 4);
    *reinterpret_cast<uint4*>(sc_buf + off) = make_uint4(hw[4 * g], hw[4 * g + 1], hw[4 * g + 2], hw[4 * g + 3]);
    *reinterpret_cast<uint4*>(sc_buf + 16384 + off) = make_uint4(lw[4 * g], lw[4 * g + 1], lw[4 * g + 2], lw[4 * g + 3]);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = i * 16 + (t >> 3), ch = t & 7;
    const int off = r * 128 + ((ch ^ (r & 7)) << 4);
    *reinterpret_cast<uint4*>(hiT + (size_t)(c0 + r) * R + r0 + ch * 16) = *reinterpret_cast<const uint4*>(sc_buf + off);
    *reinterpret_cast<uint4*>(loT + (size_t)(c0 + r) * R + r0 + ch * 16) = *reinterpret_cast<const uint4*>(sc_buf + 16384 + off);
  }
}
// exponents (zeroed before) and slices of the columns of X [R, C]
template <bool F32>
static void col_exp_launch(const void* X, int R, int C, int32_t* E, cudaStream_t st) {
  launch_after(k_col_exp<F32>, dim3(C / 128, R / 128), 128, 0, st, X, R, C, E);
}
template <bool F32>
static int slice_cols_launch(const void* X, int R, int C, const int32_t* E, int8_t* hiT, int8_t* loT, cudaStream_t st) {
  static DevOnce once = {};
  if (dev_ensure_smem(once, (const void*)k_slice_cols<F32>, SC_SMEM<F32>) != DET_OK) return DET_ERR_CUDA;
  launch_after(k_slice_cols<F32>, dim3(C / 128, R / 128), 128, SC_SMEM<F32>, st, X, R, C, E, hiT, loT);
  return DET_OK;
}

// ---- sliced contraction -------------------------------------------------------------------------------------------------
constexpr int SL_T = 128;                     // tile edge (rows of H x rows of W)
constexpr int SL_BK = 128;                    // bytes (= int8 elements) per step along K
constexpr int SL_STAGES = 3;
constexpr int SL_TILE = SL_T * SL_BK;         // one operand tile: 16 KiB
constexpr int SL_STAGE_BYTES = 4 * SL_TILE;   // H hi | H lo | W hi | W lo
constexpr int SL_EPI_WARPS = 16;              // warp & 3 = TMEM lane quarter, four warps per quarter take 32 columns each
constexpr int SL_THREADS = 64 + 32 * SL_EPI_WARPS;
constexpr size_t SL_SMEM = (size_t)SL_STAGES * SL_STAGE_BYTES + SL_EPI_WARPS * 2048 + 1024;   // ring + a staging tile per epilogue warp

// the one rounding of the definition: I 2^e as binary32, nearest even; results below 2^-126 after the rounding are zeros.
// The conversion of the integer rounds once (nearest even) and a scaling by 2^e is exact while the result stays a
// normal number, so the exponent is simply added; near the ends of the range the rounding is done in binary64 instead
// (exact product, one conversion), where the subnormal grid decides what reaches 2^-126.
__device__ __forceinline__ float round_scaled(long long I, int e) {
  if (I == 0) return 0.0f;
  const float f = __ll2float_rn(I);
  const int ef = (int)((__float_as_uint(f) >> 23) & 0xFFu) + e;
  if ((unsigned)(ef - 2) <= 252u) return __uint_as_float(__float_as_uint(f) + ((uint32_t)e << 23));
  const double v = (double)I * __longlong_as_double((long long)(e + 1023) << 52);   // exact: |I| < 2^53, e + 1023 in [745, 1253]
  float r = __double2float_rn(v);
  if (fabsf(r) < 0x1p-126f) r = copysignf(0.0f, r);
  return r;
}

// I = 2^14 hh + 2^7 cross + ll
__device__ __forceinline__ long long sl_total(uint32_t hh, uint32_t cr, uint32_t ll) {
  long long t;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(t) : "r"(cr), "r"(128), "l"((long long)(int)ll));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(t) : "r"(hh), "r"(16384));
  return t;
}
// binary32 of I, nearest even, for |I| < 2^44 (fewer than 2^16 terms of at most 16383^2): the bits above the 23 lowest and those 23 are
// integers that adding 1.5 * 2^23 and 2^23 by their bits makes floats, and one fused multiply-add joins the two with the one rounding.
// The whole kernel, polling in its waits included, executed 34.4 warp instructions for 32 results with the conversion of a 64-bit integer and a
// test of its result's range, and 30.9 with this (logits of 16 heads x 2048, 0.122 -> 0.084 ms with the earlier release below).
__device__ __forceinline__ float sl_float(long long I) {
  const float h = fadd(__int_as_float((int)(I >> 23) + 0x4b400000), -12582912.0f);
  const float l = fadd(__uint_as_float(((uint32_t)I & 0x7fffffu) | 0x4b000000u), -8388608.0f);
  return __fmaf_rn(h, 8388608.0f, l);
}
// whether every result of a row against columns with exponents lo .. hi is 0 or a normal number whatever I: 2^e and 2^(e + 44) are, with
// e = ea280 + eb.  The row's exponent comes without the flag of a non-finite row, whose results are all replaced anyway; with the flag of
// a column in hi it is false, and the sum of two flags would overflow.
__device__ __forceinline__ bool sl_plain(int ea280, int lo, int hi) { return ea280 + lo >= -126 && ea280 + hi <= 83; }

// Rounding and stores of one tile, by a warp that owns 32 rows (a lane each) and 32 columns: ready() waits for the tile's MMAs, after
// the exponents have been fetched; totals(c, T) gives the integers of columns c .. c + CH - 1; release() is called by one lane once
// all of them have been read, before the stores, so that the MMAs of the next tile run beside these (8192 x 50304 x 2048: 2.77 -> 2.43
// ms with the shorter rounding).
template <int CH, class Ready, class Totals, class Release>
__device__ __forceinline__ bool sl_tile(const SlArgs& p, int z, int row, int j0, int part, uint8_t* stage, Ready ready, Totals totals,
                                        Release release) {
  const int lane = threadIdx.x & 31;
  const int ea = p.Ea[(size_t)z * p.I + row];
  // the warp's first row: whole row segments leave through the staging tile (tc05.cuh: store_rows32)
  const size_t wbase = (size_t)(z / p.hdiv) * p.o_b + (size_t)(z % p.hdiv) * p.o_h + (size_t)(row - lane) * p.ldo + j0 + part * 32;
  const float rsc = (p.epi == SL_BF16_ROWSCALE) ? p.rowscale[(size_t)z * p.I + row] : 1.0f;
  // the exponents of the warp's 32 columns, one load per tile: lane l keeps column l's, and all of them pass through the
  // staging tile, which is free until the stores
  const int ebv = p.Eb[(size_t)z * p.J + j0 + part * 32 + lane];
  const int any_bad = __any_sync(0xffffffffu, ((ea | ebv) >> 30) != 0);
  const int ea280 = (ea & 0xFF) - 280;
  const bool plain = __all_sync(0xffffffffu, sl_plain(ea280, __reduce_min_sync(0xffffffffu, ebv), __reduce_max_sync(0xffffffffu, ebv)));
  uint32_t* cexp = reinterpret_cast<uint32_t*>(stage);
  __syncwarp();
  cexp[lane] = (uint32_t)ebv << 23;
  __syncwarp();
  if (!__all_sync(0xffffffffu, ready())) return false;
  tc_fence_after();
  float f[32];
#pragma unroll
  for (int c0 = 0; c0 < 32; c0 += CH) {
    long long T[CH];
    totals(c0, T);
    if (plain) {
      const uint32_t re = (uint32_t)(ea280 + 127) << 23;
#pragma unroll
      for (int v = 0; v < CH; v += 4) {
        const uint4 ce = *reinterpret_cast<const uint4*>(cexp + c0 + v);
        const uint32_t e4[4] = {ce.x, ce.y, ce.z, ce.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c0 + v + c] = fmul(sl_float(T[v + c]), __uint_as_float(re + e4[c]));
      }
    } else {
#pragma unroll
      for (int c = 0; c < CH; ++c) f[c0 + c] = round_scaled(T[c], ea280 + (__shfl_sync(0xffffffffu, ebv, c0 + c) & 0xFF));
    }
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) release();
  if (any_bad) {   // a row or a column of the tile holds an infinity or a NaN: its results are NaN
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if ((ea | __shfl_sync(0xffffffffu, ebv, c)) >> 30) f[c] = __int_as_float(0x7FC00000);
  }
  if (p.epi == SL_BF16_ROWSCALE) {
#pragma unroll
    for (int c = 0; c < 32; ++c) f[c] = fmul(f[c], rsc);
  }
#pragma unroll
  for (int c0 = 0; c0 < 32; c0 += 16) {
    const float* g = f + c0;
    if (p.epi != SL_F32) {
      uint4 o[2];
#pragma unroll
      for (int v = 0; v < 2; ++v)
        o[v] = make_uint4(pack_bf2(g[8 * v], g[8 * v + 1]), pack_bf2(g[8 * v + 2], g[8 * v + 3]),
                          pack_bf2(g[8 * v + 4], g[8 * v + 5]), pack_bf2(g[8 * v + 6], g[8 * v + 7]));
      store_rows32<2>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<uint16_t*>(p.out) + wbase + c0), (size_t)p.ldo * 2, o);
    } else {
      uint4 o[4];
#pragma unroll
      for (int v = 0; v < 4; ++v)
        o[v] = make_uint4(__float_as_uint(g[4 * v]), __float_as_uint(g[4 * v + 1]), __float_as_uint(g[4 * v + 2]), __float_as_uint(g[4 * v + 3]));
      store_rows32<4>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<float*>(p.out) + wbase + c0), (size_t)p.ldo * 4, o);
    }
  }
  return true;
}

// One launch covers Z independent problems of the same shape (the operands of problem z are rows z*I.. of A and z*J.. of
// B; the result goes to out + (z / hdiv) * o_b + (z % hdiv) * o_h + i * ldo + j).  causal_tiles: only the tiles with
// j0 <= i0 exist.  krange: 0 the whole contraction; 1 only the steps up to and including the row tile's own (a causal
// product whose contracted index is the key); 2 only the steps from the row tile's own on (contracted index = query).
// epi: SL_F32 | SL_BF16 | SL_BF16_ROWSCALE (the rounded result times rowscale[z*I + i] in binary32, then bf16).
// SPLIT > 1: a cluster of SPLIT CTAs computes ONE tile (krange 0, no causal filter): each takes a part of the steps, and the integers meet in
// shared memory before the one rounding.
template <int SPLIT>
__global__ void __cluster_dims__(SPLIT, 1, 1) __launch_bounds__(SL_THREADS, 1)
    k_igemm_sl(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
               const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl, const SlArgs p, int* status) {
  const int I = p.I, J = p.J, K = p.K;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bar_full[SL_STAGES], bar_empty[SL_STAGES], bar_tfull, bar_tempty;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = SPLIT > 1 ? (int)cluster_ctarank() : 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < SL_STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
    mbar_init(&bar_tfull, 1);
    mbar_init(&bar_tempty, SL_EPI_WARPS);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  grid_wait();
  const int tiles_i = I / SL_T, tiles_j = J / SL_T, per_z = tiles_i * tiles_j, num_tiles = p.Z * per_z, kblocks = K / SL_BK;
  // tile t -> problem z, row tile it, column tile jt (the rows run fastest: the CTAs resident at one time share a tile of
  // B and stream A through L2); false when the tile does not exist; [k_lo, k_hi) = its steps along the contraction
  auto tile_of = [&](int t, int& z, int& i0, int& j0, int& k_lo, int& k_hi) {
    z = t / per_z;
    const int r = t - z * per_z, it = r % tiles_i, jt = r / tiles_i;
    i0 = it * SL_T; j0 = jt * SL_T;
    k_lo = (p.krange == 2) ? it : 0;
    k_hi = (p.krange == 1) ? min(kblocks, it + 1) : kblocks;
    if (SPLIT > 1) { k_lo = kblocks * rank / SPLIT; k_hi = kblocks * (rank + 1) / SPLIT; }
    return !(p.causal_tiles && jt > it);
  };

  const int first_tile = (int)blockIdx.x / SPLIT, next_tile = (int)gridDim.x / SPLIT;
  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = first_tile; tile < num_tiles && ok; tile += next_tile) {
        int z, i0, j0, k_lo, k_hi;
        if (!tile_of(tile, z, i0, j0, k_lo, k_hi)) continue;
        for (int kb = k_lo; kb < k_hi; ++kb) {
          if (!mbar_wait(&bar_empty[stage], phase ^ 1u, abort_flag, status)) { ok = false; break; }
          mbar_expect_tx(&bar_full[stage], SL_STAGE_BYTES);
          uint8_t* sa = smem + stage * SL_STAGE_BYTES;
          tma_load_2d(sa, &tmAh, kb * SL_BK, z * I + i0, &bar_full[stage]);
          tma_load_2d(sa + SL_TILE, &tmAl, kb * SL_BK, z * I + i0, &bar_full[stage]);
          tma_load_2d(sa + 2 * SL_TILE, &tmBh, kb * SL_BK, z * J + j0, &bar_full[stage]);
          tma_load_2d(sa + 3 * SL_TILE, &tmBl, kb * SL_BK, z * J + j0, &bar_full[stage]);
          if (++stage == SL_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // instruction descriptor: D = S32, A = B = signed 8-bit, both K-major, N = 128, M = 128
      constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SL_T >> 3) << 17) | ((uint32_t)(SL_T >> 4) << 24);
      int stage = 0, it = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = first_tile; tile < num_tiles && ok; tile += next_tile) {
        int z, i0, j0, k_lo, k_hi;
        if (!tile_of(tile, z, i0, j0, k_lo, k_hi)) continue;
        if (!mbar_wait(&bar_tempty, ((uint32_t)it & 1u) ^ 1u, abort_flag, status)) { ok = false; break; }   // accumulators drained
        ++it;
        tc_fence_after();
        for (int kb = k_lo; kb < k_hi; ++kb) {
          if (!mbar_wait(&bar_full[stage], phase, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * SL_STAGE_BYTES);
          const uint64_t ah = make_smem_desc(sa), al = make_smem_desc(sa + SL_TILE);
          const uint64_t bh = make_smem_desc(sa + 2 * SL_TILE), bl = make_smem_desc(sa + 3 * SL_TILE);
#pragma unroll
          for (int k4 = 0; k4 < SL_BK / 32; ++k4) {
            const uint64_t o = (uint64_t)(k4 * 2);
            const uint32_t first = (kb != k_lo || k4) ? 1u : 0u;
            umma_i8(tmem_base, ah + o, bh + o, idesc, first);              // hh
            umma_i8(tmem_base + 128u, ah + o, bl + o, idesc, first);       // hl starts the cross accumulator ...
            umma_i8(tmem_base + 128u, al + o, bh + o, idesc, 1u);          // ... lh adds to it
            umma_i8(tmem_base + 256u, al + o, bl + o, idesc, first);       // ll
          }
          umma_commit(&bar_empty[stage]);
          if (++stage == SL_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit(&bar_tfull);
      }
    }
  } else {
    const int q = warp & 3, part = (warp - 2) >> 2;  // TMEM lane quarter this warp may read; its 32 of the 128 columns
    uint8_t* stage = smem + SL_STAGES * SL_STAGE_BYTES + (warp - 2) * 2048;
    int it = 0;
    bool ok = true;
    const uint32_t tcols = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * 32);
    // the totals of 16 of this warp's columns, of this CTA's part of the contraction
    auto totals = [&](int sub, long long (&T)[16]) {
      uint32_t hh[16], cr[16], ll[16];
      tmem_ld16_nowait(tcols + (uint32_t)(sub * 16), hh);
      tmem_ld16_nowait(tcols + 128u + (uint32_t)(sub * 16), cr);
      tmem_ld16_nowait(tcols + 256u + (uint32_t)(sub * 16), ll);
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 16; ++c) T[c] = sl_total(hh[c], cr[c], ll[c]);
    };
    // SPLIT: CTA r of the cluster finishes the columns r * 128 / SPLIT .. and gets the others' totals of them into its ring, which is free once
    // every CTA's MMAs are done: [sender][column of its share][row]
    const int owner = part * SPLIT / 4;
    constexpr int SHARE = SL_T / SPLIT;
    const uint32_t xrow = (uint32_t)((part * 32 - owner * SHARE) * SL_T + q * 32 + lane) * 8u;
    if (SPLIT > 1) {
      ok = __all_sync(0xffffffffu, mbar_wait(&bar_tfull, 0u, abort_flag, status));
      tc_fence_after();
      cluster_sync_all();
      if (ok && owner != rank) {
        const uint32_t dst = mapa_u32(smem_u32(smem), (uint32_t)owner) + (uint32_t)((rank - (rank > owner ? 1 : 0)) * SHARE * SL_T) * 8u + xrow;
#pragma unroll 1
        for (int sub = 0; sub < 2; ++sub) {
          long long T[16];
          totals(sub, T);
#pragma unroll
          for (int c = 0; c < 16; ++c)
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(dst + (uint32_t)((sub * 16 + c) * SL_T) * 8u), "l"(T[c]) : "memory");
        }
      }
      cluster_sync_all();
      ok = ok && owner == rank;
    }
    for (int tile = first_tile; tile < num_tiles && ok; tile += next_tile) {
      int z, i0, j0, k_lo, k_hi;
      if (!tile_of(tile, z, i0, j0, k_lo, k_hi)) continue;
      ok = sl_tile<16>(p, z, i0 + q * 32 + lane, j0, part, stage, [&]() { return mbar_wait(&bar_tfull, (uint32_t)it & 1u, abort_flag, status); },
                       [&](int c0, long long (&T)[16]) {
        totals(c0 / 16, T);
        if (SPLIT > 1) {
#pragma unroll
          for (int src = 0; src < SPLIT - 1; ++src)
#pragma unroll
            for (int c = 0; c < 16; ++c)
              T[c] += *reinterpret_cast<const long long*>(smem + (size_t)(src * SHARE + c0 + c) * SL_T * 8 + xrow);
        }
      }, [&]() { mbar_arrive(&bar_tempty); });
      ++it;
    }
  }
  if (SPLIT > 1 && warp < 2) {   // the two meetings of the cluster, with the epilogue warps
    __syncwarp();
    cluster_sync_all();
    cluster_sync_all();
  }
  __syncthreads();
  if (abort_s) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// CTA pairs (cta_group::2): a pair computes 256 x 128 results.  CTA r stages its own 128 rows of both slices of A and ONE slice of the
// 128 rows of B, the high one in CTA 0, the low one in CTA 1: side by side they are the 256 columns of one MMA, so that A hi times
// both is hh | hl and A lo times both lh | ll, two MMAs of 256 x 256 where a single CTA issues four of 128 x 128.  A CTA reads 48
// instead of 64 KiB per 128-deep step, and what all SMs together read from L2 is what bounds the single CTAs (some 10 TB/s; 8192 x 50304 x
// 2048: 2.43 -> 2.28 ms).  The four accumulators fill TMEM; hl and lh are added in the epilogue.
constexpr int SLP_STAGES = 4, SLP_STAGE_BYTES = 3 * SL_TILE;
static_assert(SLP_STAGES * SLP_STAGE_BYTES == SL_STAGES * SL_STAGE_BYTES, "the pair's ring is as large as the single CTA's");
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(SL_THREADS, 1)
    k_igemm_sl_pair(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                    const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmBl, const SlArgs p, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bar_full[SLP_STAGES], bar_empty[SLP_STAGES], bar_tfull, bar_tempty;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  if (threadIdx.x == 0) {
    for (int s = 0; s < SLP_STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
    mbar_init(&bar_tfull, 1);
    mbar_init(&bar_tempty, 2 * SL_EPI_WARPS);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // the peer's barriers are initialised before anything can signal them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  grid_wait();
  const int tiles_i = p.I / (2 * SL_T), per_z = tiles_i * (p.J / SL_T), num_tiles = p.Z * per_z, kblocks = p.K / SL_BK;
  const int first = (int)blockIdx.x >> 1, step = (int)gridDim.x >> 1;
  auto tile_of = [&](int t, int& z, int& i0, int& j0) {
    z = t / per_z;
    const int r = t - z * per_z;
    i0 = (r % tiles_i) * (2 * SL_T); j0 = (r / tiles_i) * SL_T;
  };
  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      const CUtensorMap* tmB = rank ? &tmBl : &tmBh;
      for (int tile = first; tile < num_tiles && ok; tile += step) {
        int z, i0, j0;
        tile_of(tile, z, i0, j0);
        const int arow = z * p.I + i0 + rank * SL_T, brow = z * p.J + j0;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait(&bar_empty[stage], phase ^ 1u, abort_flag, status)) { ok = false; break; }
          if (rank == 0) mbar_expect_tx(&bar_full[stage], 2 * SLP_STAGE_BYTES);   // both CTAs' tiles complete on this barrier
          uint8_t* sa = smem + stage * SLP_STAGE_BYTES;
          tma_load_2d_pair(sa, &tmAh, kb * SL_BK, arow, &bar_full[stage]);
          tma_load_2d_pair(sa + SL_TILE, &tmAl, kb * SL_BK, arow, &bar_full[stage]);
          tma_load_2d_pair(sa + 2 * SL_TILE, tmB, kb * SL_BK, brow, &bar_full[stage]);
          if (++stage == SLP_STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // instruction descriptor: D = S32, A = B = signed 8-bit, both K-major, N = 256, M = 256 (two CTAs x 128)
      constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      int stage = 0, it = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = first; tile < num_tiles && ok; tile += step, ++it) {
        if (!mbar_wait(&bar_tempty, ((uint32_t)it & 1u) ^ 1u, abort_flag, status)) { ok = false; break; }   // accumulators drained
        tc_fence_after();
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait(&bar_full[stage], phase, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * SLP_STAGE_BYTES);
          const uint64_t ah = make_smem_desc(sa), al = make_smem_desc(sa + SL_TILE), b = make_smem_desc(sa + 2 * SL_TILE);
#pragma unroll
          for (int k4 = 0; k4 < SL_BK / 32; ++k4) {
            const uint64_t o = (uint64_t)(k4 * 2);
            const uint32_t more = (kb || k4) ? 1u : 0u;
            umma_i8_pair(tmem_base, ah + o, b + o, idesc, more);            // hh | hl
            umma_i8_pair(tmem_base + 256u, al + o, b + o, idesc, more);     // lh | ll
          }
          umma_commit_pair(&bar_empty[stage]);
          if (++stage == SLP_STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(&bar_tfull);
      }
    }
  } else {
    const int q = warp & 3, part = (warp - 2) >> 2;  // TMEM lane quarter this warp may read; its 32 of the 128 columns
    uint8_t* stage = smem + SLP_STAGES * SLP_STAGE_BYTES + (warp - 2) * 2048;
    const uint32_t tcols = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * 32), tempty = mapa_u32(smem_u32(&bar_tempty), 0);
    int it = 0;
    for (int tile = first; tile < num_tiles; tile += step, ++it) {
      int z, i0, j0;
      tile_of(tile, z, i0, j0);
      if (!sl_tile<8>(p, z, i0 + rank * SL_T + q * 32 + lane, j0, part, stage, [&]() { return mbar_wait(&bar_tfull, (uint32_t)it & 1u, abort_flag, status); },
                      [&](int c0, long long (&T)[8]) {
        uint32_t hh[8], hl[8], lh[8], ll[8];
        tmem_ld8_nowait(tcols + (uint32_t)c0, hh);
        tmem_ld8_nowait(tcols + 128u + (uint32_t)c0, hl);
        tmem_ld8_nowait(tcols + 256u + (uint32_t)c0, lh);
        tmem_ld8_nowait(tcols + 384u + (uint32_t)c0, ll);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) T[c] = sl_total(hh[c], hl[c] + lh[c], ll[c]);
      }, [&]() { mbar_arrive_remote(tempty); })) break;
    }
  }
  // both CTAs meet before either leaves (the peer may still signal this CTA's barriers or read its tiles)
  __syncthreads();
  if (abort_s) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
  }
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

template <class Kern>
static int sl_go(Kern kern, DevOnce& once, long long ctas, const CUtensorMap& tAh, const CUtensorMap& tAl, const CUtensorMap& tBh,
                 const CUtensorMap& tBl, const SlArgs& p, int* status, cudaStream_t st) {
  if (dev_ensure_smem(once, (const void*)kern, SL_SMEM) != DET_OK) return DET_ERR_CUDA;
  launch_after(kern, (unsigned)ctas, SL_THREADS, SL_SMEM, st, tAh, tAl, tBh, tBl, p, status);
  if (cudaPeekAtLastError() != cudaSuccess) { cudaGetLastError(); return DET_ERR_CUDA; }
  return DET_OK;
}

// host: Z sliced contractions in one launch (see k_igemm_sl); the slices of problem z are rows z*I.. / z*J.. of A / B
int sliced_gemm_launch(const int8_t* Ah, const int8_t* Al, const int8_t* Bh, const int8_t* Bl, const SlArgs& p, int* status,
                       cudaStream_t st) {
  if (p.I % SL_T || p.J % SL_T || p.K % SL_BK || p.Z <= 0 || p.hdiv <= 0) return DET_ERR_SHAPE;
  if (p.K >= (1 << 16)) return DET_ERR_RANGE;   // the cross accumulator holds two products: 2 K 127^2 must stay below 2^31
  CUtensorMap tAh, tAl, tBh, tBl;
  if (!make_map(&tAh, Ah, p.Z * p.I, p.K, SL_T) || !make_map(&tAl, Al, p.Z * p.I, p.K, SL_T) ||
      !make_map(&tBh, Bh, p.Z * p.J, p.K, SL_T) || !make_map(&tBl, Bl, p.Z * p.J, p.K, SL_T))
    return DET_ERR_CUDA;
  static DevOnce once[4] = {};
  const int sms = dev_sm_count(), steps = p.K / SL_BK;
  if (sms <= 0) return DET_ERR_CUDA;
  const long long tiles = (long long)p.Z * (p.I / SL_T) * (p.J / SL_T);
  const bool whole = !p.krange && !p.causal_tiles;      // every tile takes every step
  // Few tiles with a long contraction (a token gradient of 1024 x 1024 has 64 tiles of 256 steps) leave SMs idle: two or four CTAs share a
  // tile.  A part is at least eight steps (the exchange costs about four); clusters of four find room on some seven eighths of the SMs.
  // One, two and four CTAs a tile, us: 2 tiles 16 steps 17.4, 13.9, 12.2, 32 steps 28.4, 19.5, 15.0; 64 tiles 8 steps 12.3, 11.9, 16 17.9,
  // 14.9, 256 186, 106; 36 tiles 16 steps 17.8, 14.4 and, in clusters of four that do not all find room, 23.8; 80 tiles 16 steps 18.6, 27.7.
  if (whole && tiles * 4 <= sms - sms / 8 && steps >= 32) return sl_go(k_igemm_sl<4>, once[0], tiles * 4, tAh, tAl, tBh, tBl, p, status, st);
  if (whole && tiles * 2 <= sms && steps >= 16) return sl_go(k_igemm_sl<2>, once[1], tiles * 2, tAh, tAl, tBh, tBl, p, status, st);
  // Pairs where their tile fits (causal and row-tied problems are written for tiles of 128 rows) and what a step gains has made up for the
  // launch of clusters, some 2 us, and the longer drain of four accumulators: 15 steps in all rounds together, 6 a tile.  Single CTA
  // and pair, us, one round (2048 x 1024 results) 12 steps 15.6 and 16.0, 14 17.2 and 17.1, 15 17.9 and 17.7; two (512 x 8064) 7 steps 19.5 and 19.8,
  // 8 20.9 and 21.0, 10 23.7 and 23.2; four (1024 x 8064) 4 steps 25.9 and 27.1, 6 31.3 and 31.1, 16 65.2 and 58.2; 22 (1024 x 50304)
  // 1 step 120 and 136, 4 157 and 159, 6 175 and 172, 16 390 and 335.
  const long long rounds = (tiles + sms - 1) / sms;
  if (whole && p.I % (2 * SL_T) == 0 && steps >= 6 && rounds * steps >= 15 && sms >= 2) {
    const long long pairs = tiles / 2 < sms / 2 ? tiles / 2 : sms / 2;
    return sl_go(k_igemm_sl_pair, once[2], 2 * pairs, tAh, tAl, tBh, tBl, p, status, st);
  }
  return sl_go(k_igemm_sl<1>, once[3], tiles < sms ? tiles : sms, tAh, tAl, tBh, tBl, p, status, st);
}

}  // namespace det

using namespace det;

// one sliced contraction out[i,j] = round(I 2^(Ea[i] + Eb[j] - 280)) from the slices of both operands ([I,K] and [J,K] int8)
template <bool OUT_BF16>
static int sliced_gemm(const int8_t* Ah, const int8_t* Al, const int8_t* Bh, const int8_t* Bl, const int32_t* Ea, const int32_t* Eb,
                       void* out, int I, int J, int K, int* status, cudaStream_t st) {
  SlArgs p = {};
  p.Ea = Ea; p.Eb = Eb; p.out = out; p.rowscale = nullptr;
  p.I = I; p.J = J; p.K = K; p.Z = 1; p.hdiv = 1; p.o_b = 0; p.o_h = 0; p.ldo = J;
  p.causal_tiles = 0; p.krange = 0; p.epi = OUT_BF16 ? SL_BF16 : SL_F32;
  return sliced_gemm_launch(Ah, Al, Bh, Bl, p, status, st);
}

static size_t v2_layout(int M, int V, int K, size_t* oAh, size_t* oAl, size_t* oBh, size_t* oBl, size_t* oEa, size_t* oEb) {
  size_t off = 0;
  *oAh = off; off += align_up((size_t)M * K, 256);
  *oAl = off; off += align_up((size_t)M * K, 256);
  *oBh = off; off += align_up((size_t)V * K, 256);
  *oBl = off; off += align_up((size_t)V * K, 256);
  *oEa = off; off += align_up((size_t)M * 4, 256);
  *oEb = off; off += align_up((size_t)V * 4, 256);
  return off;
}
extern "C" size_t det_lmhead_fwd_v2_ws_bytes(int M, int V, int K) {
  size_t a, b, c, d, e, f;
  return v2_layout(M, V, K, &a, &b, &c, &d, &e, &f);
}
extern "C" int det_lmhead_fwd_v2(const det_bf16* H, const det_bf16* W, int M, int V, int K, float* logits, void* ws,
                                 size_t ws_bytes, void* stream, int* status_dev) {
  if (!H || !W || !logits || M <= 0 || V <= 0 || K <= 0) return DET_ERR_ARG;
  if (M % SL_T || V % SL_T || K % SL_BK) return DET_ERR_SHAPE;
  if (K >= (1 << 16)) return DET_ERR_RANGE;   // the cross accumulator holds two products: 2 K 127^2 must stay below 2^31
  if (!aligned16(H) || !aligned16(W) || !aligned16(logits) || !aligned16(ws)) return DET_ERR_ALIGN;
  size_t oAh, oAl, oBh, oBl, oEa, oEb;
  if (!ws || ws_bytes < v2_layout(M, V, K, &oAh, &oAl, &oBh, &oBl, &oEa, &oEb)) return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  uint8_t* base = (uint8_t*)ws;
  int8_t *Ah = (int8_t*)(base + oAh), *Al = (int8_t*)(base + oAl), *Bh = (int8_t*)(base + oBh), *Bl = (int8_t*)(base + oBl);
  int32_t *Ea = (int32_t*)(base + oEa), *Eb = (int32_t*)(base + oEb);
  slice_rows_launch<false>(H, M, K, Ah, Al, Ea, st);
  slice_rows_launch<false>(W, V, K, Bh, Bl, Eb, st);
  DET_CHECK_LAUNCH();
  return sliced_gemm<false>(Ah, Al, Bh, Bl, Ea, Eb, logits, M, V, K, status_dev, st);
}

// ---- gradients (version 2): the same contraction on transposed operands -------------------------------------------------
static size_t v2b_layout(int M, int V, int K, size_t (&o)[12]) {
  size_t off = 0;
  const size_t sz[12] = {(size_t)M * V, (size_t)M * V,      // g = bf16(dlogits), rows (exponent per token): hi, lo [M,V]
                         (size_t)M * V, (size_t)M * V,      // g columns, transposed (exponent per vocabulary entry): hi, lo [V,M]
                         (size_t)V * K, (size_t)V * K,      // W columns, transposed: hi, lo [K,V]
                         (size_t)M * K, (size_t)M * K,      // H columns, transposed: hi, lo [K,M]
                         (size_t)M * 4, (size_t)V * 4, (size_t)K * 4, (size_t)K * 4};   // exponents: g rows, g columns, W columns, H columns
  for (int i = 0; i < 12; ++i) { o[i] = off; off += align_up(sz[i], 256); }
  return off;
}
extern "C" size_t det_lmhead_bwd_v2_ws_bytes(int M, int V, int K) {
  size_t o[12];
  return v2b_layout(M, V, K, o);
}
extern "C" int det_lmhead_bwd_v2(const float* dlogits, const det_bf16* H, const det_bf16* W, int M, int V, int K, det_bf16* dH,
                                 float* dW, void* ws, size_t ws_bytes, void* stream, int* status_dev) {
  if (!dlogits || !H || !W || !dH || !dW || M <= 0 || V <= 0 || K <= 0) return DET_ERR_ARG;
  if (M % SL_T || V % SL_T || K % SL_BK) return DET_ERR_SHAPE;
  if (M >= (1 << 16) || V >= (1 << 16)) return DET_ERR_RANGE;   // contraction lengths of the two gradients
  if (!aligned16(dlogits) || !aligned16(H) || !aligned16(W) || !aligned16(dH) || !aligned16(dW) || !aligned16(ws)) return DET_ERR_ALIGN;
  size_t o[12];
  if (!ws || ws_bytes < v2b_layout(M, V, K, o)) return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  uint8_t* b = (uint8_t*)ws;
  int8_t *gh = (int8_t*)(b + o[0]), *gl = (int8_t*)(b + o[1]), *gTh = (int8_t*)(b + o[2]), *gTl = (int8_t*)(b + o[3]);
  int8_t *WTh = (int8_t*)(b + o[4]), *WTl = (int8_t*)(b + o[5]), *HTh = (int8_t*)(b + o[6]), *HTl = (int8_t*)(b + o[7]);
  int32_t *Eg = (int32_t*)(b + o[8]), *EgT = (int32_t*)(b + o[9]), *EWT = (int32_t*)(b + o[10]), *EHT = (int32_t*)(b + o[11]);
  cudaMemsetAsync(EgT, 0, o[11] - o[9] + align_up((size_t)K * 4, 256), st);        // the three column-exponent arrays
  slice_rows_launch<true>(dlogits, M, V, gh, gl, Eg, st);
  col_exp_launch<true>(dlogits, M, V, EgT, st);
  col_exp_launch<false>(W, V, K, EWT, st);
  col_exp_launch<false>(H, M, K, EHT, st);
  if (slice_cols_launch<true>(dlogits, M, V, EgT, gTh, gTl, st) != DET_OK || slice_cols_launch<false>(W, V, K, EWT, WTh, WTl, st) != DET_OK ||
      slice_cols_launch<false>(H, M, K, EHT, HTh, HTl, st) != DET_OK)
    return DET_ERR_CUDA;
  DET_CHECK_LAUNCH();
  // dH[m,k] = bf16(contraction over the vocabulary of row m of g with column k of W)
  int rc = sliced_gemm<true>(gh, gl, WTh, WTl, Eg, EWT, dH, M, K, V, status_dev, st);
  if (rc != DET_OK) return rc;
  // dW[v,k] = contraction over the tokens of column v of g with column k of H
  return sliced_gemm<false>(gTh, gTl, HTh, HTl, EgT, EHT, dW, V, K, M, status_dev, st);
}
