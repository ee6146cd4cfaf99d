// The ordered FP32-ALU contractions (LM head, attention backward): C[i,j] = sum over c ascending of A(i,c) B(j,c), one
// sequential accumulator per output.  Operand slabs are staged through shared memory as f32 by producer warps, consumer
// warps hold register tiles of 8 rows and use packed two-lane arithmetic; a per-slab check decides between the
// fused and the two-instruction multiply-add (identical bits, see ogemm.cu).
#pragma once
#include "tc05.cuh"
#include "internal.h"

namespace det {

constexpr int OT = 128;  // tile edge
constexpr int OK = 16;   // slab depth
constexpr int OG_PROD = 128;  // producer threads of a CTA

// Operand access modes.  C[i,j] = sum_c A(i,c) * B(j,c).
//   CONTIG : operand stored [rows, contraction] (contraction index contiguous)
//   STRIDED: operand stored [contraction, rows] (row index contiguous)
enum { CONTIG = 0, STRIDED = 1 };

// One 16-deep slab for this thread's 8 x CT outputs: rows {ty*4 .., TM/2 + ty*4 ..}, columns g * TN*4/CT + tx*4 .. for
// g < CT/4.  FUSED: a*b+acc in one instruction, used only for slabs in which no product can be subnormal (every non-zero
// factor is at least 2^-63 in magnitude), where it gives exactly the bits of the unfused sequence because a product of
// two bf16 values is exact in binary32.  Two accumulators are processed per instruction (packed f32x2 arithmetic, each
// lane rounded on its own).
//
// The 8 x 16 and 8 x 4 tiles (FUSED) fetch the next step's operands before they multiply the current one's and keep that order
// (volatile): 302 instead of 306 cycles per step of the 128 x 256 tile, then (295 now); other orders of the 64 multiply-adds (rows outermost, zigzag,
// 2 x 2 blocks) took 302 to 326, a copy of A with every value doubled 365, and bf16 words in shared memory that the consumers unpack
// 335 to 383.  Counters say why: a packed multiply-add holds the issue port of its scheduler for two cycles, and twice the
// multiply-adds plus everything else comes to 98 % of the cycles, so each further instruction costs its cycle.
__device__ __forceinline__ float4 lds128_ordered(const float* p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(smem_u32(p)));
  return v;
}
__device__ __forceinline__ void ffma2_ordered(float a, float2 b, float2& c) {
  unsigned long long d = f2bits(c);
  asm volatile("fma.rn.ftz.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(f2bits(make_float2(a, a))), "l"(f2bits(b)));
  c = bits2f(d);
}
// CARRY: the last step of a slab fetches the first operands of the next one, n slabs in all; else one slab.  One warp per scheduler
// sees the latency of those loads (128 x 128 tiles alone on their SMs 171 -> 165 cycles per step, 32 x 64 56 -> 52), two hide it for each other
// (128 x 256: 2 % slower), and the 8 x 8 loop is best left to the compiler (64 x 128 alone: 91 -> 99).
template <bool CARRY, int TM, int TN, int CT, int LA, int LB>
__device__ __forceinline__ void slabs_ordered(const float (*As)[LA], const float (*Bs)[LB], int n, int ty, int tx, float2 (&acc)[8][CT / 2]) {
  const float *pa = &As[0][ty * 4], *pb = &Bs[0][tx * 4];
  float4 a0 = lds128_ordered(pa), a1 = lds128_ordered(pa + TM / 2), bn[CT / 4];
#pragma unroll
  for (int g = 0; g < CT / 4; ++g) bn[g] = lds128_ordered(pb + g * (TN * 4 / CT));
#pragma unroll 1
  do {
    const float *qa = CARRY && n > 1 ? pa + OK * LA : pa, *qb = CARRY && n > 1 ? pb + OK * LB : pb;   // after the last slab: its first row again
#pragma unroll
    for (int k = 0; k < OK; ++k) {
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      float2 b[CT / 2];
#pragma unroll
      for (int g = 0; g < CT / 4; ++g) { b[2 * g] = make_float2(bn[g].x, bn[g].y); b[2 * g + 1] = make_float2(bn[g].z, bn[g].w); }
      if (CARRY || k + 1 < OK) {
        const float *na = k + 1 < OK ? pa + (k + 1) * LA : qa, *nb = k + 1 < OK ? pb + (k + 1) * LB : qb;
        a0 = lds128_ordered(na);
        a1 = lds128_ordered(na + TM / 2);
#pragma unroll
        for (int g = 0; g < CT / 4; ++g) bn[g] = lds128_ordered(nb + g * (TN * 4 / CT));
      }
#pragma unroll
      for (int j = 0; j < CT / 2; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) ffma2_ordered(av[i], b[j], acc[i][j]);
    }
    pa = qa;
    pb = qb;
  } while (CARRY && --n > 0);
}
template <bool FUSED, int TM, int TN, int CT, int LA, int LB>
__device__ __forceinline__ void slab_mac(const float (*As)[LA], const float (*Bs)[LB], int ty, int tx,
                                         float2 (&acc)[8][CT / 2]) {
#pragma unroll
  for (int k = 0; k < OK; ++k) {
    const float4 a0 = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
    const float4 a1 = *reinterpret_cast<const float4*>(&As[k][TM / 2 + ty * 4]);
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    float2 b[CT / 2];
#pragma unroll
    for (int g = 0; g < CT / 4; ++g) {
      const float4 bv = *reinterpret_cast<const float4*>(&Bs[k][g * (TN * 4 / CT) + tx * 4]);
      b[2 * g] = make_float2(bv.x, bv.y);
      b[2 * g + 1] = make_float2(bv.z, bv.w);
    }
    // column pairs outermost: each pair of B values meets the eight rows back to back (measured a few percent faster
    // than rows outermost); the order in which different accumulators are visited has no effect on any result
#pragma unroll
    for (int j = 0; j < CT / 2; ++j) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (FUSED) {
          acc[i][j] = __ffma2_rn(make_float2(av[i], av[i]), b[j], acc[i][j]);
        } else {  // scalar on purpose: a packed multiply + add pair would be contracted by ptxas
          acc[i][j].x = fadd(acc[i][j].x, fmul(av[i], b[j].x));
          acc[i][j].y = fadd(acc[i][j].y, fmul(av[i], b[j].y));
        }
      }
    }
  }
}

// ---- staging ------------------------------------------------------------------------------------------------------
// The two halves of a word of bf16 values as f32.
__device__ __forceinline__ float word_lo(uint32_t u) { return __uint_as_float(__byte_perm(u, 0, 0x1044)); }
__device__ __forceinline__ float word_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
// two f32 values rounded to bf16, `lo` in the low half
__device__ __forceinline__ uint32_t word_of(uint32_t lo, uint32_t hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(__uint_as_float(hi)), "f"(__uint_as_float(lo)));
  return r;
}
// Sets bit 15 or 31 of m where a half of u is a non-zero bf16 below 2^-63 (magnitude bits 1 .. 0x1fff; a subnormal counts,
// which only selects the slower exact path): the first sum carries into the top bit of a half unless its magnitude is 0,
// the second where it is at least 0x2000, and neither carries out of its half.
__device__ __forceinline__ void word_tiny(uint32_t u, uint32_t& m) {
  const uint32_t a = u & 0x7fff7fffu;
  m |= (a + 0x7fff7fffu) & ~(a + 0x60006000u);
}
__device__ __forceinline__ bool words_tiny(uint32_t m) { return (m & 0x80008000u) != 0; }

// The same test on two instructions a word: m, which starts at ~0, becomes the smaller of itself and the magnitudes less one, in
// which a zero is the largest.
__device__ __forceinline__ void word_least(uint32_t u, uint32_t& m) { m = __viaddmin_u16x2(u & 0x7fff7fffu, 0xffffffffu, m); }
__device__ __forceinline__ bool least_tiny(uint32_t m) { return (m & 0xffffu) < 0x1fffu || (m >> 16) < 0x1fffu; }

// One producer thread's share of a slab of ROWS rows x 16 contraction steps, as raw words.  Unit u = thread + 128 i:
//   CONTIG : a 16-byte word (8 bf16 or 4 f32 contraction indices) of RPU neighbouring rows: consecutive lanes, consecutive rows.  Two
//            rows where that leaves a unit for every thread: their values go to shared memory as pairs, half the stores
//   STRIDED: four consecutive rows 4f .. 4f+3, f = u mod ROWS/4, at one contraction index: consecutive lanes read and store
//            consecutive words, so the shared-memory stores are free of bank conflicts
// All units of a thread have the same rows, so a pointer (CONTIG: one per row) is all that fetching a slab needs.  Rows past the
// last one repeat it: their results are not stored.
// Every instruction here takes an issue cycle from the consumers of its scheduler (see slabs_ordered).  Running pointers instead of
// addresses and bounds per load, the two-instruction test and the paired stores took the instructions beside the multiply-adds
// from 0.30 to 0.25 per multiply-add (128 x 256 tiles: 2 % faster in the LM head's forward, 2.6 % in the weight gradient).
template <int MODE, bool F32IN, int ROWS>
struct OgSide {
  static constexpr int EPW = F32IN ? 4 : 8, ESZ = F32IN ? 4 : 2;          // CONTIG: contraction indices of a 16-byte word
  static constexpr int RPU = MODE == STRIDED ? 4 : (ROWS * OK / EPW >= 2 * OG_PROD ? 2 : 1);
  static constexpr int LINE = ROWS / RPU;                                 // units of one group of contraction indices
  static constexpr int UNITS = LINE * (MODE == STRIDED ? OK : OK / EPW), PER = (UNITS + OG_PROD - 1) / OG_PROD;
  static constexpr int CSTEP = (OG_PROD / LINE) * (MODE == STRIDED ? 1 : EPW);   // contraction indices from one unit of a thread to the next
  static constexpr int NP = MODE == STRIDED ? 1 : RPU, WORDS = MODE == STRIDED && !F32IN ? 2 : 4;   // pointers; 32-bit words of a load
  static_assert(OG_PROD % LINE == 0 && (UNITS % OG_PROD == 0 || PER == 1), "units of a thread share their rows");
  struct Raw { uint32_t w[PER][NP][WORDS]; };
  const char* ptr[NP];
  int c;                       // contraction index of the thread's first unit, relative to the slab's

  __device__ __forceinline__ bool mine(int pt) const { return UNITS % OG_PROD == 0 || pt < UNITS; }
  __device__ __forceinline__ void init(const void* base, int rows, int ld, int r0, int c0, int pt) {
    c = (pt / LINE) * (MODE == STRIDED ? 1 : EPW);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const int r = min(r0 + RPU * (pt % LINE) + q, rows - (MODE == STRIDED ? 4 : 1));
      ptr[q] = reinterpret_cast<const char*>(base) + (MODE == CONTIG ? (size_t)r * ld + c0 + c : (size_t)(c0 + c) * ld + r) * ESZ;
    }
  }
  // the next slab, of which `left` contraction indices exist; step: bytes from one contraction index to the next (STRIDED)
  __device__ __forceinline__ void fetch(Raw& raw, int left, long long step, int pt) {
    if (!mine(pt)) return;
    const bool full = left >= OK;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        const char* src = MODE == CONTIG ? ptr[q] + i * CSTEP * ESZ : ptr[q];
        uint32_t* w = raw.w[i][q];
        if (full || c + i * CSTEP < left) {
          if (WORDS == 4) {
            const uint4 t = __ldg(reinterpret_cast<const uint4*>(src));
            w[0] = t.x; w[1] = t.y; w[WORDS - 2] = t.z; w[WORDS - 1] = t.w;
          } else {
            const uint2 t = __ldg(reinterpret_cast<const uint2*>(src));
            w[0] = t.x; w[1] = t.y;
          }
        } else {
#pragma unroll
          for (int e = 0; e < WORDS; ++e) w[e] = 0u;
        }
      }
      if (MODE == STRIDED) ptr[0] += CSTEP * step;
    }
    if (MODE == CONTIG) {
#pragma unroll
      for (int q = 0; q < NP; ++q) ptr[q] += OK * ESZ;
    }
  }
  __device__ __forceinline__ void skip(long long bytes) {
#pragma unroll
    for (int q = 0; q < NP; ++q) ptr[q] += bytes;
  }
  // unpack, test and store; m: see word_least
  template <int LD>
  __device__ __forceinline__ void store(float (*s)[LD], const Raw& raw, uint32_t& m, int pt) const {
    if (!mine(pt)) return;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      constexpr int NW = MODE == STRIDED ? 2 : EPW / 2;       // words of bf16 pairs
      uint32_t p[NP][NW];
#pragma unroll
      for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int e = 0; e < NW; ++e) {
          p[q][e] = F32IN ? word_of(raw.w[i][q][2 * e], raw.w[i][q][2 * e + 1]) : raw.w[i][q][e];
          word_least(p[q][e], m);
        }
      const int k = c + i * CSTEP, r = RPU * (pt % LINE);
      if (MODE == STRIDED) {
        *reinterpret_cast<float4*>(&s[k][r]) = make_float4(word_lo(p[0][0]), word_hi(p[0][0]), word_lo(p[0][1]), word_hi(p[0][1]));
      } else {
#pragma unroll
        for (int e = 0; e < NW; ++e) {
          if (RPU == 2) {
            *reinterpret_cast<float2*>(&s[k + 2 * e][r]) = make_float2(word_lo(p[0][e]), word_lo(p[NP - 1][e]));
            *reinterpret_cast<float2*>(&s[k + 2 * e + 1][r]) = make_float2(word_hi(p[0][e]), word_hi(p[NP - 1][e]));
          } else {
            s[k + 2 * e][r] = word_lo(p[0][e]);
            s[k + 2 * e + 1][r] = word_hi(p[0][e]);
          }
        }
      }
    }
  }
};

// f32 -> signed 64-bit fixed point with 48 fractional bits: round to nearest even, saturate, NaN -> 0
__device__ __forceinline__ long long fix48(float u) {
  const float t = fmul(u, 0x1p48f);
  if (t != t) return 0;
  if (t >= 0x1p63f) return 0x7fffffffffffffffll;
  if (t <= -0x1p63f) return (long long)0x8000000000000000ull;
  return __float2ll_rn(t);
}
__device__ __forceinline__ float unfix48(long long a) { return fmul(__ll2float_rn(a), 0x1p-48f); }

// ---- one contraction, batched ---------------------------------------------------------------------------------------
// C[i,j] = sum over c in the row tile's range ascending of A(i,c) B(j,c), one accumulator per output.
struct OgemmArgs {
  const void* A;
  const void* B;
  void* out;
  int I, J, C;          // rows of A, rows of B, contraction length
  int lda, ldb, ldo;    // leading dimensions of the stored operands / output
  int init;             // f32 output only: start from the values already in out
  int H;                // batching: batch index = b * H + h, the output belongs to head h of b
  long long a_b, a_h, b_b, b_h, o_b, o_h;  // element offsets per batch index / head index
  // grouped queries: the accumulator runs over the nG heads h * nG + g of A, g ascending, one after the other; B reads
  // head (h * nG + g) / b_div
  int nG, b_div;
  int window;           // sliding window W (multiple of 128; 0 = none): only |query - key| < W contributes
  int range_mode;       // 0: whole contraction; 1: c >= first row of the tile (causal, per key); 2: c < last row + 1 of the tile
                        // (with a window, mode 1 also stops at c < i0 + W + TM and mode 2 starts at c >= i0 - W)
  int order;            // OG_LEAD: the next launch is OG_FILL; OG_FILL: independent of the launch before, fills the SMs that it leaves;
                        // OG_BACK: a causal grid with its shortest contractions first
};
enum { OG_LEAD = 1, OG_FILL = 2, OG_BACK = 4 };

// Tile TM x TN, thread tile 8 x CT, LY lanes of a warp along the rows, ST ring slots of HS slabs, PF slabs in flight in the producers'
// registers, CPS CTAs per SM; RC / RP: registers of a consumer / producer thread after the hand-over (0: none); PAD: floats behind
// each row of a slab (four instead of none are worth 2 % in every tile; with the 64-bit totals there is no room for them).
// A hand-over costs a consumer some 35 instructions and, with one warp per scheduler, their latency; over HS slabs it is paid once.
// 64 x 128 tiles by slabs per slot, two slots: token gradient of 384 x 8064 x 1024 2: 394, 3: 394, 4: 373 us; weight gradient of 1024 x 4096 x
// 1024 189, 188, 182.  Smaller chains gain most (32 x 64 tiles of one CTA on an SM 22 % from one slab to four, 128 x 128 5 % to three), the
// 128 x 256 tiles nothing.
template <int TM_, int TN_, int CT_, int LY_, int ST_, int PF_, int CPS_, int RC_, int RP_, int HS_, bool CARRY_ = false, int PAD_ = 4>
struct OgTile {
  static constexpr int TM = TM_, TN = TN_, CT = CT_, LY = LY_, ST = ST_, PF = PF_, CPS = CPS_, RC = RC_, RP = RP_, HS = HS_;
  static constexpr int LA = TM + PAD_, LB = TN + PAD_;                    // floats of a slab row
  static constexpr bool CARRY = CARRY_;
  static constexpr int CONS = (TM / 8) * (TN / CT), THREADS = CONS + OG_PROD;
  static constexpr size_t SMEM = (size_t)ST * HS * OK * (LA + LB) * sizeof(float);
  // what the block is launched with: 65536 registers over CPS blocks, in steps of eight a thread
  static_assert(RC == 0 || CONS * RC + OG_PROD * RP <= (65536 / (CPS * THREADS) / 8 * 8) * THREADS, "register hand-over exceeds the block's allocation");
};
// Measured at 1965 MHz: cycles per step of one CTA on each SM, from 2048 and 6144 steps, and multiply-adds per cycle and SM (128 is the pipe) of
// grids of eight full rounds of 2048 steps, start and stores included.  128 x 256, 128 x 128, 64 x 128, 32 x 64 tiles:
//   head forward     290, 161, 100, 53;  111, 109, 89, 59
//   token gradient   295, 158,  86, 54;  109, 106, 97, 67
//   weight gradient  290, 153,  92, 53;  111, 112, 99, 77
// (128 x 128 spills up to 16 bytes a thread, 64 x 128 and 32 x 64 16 to 32, the head forward's 64 x 128 64 stored and 108 loaded.)
// Some 20 to 40 cycles of every step are not multiply-adds whatever the tile, so a smaller tile shortens a chain but never reaches the rate of a
// larger one.
typedef OgTile<128, 256, 16, 2, 2, 1, 1, 216, 72, 2> OgWide;
typedef OgTile<128, 128, 16, 4, 2, 1, 2, 208, 48, 3, true> OgSquare;
typedef OgTile<64, 128, 8, 2, 2, 2, 2, 0, 0, 4> OgHalf;
// Both operands CONTIG: the two halves of a row's 32 bytes of a slab are two producer warps' and meet in the first-level cache, of which two
// rings of four slabs a slot leave 28 KiB beside them, three 92 KiB.  64 x 27184 x 1680 (W comes from memory): 201 us with four, 162 with three;
// 2048 x 8064 x 2048 1355 and 1366; one CTA on each SM, 2048 steps, 112 and 116 (strided operands, read in whole rows, lose 5 % with three).
typedef OgTile<64, 128, 8, 2, 2, 2, 2, 0, 0, 3> OgHalfRows;
typedef OgTile<32, 64, 4, 2, 2, 4, 4, 0, 0, 4, true> OgSmall;
typedef OgTile<64, 128, 8, 2, 2, 1, 2, 0, 0, 2, false, 0> OgFix;       // with 64 KiB of 64-bit accumulators beside the ring
constexpr size_t OG_FIX_BYTES = (size_t)64 * 128 * 8;

// Position of a consumer thread in the tile.  A 16-byte shared-memory load takes two cycles of the port when neighbouring
// lanes read the same word (a half-warp then touches at most 128 bytes) and four when the same words are read by lanes
// eight or sixteen apart, so the column index advances every second lane and the two lanes between differ in the row.
template <class T>
__device__ __forceinline__ void og_lane(int tid, int& ty, int& tx) {
  constexpr int LX = 32 / T::LY, WX = (T::TN / T::CT) / LX;
  const int lane = tid & 31, warp = tid >> 5;
  ty = (warp / WX) * T::LY + (lane & 1) + 2 * (lane / (2 * LX));
  tx = (warp % WX) * LX + (lane >> 1) % LX;
}

// A consumer warp only multiplies; the four producer warps only stage (global loads, unpacking, the below-2^-63 test,
// shared-memory stores) into a ring of slabs.  Each ring slot has a "full" and an "empty" mbarrier: a producer warp arrives on
// "full" after its stores, a consumer warp arrives on "empty" after its last read, and everybody only waits for the
// other side, so consumer warps are not coupled to each other and the multiply pipe never waits for staging
// instructions of its own warp.  All waits are bounded.  A slot is handed over with HS slabs (first slots of 1
// and 2 slabs, so that the multiplications start earlier, gained nothing).
// FIX: the accumulators of a block of 128 contraction indices are converted (48 fractional bits) and added to 64-bit
// totals after every block.  The totals lie in shared memory, one column per thread (no conflicts): kept in registers they
// forced 128 x 128 tiles of one CTA per SM at 63 multiply-adds per cycle and SM, 72 this way (0.292 -> 0.245 ms at 16 x 4096, window 512).
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, class T, bool FIX>
__global__ void __launch_bounds__(T::THREADS, T::CPS) k_ogemm(const OgemmArgs p) {
  constexpr int TM = T::TM, TN = T::TN, LA = T::LA, LB = T::LB, CT = T::CT, ST = T::ST, PF = T::PF, HS = T::HS;
  extern __shared__ __align__(16) unsigned char osm[];
  float(*As)[OK][LA] = reinterpret_cast<float(*)[OK][LA]>(osm);
  float(*Bs)[OK][LB] = reinterpret_cast<float(*)[OK][LB]>(osm + (size_t)ST * HS * OK * LA * sizeof(float));
  __shared__ __align__(4) uint8_t tiny_s[ST][OG_PROD / 32];
  __shared__ __align__(8) uint64_t bar_full[ST], bar_empty[ST];
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  // causal grids: the row tile is the slowest grid index, longest contraction first (OG_BACK: last)
  const bool causal = p.range_mode != 0;
  const bool down = (p.range_mode == 2) != ((p.order & OG_BACK) != 0);
  const int ti = causal ? (down ? (int)(gridDim.z - 1 - blockIdx.z) : (int)blockIdx.z) : (int)blockIdx.y;
  const int zidx = causal ? (int)blockIdx.y : (int)blockIdx.z;
  const int i0 = ti * TM, j0 = blockIdx.x * TN;
  const long long zb = zidx / p.H, zh = zidx % p.H;
  int c_lo = 0, c_hi = p.C;
  if (p.range_mode == 1) { c_lo = i0; if (p.window) c_hi = min(p.C, i0 + p.window + TM); }
  if (p.range_mode == 2) {
    c_hi = min(p.C, i0 + TM);
    if (p.window) c_lo = max(0, i0 - p.window);
    if (FIX) c_lo &= ~127;                                           // a block of 128 starts at a multiple of 128
  }
  const int per_head = (c_hi - c_lo + OK - 1) / OK, nslab = per_head * p.nG;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < ST; ++s) { mbar_init(&bar_full[s], OG_PROD / 32); mbar_init(&bar_empty[s], T::CONS / 32); }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (p.order & OG_LEAD) grid_fill_begin();
  // use n of a slot completes phase n of its barriers: the consumers wait with parity n & 1, the producers, one use
  // behind, with the opposite one
  if (tid >= T::CONS) {
    // ------------------------------- producers -------------------------------
    if (T::RP) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(T::RP ? T::RP : 24));
    const int pt = tid - T::CONS, pw = pt >> 5;
    typedef OgSide<AMODE, AF32, TM> SideA;
    typedef OgSide<BMODE, false, TN> SideB;
    const long long hA = zh * p.nG, hB = hA / p.b_div, stepA = (long long)p.lda * SideA::ESZ, stepB = (long long)p.ldb * SideB::ESZ;
    SideA sa;
    SideB sb;
    sa.init(reinterpret_cast<const char*>(p.A) + (zb * p.a_b + hA * p.a_h) * SideA::ESZ, p.I, p.lda, i0, c_lo, pt);
    sb.init(reinterpret_cast<const char*>(p.B) + (zb * p.b_b + hB * p.b_h) * SideB::ESZ, p.J, p.ldb, j0, c_lo, pt);
    // from behind a head's last slab to the next head's first one
    const long long turnA = p.a_h * SideA::ESZ - (long long)per_head * OK * (AMODE == STRIDED ? stepA : SideA::ESZ);
    const long long turnB = p.b_h * SideB::ESZ - (long long)per_head * OK * (BMODE == STRIDED ? stepB : SideB::ESZ);
    typename SideA::Raw ra[PF];
    typename SideB::Raw rb[PF];
    int fetched = 0, left = c_hi - c_lo;
    auto fetch = [&](int d) {
      if (fetched == nslab) return;
      sa.fetch(ra[d], left, stepA, pt);
      sb.fetch(rb[d], left, stepB, pt);
      ++fetched;
      left -= OK;
      if (left <= 0) {                                               // on to the next head of the group
        left = c_hi - c_lo;
        sa.skip(turnA);
        sb.skip(turnB);
      }
    };
#pragma unroll
    for (int d = 0; d < PF; ++d) fetch(d);
    int slot = 0;
    uint32_t par = 1, least = ~0u;
    for (int s0 = 0; s0 < nslab; s0 += PF) {
#pragma unroll
      for (int d = 0; d < PF; ++d) {
        if (s0 + d >= nslab) return;
        const int sub = (s0 + d) % HS;
        if (sub == 0) {
          if (!mbar_wait(&bar_empty[slot], par, abort_flag, nullptr)) return;   // the consumers have left this slot
          least = ~0u;
        }
        sa.store(As[slot * HS + sub], ra[d], least, pt);
        sb.store(Bs[slot * HS + sub], rb[d], least, pt);
        fetch(d);                                                    // these words travel during the handshake
        if (sub == HS - 1 || s0 + d == nslab - 1) {
          const int any = __any_sync(0xffffffffu, least_tiny(least));
          if (lane == 0) tiny_s[slot][pw] = (uint8_t)any;
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar_full[slot]);               // slot is full (releases the warp's stores)
          if (++slot == ST) { slot = 0; par ^= 1u; }
        }
      }
    }
    return;
  }
  // --------------------------------- consumers ---------------------------------
  if (T::RC) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(T::RC ? T::RC : 24));
  int ty, tx;
  og_lane<T>(tid, ty, tx);
  const int I = p.I, J = p.J, ldo = p.ldo;
  void* out = OUT_BF16 ? (void*)(reinterpret_cast<uint16_t*>(p.out) + zb * p.o_b + zh * p.o_h)
                       : (void*)(reinterpret_cast<float*>(p.out) + zb * p.o_b + zh * p.o_h);
  float2 acc[8][CT / 2];
  unsigned long long* fx = reinterpret_cast<unsigned long long*>(osm + T::SMEM) + tid;   // element e of this thread at fx[e * CONS]
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < CT / 2; ++b) acc[a][b] = make_float2(0.0f, 0.0f);
  if (FIX) {
#pragma unroll
    for (int e = 0; e < 8 * CT; ++e) fx[e * T::CONS] = 0;
  }
  if (!OUT_BF16 && p.init) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int r = i0 + (a >> 2) * (TM / 2) + ty * 4 + (a & 3);
#pragma unroll
      for (int g = 0; g < CT / 4; ++g) {
        const int c = j0 + g * (TN * 4 / CT) + tx * 4;
        if (r < I && c < J) {
          const float4 t = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(out) + (size_t)r * ldo + c);
          acc[a][2 * g] = make_float2(t.x, t.y);
          acc[a][2 * g + 1] = make_float2(t.z, t.w);
        }
      }
    }
  }
  int slot = 0;
  uint32_t par = 0;
  for (int s = 0; s < nslab; ++s) {
    if (!mbar_wait(&bar_full[slot], par, abort_flag, nullptr)) break;   // slot is full; after a wait that ran out the outputs are undefined
    const bool tiny = *reinterpret_cast<const uint32_t*>(tiny_s[slot]) != 0;
    if (T::CARRY && !tiny) {
      const int n = min(HS, nslab - s);
      slabs_ordered<true, TM, TN, CT>(As[slot * HS], Bs[slot * HS], n, ty, tx, acc);
      s += n - 1;
    } else {
#pragma unroll 1
      for (int sub = 0;; ++sub) {
        const int at = slot * HS + sub;
        if (tiny) slab_mac<false, TM, TN, CT>(As[at], Bs[at], ty, tx, acc);
        else if constexpr (CT == 16) slabs_ordered<false, TM, TN, CT>(As[at], Bs[at], 1, ty, tx, acc);
        else slab_mac<true, TM, TN, CT>(As[at], Bs[at], ty, tx, acc);
        if (sub == HS - 1 || s == nslab - 1) break;
        ++s;
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar_empty[slot]);                    // slot may be refilled
    if (++slot == ST) { slot = 0; par ^= 1u; }
    if (FIX && ((s & 7) == 7 || s == nslab - 1)) {
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < CT / 2; ++b) {
          unsigned long long* f = fx + (a * CT + 2 * b) * T::CONS;         // integer additions wrap
          f[0] += (unsigned long long)fix48(acc[a][b].x);
          f[T::CONS] += (unsigned long long)fix48(acc[a][b].y);
          acc[a][b] = make_float2(0.0f, 0.0f);
        }
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int r = i0 + (a >> 2) * (TM / 2) + ty * 4 + (a & 3);
#pragma unroll
    for (int g = 0; g < CT / 4; ++g) {
      const int c = j0 + g * (TN * 4 / CT) + tx * 4;
      if (r < I && c < J) {
        float4 v = make_float4(acc[a][2 * g].x, acc[a][2 * g].y, acc[a][2 * g + 1].x, acc[a][2 * g + 1].y);
        if (FIX) {
          const unsigned long long* f = fx + (a * CT + 4 * g) * T::CONS;
          v = make_float4(unfix48((long long)f[0]), unfix48((long long)f[T::CONS]), unfix48((long long)f[2 * T::CONS]),
                          unfix48((long long)f[3 * T::CONS]));
        }
        if (OUT_BF16) *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(out) + (size_t)r * ldo + c) = make_uint2(pack_bf2(v.x, v.y), pack_bf2(v.z, v.w));
        else *reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + (size_t)r * ldo + c) = v;
      }
    }
  }
  if (p.order & OG_FILL) grid_fill_end();
}

template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, class T, bool FIX = false>
static int ogemm_run(const OgemmArgs& p, int batches, cudaStream_t st) {
  static DevOnce once = {};
  const auto kern = k_ogemm<AMODE, BMODE, AF32, OUT_BF16, T, FIX>;
  constexpr size_t smem = T::SMEM + (FIX ? OG_FIX_BYTES : 0);
  if (dev_ensure_smem(once, (const void*)kern, smem) != DET_OK) return DET_ERR_CUDA;
  const unsigned ni = (unsigned)((p.I + T::TM - 1) / T::TM), nj = (unsigned)((p.J + T::TN - 1) / T::TN);
  const dim3 grid = p.range_mode ? dim3(nj, (unsigned)batches, ni) : dim3(nj, ni, (unsigned)batches);
  if (p.order & OG_FILL) launch_after(kern, grid, T::THREADS, smem, st, p);
  else kern<<<DET_L(grid), T::THREADS, smem, st>>>(p);
  return DET_OK;
}

// Which tile.  Every output is one sequential chain, so a grid with fewer CTAs than SMs, or a causal grid whose longest
// chains run on a few SMs, is bound by the time of one chain, and a smaller tile shortens it: a step of the contraction
// costs a CTA alone on its SM `alone` cycles whatever the other SMs do.  A large grid is bound by the multiply rate,
// which falls with the tile (more operand loads per multiply).  Both are measured figures; the tile with the smaller
// of the larger bounds is taken.
struct OgRate { int tm, tn; float alone, full; };     // cycles per step of a CTA alone on its SM; multiply-adds per cycle and SM of a full one
// Strided operands (the gradients, and attention's contractions with them), of the order of both gradients' figures above: the weight gradient takes a
// tile 2.1 % from its best one in the mean over 264 shapes, with its own figures 2.0 %.
constexpr OgRate OG_RATES[4] = {{128, 256, 302.0f, 108.5f}, {128, 128, 165.0f, 107.0f}, {64, 128, 93.0f, 98.0f}, {32, 64, 56.0f, 76.0f}};
// Both operands CONTIG (the head's forward): staging turns both, which costs the small tiles most.  Within 2 % of the figures above but for the
// last one (its grids seldom fill an SM's four places), these take a tile 0.2 % slower than the best one in the mean over 464 shapes (8 .. 2400 x
// 320 .. 51200 x 128 .. 2560), the figures above 0.5 %, OG_RATES 1.3 % and up to 29 % (640 x 2048 x 2048: 32 x 64 tiles, 217 us, for 128 x 128, 169;
// 304 x 37424 x 1408 754 and 639).
constexpr OgRate OG_ROW_RATES[4] = {{128, 256, 290.0f, 109.0f}, {128, 128, 161.0f, 110.0f}, {64, 128, 100.0f, 90.0f}, {32, 64, 53.0f, 64.0f}};
// share: how many such contractions run side by side; beside: SM-cycles of other work that is queued to fill the SMs that a small
// grid leaves idle (the head's two gradients at 384 tokens: 96 CTAs of 64 x 128 and the weight gradient on the other SMs,
// head and loss forward and backward 4.34 ms; 384 CTAs of 32 x 64 on all of them and the weight gradient behind, 5.27 ms)
static int og_pick(const OgRate (&rates)[4], const OgemmArgs& p, int batches, int share, int widest, double beside) {
  const int sms = dev_sm_count() > 0 ? dev_sm_count() : 1;
  int best = widest;
  double best_t = 0.0;
  for (int c = widest; c < 4; ++c) {
    const OgRate r = rates[c];
    const double ni = (p.I + r.tm - 1) / r.tm, nj = (p.J + r.tn - 1) / r.tn;
    const double tiles = ni * nj * batches;
    double longest, total;           // steps of the contraction: of one tile, and summed over the tiles
    if (p.range_mode == 0) {
      longest = p.C;
      const long long rounds = ((long long)tiles + sms - 1) / sms;
      total = tiles > sms ? (double)rounds * sms * p.C : tiles * p.C;     // tiles of equal length: whole rounds
    } else {
      const double cap = p.window ? p.window + r.tm : p.C;
      longest = p.C < cap ? p.C : cap;
      total = 0.0;
      for (int i = 1; i <= (int)ni; ++i) total += (double)i * r.tm < cap ? (double)i * r.tm : cap;
      total *= nj * batches;
    }
    const double a = longest * p.nG * r.alone, b = share * total * p.nG * r.tm * r.tn / (r.full * sms);
    // the last chains of a causal grid run beside idle SMs: half a chain, on average (three contractions side by side, 16 heads
    // on 4 x 4096: 4.36 ms for the backward with square tiles, 4.07 with half ones; 16 x 16 heads x 2048: 3.43 and 3.56)
    const double full = p.range_mode ? b + 0.5 * a : b, alone = a > full ? a : full;
    // what is queued beside also fills the last round of a grid of several (8192 tokens: 512 tiles of 128 x 256 are 3.5 rounds, and
    // the head's two gradients take 1.4 ms of 55 less than with 128 x 128 tiles of dH)
    const double each = (double)p.C * p.nG * r.tm * r.tn / r.full;
    const double busy = tiles <= sms ? tiles * a : (beside > 0.0 ? tiles * each : alone * sms);
    const double t = (busy + beside) / sms > (beside > 0.0 ? a : alone) ? (busy + beside) / sms : (beside > 0.0 ? a : alone);
    if (c == widest || t < (p.range_mode ? 1.0 : 0.95) * best_t) { best = c; best_t = t; }
  }
  return best;
}
template <int WIDEST> struct OgFirst { typedef OgWide T; };
template <> struct OgFirst<1> { typedef OgSquare T; };
template <int AMODE, int BMODE> struct OgHalfOf { typedef OgHalf T; };
template <> struct OgHalfOf<CONTIG, CONTIG> { typedef OgHalfRows T; };
// WIDEST: 0, or 1 where the output has no 256 columns (the head dimension of the attention contractions is 128)
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, int WIDEST>
static int ogemm_tile(int tile, const OgemmArgs& p, int batches, cudaStream_t st) {
  switch (tile) {
    case 0: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, typename OgFirst<WIDEST>::T>(p, batches, st);
    case 1: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, OgSquare>(p, batches, st);
    case 2: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, typename OgHalfOf<AMODE, BMODE>::T>(p, batches, st);
    default: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, OgSmall>(p, batches, st);
  }
}
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, int WIDEST>
static int ogemm_launch(const OgemmArgs& p, int batches, int share, cudaStream_t st, double beside = 0.0) {
  const OgRate(&rates)[4] = AMODE == CONTIG && BMODE == CONTIG ? OG_ROW_RATES : OG_RATES;
  return ogemm_tile<AMODE, BMODE, AF32, OUT_BF16, WIDEST>(og_pick(rates, p, batches, share, WIDEST, beside), p, batches, st);
}

}  // namespace det
