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
// The 8 x 16 tiles (FUSED) fetch the next step's operands before they multiply the current one's and keep that order (volatile):
// 301 instead of 306 cycles per step of the 128 x 256 tile; other orders of the 64 multiply-adds (rows outermost, zigzag,
// 2 x 2 blocks) took 302 to 326, and a copy of A with every value doubled, which needs no register pairs to be made, 365.
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
template <int TM, int TN>
__device__ __forceinline__ void slab_mac_ordered(const float (*As)[TM + 4], const float (*Bs)[TN + 4], int ty, int tx, float2 (&acc)[8][8]) {
  float4 a0 = lds128_ordered(&As[0][ty * 4]), a1 = lds128_ordered(&As[0][TM / 2 + ty * 4]), bn[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) bn[g] = lds128_ordered(&Bs[0][g * (TN / 4) + tx * 4]);
#pragma unroll
  for (int k = 0; k < OK; ++k) {
    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    float2 b[8];
#pragma unroll
    for (int g = 0; g < 4; ++g) { b[2 * g] = make_float2(bn[g].x, bn[g].y); b[2 * g + 1] = make_float2(bn[g].z, bn[g].w); }
    if (k + 1 < OK) {
      a0 = lds128_ordered(&As[k + 1][ty * 4]);
      a1 = lds128_ordered(&As[k + 1][TM / 2 + ty * 4]);
#pragma unroll
      for (int g = 0; g < 4; ++g) bn[g] = lds128_ordered(&Bs[k + 1][g * (TN / 4) + tx * 4]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i) ffma2_ordered(av[i], b[j], acc[i][j]);
  }
}
template <bool FUSED, int TM, int TN, int CT>
__device__ __forceinline__ void slab_mac(const float (*As)[TM + 4], const float (*Bs)[TN + 4], int ty, int tx,
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

// One producer thread's share of a slab of ROWS rows x 16 contraction steps, as raw words.  Unit u = thread + 128 i:
//   CONTIG : a 16-byte word (8 bf16 or 4 f32 contraction indices) of row u mod ROWS: consecutive lanes, consecutive rows
//   STRIDED: four consecutive rows 4f .. 4f+3, f = u mod ROWS/4, at one contraction index: consecutive lanes read and store
//            consecutive words, so the shared-memory stores are free of bank conflicts
template <int MODE, bool F32IN, int ROWS>
struct OgRaw {
  static constexpr int UNITS = MODE == CONTIG ? ROWS * (F32IN ? 4 : 2) : 4 * ROWS;
  static constexpr int PER = (UNITS + OG_PROD - 1) / OG_PROD;
  uint4 w[(MODE == STRIDED && !F32IN) ? (PER + 1) / 2 : PER];   // STRIDED bf16: two units share one 16-byte register group
};
template <int MODE, bool F32IN, int ROWS>
__device__ __forceinline__ void og_fetch(const void* base, int rows, int C, int ld, int r0, int c0, int pt,
                                         OgRaw<MODE, F32IN, ROWS>& raw) {
  typedef OgRaw<MODE, F32IN, ROWS> R;
  constexpr int ESZ = F32IN ? 4 : 2;
  const char* b = reinterpret_cast<const char*>(base);
#pragma unroll
  for (int i = 0; i < R::PER; ++i) {
    const int u = pt + OG_PROD * i;
    const bool mine = R::UNITS % OG_PROD == 0 || u < R::UNITS;
    if (MODE == CONTIG) {
      const int r = r0 + u % ROWS, c = c0 + (u / ROWS) * (F32IN ? 4 : 8);
      raw.w[i] = (mine && r < rows && c < C) ? __ldg(reinterpret_cast<const uint4*>(b + ((size_t)r * ld + c) * ESZ))
                                             : make_uint4(0u, 0u, 0u, 0u);
    } else {
      const int r = r0 + 4 * (u % (ROWS / 4)), c = c0 + u / (ROWS / 4);
      const bool ok = mine && r < rows && c < C;
      const char* src = b + ((size_t)c * ld + r) * ESZ;
      if (F32IN) {
        raw.w[i] = ok ? __ldg(reinterpret_cast<const uint4*>(src)) : make_uint4(0u, 0u, 0u, 0u);
      } else {
        const uint2 t = ok ? __ldg(reinterpret_cast<const uint2*>(src)) : make_uint2(0u, 0u);
        if (i & 1) { raw.w[i >> 1].z = t.x; raw.w[i >> 1].w = t.y; }
        else { raw.w[i >> 1].x = t.x; raw.w[i >> 1].y = t.y; }
      }
    }
  }
}
// unpack, test and store one thread's share; returns the below-2^-63 flag of its values
template <int MODE, bool F32IN, int ROWS>
__device__ __forceinline__ bool og_store(float (*s)[ROWS + 4], int pt, const OgRaw<MODE, F32IN, ROWS>& raw) {
  typedef OgRaw<MODE, F32IN, ROWS> R;
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < R::PER; ++i) {
    const int u = pt + OG_PROD * i;
    if (R::UNITS % OG_PROD != 0 && u >= R::UNITS) continue;
    if (MODE == CONTIG) {
      constexpr int EPW = F32IN ? 4 : 8;
      const int r = u % ROWS, k = (u / ROWS) * EPW;
      const uint4 q = raw.w[i];
      const uint32_t p[4] = {F32IN ? word_of(q.x, q.y) : q.x, F32IN ? word_of(q.z, q.w) : q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < EPW / 2; ++e) {
        word_tiny(p[e], m);
        s[k + 2 * e][r] = word_lo(p[e]);
        s[k + 2 * e + 1][r] = word_hi(p[e]);
      }
    } else {
      const int f = u % (ROWS / 4), k = u / (ROWS / 4);
      uint32_t lo, hi;
      if (F32IN) { lo = word_of(raw.w[i].x, raw.w[i].y); hi = word_of(raw.w[i].z, raw.w[i].w); }
      else { lo = (i & 1) ? raw.w[i >> 1].z : raw.w[i >> 1].x; hi = (i & 1) ? raw.w[i >> 1].w : raw.w[i >> 1].y; }
      word_tiny(lo, m);
      word_tiny(hi, m);
      *reinterpret_cast<float4*>(&s[k][4 * f]) = make_float4(word_lo(lo), word_hi(lo), word_lo(hi), word_hi(hi));
    }
  }
  return words_tiny(m);
}

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

// Tile TM x TN, thread tile 8 x CT, LY lanes of a warp along the rows, ST ring slots, PF slabs in flight in the producers'
// registers, CPS CTAs per SM; RC / RP: registers of a consumer / producer thread after the hand-over (0: none).
template <int TM_, int TN_, int CT_, int LY_, int ST_, int PF_, int CPS_, int RC_, int RP_>
struct OgTile {
  static constexpr int TM = TM_, TN = TN_, CT = CT_, LY = LY_, ST = ST_, PF = PF_, CPS = CPS_, RC = RC_, RP = RP_;
  static constexpr int CONS = (TM / 8) * (TN / CT), THREADS = CONS + OG_PROD;
  static constexpr size_t SMEM = (size_t)ST * OK * (TM + 4 + TN + 4) * sizeof(float);
  // what the block is launched with: 65536 registers over CPS blocks, in steps of eight a thread
  static_assert(RC == 0 || CONS * RC + OG_PROD * RP <= (65536 / (CPS * THREADS) / 8 * 8) * THREADS, "register hand-over exceeds the block's allocation");
};
// Measured at 2048 contraction steps on full GPUs (multiply-adds per cycle and SM, 128 is the pipe): 106, 103, 89, 61; one CTA
// on each SM: 311, 174, 110, 71 cycles per step.  Some 30 cycles of every step are not multiply-adds whatever the tile, so
// a smaller tile shortens a chain but never reaches the rate of a larger one.
typedef OgTile<128, 256, 16, 2, 3, 1, 1, 216, 72> OgWide;
typedef OgTile<128, 128, 16, 4, 3, 1, 2, 208, 48> OgSquare;
typedef OgTile<64, 128, 8, 2, 4, 2, 2, 0, 0> OgHalf;
typedef OgTile<32, 64, 4, 2, 6, 4, 4, 0, 0> OgSmall;
typedef OgTile<64, 128, 8, 2, 3, 2, 2, 0, 0> OgFix;          // with 64 KiB of 64-bit accumulators beside the ring
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
// instructions of its own warp.  All waits are bounded.
// FIX: the accumulators of a block of 128 contraction indices are converted (48 fractional bits) and added to 64-bit
// totals after every block.  The totals lie in shared memory, one column per thread (no conflicts): kept in registers they
// forced 128 x 128 tiles of one CTA per SM at 63 multiply-adds per cycle and SM, 72 this way (0.292 -> 0.245 ms at 16 x 4096, window 512).
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, class T, bool FIX>
__global__ void __launch_bounds__(T::THREADS, T::CPS) k_ogemm(const OgemmArgs p) {
  constexpr int TM = T::TM, TN = T::TN, CT = T::CT, ST = T::ST, PF = T::PF;
  extern __shared__ __align__(16) unsigned char osm[];
  float(*As)[OK][TM + 4] = reinterpret_cast<float(*)[OK][TM + 4]>(osm);
  float(*Bs)[OK][TN + 4] = reinterpret_cast<float(*)[OK][TN + 4]>(osm + (size_t)ST * OK * (TM + 4) * sizeof(float));
  __shared__ __align__(16) int tiny_s[ST][4];
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
    const long long hA = zh * p.nG, hB = hA / p.b_div;
    const char* A = reinterpret_cast<const char*>(p.A) + (zb * p.a_b + hA * p.a_h) * (AF32 ? 4 : 2);
    const char* B = reinterpret_cast<const char*>(p.B) + (zb * p.b_b + hB * p.b_h) * 2;
    OgRaw<AMODE, AF32, TM> ra[PF];
    OgRaw<BMODE, false, TN> rb[PF];
    int fetched = 0, c_next = c_lo;
    auto fetch = [&](int d) {
      if (fetched == nslab) return;
      og_fetch<AMODE, AF32, TM>(A, p.I, c_hi, p.lda, i0, c_next, pt, ra[d]);
      og_fetch<BMODE, false, TN>(B, p.J, c_hi, p.ldb, j0, c_next, pt, rb[d]);
      ++fetched;
      c_next += OK;
      if (c_next >= c_hi) {                                          // on to the next head of the group
        c_next = c_lo;
        A += p.a_h * (AF32 ? 4 : 2);
        B += p.b_h * 2;
      }
    };
#pragma unroll
    for (int d = 0; d < PF; ++d) fetch(d);
    int slot = 0;
    uint32_t par = 1;
    for (int s0 = 0; s0 < nslab; s0 += PF) {
#pragma unroll
      for (int d = 0; d < PF; ++d) {
        if (s0 + d >= nslab) return;
        if (!mbar_wait(&bar_empty[slot], par, abort_flag, nullptr)) return;   // the consumers have left this slot
        bool tiny = og_store<AMODE, AF32, TM>(As[slot], pt, ra[d]);
        tiny |= og_store<BMODE, false, TN>(Bs[slot], pt, rb[d]);
        fetch(d);                                                    // these words travel during the handshake
        const int any = __any_sync(0xffffffffu, tiny);
        if (lane == 0) tiny_s[slot][pw] = any;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_full[slot]);                 // slot is full (releases the warp's stores)
        if (++slot == ST) { slot = 0; par ^= 1u; }
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
    const int4 t4 = *reinterpret_cast<const int4*>(tiny_s[slot]);
    if (t4.x | t4.y | t4.z | t4.w) slab_mac<false, TM, TN, CT>(As[slot], Bs[slot], ty, tx, acc);
    else if constexpr (CT == 16) slab_mac_ordered<TM, TN>(As[slot], Bs[slot], ty, tx, acc);
    else slab_mac<true, TM, TN, CT>(As[slot], Bs[slot], ty, tx, acc);
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
constexpr OgRate OG_RATES[4] = {{128, 256, 311.0f, 106.0f}, {128, 128, 174.0f, 103.0f}, {64, 128, 110.0f, 89.0f}, {32, 64, 71.0f, 61.0f}};
// share: how many such contractions run side by side; beside: SM-cycles of other work that is queued to fill the SMs that a small
// grid leaves idle (the head's two gradients at 384 tokens: 96 CTAs of 64 x 128 and the weight gradient on the other SMs,
// head and loss forward and backward 4.34 ms; 384 CTAs of 32 x 64 on all of them and the weight gradient behind, 5.27 ms)
static int og_pick(const OgemmArgs& p, int batches, int share, int widest, double beside) {
  const int sms = dev_sm_count() > 0 ? dev_sm_count() : 1;
  int best = widest;
  double best_t = 0.0;
  for (int c = widest; c < 4; ++c) {
    const OgRate r = OG_RATES[c];
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
// WIDEST: 0, or 1 where the output has no 256 columns (the head dimension of the attention contractions is 128)
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, int WIDEST>
static int ogemm_tile(int tile, const OgemmArgs& p, int batches, cudaStream_t st) {
  switch (tile) {
    case 0: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, typename OgFirst<WIDEST>::T>(p, batches, st);
    case 1: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, OgSquare>(p, batches, st);
    case 2: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, OgHalf>(p, batches, st);
    default: return ogemm_run<AMODE, BMODE, AF32, OUT_BF16, OgSmall>(p, batches, st);
  }
}
template <int AMODE, int BMODE, bool AF32, bool OUT_BF16, int WIDEST>
static int ogemm_launch(const OgemmArgs& p, int batches, int share, cudaStream_t st, double beside = 0.0) {
  return ogemm_tile<AMODE, BMODE, AF32, OUT_BF16, WIDEST>(og_pick(p, batches, share, WIDEST, beside), p, batches, st);
}

}  // namespace det
