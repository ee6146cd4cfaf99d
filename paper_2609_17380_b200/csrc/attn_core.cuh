// Pieces the attention forward kernels share: the multiply loop of a warp's 8 query rows against a 16-deep slab, and the online
// softmax of one block of 128 keys (attn.cu says how the work is laid out).
#pragma once
#include "ogemm_core.cuh"

namespace det {

#define ATT_SCALE 0x1.6a09e6p-4f
constexpr int DH = 128;

__device__ __forceinline__ void unpack8a(const uint4& u, float v[8]) {
  v[0] = bflo(u.x); v[1] = bfhi(u.x); v[2] = bflo(u.y); v[3] = bfhi(u.y);
  v[4] = bflo(u.z); v[5] = bfhi(u.z); v[6] = bflo(u.w); v[7] = bfhi(u.w);
}

// conservative test for 0 < |v| < 2^-63 (also true for subnormal v, which only selects the slower exact path)
__device__ __forceinline__ bool tiny1(float v) { return (__float_as_uint(v) * 2u - 1u) < 0x3fffffffu; }
constexpr int FK = 128;
constexpr int AF_RW = 8;                      // query rows per consumer warp
constexpr int AF_PROD = 128;
// A slab row: the first and the second four columns of a lane lie 80 apart (4t and 80 + 4t), so that a warp's loads of
// either half are 256 adjacent bytes and the key-wise stores of K stay free of bank conflicts.
constexpr int AF_HI = 80, AF_BP = 148;

// one 16-deep slab: (row i of the lane, column c) += A[k][row] * B[k][c].  The lane's four rows of step k are chunk
// `chunk` ^ (PSWZ ? swizzle of the key : 0) of row k of A.
template <bool FUSED, bool PSWZ>
__device__ __forceinline__ void mac_4x8(const float* __restrict__ ap, int a_ld, int chunk, int key0,
                                        const float (*Bs)[AF_BP], int tx, float2 (&acc)[4][4]) {
#pragma unroll
  for (int k = 0; k < OK; ++k) {
    const int sw = PSWZ ? (((key0 + k) >> 3) & 3) << 1 : 0;
    const float4 a4 = *reinterpret_cast<const float4*>(ap + (size_t)k * a_ld + ((chunk ^ sw) << 2));
    const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k][4 * tx]), b1 = *reinterpret_cast<const float4*>(&Bs[k][AF_HI + 4 * tx]);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w};
    const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (FUSED) {
          acc[i][j] = __ffma2_rn(make_float2(a[i], a[i]), b[j], acc[i][j]);
        } else {  // scalar on purpose: a packed multiply + add pair would be contracted by ptxas
          acc[i][j].x = fadd(acc[i][j].x, fmul(a[i], b[j].x));
          acc[i][j].y = fadd(acc[i][j].y, fmul(a[i], b[j].y));
        }
      }
  }
}
// Reduction of a lane's four rows over the sixteen lanes that hold them, with partners 2, 4, 8, 16 lanes apart in that
// order, which for sums is the adjacent pairwise tree over the lanes.  The first two stages halve the rows a lane carries (it
// sends its partner the half the partner keeps): 2 + 1 + 1 + 1 shuffles, and lane L ends with the result of row
// ROW_OF_LANE(L) of the warp; both operand orders of an addition or a maximum give the same bits.
#define ROW_OF_LANE(L) ((((L) & 1) << 2) | ((L) & 2) | (((L) & 4) >> 2))
#define LANE_OF_ROW(i) ((lane & 1) | ((i) & 2) | (((i) & 1) << 2))   /* a lane that holds row i of this lane's four */
template <bool SUM>
__device__ __forceinline__ float rows_reduce(const float (&x)[4], int lane) {
  auto op = [](float a, float b) { return SUM ? fadd(a, b) : fmaxf(a, b); };
  const bool b1 = lane & 2, b2 = lane & 4;
  float c[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) c[j] = op(b1 ? x[2 + j] : x[j], __shfl_xor_sync(0xffffffffu, b1 ? x[j] : x[2 + j], 2));
  float d = op(b2 ? c[1] : c[0], __shfl_xor_sync(0xffffffffu, b2 ? c[0] : c[1], 4));
  d = op(d, __shfl_xor_sync(0xffffffffu, d, 8));
  return op(d, __shfl_xor_sync(0xffffffffu, d, 16));
}
// Online softmax of one key block for the warp's 8 rows: acc (the logits of rows `row` .. row + 3 and keys `key` .. key + 7 of this
// lane, without the scale) becomes the weights exp(s - m), invisible pairs +0; the running maximum and the rescale factor of row
// ROW_OF_LANE(lane) of the warp (row `own`) are updated, and the block's row sum is returned.  before(m) gives the maximum up to the
// block before, after(m) takes the one up to this block (the identity and nothing where one warp sees all blocks).  diag: the block reaches past some row; edge: some
// row's window starts inside or after it (last: the block's last key).
template <class Before, class After>
__device__ __forceinline__ float softmax_block(float2 (&acc)[4][4], int key, int row, int own, int last, int W, bool diag, bool edge,
                                               int lane, float& m_mine, float& alpha_mine, float2 one, Before before, After after) {
  float rm[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float mt = __int_as_float(0xff800000);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[i][j] = mul2(acc[i][j], same2(ATT_SCALE));
      if ((!diag || key + 2 * j <= row + i) && (!edge || key + 2 * j > row + i - W)) mt = fmaxf(mt, acc[i][j].x);
      if ((!diag || key + 2 * j + 1 <= row + i) && (!edge || key + 2 * j + 1 > row + i - W)) mt = fmaxf(mt, acc[i][j].y);
    }
    rm[i] = mt;
  }
  // a row sees at least one key of a block it visits, so its maximum is a number; in a block that holds none of its keys its
  // statistics stay untouched
  const float m_block = rows_reduce<false>(rm, lane), m_old = before(m_mine), m_new = fmaxf(m_old, m_block);
  after(m_new);
  alpha_mine = det_exp_le0(fsub(m_old, m_new));
  if (edge && last <= own - W) alpha_mine = 1.0f;
  m_mine = m_new;
#pragma unroll
  for (int i = 0; i < 4; ++i) rm[i] = __shfl_sync(0xffffffffu, m_new, LANE_OF_ROW(i));
  // 32 independent exponentials in one straight-line block (no branch, no shuffle in between), so that their
  // dependent chains interleave; invisible pairs are zeroed afterwards (their arguments may be anything)
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = det_exp_le0_2(add2(acc[i][j], same2(-rm[i]), one), one);
  if (diag) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (key + 2 * j > row + i) acc[i][j].x = 0.0f;
        if (key + 2 * j + 1 > row + i) acc[i][j].y = 0.0f;
      }
  }
  if (edge) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (key + 2 * j <= row + i - W) acc[i][j].x = 0.0f;
        if (key + 2 * j + 1 <= row + i - W) acc[i][j].y = 0.0f;
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)   // the lane's eight adjacent slots of the block's row sum
    rm[i] = fadd(fadd(fadd(acc[i][0].x, acc[i][0].y), fadd(acc[i][1].x, acc[i][1].y)),
                 fadd(fadd(acc[i][2].x, acc[i][2].y), fadd(acc[i][3].x, acc[i][3].y)));
  // the rest of the adjacent tree over the block's 128 slots: lanes 2, 4, 8, 16 apart
  return rows_reduce<true>(rm, lane);
}

}  // namespace det
