// RMSNorm forward/backward and cross-entropy (+ z-loss) forward/backward: HBM-bound kernels whose
// reductions are the fixed pairwise tree with 256-element leaves (a lane owns 8 adjacent elements,
// a warp owns a leaf).
#include "common.cuh"
#include "internal.h"

namespace det {

template <bool BF>
__device__ __forceinline__ void load8(const void* p, size_t idx, float v[8]) {
  if (BF) {
    uint4 u = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(p) + idx);
    v[0] = bflo(u.x); v[1] = bfhi(u.x); v[2] = bflo(u.y); v[3] = bfhi(u.y);
    v[4] = bflo(u.z); v[5] = bfhi(u.z); v[6] = bflo(u.w); v[7] = bfhi(u.w);
  } else {
    const float4* q = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + idx);
    float4 a = q[0], b = q[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
}
template <bool BF>
__device__ __forceinline__ void store8(void* p, size_t idx, const float v[8]) {
  if (BF) {
    uint4 u;
    u.x = pack_bf2(v[0], v[1]); u.y = pack_bf2(v[2], v[3]); u.z = pack_bf2(v[4], v[5]); u.w = pack_bf2(v[6], v[7]);
    *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(p) + idx) = u;
  } else {
    float4* q = reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + idx);
    q[0] = make_float4(v[0], v[1], v[2], v[3]);
    q[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// ------------------------------------------------------------------------------------------------
// RMSNorm.  Rows of at most 2048 elements (8 leaves) are held in registers between the sum of squares and
// the output (k_rmsnorm_fwd8); longer rows use the two-pass variant that reads the row again.
// ------------------------------------------------------------------------------------------------
// A warp per LEAF (256 columns, 8 adjacent columns per lane), a CTA of 8 warps per block of 8 rows in two passes of four
// rows: 16 values and 8 loads in flight per lane, four CTAs per SM; the leaf sums of a row meet in shared memory (one
// barrier per pass) and every thread forms the row's tree over its leaves itself.  Rows of at most 1024 columns need only some of
// the warps: the eight rows are then dealt out to 2, 4 or 8 groups of warps and take one pass (cold, 128 rows of 256: 10.3 -> 4.1 us;
// 1664 of 1024: 12.6 -> 8.9).
// WPR warps per row; RowGroups: groups per CTA, rows per group and pass.
template <int WPR>
struct RowGroups { static constexpr int GROUPS = 8 / WPR, ROWS = WPR < 4 ? WPR : 4; };
template <bool BF, int WPR>
__global__ void __launch_bounds__(256, 4) k_rmsnorm_fwd8(const void* __restrict__ x, const void* __restrict__ gamma, int rows,
                                                         int D, float eps, float invD, void* __restrict__ y,
                                                         float* __restrict__ rstd, const float* __restrict__ s_q = nullptr,
                                                         int8_t* __restrict__ qy = nullptr, const void* __restrict__ res = nullptr,
                                                         void* __restrict__ sum = nullptr) {
  grid_dep();
  __shared__ float leaf_sum[8][8];
  constexpr int ROWS = RowGroups<WPR>::ROWS, STEP = RowGroups<WPR>::GROUPS * ROWS;
  const int grp = (threadIdx.x >> 5) / WPR, warp = (threadIdx.x >> 5) % WPR, lane = threadIdx.x & 31;
  const int e0 = warp * 256 + lane * 8;
  const bool have = e0 < D;
  const bool full = (D & 255) == 0;
  const long long r0 = (long long)blockIdx.x * 8;
  const float inv_q = (BF && qy) ? fdiv(1.0f, s_q[0]) : 0.0f;
#pragma unroll 1
  for (int first = grp * ROWS; first < 8; first += STEP) {   // this group's rows of the pass
    float xr[ROWS][8];
#pragma unroll
    for (int a = 0; a < ROWS; ++a) {
      const long long row = r0 + first + a;
      if (row < rows && have) load8<BF>(x, (size_t)row * D + e0, xr[a]);
      else {
#pragma unroll
        for (int t = 0; t < 8; ++t) xr[a][t] = 0.0f;
      }
    }
    if (BF && res) {   // the residual sum in front of the norm: x + res, rounded and stored, is what is normalised
#pragma unroll
      for (int a = 0; a < ROWS; ++a) {
        const long long row = r0 + first + a;
        if (row >= rows || !have) continue;
        float b[8];
        load8<BF>(res, (size_t)row * D + e0, b);
#pragma unroll
        for (int t = 0; t < 8; ++t) xr[a][t] = fadd(xr[a][t], b[t]);
        store8<BF>(sum, (size_t)row * D + e0, xr[a]);
#pragma unroll
        for (int t = 0; t < 8; ++t) xr[a][t] = bf2f(f2bf(xr[a][t]));
      }
    }
#pragma unroll
    for (int a = 0; a < ROWS; ++a) {
      float sq[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) sq[t] = fmul(xr[a][t], xr[a][t]);
      const float t8 = tree8_full(sq);
      const float leaf = full ? warp_tree_full(t8) : warp_tree(t8, (long long)warp * 256, 8, D);
      if (lane == 0) leaf_sum[first + a][warp] = leaf;
    }
    __syncthreads();
    float g[8];
    if (gamma && have) load8<BF>(gamma, e0, g);
#pragma unroll
    for (int a = 0; a < ROWS; ++a) {
      const long long row = r0 + first + a;
      float L[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) L[j] = leaf_sum[first + a][j];
      const float ss = reg_tree<8>(L, 0, 256, D);          // a leaf beyond D does not exist
      const float rs = fdiv(1.0f, fsqrt(fadd(fmul(ss, invD), eps)));
      if (row >= rows) continue;
      if (warp == 0 && lane == a) rstd[row] = rs;
      if (!have) continue;
      float o[8];
      if (gamma) {
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = fmul(fmul(xr[a][t], rs), g[t]);
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = fmul(xr[a][t], rs);
      }
      store8<BF>(y, (size_t)row * D + e0, o);
      if (BF && qy) {   // the next linear's quantiser, applied to the bf16 values just stored
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = bf2f(f2bf(o[t]));
        *reinterpret_cast<uint2*>(qy + (size_t)row * D + e0) = quant8(o, inv_q);
      }
    }
  }
}

// Backward for rows of at most 2048 elements.  A CTA of 8 warps takes a block of 8 adjacent rows in four passes of two
// rows; warp j holds columns 256 j .. 256 j + 255 (one leaf of the fixed tree) of both rows, 8 adjacent columns per lane;
// three CTAs per SM, so that one loads or stores while another stands at its barrier (one CTA of 8 rows x 4 warps per SM
// ran 20 % slower).  A lane sees the same 8 columns of all 8 rows of the block, one pair of rows after the other, so with
// DG the column tree over the 8 rows of dy*xhat (the first three levels of the gain gradient's row-direction tree,
// written to partial8[block][D]) runs in its registers: no shared-memory copy of the products and no barrier of its own
// (0.080 ms with the products staged through shared memory by warps that each owned a quarter row, 0.070 ms now;
// 0.065-0.070 ms without the gain gradient, i.e. 0.9 of the copy bandwidth).  The row sums go through shared memory: one
// value per leaf and row, one barrier per pass.
// RPP rows per pass: 2 for f32 rows, 4 for bf16 rows (16 values and 64 bytes of loads in flight per lane and tensor either way).
// bf16 rows of at most 1024 columns: groups of warps as in the forward kernel, one pass; the groups' nodes of the column tree meet in
// shared memory (cold, 128 rows of 256: 13.3 -> 4.1 us; 1024 of 1024: 14.3 -> 8.7).
template <bool BF, bool DG, int WPR>
__global__ void __launch_bounds__(256, 3) k_rmsnorm_bwd8(const void* __restrict__ dy, const void* __restrict__ x,
                                                        const void* __restrict__ gamma, const float* __restrict__ rstd,
                                                        int rows, int D, float invD, void* dx, const void* res,
                                                        float* __restrict__ partial8, int* __restrict__ tickets) {
  grid_dep();
  static_assert(BF || WPR == 8, "f32 rows take the passes one after the other");
  constexpr int RPP = BF ? RowGroups<WPR>::ROWS : 2, GROUPS = RowGroups<WPR>::GROUPS;
  __shared__ float leaf_sum[8][8];
  __shared__ __align__(16) float nodes[DG && GROUPS > 1 ? 8 : 1][32][8];
  const int grp = (threadIdx.x >> 5) / WPR, warp = (threadIdx.x >> 5) % WPR, lane = threadIdx.x & 31;
  const int e0 = warp * 256 + lane * 8;
  const bool have = e0 < D;                       // this lane's 8 columns exist (D is a multiple of 8)
  const bool full = (D & 255) == 0;
  const long long r0 = (long long)blockIdx.x * 8;
  if (DG && blockIdx.x == 0 && (int)threadIdx.x < ((D + 255) >> 8)) tickets[threadIdx.x] = 0;   // for the kernel that follows
  float pair0[8], node[8];                        // column tree: a pair of rows waiting for the next pair; rows 0 .. 3
#pragma unroll
  for (int t = 0; t < 8; ++t) { pair0[t] = 0.0f; node[t] = 0.0f; }
#pragma unroll 1
  for (int pass = 0, f = grp * RPP; f < 8; f += GROUPS * RPP, ++pass) {
    const long long first = r0 + f;
    float w[RPP][8], xh[RPP][8], rs[RPP];
#pragma unroll
    for (int a = 0; a < RPP; ++a) {
      const long long row = first + a;
      if (row < rows && have) {
        load8<BF>(dy, (size_t)row * D + e0, w[a]);
        load8<BF>(x, (size_t)row * D + e0, xh[a]);
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) { w[a][t] = 0.0f; xh[a][t] = 0.0f; }
      }
      rs[a] = row < rows ? rstd[row] : 0.0f;
    }
#pragma unroll
    for (int a = 0; a < RPP; ++a)
#pragma unroll
      for (int t = 0; t < 8; ++t) xh[a][t] = fmul(xh[a][t], rs[a]);
    if (DG) {   // rows in pairs; pairs 0, 1 and 2, 3 -> nodes of four rows; those two -> the node of eight (a right node exists
                // iff its first row does, else the left one is carried up unchanged)
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const float d0 = fmul(w[0][t], xh[0][t]);
        float pa = d0;
        if (RPP > 1) pa = (first + 1 < rows) ? fadd(d0, fmul(w[RPP > 1][t], xh[RPP > 1][t])) : d0;
        if (BF) {
          float four = pa;
          if (RPP == 4) {
            const float d2 = fmul(w[RPP / 2][t], xh[RPP / 2][t]), d3 = fmul(w[RPP - 1][t], xh[RPP - 1][t]);
            const float pb = (first + 3 < rows) ? fadd(d2, d3) : d2;
            four = (first + 2 < rows) ? fadd(pa, pb) : pa;
          }
          node[t] = (pass == 0) ? four : ((r0 + 4 < rows) ? fadd(node[t], four) : node[t]);
        } else if ((pass & 1) == 0) {
          pair0[t] = pa;
        } else {
          const float four = (first < rows) ? fadd(pair0[t], pa) : pair0[t];
          node[t] = (pass == 1) ? four : ((r0 + 4 < rows) ? fadd(node[t], four) : node[t]);
        }
      }
      if (GROUPS > 1) {
        float4* mine = reinterpret_cast<float4*>(nodes[threadIdx.x >> 5][lane]);
        mine[0] = make_float4(node[0], node[1], node[2], node[3]);
        mine[1] = make_float4(node[4], node[5], node[6], node[7]);
      }
    }
    if (gamma && have) {
      float g[8];
      load8<BF>(gamma, e0, g);
#pragma unroll
      for (int a = 0; a < RPP; ++a)
#pragma unroll
        for (int t = 0; t < 8; ++t) w[a][t] = fmul(w[a][t], g[t]);
    }
#pragma unroll
    for (int a = 0; a < RPP; ++a) {
      float pr[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) pr[t] = fmul(w[a][t], xh[a][t]);
      const float t8 = tree8_full(pr);
      const float leaf = full ? warp_tree_full(t8) : warp_tree(t8, (long long)warp * 256, 8, D);
      if (lane == 0) leaf_sum[f + a][warp] = leaf;
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < RPP; ++a) {
      const long long row = first + a;
      float L[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) L[j] = leaf_sum[f + a][j];
      const float c = fmul(reg_tree<8>(L, 0, 256, D), invD);   // the row's tree over its leaves (a leaf beyond D does not exist)
      if (row < rows && have) {
        float o[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) o[t] = fmul(rs[a], fsub(w[a][t], fmul(xh[a][t], c)));
        if (BF && res) {   // the gradient that bypasses the norm, added to the rounded one (res may be dx)
          float b[8];
          load8<BF>(res, (size_t)row * D + e0, b);
#pragma unroll
          for (int t = 0; t < 8; ++t) o[t] = fadd(b[t], bf2f(f2bf(o[t])));
        }
        store8<BF>(dx, (size_t)row * D + e0, o);
      }
    }
  }
  if (DG && GROUPS > 1) {   // the tree over the groups' nodes, each of RPP rows
    __syncthreads();
    if (grp) return;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      float n[GROUPS];
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) n[g] = nodes[g * WPR + warp][lane][t];
      node[t] = reg_tree<GROUPS>(n, r0, RPP, rows);
    }
  }
  if (DG && have) {
    float* dst = partial8 + (size_t)blockIdx.x * D + e0;
    *reinterpret_cast<float4*>(dst) = make_float4(node[0], node[1], node[2], node[3]);
    *reinterpret_cast<float4*>(dst + 4) = make_float4(node[4], node[5], node[6], node[7]);
  }
}
// partial8 [nb8][D] (node = 8 rows) -> partial256 [nb256][D]: tree over 32 adjacent 8-row nodes per column; the CTA
// that completes a block of 256 columns (a ticket counter per column block, zeroed by the kernel before, says which
// one it is) goes on to the levels above for those columns, 32 nodes at a time, and writes dgamma.  The counter
// decides only WHO evaluates those levels; operands and order are the fixed tree's.
__global__ void __launch_bounds__(256) k_colsum32(const float* __restrict__ partial8, int nb8, int rows, int D,
                                                  float* __restrict__ partial256, int nb256, int* __restrict__ tickets,
                                                  float* __restrict__ dgamma) {
  __shared__ int last_s;
  const int col = blockIdx.x * 256 + threadIdx.x;
  const int g = blockIdx.y;
  grid_dep();
  if (col < D) {
    float s[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int b = g * 32 + i;
      s[i] = (b < nb8) ? partial8[(size_t)b * D + col] : 0.0f;
    }
    partial256[(size_t)g * D + col] = reg_tree<32>(s, (long long)g * 256, 8, rows);
  }
  __syncthreads();
  if (threadIdx.x == 0) {   // the barrier orders the CTA's stores before this thread's fence, which is cumulative
    __threadfence();
    last_s = (atomicAdd(&tickets[blockIdx.x], 1) == nb256 - 1);
    __threadfence();
  }
  __syncthreads();
  if (!last_s || col >= D) return;
  int n = nb256;
  long long stride = 256;
  while (n > 1) {
    const int groups = (n + 31) / 32;
    for (int gg = 0; gg < groups; ++gg) {
      float s[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) s[i] = (gg * 32 + i < n) ? __ldcg(&partial256[(size_t)(gg * 32 + i) * D + col]) : 0.0f;
      partial256[(size_t)gg * D + col] = reg_tree<32>(s, (long long)gg * 32 * stride, stride, rows);
    }
    n = groups;
    stride *= 32;
  }
  dgamma[col] = __ldcg(&partial256[col]);
}

// generic two-pass variants (rows longer than 2048 elements)
template <bool BF, int NL>  // NL = leaves held in registers (0: re-read)
__global__ void __launch_bounds__(256) k_rmsnorm_fwd(const void* __restrict__ x, const void* __restrict__ gamma, int rows,
                                                     int D, float eps, float invD, void* __restrict__ y,
                                                     float* __restrict__ rstd) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 8 + warp;
  if (row >= rows) return;
  const size_t rb = (size_t)row * D;
  const int nl = (D + 255) >> 8;
  float keep[NL > 0 ? NL : 1][8];
  float mine = 0.0f;
#pragma unroll
  for (int j = 0; j < (NL > 0 ? NL : 32); ++j) {
    if (j >= nl) break;
    const int e0 = j * 256 + lane * 8;
    float v[8], sq[8];
    if (e0 < D) load8<BF>(x, rb + e0, v);
    else {
#pragma unroll
      for (int t = 0; t < 8; ++t) v[t] = 0.0f;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) sq[t] = fmul(v[t], v[t]);
    if (NL > 0) {
#pragma unroll
      for (int t = 0; t < 8; ++t) keep[j][t] = v[t];
    }
    float leaf = warp_tree(tree8_full(sq), (long long)j * 256, 8, D);
    if (lane == j) mine = leaf;
  }
  float ss = warp_tree(mine, 0, 256, D);
  float rs = fdiv(1.0f, fsqrt(fadd(fmul(ss, invD), eps)));
  if (lane == 0) rstd[row] = rs;
#pragma unroll
  for (int j = 0; j < (NL > 0 ? NL : 32); ++j) {
    if (j >= nl) break;
    const int e0 = j * 256 + lane * 8;
    if (e0 >= D) continue;
    float v[8], o[8];
    if (NL > 0) {
#pragma unroll
      for (int t = 0; t < 8; ++t) v[t] = keep[j][t];
    } else {
      load8<BF>(x, rb + e0, v);
    }
    if (gamma) {
      float g[8];
      load8<BF>(gamma, e0, g);
#pragma unroll
      for (int t = 0; t < 8; ++t) o[t] = fmul(fmul(v[t], rs), g[t]);
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) o[t] = fmul(v[t], rs);
    }
    store8<BF>(y, rb + e0, o);
  }
}

template <bool BF, int NL>
__global__ void __launch_bounds__(256) k_rmsnorm_bwd(const void* __restrict__ dy, const void* __restrict__ x,
                                                     const void* __restrict__ gamma, const float* __restrict__ rstd,
                                                     int rows, int D, float invD, void* __restrict__ dx) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 8 + warp;
  if (row >= rows) return;
  const size_t rb = (size_t)row * D;
  const int nl = (D + 255) >> 8;
  const float rs = rstd[row];
  float kw[NL > 0 ? NL : 1][8], kx[NL > 0 ? NL : 1][8];
  float mine = 0.0f;
#pragma unroll
  for (int j = 0; j < (NL > 0 ? NL : 32); ++j) {
    if (j >= nl) break;
    const int e0 = j * 256 + lane * 8;
    float w[8], xh[8], pr[8];
    if (e0 < D) {
      load8<BF>(dy, rb + e0, w);
      load8<BF>(x, rb + e0, xh);
      if (gamma) {
        float g[8];
        load8<BF>(gamma, e0, g);
#pragma unroll
        for (int t = 0; t < 8; ++t) w[t] = fmul(w[t], g[t]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) xh[t] = fmul(xh[t], rs);
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) { w[t] = 0.0f; xh[t] = 0.0f; }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) pr[t] = fmul(w[t], xh[t]);
    if (NL > 0) {
#pragma unroll
      for (int t = 0; t < 8; ++t) { kw[j][t] = w[t]; kx[j][t] = xh[t]; }
    }
    float leaf = warp_tree(tree8_full(pr), (long long)j * 256, 8, D);
    if (lane == j) mine = leaf;
  }
  const float c = fmul(warp_tree(mine, 0, 256, D), invD);
#pragma unroll
  for (int j = 0; j < (NL > 0 ? NL : 32); ++j) {
    if (j >= nl) break;
    const int e0 = j * 256 + lane * 8;
    if (e0 >= D) continue;
    float w[8], xh[8], o[8];
    if (NL > 0) {
#pragma unroll
      for (int t = 0; t < 8; ++t) { w[t] = kw[j][t]; xh[t] = kx[j][t]; }
    } else {
      load8<BF>(dy, rb + e0, w);
      load8<BF>(x, rb + e0, xh);
      if (gamma) {
        float g[8];
        load8<BF>(gamma, e0, g);
#pragma unroll
        for (int t = 0; t < 8; ++t) w[t] = fmul(w[t], g[t]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) xh[t] = fmul(xh[t], rs);
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) o[t] = fmul(rs, fsub(w[t], fmul(xh[t], c)));
    store8<BF>(dx, rb + e0, o);
  }
}

// dgamma partials: CTA = 256 rows (one leaf of the row-direction tree) x 32 columns.
template <bool BF>
__global__ void __launch_bounds__(256) k_dgamma_partial(const void* __restrict__ dy, const void* __restrict__ x,
                                                        const float* __restrict__ rstd, int rows, int D,
                                                        float* __restrict__ partial) {
  __shared__ float sm[8][33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int col = blockIdx.x * 32 + lane;
  const long long r0 = (long long)blockIdx.y * 256 + warp * 32;
  float s[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    long long r = r0 + i;
    float v = 0.0f;
    if (r < rows && col < D) {
      size_t idx = (size_t)r * D + col;
      float a, b;
      if (BF) { a = bf2f(reinterpret_cast<const uint16_t*>(dy)[idx]); b = bf2f(reinterpret_cast<const uint16_t*>(x)[idx]); }
      else { a = reinterpret_cast<const float*>(dy)[idx]; b = reinterpret_cast<const float*>(x)[idx]; }
      v = fmul(a, fmul(b, rstd[r]));
    }
    s[i] = v;
  }
  sm[warp][lane] = reg_tree<32>(s, r0, 1, rows);
  __syncthreads();
  if (warp == 0 && col < D) {
    float w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = sm[j][lane];
    partial[(size_t)blockIdx.y * D + col] = reg_tree<8>(w, (long long)blockIdx.y * 256, 32, rows);
  }
}
// tree over the nb row-block partials (each a node of 256 rows) of every column, 32 nodes at a time from independent
// loads; the partial buffer is reused for the intermediate levels
__global__ void k_col_tree(float* __restrict__ partial, int nb, int D, float* __restrict__ out, int rows) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= D) return;
  int n = nb;
  long long stride = 256;
  while (n > 1) {
    const int groups = (n + 31) / 32;
    for (int g = 0; g < groups; ++g) {
      float s[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) s[i] = (g * 32 + i < n) ? partial[(size_t)(g * 32 + i) * D + col] : 0.0f;
      partial[(size_t)g * D + col] = reg_tree<32>(s, (long long)g * 32 * stride, stride, rows);
    }
    n = groups;
    stride *= 32;
  }
  out[col] = partial[col];
}

// ------------------------------------------------------------------------------------------------
// Cross-entropy.  One CTA (512 threads) per row: max, then exp and the leaf sums, then the tree over
// leaf sums in shared memory.
// ------------------------------------------------------------------------------------------------
constexpr int XT = 512;
__global__ void __launch_bounds__(XT) k_xent_fwd(const float* __restrict__ logits, const int32_t* __restrict__ target,
                                                 int V, float* __restrict__ loss_row, float* __restrict__ lse_out,
                                                 float* __restrict__ zsq_row, int* status) {
  extern __shared__ float leafs[];  // ceil(V/256) floats, >= 32
  __shared__ float red[XT / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* z = logits + (size_t)(blockIdx.x + grid_dep()) * V;
  float m = __int_as_float(0xff800000);
  {
    auto ld4 = [&](const float* p) { return *reinterpret_cast<const float4*>(p); };
    int i = threadIdx.x * 4;
    for (; i + 3 * XT * 4 < V; i += 4 * XT * 4) {      // four loads in flight per thread
      float4 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = ld4(z + i + u * XT * 4);
#pragma unroll
      for (int u = 0; u < 4; ++u) m = fmaxf(fmaxf(m, fmaxf(a[u].x, a[u].y)), fmaxf(a[u].z, a[u].w));
    }
    for (; i < V; i += XT * 4) {
      float4 a = ld4(z + i);
      m = fmaxf(fmaxf(m, fmaxf(a.x, a.y)), fmaxf(a.z, a.w));
    }
  }
#pragma unroll
  for (int w = 16; w; w >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, w));
  if (lane == 0) red[warp] = m;
  __syncthreads();
  m = red[0];
#pragma unroll
  for (int w = 1; w < XT / 32; ++w) m = fmaxf(m, red[w]);
  const int nl = (V + 255) >> 8;
  // every argument z - m is <= 0 (or NaN), so the exponential without the overflow range applies
  const float2 one = same2(c_one);
  const int nfull = V >> 8;  // leaves that lie wholly inside the row: no existence tests in their tree
  // Second and last read of the row, from its end: the lines that the first sweep read last are those still in L2 (the rows in flight
  // on all SMs together fill it from some 50000 columns on: 4096 x 128256 0.606 ms, 0.790 from the start of the row; 4096 x 50304 0.223
  // and 0.233), and by streaming loads, so that lines leave L2 before those of rows still waiting between their two sweeps (ordinary
  // loads 0.641 and 0.248).
  for (int leaf = nfull - 1 - warp; leaf >= 0; leaf -= XT / 32) {
    const int e0 = leaf * 256 + lane * 8;
    const float4 a0 = __ldcs(reinterpret_cast<const float4*>(z + e0)), a1 = __ldcs(reinterpret_cast<const float4*>(z + e0 + 4));
    const float2 z8[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
    float e[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {          // branch-free, two at a time: the chains interleave
      const float2 v = det_exp_le0_2(add2(z8[t], same2(-m), one), one);
      e[2 * t] = v.x;
      e[2 * t + 1] = v.y;
    }
    const float s = warp_tree_full(tree8_full(e));
    if (lane == 0) leafs[leaf] = s;
  }
  if (nfull < nl && warp == (nfull % (XT / 32))) {  // the ragged last leaf
    const int leaf = nfull;
    const int e0 = leaf * 256 + lane * 8;
    float e[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (e0 + 4 * h < V) {
        float4 a = *reinterpret_cast<const float4*>(z + e0 + 4 * h);
        e[4 * h] = det_exp_le0(fsub(a.x, m)); e[4 * h + 1] = det_exp_le0(fsub(a.y, m));
        e[4 * h + 2] = det_exp_le0(fsub(a.z, m)); e[4 * h + 3] = det_exp_le0(fsub(a.w, m));
      } else {
        e[4 * h] = e[4 * h + 1] = e[4 * h + 2] = e[4 * h + 3] = 0.0f;
      }
    }
    float s = warp_tree(tree8(e, e0, V), (long long)leaf * 256, 8, V);
    if (lane == 0) leafs[leaf] = s;
  }
  __syncthreads();
  smem_tree(leafs, nl);
  if (threadIdx.x == 0) {
    float l = fadd(m, det_log(leafs[0]));
    lse_out[blockIdx.x] = l;
    int t = target[blockIdx.x];
    if (t < 0 || t >= V) {
      loss_row[blockIdx.x] = 0.0f;
      zsq_row[blockIdx.x] = 0.0f;
      or_status(status, DET_DEV_TARGET);
    } else {
      loss_row[blockIdx.x] = fsub(l, z[t]);
      zsq_row[blockIdx.x] = fmul(l, l);
    }
  }
}

// the last levels of both sums (n <= SUM_CHUNK nodes each) and the means
__global__ void __launch_bounds__(256) k_xent_finish(const float* __restrict__ ce, const float* __restrict__ zsq, int n, float inv_rows,
                                                     float z_weight, float* loss_mean, float* z_mean) {
  grid_dep();
  __shared__ float wsum[SUM_LEAVES];
  const float c = fmul(chunk_sum<false>(ce, 0, n, wsum), inv_rows);
  __syncthreads();
  const float zm = fmul(chunk_sum<false>(zsq, 0, n, wsum), inv_rows);
  if (threadIdx.x) return;
  z_mean[0] = zm;
  loss_mean[0] = (z_weight != 0.0f) ? fadd(c, fmul(z_weight, zm)) : c;
}

// Each thread takes two groups of four adjacent logits of a row, 1024 columns apart (every access of a warp covers whole
// lines).  The argument z - lse is at most 0 whenever lse is the row's own logsumexp, and then the exponential without the
// overflow range applies (same bits); lse is an input, though, so a thread that sees a positive argument takes the
// general form for its eight values.
__global__ void __launch_bounds__(256) k_xent_bwd(float* __restrict__ logits, const int32_t* __restrict__ target,
                                                  const float* __restrict__ lse, int rows, int V, float z_weight, float scale) {
  grid_dep();
  const int i0 = blockIdx.x * 2048 + threadIdx.x * 4;
  if (i0 >= V) return;
  const bool two = i0 + 1024 < V;
  const float2 one = same2(c_one);
  for (int row = blockIdx.y; row < rows; row += gridDim.y) {
    float* z = logits + (size_t)row * V;
    const int t = target[row];
    const bool ok = t >= 0 && t < V;
    const float l = lse[row];
    const float zc = fmul(fmul(2.0f, z_weight), l);
    const float4 a = *reinterpret_cast<float4*>(z + i0);
    const float4 b = two ? *reinterpret_cast<float4*>(z + i0 + 1024) : make_float4(0.f, 0.f, 0.f, 0.f);
    float x[8] = {fsub(a.x, l), fsub(a.y, l), fsub(a.z, l), fsub(a.w, l), fsub(b.x, l), fsub(b.y, l), fsub(b.z, l), fsub(b.w, l)};
    bool pos = false;
#pragma unroll
    for (int k = 0; k < 8; ++k) pos |= x[k] > 0.0f;
    float p[8];
    if (!pos) {
#pragma unroll
      for (int k = 0; k < 8; k += 2) {
        const float2 v = det_exp_le0_2(make_float2(x[k], x[k + 1]), one);
        p[k] = v.x;
        p[k + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) p[k] = det_exp(x[k]);
    }
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int col = i0 + (k >> 2) * 1024 + (k & 3);
      float d = fsub(p[k], (col == t) ? 1.0f : 0.0f);
      if (z_weight != 0.0f) d = fadd(d, fmul(zc, p[k]));
      v[k] = ok ? fmul(d, scale) : 0.0f;
    }
    *reinterpret_cast<float4*>(z + i0) = make_float4(v[0], v[1], v[2], v[3]);
    if (two) *reinterpret_cast<float4*>(z + i0 + 1024) = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// the variant for rows of D columns
template <bool BF>
static auto fwd8_kernel(int D) {
  return D <= 256 ? k_rmsnorm_fwd8<BF, 1> : (D <= 512 ? k_rmsnorm_fwd8<BF, 2> : (D <= 1024 ? k_rmsnorm_fwd8<BF, 4> : k_rmsnorm_fwd8<BF, 8>));
}
template <bool BF, bool DG>
static auto bwd8_kernel(int D) {
  if constexpr (BF)
    return D <= 256 ? k_rmsnorm_bwd8<BF, DG, 1> : (D <= 512 ? k_rmsnorm_bwd8<BF, DG, 2> : (D <= 1024 ? k_rmsnorm_bwd8<BF, DG, 4> : k_rmsnorm_bwd8<BF, DG, 8>));
  else
    return &k_rmsnorm_bwd8<BF, DG, 8>;
}

}  // namespace det

using namespace det;

extern "C" int det_rmsnorm_fwd(int io, const void* x, const void* gamma, int rows, int D, float eps, void* y,
                               float* rstd, void* stream) {
  if (!x || !y || !rstd || rows < 0 || D <= 0 || (io != DET_F32 && io != DET_BF16)) return DET_ERR_ARG;
  if (D % 8 || D > 8192) return DET_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(y) || (gamma && !aligned16(gamma))) return DET_ERR_ALIGN;
  if (rows == 0) return DET_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const float invD = (float)(1.0 / (double)D);
  dim3 grid((rows + 7) / 8);
  if (io == DET_BF16) {
    if (D <= 2048) launch_after(fwd8_kernel<true>(D), grid, 256, 0, st, x, gamma, rows, D, eps, invD, y, rstd, nullptr, nullptr, nullptr, nullptr);
    else k_rmsnorm_fwd<true, 0><<<DET_L(grid), 256, 0, st>>>(x, gamma, rows, D, eps, invD, y, rstd);
  } else {
    if (D <= 2048) launch_after(fwd8_kernel<false>(D), grid, 256, 0, st, x, gamma, rows, D, eps, invD, y, rstd, nullptr, nullptr, nullptr, nullptr);
    else k_rmsnorm_fwd<false, 0><<<DET_L(grid), 256, 0, st>>>(x, gamma, rows, D, eps, invD, y, rstd);
  }
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_rmsnorm_fwd_q(const det_bf16* x, const det_bf16* gamma, int rows, int D, float eps, det_bf16* y,
                                 float* rstd, const float* s_q, int8_t* qy, void* stream) {
  if (!x || !y || !rstd || !s_q || !qy || rows < 0 || D <= 0) return DET_ERR_ARG;
  if (D % 8 || D > 2048) return DET_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(y) || (gamma && !aligned16(gamma)) || (((uintptr_t)qy) & 7u)) return DET_ERR_ALIGN;
  if (rows == 0) return DET_OK;
  launch_after(fwd8_kernel<true>(D), (rows + 7) / 8, 256, 0, (cudaStream_t)stream, x, gamma, rows, D, eps, (float)(1.0 / (double)D), y,
                                                                              rstd, s_q, qy, nullptr, nullptr);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" size_t det_rmsnorm_bwd_ws_bytes(int rows, int D) {
  const size_t nb8 = (size_t)((rows + 7) / 8), nb256 = (size_t)((rows + 255) / 256);
  return align_up(nb8 * (size_t)D * sizeof(float), 256) + align_up(nb256 * (size_t)D * sizeof(float), 256) + 256;
}

template <bool BF>
static int rmsnorm_bwd8_launch(const void* dy, const void* x, const void* gamma, const float* rstd, int rows, int D,
                               float invD, void* dx, const void* res, float* dgamma, float* ws, cudaStream_t st) {
  const int nb8 = (rows + 7) / 8, nb256 = (rows + 255) / 256;
  if (!dgamma) {
    launch_after(bwd8_kernel<BF, false>(D), nb8, 256, 0, st, dy, x, gamma, rstd, rows, D, invD, dx, res, nullptr, nullptr);
    return DET_OK;
  }
  float* partial8 = ws;
  float* partial256 = ws + align_up((size_t)nb8 * D, 64);
  int* tickets = reinterpret_cast<int*>(partial256 + align_up((size_t)nb256 * D, 64));   // one per block of 256 columns (<= 8)
  launch_after(bwd8_kernel<BF, true>(D), nb8, 256, 0, st, dy, x, gamma, rstd, rows, D, invD, dx, res, partial8, tickets);
  // the second launch overlaps its start-up with the first kernel's tail (programmatic dependent launch); the kernel
  // itself waits for the first grid to complete before it reads anything
  launch_after(k_colsum32, dim3((D + 255) / 256, nb256), 256, 0, st, (const float*)partial8, nb8, rows, D, partial256, nb256, tickets, dgamma);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_rmsnorm_bwd(int io, const void* dy, const void* x, const void* gamma, const float* rstd, int rows,
                               int D, void* dx, float* dgamma, void* ws, size_t ws_bytes, void* stream) {
  if (!dy || !x || !rstd || !dx || rows < 0 || D <= 0 || (io != DET_F32 && io != DET_BF16)) return DET_ERR_ARG;
  if (D % 8 || D > 8192) return DET_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(dy) || !aligned16(dx) || (gamma && !aligned16(gamma))) return DET_ERR_ALIGN;
  if (dgamma && (!ws || !aligned16(ws) || ws_bytes < det_rmsnorm_bwd_ws_bytes(rows, D))) return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (rows == 0) {
    if (dgamma) cudaMemsetAsync(dgamma, 0, (size_t)D * sizeof(float), st);
    return DET_OK;
  }
  const float invD = (float)(1.0 / (double)D);
  if (D <= 2048) {
    int rc = (io == DET_BF16) ? rmsnorm_bwd8_launch<true>(dy, x, gamma, rstd, rows, D, invD, dx, nullptr, dgamma, (float*)ws, st)
                              : rmsnorm_bwd8_launch<false>(dy, x, gamma, rstd, rows, D, invD, dx, nullptr, dgamma, (float*)ws, st);
    if (rc != DET_OK) return rc;
    DET_CHECK_LAUNCH();
    return DET_OK;
  }
  dim3 grid((rows + 7) / 8);
  if (io == DET_BF16) k_rmsnorm_bwd<true, 0><<<DET_L(grid), 256, 0, st>>>(dy, x, gamma, rstd, rows, D, invD, dx);
  else k_rmsnorm_bwd<false, 0><<<DET_L(grid), 256, 0, st>>>(dy, x, gamma, rstd, rows, D, invD, dx);
  if (dgamma) {
    const int nb = (rows + 255) / 256;
    dim3 g2((D + 31) / 32, nb);
    if (io == DET_BF16) k_dgamma_partial<true><<<DET_L(g2), 256, 0, st>>>(dy, x, rstd, rows, D, (float*)ws);
    else k_dgamma_partial<false><<<DET_L(g2), 256, 0, st>>>(dy, x, rstd, rows, D, (float*)ws);
    k_col_tree<<<DET_L((D + 127) / 128), 128, 0, st>>>((float*)ws, nb, D, dgamma, rows);
  }
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_residual_rmsnorm_fwd(const det_bf16* a, const det_bf16* b, const det_bf16* gamma, int rows, int D, float eps,
                                        det_bf16* sum, det_bf16* y, float* rstd, const float* s_q, int8_t* qy, void* stream) {
  if (!a || !b || !sum || !y || !rstd || (qy && !s_q) || rows < 0 || D <= 0) return DET_ERR_ARG;
  if (D % 8 || D > 2048) return DET_ERR_SHAPE;
  if (!aligned16(a) || !aligned16(b) || !aligned16(sum) || !aligned16(y) || (gamma && !aligned16(gamma)) || (((uintptr_t)qy) & 7u))
    return DET_ERR_ALIGN;
  if (rows == 0) return DET_OK;
  launch_after(fwd8_kernel<true>(D), (rows + 7) / 8, 256, 0, (cudaStream_t)stream, a, gamma, rows, D, eps, (float)(1.0 / (double)D), y,
                                                                              rstd, s_q, qy, b, sum);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_rmsnorm_bwd_residual(const det_bf16* dy, const det_bf16* x, const det_bf16* gamma, const float* rstd, int rows,
                                        int D, const det_bf16* res, det_bf16* dx, float* dgamma, void* ws, size_t ws_bytes, void* stream) {
  if (!dy || !x || !rstd || !res || !dx || rows < 0 || D <= 0) return DET_ERR_ARG;
  if (D % 8 || D > 2048) return DET_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(dy) || !aligned16(res) || !aligned16(dx) || (gamma && !aligned16(gamma))) return DET_ERR_ALIGN;
  if (dgamma && (!ws || !aligned16(ws) || ws_bytes < det_rmsnorm_bwd_ws_bytes(rows, D))) return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (rows == 0) {
    if (dgamma) cudaMemsetAsync(dgamma, 0, (size_t)D * sizeof(float), st);
    return DET_OK;
  }
  int rc = rmsnorm_bwd8_launch<true>(dy, x, gamma, rstd, rows, D, (float)(1.0 / (double)D), dx, res, dgamma, (float*)ws, st);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" size_t det_xent_ws_bytes(int rows, int V) {
  (void)V;
  size_t r = align_up((size_t)(rows > 0 ? rows : 1), 64);
  return (r + 2 * sum_ws_floats((size_t)rows)) * sizeof(float);
}

extern "C" int det_xent_fwd(const float* logits, const int32_t* target, int rows, int V, float z_weight,
                            float* loss_row, float* lse, float* loss_mean, float* z_mean, void* ws, size_t ws_bytes,
                            void* stream, int* status_dev) {
  if (!logits || !target || !loss_row || !lse || !loss_mean || !z_mean || rows <= 0 || V <= 0 || !ws) return DET_ERR_ARG;
  if (V % 4 || V > 2 * XT * 256) return DET_ERR_SHAPE;
  if (!aligned16(logits)) return DET_ERR_ALIGN;
  if (ws_bytes < det_xent_ws_bytes(rows, V)) return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* zsq = (float*)ws;
  float* scratch = zsq + align_up((size_t)rows, 64);
  const int nl = (V + 255) / 256;
  size_t sh = (size_t)(nl < 32 ? 32 : nl) * sizeof(float);
  launch_after(k_xent_fwd, rows, XT, sh, st, logits, target, V, loss_row, lse, zsq, status_dev);
  const float* ce = loss_row;
  const float* zs = zsq;
  size_t n = (size_t)rows, nz = (size_t)rows;
  sum_to_chunk(ce, n, scratch, st);
  sum_to_chunk(zs, nz, scratch, st);
  launch_after(k_xent_finish, 1, 256, 0, st, ce, zs, (int)n, (float)(1.0 / (double)rows), z_weight, loss_mean, z_mean);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_xent_bwd(float* logits_inout, const int32_t* target, const float* lse, int rows, int V,
                            float z_weight, float scale, void* stream) {
  if (!logits_inout || !target || !lse || rows <= 0 || V <= 0) return DET_ERR_ARG;
  if (V % 4) return DET_ERR_SHAPE;
  if (!aligned16(logits_inout)) return DET_ERR_ALIGN;
  dim3 grid((V + 2047) / 2048, rows < 65535 ? rows : 65535);
  launch_after(k_xent_bwd, grid, 256, 0, (cudaStream_t)stream, logits_inout, target, lse, rows, V, z_weight, scale);
  DET_CHECK_LAUNCH();
  return DET_OK;
}
