// int8 x int8 -> int32 contraction on the 5th-generation tensor cores (tcgen05), used by the three GEMMs
// of every LSQ linear layer (Sec. 3.2 "int8 computation": forward, grad-x and grad-W all run in int8 and
// accumulate in int32, which is exact and therefore order-free).
//
//   C[i,j] = sum_k A[i,k] * B[j,k]        A: int8 [I,K] row-major, B: int8 [J,K] row-major (both K-major)
//
// One persistent CTA per SM, tiles of 128 x BN (BN = 256, 128 or 64):
//   warp 0    TMA producer: 128-byte-swizzled tiles of A (128 x 128 B) and B (BN x 128 B) into a ring of 4 to 8 stages
//   warp 1    allocates TMEM (two BN-column accumulators) and issues tcgen05.mma.kind::i8
//             (M=128, N=BN, K=32 per instruction, 4 per stage); tcgen05.commit releases ring slots
//   the rest  epilogue: tcgen05.ld of the int32 accumulator (lane = row), dequantise / mask in registers, stores in whole
//             row segments through a staging tile; overlaps with the next tile's MMAs through the second accumulator
// Every mbarrier wait is bounded: on expiry the kernel raises DET_DEV_TIMEOUT in *status, stops issuing
// work, lets in-flight copies land, frees its TMEM and returns.
#include "tc05.cuh"
#include "internal.h"
#include "../../include/det_test.h"

namespace det {

constexpr int BM = 128;
constexpr int BK = 128;  // bytes (= int8 elements) per stage along K
// eight epilogue warps (two per TMEM lane quarter, half of the columns each), four for the narrow tile
template <int BN> struct IgTile {
  static constexpr int STAGES = BN == 256 ? 4 : (BN == 128 ? 6 : 8), EW = BN == 64 ? 4 : 8, CW = BN / (EW / 4);
  static constexpr int THREADS = 64 + 32 * EW, TCOLS = 2 * BN;
  static constexpr size_t SMEM = (size_t)STAGES * (BM * BK + BN * BK) + EW * 4096 + 1024;
};
// Tile order: the dimension with fewer tiles runs fastest, so that the CTAs resident at one time share the smaller
// operand's tiles and the larger operand streams through L2 once.
__device__ __forceinline__ void tile_origin(int tile, int tiles_i, int tiles_j, int bn, int& i0, int& j0) {
  if (tiles_j <= tiles_i) { j0 = (tile % tiles_j) * bn; i0 = (tile / tiles_j) * BM; }
  else { i0 = (tile % tiles_i) * BM; j0 = (tile / tiles_i) * bn; }
}

// data-dependent scalars of the epilogue, read once per CTA from device memory
template <int EPI>
__device__ __forceinline__ void epi_scalars(const EpiParams& ep, float& cscale, float& inv_s, float& sx) {
  cscale = 1.0f; inv_s = 1.0f; sx = 1.0f;
    if (EPI == EPI_FWD) sx = ep.s_x[0];
    if (EPI == EPI_DX) {
      const float am = __uint_as_float(ep.amax1[0]);
      const float s_a = (am > 0.0f) ? fdiv(am, 127.0f) : 0.0f;
      cscale = fmul(fmul(s_a, ep.s_u[0]), ep.rot);
      inv_s = fdiv(1.0f, ep.s_x[0]);
    }
    if (EPI == EPI_DW) {
      const float am = __uint_as_float(ep.amax1[0]);
      const float s_g = (am > 0.0f) ? fdiv(am, 127.0f) : 0.0f;
      float s_z = 1.0f;
      if (ep.amax2) {
        const int az = (int)ep.amax2[0];
        s_z = (az > 0) ? fdiv(__int2float_rn(az), 127.0f) : 0.0f;
      }
      cscale = fmul(fmul(fmul(s_g, s_z), ep.s_x[0]), ep.rot);
    }
}

// The reverse for the bf16 reference operand of the gradient epilogues: `pre` holds sixteen-byte pieces fetched with whole
// 64-byte row segments per quad of lanes (fetch_rows32); rows32_to_lanes hands every lane the four words of its own row.
__device__ __forceinline__ void fetch_rows32(const uint8_t* gbase, size_t row_pitch_bytes, uint4 (&pre)[4]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    pre[i] = __ldg(reinterpret_cast<const uint4*>(gbase + (size_t)(i * 8 + (lane >> 2)) * row_pitch_bytes + (lane & 3) * 16));
}
__device__ __forceinline__ void rows32_to_lanes(uint8_t* stage, const uint4 (&pre)[4], uint4 (&w)[4]) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = i * 8 + (lane >> 2), piece = lane & 3;
    *reinterpret_cast<uint4*>(stage + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4)) = pre[i];
  }
  __syncwarp();
#pragma unroll
  for (int v = 0; v < 4; ++v) w[v] = *reinterpret_cast<const uint4*>(stage + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4));
}

// Epilogue of one accumulator row: this lane owns TMEM lane `taddr`'s row (output row `row`), columns j0 .. j0+CW.
// The outputs are written through store_rows32 and the reference operand is read the same way, one chunk of 32 ahead (`stage`: 4 KiB
// per warp).  DX leaves the partial sums of dXhat * phi of every 64 columns (an aligned subtree of the fixed tree).
template <int CW, int EPI>
__device__ __forceinline__ void epi_row(const EpiParams& ep, uint32_t taddr, int row, int J, int j0, float cscale,
                                        float inv_s, float sx, uint8_t* stage) {
  const size_t wbase = (size_t)(row - (int)(threadIdx.x & 31)) * J + j0;  // the warp's first row
  constexpr bool REF = EPI == EPI_DX || EPI == EPI_DW;
  if (EPI == EPI_DW) inv_s = fdiv(1.0f, ep.s_w[row]);
  uint4 pre[4];
  if (REF) fetch_rows32(reinterpret_cast<const uint8_t*>(ep.ref + wbase), (size_t)J * 2, pre);
#pragma unroll 1
  for (int h = 0; h < CW / 64; ++h) {
    float grp[2];
#pragma unroll
    for (int cc = 0; cc < 2; ++cc) {
      const int c0 = h * 64 + cc * 32;
      uint32_t r[32];
      tmem_ld32(taddr + (uint32_t)c0, r);
      uint4 refw[4];
      if (REF) {
        rows32_to_lanes(stage, pre, refw);
        if (c0 + 32 < CW) fetch_rows32(reinterpret_cast<const uint8_t*>(ep.ref + wbase + c0 + 32), (size_t)J * 2, pre);
      }
      if (EPI == EPI_RAW) {
        uint4 o[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) o[v] = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
        store_rows32<8>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<int32_t*>(ep.out) + wbase + c0), (size_t)J * 4, o);
      } else if (EPI == EPI_FWD) {
        const float4* sw = reinterpret_cast<const float4*>(ep.s_w + j0 + c0);
        uint4 o[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          float4 w0 = __ldg(sw + 2 * v), w1 = __ldg(sw + 2 * v + 1);
          float f[8];
          f[0] = fmul(__int2float_rn((int)r[8 * v + 0]), fmul(sx, w0.x));
          f[1] = fmul(__int2float_rn((int)r[8 * v + 1]), fmul(sx, w0.y));
          f[2] = fmul(__int2float_rn((int)r[8 * v + 2]), fmul(sx, w0.z));
          f[3] = fmul(__int2float_rn((int)r[8 * v + 3]), fmul(sx, w0.w));
          f[4] = fmul(__int2float_rn((int)r[8 * v + 4]), fmul(sx, w1.x));
          f[5] = fmul(__int2float_rn((int)r[8 * v + 5]), fmul(sx, w1.y));
          f[6] = fmul(__int2float_rn((int)r[8 * v + 6]), fmul(sx, w1.z));
          f[7] = fmul(__int2float_rn((int)r[8 * v + 7]), fmul(sx, w1.w));
          o[v] = make_uint4(pack_bf2(f[0], f[1]), pack_bf2(f[2], f[3]), pack_bf2(f[4], f[5]), pack_bf2(f[6], f[7]));
        }
        store_rows32<4>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<uint16_t*>(ep.out) + wbase + c0), (size_t)J * 2, o);
      } else if (EPI == EPI_DX) {
        uint4 o[4];
        float term[32];
        const float2 one = same2(c_one);
#pragma unroll
        for (int v = 0; v < 16; ++v) {
          const uint32_t xs = reinterpret_cast<const uint32_t*>(refw)[v];
          const float2 gx = mul2(make_float2(__int2float_rn((int)r[2 * v]), __int2float_rn((int)r[2 * v + 1])), same2(cscale));
          const float2 t = mul2(make_float2(bflo(xs), bfhi(xs)), same2(inv_s));
          // t held to [-128, 127]; rne(t) - t where it holds t itself (a NaN included: it compares neither below nor above)
          const float2 tc = make_float2(fminf(fmaxf(t.x, -128.0f), 127.0f), fminf(fmaxf(t.y, -128.0f), 127.0f));
          const float2 d = add2(add2(add2(t, same2(12582912.0f), one), same2(-12582912.0f), one), make_float2(-t.x, -t.y), one);
          const float2 phi = make_float2((t.x < tc.x || t.x > tc.x) ? tc.x : d.x, (t.y < tc.y || t.y > tc.y) ? tc.y : d.y);
          reinterpret_cast<uint32_t*>(o)[v] = pack_bf2(t.x == tc.x ? gx.x : 0.0f, t.y == tc.y ? gx.y : 0.0f);
          const float2 p = mul2(gx, phi);
          term[2 * v] = p.x;
          term[2 * v + 1] = p.y;
        }
        store_rows32<4>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<uint16_t*>(ep.out) + wbase + c0), (size_t)J * 2, o);
        // adjacent tree over this lane's 32 columns
#pragma unroll
        for (int w = 1; w < 32; w <<= 1)
#pragma unroll
          for (int e = 0; e < 32; e += 2 * w) term[e] = fadd(term[e], term[e + w]);
        grp[cc] = term[0];
      } else {  // EPI_DW
        uint4 o[8];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          uint4 wu = refw[v];
          const uint32_t wsr[4] = {wu.x, wu.y, wu.z, wu.w};
          float g[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float wv = (e & 1) ? bfhi(wsr[e >> 1]) : bflo(wsr[e >> 1]);
            const float t = fmul(wv, inv_s);
            const bool in_range = (t >= -128.0f) && (t <= 127.0f);
            g[e] = in_range ? fmul(__int2float_rn((int)r[8 * v + e]), cscale) : 0.0f;
          }
          o[2 * v] = make_uint4(__float_as_uint(g[0]), __float_as_uint(g[1]), __float_as_uint(g[2]), __float_as_uint(g[3]));
          o[2 * v + 1] = make_uint4(__float_as_uint(g[4]), __float_as_uint(g[5]), __float_as_uint(g[6]), __float_as_uint(g[7]));
        }
        store_rows32<8>(stage, reinterpret_cast<uint8_t*>(reinterpret_cast<float*>(ep.out) + wbase + c0), (size_t)J * 4, o);
      }
    }
    if (EPI == EPI_DX) ep.ds_partial[(size_t)row * (J / 64) + (j0 / 64) + h] = fadd(grp[0], grp[1]);
  }
}

// A product of a launch that has two of them, with the same columns J
struct IgProduct {
  CUtensorMap a, b;
  EpiParams ep;
  int I, K;
};
// The tiles of CTA `b` of `g`, one after the other: from `at`, the tile before, to tile `it`.  One product steps on; computed from `it` like
// two, that cost its kernel more registers and 1 % (8192 x 384 x 384, a backward pass of two launches: 47.4 and 47.8 us).
template <bool TWO>
struct IgWalk {
  int n0, n1, b, g, lead;
  __device__ __forceinline__ int before() const { return b - g; }
  __device__ __forceinline__ bool tile(int it, int& job, int& at) const {
    job = 0;
    at += g;
    return at < n0;
  }
};
// Two products: the tiles of the second (n1) come behind those of the first (n0), and the CTAs that have one tile of the first less take `lead` tiles
// of the second while the others are at it.
template <>
struct IgWalk<true> {
  int n0, n1, b, g, lead;
  __device__ __forceinline__ int before() const { return b - g; }
  __device__ __forceinline__ bool tile(int it, int& job, int& at) const {
    job = 0;
    at = b + it * g;
    if (at < n0) return true;
    if (n1 == 0) return false;
    const int own = b < n0 ? (n0 - b + g - 1) / g : 0, rest = n0 % g, mine = b >= rest ? lead : 0;
    job = 1;
    it -= own;
    at = it < mine ? it * (g - rest) + b - rest : lead * (g - rest) + (it - mine) * g + b;
    return at < n1;
  }
};

template <int BN, int EPI, int EPI2>
__device__ __forceinline__ void ig_body(const CUtensorMap& tmA, const CUtensorMap& tmB, const EpiParams& ep, int I, int J, int K,
                                        int* status, int fill, const IgProduct* second, int lead) {
  constexpr int STAGE_A = BM * BK, STAGE_B = BN * BK, STAGE_BYTES = STAGE_A + STAGE_B;
  constexpr int STAGES = IgTile<BN>::STAGES, EW = IgTile<BN>::EW, CW = IgTile<BN>::CW;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bar_full[STAGES], bar_empty[STAGES], bar_tfull[2], bar_tempty[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(&bar_tfull[a], 1); mbar_init(&bar_tempty[a], EW); }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)IgTile<BN>::TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  if (fill) grid_fill_begin();
  else grid_dep();

  constexpr bool TWO = EPI2 >= 0;
  const int tiles_j = J / BN, tiles_i[2] = {I / BM, TWO ? second->I / BM : 0}, kblocks[2] = {K / BK, TWO ? second->K / BK : 0};
  const IgWalk<TWO> walk = {tiles_i[0] * tiles_j, tiles_i[1] * tiles_j, (int)blockIdx.x, (int)gridDim.x, lead};

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, job, tile = walk.before();
      uint32_t phase = 0;
      bool ok = true;
      for (int it = 0; ok && walk.tile(it, job, tile); ++it) {
        const bool w = TWO && job;
        int i0, j0;
        tile_origin(tile, w ? tiles_i[1] : tiles_i[0], tiles_j, BN, i0, j0);
        const CUtensorMap *ma = w ? &second->a : &tmA, *mb = w ? &second->b : &tmB;
        for (int kb = 0, nk = w ? kblocks[1] : kblocks[0]; kb < nk; ++kb) {
          if (!mbar_wait(&bar_empty[stage], phase ^ 1u, abort_flag, status)) { ok = false; break; }
          mbar_expect_tx(&bar_full[stage], STAGE_BYTES);
          uint8_t* sa = smem + stage * STAGE_BYTES;
          tma_load_2d(sa, ma, kb * BK, i0, &bar_full[stage]);
          tma_load_2d(sa + STAGE_A, mb, kb * BK, j0, &bar_full[stage]);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // instruction descriptor: D = S32, A = B = signed 8-bit, both K-major, N = BN, M = 128
      constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      int stage = 0, job, tile = walk.before();
      uint32_t phase = 0;
      bool ok = true;
      for (int it = 0; ok && walk.tile(it, job, tile); ++it) {
        const int acc = it & 1;
        const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
        if (!mbar_wait(&bar_tempty[acc], acc_phase ^ 1u, abort_flag, status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(acc * BN);
        for (int kb = 0, nk = TWO && job ? kblocks[1] : kblocks[0]; kb < nk; ++kb) {
          if (!mbar_wait(&bar_full[stage], phase, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * STAGE_BYTES);
          const uint64_t da = make_smem_desc(sa), db = make_smem_desc(sa + STAGE_A);
#pragma unroll
          for (int k4 = 0; k4 < BK / 32; ++k4)
            umma_i8(tmem_d, da + (uint64_t)(k4 * 2), db + (uint64_t)(k4 * 2), idesc, (kb | k4) ? 1u : 0u);
          umma_commit(&bar_empty[stage]);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit(&bar_tfull[acc]);
      }
    }
  } else {
    const int q = warp & 3, part = (warp - 2) >> 2;  // TMEM lane quarter this warp may read; its share of the columns
    uint8_t* stage = smem + STAGES * STAGE_BYTES + (warp - 2) * 4096;  // this warp's 32 x 128-byte staging tile
    int job, tile = walk.before();
    float cscale, inv_s, sx, cscale2 = 1.0f, inv_s2 = 1.0f, sx2 = 1.0f;
    epi_scalars<EPI>(ep, cscale, inv_s, sx);
    if constexpr (TWO) epi_scalars<EPI2>(second->ep, cscale2, inv_s2, sx2);
    // A wait that ran out is passed over and the loop runs to its end: a tile's loads and stores are the warp's, and lanes that have given up must
    // not leave the others in them (later waits see the abort flag after a few polls; the output is undefined then).  A vote of the warp instead
    // costs up to 2 % where the epilogue bounds (forward of 1792 x 14336 x 256 20.1 and 20.5 us).
    for (int it = 0; walk.tile(it, job, tile); ++it) {
      const int acc = it & 1;
      const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
      int i0, j0;
      tile_origin(tile, TWO && job ? tiles_i[1] : tiles_i[0], tiles_j, BN, i0, j0);
      mbar_wait(&bar_tfull[acc], acc_phase, abort_flag, status);
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + part * CW);
      if (!TWO || !job) epi_row<CW, EPI>(ep, taddr, i0 + q * 32 + lane, J, j0 + part * CW, cscale, inv_s, sx, stage);
      if constexpr (TWO)
        if (job) epi_row<CW, EPI2>(second->ep, taddr, i0 + q * 32 + lane, J, j0 + part * CW, cscale2, inv_s2, sx2, stage);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_tempty[acc]);
    }
  }

  // teardown: everyone meets here; after a timeout give in-flight copies time to land first
  __syncthreads();
  if (abort_s) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)IgTile<BN>::TCOLS) : "memory");
  }
}
template <int BN, int EPI>
__global__ void __launch_bounds__(IgTile<BN>::THREADS, 1)
    k_igemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, EpiParams ep, int I, int J, int K,
            int* status, int fill) {
  ig_body<BN, EPI, -1>(tmA, tmB, ep, I, J, K, status, fill, nullptr, 0);
  if (fill) grid_fill_end();
}
// both gradient products of a linear layer, dX [M, K] over N and dW [N, K] over M, `p` before `s`; two epilogues in one kernel spill 28, 48 and 88 bytes
// a thread with 64, 128 and 256 columns
template <int BN, bool W_FIRST>
__global__ void __launch_bounds__(IgTile<BN>::THREADS, 1)
    k_igemm_grads(const __grid_constant__ IgProduct p, const __grid_constant__ IgProduct s, int J, int* status, int lead) {
  ig_body<BN, W_FIRST ? EPI_DW : EPI_DX, W_FIRST ? EPI_DX : EPI_DW>(p.a, p.b, p.ep, p.I, J, p.K, status, 0, &s, lead);
}

// ------------------------------------------------------------------------------------------------------------
// Two-CTA variant (tcgen05 cta_group::2).  A cluster of two CTAs on neighbouring SMs computes one 256 x 256 tile:
// CTA r owns rows r*128 .. r*128+127 of the tile (its own A rows and its own 128 x 256 accumulator in TMEM) and stages
// only half of the B tile (rows r*128 .. of the 256 B rows); the MMA, issued by the leader CTA for both, reads the two
// halves of B from the two CTAs' shared memory.  Per CTA and K step that is 32 KiB staged and 32 KiB read by the tensor
// core instead of 48 + 48 KiB, which matters because TMA writes and MMA operand reads share the shared-memory port.
//   * each CTA's producer thread loads its own A / B-half tiles; the loads complete on the LEADER's full barrier
//   * the leader's MMA thread waits on that barrier, issues the MMAs, and releases the ring slot in BOTH CTAs with a
//     multicast tcgen05.commit; the same for "accumulator ready"
//   * the epilogue warps of both CTAs drain their own TMEM and arrive on the leader's "accumulator free" barrier
// No load uses cluster multicast.  All waits are bounded as in the one-CTA kernel.
// ------------------------------------------------------------------------------------------------------------
constexpr int STAGES2 = 6;
constexpr int BN2 = 256;
// warps 0 / 1 load and multiply; eight epilogue warps: warp & 3 is the TMEM lane quarter a warp may read, the two
// warps of a quarter take one half (128 columns) of the accumulator each
constexpr int GEMM2_THREADS = 64 + 8 * 32;

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM2_THREADS, 1)
    k_igemm2(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, EpiParams ep, int I, int J,
             int K, int* status, int fill) {
  constexpr int STAGE_A = 128 * BK, STAGE_B = 128 * BK, STAGE_BYTES = STAGE_A + STAGE_B;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bar_full[STAGES2], bar_empty[STAGES2], bar_tfull[2], bar_tempty[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES2; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(&bar_tfull[a], 1); mbar_init(&bar_tempty[a], 16); }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers are initialised before anything can signal them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  if (fill) grid_fill_begin();
  else grid_dep();

  const int tiles_i = I / 256, tiles_j = J / BN2;
  const int num_tiles = tiles_i * tiles_j;
  const int kblocks = K / BK;
  const int cluster_id = blockIdx.x >> 1, nclusters = gridDim.x >> 1;

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = cluster_id; tile < num_tiles && ok; tile += nclusters) {
        int i0, j0;
        if (tiles_j <= tiles_i) { j0 = (tile % tiles_j) * BN2; i0 = (tile / tiles_j) * 256; }
        else { i0 = (tile % tiles_i) * 256; j0 = (tile / tiles_i) * BN2; }
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait(&bar_empty[stage], phase ^ 1u, abort_flag, status)) { ok = false; break; }
          if (leader) mbar_expect_tx(&bar_full[stage], 2 * STAGE_BYTES);  // both CTAs' tiles complete on this barrier
          uint8_t* sa = smem + stage * STAGE_BYTES;
          tma_load_2d_pair(sa, &tmA, kb * BK, i0 + (int)rank * 128, &bar_full[stage]);
          tma_load_2d_pair(sa + STAGE_A, &tmB, kb * BK, j0 + (int)rank * 128, &bar_full[stage]);
          if (++stage == STAGES2) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // instruction descriptor: D = S32, A = B = signed 8-bit, both K-major, N = 256, M = 256 (two CTAs x 128)
      constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN2 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      for (int tile = cluster_id; tile < num_tiles && ok; tile += nclusters, ++it) {
        const int acc = it & 1;
        const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
        if (!mbar_wait(&bar_tempty[acc], acc_phase ^ 1u, abort_flag, status)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(acc * BN2);
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait(&bar_full[stage], phase, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * STAGE_BYTES);
          const uint64_t da = make_smem_desc(sa), db = make_smem_desc(sa + STAGE_A);
#pragma unroll
          for (int k4 = 0; k4 < BK / 32; ++k4)
            umma_i8_pair(tmem_d, da + (uint64_t)(k4 * 2), db + (uint64_t)(k4 * 2), idesc, (kb | k4) ? 1u : 0u);
          umma_commit_pair(&bar_empty[stage]);
          if (++stage == STAGES2) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(&bar_tfull[acc]);
      }
    }
  } else {
    const int q = warp & 3, half = (warp - 2) >> 2;
    uint8_t* stage = smem + STAGES2 * STAGE_BYTES + (warp - 2) * 4096;  // this warp's 32 x 128-byte staging tile
    int it = 0;
    float cscale, inv_s, sx;
    epi_scalars<EPI>(ep, cscale, inv_s, sx);
    const uint32_t tempty_leader0 = mapa_u32(smem_u32(&bar_tempty[0]), 0), tempty_leader1 = mapa_u32(smem_u32(&bar_tempty[1]), 0);
    for (int tile = cluster_id; tile < num_tiles; tile += nclusters, ++it) {
      const int acc = it & 1;
      const uint32_t acc_phase = (uint32_t)(it >> 1) & 1u;
      int i0, j0;
      if (tiles_j <= tiles_i) { j0 = (tile % tiles_j) * BN2; i0 = (tile / tiles_j) * 256; }
      else { i0 = (tile % tiles_i) * 256; j0 = (tile / tiles_i) * BN2; }
      mbar_wait(&bar_tfull[acc], acc_phase, abort_flag, status);   // passed over when it ran out, as in the one-CTA kernel
      tc_fence_after();
      epi_row<BN2 / 2, EPI>(ep, tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN2 + half * (BN2 / 2)),
                            i0 + (int)rank * 128 + q * 32 + lane, J, j0 + half * (BN2 / 2), cscale, inv_s, sx, stage);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(acc ? tempty_leader1 : tempty_leader0);
    }
  }

  // teardown: both CTAs meet before either leaves (the peer may still signal this CTA's barriers or read its tiles)
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
  if (fill) grid_fill_end();
}

// ---- host side -------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = (EncodeTiledFn)p;
  }
  return fn;
}
bool make_map(CUtensorMap* tm, const int8_t* base, int rows, int K, int box_rows) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  cuuint64_t gdim[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t gstr[1] = {(cuuint64_t)K};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void*)base, gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int EPI>
static int launch_one(const CUtensorMap& ta, const CUtensorMap& tb, const EpiParams& ep, int I, int J, int K, int* status,
                      cudaStream_t st, int fill) {
  typedef IgTile<BN> T;
  static DevOnce once = {};
  if (dev_ensure_smem(once, (const void*)k_igemm<BN, EPI>, T::SMEM) != DET_OK) return DET_ERR_CUDA;
  const int sms = dev_sm_count();
  if (sms <= 0) return DET_ERR_CUDA;
  const int tiles = (I / BM) * (J / BN);
  const int grid = tiles < sms ? tiles : sms;
  launch_after(k_igemm<BN, EPI>, grid, T::THREADS, T::SMEM, st, ta, tb, ep, I, J, K, status, fill);
  if (cudaPeekAtLastError() != cudaSuccess) { cudaGetLastError(); return DET_ERR_CUDA; }
  return DET_OK;
}

template <int EPI>
static int launch_pair(const CUtensorMap& ta, const CUtensorMap& tb, const EpiParams& ep, int I, int J, int K, int* status,
                       cudaStream_t st, int fill) {
  constexpr size_t smem = (size_t)STAGES2 * (2 * 128 * BK) + 8 * 4096 + 1024;
  static DevOnce once = {};
  if (dev_ensure_smem(once, (const void*)k_igemm2<EPI>, smem) != DET_OK) return DET_ERR_CUDA;
  const int sms = dev_sm_count();
  if (sms < 2) return DET_ERR_CUDA;
  const int tiles = (I / 256) * (J / BN2);
  int clusters = sms / 2;
  if (tiles < clusters) clusters = tiles;
  launch_after(k_igemm2<EPI>, 2 * clusters, GEMM2_THREADS, smem, st, ta, tb, ep, I, J, K, status, fill);
  if (cudaPeekAtLastError() != cudaSuccess) { cudaGetLastError(); return DET_ERR_CUDA; }
  return DET_OK;
}

// Which tile: whole rounds of tiles over the SMs, each the longer of its multiply loop and its epilogue, and once the other of the
// two.  Measured, in microseconds: a 128-deep step costs 0.37 with 256-column tiles and 0.30 with narrower ones (bound by the
// tensor pipe and by L2), the epilogue of a tile what the table says.  A small grid is bound by the epilogue of one tile, which a
// narrow tile shortens and spreads over more SMs (1024 x 1024 x 1024: 11.1, 10.6, 8.5, 8.5 forward and 16.7, 15.3, 12.6, 10.5
// input gradient for 256 x 256 pairs and 256, 128, 64 columns); over many rounds the pairs run a few percent faster
// than their rounds say (16384 x 2048 x 8192: 166, 171, 265, 520), over few of them the 256-column tiles of one CTA.
// bn: the columns of a one-CTA tile, or 512 for the CTA pair (256 x 256); work: its time on a full GPU without the last round's loss.
struct IgCost { int bn, bi, bj, pair; double step, turn, epi[4]; };               // epi: RAW, FWD, DX, DW
constexpr IgCost IG_COST[4] = {{512, 256, 256, 1, 0.365, 0.9, {6.6, 4.2, 10.0, 6.6}}, {256, 128, 256, 0, 0.375, 0.5, {8.4, 4.0, 9.3, 6.2}},
                               {128, 128, 128, 0, 0.30, 0.5, {3.8, 1.7, 5.7, 3.8}}, {64, 128, 64, 0, 0.30, 0.5, {1.8, 1.7, 3.7, 1.8}}};
struct IgPlan { int bn, tiles; double each, tail, work; };                        // each: a tile's time, tail: what the last one takes longer
static IgPlan igemm_pick(int epi, int I, int J, int K, int force_one_cta) {
  const int sms = dev_sm_count() > 0 ? dev_sm_count() : 1;
  const IgCost* c = IG_COST;
  IgPlan best = {};
  double best_t = 0.0;
  for (int i = force_one_cta ? 1 : 0; i < 4; ++i) {
    const int units = c[i].pair ? sms / 2 : sms;
    if (I % c[i].bi || J % c[i].bj || !units) continue;
    const long long tiles = (long long)(I / c[i].bi) * (J / c[i].bj), rounds = (tiles + units - 1) / units;
    const double loop = (K / BK) * c[i].step, e = c[i].epi[epi], each = (loop > e ? loop : e) + c[i].turn, tail = loop > e ? e : loop;
    double t = rounds * each + tail;
    if (c[i].bn == 512 && rounds >= 6) t *= 0.95;
    if (!best.bn || t < best_t) {
      best = {c[i].bn, (int)tiles, each, tail, tiles * each / units};
      best_t = t;
    }
  }
  return best;
}
template <int EPI>
static int igemm_tile(int bn, const CUtensorMap& ta, const CUtensorMap& tb, const EpiParams& ep, int I, int J, int K, int* status,
                      cudaStream_t st, int fill) {
  switch (bn) {
    case 512: return launch_pair<EPI>(ta, tb, ep, I, J, K, status, st, fill);
    case 256: return launch_one<256, EPI>(ta, tb, ep, I, J, K, status, st, fill);
    case 128: return launch_one<128, EPI>(ta, tb, ep, I, J, K, status, st, fill);
    default: return launch_one<64, EPI>(ta, tb, ep, I, J, K, status, st, fill);
  }
}
int igemm_launch(int epi, const int8_t* A, const int8_t* B, int I, int J, int K, const EpiParams& ep, int* status,
                 cudaStream_t st, int force_one_cta, int fill) {
  if (!A || !B || I <= 0 || J <= 0 || K <= 0) return DET_ERR_ARG;
  if (I % BM || J % 128 || K % BK) return DET_ERR_SHAPE;
  if (K >= (1 << 17)) return DET_ERR_RANGE;
  if (!aligned16(A) || !aligned16(B)) return DET_ERR_ALIGN;
  const int bn = igemm_pick(epi, I, J, K, force_one_cta).bn;
  CUtensorMap ta, tb;
  if (!make_map(&ta, A, I, K, 128) || !make_map(&tb, B, J, K, bn == 512 ? 128 : bn)) return DET_ERR_CUDA;
  switch (epi) {
    case EPI_RAW: return igemm_tile<EPI_RAW>(bn, ta, tb, ep, I, J, K, status, st, fill);
    case EPI_FWD: return igemm_tile<EPI_FWD>(bn, ta, tb, ep, I, J, K, status, st, fill);
    case EPI_DX: return igemm_tile<EPI_DX>(bn, ta, tb, ep, I, J, K, status, st, fill);
    case EPI_DW: return igemm_tile<EPI_DW>(bn, ta, tb, ep, I, J, K, status, st, fill);
  }
  return DET_ERR_ARG;
}

template <int BN>
static int grads_tile(bool w_first, const IgProduct& p, const IgProduct& s, int J, int grid, int lead, int* status, cudaStream_t st) {
  typedef IgTile<BN> T;
  static DevOnce once[2] = {};
  const auto kern = w_first ? k_igemm_grads<BN, true> : k_igemm_grads<BN, false>;
  if (dev_ensure_smem(once[w_first], (const void*)kern, T::SMEM) != DET_OK) return DET_ERR_CUDA;
  launch_after(kern, grid, T::THREADS, T::SMEM, st, p, s, J, status, lead);
  if (cudaPeekAtLastError() != cudaSuccess) { cudaGetLastError(); return DET_ERR_CUDA; }
  return DET_OK;
}
// When the last CTA of product `w` is done whose CTAs move in behind those of product `x`, first on the SMs that it leaves idle, then as they end
static double behind_each_other(const IgPlan& x, const IgPlan& w, int sms) {
  const int gx = x.tiles < sms ? x.tiles : sms, gw = w.tiles < sms ? w.tiles : sms, rest = w.tiles % gw;
  auto free = [&](int j) {                                            // of the j-th SM to be free
    j -= sms - gx;
    return j < 0 ? 0.0 : (x.tiles / gx + (j >= gx - x.tiles % gx)) * x.each + x.tail;
  };
  const double few = free(gw - 1) + (w.tiles / gw) * w.each, many = rest ? free(rest - 1) + (w.tiles / gw + 1) * w.each : 0.0;
  const double wt = (few > many ? few : many) + w.tail, xt = free(sms - 1);
  return wt > xt ? wt : xt;
}
// Both gradient products in one launch, *did, instead of two; fork: the two would be on two streams, else one behind the other.  The product with
// the longer tiles comes first; the time of a tile width is that of the CTA that has most to do.  Whole input passes, tokens, rows and columns,
// microseconds, two launches and one, 445 shapes measured:
//   on one stream one launch is the better one nearly always (512 x 512 x 512 18.6 and 17.4, 1024 x 1024 x 1024 26.2 and 21.6, 2560 x 3584 x 256 53.6
//     and 45.5), unless its one width costs much more than the two widths of the others (128 x 7424 x 256 32.7 and 33.9);
//   instead of a fork and a join one launch has to be faster by what it loses: the sum of the step gradient, which runs beside the weight
//     gradient otherwise, from 16384 partial sums on in two launches (1024 x 5632 x 1024 52.6 and 46.0, 512 x 9216 x 1408 78.7 and 61.8; but 384 x 1408 x
//     3328 29.0 and 33.8, 3840 x 384 x 768 30.9 and 35.8, 1024 x 2048 x 2816 41.4 and 43.0).  Long columns in wide tiles (768 x 4864 x 3328 71.3 and 77.9,
//     128 x 6016 x 2048 40.8 and 43.3) and long work (896 x 16384 x 2432 162 and 168) stay apart.
// Of the 328 forks 109 are joined, four of them to their loss (6 % at most); the joined ones gain 6 % in the mean.
int igemm_grads_launch(const int8_t* A, const int8_t* Ut, const EpiParams& ex, const int8_t* Gt, const int8_t* Zt, const EpiParams& ew,
                       int M, int N, int K, bool fork, int* status, cudaStream_t st, bool* did) {
  *did = false;
  const int sms = dev_sm_count();
  if (sms <= 0) return DET_ERR_CUDA;
  const IgPlan px = igemm_pick(EPI_DX, M, K, N, 0), pw = igemm_pick(EPI_DW, N, K, M, 0);
  if (px.bn == 512 || pw.bn == 512) return DET_OK;
  int bn = 0, lead = 0, grid = 0;
  bool w_first = false;
  double best = 0.0;
  for (int i = 1; i < 4; ++i) {
    const IgCost& c = IG_COST[i];
    if (K % c.bn) continue;
    const double loop[2] = {(N / BK) * c.step, (M / BK) * c.step}, epi[2] = {c.epi[EPI_DX], c.epi[EPI_DW]};
    const int tiles[2] = {(M / BM) * (K / c.bn), (N / BM) * (K / c.bn)};
    double each[2];
    for (int k = 0; k < 2; ++k) each[k] = (loop[k] > epi[k] ? loop[k] : epi[k]) + c.turn;
    const int f = each[1] > each[0], g = tiles[0] + tiles[1] < sms ? tiles[0] + tiles[1] : sms;    // f: the first product
    const int rest = tiles[f] % g, spare = g - rest, n = tiles[1 - f];
    int l = 0;
    if (rest) {
      l = (int)(each[f] / each[1 - f] + 0.5);
      if (l > (n + spare - 1) / spare) l = (n + spare - 1) / spare;
    }
    const int left = n > l * spare ? n - l * spare : 0;
    const double part = rest ? (each[f] > l * each[1 - f] ? each[f] : l * each[1 - f]) : 0.0;
    const double tail = loop[1 - f] < epi[1 - f] ? loop[1 - f] : epi[1 - f];
    const double t = (tiles[f] / g) * each[f] + part + ((left + g - 1) / g) * each[1 - f] + tail;
    if (!bn || t < best) { bn = c.bn; best = t; lead = l; grid = g; w_first = f; }
  }
  const double work = px.work + pw.work;
  if (fork ? best > behind_each_other(px, pw, sms) - ((size_t)M * (K / 64) <= SUM_CHUNK ? 5.0 : 9.0) || (bn == 256 && K >= 2048) || work > 70.0
           : best > work + 5.5)
    return DET_OK;
  IgProduct x = {}, w = {};
  if (!make_map(&x.a, A, M, N, 128) || !make_map(&x.b, Ut, K, N, bn) || !make_map(&w.a, Gt, N, M, 128) || !make_map(&w.b, Zt, K, M, bn))
    return DET_ERR_CUDA;
  x.ep = ex; x.I = M; x.K = N;
  w.ep = ew; w.I = N; w.K = M;
  *did = true;
  const IgProduct &p = w_first ? w : x, &s = w_first ? x : w;
  switch (bn) {
    case 256: return grads_tile<256>(w_first, p, s, K, grid, lead, status, st);
    case 128: return grads_tile<128>(w_first, p, s, K, grid, lead, status, st);
    default: return grads_tile<64>(w_first, p, s, K, grid, lead, status, st);
  }
}

}  // namespace det

using namespace det;

// Self-test of the bounded wait every tensor-core kernel relies on: one warp waits on an mbarrier that nothing ever
// completes; after `limit_cycles` the wait gives up, raises DET_DEV_TIMEOUT in *status_dev and the kernel returns.
__global__ void k_selftest_wait(int* status, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_s;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  mbar_wait(&bar, 0, &abort_s, status, limit);
}

extern "C" int det_test_wait_timeout(int* status_dev, long long limit_cycles, void* stream) {
  if (!status_dev || limit_cycles <= 0 || limit_cycles > 4000000000ll) return DET_ERR_ARG;
  k_selftest_wait<<<DET_L(1), 32, 0, (cudaStream_t)stream>>>(status_dev, limit_cycles);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

// Self-test of the wait of a whole warp: even lanes wait for a phase that is over, odd ones for one that nothing completes.
__global__ void k_selftest_wait_warp(int* gone_on, long long limit) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_s;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  gone_on[threadIdx.x] = mbar_wait_warp(&bar, threadIdx.x & 1 ? 0u : 1u, &abort_s, nullptr, limit);
}

extern "C" int det_test_wait_warp(int* gone_on, long long limit_cycles, void* stream) {
  if (!gone_on || limit_cycles <= 0 || limit_cycles > 4000000000ll) return DET_ERR_ARG;
  k_selftest_wait_warp<<<DET_L(1), 32, 0, (cudaStream_t)stream>>>(gone_on, limit_cycles);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_test_igemm_tn(const int8_t* A, const int8_t* B, int I, int J, int K, int32_t* C, int force_one_cta,
                                 void* stream, int* status_dev) {
  if (!C) return DET_ERR_ARG;
  if (!aligned16(C)) return DET_ERR_ALIGN;
  EpiParams ep = {};
  ep.out = C;
  return igemm_launch(EPI_RAW, A, B, I, J, K, ep, status_dev, (cudaStream_t)stream, force_one_cta);
}
