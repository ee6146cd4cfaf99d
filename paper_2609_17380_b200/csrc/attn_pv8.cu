// Attention forward with the P.V product of every block of 128 keys on the int8 tensor cores (Sec. 3.2: "int8 P.V per
// block; QK^T and softmax in higher precision").
//
// Per (batch, key/value head, block of 128 keys): s_v = absmax(V block) / 127, q_v = rne(clamp(v * (127 / absmax))).
// Per query row and block: q_p = rne(p * 127), p = exp(s - m) in [0, 1].  u = float(sum_j q_p q_v) * (s_v / 127): the
// integer sum is exact, so the tensor core's accumulation order does not matter.  Logits, running maximum, row sums
// and the rescale o = o * alpha + u stay in ordered f32 exactly as in the full-precision kernel (attn.cu); lse is the
// same as there.
//
// CTA = 128 queries of one (batch, head), one CTA per SM, warp-specialised like the full-precision kernel (attn.cu):
//   warps 0-15   consumers: 8 whole query rows each; logits on the FP32 pipe from the slab ring, softmax, quantised weights
//                (A operand, [query][key]) into shared memory in the 128-byte-swizzled K-major layout the MMA expects
//   warps 16-19  producers: the key block as eight 16-deep slabs into the ring, then the block absmax of V and the
//                quantised, transposed values (B operand, [dim][key]), double-buffered; between the two one thread issues
//                four tcgen05.mma.kind::i8 (M = N = 128, K = 32 each) of the block before into a 128-column TMEM accumulator
//                once both its operands are there, and commits to an mbarrier
// A consumer warp collects the product of block t after its logits of block t + 1, so the tensor-core product, the other warps'
// softmax and the quantisation of V run behind the multiply loop (with block-wide phases, each waiting for the one before,
// forward and backward of 16 heads x 4096 at window 512 took 1.69 ms, 1.55 now).  In that step a thread owns one query row and 32 output
// dimensions.  Every wait on an mbarrier is bounded: on expiry the kernel raises DET_DEV_TIMEOUT in *status, all roles skip what
// is left, and the kernel frees its TMEM and returns.
#include "attn_core.cuh"

namespace det {

constexpr int PQ = 128, PK = 128, PLQ = PQ + 4, PV_SLOTS = 4, PV_HS = 2;   // ring slots, 16-deep slabs of a slot
constexpr int PV_CONS = 512, PV_PROD = 128, PV_THREADS = PV_CONS + PV_PROD;
// shared memory: Q f32 [dim][query], the slab ring, then (1024-byte aligned) q_p int8 [query][key], q_v int8 [2][dim][key]
constexpr size_t PV8_SMEM = (size_t)(DH * PLQ + PV_SLOTS * PV_HS * OK * AF_BP) * sizeof(float) + 1024 + 3 * PQ * PK;
// setmaxnreg: 104 registers for consumers, 64 for producers
static_assert(PV_CONS * 104 + PV_PROD * 64 <= (65536 / PV_THREADS / 8 * 8) * PV_THREADS, "register hand-over exceeds the block's allocation");

// byte offset of element (row, col) of a 128 x 128 int8 K-major tile with 128-byte swizzle (16-byte chunks of a row
// are permuted by the row index modulo 8)
__device__ __forceinline__ int swz(int row, int col) { return row * 128 + ((((col >> 4) ^ (row & 7))) << 4) + (col & 15); }

__global__ void __launch_bounds__(PV_THREADS, 1)
    k_attn_fwd_pv8(const uint16_t* __restrict__ q, const uint16_t* __restrict__ k, const uint16_t* __restrict__ v, int ld, int H,
                   int Hkv, int S, int W, uint16_t* __restrict__ out, int ld_out, float* __restrict__ lse, int* status) {
  extern __shared__ __align__(16) unsigned char psm8[];
  float(*Qs)[PLQ] = reinterpret_cast<float(*)[PLQ]>(psm8);
  float(*Ring)[OK][AF_BP] = reinterpret_cast<float(*)[OK][AF_BP]>(psm8 + (size_t)DH * PLQ * sizeof(float));
  uint8_t* ops = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(psm8 + (size_t)(DH * PLQ + PV_SLOTS * PV_HS * OK * AF_BP) * sizeof(float)) + 1023) & ~(uintptr_t)1023);
  int8_t* Pq = reinterpret_cast<int8_t*>(ops);              // A operand: [query][key]
  int8_t* Vq = reinterpret_cast<int8_t*>(ops + PQ * PK);    // B operand: two buffers [dim][key]
  __shared__ float alpha_s[2][PQ], l_s[PQ], cs_s[4], vmax_s[2][4];
  __shared__ __align__(4) uint8_t tiny_s[PV_SLOTS][4];
  __shared__ int tiny_q_s, abort_s;
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bar_full[PV_SLOTS], bar_empty[PV_SLOTS], bar_p, bar_v[2], bar_mma;
  volatile int* abort_flag = &abort_s;

  const int qb = gridDim.y - 1 - blockIdx.y;  // longest rows first
  const int h = blockIdx.x % H, b = blockIdx.x / H, hk = h / (H / Hkv);
  const int q0 = qb * PQ;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t row0 = (size_t)b * S;
  const uint16_t* qp = q + row0 * ld + (size_t)h * DH;
  const uint16_t* kp = k + row0 * ld + (size_t)hk * DH;
  const uint16_t* vp = v + row0 * ld + (size_t)hk * DH;
  const int jt0 = (W > 0 && q0 > W) ? (q0 - W) / PK : 0, nt = q0 / PK + 1 - jt0;     // key blocks of this CTA

  if (tid == 0) {
    for (int s = 0; s < PV_SLOTS; ++s) { mbar_init(&bar_full[s], 4); mbar_init(&bar_empty[s], PV_CONS / 32); }
    mbar_init(&bar_p, PV_CONS / 32);
    mbar_init(&bar_v[0], 4);
    mbar_init(&bar_v[1], 4);
    mbar_init(&bar_mma, 1);
    abort_s = 0;
    tiny_q_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 16) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(128u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  {  // q^T of the query block, staged once by everybody
    bool tq = false;
    for (int idx = tid; idx < PQ * 16; idx += PV_THREADS) {
      const int r = idx % PQ, ch = idx / PQ;
      float t[8];
      if (q0 + r < S) unpack8a(__ldg(reinterpret_cast<const uint4*>(qp + (size_t)(q0 + r) * ld + ch * 8)), t);
      else {
#pragma unroll
        for (int x = 0; x < 8; ++x) t[x] = 0.0f;
      }
#pragma unroll
      for (int x = 0; x < 8; ++x) { tq |= tiny1(t[x]); Qs[ch * 8 + x][r] = t[x]; }
    }
    if (__any_sync(__activemask(), tq) && lane == 0) atomicOr(&tiny_q_s, 1);
  }
  __syncthreads();

  if (warp >= 16) {
    // ------------------------------- producers -------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const int pt = tid - PV_CONS, pw = pt >> 5;
    const int kk = 2 * (pt & 63), kd = (pt >> 6) * 8;   // K: keys kk and kk + 1 of a block, dimensions kd .. kd + 7 of a slab
    const int kcol = (kk & 4 ? AF_HI : 0) + (kk >> 3) * 4 + (kk & 3);
    int slot = 0;
    uint32_t par = 1;
    bool ok = true;                                  // after a failed wait nothing is staged, but every barrier below is still met
    constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(DH >> 3) << 17) | ((uint32_t)(PQ >> 4) << 24);
    auto product = [&](int t) {                      // of block t, by one thread, once weights and values are there
      if (pt == 0 && mbar_wait(&bar_v[t & 1], (uint32_t)(t >> 1) & 1u, abort_flag, status) &&
          mbar_wait(&bar_p, (uint32_t)t & 1u, abort_flag, status)) {
        tc_fence_after();
        const uint64_t da = make_smem_desc(smem_u32(Pq)), db = make_smem_desc(smem_u32(Vq + (t & 1) * (PQ * PK)));
#pragma unroll
        for (int k4 = 0; k4 < PK / 32; ++k4) umma_i8(tmem_base, da + (uint64_t)(k4 * 2), db + (uint64_t)(k4 * 2), idesc, k4 ? 1u : 0u);
        umma_commit(&bar_mma);
      }
      __syncwarp();
    };
    for (int t = 0; t < nt; ++t) {
      const int j0 = (jt0 + t) * PK;
      {  // K: slab sl holds head dimensions 16 sl .. of the 128 keys, four slabs in flight; keys past the last one repeat it, they are never visible
        const uint4* src0 = reinterpret_cast<const uint4*>(kp + (size_t)min(j0 + kk, S - 1) * ld + kd);
        const uint4* src1 = reinterpret_cast<const uint4*>(kp + (size_t)min(j0 + kk + 1, S - 1) * ld + kd);
        uint4 raw[4][2];
        auto fetch = [&](int sl, uint4 (&w)[2]) { w[0] = __ldg(src0 + 2 * sl); w[1] = __ldg(src1 + 2 * sl); };
#pragma unroll
        for (int d = 0; d < 4; ++d) fetch(d, raw[d]);
        uint32_t least = ~0u;
#pragma unroll
        for (int sl = 0; sl < 8; ++sl) {
          const int sub = sl % PV_HS;
          if (sub == 0) {
            ok = ok && mbar_wait(&bar_empty[slot], par, abort_flag, status);
            least = ~0u;
          }
          const uint4 w0 = raw[sl & 3][0], w1 = raw[sl & 3][1];
          const uint32_t words[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
          if (ok) {
            float(*dst)[AF_BP] = Ring[slot * PV_HS + sub];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              word_least(words[i], least);
              word_least(words[4 + i], least);
              *reinterpret_cast<float2*>(&dst[kd + 2 * i][kcol]) = make_float2(word_lo(words[i]), word_lo(words[4 + i]));
              *reinterpret_cast<float2*>(&dst[kd + 2 * i + 1][kcol]) = make_float2(word_hi(words[i]), word_hi(words[4 + i]));
            }
          }
          if (sl < 4) fetch(sl + 4, raw[sl & 3]);
          if (sub < PV_HS - 1) continue;
          const int any = __any_sync(0xffffffffu, least_tiny(least));
          if (lane == 0) { tiny_s[slot][pw] = (uint8_t)any; }
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar_full[slot]);
          if (++slot == PV_SLOTS) { slot = 0; par ^= 1u; }
        }
      }
      if (t > 0) product(t - 1);
      // V: block absmax (128 keys x 128 dims), then the quantised transposed operand
      float vm = 0.0f;
#pragma unroll 8
      for (int it = 0; it < 16; ++it) {
        const int key = j0 + it * 8 + (pt >> 4);
        if (key < S) {
          float x[8];
          unpack8a(__ldg(reinterpret_cast<const uint4*>(vp + (size_t)key * ld + (pt & 15) * 8)), x);
#pragma unroll
          for (int e = 0; e < 8; ++e) vm = fmaxf(vm, fabsf(x[e]));
        }
      }
#pragma unroll
      for (int w = 16; w; w >>= 1) vm = fmaxf(vm, __shfl_xor_sync(0xffffffffu, vm, w));
      if (lane == 0) vmax_s[t & 1][pw] = vm;
      // past this barrier the products up to block t - 2 are done and buffer t & 1 is free: the first warp has been through
      // product(t - 1), which every consumer warp announced only after it had collected block t - 2
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const float am = fmaxf(fmaxf(vmax_s[t & 1][0], vmax_s[t & 1][1]), fmaxf(vmax_s[t & 1][2], vmax_s[t & 1][3]));
      const float s_v = (am > 0.0f) ? fdiv(am, 127.0f) : 0.0f, inv_v = (am > 0.0f) ? fdiv(127.0f, am) : 0.0f;
      if (ok) {
        if (pt == 0) cs_s[t & 3] = fdiv(s_v, 127.0f);
        int8_t* dst = Vq + (t & 1) * (PQ * PK);
        const int key = j0 + 4 * lane;               // four adjacent keys x eight dimensions a step: one word per dimension
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int ch = pw * 4 + c;
          uint4 u[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            u[i] = key + i < S ? __ldg(reinterpret_cast<const uint4*>(vp + (size_t)(key + i) * ld + ch * 8)) : make_uint4(0u, 0u, 0u, 0u);
          float x[4][8];
#pragma unroll
          for (int i = 0; i < 4; ++i) unpack8a(u[i], x[i]);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            uint32_t w = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) w |= (uint32_t)(uint8_t)quant1(x[i][e], inv_v) << (8 * i);
            *reinterpret_cast<uint32_t*>(dst + swz(ch * 8 + e, 4 * lane)) = w;
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_v[t & 1]);
    }
    product(nt - 1);
  } else {
    // ------------------------------- consumers -------------------------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int tiny_q = tiny_q_s;
    const int wrow = warp * AF_RW, r2 = lane & 1, tx = lane >> 1, lrow = wrow + 4 * r2;
    // accumulator phase: this thread owns query row orow and the 32 output dimensions starting at ocol
    const int orow = (warp & 3) * 32 + lane, ocol = (warp >> 2) * 32;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ocol;
    const float2 one = same2(c_one);
    float m_mine = __int_as_float(0xff800000), l_mine = 0.0f, alpha_mine = 0.0f;   // row ROW_OF_LANE(lane) of the warp
    float2 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = make_float2(0.0f, 0.0f);
    // o = o * alpha + u of block t, once its product is there
    auto collect = [&](int t) -> bool {
      // the TMEM load below is warp-collective
      if (!mbar_wait_warp(&bar_p, (uint32_t)t & 1u, abort_flag, status) || !mbar_wait_warp(&bar_mma, (uint32_t)t & 1u, abort_flag, status)) return false;
      tc_fence_after();
      const float2 al = same2(alpha_s[t & 1][orow]), cs = same2(cs_s[t & 3]);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t r[16];
        tmem_ld16_nowait(taddr + 16 * hf, r);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float2 u = make_float2(__int2float_rn((int)r[2 * c]), __int2float_rn((int)r[2 * c + 1]));
          o[8 * hf + c] = add2(mul2(o[8 * hf + c], al), mul2(u, cs), one);
        }
      }
      tc_fence_before();
      return true;
    };
    bool ok = true;
    int slot = 0;
    uint32_t par = 0;
    for (int t = 0; t < nt && ok; ++t) {
      const int j0 = (jt0 + t) * PK;
      const bool diag = t == nt - 1;                 // only the last block of a row block reaches past the diagonal
      const bool edge = W > 0 && j0 <= q0 + PQ - 1 - W;  // some row's window starts inside or after this block
      float2 acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
      for (int sl = 0; sl < 8; sl += PV_HS) {
        ok = mbar_wait_warp(&bar_full[slot], par, abort_flag, status);
        if (!ok) break;
        const bool tiny = tiny_q != 0 || *reinterpret_cast<const uint32_t*>(tiny_s[slot]) != 0;
#pragma unroll 1
        for (int sub = 0; sub < PV_HS; ++sub) {
          const float* ap = &Qs[(sl + sub) * OK][lrow];
          if (tiny) mac_4x8<false, false>(ap, PLQ, 0, 0, Ring[slot * PV_HS + sub], tx, acc);
          else mac_4x8<true, false>(ap, PLQ, 0, 0, Ring[slot * PV_HS + sub], tx, acc);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_empty[slot]);
        if (++slot == PV_SLOTS) { slot = 0; par ^= 1u; }
      }
      if (ok && t > 0) ok = collect(t - 1);
      if (!ok) break;
      const float sum = softmax_block(acc, j0 + 8 * tx, q0 + lrow, q0 + wrow + ROW_OF_LANE(lane), j0 + PK - 1, W, diag, edge, lane,
                                      m_mine, alpha_mine, one, [](float m) { return m; }, [](float) {});
      l_mine = fadd(fmul(l_mine, alpha_mine), sum);
      if (lane < AF_RW) alpha_s[t & 1][wrow + ROW_OF_LANE(lane)] = alpha_mine;
      // q_p = rne(127 p) of the lane's 4 x 8 weights (0 <= 127 p <= 127: adding 1.5 2^23 leaves the integer in the low byte)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t w[2];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const float2 x = add2(mul2(acc[i][2 * g], same2(127.0f)), same2(12582912.0f), one);
          const float2 y = add2(mul2(acc[i][2 * g + 1], same2(127.0f)), same2(12582912.0f), one);
          w[g] = __byte_perm(__byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x0040),
                             __byte_perm(__float_as_uint(y.x), __float_as_uint(y.y), 0x0040), 0x5410);
        }
        *reinterpret_cast<uint2*>(Pq + swz(lrow + i, 8 * tx)) = make_uint2(w[0], w[1]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_p);
    }
    if (ok) ok = collect(nt - 1);
    // row sums travel from the logit mapping (a lane per row) to the accumulator mapping (a row per thread)
    if (lane < AF_RW) {
      const int r = wrow + ROW_OF_LANE(lane);
      l_s[r] = l_mine;
      if (q0 + r < S && ok) lse[((size_t)b * H + h) * S + q0 + r] = fadd(m_mine, det_log(l_mine));
    }
    asm volatile("bar.sync 2, 512;" ::: "memory");
    const int row = q0 + orow;
    if (row < S && ok) {
      const float il = fdiv(1.0f, l_s[orow]);
      uint16_t* op = out + (row0 + row) * ld_out + (size_t)h * DH + ocol;
#pragma unroll
      for (int c = 0; c < 16; c += 4) {
        uint4 w;
        w.x = pack_bf2(fmul(o[c].x, il), fmul(o[c].y, il));
        w.y = pack_bf2(fmul(o[c + 1].x, il), fmul(o[c + 1].y, il));
        w.z = pack_bf2(fmul(o[c + 2].x, il), fmul(o[c + 2].y, il));
        w.w = pack_bf2(fmul(o[c + 3].x, il), fmul(o[c + 3].y, il));
        *reinterpret_cast<uint4*>(op + 2 * c) = w;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (abort_s) {   // give copies and products in flight time to land before the TMEM goes
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
    __syncthreads();
  }
  if (warp == 16) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(128u) : "memory");
  }
}

}  // namespace det

using namespace det;

extern "C" int det_attn_fwd_int8pv(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S,
                                   int window, det_bf16* out, int ld_out, float* lse, void* stream, int* status_dev) {
  if (!q || !k || !v || !out || !lse || B <= 0 || H <= 0 || Hkv <= 0 || S <= 0 || window < 0) return DET_ERR_ARG;
  if (S % 64 || ld % 8 || ld_out % 8 || ld < H * DH || ld_out < H * DH || H % Hkv || window % 128) return DET_ERR_SHAPE;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out)) return DET_ERR_ALIGN;
  static DevOnce once = {};
  if (dev_ensure_smem(once, (const void*)k_attn_fwd_pv8, PV8_SMEM) != DET_OK) return DET_ERR_CUDA;
  dim3 grid(H * B, (S + PQ - 1) / PQ);
  k_attn_fwd_pv8<<<DET_L(grid), PV_THREADS, PV8_SMEM, (cudaStream_t)stream>>>(q, k, v, ld, H, Hkv, S, window, out, ld_out, lse, status_dev);
  DET_CHECK_LAUNCH();
  return DET_OK;
}
