// Causal attention, head_dim 128, in a fixed order on the FP32 ALUs (Sec. 3.2: QK^T and softmax stay in
// higher precision; the backward recomputes the weights in full precision and is not quantised).
//
// Forward: online softmax over KV tiles of 128 keys in ascending order.  Each logit is a sequential
// ascending sum over the 128 head dimensions of exact bf16 products; the tile's row sum is the adjacent
// pairwise tree over its 128 slots (masked slots are +0); P is rounded to bf16 before P.V; P.V is a
// sequential ascending sum over the tile's keys from +0, then o = o*alpha + u.
// Backward: P = exp(S*scale - L) recomputed; every one of the five contractions (S, dP, dV, dK, dQ) is a batched
// ordered contraction with one sequential accumulator per output (ogemm_core.cuh); bf16(P) and bf16(dS) go through
// global scratch, so nothing is accumulated with atomics.
#include <math.h>
#include "attn_core.cuh"

namespace det {

// ---------------------------------------------------------------------------------------------
// forward, warp-specialised; CTA = FQ queries of one (batch, head).
//
// A consumer warp owns 8 whole query rows: lane 2t + r holds rows 4r .. 4r+3 and 8 columns (keys 8t .. 8t+7 while the logits
// are formed, head dimensions {4t.., 64 + 4t..} during P.V).  The row operand (q^T [dim][query], P~ [key][query] in
// shared memory) is one 16-byte load of two cycles, the column operand two loads of two cycles (neighbouring lanes read the
// same word), for 16 packed multiply-adds; with 8 rows x 4 columns a lane the column load alone took four cycles and the
// shared-memory port was busy all the time (4 x 16 heads x 2048: 1.56 -> 1.48 ms).  A row's 128 logits of a key block sit in one warp, so its
// maximum and its row sum (the adjacent pairwise tree: eight slots in the lane, then lanes 2, 4, 8, 16 apart) are warp
// shuffles, P~ of the warp's rows is written and read by that warp alone, and the running maximum, sum and rescale factor
// of a row live in one lane.
// K and V arrive through an mbarrier-guarded ring of 16-deep slabs filled by four producer warps (K: 16 head dimensions
// x 128 keys, eight per block; V: 16 keys x 128 dimensions, eight per block), so no block-wide barrier is left in the
// loop and consumer warps are not coupled to each other.  The softmax evaluates its 32 exponentials per lane two at a time
// as one straight-line block of branch-free chains and reduces the 8 rows with 5 shuffles per reduction.
// On the diagonal block a warp stops P.V after the last key any of its rows may see.
// WIN: row i sees the keys j in (i - W, i] (W a multiple of 128): the tile loop starts at the tile of q0 - W, and a row
// skips a tile that holds none of its keys (its statistics stay untouched: alpha = 1, all weights 0).
// Hkv key/value heads serve H query heads (head h reads key/value head h / (H/Hkv)).
// ---------------------------------------------------------------------------------------------
// Rows per CTA, ring slots, slabs in flight in the producers' registers, CTAs per SM, registers per consumer and producer thread after the hand-over.
// The registers go to the consumers, whose loops spill and reload with fewer: one slab in flight leaves them eight to sixteen more than
// three or four did (64 heads x 2048, 128 rows, 104 and 112: 1447 and 1415 us; 4 x 4096, 64 rows, 96 and 104: 494 and 479; 20 x 1024,
// 32 rows, 104, 112 and 120: 170, 153 and 149; 8 x 1024, two groups, 136 and 160: 78.3 and 76.5), and the other warps cover the loads.
// A CTA of 128 rows has the best rate (23.9 us per row block and key block on a full GPU, against 12.1 us for 64 rows and
// 6.5 us for 32), but its chain of key blocks is the longest: alone on its SM 23.5, 15.0 and 9.8 us per key block.
// GR groups of consumer and producer warps take the key blocks of the CTA's rows in turn: logits and P.V of a block need nothing of
// the block before but its running maximum, which passes from warp to warp through shared memory, and group 1 hands its u, row
// sums and rescale factors to group 0, which alone forms o and l, in block order.  Two groups shorten the chain, 9.8 to 8.6 us per
// key block, and lose rate (8.6 against 6.5 us per 32 rows and key block): 8 heads x 1024 98 us with 32 rows, 76 with two groups;
// 16 x 832 106 and 102; 16 x 1088 151 and 163.
// Slabs of a ring slot.  The kernel is bound by issue slots (twice the packed multiply-adds plus all other instructions come to 98 % of the
// cycles), and a hand-over takes a consumer warp some 70 of them: one for two slabs instead of one a slab, waited for where it is needed
// instead of a slab ahead, with two keys a store in the producers (see OgSide) took 16 heads x 832 from 116 to 107 us.
constexpr int AF_HS = 2;
template <int FQ_, int SLOTS_, int PF_, int CPS_, int RC_, int RP_, int GR_ = 1>
struct AfTile {
  static constexpr int FQ = FQ_, LQ = FQ_ + 4, SLOTS = SLOTS_, PF = PF_, CPS = CPS_, RC = RC_, RP = RP_, GR = GR_;
  static constexpr int GCONS = (FQ / AF_RW) * 32, CONS = GR * GCONS, THREADS = CONS + GR * AF_PROD;
  static constexpr size_t SMEM = (size_t)(DH * LQ + GR * (FK * FQ + SLOTS * AF_HS * OK * AF_BP) + (GR - 1) * FQ * DH) * sizeof(float);
  static_assert(FQ % (AF_HS * OK) == 0, "the last slot of value rows is whole");
  // setmaxnreg: the counts after the hand-over must fit into what the block was launched with, or the increase never returns
  static_assert(CONS * RC + GR * AF_PROD * RP <= (65536 / (CPS * THREADS) / 8 * 8) * THREADS, "register hand-over exceeds the block's allocation");
};
typedef AfTile<128, 4, 1, 1, 112, 32> AfTall;
typedef AfTile<64, 2, 1, 2, 104, 32> AfHalf;
typedef AfTile<32, 2, 1, 3, 120, 40> AfShort;
typedef AfTile<32, 2, 3, 1, 160, 96, 2> AfPair;

template <class T, bool WIN>
__global__ void __launch_bounds__(T::THREADS, T::CPS)
    k_attn_fwd(const uint16_t* __restrict__ q, const uint16_t* __restrict__ k, const uint16_t* __restrict__ v, int ld,
               int H, int Hkv, int S, int Warg, uint16_t* __restrict__ out, int ld_out, float* __restrict__ lse,
               const float* __restrict__ s_q, int8_t* __restrict__ qout, int sms) {
  constexpr int FQ = T::FQ, LQ = T::LQ, AF_SLOTS = T::SLOTS, AF_PF = T::PF, AF_CONS = T::CONS, AF_THREADS = T::THREADS, GR = T::GR;
  constexpr int GWARPS = T::GCONS / 32;
  const int W = WIN ? Warg : 0;
  extern __shared__ __align__(16) float sm[];
  float(*Qs)[LQ] = reinterpret_cast<float(*)[LQ]>(sm);                         // [dim][query]
  __shared__ __align__(4) uint8_t tiny_g[GR][AF_SLOTS][AF_PROD / 32];
  __shared__ int tiny_q_s, abort_s;
  __shared__ __align__(8) uint64_t full_g[GR][AF_SLOTS], empty_g[GR][AF_SLOTS];
  // between the two groups, per warp: maxima passed on by either, group 1's sums and factors, "u is there", "u has been read"
  __shared__ float max_g[GR][FQ], sum_g[FQ], alpha_g[FQ];
  __shared__ __align__(8) uint64_t bar_max[GR][GWARPS], bar_u[GWARPS], bar_ufree[GWARPS];
  volatile int* abort_flag = &abort_s;
  // Longest rows first.  With two CTAs per SM the first two rounds over the SMs are resident together, one of each on an SM: the
  // second one runs backwards, so that a long row has a short one beside it (two sequences of 8 heads x 1088, 64 rows: 0.181 -> 0.157
  // ms; 32 heads x 512 0.090 -> 0.078; with three CTAs per SM the order of placement is another one, 16 heads x 832, 32 rows: 0.119 and 0.129)
  int c = blockIdx.y * gridDim.x + blockIdx.x;
  if (T::CPS == 2 && c >= sms && c < 2 * sms) c = sms + min(2 * sms, (int)(gridDim.x * gridDim.y)) - 1 - c;
  const int qb = gridDim.y - 1 - c / gridDim.x, bh = c % gridDim.x;
  const int h = bh % H, b = bh / H, hk = h / (H / Hkv);
  const int q0 = qb * FQ;
  const int tid = threadIdx.x, lane = tid & 31;
  const int grp = GR == 1 ? 0 : (tid < AF_CONS ? tid / T::GCONS : (tid - AF_CONS) / AF_PROD), warp = (tid >> 5) - grp * GWARPS;   // consumers' warp
  float* Ps = sm + DH * LQ + grp * (FK * FQ);                                  // [key][query], 16-byte chunks swizzled
  float(*Ring)[OK][AF_BP] = reinterpret_cast<float(*)[OK][AF_BP]>(sm + DH * LQ + GR * FK * FQ) + grp * (AF_SLOTS * AF_HS);
  float4* U = reinterpret_cast<float4*>(sm + DH * LQ + GR * (FK * FQ + AF_SLOTS * AF_HS * OK * AF_BP));   // [4][thread of the group]
  uint8_t(*tiny_s)[AF_PROD / 32] = tiny_g[grp];
  uint64_t *bar_full = full_g[grp], *bar_empty = empty_g[grp];
  const size_t row0 = (size_t)b * S;
  const uint16_t* qp = q + row0 * ld + (size_t)h * DH;
  const uint16_t* kp = k + row0 * ld + (size_t)hk * DH;
  const uint16_t* vp = v + row0 * ld + (size_t)hk * DH;
  const int jt0 = ((WIN && q0 > W) ? (q0 - W) / FK : 0) + grp, ntiles = q0 / FK + 1;   // this group's first block
  // the last block ends with the last slab of 16 value rows that the CTA's last query may see, and with that a slot (FQ % 32 = 0)
  const int mine = ntiles > jt0 ? (ntiles - jt0 + GR - 1) / GR : 0;
  const int nslab = mine * 16 - ((ntiles - 1 - jt0) % GR == 0 && mine ? 7 - (q0 % FK + FQ - 1) / OK : 0);
  if (tid == 0) {
    for (int g = 0; g < GR; ++g)
      for (int s = 0; s < AF_SLOTS; ++s) { mbar_init(&full_g[g][s], AF_PROD / 32); mbar_init(&empty_g[g][s], GWARPS); }
    if (GR > 1)
      for (int w = 0; w < GWARPS; ++w) { mbar_init(&bar_max[0][w], 1); mbar_init(&bar_max[GR - 1][w], 1); mbar_init(&bar_u[w], 1); mbar_init(&bar_ufree[w], 1); }
    tiny_q_s = 0;
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  {  // q^T of the query block, staged once by everybody
    bool tq = false;
    for (int idx = tid; idx < FQ * 16; idx += AF_THREADS) {
      const int r = idx % FQ, ch = idx / FQ;
      float t[8];
      if (q0 + r < S) unpack8a(__ldg(reinterpret_cast<const uint4*>(qp + (size_t)(q0 + r) * ld + ch * 8)), t);
      else {
#pragma unroll
        for (int x = 0; x < 8; ++x) t[x] = 0.0f;
      }
#pragma unroll
      for (int x = 0; x < 8; ++x) { tq |= tiny1(t[x]); Qs[ch * 8 + x][r] = t[x]; }
    }
    if (__any_sync(0xffffffffu, tq) && lane == 0) atomicOr(&tiny_q_s, 1);
  }
  __syncthreads();
  if (tid >= AF_CONS) {
    // ------------------------------- producers -------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(T::RP));
    const int pt = (tid - AF_CONS) % AF_PROD, pw = pt >> 5;
    // Slab s of the block sequence: block s / 16; s % 16 < 8: K, head dimensions 16 (s % 16) .. (thread = eight of them, of two
    // neighbouring keys); else V, keys 16 (s % 16 - 8) .. (thread = four dimensions of keys kk, kk + 4, kk + 8, kk + 12).
    // AF_PF slabs are in flight in registers, so that the latency of a global load is spread over several slabs.
    // Both kinds are two 16-byte words per thread, so one register array holds whichever kind slab s is.
    uint4 raw[AF_PF][2];
    const int vf = pt & 31, vk = pt >> 5;            // V: dimensions 4 vf .. 4 vf + 3 of keys vk, vk + 4, vk + 8, vk + 12
    const int kk = 2 * (pt & 63), kd = (pt >> 6) * 8;   // K: keys kk and kk + 1, dimensions kd .. kd + 7 of the slab
    const size_t row = (size_t)ld * 2;
    // keys past the last one repeat it: they are never visible.  ksrc, vsrc: this thread's words of the block's first slab
    const char *ksrc0, *ksrc1, *vsrc;
    int vleft;                                       // keys of the sequence from the thread's first one on
    auto block = [&](int j0n) {
      ksrc0 = reinterpret_cast<const char*>(kp + kd) + min(j0n + kk, S - 1) * row;
      ksrc1 = reinterpret_cast<const char*>(kp + kd) + min(j0n + kk + 1, S - 1) * row;
      vsrc = reinterpret_cast<const char*>(vp + 4 * vf) + (j0n + vk) * row;
      vleft = S - (j0n + vk);
    };
    block(jt0 * FK);
    auto fetch = [&](int sn, uint4 (&w)[2]) {
      if (sn >= nslab) return;
      const int phn = sn & 15;
      if (phn == 0 && sn) block((jt0 + GR * (sn >> 4)) * FK);
      if (phn < 8) {
        w[0] = __ldg(reinterpret_cast<const uint4*>(ksrc0));
        w[1] = __ldg(reinterpret_cast<const uint4*>(ksrc1));
        ksrc0 += 2 * OK;
        ksrc1 += 2 * OK;
      } else {
        uint2 u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          u[i] = 4 * i < vleft ? __ldg(reinterpret_cast<const uint2*>(vsrc)) : make_uint2(0u, 0u);
          vsrc += 4 * row;
        }
        vleft -= OK;
        w[0] = make_uint4(u[0].x, u[0].y, u[1].x, u[1].y);
        w[1] = make_uint4(u[2].x, u[2].y, u[3].x, u[3].y);
      }
    };
    // unpack, test for factors below 2^-63 and store: K as [dimension][key], two keys at a time, V as [key][dimension]
    const int kcol = (kk & 4 ? AF_HI : 0) + (kk >> 3) * 4 + (kk & 3), vcol = 4 * vf + (vf >= 16 ? AF_HI - 64 : 0);
    auto store = [&](int ph, float (*dst)[AF_BP], const uint4 (&w)[2], uint32_t& least) {
      const uint32_t words[8] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w};
#pragma unroll
      for (int i = 0; i < 8; ++i) word_least(words[i], least);
      if (ph < 8) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          *reinterpret_cast<float2*>(&dst[kd + 2 * i][kcol]) = make_float2(word_lo(words[i]), word_lo(words[4 + i]));
          *reinterpret_cast<float2*>(&dst[kd + 2 * i + 1][kcol]) = make_float2(word_hi(words[i]), word_hi(words[4 + i]));
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          *reinterpret_cast<float4*>(&dst[vk + 4 * i][vcol]) =
              make_float4(word_lo(words[2 * i]), word_hi(words[2 * i]), word_lo(words[2 * i + 1]), word_hi(words[2 * i + 1]));
      }
    };
#pragma unroll
    for (int d = 0; d < AF_PF; ++d) fetch(d, raw[d]);
    int slot = 0;
    uint32_t par = 1, least = ~0u;
    for (int s0 = 0; s0 < nslab; s0 += AF_PF) {
#pragma unroll
      for (int d = 0; d < AF_PF; ++d) {
        const int s = s0 + d, sub = s % AF_HS;
        if (s >= nslab) return;
        if (sub == 0) {
          if (!mbar_wait(&bar_empty[slot], par, abort_flag, nullptr)) return;
          least = ~0u;
        }
        store(s & 15, Ring[slot * AF_HS + sub], raw[d], least);
        fetch(s + AF_PF, raw[d]);
        if (sub < AF_HS - 1) continue;
        const int any = __any_sync(0xffffffffu, least_tiny(least));
        if (lane == 0) tiny_s[slot][pw] = (uint8_t)any;
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_full[slot]);
        if (++slot == AF_SLOTS) { slot = 0; par ^= 1u; }
      }
    }
    return;
  }
  // --------------------------------- consumers ---------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(T::RC));
  const int tiny_q = tiny_q_s;
  const int wrow = warp * AF_RW;                      // first row of this warp inside the query block
  float m_mine = __int_as_float(0xff800000), l_mine = 0.0f, alpha_mine = 0.0f;   // row ROW_OF_LANE(lane) of the warp
  const int r2 = lane & 1, tx = lane >> 1, lrow = wrow + 4 * r2;   // this lane's rows lrow .. lrow + 3, columns of tx
  const float2 one = same2(c_one);
  float2 o[4][4];                                     // row lrow + i, column pair j
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) o[i][j] = make_float2(0.0f, 0.0f);
  bool ok = true;
  int slot = 0;
  uint32_t par = 0;
  // the next slot is full: its below-2^-63 flags
  auto acquire = [&](bool& tiny) -> bool {
    if (!mbar_wait(&bar_full[slot], par, abort_flag, nullptr)) return false;
    tiny = *reinterpret_cast<const uint32_t*>(tiny_s[slot]) != 0;
    return true;
  };
  auto release = [&]() {
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar_empty[slot]);
    if (++slot == AF_SLOTS) { slot = 0; par ^= 1u; }
  };
  // o = o * alpha + u and l = l * alpha + sum of group 1's block of round `rd`
  auto take = [&](int rd) -> bool {
    if (!mbar_wait_warp(&bar_u[warp], (uint32_t)rd & 1u, abort_flag, nullptr)) return false;
    const int own = wrow + ROW_OF_LANE(lane);
    l_mine = fadd(fmul(l_mine, alpha_g[own]), sum_g[own]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 al = same2(alpha_g[lrow + i]);
      const float4 x = U[(2 * i) * T::GCONS + tid], y = U[(2 * i + 1) * T::GCONS + tid];
      const float2 u[4] = {make_float2(x.x, x.y), make_float2(x.z, x.w), make_float2(y.x, y.y), make_float2(y.z, y.w)};
#pragma unroll
      for (int j = 0; j < 4; ++j) o[i][j] = add2(mul2(o[i][j], al), u[j], one);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&bar_ufree[warp]);
    return true;
  };
  int rd = 0;
  for (int jt = jt0; jt < ntiles && ok; jt += GR, ++rd) {
    const int j0 = jt * FK;
    const bool diag = (jt == ntiles - 1);           // only the last block of a row block reaches past the diagonal
    const bool edge = WIN && j0 <= q0 + FQ - 1 - W;  // some row's window starts inside or after this block
    // ---- logits: sum over the 128 dimensions ascending of q[row][d] k[key][d], keys 8 tx .. 8 tx + 7 ----
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
    for (int sl = 0; sl < 8; sl += AF_HS) {
      bool tiny;
      if (!acquire(tiny)) { ok = false; break; }
      tiny |= tiny_q != 0;
#pragma unroll 1
      for (int sub = 0; sub < AF_HS; ++sub) {
        const float* ap = &Qs[(sl + sub) * OK][lrow];
        if (tiny) mac_4x8<false, false>(ap, LQ, 0, 0, Ring[slot * AF_HS + sub], tx, acc);
        else mac_4x8<true, false>(ap, LQ, 0, 0, Ring[slot * AF_HS + sub], tx, acc);
      }
      release();
    }
    if (!ok) break;
    // ---- online softmax of the warp's 8 rows; the row sums take the weights before their rounding to bf16 ----
    const float sum = softmax_block(
        acc, j0 + 8 * tx, q0 + lrow, q0 + wrow + ROW_OF_LANE(lane), j0 + FK - 1, W, diag, edge, lane, m_mine, alpha_mine, one,
        [&](float m) {
          if (GR == 1 || (grp == 0 && rd == 0)) return m;
          ok = mbar_wait_warp(&bar_max[GR - 1 - grp][warp], (uint32_t)(grp ? rd : rd - 1) & 1u, abort_flag, nullptr);
          return max_g[GR - 1 - grp][wrow + ROW_OF_LANE(lane)];
        },
        [&](float m) {
          if (GR == 1) return;
          if (lane < AF_RW) max_g[grp][wrow + ROW_OF_LANE(lane)] = m;
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar_max[grp][warp]);
        });
    if (!ok) break;
    uint32_t tw = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t w = pack_bf2(acc[i][j].x, acc[i][j].y);
        word_tiny(w, tw);
        acc[i][j] = make_float2(word_lo(w), word_hi(w));
      }
    const bool tp = words_tiny(tw);
    // P~ of the lane's rows: key rows 8 tx + c, one chunk of four rows each
    __syncwarp();                                    // the previous block's P.V loads are done
    float* pchunk = Ps + (size_t)(8 * tx) * FQ + (((lrow >> 2) ^ ((tx & 3) << 1)) << 2);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      *reinterpret_cast<float4*>(pchunk + (2 * j) * FQ) = make_float4(acc[0][j].x, acc[1][j].x, acc[2][j].x, acc[3][j].x);
      *reinterpret_cast<float4*>(pchunk + (2 * j + 1) * FQ) = make_float4(acc[0][j].y, acc[1][j].y, acc[2][j].y, acc[3][j].y);
    }
    const int tiny_p = __any_sync(0xffffffffu, tp);  // also orders the stores before the loads below
    __syncwarp();
    // ---- u = P~ . V over the block's keys ascending from +0, then o = o * alpha + u ----
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
    // on the diagonal the warp's rows see no key beyond its last row, the CTA's none beyond its own last row
    const int last_slab = diag ? (q0 - j0 + wrow + AF_RW - 1) / OK : 7, last_block = diag ? (q0 - j0 + FQ - 1) / OK : 7;
    for (int sl = 0; sl <= last_block; sl += AF_HS) {
      bool tiny;
      if (!acquire(tiny)) { ok = false; break; }
      tiny |= tiny_p != 0;
#pragma unroll 1
      for (int sub = 0; sub < AF_HS && sl + sub <= last_slab; ++sub) {
        const float* ap = Ps + (size_t)((sl + sub) * OK) * FQ;
        if (tiny) mac_4x8<false, true>(ap, FQ, lrow >> 2, sub * OK, Ring[slot * AF_HS + sub], tx, acc);
        else mac_4x8<true, true>(ap, FQ, lrow >> 2, sub * OK, Ring[slot * AF_HS + sub], tx, acc);
      }
      release();
    }
    if (!ok) break;
    if (GR > 1 && grp == 1) {   // hand u over once the last one has been read
      if (rd > 0 && !mbar_wait_warp(&bar_ufree[warp], (uint32_t)(rd - 1) & 1u, abort_flag, nullptr)) { ok = false; break; }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        U[(2 * i) * T::GCONS + tid - T::GCONS] = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
        U[(2 * i + 1) * T::GCONS + tid - T::GCONS] = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
      }
      if (lane < AF_RW) { sum_g[wrow + ROW_OF_LANE(lane)] = sum; alpha_g[wrow + ROW_OF_LANE(lane)] = alpha_mine; }
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_u[warp]);
      continue;
    }
    if (GR > 1 && rd > 0 && !take(rd - 1)) { ok = false; break; }
    l_mine = fadd(fmul(l_mine, alpha_mine), sum);
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // the product o * alpha is rounded before the add
      const float2 al = same2(__shfl_sync(0xffffffffu, alpha_mine, LANE_OF_ROW(i)));
#pragma unroll
      for (int j = 0; j < 4; ++j) o[i][j] = add2(mul2(o[i][j], al), acc[i][j], one);
    }
  }
  if (!ok || grp) return;
  if (GR > 1 && (ntiles - jt0) % GR == 0) {   // the last block was group 1's
    if (!take(rd - 1)) return;
    m_mine = max_g[GR - 1][wrow + ROW_OF_LANE(lane)];
  }
  const float il_mine = fdiv(1.0f, l_mine);
  const float lse_mine = fadd(m_mine, det_log(l_mine));
  if (lane < AF_RW && q0 + wrow + ROW_OF_LANE(lane) < S) lse[((size_t)b * H + h) * S + q0 + wrow + ROW_OF_LANE(lane)] = lse_mine;
  const float inv_q = qout ? fdiv(1.0f, s_q[0]) : 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = q0 + lrow + i;
    const float il = __shfl_sync(0xffffffffu, il_mine, LANE_OF_ROW(i));
    if (row >= S) continue;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const float2 x = o[i][2 * g], y = o[i][2 * g + 1];
      const uint2 w = make_uint2(pack_bf2(fmul(x.x, il), fmul(x.y, il)), pack_bf2(fmul(y.x, il), fmul(y.y, il)));
      const size_t off = (row0 + row) * ld_out + (size_t)h * DH + 64 * g + 4 * tx;
      *reinterpret_cast<uint2*>(out + off) = w;
      if (qout)   // the output projection's quantiser, applied to the bf16 values just stored
        *reinterpret_cast<uint32_t*>(qout + off) =
            ((uint32_t)(uint8_t)quant1(bflo(w.x), inv_q)) | ((uint32_t)(uint8_t)quant1(bfhi(w.x), inv_q) << 8) |
            ((uint32_t)(uint8_t)quant1(bflo(w.y), inv_q) << 16) | ((uint32_t)(uint8_t)quant1(bfhi(w.y), inv_q) << 24);
    }
  }
}


// ---------------------------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------------------------
// Delta_i = adjacent tree over the 128 dims of dO_ic * O_ic; one warp per (b, h, i)
__global__ void __launch_bounds__(256) k_attn_delta(const uint16_t* __restrict__ dout, const uint16_t* __restrict__ out,
                                                    int ld_out, int H, int S, size_t nrows, float* __restrict__ delta) {
  grid_dep();
  const size_t w = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= nrows) return;  // w = (b*H + h)*S + i
  const size_t i = w % S, bh = w / S, b = bh / H, h = bh % H;
  const size_t off = (b * S + i) * ld_out + h * DH + lane * 4;
  const uint2 a = __ldg(reinterpret_cast<const uint2*>(dout + off));
  const uint2 c = __ldg(reinterpret_cast<const uint2*>(out + off));
  float t = fadd(fadd(fmul(bflo(a.x), bflo(c.x)), fmul(bfhi(a.x), bfhi(c.x))),
                 fadd(fmul(bflo(a.y), bflo(c.y)), fmul(bfhi(a.y), bfhi(c.y))));
  t = warp_tree_full(t);
  if (lane == 0) delta[w] = t;
}

// ---------------------------------------------------------------------------------------------
// backward, first half: P and dS of every block of TM queries against every visible block of 128 keys.
// Warp-specialised like the LM-head kernel: the CTA keeps q^T and dO^T of its query block in shared memory; four
// producer warps stream the key and value blocks through a three-slot ring of 16-dimension slabs (a "full" and an
// "empty" mbarrier per slot, bounded waits); eight consumer warps accumulate S = q.k^T and dP = dO.v^T together (two
// 8 x 8 register tiles per thread, each logit one ascending sum over the 128 dimensions).  Per key block
// P = exp(S*scale - L) and dS = (P (dP - Delta)) scale are formed and bf16(P) and bf16(dS) stored.  Consumer warps are not coupled to
// each other.
// EPI: that epilogue belongs to four more warps, and the 128 sums of a thread go to them through tensor memory, which is idle
// otherwise (a store of four instructions; two buffers of 128 columns per consumer warp).  Two consumer warps on a scheduler fall
// into step and left it idle during their epilogues, a latency-bound 12.5 of 52 thousand cycles a key block; now one multiplies on
// while the exponentials fill the issue slots it leaves: 16 heads x 2048 0.453 -> 0.406 ms; the whole windowed attention (16 x 4096, forward and
// backward) 1.380 -> 1.348 ms, two sequences of 8 x 1088 0.478 -> 0.460.  A fourth slot (1.381) and slots of two slabs (1.372) leave less of the
// memory to the first-level cache and were slower.  158 bytes of the consumers' 184 and the producers' 56 registers' work are spilled, half by
// either (none by the epilogue: without its arithmetic as many, without the staging 84, without the multiply loops none); with 216 and 72 and
// no epilogue warps it is 48.
// Without EPI a consumer thread works on its own sums, which is the shorter way where a CTA has a key block or two.
// Nothing is carried from one key block to the next, so the blocks of all heads are numbered (head, query block, key block) and
// every CTA of a resident grid takes an equal run of them; where a run enters another query block the consumers stage its rows.
// One query block per CTA, 4 x 16 heads x 2048 (query blocks of up to 16 key blocks, 1024 of them): 1.564 ms, equal runs 1.597; but
// 16 x 4096 at window 512 0.545 and 0.478 ms, 2 x 8 x 1088 0.215 and 0.145, 8 x 1024 0.210 and 0.066, 16 x 832 0.166 and 0.099; 16 x 4096
// 1.528, 1.547 and with the short runs at the end 1.526.
// ---------------------------------------------------------------------------------------------
// Rows per block (TM), ring slots, CTAs per SM, registers per consumer, producer and epilogue thread.  A block of 128 rows takes 24.5 us, one
// of 64 rows 18.4 alone and 15.8 beside another; both 12 us for the launch, the first rows and the first slabs.
template <int TM_, int SLOTS_, int CPS_, int RC_, int RP_, int RE_ = 0>
struct SdpTile {
  static constexpr int TM = TM_, SLOTS = SLOTS_, CPS = CPS_, RC = RC_, RP = RP_, RE = RE_;
  static constexpr bool EPI = RE > 0;
  static constexpr int CONS = TM * 2, THREADS = CONS + OG_PROD + (EPI ? 128 : 0);
  static constexpr int COLS = CONS;                // tensor memory columns of a buffer: 128 for every four consumer warps
  static constexpr size_t SMEM = (size_t)(2 * DH * (TM + 4) + 2 * SLOTS * OK * (OT + 4)) * sizeof(float);
  static_assert(CONS * RC + OG_PROD * RP + 128 * RE <= (65536 / (CPS * THREADS) / 8 * 8) * THREADS, "register hand-over exceeds the block's allocation");
  static_assert(!EPI || (CPS == 1 && 2 * COLS <= 512), "two buffers in tensor memory");
};
typedef SdpTile<128, 3, 1, 184, 56, 88> SdpTall;
typedef SdpTile<128, 3, 1, 216, 72> SdpLone;
typedef SdpTile<64, 2, 2, 200, 56> SdpHalf;

// named barrier of the first `threads` threads; the second form also tells whether any of them came with `x`
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ int bar_or(int id, int threads, bool x) {
  int any;
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.s32 p, %1, 0;\nbar.red.or.pred q, %2, %3, p;\nselp.s32 %0, 1, 0, q;\n}"
               : "=r"(any) : "r"((int)x), "r"(id), "r"(threads) : "memory");
  return any;
}
// key blocks that the query block at i0 sees: first one, and how many
__host__ __device__ __forceinline__ int sdp_first(int i0, int W) { return W > 0 && i0 > W ? (i0 - W) / OT : 0; }
__host__ __device__ __forceinline__ int sdp_blocks(int i0, int W) { return i0 / OT + 1 - sdp_first(i0, W); }
// runs of blocks: n_long equal ones over the first `head` blocks, then n_short equal ones over the rest; or (heads != 0) one
// run per query block of the `heads` heads, the last query blocks first
struct SdpRuns {
  int n_long, head, n_short, total, heads;
  __device__ __forceinline__ int start(int c) const {
    return c <= n_long ? (int)((long long)head * c / n_long) : head + (int)((long long)(total - head) * (c - n_long) / n_short);
  }
};
// position in the numbering of the blocks
struct SdpAt {
  int bh, i0, jt;
  __device__ __forceinline__ SdpAt(int bh_, int i0_, int jt_) : bh(bh_), i0(i0_), jt(jt_) {}
  __device__ __forceinline__ SdpAt(int w, int per_head, int tm, int W) {
    bh = w / per_head;
    w -= bh * per_head;
    i0 = 0;
    for (int n = sdp_blocks(0, W); w >= n; n = sdp_blocks(i0, W)) { w -= n; i0 += tm; }
    jt = sdp_first(i0, W) + w;
  }
  __device__ __forceinline__ bool next(int S, int tm, int W) {   // true: another query block
    if (++jt <= i0 / OT) return false;
    i0 += tm;
    if (i0 >= S) { i0 = 0; ++bh; }
    jt = sdp_first(i0, W);
    return true;
  }
};

// P and dS of eight keys j0 + 64 g + 4 tx + 0 .. 3 (g = 0, 1) of row i from the sums s = q.k and d = dO.v; P and dS point to the row.
// The argument of the exponential is at most 0 whenever L is the row's own logsumexp, and then the form without the overflow range
// applies (same bits), but L is an input, so eight values that hold a positive argument take the general form.
__device__ __forceinline__ void sdp_row(const float2 (&s)[4], const float2 (&d)[4], float L, float D, int i, int j0, int tx, int S, int W,
                                        bool masked, float2 one, uint16_t* __restrict__ P, uint16_t* __restrict__ dS) {
  const float2 L2 = same2(-L), D2 = same2(-D);
  float2 x[4], pv[4], ds[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) x[t] = add2(mul2(s[t], same2(ATT_SCALE)), L2, one);
  uint32_t vis = 0xff;
  if (masked) {
    vis = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int key = j0 + (e >> 2) * 64 + tx * 4 + (e & 3);
      if (key <= i && (W == 0 || key > i - W)) vis |= 1u << e;
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) x[t] = make_float2(vis >> (2 * t) & 1 ? x[t].x : 0.0f, vis >> (2 * t + 1) & 1 ? x[t].y : 0.0f);
  }
  float top = x[0].x;
#pragma unroll
  for (int t = 0; t < 4; ++t) top = fmaxf(top, fmaxf(x[t].x, x[t].y));
  if (top > 0.0f) {
#pragma unroll
    for (int t = 0; t < 4; ++t) pv[t] = make_float2(det_exp(x[t].x), det_exp(x[t].y));
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) pv[t] = det_exp_le0_2(x[t], one);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) ds[t] = mul2(mul2(pv[t], add2(d[t], D2, one)), same2(ATT_SCALE));
  if (masked) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      pv[t] = make_float2(vis >> (2 * t) & 1 ? pv[t].x : 0.0f, vis >> (2 * t + 1) & 1 ? pv[t].y : 0.0f);
      ds[t] = make_float2(vis >> (2 * t) & 1 ? ds[t].x : 0.0f, vis >> (2 * t + 1) & 1 ? ds[t].y : 0.0f);
    }
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int jb = j0 + g * 64 + tx * 4;
    if (jb >= S) continue;
    // P~ = bf16(P) is all the value gradient needs
    *reinterpret_cast<uint2*>(P + jb) = make_uint2(pack_bf2(pv[2 * g].x, pv[2 * g].y), pack_bf2(pv[2 * g + 1].x, pv[2 * g + 1].y));
    *reinterpret_cast<uint2*>(dS + jb) = make_uint2(pack_bf2(ds[2 * g].x, ds[2 * g].y), pack_bf2(ds[2 * g + 1].x, ds[2 * g + 1].y));
  }
}

// two rows of a thread's sums, S and dP of each, to 32 columns of its lane
__device__ __forceinline__ void tmem_st_rows(uint32_t taddr, const float2 (&s0)[4], const float2 (&d0)[4], const float2 (&s1)[4],
                                             const float2 (&d1)[4]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "f"(s0[0].x), "f"(s0[0].y), "f"(s0[1].x), "f"(s0[1].y), "f"(s0[2].x), "f"(s0[2].y), "f"(s0[3].x), "f"(s0[3].y),
      "f"(d0[0].x), "f"(d0[0].y), "f"(d0[1].x), "f"(d0[1].y), "f"(d0[2].x), "f"(d0[2].y), "f"(d0[3].x), "f"(d0[3].y),
      "f"(s1[0].x), "f"(s1[0].y), "f"(s1[1].x), "f"(s1[1].y), "f"(s1[2].x), "f"(s1[2].y), "f"(s1[3].x), "f"(s1[3].y),
      "f"(d1[0].x), "f"(d1[0].y), "f"(d1[1].x), "f"(d1[1].y), "f"(d1[2].x), "f"(d1[2].y), "f"(d1[3].x), "f"(d1[3].y)
      : "memory");
}
// the wait behind tmem_ld16_nowait, with the registers it is for
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                 "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

template <class T>
__global__ void __launch_bounds__(T::THREADS, T::CPS)
    k_attn_sdp(const uint16_t* __restrict__ dout, const uint16_t* __restrict__ q, const uint16_t* __restrict__ k,
               const uint16_t* __restrict__ v, const float* __restrict__ lse, const float* __restrict__ delta, int ld,
               int ld_out, int H, int Hkv, int S, int W, int per_head, const SdpRuns runs, uint16_t* __restrict__ Pb,
               uint16_t* __restrict__ dSt) {
  constexpr int TM = T::TM, SDP_SLOTS = T::SLOTS, SDP_CONS = T::CONS;
  extern __shared__ __align__(16) unsigned char osm[];
  typedef float(*Full)[TM + 4];
  Full Qs = reinterpret_cast<Full>(osm);                                            // [dim][query]
  Full Os = reinterpret_cast<Full>(osm + (size_t)DH * (TM + 4) * sizeof(float));    // [dim][query] of dO
  float(*Ks)[OK][OT + 4] = reinterpret_cast<float(*)[OK][OT + 4]>(osm + (size_t)2 * DH * (TM + 4) * sizeof(float));
  float(*Vs)[OK][OT + 4] = Ks + SDP_SLOTS;
  __shared__ __align__(4) uint8_t tiny_s[SDP_SLOTS][OG_PROD / 32];
  __shared__ int abort_s;
  __shared__ __align__(8) uint64_t bar_full[SDP_SLOTS], bar_empty[SDP_SLOTS];
  __shared__ __align__(8) uint64_t sum_full[2][SDP_CONS / 32], sum_empty[2][SDP_CONS / 32];   // the sums of a consumer warp, per buffer
  __shared__ uint32_t tmem_base_s;
  volatile int* abort_flag = &abort_s;
  const int tid = threadIdx.x, lane = tid & 31;
  int w_lo = 0, w_hi;
  SdpAt at(0, 0, 0);
  if (runs.heads) {
    const int c = blockIdx.x, i0 = ((int)gridDim.x - 1 - c) / runs.heads * TM;
    at = SdpAt(c % runs.heads, i0, sdp_first(i0, W));
    w_hi = sdp_blocks(i0, W);
  } else {
    w_lo = runs.start(blockIdx.x);
    w_hi = runs.start(blockIdx.x + 1);
    at = SdpAt(w_lo, per_head, TM, W);
  }
  if (tid == 0) {
    for (int s = 0; s < SDP_SLOTS; ++s) { mbar_init(&bar_full[s], OG_PROD / 32); mbar_init(&bar_empty[s], SDP_CONS / 32); }
    for (int w = 0; w < SDP_CONS / 32; ++w)
      for (int b = 0; b < 2; ++b) { mbar_init(&sum_full[b][w], 1); mbar_init(&sum_empty[b][w], 1); }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (T::EPI && tid >> 5 == (SDP_CONS + OG_PROD) / 32) {   // first epilogue warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)(2 * T::COLS)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (T::EPI) tc_fence_before();
  __syncthreads();
  if (T::EPI) tc_fence_after();
  // the sums of consumer warp w: lanes 32 (w % 4) .., columns 128 (w / 4) .. of a buffer; row a of a thread in columns 16 a ..
  auto sums_at = [&](int w, int buf) { return tmem_base_s + ((uint32_t)(w & 3) << 21) + (uint32_t)(buf * T::COLS + (w >> 2) * 128); };
  const float2 one = same2(c_one);
  if (T::EPI && tid >= SDP_CONS + OG_PROD) {
    // ------------------------------- epilogue -------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(T::EPI ? T::RE : 24));
    const int tx = lane >> 1;
    int buf = 0;
    uint32_t par = 0;
    bool ok = true;
    for (int blk = w_lo; blk < w_hi && ok; ++blk) {
      const int i0 = at.i0, j0 = at.jt * OT;
      const size_t r0 = (size_t)at.bh * S;
      const bool masked = j0 + OT - 1 > i0 || (W > 0 && j0 <= i0 + TM - 1 - W);   // the block at the diagonal and those at the window's start
#pragma unroll 1
      for (int w = (tid >> 5) & 3; w < SDP_CONS / 32; w += 4) {
        const int first = i0 + (w * 2 + (lane & 1)) * 4;               // rows first + 0 .. 3 and first + TM / 2 + 0 .. 3
        // rows past the last one exist only where S is no multiple of TM: their L and Delta are never used
        float L = first < S ? __ldg(lse + r0 + first) : 0.0f, D = first < S ? __ldg(delta + r0 + first) : 0.0f;
        ok = mbar_wait_warp(&sum_full[buf][w], par, abort_flag, nullptr);
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = sums_at(w, buf);
        uint32_t r[16];
        tmem_ld16_nowait(taddr, r);
        tmem_wait_ld16(r);
#pragma unroll 1
        for (int a = 0; a < 8; ++a) {
          const int i = first + (a >> 2) * (TM / 2) + (a & 3);
          float2 sv[4], dv[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            sv[t] = make_float2(__uint_as_float(r[2 * t]), __uint_as_float(r[2 * t + 1]));
            dv[t] = make_float2(__uint_as_float(r[8 + 2 * t]), __uint_as_float(r[9 + 2 * t]));
          }
          const float La = L, Da = D;
          if (a < 7) {                                                  // the next row travels during this one's arithmetic
            const int n = first + ((a + 1) >> 2) * (TM / 2) + ((a + 1) & 3);
            tmem_ld16_nowait(taddr + 16 * (a + 1), r);
            if (n < S) { L = __ldg(lse + r0 + n); D = __ldg(delta + r0 + n); }
          }
          if (i < S) sdp_row(sv, dv, La, Da, i, j0, tx, S, W, masked, one, Pb + (r0 + i) * S, dSt + (r0 + i) * S);
          __syncwarp();
          if (a < 7) tmem_wait_ld16(r);
          if (a == 6) {                                                 // everything has been read
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sum_empty[buf][w]);
          }
        }
      }
      at.next(S, TM, W);
      if ((buf ^= 1) == 0) par ^= 1u;
    }
  } else if (tid >= SDP_CONS) {
    // ------------------------------- producers -------------------------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(T::RP));
    const int pt = tid - SDP_CONS, pw = pt >> 5;
    typedef OgSide<CONTIG, false, OT> Side;
    Side sk, sv;
    Side::Raw rk, rv;
    auto block = [&]() {                             // the key block `at`
      const size_t o = (size_t)(at.bh / H) * S * ld + (size_t)(at.bh % H / (H / Hkv)) * DH;
      sk.init(k + o, S, ld, at.jt * OT, 0, pt);
      sv.init(v + o, S, ld, at.jt * OT, 0, pt);
    };
    block();
    sk.fetch(rk, OK, 0, pt);
    sv.fetch(rv, OK, 0, pt);
    int slot = 0;
    uint32_t par = 1;
    const int nslab = (w_hi - w_lo) * (DH / OK);
    for (int s = 0; s < nslab; ++s) {
      if (!mbar_wait_warp(&bar_empty[slot], par, abort_flag, nullptr)) break;   // the block's last barrier is for whole warps
      uint32_t least = ~0u;
      sk.store(Ks[slot], rk, least, pt);
      sv.store(Vs[slot], rv, least, pt);
      if (s + 1 < nslab) {
        if ((s + 1) % (DH / OK) == 0) {
          at.next(S, TM, W);
          block();
        }
        sk.fetch(rk, OK, 0, pt);
        sv.fetch(rv, OK, 0, pt);
      }
      const int any = __any_sync(0xffffffffu, least_tiny(least));
      if (lane == 0) tiny_s[slot][pw] = (uint8_t)any;
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_full[slot]);
      if (++slot == SDP_SLOTS) { slot = 0; par ^= 1u; }
    }
  } else {
  // --------------------------------- consumers ---------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(T::RC));
  const int ty = (tid >> 5) * 2 + (tid & 1), tx = (lane >> 1);   // neighbouring lanes share their columns (see og_lane)
  int tqo = 0;                                     // a value below 2^-63 among the rows
  float Lr[8], Dr[8];
  // q^T and dO^T of the query block, and its rows' logsumexp and Delta: everything is on its way before the barrier
  auto stage = [&](int bh, int i0) {
    const size_t row = (size_t)(bh / H) * S + i0;
    const int h = bh % H;
    uint4 u[2][8];                                 // TM x 16 pieces of 16 bytes each: eight per thread
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int e = c * SDP_CONS + tid, x = e % TM, ch = e / TM;
      const bool in = i0 + x < S;
      u[0][c] = in ? __ldg(reinterpret_cast<const uint4*>(q + (row + x) * ld + (size_t)h * DH + ch * 8)) : make_uint4(0u, 0u, 0u, 0u);
      u[1][c] = in ? __ldg(reinterpret_cast<const uint4*>(dout + (row + x) * ld_out + (size_t)h * DH + ch * 8)) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      if (T::EPI) break;
      const int i = i0 + (a >> 2) * (TM / 2) + ty * 4 + (a & 3);
      Lr[a] = i < S ? lse[(size_t)bh * S + i] : 0.0f;
      Dr[a] = i < S ? delta[(size_t)bh * S + i] : 0.0f;
    }
    bool tq = false;
    bar_sync(1, SDP_CONS);                         // the rows before are not needed any more
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int e = c * SDP_CONS + tid, x = e % TM, ch = e / TM;
      float t[8];
      unpack8a(u[0][c], t);
#pragma unroll
      for (int y = 0; y < 8; ++y) { tq |= tiny1(t[y]); Qs[ch * 8 + y][x] = t[y]; }
      unpack8a(u[1][c], t);
#pragma unroll
      for (int y = 0; y < 8; ++y) { tq |= tiny1(t[y]); Os[ch * 8 + y][x] = t[y]; }
    }
    tqo = bar_or(1, SDP_CONS, tq);
  };
  int slot = 0, buf = 0;
  uint32_t par = 0, spar = 1;
  bool ok = true;
  for (int w = w_lo; w < w_hi;) {
    const int i0 = at.i0, jt0 = at.jt, jt1 = min(jt0 + w_hi - w, i0 / OT + 1);
    const size_t bh = (size_t)at.bh;
    stage(at.bh, i0);                              // after a wait that ran out, too: the other warps stand at its barriers
    w += jt1 - jt0;
    at.jt = jt1 - 1;
    at.next(S, TM, W);
    for (int jt = jt0; jt < jt1 && ok; ++jt) {
      const int j0 = jt * OT;
      float2 sa[8][4], da[8][4];
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) { sa[a][c] = make_float2(0.f, 0.f); da[a][c] = make_float2(0.f, 0.f); }
      for (int sl = 0; sl < DH / OK && ok; ++sl) {
        ok = mbar_wait_warp(&bar_full[slot], par, abort_flag, nullptr);
        if (!ok) break;
        if (tqo | *reinterpret_cast<const uint32_t*>(tiny_s[slot])) { slab_mac<false, TM, OT, 8>(Qs + sl * OK, Ks[slot], ty, tx, sa); slab_mac<false, TM, OT, 8>(Os + sl * OK, Vs[slot], ty, tx, da); }
        else { slab_mac<true, TM, OT, 8>(Qs + sl * OK, Ks[slot], ty, tx, sa); slab_mac<true, TM, OT, 8>(Os + sl * OK, Vs[slot], ty, tx, da); }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_empty[slot]);
        if (++slot == SDP_SLOTS) { slot = 0; par ^= 1u; }
      }
      if (!ok) break;
      if (T::EPI) {
        const int w = tid >> 5;
        ok = mbar_wait_warp(&sum_empty[buf][w], spar, abort_flag, nullptr);   // two blocks ago has been read
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = sums_at(w, buf);
#pragma unroll
        for (int a = 0; a < 8; a += 2) tmem_st_rows(taddr + 16 * a, sa[a], da[a], sa[a + 1], da[a + 1]);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sum_full[buf][w]);
        if ((buf ^= 1) == 0) spar ^= 1u;
      } else {
        const bool masked = j0 + OT - 1 > i0 || (W > 0 && j0 <= i0 + TM - 1 - W);   // the block at the diagonal and those at the window's start
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const int i = i0 + (a >> 2) * (TM / 2) + ty * 4 + (a & 3);
          if (i < S) sdp_row(sa[a], da[a], Lr[a], Dr[a], i, j0, tx, S, W, masked, one, Pb + (bh * S + i) * S, dSt + (bh * S + i) * S);
        }
      }
    }
  }
  }
  if (T::EPI) {
    tc_fence_before();
    __syncthreads();
    if (tid >> 5 == (SDP_CONS + OG_PROD) / 32) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base_s), "r"((uint32_t)(2 * T::COLS)) : "memory");
    }
  }
}


}  // namespace det

using namespace det;

template <class T, bool WIN>
static int attn_fwd_go(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S, int window,
                       det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, cudaStream_t st) {
  static DevOnce once = {};
  const auto kern = k_attn_fwd<T, WIN>;
  if (dev_ensure_smem(once, (const void*)kern, T::SMEM) != DET_OK) return DET_ERR_CUDA;
  const dim3 grid(H * B, (S + T::FQ - 1) / T::FQ);
  kern<<<DET_L(grid), T::THREADS, T::SMEM, st>>>(q, k, v, ld, H, Hkv, S, window, out, ld_out, lse, s_q, qout, dev_sm_count());
  return DET_OK;
}
template <class T>
static int attn_fwd_run(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S, int window,
                        det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, cudaStream_t st) {
  return window ? attn_fwd_go<T, true>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, st)
                : attn_fwd_go<T, false>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, st);
}
// Rows per CTA: the longest chain of key blocks runs on one SM whatever the others do, and all chains together share the GPU; the
// figures are the microseconds per key block of a CTA alone on its SM and of one among many, the CTAs per SM, and the part of a
// chain by which the shared time is exceeded in the end, which shrinks with the rounds of CTAs over the GPU's places (with 128 rows a key
// block's time); nothing while long and short rows are paired on the SMs (two CTAs each, none left over).  The row count with the smallest of
// the larger bounds is taken.  Measured with 128, 64, 32 rows and two groups: 16 heads x 2048 378, 405, 400, 513; 48 x 832 241, 214, 218, 294; 20 x 1024 194, 187, 151, 181;
// 16 x 1088 216, 140, 150, 163; 16 x 832 169, 112, 104, 101; 8 x 1024 192, 124, 95, 77 us.
struct RowCost { int rows; double alone, full; int cps; double over, decay, tail; };   // rows: 33 for 32 rows with two groups; tail: in key blocks
// With a window that is shorter than the sequence all rows but the first ones have chains of one length, so they run in rounds of equal CTAs and
// a last round costs what the CTAs beside each other on an SM then need: 20 heads x 832 at window 128 take one round of 128 rows
// (54 us; 64 rows, two CTAs on each SM, 64), 16 x 2048 two (103; 64 rows in two rounds of two CTAs 116, 32 rows 111), 8 x 512 one of
// two groups (24; 32 rows 30, 128 rows 54).  Forms with one CTA on an SM: the CTAs are dealt out in their order, the longest first, to the SM
// that is free first.  Forms with several: the larger one of the rounds of the longest chains and of all chains shared out evenly, a part of a
// mean chain more in the end.  Microseconds of a launch, of a key block and of a CTA beside its key blocks (odd: one more where the second group has a
// block less), by the CTAs on the SM.  Fitted to 208 shapes (2 to 96 heads x 320 to 4096, windows of 128 to 2048), all four forms measured
// of each: the form taken is 0.2 % slower than the best one in the mean and 4 % with three exceptions (12 x 832 at window 512 takes 64 or 32 rows,
// 91 us, two groups 81).  The rule below, which counts on chains of all lengths, was 6 % off in the mean.
struct WindowCost { int rows, cps; double launch, tail, block[3], cta[3], odd; };
constexpr int WIN_LENGTHS = 64;
static int attn_rows_window(int heads, int S, int window) {
  const WindowCost forms[4] = {{128, 1, 3.58, 0.0, {23.48}, {3.08}, 0.0},
                               {64, 2, 14.46, 0.32, {16.21, 26.92}, {-6.19, -3.23}, 0.0},
                               {32, 3, 10.71, 0.24, {11.72, 17.03, 20.96}, {-4.54, -4.94, -0.05}, 0.0},
                               {33, 1, 3.87, 0.0, {8.63}, {1.9}, 2.14}};
  const int sms = dev_sm_count() > 0 ? dev_sm_count() : 1;
  int best = 0;
  double best_t = 0.0;
  for (const WindowCost& f : forms) {
    const int step = f.rows & ~1;
    int longest = 0;
    long long count[WIN_LENGTHS] = {}, ctas = 0, blocks = 0;         // CTAs with a chain of so many blocks
    for (int q0 = 0; q0 < S; q0 += step) {
      const int n = q0 / FK + 1 - (q0 > window ? (q0 - window) / FK : 0);
      if (n > longest) longest = n;
      count[n] += heads;
      ctas += heads;
      blocks += (long long)n * heads;
    }
    auto chain = [&](double n, int beside) { return n * f.block[beside - 1] + f.cta[beside - 1]; };
    double t = 0.0;
    if (f.cps == 1) {
      struct { double at; long long sms; } free[WIN_LENGTHS + 1] = {{0.0, sms}};   // SMs by the time they are free; a length adds one entry at most
      int m = 1;
      for (int n = longest; n > 0; --n)
        for (long long left = count[n]; left > 0;) {
          const long long take = left < free[0].sms ? left : free[0].sms;
          const double end = free[0].at + chain(n, 1) + (n > 1 && n % 2 ? f.odd : 0.0);
          left -= take;
          if (take < free[0].sms) {
            free[0].sms -= take;
          } else {
            --m;
            for (int i = 0; i < m; ++i) free[i] = free[i + 1];
          }
          int i = m;
          for (; i > 0 && free[i - 1].at > end; --i) free[i] = free[i - 1];
          free[i] = {end, take};
          ++m;
        }
      t = free[m - 1].at;
    } else {
      const long long places = (long long)sms * f.cps, full = count[longest], rest = full % places;
      const double rounds = (full / places) * chain(longest, f.cps) + (rest ? chain(longest, (int)((rest + sms - 1) / sms)) : 0.0);
      const double shared = (blocks * f.block[f.cps - 1] + ctas * f.cta[f.cps - 1]) / places + f.tail * chain((double)blocks / ctas, 1);
      t = chain(longest, 1);
      if (rounds > t) t = rounds;
      if (ctas > sms && shared > t) t = shared;
    }
    t += f.launch;
    if (!best || t < best_t) { best = f.rows; best_t = t; }
  }
  return best;
}
static int attn_rows(int heads, int S, int window) {
  if (window && window / FK + 1 < WIN_LENGTHS) return attn_rows_window(heads, S, window);
  const RowCost c[4] = {{128, 23.5, 23.9, 1, 0.0, 0.0, 0.9}, {64, 15.0, 12.1, 2, 0.55, 2.0, 0.0}, {32, 9.8, 6.5, 3, 0.5, 1.5, 0.0}, {33, 8.6, 8.6, 1, 0.15, 0.0, 0.0}};
  const int sms = dev_sm_count() > 0 ? dev_sm_count() : 1;
  int best = c[0].rows;
  double best_t = 0.0;
  for (int i = 0; i < 4; ++i) {
    const int step = c[i].rows & ~1;
    double longest = 0.0, total = 0.0;
    for (int q0 = 0; q0 < S; q0 += step) {
      const double tiles = q0 / FK + 1 - (window && q0 > window ? (q0 - window) / FK : 0);
      total += tiles;
      if (tiles > longest) longest = tiles;
    }
    const double rounds = (double)heads * ((S + step - 1) / step) / ((double)c[i].cps * sms);
    const double over = rounds > 1.0 ? c[i].over * pow(rounds, -c[i].decay) : (c[i].cps == 2 ? 0.0 : c[i].over);
    const double a = longest * c[i].alone, b = total * heads * c[i].full / sms + over * a + (rounds > 1.0 ? c[i].tail * c[i].alone : 0.0);
    const double t = a > b ? a : b;
    if (i == 0 || t < 0.97 * best_t) { best = c[i].rows; best_t = t; }
  }
  return best;
}

static int attn_fwd_impl(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S, int window,
                         det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, void* stream, int rows = 0) {
  if (!q || !k || !v || !out || !lse || B <= 0 || H <= 0 || Hkv <= 0 || S <= 0 || window < 0) return DET_ERR_ARG;
  if (qout && (!s_q || (((uintptr_t)qout) & 3u))) return qout && !s_q ? DET_ERR_ARG : DET_ERR_ALIGN;
  if (S % 64 || ld % 8 || ld_out % 8 || ld < H * DH || ld_out < H * DH || H % Hkv || window % 128) return DET_ERR_SHAPE;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out)) return DET_ERR_ALIGN;
  if (window >= S) window = 0;                     // no row has a key that far behind it
  int rc;
  switch (rows ? rows : attn_rows(B * H, S, window)) {
    case 128: rc = attn_fwd_run<AfTall>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, (cudaStream_t)stream); break;
    case 64: rc = attn_fwd_run<AfHalf>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, (cudaStream_t)stream); break;
    case 33: rc = attn_fwd_run<AfPair>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, (cudaStream_t)stream); break;
    default: rc = attn_fwd_run<AfShort>(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, (cudaStream_t)stream);
  }
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_attn_fwd(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S,
                            int window, det_bf16* out, int ld_out, float* lse, void* stream) {
  return attn_fwd_impl(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, nullptr, nullptr, stream);
}
extern "C" int det_attn_fwd_q(const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S,
                              int window, det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, void* stream) {
  if (!s_q || !qout) return DET_ERR_ARG;
  return attn_fwd_impl(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, stream);
}
extern "C" int det_test_attn_fwd(int rows, const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S,
                                 int window, det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, void* stream) {
  if (!s_q || !qout || (rows != 128 && rows != 64 && rows != 32 && rows != 33)) return DET_ERR_ARG;
  return attn_fwd_impl(q, k, v, ld, B, H, Hkv, S, window, out, ld_out, lse, s_q, qout, stream, rows);
}
extern "C" int det_test_attn_rows(int heads, int S, int window) {
  return heads > 0 && S > 0 && window >= 0 && window % 128 == 0 ? attn_rows(heads, S, window >= S ? 0 : window) : 0;
}

// workspace: bf16(P) and bf16(dS), [B*H, S, S] each, and Delta f32 [B*H, S]
extern "C" size_t det_attn_bwd_ws_bytes(int B, int H, int Hkv, int S) {
  (void)Hkv;
  return 2 * align_up((size_t)B * H * S * S * 2, 256) + align_up((size_t)B * H * S * 4, 256);
}

// the fixed-point variant keeps its 64-bit totals in shared memory (k_ogemm): no extra scratch
extern "C" size_t det_attn_bwd_fixq_ws_bytes(int B, int H, int Hkv, int S) { return det_attn_bwd_ws_bytes(B, H, Hkv, S); }

template <class T>
static int sdp_run(const det_bf16* dout, const det_bf16* q, const det_bf16* k, const det_bf16* v, const float* lse,
                   const float* delta, int ld, int ld_out, int B, int H, int Hkv, int S, int window, int per_head, uint16_t* Pb,
                   uint16_t* dSt, cudaStream_t st) {
  static DevOnce once = {};
  if (dev_ensure_smem(once, (const void*)k_attn_sdp<T>, T::SMEM) != DET_OK) return DET_ERR_CUDA;
  const int total = B * H * per_head, slots = dev_sm_count() * T::CPS;
  // Runs of equal length, with a sixteenth of the blocks left for the SMs that finish first where a run is long; whole query blocks
  // only where those are long (the start of a CTA weighs little) and many (the hardware's order balances them)
  const int rows = (S + T::TM - 1) / T::TM, longest = sdp_blocks((rows - 1) * T::TM, window);
  SdpRuns runs = {total < slots ? total : slots, total, 0, total, 0};
  int ctas = runs.n_long;
  if (longest >= 12 && (long long)rows * B * H >= 6 * slots) {
    runs.heads = B * H;
    ctas = rows * B * H;
  } else if (total >= 16 * slots) {
    runs.head = total - total / 16;
    runs.n_short = 2 * slots;
    ctas += runs.n_short;
  }
  k_attn_sdp<T><<<DET_L(ctas), T::THREADS, T::SMEM, st>>>(dout, q, k, v, lse, delta, ld, ld_out, H, Hkv, S, window, per_head, runs, Pb,
                                                          dSt);
  return DET_OK;
}

static int attn_bwd_impl(const det_bf16* dout, const det_bf16* q, const det_bf16* k, const det_bf16* v,
                         const det_bf16* out, const float* lse, int ld, int ld_out, int B, int H, int Hkv, int S,
                         int window, det_bf16* dq, det_bf16* dk, det_bf16* dv, int ld_d, void* ws, size_t ws_bytes,
                         void* stream, bool fixq) {
  if (!dout || !q || !k || !v || !out || !lse || !dq || !dk || !dv || B <= 0 || H <= 0 || Hkv <= 0 || S <= 0 || window < 0)
    return DET_ERR_ARG;
  if (S % 64 || ld % 8 || ld_out % 8 || ld_d % 8 || (long long)B * H > 65535 || H % Hkv || window % 128) return DET_ERR_SHAPE;
  if (!aligned16(dout) || !aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(dq) ||
      !aligned16(dk) || !aligned16(dv) || !aligned16(ws))
    return DET_ERR_ALIGN;
  if (!ws || ws_bytes < (fixq ? det_attn_bwd_fixq_ws_bytes(B, H, Hkv, S) : det_attn_bwd_ws_bytes(B, H, Hkv, S)))
    return DET_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  const int G = H / Hkv;
  const size_t matP = align_up((size_t)B * H * S * S * 2, 256), matS = matP;
  uint16_t* Pb = (uint16_t*)ws;
  uint16_t* dSt = (uint16_t*)((uint8_t*)ws + matP);
  float* delta = (float*)((uint8_t*)ws + matP + matS);
  const size_t nrows = (size_t)B * H * S;
  launch_after(k_attn_delta, (unsigned)((nrows + 7) / 8), 256, 0, st, dout, out, ld_out, H, S, nrows, delta);
  DET_CHECK_LAUNCH();
  // P[i,j] = exp(scale * sum_d q[i,d] k[j,d] - L_i) for visible (i,j) (f32; tiles without a visible pair are never
  // touched) and dS[i,j] = bf16((P[i,j] * (sum_d dO[i,d] v[j,d] - Delta_i)) * scale); both sums ascend over the 128 dims
  // blocks of 64 rows where those leave every CTA with one block at most (2 heads x 128: 0.027 against 0.035 ms); with more of them
  // the tall ones have the better rate (8 x 1024: 0.076 and 0.066 ms).  Up to a block and three quarters per CTA there is little to multiply
  // behind the epilogue and the multiplying warps do it themselves (whole backward, with epilogue warps and without: 16 heads x 384, 96
  // blocks, 82.9 and 79.0 us; 24 x 512, 240 blocks, 138.3 and 137.9; 90 x 256, 270 blocks, 136.4 and 138.5)
  int tall = 0, half = 0;
  for (int i0 = 0; i0 < S; i0 += 64) {
    half += sdp_blocks(i0, window);
    if (i0 % 128 == 0) tall += sdp_blocks(i0, window);
  }
  int rc = (long long)B * H * half <= dev_sm_count()
               ? sdp_run<SdpHalf>(dout, q, k, v, lse, delta, ld, ld_out, B, H, Hkv, S, window, half, Pb, dSt, st)
           : 4ll * B * H * tall <= 7ll * dev_sm_count()
               ? sdp_run<SdpLone>(dout, q, k, v, lse, delta, ld, ld_out, B, H, Hkv, S, window, tall, Pb, dSt, st)
               : sdp_run<SdpTall>(dout, q, k, v, lse, delta, ld, ld_out, B, H, Hkv, S, window, tall, Pb, dSt, st);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  // dV[j,c] = sum over the query heads g of the group, then over queries i >= j ascending, of P~[i,j] dO[i,c];
  // dK[j,c] likewise with dS~ and q; dQ[i,c] = sum over visible keys j ascending of dS~[i,j] k[j,c].  The three are
  // independent of each other: each fills the SMs that the one before it leaves, so that the short blocks at the end of one grid
  // overlap with the long blocks at the start of the next (on three streams, 16 heads x 4096 with window 512: 1.472 ms forward and backward
  // against 1.425, two sequences of 8 x 1088 0.514 against 0.511).
  // While dV has at most two 64-row tiles per SM (whatever tile og_pick takes), all of them resident at once, the dK tiles that join them
  // start with the shortest, so that long and short ones share
  // an SM: 8 heads x 1024 0.174 -> 0.163 ms for the whole backward, two sequences of 8 x 1088 0.344 -> 0.330; with more tiles, or with
  // the long chains of grouped heads, the longest dK must not come last (16 heads on 4 x 4096: 3.40 and 3.80 ms).  Grids of 128-row
  // tiles that are resident although they have more 64-row tiles than that (8 heads x 2432 to 4096) keep the longest first.
  const bool pair = G == 1 && (long long)B * H * ((S + 63) / 64) <= 2 * dev_sm_count();
  for (int which = 0; which < 2; ++which) {
    OgemmArgs p = {};
    p.I = S; p.J = DH; p.C = S; p.lda = S; p.H = Hkv; p.a_b = (long long)H * S * S; p.a_h = (long long)S * S;
    p.nG = G; p.b_div = 1; p.range_mode = 1; p.window = window;
    p.A = which == 0 ? Pb : dSt;
    p.B = which == 0 ? dout : q;
    p.ldb = which == 0 ? ld_out : ld;
    p.b_b = (long long)S * p.ldb; p.b_h = DH;
    p.out = which == 0 ? dv : dk; p.ldo = ld_d; p.o_b = (long long)S * ld_d; p.o_h = DH;
    p.order = which == 0 ? OG_LEAD : OG_LEAD | OG_FILL | (pair ? OG_BACK : 0);
    rc = ogemm_launch<STRIDED, STRIDED, false, true, 1>(p, B * Hkv, 3, st);
    if (rc != DET_OK) return rc;
  }
  OgemmArgs p = {};
  p.I = S; p.J = DH; p.C = S; p.lda = S; p.H = H; p.a_b = (long long)H * S * S; p.a_h = (long long)S * S;
  p.A = dSt; p.B = k; p.ldb = ld; p.b_b = (long long)S * ld; p.b_h = DH; p.nG = 1; p.b_div = G;
  p.out = dq; p.ldo = ld_d; p.o_b = (long long)S * ld_d; p.o_h = DH; p.range_mode = 2; p.window = window;
  // fixq: per block of 128 keys the ordered f32 sum, accumulated over the blocks in 64-bit fixed point (Sec. 3.2)
  p.order = OG_FILL;
  if (fixq) rc = ogemm_run<CONTIG, STRIDED, false, true, OgFix, true>(p, B * H, st);
  else rc = ogemm_launch<CONTIG, STRIDED, false, true, 1>(p, B * H, 3, st);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_attn_bwd(const det_bf16* dout, const det_bf16* q, const det_bf16* k, const det_bf16* v,
                            const det_bf16* out, const float* lse, int ld, int ld_out, int B, int H, int Hkv, int S,
                            int window, det_bf16* dq, det_bf16* dk, det_bf16* dv, int ld_d, void* ws, size_t ws_bytes,
                            void* stream) {
  return attn_bwd_impl(dout, q, k, v, out, lse, ld, ld_out, B, H, Hkv, S, window, dq, dk, dv, ld_d, ws, ws_bytes, stream, false);
}
extern "C" int det_attn_bwd_fixq(const det_bf16* dout, const det_bf16* q, const det_bf16* k, const det_bf16* v,
                                 const det_bf16* out, const float* lse, int ld, int ld_out, int B, int H, int Hkv, int S,
                                 int window, det_bf16* dq, det_bf16* dk, det_bf16* dv, int ld_d, void* ws,
                                 size_t ws_bytes, void* stream) {
  return attn_bwd_impl(dout, q, k, v, out, lse, ld, ld_out, B, H, Hkv, S, window, dq, dk, dv, ld_d, ws, ws_bytes, stream, true);
}
