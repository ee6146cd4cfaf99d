// Chunked SHA-256 tensor hash (Appendix B: per-step state hash), many tensors per launch.
//
// Level 1 hashes every 4 KiB chunk of every tensor, the levels above it the concatenated digests of the level below while
// more than 128 remain, and the root is SHA-256(remaining digests || u64le(nbytes)).  A chunk is one sequential chain of
// 64 + 1 compressions, so what a level costs is either the integer pipes (many chunks: k_sha_chunks, a thread per
// chunk) or the latency of one chain (few chunks: k_sha_few, four lanes per chunk), and never its launch: the levels of
// all tensors of a call run together.
#include "common.cuh"
#include "internal.h"

namespace det {

constexpr int HASH_JOBS = 256;   // tensors per launch
constexpr size_t HASH_CHUNK = 4096;

// Job j covers the bytes base[j] .. base[j] + nbytes[j]; its chunks have the numbers first[j] .. first[j + 1] - 1 of the
// launch, and chunk i leaves its digest at out + 32 i.  total: the tensor's byte count, appended to the message of a root.
struct HashJobs {
  int n;
  uint32_t first[HASH_JOBS + 1];
  const uint8_t* base[HASH_JOBS];
  unsigned long long nbytes[HASH_JOBS];
  unsigned long long total[HASH_JOBS];
};

__device__ __forceinline__ uint32_t rotr32(uint32_t x, int r) { return __funnelshift_r(x, x, r); }
__device__ __forceinline__ uint32_t bswap(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

#define SHA_K_LIST \
    0x428a2f98, 0x71374491, 0xb5c0fbcf, 0xe9b5dba5, 0x3956c25b, 0x59f111f1, 0x923f82a4, 0xab1c5ed5, 0xd807aa98, \
    0x12835b01, 0x243185be, 0x550c7dc3, 0x72be5d74, 0x80deb1fe, 0x9bdc06a7, 0xc19bf174, 0xe49b69c1, 0xefbe4786, \
    0x0fc19dc6, 0x240ca1cc, 0x2de92c6f, 0x4a7484aa, 0x5cb0a9dc, 0x76f988da, 0x983e5152, 0xa831c66d, 0xb00327c8, \
    0xbf597fc7, 0xc6e00bf3, 0xd5a79147, 0x06ca6351, 0x14292967, 0x27b70a85, 0x2e1b2138, 0x4d2c6dfc, 0x53380d13, \
    0x650a7354, 0x766a0abb, 0x81c2c92e, 0x92722c85, 0xa2bfe8a1, 0xa81a664b, 0xc24b8b70, 0xc76c51a3, 0xd192e819, \
    0xd6990624, 0xf40e3585, 0x106aa070, 0x19a4c116, 0x1e376c08, 0x2748774c, 0x34b0bcb5, 0x391c0cb3, 0x4ed8aa4a, \
    0x5b9cca4f, 0x682e6ff3, 0x748f82ee, 0x78a5636f, 0x84c87814, 0x8cc70208, 0x90befffa, 0xa4506ceb, 0xbef9a3f7, \
    0xc67178f2

__device__ __forceinline__ uint32_t big_s1(uint32_t e) { return rotr32(e, 6) ^ rotr32(e, 11) ^ rotr32(e, 25); }
__device__ __forceinline__ uint32_t big_s0(uint32_t a) { return rotr32(a, 2) ^ rotr32(a, 13) ^ rotr32(a, 22); }
__device__ __forceinline__ uint32_t sha_ch(uint32_t e, uint32_t f, uint32_t g) { return (e & f) ^ (~e & g); }
__device__ __forceinline__ uint32_t sha_maj(uint32_t a, uint32_t b, uint32_t c) { return (a & b) ^ (a & c) ^ (b & c); }
__device__ __forceinline__ uint32_t small_s0(uint32_t w) { return rotr32(w, 7) ^ rotr32(w, 18) ^ (w >> 3); }
__device__ __forceinline__ uint32_t small_s1(uint32_t w) { return rotr32(w, 17) ^ rotr32(w, 19) ^ (w >> 10); }

// a + b on the multiply-add pipe, with `one` a 1 that the compiler does not know
__constant__ uint32_t c_one_u = 1u;
__device__ __forceinline__ uint32_t opaque_one() {
  uint32_t one;
  asm volatile("mov.u32 %0, %1;" : "=r"(one) : "r"(c_one_u));
  return one;
}
template <bool MAD>
__device__ __forceinline__ uint32_t add_mad(uint32_t a, uint32_t b, uint32_t one) {
  if (!MAD) return a + b;
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(one), "r"(b));
  return d;
}
// one compression: 64 rounds with the message schedule kept in a rolling window of 16 words.  The integer pipe is what a
// thread per chunk is bound by (96 % busy with 21 logic, shift and add instructions a round, 1 GiB at 0.86 TB/s), while the
// multiply-add pipe idles, so most additions go there: 1.03 TB/s with the ones below, 0.86 to 1.02 with other choices (all
// of the schedule 1.02, without the schedule 1.01, the round constant's too 0.92).
template <bool MAD>
__device__ __forceinline__ void sha_rounds(uint32_t (&h)[8], uint32_t (&w)[16], uint32_t one) {
  constexpr uint32_t K[64] = {SHA_K_LIST};
  auto add = [one](uint32_t x, uint32_t y) { return add_mad<MAD>(x, y, one); };
  uint32_t a = h[0], b = h[1], c = h[2], d = h[3], e = h[4], f = h[5], g = h[6], hh = h[7];
#pragma unroll
  for (int i = 0; i < 64; ++i) {
    if (i >= 16)
      w[i & 15] = add(add(w[(i + 9) & 15], small_s1(w[(i + 14) & 15])), w[i & 15] + small_s0(w[(i + 1) & 15]));
    const uint32_t t1 = add(big_s1(e), add(sha_ch(e, f, g), add(hh, w[i & 15] + K[i])));
    const uint32_t t2 = add(big_s0(a), sha_maj(a, b, c));
    hh = g; g = f; f = e; e = add(d, t1); d = c; c = b; b = a; a = add(t2, t1);
  }
  h[0] += a; h[1] += b; h[2] += c; h[3] += d; h[4] += e; h[5] += f; h[6] += g; h[7] += hh;
}

__device__ __forceinline__ void sha_init(uint32_t (&h)[8]) {
  h[0] = 0x6a09e667; h[1] = 0xbb67ae85; h[2] = 0x3c6ef372; h[3] = 0xa54ff53a;
  h[4] = 0x510e527f; h[5] = 0x9b05688c; h[6] = 0x1f83d9ab; h[7] = 0x5be0cd19;
}
__device__ __forceinline__ void sha_store(uint8_t* out, const uint32_t (&h)[8]) {
  uint4* o = reinterpret_cast<uint4*>(out);
  o[0] = make_uint4(bswap(h[0]), bswap(h[1]), bswap(h[2]), bswap(h[3]));
  o[1] = make_uint4(bswap(h[4]), bswap(h[5]), bswap(h[6]), bswap(h[7]));
}
// A message: `len` bytes at p (4-byte aligned), then for a root the 8 bytes of `total`, then the padding of SHA-256.
struct ShaMsg {
  const uint8_t* p;
  uint32_t len, sfx;
  unsigned long long total;
  __device__ __forceinline__ uint32_t blocks() const { return (len + sfx + 9 + 63) / 64; }
  // block b where it is not wholly message bytes, a word at a time (a byte at a time, through a test per byte, the two short chains
  // of a tensor of 16 bytes took 19.0 us).  A root's digests end on a word, so only a message without suffix has a word that
  // holds message bytes and padding.
  __device__ __noinline__ void ragged_block(uint32_t b, uint32_t* w) const {
    const uint32_t end = 64 * blocks();
    const unsigned long long bits = (unsigned long long)(len + sfx) * 8ull;
    for (int k = 0; k < 16; ++k) {
      const uint32_t i = b * 64 + 4 * k;
      uint32_t v = 0;
      if (i + 4 <= len) v = bswap(*reinterpret_cast<const uint32_t*>(p + i));
      else if (i + 8 >= end) v = (uint32_t)(i + 8 == end ? bits >> 32 : bits);
      else if (i < len + sfx && sfx) v = bswap((uint32_t)(i == len ? total : total >> 32));
      else if (i <= len + sfx && i + 4 > len + sfx) {
        v = 0x80000000u;
        for (uint32_t e = len + sfx; e > i; --e) v = (v >> 8) | ((uint32_t)p[e - 1] << 24);
      }
      w[k] = v;
    }
  }
};
template <bool ROOT>
__device__ __forceinline__ ShaMsg sha_msg(const HashJobs& jobs, uint32_t chunk) {
  int lo = 0, hi = jobs.n - 1;         // the last job whose first chunk is <= chunk
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs.first[mid] <= chunk) lo = mid; else hi = mid - 1;
  }
  const size_t off = (size_t)(chunk - jobs.first[lo]) * HASH_CHUNK;
  const size_t left = jobs.nbytes[lo] - off;
  ShaMsg m;
  m.p = jobs.base[lo] + off;
  m.len = (uint32_t)(left < HASH_CHUNK ? left : HASH_CHUNK);
  m.sfx = ROOT ? 8 : 0;
  m.total = ROOT ? jobs.total[lo] : 0;
  return m;
}

// Many chunks: a thread per chunk, the next 64-byte block on its way while the rounds of the current one run (sha_rounds says what
// bounds it).  A plain launch that lets nothing in early: the few CTAs of the next level would be packed on two or three SMs (grid_wait in
// common.cuh) and their chains share the schedulers there (whole hash of 10240 chunks 0.463 -> 0.228 ms, of 65536 0.784 -> 0.485, of 262144
// 1.53 -> 1.23).
template <bool MAD>
__global__ void __launch_bounds__(64) k_sha_chunks(const __grid_constant__ HashJobs jobs, uint8_t* __restrict__ out) {
  const uint32_t c = blockIdx.x * 64 + threadIdx.x;
  if (c >= jobs.first[jobs.n]) return;
  const ShaMsg msg = sha_msg<false>(jobs, c);
  const uint32_t one = opaque_one();
  uint32_t h[8], w[16];
  sha_init(h);
  const uint32_t full = msg.len / 64, nb = msg.blocks();
  // the next 64-byte block is fetched while the 64 rounds of the current one run
  uint4 nx[4];
  if (full) {
#pragma unroll
    for (int k = 0; k < 4; ++k) nx[k] = __ldg(reinterpret_cast<const uint4*>(msg.p) + k);
  }
  for (uint32_t b = 0; b < nb; ++b) {
    if (b < full) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint4 u = nx[k];
        w[4 * k] = bswap(u.x); w[4 * k + 1] = bswap(u.y); w[4 * k + 2] = bswap(u.z); w[4 * k + 3] = bswap(u.w);
      }
      if (b + 1 < full) {
        const uint4* q = reinterpret_cast<const uint4*>(msg.p + (b + 1) * 64);
#pragma unroll
        for (int k = 0; k < 4; ++k) nx[k] = __ldg(q + k);
      }
    } else {
      uint32_t t[16];
      msg.ragged_block(b, t);
#pragma unroll
      for (int k = 0; k < 16; ++k) w[k] = t[k];
    }
    sha_rounds<MAD>(h, w, one);
  }
  sha_store(out + (size_t)c * 32, h);
}

// Few chunks: eight chains per CTA, four lanes each.  Only the 64 rounds of a block depend on the block before, so the four lanes
// of a chain expand the schedules of its next four blocks side by side (schedule word + round constant, through shared memory)
// and the chain itself is rounds alone: 12 instructions a round on the half-rate integer pipe instead of 22, ordered so that a and
// e depend on the round before through one rotation, one exclusive or and one addition each.  A warp alone on its scheduler is bound by
// that pipe, two cycles an instruction, so the additions that nothing waits for (schedule word + h + d, maj - d) go to the
// multiply-add pipe: all levels of 1 MiB 138.6 -> 133.0 us, one chunk 72.7 -> 69.9 (all additions there: slower, by their latency).  Their 1 is
// the grid's height: from constant memory it was a miss that short chains wait for (60 bytes 13.7 -> 14.1 us, 13.8 with this).  While there
// are schedulers to spare a second warp does the expanding, double-buffered.  65 blocks: 0.119 ms with a thread per chunk, 0.074 with
// one warp per CTA, 0.063 with two.
constexpr int SF_CH = 8, SF_PITCH = 68;
template <bool ROOT>
__global__ void __launch_bounds__(64) k_sha_few(const __grid_constant__ HashJobs jobs, uint8_t* __restrict__ out) {
  grid_dep();
  __shared__ __align__(16) uint32_t ws[2][4 * SF_CH * SF_PITCH];
  constexpr uint32_t K[64] = {SHA_K_LIST};
  const int ch = (threadIdx.x & 31) >> 2, sub = threadIdx.x & 3;
  const bool pair = blockDim.x == 64, expand = threadIdx.x >= 32;
  const uint32_t c = blockIdx.x * SF_CH + ch;
  const bool have = c < jobs.first[jobs.n];
  ShaMsg msg = {};
  uint32_t nb = 0;
  if (have) { msg = sha_msg<ROOT>(jobs, c); nb = msg.blocks(); }
  const uint32_t full = have ? msg.len / 64 : 0, nbmax = __reduce_max_sync(0xffffffffu, nb);
  uint4 nx[4];
  auto fetch = [&](uint32_t b) {
    if (b < full) {
#pragma unroll
      for (int k = 0; k < 4; ++k) nx[k] = __ldg(reinterpret_cast<const uint4*>(msg.p + (size_t)b * 64) + k);
    }
  };
  auto schedule = [&](uint32_t b, uint32_t* row) {   // of block b, whose words are in nx
    if (b >= nb) return;
    uint32_t w[16];
    if (b < full) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint4 u = nx[k];
        w[4 * k] = bswap(u.x); w[4 * k + 1] = bswap(u.y); w[4 * k + 2] = bswap(u.z); w[4 * k + 3] = bswap(u.w);
      }
    } else {
      uint32_t t[16];
      msg.ragged_block(b, t);
#pragma unroll
      for (int k = 0; k < 16; ++k) w[k] = t[k];
    }
    fetch(b + 4);
#pragma unroll
    for (int i = 0; i < 64; i += 4) {
      uint32_t t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int j = i + k;
        if (j >= 16) w[j & 15] += small_s0(w[(j + 1) & 15]) + w[(j + 9) & 15] + small_s1(w[(j + 14) & 15]);
        t[k] = w[j & 15] + K[j];
      }
      *reinterpret_cast<uint4*>(row + i) = make_uint4(t[0], t[1], t[2], t[3]);
    }
  };
  const uint32_t one = gridDim.y, minus_one = 0u - one;   // 1, which the compiler does not know
  uint32_t h[8];
  sha_init(h);
  // a pair: the expanding warp is four blocks ahead; a single warp does one after the other
  if (!pair || expand) fetch(sub);
  for (int b0 = pair ? -4 : 0; b0 < (int)nbmax; b0 += 4) {
    uint32_t* next = ws[pair ? (b0 / 4 + 1) & 1 : 0];
    const uint32_t* cur = ws[pair ? (b0 / 4) & 1 : 0];
    if (!pair || expand) schedule((uint32_t)(b0 + (pair ? 4 : 0) + sub), next + (sub * SF_CH + ch) * SF_PITCH);
    if (!pair) __syncwarp();
    if (!expand && b0 >= 0) {
#pragma unroll 1
      for (int s = 0; s < 4; ++s) {
        if ((uint32_t)(b0 + s) < nb) {
          const uint32_t* row = cur + (s * SF_CH + ch) * SF_PITCH;
          uint32_t a = h[0], b = h[1], cc = h[2], d = h[3], e = h[4], f = h[5], g = h[6], hh = h[7];
#pragma unroll
          for (int i = 0; i < 64; i += 4) {
            const uint4 u = *reinterpret_cast<const uint4*>(row + i);
            const uint32_t wk[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t dx = add_mad<true>(add_mad<true>(wk[k], hh, one), d, one);
              const uint32_t en = big_s1(e) + sha_ch(e, f, g) + dx;
              const uint32_t an = big_s0(a) + add_mad<true>(d, sha_maj(a, b, cc), minus_one) + en;
              hh = g; g = f; f = e; e = en; d = cc; cc = b; b = a; a = an;
            }
          }
          h[0] += a; h[1] += b; h[2] += cc; h[3] += d; h[4] += e; h[5] += f; h[6] += g; h[7] += hh;
        }
      }
    }
    __syncthreads();
  }
  if (have && !expand && sub == 0) sha_store(out + (size_t)c * 32, h);
}

// The rule, 65 blocks a chunk, 148 SMs of four schedulers.  Where the latency of a chain is what counts the form with the shorter chain
// is taken: four lanes per chunk and a second warp while there are schedulers to spare (8 to 2368 chunks: 0.063 ms, one warp 0.074, a
// thread per chunk 0.119), one warp while its warps do not outnumber the schedulers (up to 4736 chunks: 0.077, 0.120, 0.120), then
// a thread per chunk with plain additions up to one warp per scheduler (6000: 0.121, four lanes 0.139, the multiply-add pipe's longer
// latency 0.129; 18944: 0.123, 0.270, 0.131).  Beyond that the integer pipe is what counts (20480: 0.215 plain, 0.181; 65536: 0.410, 0.342;
// 262144: 1.33, 1.08).
static void sha_few_launch(bool root, const HashJobs& jobs, uint32_t n, uint8_t* out, int sms, cudaStream_t st) {
  const unsigned ctas = (n + SF_CH - 1) / SF_CH;
  launch_after(root ? k_sha_few<true> : k_sha_few<false>, ctas, ctas <= 2u * (unsigned)sms ? 64 : 32, 0, st, jobs, out);
}
static int hash_level(const HashJobs& jobs, uint8_t* out, cudaStream_t st) {
  const uint32_t n = jobs.first[jobs.n];
  if (!n) return DET_OK;
  const int sms = dev_sm_count();
  if (sms <= 0) return DET_ERR_CUDA;
  if (n <= (uint32_t)sms * 4 * SF_CH) sha_few_launch(false, jobs, n, out, sms, st);
  else if (n <= (uint32_t)sms * 4 * 32) k_sha_chunks<false><<<DET_L((n + 63) / 64), 64, 0, st>>>(jobs, out);
  else k_sha_chunks<true><<<DET_L((n + 63) / 64), 64, 0, st>>>(jobs, out);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

static inline size_t chunks_of(size_t nbytes) { return (nbytes + HASH_CHUNK - 1) / HASH_CHUNK; }

}  // namespace det

using namespace det;

// The digests of every level of every tensor of a group lie one after the other: 32 bytes per chunk.
extern "C" size_t det_tensor_hash_batch_ws_bytes(const size_t* nbytes, int ntensors) {
  size_t most = 0;
  for (int t0 = 0; t0 < ntensors; t0 += HASH_JOBS) {
    size_t need = 0;
    for (int t = t0; t < ntensors && t < t0 + HASH_JOBS; ++t) {
      size_t nc = chunks_of(nbytes[t]);
      need += nc;
      while (nc > 128) { nc = chunks_of(nc * 32); need += nc; }
    }
    most = need > most ? need : most;
  }
  return most * 32 + 256;
}
extern "C" int det_tensor_hash_batch(const void* const* ptrs, const size_t* nbytes, int ntensors, uint8_t* roots_dev, void* ws,
                                     size_t ws_bytes, void* stream) {
  if (ntensors < 0 || (ntensors && (!ptrs || !nbytes || !roots_dev))) return DET_ERR_ARG;
  if (ntensors == 0) return DET_OK;
  for (int t = 0; t < ntensors; ++t) {
    if (nbytes[t] && !ptrs[t]) return DET_ERR_ARG;
    if (nbytes[t] && !aligned16(ptrs[t])) return DET_ERR_ALIGN;
  }
  if (!aligned16(roots_dev)) return DET_ERR_ALIGN;
  if (!ws || !aligned16(ws) || ws_bytes < det_tensor_hash_batch_ws_bytes(nbytes, ntensors)) return DET_ERR_WORKSPACE;
  const int sms = dev_sm_count();
  if (sms <= 0) return DET_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)stream;
  for (int t0 = 0; t0 < ntensors; t0 += HASH_JOBS) {
    const int n = ntensors - t0 < HASH_JOBS ? ntensors - t0 : HASH_JOBS;
    uint8_t* out = (uint8_t*)ws;
    HashJobs root, lv;                // lv: the tensors that still have a level to go, with their current bytes
    int who[HASH_JOBS];
    root.n = n;
    lv.n = n;
    for (int t = 0; t < n; ++t) {
      who[t] = t;
      lv.base[t] = (const uint8_t*)ptrs[t0 + t];
      lv.nbytes[t] = nbytes[t0 + t];
      root.first[t] = (uint32_t)t;
      root.total[t] = nbytes[t0 + t];
    }
    root.first[n] = (uint32_t)n;
    while (lv.n) {
      size_t c = 0;
      for (int j = 0; j < lv.n; ++j) { lv.first[j] = (uint32_t)c; c += chunks_of(lv.nbytes[j]); }
      if (c > 0xffffffffull) return DET_ERR_SHAPE;
      lv.first[lv.n] = (uint32_t)c;
      const int rc = hash_level(lv, out, st);
      if (rc != DET_OK) return rc;
      // a tensor with at most 128 digests goes to its root, the others to the next level
      int m = 0;
      for (int j = 0; j < lv.n; ++j) {
        const size_t nc = chunks_of(lv.nbytes[j]);
        const uint8_t* dig = out + (size_t)lv.first[j] * 32;
        if (nc <= 128) { root.base[who[j]] = dig; root.nbytes[who[j]] = nc * 32; }
        else { lv.base[m] = dig; lv.nbytes[m] = nc * 32; who[m] = who[j]; ++m; }
      }
      out += c * 32;
      lv.n = m;
    }
    sha_few_launch(true, root, (uint32_t)n, roots_dev + (size_t)t0 * 32, sms, st);
    DET_CHECK_LAUNCH();
  }
  return DET_OK;
}

// One tensor: the batch of one, and 256 bytes for the root of the synchronising call.
extern "C" size_t det_tensor_hash_ws_bytes(size_t nbytes) {
  return align_up(det_tensor_hash_batch_ws_bytes(&nbytes, 1), 256) + 256;
}
extern "C" int det_tensor_hash_async(const void* p, size_t nbytes, uint8_t* out32_dev, void* ws, size_t ws_bytes,
                                     void* stream) {
  if ((nbytes && !p) || !out32_dev) return DET_ERR_ARG;
  if (ws_bytes < det_tensor_hash_ws_bytes(nbytes) || !ws || !aligned16(ws)) return DET_ERR_WORKSPACE;
  return det_tensor_hash_batch(&p, &nbytes, 1, out32_dev, ws, ws_bytes, stream);
}
extern "C" int det_tensor_hash(const void* p, size_t nbytes, uint8_t* out32_host, void* ws, size_t ws_bytes,
                               void* stream) {
  if (!out32_host) return DET_ERR_ARG;
  if (ws_bytes < det_tensor_hash_ws_bytes(nbytes) || !ws || !aligned16(ws)) return DET_ERR_WORKSPACE;
  uint8_t* root = (uint8_t*)ws + det_tensor_hash_ws_bytes(nbytes) - 256;
  int rc = det_tensor_hash_async(p, nbytes, root, ws, ws_bytes, stream);
  if (rc != DET_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(out32_host, root, 32, cudaMemcpyDeviceToHost, st) != cudaSuccess) return DET_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DET_ERR_CUDA;
  return DET_OK;
}
