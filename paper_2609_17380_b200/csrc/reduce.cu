// Order-fixed sums on CUDA cores: det_sum, global gradient norm, clip scaling, primitive test hook.
//
// A CTA reduces one aligned chunk of 16384 elements (64 leaves of 256) as a perfect subtree of the
// fixed pairwise tree: a lane reads 8 adjacent floats (two 128-bit loads) and pairs them in registers,
// a warp butterfly finishes the 256-element leaf, eight leaf sums are paired in registers, and the
// eight warp sums in shared memory.  The chunk sums are reduced by the same kernel until one value
// is left, so the tree depends on n only.
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "internal.h"
#include "../../include/det_test.h"

namespace det {

static std::atomic<unsigned long long> g_launches{0};
int note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); return 0; }

static std::mutex g_dev_mutex;

AuxStreams* aux_fork(cudaStream_t st) {
  static AuxStreams table[MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return nullptr;
  AuxStreams* a = &table[dev];
  {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!a->ok) {
      // all or nothing: what a failed attempt created is destroyed again, so a later call starts from scratch
      AuxStreams t = {};
      int ns = 0, ne = 0;
      bool good = true, have_fork = false;
      for (int i = 0; i < 2 && good; ++i) {
        good = cudaStreamCreateWithFlags(&t.s[i], cudaStreamNonBlocking) == cudaSuccess;
        if (good) ++ns;
        if (good) { good = cudaEventCreateWithFlags(&t.join[i], cudaEventDisableTiming) == cudaSuccess; if (good) ++ne; }
      }
      if (good) { good = cudaEventCreateWithFlags(&t.fork, cudaEventDisableTiming) == cudaSuccess; have_fork = good; }
      if (!good) {
        for (int i = 0; i < ns; ++i) cudaStreamDestroy(t.s[i]);
        for (int i = 0; i < ne; ++i) cudaEventDestroy(t.join[i]);
        if (have_fork) cudaEventDestroy(t.fork);
        cudaGetLastError();
        return nullptr;
      }
      t.ok = true;
      *a = t;
    }
  }
  if (cudaEventRecord(a->fork, st) != cudaSuccess) return nullptr;
  // if the second wait fails the first auxiliary stream already depends on `st`: still hand the streams out, the
  // join below is what the caller's stream order needs
  for (int i = 0; i < 2; ++i)
    if (cudaStreamWaitEvent(a->s[i], a->fork, 0) != cudaSuccess) { cudaGetLastError(); return nullptr; }
  return a;
}
bool aux_join(cudaStream_t st, AuxStreams* a) {
  if (!a) return true;
  bool ok = true;
  for (int i = 0; i < 2; ++i)
    if (cudaEventRecord(a->join[i], a->s[i]) != cudaSuccess || cudaStreamWaitEvent(st, a->join[i], 0) != cudaSuccess) ok = false;
  return ok;
}

int dev_ensure_smem(DevOnce& once, const void* fn, size_t bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return DET_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  if (!once.done[dev]) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) {
      cudaGetLastError();
      return DET_ERR_CUDA;
    }
    once.done[dev] = true;
  }
  return DET_OK;
}
int dev_sm_count() {
  static int sms[MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return 0;
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms[dev] = 0;
  return sms[dev];
}
unsigned long long launches() { return g_launches.load(std::memory_order_relaxed); }

template <bool SQ>
__global__ void __launch_bounds__(256) k_sum_chunk(const float* __restrict__ x, long long n, float* __restrict__ partial) {
  grid_dep();
  __shared__ float wsum[SUM_LEAVES];
  const float r = chunk_sum<SQ>(x, (long long)blockIdx.x * SUM_CHUNK, n, wsum);
  if (threadIdx.x == 0) partial[blockIdx.x] = r;
}

// One level of the sums of many tensors: job j is x[j][0..len[j]), its chunks are the blocks from first[j] on (a multiple of
// four where there are several, so that the next level's loads are aligned), and block c leaves its sum in out[c], or in
// per[who[j]] where the job has no other chunk.
constexpr int SUM_JOBS = 256;
struct SumJobs {
  int n;
  uint32_t first[SUM_JOBS + 1];
  const float* x[SUM_JOBS];
  long long len[SUM_JOBS];
  int who[SUM_JOBS];
};
template <bool SQ>
__global__ void __launch_bounds__(256) k_sum_jobs(const __grid_constant__ SumJobs jobs, float* __restrict__ out, float* __restrict__ per) {
  grid_dep();
  __shared__ float wsum[SUM_LEAVES];
  int lo = 0, hi = jobs.n - 1;         // the last job whose first block is <= this one
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs.first[mid] <= blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const long long base = (long long)(blockIdx.x - jobs.first[lo]) * SUM_CHUNK;
  if (base >= jobs.len[lo]) return;    // a block that only aligns the next job
  const float r = chunk_sum<SQ>(jobs.x[lo], base, jobs.len[lo], wsum);
  if (threadIdx.x == 0) {
    if (jobs.len[lo] <= SUM_CHUNK) per[jobs.who[lo]] = r;
    else out[blockIdx.x] = r;
  }
}

static inline long long nchunks(long long n) { return (n + SUM_CHUNK - 1) / SUM_CHUNK; }

// runs the multi-level reduction; result lands in out[0] (device).  ws must hold sum_ws floats.
size_t sum_ws_floats(size_t n) {
  size_t tot = 0;
  long long c = nchunks((long long)n);
  while (c > 1) { tot += align_up((size_t)c, 64); c = nchunks(c); }
  return tot + 64;
}

int sum_launch(const float* x, size_t n, int squares, float* out, float* ws, cudaStream_t st) {
  if (n == 0) { cudaMemsetAsync(out, 0, sizeof(float), st); return DET_OK; }
  const float* src = x;
  long long cur = (long long)n;
  bool sq = squares != 0;
  float* w = ws;
  while (true) {
    long long c = nchunks(cur);
    float* dst = (c == 1) ? out : w;
    if (sq) launch_after(k_sum_chunk<true>, (unsigned)c, 256, 0, st, src, cur, dst);
    else launch_after(k_sum_chunk<false>, (unsigned)c, 256, 0, st, src, cur, dst);
    if (c == 1) break;
    w += align_up((size_t)c, 64);
    src = dst;
    cur = c;
    sq = false;
  }
  return DET_OK;
}

// det_sum(x[0..n)), n <= SUM_CHUNK, times gs (the last levels of a sum and the scaling that follows it, in one launch)
__global__ void __launch_bounds__(256) k_sum_scaled(const float* __restrict__ x, int n, float gs, float* __restrict__ out) {
  grid_dep();
  __shared__ float wsum[SUM_LEAVES];
  const float r = chunk_sum<false>(x, 0, n, wsum);
  if (threadIdx.x == 0) out[0] = fmul(gs, r);
}
// Reduces x[0..n) until at most SUM_CHUNK nodes are left; x and n become what is left, ws what is free of the scratch.
void sum_to_chunk(const float*& x, size_t& n, float*& ws, cudaStream_t st) {
  while (n > (size_t)SUM_CHUNK) {
    const size_t c = (size_t)nchunks((long long)n);
    launch_after(k_sum_chunk<false>, (unsigned)c, 256, 0, st, x, (long long)n, ws);
    x = ws;
    ws += align_up(c, 64);
    n = c;
  }
}
int sum_scaled_launch(const float* x, size_t n, float gs, float* out, float* ws, cudaStream_t st) {
  sum_to_chunk(x, n, ws, st);
  launch_after(k_sum_scaled, 1, 256, 0, st, x, (int)n, gs, out);
  return DET_OK;
}

// the tree over the per-tensor sums (n <= SUM_CHUNK), the norm and the clip coefficient
__global__ void __launch_bounds__(256) k_norm_finish(const float* __restrict__ per, int n, float max_norm, float* norm_out,
                                                     float* coef_out, int* status) {
  grid_dep();
  __shared__ float wsum[SUM_LEAVES];
  const float total = n ? chunk_sum<false>(per, 0, n, wsum) : 0.0f;
  if (threadIdx.x) return;
  float nrm = fsqrt(total);
  norm_out[0] = nrm;
  float coef = 1.0f;
  if (max_norm > 0.0f) coef = fminf(1.0f, fdiv(max_norm, fadd(nrm, 1e-6f)));
  coef_out[0] = coef;
  if (!(fabsf(nrm) <= 3.4028234e38f)) or_status(status, DET_DEV_NONFINITE);
}

__global__ void __launch_bounds__(256) k_scale(float* __restrict__ g, size_t n, const float* __restrict__ coef) {
  const float c = coef[0];
  size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) * 4;
  if (i + 4 <= n) {
    float4 v = *reinterpret_cast<float4*>(g + i);
    v.x = fmul(v.x, c); v.y = fmul(v.y, c); v.z = fmul(v.z, c); v.w = fmul(v.w, c);
    *reinterpret_cast<float4*>(g + i) = v;
  } else {
    for (; i < n; ++i) g[i] = fmul(g[i], c);
  }
}

__global__ void k_prim(int op, const float* a, const float* b, float* out, size_t n) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x = a[i], y = b ? b[i] : 0.0f, r;
  switch (op) {
    case 0: r = fadd(x, y); break;
    case 1: r = fsub(x, y); break;
    case 2: r = fmul(x, y); break;
    case 3: r = fdiv(x, y); break;
    case 4: r = fsqrt(x); break;
    case 5: r = det_exp(x); break;
    case 6: r = det_log(x); break;
    case 7: r = fmaxf(x, y); break;
    case 8: {  // narrowing is only ever applied to flushed values; flush the raw input here
      uint32_t u = __float_as_uint(x);
      if (!(u & 0x7f800000u)) x = __uint_as_float(u & 0x80000000u);
      r = bf2f(f2bf(x));
      break;
    }
    case 9: r = fadd(fmul(x, y), y); break;
    case 10: r = det_exp_le0(x); break;
    case 11: {   // the two-lane form: this element in one lane, another argument in the other
      const float2 v = det_exp_le0_2((i & 1) ? make_float2(-0.75f, x) : make_float2(x, -1.5f), same2(c_one));
      r = (i & 1) ? v.y : v.x;
      break;
    }
    default: r = 0.0f;
  }
  out[i] = r;
}

}  // namespace det

using namespace det;

extern "C" unsigned long long det_launch_count(void) { return det::launches(); }

extern "C" int det_device_sm_count(void) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DET_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return DET_ERR_CUDA;
  return sms;
}

extern "C" int det_test_prim(int op, const float* a, const float* b, float* out, size_t n, void* stream) {
  if (!a || !out || op < 0 || op > 11) return DET_ERR_ARG;
  if (n == 0) return DET_OK;
  k_prim<<<DET_L((unsigned)((n + 255) / 256)), 256, 0, (cudaStream_t)stream>>>(op, a, b, out, n);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" size_t det_sum_ws_bytes(size_t n) { return sum_ws_floats(n) * sizeof(float); }

extern "C" int det_sum(const float* x, size_t n, int squares, float* out, void* ws, size_t ws_bytes, void* stream) {
  if (!out || (n && !x)) return DET_ERR_ARG;
  if (n && !aligned16(x)) return DET_ERR_ALIGN;
  if (ws_bytes < det_sum_ws_bytes(n) || (!ws && n > (size_t)SUM_CHUNK)) return DET_ERR_WORKSPACE;
  int rc = sum_launch(x, n, squares, out, (float*)ws, (cudaStream_t)stream);
  DET_CHECK_LAUNCH();
  return rc;
}

// Workspace: the per-tensor sums, then the chunk sums of one group of tensors (all levels), then the levels above
// SUM_CHUNK tensors.
extern "C" size_t det_grad_norm_ws_bytes(const size_t* n_elems, int ntensors) {
  size_t most = 0;
  for (int t0 = 0; t0 < ntensors; t0 += SUM_JOBS) {
    size_t need = 0;
    for (int t = t0; t < ntensors && t < t0 + SUM_JOBS; ++t) {
      long long c = (long long)n_elems[t];
      do { c = nchunks(c); need += (size_t)c + 4; } while (c > 1);
    }
    most = need + 4 * 64 > most ? need + 4 * 64 : most;                 // every level starts at a multiple of 64
  }
  const size_t nt = (size_t)(ntensors > 0 ? ntensors : 1);
  return (align_up(nt, 64) + 64 + align_up(most, 64) + sum_ws_floats(nt)) * sizeof(float);
}

// The sums of squares of all tensors run level by level together: a launch of its own per tensor and level (138 for a
// model of 87 tensors, 4 us each and one after the other) cost more than the 187 M values take to read.
extern "C" int det_grad_norm(const float* const* g_ptrs, const size_t* n_elems, int ntensors, float max_norm,
                             float* norm_out, float* coef_out, void* ws, size_t ws_bytes, void* stream,
                             int* status_dev) {
  if (ntensors < 0 || !norm_out || !coef_out || (ntensors && (!g_ptrs || !n_elems)) || !ws) return DET_ERR_ARG;
  if (ws_bytes < det_grad_norm_ws_bytes(n_elems, ntensors)) return DET_ERR_WORKSPACE;
  for (int t = 0; t < ntensors; ++t)
    if (n_elems[t] && (!g_ptrs[t] || !aligned16(g_ptrs[t]))) return g_ptrs[t] ? DET_ERR_ALIGN : DET_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  float* per = (float*)ws;
  float* total = per + align_up((size_t)(ntensors > 0 ? ntensors : 1), 64);
  float* scratch = total + 64;
  bool empty = false;
  for (int t = 0; t < ntensors; ++t) empty |= n_elems[t] == 0;
  if (empty) cudaMemsetAsync(per, 0, (size_t)ntensors * sizeof(float), st);   // a tensor without elements has the sum +0
  for (int t0 = 0; t0 < ntensors; t0 += SUM_JOBS) {
    SumJobs jobs;
    jobs.n = 0;
    for (int t = t0; t < ntensors && t < t0 + SUM_JOBS; ++t) {
      if (!n_elems[t]) continue;
      jobs.x[jobs.n] = g_ptrs[t];
      jobs.len[jobs.n] = (long long)n_elems[t];
      jobs.who[jobs.n++] = t;
    }
    float* out = scratch;
    bool sq = true;
    while (jobs.n) {
      long long c = 0;
      for (int j = 0; j < jobs.n; ++j) {
        if (jobs.len[j] > SUM_CHUNK) c = (c + 3) / 4 * 4;
        jobs.first[j] = (uint32_t)c;
        c += nchunks(jobs.len[j]);
      }
      if (c > 0x7fffffffll) return DET_ERR_SHAPE;
      jobs.first[jobs.n] = (uint32_t)c;
      if (sq) launch_after(k_sum_jobs<true>, (unsigned)c, 256, 0, st, jobs, out, per);
      else launch_after(k_sum_jobs<false>, (unsigned)c, 256, 0, st, jobs, out, per);
      int m = 0;
      for (int j = 0; j < jobs.n; ++j)
        if (jobs.len[j] > SUM_CHUNK) { jobs.x[m] = out + jobs.first[j]; jobs.len[m] = nchunks(jobs.len[j]); jobs.who[m] = jobs.who[j]; ++m; }
      jobs.n = m;
      out += align_up((size_t)c, 64);
      sq = false;
    }
  }
  int n = ntensors;
  const float* src = per;
  if (n > SUM_CHUNK) {
    sum_launch(per, (size_t)n, 0, total, scratch, st);
    src = total;
    n = 1;
  }
  launch_after(k_norm_finish, 1, 256, 0, st, src, n, max_norm, norm_out, coef_out, status_dev);
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_scale_inplace(float* g, size_t n, const float* coef_dev, void* stream) {
  if ((n && !g) || !coef_dev) return DET_ERR_ARG;
  if (n && !aligned16(g)) return DET_ERR_ALIGN;
  if (n == 0) return DET_OK;
  k_scale<<<DET_L((unsigned)((n + 1023) / 1024)), 256, 0, (cudaStream_t)stream>>>(g, n, coef_dev);
  DET_CHECK_LAUNCH();
  return DET_OK;
}
