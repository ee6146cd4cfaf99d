// Ordered full-precision contractions for the LM head (Sec. 3.2: the head stays out of quantisation).
//
// Every output is ONE f32 accumulator that starts at +0 (or at the value already in the output) and
// receives its terms in ascending order of the contraction index, each term an exact bf16 x bf16 product
// added with a separate rounding.  That fixes the order, so these GEMMs run on the FP32 ALUs:
// 128x256 output tile per CTA (smaller ones where those leave SMs idle: og_pick), 8x16 register tile per consumer thread,
// 16-deep slabs staged through a shared-memory ring as f32 by dedicated producer warps (k_ogemm in ogemm_core.cuh), packed
// two-lane FP32 instructions.  Because the product of two
// bf16 values is exact in binary32, "multiply, then add" and a fused multiply-add round the same exact sum
// once and give the same bits, unless the product is subnormal (the unfused product is then flushed to zero,
// the fused one is not).  Each slab is therefore checked for factors below 2^-63 while it is staged; clean
// slabs use the fused instruction, the others the two-instruction sequence.
#include "ogemm_core.cuh"
#include "../../include/det_test.h"

using namespace det;

static OgemmArgs plain_args(const void* A, const void* B, void* out, int I, int J, int C, int lda, int ldb, int ldo, int init) {
  OgemmArgs p = {};
  p.A = A; p.B = B; p.out = out; p.I = I; p.J = J; p.C = C; p.lda = lda; p.ldb = ldb; p.ldo = ldo; p.init = init;
  p.H = 1; p.nG = 1; p.b_div = 1;
  return p;
}

extern "C" int det_lmhead_fwd(const det_bf16* H, const det_bf16* W, int M, int V, int K, float* logits, void* stream) {
  if (!H || !W || !logits || M <= 0 || V <= 0 || K <= 0) return DET_ERR_ARG;
  if (K % 16 || V % 4) return DET_ERR_SHAPE;
  if (!aligned16(H) || !aligned16(W) || !aligned16(logits)) return DET_ERR_ALIGN;
  int rc = ogemm_launch<CONTIG, CONTIG, false, false, 0>(plain_args(H, W, logits, M, V, K, K, K, V, 0), 1, 1, (cudaStream_t)stream);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_lmhead_bwd(const float* dlogits, const det_bf16* H, const det_bf16* W, int M, int V, int K, det_bf16* dH,
                              float* dW, int first_chunk, void* stream) {
  if (!dlogits || !H || !W || !dH || !dW || M <= 0 || V <= 0 || K <= 0) return DET_ERR_ARG;
  if (K % 16 || V % 16 || M % 8) return DET_ERR_SHAPE;
  if (!aligned16(dlogits) || !aligned16(H) || !aligned16(W) || !aligned16(dH) || !aligned16(dW)) return DET_ERR_ALIGN;
  cudaStream_t st = (cudaStream_t)stream;
  // dH[m,k] = sum over v ascending of bf16(dlogits[m,v]) * W[v,k]; dW[v,k] (+)= sum over m ascending of bf16(dlogits[m,v]) * H[m,k].
  // The two are independent, and dW fills the SMs that dH leaves.  It must come second: with its CTAs first on the SMs the chains of dH
  // start when dW is nearly done (384 tokens: 7.3 instead of 4.3 ms for head and loss, which two streams left to chance).
  OgemmArgs h = plain_args(dlogits, W, dH, M, K, V, V, K, K, 0), w = plain_args(dlogits, H, dW, V, K, M, V, K, K, first_chunk ? 0 : 1);
  h.order = OG_LEAD;
  w.order = OG_FILL;
  int rc = ogemm_launch<CONTIG, STRIDED, true, true, 0>(h, 1, 1, st, (double)M * V * K / OG_RATES[0].full);
  if (rc != DET_OK) return rc;
  rc = ogemm_launch<STRIDED, STRIDED, true, false, 0>(w, 1, 1, st);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

// The three contractions of the head one by one, with the tile (an index into OG_RATES) given instead of picked
extern "C" int det_test_lmhead_tile(int which, int tile, const void* A, const det_bf16* B, int M, int V, int K, void* out, int first_chunk,
                                    void* stream) {
  if (!A || !B || !out || M <= 0 || V <= 0 || K <= 0 || which < 0 || which > 2 || tile < 0 || tile > 3) return DET_ERR_ARG;
  if (K % 16 || V % (which ? 16 : 4) || (which && M % 8)) return DET_ERR_SHAPE;
  if (!aligned16(A) || !aligned16(B) || !aligned16(out)) return DET_ERR_ALIGN;
  cudaStream_t st = (cudaStream_t)stream;
  int rc;
  if (which == 0) rc = ogemm_tile<CONTIG, CONTIG, false, false, 0>(tile, plain_args(A, B, out, M, V, K, K, K, V, 0), 1, st);
  else if (which == 1) rc = ogemm_tile<CONTIG, STRIDED, true, true, 0>(tile, plain_args(A, B, out, M, K, V, V, K, K, 0), 1, st);
  else rc = ogemm_tile<STRIDED, STRIDED, true, false, 0>(tile, plain_args(A, B, out, V, K, M, V, K, K, first_chunk ? 0 : 1), 1, st);
  if (rc != DET_OK) return rc;
  DET_CHECK_LAUNCH();
  return DET_OK;
}

extern "C" int det_test_lmhead_pick(int M, int V, int K) {
  if (M <= 0 || V <= 0 || K <= 0 || K % 16 || V % 4) return -1;
  return og_pick(OG_ROW_RATES, plain_args(nullptr, nullptr, nullptr, M, V, K, K, K, V, 0), 1, 1, 0, 0.0);
}
