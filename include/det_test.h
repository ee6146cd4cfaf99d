/* det_test.h -- test hooks of libdet.  Not part of the product boundary (include/det.h): these calls exist so that
 * tests can reach pieces that no product call exposes on their own.  Same conventions as det.h (device pointers,
 * stream-ordered, status codes). */
#ifndef DET_TEST_H
#define DET_TEST_H
#include "det.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Elementwise evaluation of one primitive of Sec. 2.1 ("Reproducible Operations") on device arrays: op 0 add, 1 sub,
 * 2 mul, 3 div, 4 sqrt(a), 5 det_exp(a), 6 det_log(a), 7 max, 8 bf16 round trip of a, 9 unfused a*b+b, 10 the form of
 * det_exp the softmax kernels use for arguments a <= 0 or NaN (same bits as op 5 there), 11 its two-lane form.  b may be NULL for unary ops.  Lets a test compare the device arithmetic with the CPU statement of the same rule. */
int det_test_prim(int op, const float* a, const float* b, float* out, size_t n, void* stream);

/* The GEMM core of the LSQ linears alone (Sec. 3.2 "int8 computation"): exact int8 x int8 -> int32 contraction
 * C[i,j] = sum_k A[i,k] B[j,k] on tcgen05.  I % 128 == 0, J % 128 == 0, K % 128 == 0, K < 2^17.  force_one_cta != 0
 * keeps the one-CTA kernel where the two-CTA 256 x 256 tiles (cta_group::2) would otherwise be chosen (both output
 * dimensions multiples of 256); integer accumulation is exact, so both give the same result. */
int det_test_igemm_tn(const int8_t* A, const int8_t* B, int I, int J, int K, int32_t* C, int force_one_cta, void* stream,
                      int* status_dev);

/* The bounded wait used by every kernel that waits on an mbarrier (TMA loads, tensor-core commits): one warp waits on a
 * barrier that nothing completes; after limit_cycles SM clocks (at most 4e9) the wait gives up, ORs DET_DEV_TIMEOUT into
 * *status_dev (device int) and the kernel returns, leaving the context usable.  No counterpart in the paper: it exists
 * so that the time-out path can be exercised without making a real kernel hang. */
int det_test_wait_timeout(int* status_dev, long long limit_cycles, void* stream);

/* The same wait by a whole warp of which only every other lane waits for nothing: gone_on (device, 32 ints) says for each lane whether it
 * would go on.  After limit_cycles all of them must have given up together. */
int det_test_wait_warp(int* gone_on, long long limit_cycles, void* stream);

/* One contraction of the LM head with a tile of the caller's choice (0: 128 x 256, 1: 128 x 128, 2: 64 x 128, 3: 32 x 64), so that a test can
 * run every tile at any size; the result does not depend on it.  which 0: logits f32 [M,V] of A = H, B = W as det_lmhead_fwd; 1: dH bf16
 * [M,K] of A = dlogits (f32), B = W; 2: dW f32 [V,K] of A = dlogits, B = H (first_chunk as there), as det_lmhead_bwd.  Same shape limits. */
int det_test_lmhead_tile(int which, int tile, const void* A, const det_bf16* B, int M, int V, int K, void* out, int first_chunk,
                         void* stream);

/* The tile (numbers as above) that det_lmhead_fwd takes on this device; -1 for sizes that it refuses. */
int det_test_lmhead_pick(int M, int V, int K);

/* det_attn_fwd_q with a form of the caller's choice: rows per CTA 128, 64 or 32, or 33 for 32 rows with two groups of warps; the result does not
 * depend on it. */
int det_test_attn_fwd(int rows, const det_bf16* q, const det_bf16* k, const det_bf16* v, int ld, int B, int H, int Hkv, int S, int window,
                      det_bf16* out, int ld_out, float* lse, const float* s_q, int8_t* qout, void* stream);

/* The form that det_attn_fwd takes on this device for that many heads (of all sequences together); 0 for sizes that it refuses. */
int det_test_attn_rows(int heads, int S, int window);

#ifdef __cplusplus
}
#endif
#endif
