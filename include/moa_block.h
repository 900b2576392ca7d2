/*
 * moa_block.h -- C ABI of the token-wise pieces of the transformer block for NVIDIA B200
 * (sm_100a): RMSNorm and the gated MLP, each forward and backward, and the GEMM of the projections.
 *
 * These are the pieces the paper's block section puts around attention ("RMSNorm, gated MLP",
 * hidden width d_ff, with the gated-MLP backward the dominant kernel of its block profile).
 * The paper names them and counts the block's traffic but prints no formula for either; the
 * definitions taken here are the usual ones and are stated with each call.
 *
 * Conventions (the same as moa_attn.h): every tensor argument is a DEVICE pointer to a
 * contiguous row-major array, 16-byte aligned; the caller owns every buffer, workspace
 * included; calls enqueue kernels on `stream` (a cudaStream_t passed as void*) and return
 * without synchronising; outputs are overwritten; errors come back only as moa_status.  When an argument, workspace or
 * architecture error is returned nothing has been enqueued -- except by moa_block_fwd and moa_block_bwd, which are sequences
 * of calls and return the first error of any of them, with the calls in front of it enqueued.  Where an output lies over an
 * input (dx over dy, say), a call gives what its steps, in the order of the formulas below, give one after the other.  bf16
 * storage, fp32 arithmetic.
 */
#ifndef MOA_BLOCK_H
#define MOA_BLOCK_H

#include "moa_attn.h"

#ifdef __cplusplus
extern "C" {
#endif

/* ------------------------------------------------------------------------- RMSNorm
 *   r_i  = 1 / sqrt( (1/d) sum_k x_ik^2 + eps )          y_ik = x_ik r_i g_k
 *   dg_k = sum_i dy_ik x_ik r_i
 *   dx_ik = r_i g_k dy_ik - x_ik r_i^3 (1/d) sum_m x_im g_m dy_im
 * x, y, dy, dx: [n,d]; g, dg: [d]; r: [n] fp32.  n >= 1; d a multiple of 8, 8 <= d <= 8192;
 * dtype MOA_BF16 (others: MOA_ERR_UNSUPPORTED).  HBM-bound: the forward reads x and writes y
 * once, the backward reads x and dy and writes dx once. */
typedef struct {
    int32_t n, d;
    float   eps;
    int32_t dtype;       /* moa_dtype of x, g, y, dy, dx, dg */
} moa_rmsnorm_desc;

/* Workspace of the backward: per-CTA partial sums of dg, reduced in a fixed order (so the
 * result does not depend on timing).  0 for an invalid desc. */
size_t moa_rmsnorm_workspace_bytes(const moa_rmsnorm_desc *desc);

/* Reads x, g; writes y and, when r != NULL, r (which the backward wants). */
moa_status moa_rmsnorm_fwd(const moa_rmsnorm_desc *desc, const void *x, const void *g,
                           void *y, float *r, void *stream);

/* Reads x, g, dy and r (as written by the forward for the same x; NULL: recomputed from x);
 * writes dx and dg.  dx_add (NULL or [n,d]) is added to dx: the gradient that reaches x past the
 * norm, along a residual connection. */
moa_status moa_rmsnorm_bwd(const moa_rmsnorm_desc *desc, const void *x, const void *g, const float *r,
                           const void *dy, const void *dx_add, void *dx, void *dg,
                           void *ws, size_t ws_bytes, void *stream);

/* ----------------------------------------------------------------------- gated MLP
 * SiLU-gated MLP without biases, weights stored [out, in]:
 *   a = x W1^T, u = x W3^T   [n,d_ff]      h = silu(a) * u,  silu(a) = a / (1 + exp(-a))
 *   y = h W2^T               [n,d]
 *   dh = dy W2,  da = dh u s (1 + a (1 - s)) with s = 1/(1+exp(-a)),  du = dh a s
 *   dW2 = dy^T h,  dW1 = da^T x,  dW3 = du^T x,  dx = da W1 + du W3
 * x, y, dy, dx: [n,d]; W1, W3, dW1, dW3: [d_ff,d]; W2, dW2: [d,d_ff]; a, u, h: [n,d_ff].
 * The contractions run on the tensor cores (tcgen05, fp32 accumulation in TMEM) with the
 * gate arithmetic fused into the epilogues of the GEMMs that produce a|u and dh, so dh is
 * never written to memory.  n >= 1; d and d_ff multiples of 8 (rows stay 16-byte aligned);
 * d_ff >= 8, d >= 8; dtype MOA_BF16. */
typedef struct {
    int32_t n, d, d_ff;
    int32_t dtype;
} moa_mlp_desc;

/* Forward.  Reads x, W1, W3, W2; writes a, u, h (kept for the backward, bf16) and y.  res (NULL or
 * [n,d]) is added to y in the epilogue of the last GEMM: the block's residual connection. */
moa_status moa_gated_mlp_fwd(const moa_mlp_desc *desc, const void *x, const void *W1, const void *W3,
                             const void *W2, const void *res, void *a, void *u, void *h, void *y, void *stream);

/* Workspace of the backward: da and du, [n,d_ff] each in the storage type.  0 for an invalid desc. */
size_t moa_gated_mlp_workspace_bytes(const moa_mlp_desc *desc);

/* Backward.  Reads x, the weights, a, u, h (as written by the forward) and dy; writes dx, dW1,
 * dW3, dW2.  Weight gradients are overwritten (not accumulated into). */
moa_status moa_gated_mlp_bwd(const moa_mlp_desc *desc, const void *x, const void *W1, const void *W3,
                             const void *W2, const void *a, const void *u, const void *h, const void *dy,
                             void *dx, void *dW1, void *dW3, void *dW2,
                             void *ws, size_t ws_bytes, void *stream);

/* ------------------------------------------------------------------------------ GEMM
 * The product the block's projections and their backward passes need, on the same tensor-core
 * kernel as the gated MLP:   C[M,N] = A B^T (+ R)
 * A is given as [M,K] row-major (a_layout = 0) or as [K,M] row-major (a_layout = 1); B as [N,K]
 * row-major (b_layout = 0) or as [K,N] row-major (b_layout = 1); C and the optional R are [M,N].
 * With weights stored [out,in]:  y = x W^T is (0,0);  dx = dy W is (0,1);  dW = dy^T x is (1,1) with
 * M = out, N = in, K = tokens.  R (NULL or [M,N]) is added in the epilogue: a residual connection, or
 * the running sum of a chain of products.  M, N, K >= 1; the row length of every array a multiple of
 * 8 (rows stay 16-byte aligned); dtype MOA_BF16; fp32 accumulation.
 * Tiling: 256 x 256 tiles on pairs of CTAs (one cluster of two, UMMAs of M = 256 reading half of B from each CTA's
 * shared memory), 128 x 256 output tiles on single CTAs where M is so small that pairs would need more waves, or 128 x 128 and
 * 128 x 64 where the wider ones would leave SMs idle; a small block's or gated MLP's backward sends out several products as one launch.
 * The environment variable MOA_GEMM_PAIR, read once per process, overrides the choice for
 * tests and measurements: 0 = never pairs, 2 = always pairs (no narrow tiles and no joint launches); the results do not depend on it beyond rounding order
 * (they are the same bits: every output element is one fp32 accumulation over K in the same order). */
typedef struct {
    int32_t M, N, K;
    int32_t a_layout, b_layout;
    int32_t dtype;
} moa_gemm_desc;
moa_status moa_gemm(const moa_gemm_desc *desc, const void *A, const void *B, const void *R, void *C, void *stream);

/* ---------------------------------------------------------------------- the block
 * A whole pre-norm transformer block as one call per direction: the sequence of the calls above with a packed Q/K/V
 * projection (host work only: a step of a small block spent more time between the calls than in them).
 *     h1 = RMSNorm(x; g1)    qkv = h1 Wqkv^T ([T, 3 H d], T = B n: its thirds are Q, K, V of a [B,n,3,H,d] array)
 *     o = attention(Q, K, V)    x2 = x + o Wo^T    h2 = RMSNorm(x2; g2)    y = x2 + gated_mlp(h2)
 * Every array is [T, H d] unless said otherwise; weights are stored [out,in].  The forward reads x and the weights and writes
 * the activations; the backward reads those, the weights and dy and writes the gradients.  Workspaces as for the single calls
 * (attention: MOA_OP_BWD).  The first error of a call of the sequence is returned; the calls in front of it have been enqueued. */
typedef struct {
    int32_t B, n, H, d, d_ff;
    int32_t causal;
    float   eps, scale;
} moa_block_desc;
typedef struct {
    const void *x, *g1, *g2, *Wqkv /* [3 H d, H d] */, *Wo, *W1 /* [d_ff, H d] */, *W3, *W2 /* [H d, d_ff] */;
    void *h1, *qkv /* [T, 3 H d] */, *o, *x2, *h2, *a /* [T, d_ff] */, *u, *h, *y;
    float *r1 /* [T] */, *r2, *L /* [B,H,n] */;
    const void *dy;                                                     /* from here on: backward only */
    void *dh2, *dx2, *dout /* gradient of o */, *dqkv, *dh1, *dx;
    void *dg1, *dg2, *dWqkv, *dWo, *dW1, *dW3, *dW2;
    void *norm_ws, *attn_ws, *mlp_ws;
    size_t norm_ws_bytes, attn_ws_bytes, mlp_ws_bytes;
} moa_block_arrays;
moa_status moa_block_fwd(const moa_block_desc *desc, const moa_block_arrays *arrays, void *stream);
moa_status moa_block_bwd(const moa_block_desc *desc, const moa_block_arrays *arrays, void *stream);

#ifdef __cplusplus
}
#endif
#endif /* MOA_BLOCK_H */
