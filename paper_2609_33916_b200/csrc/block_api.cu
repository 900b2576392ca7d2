// C-ABI entry points of the block pieces (include/moa_block.h): argument checks and the sequence
// of kernel launches of each operation.  No arithmetic here.
#include "common.cuh"
#include "moa_block.h"

using namespace moa;

namespace {

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool finite(float v) { return v == v && v - v == 0.f; }

moa_status check_rmsnorm(const moa_rmsnorm_desc *d)
{
    if (!d) return MOA_ERR_INVALID_ARG;
    if (d->n <= 0 || d->d <= 0) return MOA_ERR_INVALID_ARG;
    if (!finite(d->eps) || d->eps < 0.f) return MOA_ERR_INVALID_ARG;
    if (d->dtype != MOA_BF16 && d->dtype != MOA_F32) return MOA_ERR_INVALID_ARG;
    if (d->dtype != MOA_BF16) return MOA_ERR_UNSUPPORTED;
    if (d->d % 8 != 0 || d->d > 8192) return MOA_ERR_UNSUPPORTED;
    return MOA_OK;
}

moa_status check_mlp(const moa_mlp_desc *d)
{
    if (!d) return MOA_ERR_INVALID_ARG;
    if (d->n <= 0 || d->d <= 0 || d->d_ff <= 0) return MOA_ERR_INVALID_ARG;
    if (d->dtype != MOA_BF16 && d->dtype != MOA_F32) return MOA_ERR_INVALID_ARG;
    if (d->dtype != MOA_BF16) return MOA_ERR_UNSUPPORTED;
    if (d->d % 8 != 0 || d->d_ff % 8 != 0) return MOA_ERR_UNSUPPORTED;       // rows of every array stay 16-byte aligned
    if ((long long)d->n * d->d_ff >= (1LL << 40)) return MOA_ERR_UNSUPPORTED;
    return MOA_OK;
}

size_t mlp_half_ws(const moa_mlp_desc *d) { return ((size_t)d->n * d->d_ff * 2 + 255) / 256 * 256; }

}  // namespace

extern "C" {

size_t moa_rmsnorm_workspace_bytes(const moa_rmsnorm_desc *desc)
{
    if (check_rmsnorm(desc) != MOA_OK) return 0;
    return rmsnorm_workspace_bytes(desc->n, desc->d);
}

moa_status moa_rmsnorm_fwd(const moa_rmsnorm_desc *desc, const void *x, const void *g, void *y, float *r, void *stream)
{
    moa_status s = check_rmsnorm(desc);
    if (s != MOA_OK) return s;
    if (!x || !g || !y) return MOA_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(g) || !aligned16(y) || (r && !aligned16(r))) return MOA_ERR_INVALID_ARG;
    if ((s = check_device_arch()) != MOA_OK) return s;
    return rmsnorm_fwd(desc->n, desc->d, desc->eps, x, g, y, r, (cudaStream_t)stream) == cudaSuccess ? MOA_OK : MOA_ERR_CUDA;
}

moa_status moa_rmsnorm_bwd(const moa_rmsnorm_desc *desc, const void *x, const void *g, const float *r,
                           const void *dy, const void *dx_add, void *dx, void *dg, void *ws, size_t ws_bytes, void *stream)
{
    moa_status s = check_rmsnorm(desc);
    if (s != MOA_OK) return s;
    if (!x || !g || !dy || !dx || !dg) return MOA_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(g) || !aligned16(dy) || !aligned16(dx) || !aligned16(dg) || (r && !aligned16(r)) ||
        (dx_add && !aligned16(dx_add)))
        return MOA_ERR_INVALID_ARG;
    if (!ws || ws_bytes < rmsnorm_workspace_bytes(desc->n, desc->d)) return MOA_ERR_WORKSPACE;
    if (!aligned16(ws)) return MOA_ERR_INVALID_ARG;
    if ((s = check_device_arch()) != MOA_OK) return s;
    return rmsnorm_bwd(desc->n, desc->d, desc->eps, x, g, r, dy, dx_add, dx, dg, ws, (cudaStream_t)stream) == cudaSuccess
               ? MOA_OK : MOA_ERR_CUDA;
}

size_t moa_gated_mlp_workspace_bytes(const moa_mlp_desc *desc)
{
    if (check_mlp(desc) != MOA_OK) return 0;
    return 2 * mlp_half_ws(desc);
}

moa_status moa_gated_mlp_fwd(const moa_mlp_desc *desc, const void *x, const void *W1, const void *W3, const void *W2,
                             const void *res, void *a, void *u, void *h, void *y, void *stream)
{
    moa_status s = check_mlp(desc);
    if (s != MOA_OK) return s;
    if (!x || !W1 || !W3 || !W2 || !a || !u || !h || !y) return MOA_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(W1) || !aligned16(W3) || !aligned16(W2) || !aligned16(a) || !aligned16(u) ||
        !aligned16(h) || !aligned16(y) || (res && !aligned16(res)))
        return MOA_ERR_INVALID_ARG;
    if ((s = check_device_arch()) != MOA_OK) return s;
    return gated_mlp_fwd(desc->n, desc->d, desc->d_ff, x, W1, W3, W2, res, a, u, h, y, (cudaStream_t)stream) == cudaSuccess
               ? MOA_OK : MOA_ERR_CUDA;
}

moa_status moa_gated_mlp_bwd(const moa_mlp_desc *desc, const void *x, const void *W1, const void *W3, const void *W2,
                             const void *a, const void *u, const void *h, const void *dy,
                             void *dx, void *dW1, void *dW3, void *dW2, void *ws, size_t ws_bytes, void *stream)
{
    moa_status s = check_mlp(desc);
    if (s != MOA_OK) return s;
    if (!x || !W1 || !W3 || !W2 || !a || !u || !h || !dy || !dx || !dW1 || !dW3 || !dW2) return MOA_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(W1) || !aligned16(W3) || !aligned16(W2) || !aligned16(a) || !aligned16(u) ||
        !aligned16(h) || !aligned16(dy) || !aligned16(dx) || !aligned16(dW1) || !aligned16(dW3) || !aligned16(dW2))
        return MOA_ERR_INVALID_ARG;
    if (!ws || ws_bytes < 2 * mlp_half_ws(desc)) return MOA_ERR_WORKSPACE;
    if (!aligned16(ws)) return MOA_ERR_INVALID_ARG;
    if ((s = check_device_arch()) != MOA_OK) return s;
    void *da = ws, *du = (char *)ws + mlp_half_ws(desc);
    return gated_mlp_bwd(desc->n, desc->d, desc->d_ff, x, W1, W3, W2, a, u, h, dy, da, du, dx, dW1, dW3, dW2,
                         (cudaStream_t)stream) == cudaSuccess ? MOA_OK : MOA_ERR_CUDA;
}

moa_status moa_gemm(const moa_gemm_desc *desc, const void *A, const void *B, const void *R, void *C, void *stream)
{
    if (!desc) return MOA_ERR_INVALID_ARG;
    if (desc->M <= 0 || desc->N <= 0 || desc->K <= 0) return MOA_ERR_INVALID_ARG;
    if ((desc->a_layout != 0 && desc->a_layout != 1) || (desc->b_layout != 0 && desc->b_layout != 1)) return MOA_ERR_INVALID_ARG;
    if (desc->dtype != MOA_BF16 && desc->dtype != MOA_F32) return MOA_ERR_INVALID_ARG;
    if (desc->dtype != MOA_BF16) return MOA_ERR_UNSUPPORTED;
    // row lengths: A [M,K] or [K,M]; B [N,K] or [K,N]; C, R [M,N]
    const int a_cols = desc->a_layout ? desc->M : desc->K, b_cols = desc->b_layout ? desc->N : desc->K;
    if (a_cols % 8 != 0 || b_cols % 8 != 0 || desc->N % 8 != 0) return MOA_ERR_UNSUPPORTED;
    if (!A || !B || !C) return MOA_ERR_INVALID_ARG;
    if (!aligned16(A) || !aligned16(B) || !aligned16(C) || (R && !aligned16(R))) return MOA_ERR_INVALID_ARG;
    moa_status s = check_device_arch();
    if (s != MOA_OK) return s;
    return gemm_bf16(desc->a_layout, desc->b_layout, desc->M, desc->N, desc->K, A, B, R, C, (cudaStream_t)stream) == cudaSuccess
               ? MOA_OK : MOA_ERR_CUDA;
}

namespace {

// the descriptors of the block's calls
struct BlockCalls {
    moa_rmsnorm_desc norm;
    moa_attn_desc attn;
    moa_mlp_desc mlp;
    int T, dm;
    explicit BlockCalls(const moa_block_desc &b) : norm{}, attn{}, mlp{}, T(b.B * b.n), dm(b.H * b.d)
    {
        norm = moa_rmsnorm_desc{T, dm, b.eps, MOA_BF16};
        attn.B = b.B; attn.H = b.H; attn.n = b.n; attn.d = b.d; attn.causal = b.causal; attn.scale = b.scale;
        attn.layout = MOA_LAYOUT_STRIDED;
        const int64_t third[3] = {3LL * dm, b.d, (int64_t)b.n * 3 * dm}, whole[3] = {dm, b.d, (int64_t)b.n * dm};
        for (int i = 0; i < 3; ++i) { attn.q_stride[i] = attn.kv_stride[i] = third[i]; attn.o_stride[i] = whole[i]; }
        mlp = moa_mlp_desc{T, dm, b.d_ff, MOA_BF16};
    }
    moa_gemm_desc gemm(int M, int N, int K, int a_layout, int b_layout) const { return moa_gemm_desc{M, N, K, a_layout, b_layout, MOA_BF16}; }
    // two products that do not depend on each other
    moa_status two(const moa_gemm_desc &g, const void *A, const void *B, void *C, const moa_gemm_desc &h, const void *D, const void *E, void *F,
                   void *stream) const
    {
        for (const void *p : {A, B, (const void *)C, D, E, (const void *)F})
            if (!p || !aligned16(p)) return MOA_ERR_INVALID_ARG;
        if (dm % 8 != 0) return MOA_ERR_UNSUPPORTED;
        const moa_status s = check_device_arch();
        if (s != MOA_OK) return s;
        return gemm_bf16_two(GemmArgs{g.a_layout, g.b_layout, g.M, g.N, g.K, A, B, C}, GemmArgs{h.a_layout, h.b_layout, h.M, h.N, h.K, D, E, F},
                             (cudaStream_t)stream) == cudaSuccess ? MOA_OK : MOA_ERR_CUDA;
    }
    char *third(void *packed, int i) const { return packed ? (char *)packed + (size_t)i * dm * 2 : nullptr; }
};

bool block_desc_ok(const moa_block_desc *b, const moa_block_arrays *r)
{
    // (products of sizes that have to be countable in an int; everything else is checked by the calls)
    return b && r && b->B > 0 && b->n > 0 && b->H > 0 && b->d > 0 && b->d_ff > 0 && (long long)b->B * b->n < (1LL << 31) &&
           3LL * b->H * b->d < (1LL << 31);
}

}  // namespace

#define MOA_STEP(call) do { const moa_status step = (call); if (step != MOA_OK) return step; } while (0)

moa_status moa_block_fwd(const moa_block_desc *desc, const moa_block_arrays *r, void *stream)
{
    if (!block_desc_ok(desc, r)) return MOA_ERR_INVALID_ARG;
    const BlockCalls c(*desc);
    MOA_STEP(moa_rmsnorm_fwd(&c.norm, r->x, r->g1, r->h1, r->r1, stream));
    const moa_gemm_desc proj3 = c.gemm(c.T, 3 * c.dm, c.dm, 0, 0), proj = c.gemm(c.T, c.dm, c.dm, 0, 0);
    MOA_STEP(moa_gemm(&proj3, r->h1, r->Wqkv, nullptr, r->qkv, stream));
    MOA_STEP(moa_attn_fwd(&c.attn, c.third(r->qkv, 0), c.third(r->qkv, 1), c.third(r->qkv, 2), r->o, r->L, nullptr, 0, stream));
    MOA_STEP(moa_gemm(&proj, r->o, r->Wo, r->x, r->x2, stream));
    MOA_STEP(moa_rmsnorm_fwd(&c.norm, r->x2, r->g2, r->h2, r->r2, stream));
    return moa_gated_mlp_fwd(&c.mlp, r->h2, r->W1, r->W3, r->W2, r->x2, r->a, r->u, r->h, r->y, stream);
}

moa_status moa_block_bwd(const moa_block_desc *desc, const moa_block_arrays *r, void *stream)
{
    if (!block_desc_ok(desc, r)) return MOA_ERR_INVALID_ARG;
    const BlockCalls c(*desc);
    MOA_STEP(moa_gated_mlp_bwd(&c.mlp, r->h2, r->W1, r->W3, r->W2, r->a, r->u, r->h, r->dy, r->dh2, r->dW1, r->dW3, r->dW2, r->mlp_ws,
                               r->mlp_ws_bytes, stream));
    MOA_STEP(moa_rmsnorm_bwd(&c.norm, r->x2, r->g2, r->r2, r->dh2, r->dy, r->dx2, r->dg2, r->norm_ws, r->norm_ws_bytes, stream));
    MOA_STEP(c.two(c.gemm(c.dm, c.dm, c.T, 1, 1), r->dx2, r->o, r->dWo, c.gemm(c.T, c.dm, c.dm, 0, 1), r->dx2, r->Wo, r->dout, stream));
    MOA_STEP(moa_attn_bwd(&c.attn, c.third(r->qkv, 0), c.third(r->qkv, 1), c.third(r->qkv, 2), r->o, r->L, r->dout, c.third(r->dqkv, 0),
                          c.third(r->dqkv, 1), c.third(r->dqkv, 2), r->attn_ws, r->attn_ws_bytes, stream));
    MOA_STEP(c.two(c.gemm(c.T, c.dm, 3 * c.dm, 0, 1), r->dqkv, r->Wqkv, r->dh1, c.gemm(3 * c.dm, c.dm, c.T, 1, 1), r->dqkv, r->h1, r->dWqkv, stream));
    return moa_rmsnorm_bwd(&c.norm, r->x, r->g1, r->r1, r->dh1, r->dx2, r->dx, r->dg1, r->norm_ws, r->norm_ws_bytes, stream);
}

}  // extern "C"
