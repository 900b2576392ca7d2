// fp32 SIMT kernels: the MOA_F32 path, and a generic path for any dtype/shape.
//
// Online softmax in the forward; the backward recomputes P from the stored logsumexp,
// one CTA or cluster per key tile (each dK/dV element has exactly one writer), dQ either
// by fp32 atomics or by a separate query-parallel kernel.  The forward and the key-parallel
// backward are register-tiled (below); the two comparison variants (the query-parallel dQ
// pass and the row-parallel single kernel) keep plain tiles of 64 query rows x 64 keys,
// 256 threads as a 16 x 16 grid; thread (ty,tx) owns score rows ty*4..ty*4+3 and score
// columns tx, tx+16, tx+32, tx+48, and the output columns tx+16c.
#include "common.cuh"
#include "ptx.cuh"
#include <math.h>

namespace moa {
namespace {

constexpr int BM = 64;       // query rows per tile
constexpr int BN = 64;       // keys per tile
constexpr int NTHREADS = 256;
constexpr int SLD = BN + 1;  // leading dimension of the 64x64 score tiles in shared memory

template <typename T, int D>
__device__ __forceinline__ void load_tile(float *dst, const T *src, int row0, int n)
{
    constexpr int LD = D + 1;
    for (int idx = threadIdx.x; idx < BM * D; idx += NTHREADS) {
        const int r = idx / D, c = idx % D;
        const int row = row0 + r;
        dst[r * LD + c] = row < n ? to_float<T>(src[(size_t)row * D + c]) : 0.f;
    }
}

__device__ __forceinline__ float group16_max(float v)
{
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float group16_sum(float v)
{
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------- register-tiled kernels: shared pieces
// What bounds the two kernels below is the FMA pipe (fp32 in, fp32 accumulate: no tensor-core form keeps 24 bits), so
// everything is arranged to feed it from as few instructions as possible:
//   * the products run on packed pairs (fma.rn.f32x2: one instruction for two multiply-adds), operands come from shared
//     memory 16 bytes at a time, a thread computes R x 4 or more outputs: 3 loads per 16 packed multiply-adds at R = 8;
//   * a contraction over d reads both operands along their rows and keeps even and odd partial sums in the two halves of
//     a pair; a contraction over keys or queries packs two neighbouring rows of the output, so one operand is a pair as it
//     lies in memory and the other a duplicated scalar;
//   * rows are padded by 16 bytes: the 16 lanes that read 16 rows at one column fall on different banks;
//   * P (and dS) go through shared memory only between the lanes of one warp, and the loads of the next tile are
//     asynchronous and run under the product that does not need their buffer;
//   * a CTA cluster shares one output tile when there are fewer tiles than the chip has room for: the ranks take the tiles
//     of the other axis in turn, and their partial results are added through distributed shared memory, in rank order.
constexpr int SNT = 128;         // threads per CTA: lane tx = tid % 16 along columns, ty = tid / 16 along rows
constexpr int STY = SNT / 16;
constexpr float kLazyMax = 5.f;  // (e^5: far from where fp32 sums of such terms would lose anything)

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool live)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int bytes = live ? 16 : 0;      // 0: zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ROWS x D tile of src (row row0 first, rows past n zero) into padded rows of D + 4 floats.  fp32: asynchronous copies, to
// be committed by the caller; bf16: widened on the way.
template <typename T, int ROWS, int D>
__device__ __forceinline__ void tile_in(float *dst, const T *src, int row0, int n)
{
    constexpr int V = 16 / (int)sizeof(T), PER_ROW = D / V;
#pragma unroll
    for (int it = 0; it < ROWS * PER_ROW / SNT; ++it) {
        const int idx = it * SNT + threadIdx.x, r = idx / PER_ROW, c = (idx % PER_ROW) * V;
        const bool live = row0 + r < n;
        const T *from = src + (size_t)(live ? row0 + r : 0) * D + c;
        float *to = dst + r * (D + 4) + c;
        if (sizeof(T) == 4) {
            cp_async16(to, reinterpret_cast<const float *>(from), live);
        } else {
            uint4 u = make_uint4(0, 0, 0, 0);
            if (live) u = *reinterpret_cast<const uint4 *>(from);
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
            float f[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {      // bf16 -> fp32 is a shift
                f[2 * i] = __uint_as_float(w[i] << 16);
                f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
            }
            *reinterpret_cast<float4 *>(to) = make_float4(f[0], f[1], f[2], f[3]);
            *reinterpret_cast<float4 *>(to + 4) = make_float4(f[4], f[5], f[6], f[7]);
        }
    }
}

// four consecutive outputs of a row
__device__ __forceinline__ void store4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16 *p, float4 v)
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
}
__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p)
{
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xFFFF0000u));
}

template <typename T> __device__ __forceinline__ float4 as_stored(float4 v)
{
    return make_float4(to_float(from_float<T>(v.x)), to_float(from_float<T>(v.y)), to_float(from_float<T>(v.z)),
                       to_float(from_float<T>(v.w)));
}

// kDeep: many steps of the products unrolled, their loads in flight together.  For launches of one tile per CTA and at most a CTA (a warp per
// scheduler) per SM, where the time is that tile's latency: fused B1 H1 n128 d64 12.3 -> 11.2 us, B1 H1 n128 d128 15.3 -> 14.1, B1 H8 n64 d64
// 11.6 -> 10.5.  From two tiles per CTA on it was slower (B1 H2 n300 d64 21.7 -> 27.9).
// out[i][b] = A[a_row0 + i][:] . B[tx + 16 b][:], contraction over D; rows of D + 4 floats
template <int R, int NB, int D, bool kDeep>
__device__ __forceinline__ void dot_rows(float (&out)[R][NB], const float *A, const float *B, int a_row0, int tx)
{
    constexpr int LD = D + 4;
    uint64_t acc[R][NB];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[i][b] = 0ull;
    const float *ap = A + a_row0 * LD, *bp = B + tx * LD;
#pragma unroll (kDeep ? 8 : 2)
    for (int k = 0; k < D; k += 4) {
        ulonglong2 av[R], bv[NB];
#pragma unroll
        for (int i = 0; i < R; ++i) av[i] = *reinterpret_cast<const ulonglong2 *>(ap + i * LD + k);
#pragma unroll
        for (int b = 0; b < NB; ++b) bv[b] = *reinterpret_cast<const ulonglong2 *>(bp + 16 * b * LD + k);
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                acc[i][b] = ptx::fma_f32x2(av[i].x, bv[b].x, acc[i][b]);
                acc[i][b] = ptx::fma_f32x2(av[i].y, bv[b].y, acc[i][b]);
            }
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            float lo, hi;
            ptx::unpack_f32x2(acc[i][b], lo, hi);
            out[i][b] = lo + hi;
        }
}

// acc[i2][c] (rows 2 i2 and 2 i2 + 1 of the thread's R rows, packed) += sum_{j < K} W[j][R rows] X[j][4 tx + 64 v + 0..3];
// W: rows of LW floats, the thread's R rows consecutive at w0; X: rows of D + 4 floats
template <int R, int K, int D, bool kDeep>
__device__ __forceinline__ void add_rows(uint64_t (&acc)[R / 2][D / 16], const float *W, int LW, int w0, const float *X, int tx)
{
    static_assert(R == 2 || R % 4 == 0, "a thread's rows are read 8 or 16 bytes at a time");
    constexpr int LD = D + 4;
    const float *wp = W + w0, *xp = X + 4 * tx;
#pragma unroll (kDeep ? 16 : 4)
    for (int j = 0; j < K; ++j) {
        uint64_t wv[R / 2], xv[D / 16];
        if (R == 2) {
            wv[0] = *reinterpret_cast<const uint64_t *>(wp + j * LW);
        } else {
#pragma unroll
            for (int i = 0; i < R / 4; ++i) {
                const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(wp + j * LW + 4 * i);
                wv[2 * i] = u.x;
                wv[2 * i + 1] = u.y;
            }
        }
#pragma unroll
        for (int v = 0; v < D / 64; ++v) {
            const float4 f = *reinterpret_cast<const float4 *>(xp + j * LD + 64 * v);
            xv[4 * v] = ptx::pack_f32x2(f.x, f.x);
            xv[4 * v + 1] = ptx::pack_f32x2(f.y, f.y);
            xv[4 * v + 2] = ptx::pack_f32x2(f.z, f.z);
            xv[4 * v + 3] = ptx::pack_f32x2(f.w, f.w);
        }
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
#pragma unroll
            for (int c = 0; c < D / 16; ++c) acc[i][c] = ptx::fma_f32x2(wv[i], xv[c], acc[i][c]);
    }
}

// rows 2 i2, 2 i2 + 1 of a packed accumulator -> two float4 of column group v
template <int C>
__device__ __forceinline__ void unpack_rows(const uint64_t (&acc)[C], int v, float4 &even, float4 &odd)
{
    ptx::unpack_f32x2(acc[4 * v], even.x, odd.x);
    ptx::unpack_f32x2(acc[4 * v + 1], even.y, odd.y);
    ptx::unpack_f32x2(acc[4 * v + 2], even.z, odd.z);
    ptx::unpack_f32x2(acc[4 * v + 3], even.w, odd.w);
}

// ------------------------------------------------------------------------- forward
// CTA: BM = 8 R query rows; a warp has 2 R rows to itself, a thread R rows x 4 keys of the score tile and R rows x D / 16
// columns of O.  The `split` ranks of a cluster take the key tiles of their rows in turn (rank r: tiles r, r + split, ...), each
// with its own online softmax; at the end rank r merges rows r BM / split ... of all ranks' partial results.
// In a fused call (dO != nullptr) the merge also gives D = rowsum(dO o O) and clears its rows of dQ.
template <int R, int D>
struct SimtFwd {
    static constexpr int BM = STY * R, LD = D + 4, LP = 2 * R + 4;
    static constexpr int kFloats = (BM + 2 * BN) * LD + 4 * BN * LP;      // Q, K, V, P^T of the four warps
    static constexpr size_t kSmem = kFloats * sizeof(float);
};

template <typename T, int R, int D, bool kDeep>
__global__ void __launch_bounds__(SNT, R == 8 ? 3 : D == 128 ? 2 : 4)
simt_fwd_kernel(const T *__restrict__ Q, const T *__restrict__ K, const T *__restrict__ V, T *__restrict__ O,
                float *__restrict__ L, const T *__restrict__ dO, float *__restrict__ Dv, float *__restrict__ dQzero, int n,
                int causal, float scale, int nqt, int split)
{
    using S = SimtFwd<R, D>;
    constexpr int BM = S::BM, LD = S::LD, LP = S::LP, NC = D / 16;
    extern __shared__ float smem[];
    float *Qs = smem, *Ks = Qs + BM * LD, *Vs = Ks + BN * LD;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16, warp = tid / 32;
    float *Pw = Vs + BN * LD + warp * BN * LP;      // this warp's P^T: [key][2 R rows]
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    Q = ptx::after_wait(Q); K = ptx::after_wait(K); V = ptx::after_wait(V); dO = ptx::after_wait(dO);

    const int rank = split > 1 ? (int)ptx::cluster_ctarank() : 0;
    const int job = (int)blockIdx.x / split;
    int qt = job % nqt;
    const int bh = job / nqt;
    if (causal) qt = nqt - 1 - qt;  // longest rows first
    const int q0 = qt * BM;
    const size_t base = (size_t)bh * n * D;
    Q += base; K += base; V += base; O += base; L += (size_t)bh * n;

    float m[R], l[R];
    uint64_t o[R / 2][NC];
#pragma unroll
    for (int i = 0; i < R; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) o[i][c] = 0ull;
    const int kend = causal ? min(n, q0 + BM) : n;
    const int step = BN * split;
    int k0 = rank * BN;
    if (k0 < kend) {
        tile_in<T, BM, D>(Qs, Q, q0, n);
        tile_in<T, BN, D>(Ks, K, k0, n);
        cp_commit();
        tile_in<T, BN, D>(Vs, V, k0, n);
        cp_commit();
    }
    for (; k0 < kend; k0 += step) {
        const bool more = k0 + step < kend;
        cp_wait<1>();                 // K (and Q) are here; V may still be on its way
        __syncthreads();
        float s[R][4];
        dot_rows<R, 4, D, kDeep>(s, Qs, Ks, ty * R, tx);
        __syncthreads();
        if (more) tile_in<T, BN, D>(Ks, K, k0 + step, n);      // runs under the softmax and the P V product
        cp_commit();
        const bool mask = k0 + BN > n || (causal && k0 + BN - 1 > q0);
        // A row's reference is raised only when a score exceeds it by more than kLazyMax, so that most tiles pass without the
        // exchange of maxima between lanes and the rescaling of O; row sums stay per lane until the end.
        float mx[R];
        bool grow = false;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int row = q0 + ty * R + i;
            mx[i] = -INFINITY;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                float v = s[i][b] * scale;
                if (mask) {
                    const int col = k0 + tx + 16 * b;
                    if (col >= n || (causal && col > row)) v = -INFINITY;
                }
                s[i][b] = v;
                mx[i] = fmaxf(mx[i], v);
            }
            grow |= mx[i] > m[i] + kLazyMax;
        }
        if (__any_sync(0xffffffffu, grow)) {
            uint64_t al[R / 2];
#pragma unroll
            for (int i = 0; i < R; i += 2) {
                float alpha[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float mn = fmaxf(m[i + e], group16_max(mx[i + e]));
                    alpha[e] = expf(m[i + e] - (mn == -INFINITY ? 0.f : mn));
                    l[i + e] *= alpha[e];
                    m[i + e] = mn;
                }
                al[i / 2] = ptx::pack_f32x2(alpha[0], alpha[1]);
            }
#pragma unroll
            for (int i = 0; i < R / 2; ++i)
#pragma unroll
                for (int c = 0; c < NC; ++c) o[i][c] = ptx::mul_f32x2(o[i][c], al[i]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float ref = m[i] == -INFINITY ? 0.f : m[i];      // (-inf: no key visible so far)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[i][b] = expf(s[i][b] - ref);
                l[i] += s[i][b];
            }
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            float *dst = Pw + (tx + 16 * b) * LP + (ty % 2) * R;
            if (R == 2) {
                *reinterpret_cast<float2 *>(dst) = make_float2(s[0][b], s[R - 1][b]);
            } else {
#pragma unroll
                for (int i = 0; i + 3 < R; i += 4)
                    *reinterpret_cast<float4 *>(dst + i) = make_float4(s[i][b], s[i + 1][b], s[i + 2][b], s[i + 3][b]);
            }
        }
        cp_wait<1>();                 // V is here; the next K may still be on its way
        __syncthreads();              // (also: every lane's part of P^T is written)
        add_rows<R, BN, D, kDeep>(o, Pw, LP, (ty % 2) * R, Vs, tx);
        __syncthreads();
        if (more) tile_in<T, BN, D>(Vs, V, k0 + step, n);
        cp_commit();
    }
    cp_wait<0>();
    __syncthreads();
    // partial results into shared memory: O [BM][LD] over Q, then m, l
    float *Om = smem, *Mm = Ks, *Lm = Ks + BM;
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int v = 0; v < D / 64; ++v) {
            float4 e, od;
            unpack_rows<NC>(o[i], v, e, od);
            *reinterpret_cast<float4 *>(Om + (ty * R + 2 * i) * LD + 64 * v + 4 * tx) = e;
            *reinterpret_cast<float4 *>(Om + (ty * R + 2 * i + 1) * LD + 64 * v + 4 * tx) = od;
        }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const float li = group16_sum(l[i]);
        if (tx == 0) { Mm[ty * R + i] = m[i]; Lm[ty * R + i] = li; }
    }
    if (split > 1) ptx::cluster_sync_all();
    else __syncthreads();
    constexpr int LPR = D / 4;         // lanes per row, 16 bytes each
    const int per = (BM + split - 1) / split;        // rows this rank finishes (the last rank: what is left)
    for (int r = tid / LPR; r < per && rank * per + r < BM; r += SNT / LPR) {
        const int rr = rank * per + r, row = q0 + rr, c = (tid % LPR) * 4;
        float mt = -INFINITY, mk[ptx::kMaxRanks], lk[ptx::kMaxRanks];
        float4 vk[ptx::kMaxRanks];
#pragma unroll
        for (int k = 0; k < ptx::kMaxRanks; ++k) {
            mk[k] = ptx::peer_f1(ptx::smem_u32(Mm + rr), k, split, -INFINITY);
            lk[k] = ptx::peer_f1(ptx::smem_u32(Lm + rr), k, split, 0.f);
            vk[k] = ptx::peer_f4(ptx::smem_u32(Om + rr * LD + c), k, split);
        }
#pragma unroll
        for (int k = 0; k < ptx::kMaxRanks; ++k) mt = fmaxf(mt, mk[k]);
        const float ref = mt == -INFINITY ? 0.f : mt;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        float lt = 0.f;
#pragma unroll
        for (int k = 0; k < ptx::kMaxRanks; ++k) {      // (a rank that does not exist has weight 0)
            const float w = expf(mk[k] - ref);
            const float4 v = vk[k];
            lt = fmaf(lk[k], w, lt);
            a.x = fmaf(v.x, w, a.x); a.y = fmaf(v.y, w, a.y); a.z = fmaf(v.z, w, a.z); a.w = fmaf(v.w, w, a.w);
        }
        const bool live = row < n;
        const float inv = 1.f / lt;
        a.x *= inv; a.y *= inv; a.z *= inv; a.w *= inv;
        const size_t at = (size_t)row * D + c;
        if (live) {
            store4(O + at, a);
            if (c == 0) L[row] = mt + logf(lt);
        }
        if (dO != nullptr) {
            float dot = 0.f;
            if (live) {
                // (from O as stored, like the separate backward call: the same gradients either way, bit for bit)
                const float4 g = load4(dO + base + at), r = as_stored<T>(a);
                dot = fmaf(g.x, r.x, fmaf(g.y, r.y, fmaf(g.z, r.z, g.w * r.w)));
                if (dQzero) store4(dQzero + base + at, make_float4(0.f, 0.f, 0.f, 0.f));
            }
            // the lanes of a row, 16 (D = 64) or 32 consecutive ones, go through this loop together
            const uint32_t who = D == 64 ? 0xFFFFu << (tid & 16) : 0xFFFFFFFFu;
#pragma unroll
            for (int d = LPR / 2; d >= 1; d >>= 1) dot += __shfl_xor_sync(who, dot, d);
            if (live && c == 0) Dv[(size_t)bh * n + row] = dot;
        }
    }
    if (split > 1) ptx::cluster_sync_all();      // nobody leaves while another rank may still read its shared memory
}

// ---------------------------------------- rowsum(dO o O), and dQ (or its accumulator) cleared: one warp per row
template <typename T>
__global__ void row_dot_kernel(const T *__restrict__ dO, const T *__restrict__ O,
                               float *__restrict__ Dv, float *__restrict__ dQzero, size_t rows, int d)
{
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    dO = ptx::after_wait(dO); O = ptx::after_wait(O);
    const size_t row = (size_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    if (row >= rows) return;
    const int lane = threadIdx.x % 32;
    float acc = 0.f;
    for (int c = 4 * lane; c < d; c += 128) {
        const float4 a = load4(dO + row * d + c), b = load4(O + row * d + c);
        acc = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc))));
        if (dQzero) store4(dQzero + row * d + c, make_float4(0.f, 0.f, 0.f, 0.f));
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) Dv[row] = acc;
}

// --------------------------------------------- shared by the two backward kernels
// scores and dP of a 64x64 tile -> P and scale*dS in shared memory
template <int D>
__device__ __forceinline__ void bwd_tile_p_ds(const float *Qs, const float *dOs, const float *Ks,
                                              const float *Vs, const float *Ls, const float *Ds,
                                              float *Ps, float *dSs, int q0, int k0, int n,
                                              int causal, float scale, int tx, int ty)
{
    constexpr int LD = D + 1;
    float s[4][4], dp[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) { s[a][b] = 0.f; dp[a][b] = 0.f; }
#pragma unroll 2
    for (int k = 0; k < D; ++k) {
        float qv[4], gv[4], kv[4], vv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) { qv[a] = Qs[(ty * 4 + a) * LD + k]; gv[a] = dOs[(ty * 4 + a) * LD + k]; }
#pragma unroll
        for (int b = 0; b < 4; ++b) { kv[b] = Ks[(tx + 16 * b) * LD + k]; vv[b] = Vs[(tx + 16 * b) * LD + k]; }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                s[a][b] = fmaf(qv[a], kv[b], s[a][b]);
                dp[a][b] = fmaf(gv[a], vv[b], dp[a][b]);
            }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int r = ty * 4 + a, row = q0 + r;
        const float Li = Ls[r], Di = Ds[r];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int cidx = tx + 16 * b, col = k0 + cidx;
            const bool live = row < n && col < n && !(causal && col > row);
            const float pv = live ? expf(s[a][b] * scale - Li) : 0.f;
            Ps[r * SLD + cidx] = pv;
            if (dSs) dSs[r * SLD + cidx] = pv * (dp[a][b] - Di) * scale;
        }
    }
}

__device__ __forceinline__ void load_rowvec(float *dst, const float *src, int row0, int n)
{
    for (int r = threadIdx.x; r < BM; r += NTHREADS) dst[r] = (row0 + r) < n ? src[row0 + r] : 0.f;
}

// ----------------------------------------- backward, one CTA (or cluster) per key tile: dK, dV (+dQ red)
// CTA: BN = 8 R keys against query tiles of BM rows; a warp has 2 R keys to itself, a thread R keys x BM / 16 queries of the
// score tile, R keys x D / 16 columns of dK and dV, and BM / 8 queries x D / 16 columns of the dQ tile.  P, then dS in its
// place, is exchanged inside a warp ([query][key], the warp's own keys); dQ needs the dS of all warps, so a transposed copy
// ([key][query]) goes through a CTA barrier, behind which the next Q and dO tiles are requested: they arrive under the dQ
// product.  The `split` ranks of a cluster take the query tiles of their keys in turn and add their dK, dV at the end.
template <int R, int D>
struct SimtBwd {
    static constexpr int BN = STY * R, BM = D == 64 ? 64 : 32, LD = D + 4;
    static constexpr int LPS = BN + 4, LST = BM + 4;      // rows of P / dS [query][key] and of dS^T [key][query]
    static constexpr int kFloats = 2 * (BN + BM) * LD + BM * LPS + BN * LST + 2 * BM;
    static constexpr size_t kSmem = kFloats * sizeof(float);
    static_assert(BN <= BM, "the partial dK, dV are staged over Q, dO");
};

template <typename T, int R, int D, bool kDeep>
__global__ void __launch_bounds__(SNT, 2)
simt_bwd_kv_kernel(const T *__restrict__ Q, const T *__restrict__ K, const T *__restrict__ V,
                   const T *__restrict__ dO, const float *__restrict__ L, const float *__restrict__ Dv,
                   T *__restrict__ dK, T *__restrict__ dV, float *__restrict__ dQacc,
                   int n, int causal, float scale, int nkt, int split)
{
    using S = SimtBwd<R, D>;
    constexpr int BN = S::BN, BM = S::BM, LD = S::LD, LPS = S::LPS, LST = S::LST, NC = D / 16, QB = BM / 16, RQ = BM / STY;
    extern __shared__ float smem[];
    float *Ks = smem, *Vs = Ks + BN * LD, *Qs = Vs + BN * LD, *dOs = Qs + BM * LD;
    float *Ps = dOs + BM * LD, *dSt = Ps + BM * LPS, *Ls = dSt + BN * LST, *Ds = Ls + BM;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;

    const int rank = split > 1 ? (int)ptx::cluster_ctarank() : 0;
    const int job = (int)blockIdx.x / split;
    const int kt = job % nkt;   // causal: key tile 0 has the most work and comes first
    const int bh = job / nkt;
    const int k0 = kt * BN;
    const size_t base = (size_t)bh * n * D;
    Q += base; K += base; V += base; dO += base; dV += base;
    if (dK) dK += base;
    L += (size_t)bh * n; Dv += (size_t)bh * n;
    if (dQacc) dQacc += base;

    uint64_t dk[R / 2][NC], dv[R / 2][NC];
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) { dk[i][c] = 0ull; dv[i][c] = 0ull; }

    const int step = BM * split;
    int q0 = (causal ? k0 / BM * BM : 0) + rank * BM;
    if (q0 < n) {
        tile_in<T, BN, D>(Ks, K, k0, n);
        tile_in<T, BN, D>(Vs, V, k0, n);
        tile_in<T, BM, D>(Qs, Q, q0, n);
        tile_in<T, BM, D>(dOs, dO, q0, n);
        cp_commit();
    }
    // (the tiles above are the call's inputs; L, D and the cleared dQ come from the kernel in front)
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    L = ptx::after_wait(L); Dv = ptx::after_wait(Dv);
    for (; q0 < n; q0 += step) {
        if (tid < BM) {
            const bool live = q0 + tid < n;
            Ls[tid] = live ? L[q0 + tid] : 0.f;
            Ds[tid] = live ? Dv[q0 + tid] : 0.f;
        }
        cp_wait<0>();
        __syncthreads();
        const bool mask = k0 + BN > n || q0 + BM > n || (causal && k0 + BN - 1 > q0);
        float p[R][QB];
        dot_rows<R, QB, D, kDeep>(p, Ks, Qs, ty * R, tx);
#pragma unroll
        for (int b = 0; b < QB; ++b) {
            const int q = tx + 16 * b, row = q0 + q;
            const float Li = Ls[q];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                p[i][b] = expf(p[i][b] * scale - Li);
                if (mask) {
                    const int col = k0 + ty * R + i;
                    if (row >= n || col >= n || (causal && col > row)) p[i][b] = 0.f;
                }
            }
        }
        auto put_rows = [&](const float (&v)[R][QB]) {      // [query][key]: this thread's R keys of each of its queries
#pragma unroll
            for (int b = 0; b < QB; ++b) {
                float *dst = Ps + (tx + 16 * b) * LPS + ty * R;
                if (R == 2) {
                    *reinterpret_cast<float2 *>(dst) = make_float2(v[0][b], v[R - 1][b]);
                } else {
#pragma unroll
                    for (int i = 0; i + 3 < R; i += 4)
                        *reinterpret_cast<float4 *>(dst + i) = make_float4(v[i][b], v[i + 1][b], v[i + 2][b], v[i + 3][b]);
                }
            }
            __syncwarp();
        };
        put_rows(p);
        add_rows<R, BM, D, kDeep>(dv, Ps, LPS, ty * R, dOs, tx);
        if (dK != nullptr || dQacc != nullptr) {
            float ds[R][QB];
            dot_rows<R, QB, D, kDeep>(ds, Vs, dOs, ty * R, tx);
#pragma unroll
            for (int b = 0; b < QB; ++b) {
                const int q = tx + 16 * b;
                const float Di = Ds[q];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    ds[i][b] = p[i][b] * (ds[i][b] - Di) * scale;
                    dSt[(ty * R + i) * LST + q] = ds[i][b];
                }
            }
            __syncwarp();              // the warp's lanes have read P
            put_rows(ds);
            add_rows<R, BM, D, kDeep>(dk, Ps, LPS, ty * R, Qs, tx);
        }
        __syncthreads();
        if (q0 + step < n) {           // arrives under the dQ product
            tile_in<T, BM, D>(Qs, Q, q0 + step, n);
            tile_in<T, BM, D>(dOs, dO, q0 + step, n);
            cp_commit();
        }
        if (dQacc != nullptr) {
            uint64_t dq[RQ / 2][NC];
#pragma unroll
            for (int i = 0; i < RQ / 2; ++i)
#pragma unroll
                for (int c = 0; c < NC; ++c) dq[i][c] = 0ull;
            add_rows<RQ, BN, D, kDeep>(dq, dSt, LST, ty * RQ, Ks, tx);
#pragma unroll
            for (int i = 0; i < RQ / 2; ++i)
#pragma unroll
                for (int v = 0; v < D / 64; ++v) {
                    float4 r[2];
                    unpack_rows<NC>(dq[i], v, r[0], r[1]);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int row = q0 + ty * RQ + 2 * i + e;
                        if (row < n)       // 16 lanes cover 256 consecutive bytes of the row
                            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dQacc + (size_t)row * D + 64 * v + 4 * tx),
                                         "f"(r[e].x), "f"(r[e].y), "f"(r[e].z), "f"(r[e].w) : "memory");
                    }
                }
        }
    }
    if (split == 1) {
#pragma unroll
        for (int i = 0; i < R / 2; ++i)
#pragma unroll
            for (int v = 0; v < D / 64; ++v) {
                float4 a[2], g[2];
                unpack_rows<NC>(dk[i], v, a[0], a[1]);
                unpack_rows<NC>(dv[i], v, g[0], g[1]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int row = k0 + ty * R + 2 * i + e;
                    if (row >= n) continue;
                    const size_t at = (size_t)row * D + 64 * v + 4 * tx;
                    if (dK) store4(dK + at, a[e]);   // nullptr: dV only
                    store4(dV + at, g[e]);
                }
            }
        return;
    }
    // partial dK over Q, dV over dO (all tiles are done with them: the barrier in front of the last dQ product)
    __syncthreads();
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int v = 0; v < D / 64; ++v) {
            float4 a[2], g[2];
            unpack_rows<NC>(dk[i], v, a[0], a[1]);
            unpack_rows<NC>(dv[i], v, g[0], g[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int at = (ty * R + 2 * i + e) * LD + 64 * v + 4 * tx;
                *reinterpret_cast<float4 *>(Qs + at) = a[e];
                *reinterpret_cast<float4 *>(dOs + at) = g[e];
            }
        }
    ptx::cluster_sync_all();
    constexpr int LPR = D / 4;
    const int per = (BN + split - 1) / split;
    for (int r = tid / LPR; r < per && rank * per + r < BN; r += SNT / LPR) {
        const int rr = rank * per + r, row = k0 + rr, c = (tid % LPR) * 4;
        if (row >= n) continue;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), g = a;
        const uint32_t at_k = ptx::smem_u32(Qs + rr * LD + c), at_v = ptx::smem_u32(dOs + rr * LD + c);
#pragma unroll 1
        for (int k0 = 0; k0 < split; k0 += 4) {
            float4 x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { x[u] = ptx::peer_f4(at_k, k0 + u, split); y[u] = ptx::peer_f4(at_v, k0 + u, split); }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a.x += x[u].x; a.y += x[u].y; a.z += x[u].z; a.w += x[u].w;
                g.x += y[u].x; g.y += y[u].y; g.z += y[u].z; g.w += y[u].w;
            }
        }
        if (dK) store4(dK + (size_t)row * D + c, a);
        store4(dV + (size_t)row * D + c, g);
    }
    ptx::cluster_sync_all();
}

// ----------------------------------------- backward, one CTA per query tile: dQ, no atomics
template <typename T, int D>
__global__ void __launch_bounds__(NTHREADS)
simt_bwd_dq_kernel(const T *__restrict__ Q, const T *__restrict__ K, const T *__restrict__ V,
                   const T *__restrict__ dO, const float *__restrict__ L, const float *__restrict__ Dv,
                   T *__restrict__ dQ, int n, int causal, float scale, int nqt)
{
    constexpr int LD = D + 1;
    constexpr int NC = D / 16;
    extern __shared__ float smem[];
    float *Ks = smem, *Vs = Ks + BN * LD, *Qs = Vs + BN * LD, *dOs = Qs + BM * LD;
    float *Ps = dOs + BM * LD, *dSs = Ps + BM * SLD, *Ls = dSs + BM * SLD, *Ds = Ls + BM;

    int qt = blockIdx.x % nqt;
    const int bh = blockIdx.x / nqt;
    if (causal) qt = nqt - 1 - qt;
    const int q0 = qt * BM;
    const size_t base = (size_t)bh * n * D;
    Q += base; K += base; V += base; dO += base; dQ += base;
    L += (size_t)bh * n; Dv += (size_t)bh * n;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;

    load_tile<T, D>(Qs, Q, q0, n);
    load_tile<T, D>(dOs, dO, q0, n);
    load_rowvec(Ls, L, q0, n);
    load_rowvec(Ds, Dv, q0, n);
    float dq[4][NC];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) dq[a][c] = 0.f;
    const int kend = causal ? min(n, q0 + BM) : n;
    for (int k0 = 0; k0 < kend; k0 += BN) {
        __syncthreads();
        load_tile<T, D>(Ks, K, k0, n);
        load_tile<T, D>(Vs, V, k0, n);
        __syncthreads();
        bwd_tile_p_ds<D>(Qs, dOs, Ks, Vs, Ls, Ds, Ps, dSs, q0, k0, n, causal, scale, tx, ty);
        __syncthreads();
#pragma unroll 2
        for (int j = 0; j < BN; ++j) {
            float gv[4], kk[NC];
#pragma unroll
            for (int a = 0; a < 4; ++a) gv[a] = dSs[(ty * 4 + a) * SLD + j];
#pragma unroll
            for (int c = 0; c < NC; ++c) kk[c] = Ks[j * LD + tx + 16 * c];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) dq[a][c] = fmaf(gv[a], kk[c], dq[a][c]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int row = q0 + ty * 4 + a;
        if (row >= n) continue;
#pragma unroll
        for (int c = 0; c < NC; ++c) dQ[(size_t)row * D + tx + 16 * c] = from_float<T>(dq[a][c]);
    }
}

// ------------------ row-parallel fused forward+backward in one kernel, dK/dV by atomics
// The paper's own fused design (Sec. 4, its first GPU version): one kernel, parallel over query
// rows.  A CTA runs the forward of its 64 query rows (online softmax; O, L), takes D = rowsum(dO o O)
// from the O it holds, and runs the backward of the same rows straight away: every row statistic it
// needs is its own, so no other CTA is waited for.  dQ stays local; the dV and dK contributions of
// every (query tile, key tile) pair are added into global fp32 accumulators with atomics -- the
// paper's GV and GK atomic sites.  kSites = 2: both sites (the paper's v1).  kSites = 1: only dK;
// dV then comes from an atomic-free key-parallel kernel of its own, as in the paper's v3.
template <typename T, int D, int kSites>
__global__ void __launch_bounds__(NTHREADS)
simt_rowpar_kernel(const T *__restrict__ Q, const T *__restrict__ K, const T *__restrict__ V,
                   const T *__restrict__ dO, T *__restrict__ O, float *__restrict__ L, float *__restrict__ Dv,
                   T *__restrict__ dQ, float *__restrict__ dKacc, float *__restrict__ dVacc,
                   int n, int causal, float scale, int nqt)
{
    constexpr int LD = D + 1;
    constexpr int NC = D / 16;
    extern __shared__ float smem[];
    float *Ks = smem, *Vs = Ks + BN * LD, *Qs = Vs + BN * LD, *dOs = Qs + BM * LD;
    float *Ps = dOs + BM * LD, *dSs = Ps + BM * SLD, *Ls = dSs + BM * SLD, *Ds = Ls + BM;

    int qt = blockIdx.x % nqt;
    const int bh = blockIdx.x / nqt;
    if (causal) qt = nqt - 1 - qt;  // longest rows first
    const int q0 = qt * BM;
    const size_t base = (size_t)bh * n * D;
    Q += base; K += base; V += base; dO += base; O += base; dQ += base; dKacc += base;
    if (kSites == 2) dVacc += base;
    L += (size_t)bh * n; Dv += (size_t)bh * n;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    load_tile<T, D>(Qs, Q, q0, n);
    load_tile<T, D>(dOs, dO, q0, n);
    const int kend = causal ? min(n, q0 + BM) : n;

    // ---- forward of these rows (as simt_fwd_kernel; the P tile goes through Ps)
    {
        float m[4], l[4], o[4][NC];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            m[a] = -INFINITY; l[a] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) o[a][c] = 0.f;
        }
        for (int k0 = 0; k0 < kend; k0 += BN) {
            __syncthreads();
            load_tile<T, D>(Ks, K, k0, n);
            load_tile<T, D>(Vs, V, k0, n);
            __syncthreads();
            float s[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) s[a][b] = 0.f;
#pragma unroll 4
            for (int k = 0; k < D; ++k) {
                float qv[4], kv[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) qv[a] = Qs[(ty * 4 + a) * LD + k];
#pragma unroll
                for (int b = 0; b < 4; ++b) kv[b] = Ks[(tx + 16 * b) * LD + k];
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) s[a][b] = fmaf(qv[a], kv[b], s[a][b]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const int row = q0 + ty * 4 + a;
                float mx = -INFINITY;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int col = k0 + tx + 16 * b;
                    float v = s[a][b] * scale;
                    if (col >= n || (causal && col > row)) v = -INFINITY;
                    s[a][b] = v;
                    mx = fmaxf(mx, v);
                }
                mx = group16_max(mx);
                float mn = fmaxf(m[a], mx);
                if (mn == -INFINITY) mn = 0.f;  // whole row masked so far (padding rows only)
                const float alpha = expf(m[a] - mn);
                float sum = 0.f;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float pv = expf(s[a][b] - mn);
                    sum += pv;
                    Ps[(ty * 4 + a) * SLD + tx + 16 * b] = pv;
                }
                sum = group16_sum(sum);
                l[a] = l[a] * alpha + sum;
                m[a] = mn;
#pragma unroll
                for (int c = 0; c < NC; ++c) o[a][c] *= alpha;
            }
            __syncthreads();
#pragma unroll 4
            for (int j = 0; j < BN; ++j) {
                float pv[4], vv[NC];
#pragma unroll
                for (int a = 0; a < 4; ++a) pv[a] = Ps[(ty * 4 + a) * SLD + j];
#pragma unroll
                for (int c = 0; c < NC; ++c) vv[c] = Vs[j * LD + tx + 16 * c];
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int c = 0; c < NC; ++c) o[a][c] = fmaf(pv[a], vv[c], o[a][c]);
            }
        }
        // O, L, and D = rowsum(dO o O) from the fp32 O held here (the paper's precompute pass)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int r = ty * 4 + a, row = q0 + r;
            const float inv = row < n ? 1.f / l[a] : 0.f;
            float dsum = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float ov = o[a][c] * inv;
                dsum = fmaf(ov, dOs[r * LD + tx + 16 * c], dsum);
                if (row < n) O[(size_t)row * D + tx + 16 * c] = from_float<T>(ov);
            }
            dsum = group16_sum(dsum);
            if (tx == 0) {
                const float lse = row < n ? m[a] + logf(l[a]) : 0.f;
                Ls[r] = lse;
                Ds[r] = row < n ? dsum : 0.f;
                if (row < n) { L[row] = lse; Dv[row] = dsum; }
            }
        }
    }

    // ---- backward of the same rows
    float dq[4][NC];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) dq[a][c] = 0.f;
    for (int k0 = 0; k0 < kend; k0 += BN) {
        __syncthreads();
        load_tile<T, D>(Ks, K, k0, n);
        load_tile<T, D>(Vs, V, k0, n);
        __syncthreads();
        bwd_tile_p_ds<D>(Qs, dOs, Ks, Vs, Ls, Ds, Ps, dSs, q0, k0, n, causal, scale, tx, ty);
        __syncthreads();
#pragma unroll 2
        for (int j = 0; j < BN; ++j) {
            float gv[4], kk[NC];
#pragma unroll
            for (int a = 0; a < 4; ++a) gv[a] = dSs[(ty * 4 + a) * SLD + j];
#pragma unroll
            for (int c = 0; c < NC; ++c) kk[c] = Ks[j * LD + tx + 16 * c];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) dq[a][c] = fmaf(gv[a], kk[c], dq[a][c]);
        }
        // this tile pair's dK (and dV) contribution: [keys][d], thread (ty,tx) owns keys ty*4+a
        float dk[4][NC], dv[4][NC];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < NC; ++c) { dk[a][c] = 0.f; dv[a][c] = 0.f; }
#pragma unroll 2
        for (int q = 0; q < BM; ++q) {
            float pv[4], gv[4], gq[NC], qq[NC];
#pragma unroll
            for (int a = 0; a < 4; ++a) { pv[a] = Ps[q * SLD + ty * 4 + a]; gv[a] = dSs[q * SLD + ty * 4 + a]; }
#pragma unroll
            for (int c = 0; c < NC; ++c) { gq[c] = dOs[q * LD + tx + 16 * c]; qq[c] = Qs[q * LD + tx + 16 * c]; }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (kSites == 2) dv[a][c] = fmaf(pv[a], gq[c], dv[a][c]);
                    dk[a][c] = fmaf(gv[a], qq[c], dk[a][c]);
                }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int row = k0 + ty * 4 + a;
            if (row >= n) continue;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                atomicAdd(&dKacc[(size_t)row * D + tx + 16 * c], dk[a][c]);                     // atomic site GK
                if (kSites == 2) atomicAdd(&dVacc[(size_t)row * D + tx + 16 * c], dv[a][c]);    // atomic site GV
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int row = q0 + ty * 4 + a;
        if (row >= n) continue;
#pragma unroll
        for (int c = 0; c < NC; ++c) dQ[(size_t)row * D + tx + 16 * c] = from_float<T>(dq[a][c]);
    }
}

// HBM-bound (4 bytes read, 2 written per element): grid-stride over float4 groups, four
// independent loads in flight per thread, streaming loads (the accumulator is not read again).
__global__ void __launch_bounds__(256)
convert_kernel(const float *__restrict__ src, __nv_bfloat16 *__restrict__ dst, size_t count, float mul)
{
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    src = ptx::after_wait(src);
    const size_t quads = count / 4;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    auto put = [&](size_t at, const float4 v) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x * mul, v.y * mul), b = __floats2bfloat162_rn(v.z * mul, v.w * mul);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t *>(&a);
        u.y = *reinterpret_cast<uint32_t *>(&b);
        *reinterpret_cast<uint2 *>(dst + 4 * at) = u;
    };
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
    for (; q + 3 * stride < quads; q += 4 * stride) {
        const float4 v0 = __ldcs(s4 + q), v1 = __ldcs(s4 + q + stride), v2 = __ldcs(s4 + q + 2 * stride),
                     v3 = __ldcs(s4 + q + 3 * stride);
        put(q, v0); put(q + stride, v1); put(q + 2 * stride, v2); put(q + 3 * stride, v3);
    }
    for (; q < quads; q += stride) put(q, __ldcs(s4 + q));
    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (size_t i = quads * 4; i < count; ++i) dst[i] = __float2bfloat16_rn(src[i] * mul);
}

// The same conversion row by row, for an accumulator [B*H, n, src_ld] whose rows are wider than d
// and / or a [B,n,H,d] destination; one thread converts four consecutive elements of a row.
__global__ void __launch_bounds__(256)
convert_rows_kernel(const float *__restrict__ src, int src_ld, __nv_bfloat16 *__restrict__ dst, size_t rows, int n, int H,
                    int d, Strides ds, float mul)
{
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    src = ptx::after_wait(src);
    const int quads_per_row = d / 4;
    const size_t total = rows * (size_t)quads_per_row;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += stride) {
        const size_t row = q / quads_per_row;             // flat (b*H + h)*n + r
        const int c4 = (int)(q - row * quads_per_row);
        const size_t bh = row / (size_t)n;
        const size_t r = row - bh * (size_t)n, bb = bh / (size_t)H, h = bh - bb * (size_t)H;
        const size_t doff = ds.at((long long)bb, (long long)h, (long long)r);
        const float4 v = __ldcs(reinterpret_cast<const float4 *>(src + row * (size_t)src_ld) + c4);
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x * mul, v.y * mul), b = __floats2bfloat162_rn(v.z * mul, v.w * mul);
        uint2 u;
        u.x = *reinterpret_cast<uint32_t *>(&a);
        u.y = *reinterpret_cast<uint32_t *>(&b);
        *reinterpret_cast<uint2 *>(dst + doff + 4 * c4) = u;
    }
}

constexpr size_t bwd_smem(int D) { return (size_t)(4 * BM * (D + 1) + 2 * BM * SLD + 2 * BM) * sizeof(float); }

// How many ranks share an output tile; set-up and merge are small beside these kernels' tiles.
// Equal tiles (no causal mask): one CTA alone brings an SM to 82 % of what any number of them reach, so k CTAs on an SM take 0.82 k times
// as long as one, together or in turn, and the time is that of the fullest SM.  Any number of ranks up to 8: B2 H1 n2048 d64's 64 tiles
// take 156, 82, 94, 70, 85, 75, 82, 76 us with 1 ... 8 ranks (estimate 32, 16.5, 18.9, 13.9, 18.5, 16, 18.5, 14.8 tiles).
// Causal: the longest job against the packing of all of them (bwd_split for `per_sm` CTAs on an SM; B2 H2 n1817 d128: 207, 146, 126, 152
// us with 1, 2, 4, 8).
int simt_split(long long jobs, int own_tiles, int others, int own_rows, int other_rows, bool causal, int per_sm)
{
    if (causal) {
        // the tiles of the other axis that tile t meets, summed over t (both axes are cut from the same n rows)
        long long total = 0;
        for (int t = 0; t < own_tiles; ++t) {
            const long long c = ((long long)(t + 1) * own_rows + other_rows - 1) / other_rows;
            total += c < others ? c : others;
        }
        return bwd_split(jobs, others, jobs / own_tiles * total, true, 0.2, 0.1, per_sm);
    }
    const long long sms = device_info().sms;
    int best = 1;
    double best_cost = 0;
    for (int s = 1; s <= 8 && s <= others; ++s) {
        const long long k = (jobs * s + sms - 1) / sms;
        const double cost = ((others + s - 1) / s + (s > 1 ? 0.5 : 0.3)) * (k > 1 ? 0.82 * k : 1.0);
        if (s == 1 || cost < 0.95 * best_cost) { best = s; best_cost = cost; }
    }
    return best;
}

// Rows per thread: the widest tile (fewest shared-memory loads per multiply-add) whose tiles, shared by clusters as far as
// that goes, still give most SMs a CTA; narrower tiles below that, where the time is one CTA's latency.
template <typename T, int R, int D>
cudaError_t fwd_r(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const SimtPrep &pr,
                  cudaStream_t st)
{
    using S = SimtFwd<R, D>;
    const int nqt = (p.n + S::BM - 1) / S::BM, nkt = (p.n + BN - 1) / BN;
    const long long tiles = (long long)nqt * p.BH();
    if (R > 2 && tiles * (nkt < 8 ? nkt : 8) < device_info().sms)
        return fwd_r<T, (R > 2 ? R / 2 : 2), D>(p, Q, K, V, O, L, pr, st);
    const int split = simt_split(tiles, nqt, nkt, S::BM, BN, p.causal, R == 8 ? 3 : D == 128 ? 2 : 4);
    // Not a programmatic dependent where an SM gets more than one CTA: those placed while the kernel in front drains pile up on
    // the SMs it leaves first (B2 H1 n2048 d64: 252 us per fused call against 219).
    const bool alone = tiles * split <= device_info().sms;
    auto go = [&](auto kernel, cudaError_t e) {
        if (e != cudaSuccess) return e;
        LaunchScope scope(MOA_KERNEL_FWD, st);
        return launch_cluster_as(alone, kernel, (unsigned)split, dim3((unsigned)(tiles * split)), dim3(SNT), S::kSmem, st, (const T *)Q, (const T *)K,
                                 (const T *)V, (T *)O, L, (const T *)pr.dO, pr.Dv, pr.dQzero, p.n, p.causal, p.scale, nqt, split);
    };
    if constexpr (R == 2)
        if (alone && split >= nkt) return go(simt_fwd_kernel<T, R, D, true>, allow_smem<simt_fwd_kernel<T, R, D, true>>(S::kSmem));
    return go(simt_fwd_kernel<T, R, D, false>, allow_smem<simt_fwd_kernel<T, R, D, false>>(S::kSmem));
}
template <typename T, int D>
cudaError_t fwd_t(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const SimtPrep &pr,
                  cudaStream_t st)
{
    return fwd_r<T, D == 64 ? 8 : 4, D>(p, Q, K, V, O, L, pr, st);
}

template <typename T, int R, int D>
cudaError_t bwd_kv_r(const Problem &p, const void *Q, const void *K, const void *V, const void *dO, const float *L,
                     const float *Dv, void *dK, void *dV, float *dQacc, cudaStream_t st)
{
    using S = SimtBwd<R, D>;
    const int nkt = (p.n + S::BN - 1) / S::BN, nqt = (p.n + S::BM - 1) / S::BM;
    const long long tiles = (long long)nkt * p.BH();
    if (R > 2 && tiles * (nqt < 8 ? nqt : 8) < device_info().sms)
        return bwd_kv_r<T, (R > 2 ? R / 2 : 2), D>(p, Q, K, V, dO, L, Dv, dK, dV, dQacc, st);
    const int split = simt_split(tiles, nkt, nqt, S::BN, S::BM, p.causal, 2);
    auto go = [&](auto kernel, cudaError_t e) {
        if (e != cudaSuccess) return e;
        LaunchScope scope(MOA_KERNEL_BWD_KV, st);
        return launch_cluster(kernel, (unsigned)split, dim3((unsigned)(tiles * split)), dim3(SNT), S::kSmem, st, (const T *)Q, (const T *)K, (const T *)V,
                              (const T *)dO, L, Dv, (T *)dK, (T *)dV, dQacc, p.n, p.causal, p.scale, nkt, split);
    };
    if constexpr (R == 2)
        if (tiles * split <= device_info().sms && split >= nqt)
            return go(simt_bwd_kv_kernel<T, R, D, true>, allow_smem<simt_bwd_kv_kernel<T, R, D, true>>(S::kSmem));
    return go(simt_bwd_kv_kernel<T, R, D, false>, allow_smem<simt_bwd_kv_kernel<T, R, D, false>>(S::kSmem));
}
template <typename T, int D>
cudaError_t bwd_kv_t(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                     const float *L, const float *Dv, void *dK, void *dV, float *dQacc, cudaStream_t st)
{
    return bwd_kv_r<T, D == 64 ? 8 : 4, D>(p, Q, K, V, dO, L, Dv, dK, dV, dQacc, st);
}

template <typename T, int D>
cudaError_t bwd_dq_t(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                     const float *L, const float *Dv, void *dQ, cudaStream_t st)
{
    const int nqt = (p.n + BM - 1) / BM;
    cudaError_t e = allow_smem<simt_bwd_dq_kernel<T, D>>(bwd_smem(D));
    if (e != cudaSuccess) return e;
    LaunchScope scope(MOA_KERNEL_BWD_DQ, st);
    simt_bwd_dq_kernel<T, D><<<(unsigned)(nqt * p.BH()), NTHREADS, bwd_smem(D), st>>>(
        (const T *)Q, (const T *)K, (const T *)V, (const T *)dO, L, Dv, (T *)dQ, p.n, p.causal, p.scale, nqt);
    return cudaGetLastError();
}

template <typename T, int D>
cudaError_t rowpar_t(const Problem &p, const void *Q, const void *K, const void *V, const void *dO, void *O, float *L,
                     float *Dv, void *dQ, float *dKacc, float *dVacc, int sites, cudaStream_t st)
{
    const int nqt = (p.n + BM - 1) / BM;
    cudaError_t e = allow_smem<simt_rowpar_kernel<T, D, 1>>(bwd_smem(D));
    if (e == cudaSuccess) e = allow_smem<simt_rowpar_kernel<T, D, 2>>(bwd_smem(D));
    if (e != cudaSuccess) return e;
    LaunchScope scope(MOA_KERNEL_OTHER, st);
    if (sites == 2)
        simt_rowpar_kernel<T, D, 2><<<(unsigned)(nqt * p.BH()), NTHREADS, bwd_smem(D), st>>>(
            (const T *)Q, (const T *)K, (const T *)V, (const T *)dO, (T *)O, L, Dv, (T *)dQ, dKacc, dVacc,
            p.n, p.causal, p.scale, nqt);
    else
        simt_rowpar_kernel<T, D, 1><<<(unsigned)(nqt * p.BH()), NTHREADS, bwd_smem(D), st>>>(
            (const T *)Q, (const T *)K, (const T *)V, (const T *)dO, (T *)O, L, Dv, (T *)dQ, dKacc, dVacc,
            p.n, p.causal, p.scale, nqt);
    return cudaGetLastError();
}

#define MOA_DISPATCH(FN, ...)                                                         \
    do {                                                                              \
        if (dtype == MOA_F32) {                                                       \
            if (p.d == 64) return FN<float, 64>(__VA_ARGS__);                         \
            if (p.d == 128) return FN<float, 128>(__VA_ARGS__);                       \
        } else {                                                                      \
            if (p.d == 64) return FN<__nv_bfloat16, 64>(__VA_ARGS__);                 \
            if (p.d == 128) return FN<__nv_bfloat16, 128>(__VA_ARGS__);               \
        }                                                                             \
        return cudaErrorInvalidValue;                                                 \
    } while (0)

}  // namespace

cudaError_t simt_fwd(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                     void *O, float *L, const SimtPrep &pr, cudaStream_t st)
{
    MOA_DISPATCH(fwd_t, p, Q, K, V, O, L, pr, st);
}

cudaError_t simt_bwd_kv(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                        const void *dO, const float *L, const float *Dv,
                        void *dK, void *dV, float *dQacc, cudaStream_t st)
{
    MOA_DISPATCH(bwd_kv_t, p, Q, K, V, dO, L, Dv, dK, dV, dQacc, st);
}

cudaError_t simt_rowpar(const Problem &p, int dtype, const void *Q, const void *K, const void *V, const void *dO,
                        void *O, float *L, float *Dv, void *dQ, float *dKacc, float *dVacc, int sites, cudaStream_t st)
{
    MOA_DISPATCH(rowpar_t, p, Q, K, V, dO, O, L, Dv, dQ, dKacc, dVacc, sites, st);
}

cudaError_t simt_bwd_dq(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                        const void *dO, const float *L, const float *Dv, void *dQ, cudaStream_t st)
{
    MOA_DISPATCH(bwd_dq_t, p, Q, K, V, dO, L, Dv, dQ, st);
}

cudaError_t row_dot(const Problem &p, int dtype, const void *dO, const void *O, float *Dv, float *dQzero, cudaStream_t st)
{
    const size_t rows = (size_t)p.BH() * p.n;
    const int wpb = 8;
    const unsigned grid = (unsigned)((rows + wpb - 1) / wpb);
    LaunchScope scope(MOA_KERNEL_PREPROCESS, st);
    if (dtype == MOA_F32)
        return launch_dependent(row_dot_kernel<float>, dim3(grid), dim3(wpb * 32), (size_t)0, st, (const float *)dO, (const float *)O,
                                Dv, dQzero, rows, p.d);
    return launch_dependent(row_dot_kernel<__nv_bfloat16>, dim3(grid), dim3(wpb * 32), (size_t)0, st, (const __nv_bfloat16 *)dO,
                            (const __nv_bfloat16 *)O, Dv, dQzero, rows, p.d);
}

cudaError_t convert_f32_to_bf16(const float *src, void *dst, size_t count, float mul, cudaStream_t st)
{
    const size_t quads = (count + 3) / 4;
    size_t blocks = (quads + 4 * 256 - 1) / (4 * 256);
    if (blocks < 1) blocks = 1;
    if (blocks > 16LL * device_info().sms) blocks = 16LL * device_info().sms;     // grid-stride beyond 16 blocks per SM
    const unsigned grid = (unsigned)blocks;
    LaunchScope scope(MOA_KERNEL_CONVERT, st);
    return launch_dependent(convert_kernel, dim3(grid), dim3(256), (size_t)0, st, src, (__nv_bfloat16 *)dst, count, mul);
}

cudaError_t convert_f32_to_bf16_rows(const float *src, int src_ld, void *dst, int B, int H, int n, int d, Strides ds,
                                     float mul, cudaStream_t st)
{
    const size_t rows = (size_t)B * H * n, quads = rows * (size_t)(d / 4);
    size_t blocks = (quads + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > 16LL * device_info().sms) blocks = 16LL * device_info().sms;
    LaunchScope scope(MOA_KERNEL_CONVERT, st);
    return launch_dependent(convert_rows_kernel, dim3((unsigned)blocks), dim3(256), (size_t)0, st, src, src_ld, (__nv_bfloat16 *)dst, rows, n, H, d,
                            ds, mul);
}

}  // namespace moa
