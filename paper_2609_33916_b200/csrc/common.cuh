// Shared declarations of the CUDA library's translation units (internal; the
// public interface is include/moa_attn.h).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include <mutex>
#include "moa_attn.h"

namespace moa {

// Where element (b, h, row, 0) of one of the caller's tensors lives: b * batch + h * head + row * row elements past
// its base pointer (the d elements of a row are contiguous).
struct Strides {
    long long row, head, batch;
    __host__ __device__ size_t at(long long b, long long h, long long r) const { return (size_t)(b * batch + h * head + r * row); }
};

struct Problem {
    int B, H, n, d;
    int causal;
    float scale;
    int Hkv = 0;                                   // key/value heads; 0: same as H
    int bnhd = 0;                                  // 1: the caller's tensors are [B,n,H,d] in memory (L stays [B,H,n])
    // strides of the three tensor classes: Q, dQ | K, V, dK, dV | O, dO.  Filled by with_layout() from the fixed
    // layouts, or taken from the descriptor (MOA_LAYOUT_STRIDED).
    Strides sq{0, 0, 0}, skv{0, 0, 0}, so{0, 0, 0};
    Problem &with_layout()
    {
        const long long hk = kv_heads();
        if (bnhd) {
            sq = so = Strides{(long long)H * d, d, (long long)n * H * d};
            skv = Strides{hk * d, d, (long long)n * hk * d};
        } else {
            sq = so = Strides{d, (long long)n * d, (long long)H * n * d};
            skv = Strides{d, (long long)n * d, hk * n * d};
        }
        return *this;
    }
    bool contiguous_bhnd() const     // every tensor is a plain [B,heads,n,d] array
    {
        return sq.row == d && sq.head == (long long)n * d && sq.batch == (long long)H * n * d && so.row == sq.row &&
               so.head == sq.head && so.batch == sq.batch;
    }
    int BH() const { return B * H; }
    int kv_heads() const { return Hkv > 0 ? Hkv : H; }
    int group() const { return H / kv_heads(); }    // query heads per key/value head
    int BHkv() const { return B * kv_heads(); }
};

// Head dimension the tensor-core kernels are compiled for: a head of d columns (a multiple of 8, so
// that rows stay 16-byte aligned) runs in the 64-, 128- or 256-column kernels; the TMA loads fill the
// columns past d with zeros and the TMA stores drop them, which leaves every result unchanged.
// 256: the kernels for head dimensions 136..256 (tc_fwd_wide.cu, tc_bwd_192.cu, tc_bwd_wide.cu).
inline int kernel_d(int d) { return d <= 64 ? 64 : d <= 128 ? 128 : 256; }

// Block order of the tile-parallel kernels.  Heads are taken in groups of `hpg`; inside a group
// the blocks go tile-major (every head's tile 0, then every head's tile 1, ...).  With causal
// masking tile t is the t-th longest job, so the hardware's in-order block dispatch becomes
// longest-job-first inside a group and the last blocks to start are the shortest: head-major
// order left SMs idle for ~12 % of a causal backward, waiting for long jobs that started late.
// hpg = 1 is head-major order (best L2 locality), used whenever all jobs have the same length.
__device__ __forceinline__ void job_from_block(int block, int tiles, int heads, int hpg, int &bh, int &t)
{
    const int per_group = hpg * tiles;
    const int group = block / per_group, r = block - group * per_group;
    const int cur = min(hpg, heads - group * hpg);
    t = r / cur;
    bh = group * hpg + (r - t * cur);
}

// What the launch arithmetic needs to know about the current device, read once per device
// (cudaDevAttrMultiProcessorCount, cudaDevAttrL2CacheSize); a B200 gives 148 SMs and 126 MB.
struct DeviceInfo {
    int sms;             // streaming multiprocessors
    long long l2_bytes;  // L2 cache
};
const DeviceInfo &device_info();

// Heads per group: enough jobs per group that its longest job (tiles iterations) is shorter than
// the group's share of the SMs, and as many heads as keep Q, K, V, dO of a group within half of L2.
inline int heads_per_group(const Problem &p, int tiles)
{
    if (!p.causal) return 1;
    const DeviceInfo &dev = device_info();
    const long long per_head = 4LL * p.n * p.d * 2;
    const long long fit = (dev.l2_bytes / 2 + per_head / 2) / (per_head > 0 ? per_head : 1);     // to the nearest head
    long long g = (2 * dev.sms + tiles) / (tiles + 1);
    if (fit > g) g = fit;
    if (g < 1) g = 1;
    if (g > p.BH()) g = p.BH();
    const long long groups = (p.BH() + g - 1) / g;      // groups of equal size (to within one head)
    g = (p.BH() + groups - 1) / groups;
    return (int)g;
}

// CTAs that share a key tile of the backward (a cluster; each takes a contiguous part of the tile's query tiles and the partial
// dK, dV are added through distributed shared memory).  One CTA per key tile leaves SMs idle when there are few tiles, and with
// shared K/V heads or the causal mask the longest tile alone can outlast the average SM's share by far.  Estimated in units
// of one query tile: a CTA costs `fixed` beside its tiles, a merge `merge` more; equal jobs go in rounds, causal ones longest first,
// which packs to within a part of an average job.  A cluster has to beat the next smaller one by 5 %.
//   jobs: key tiles of all K/V heads (times the passes over d); longest, total: query tiles of the longest job, of all jobs;
//   per_sm: CTAs that an SM holds at once
inline int bwd_split(long long jobs, long long longest, long long total, bool causal, double fixed, double merge, int per_sm = 1)
{
    const double sms = (double)device_info().sms * per_sm;
    int best = 1;
    double best_cost = 0;
    for (int s = 1; s <= 8; s *= 2) {
        if (s > 1 && (longest < s || jobs * s > 8 * (long long)sms)) break;
        // (clusters of 4 and 8 leave SMs of a GPC over; less so where an SM holds several CTAs)
        const double slots = s <= 2 ? sms : s == 4 ? (per_sm > 1 ? 1.0 : 0.9) * sms : (per_sm > 1 ? 0.89 : 0.85) * sms;
        const double extra = fixed + (s > 1 ? merge : 0.0), job = (double)longest / s + extra;
        const double avg = ((double)total + (double)jobs * s * extra) / slots, mean = (double)total / (jobs * s) + extra;
        const long long n = jobs * s, rounds = (n + (long long)slots - 1) / (long long)slots;
        const double even = (double)rounds * job, packed = avg + 0.5 * mean;
        const double cost = causal ? (job > packed ? job : packed < even ? packed : even) : even;
        if (s == 1 || cost < 0.95 * best_cost) { best = s; best_cost = cost; }
    }
    return best;
}

// Decode through the tensor-core forward kernel (tc_fwd.cu): the G query heads of a K/V head are
// the rows of one query tile, the cache is split among CTAs; partial results to be merged.
cudaError_t tc_fwd_decode(int B, int Hkv, int G, int n, int d, float scale, const void *q, const void *K, const void *V,
                          void *O_part, float *L_part, int splits, int tiles_per_split, cudaStream_t st);

// ---- decode attention (decode.cu) ----------------------------------------------------
struct DecodeProblem {
    int B, H, Hkv, n, d;     // Hkv resolved (never 0)
    float scale;
};
size_t decode_workspace_bytes(const DecodeProblem &p, int dtype);    // partial results of all segments
// q [B,H,d], K, V [B,Hkv,n,d] -> out [B,H,d] (dtype of the inputs), lse [B,H] fp32 (may be null)
cudaError_t decode_attn(const DecodeProblem &p, int dtype, const void *q, const void *K, const void *V, void *out,
                        float *lse, void *ws, cudaStream_t st);

// groups of query heads on warp-level tensor-core instructions (decode_mma.cu)
bool decode_uses_mma(const DecodeProblem &p, int dtype);
size_t decode_mma_workspace_bytes(const DecodeProblem &p);
cudaError_t decode_mma(const DecodeProblem &p, const void *q, const void *K, const void *V, void *out, float *lse, void *ws,
                       cudaStream_t st);
// counters of a merge by the last CTA to zero, in stream order
cudaError_t decode_clear(unsigned int *counters, int count, cudaStream_t st);

// Host-side launch counter (moa_launch_count).
void count_launch(int k = 1);

// Brackets one kernel launch with an event pair when profiling is enabled
// (moa_profile_enable); also counts the launch.
struct LaunchScope {
    LaunchScope(int kind, cudaStream_t st);
    ~LaunchScope();
    int slot;
    cudaStream_t st;
};

// Launch `kernel` so that it may start before the kernel in front of it in the stream has finished (programmatic
// dependent launch), in clusters of `cluster` CTAs.  Every kernel launched like this keeps to two rules, which together
// make the early start invisible:
//   * it calls ptx::grid_dependency_wait() before it reads or writes global memory -- except that a kernel that is never the
//     first of a call may read the call's own inputs before that: the attention backward kernels, and decode's streaming kernels where they
//     merge through memory.  (The latter rest on decode_clear_kernel in front of them, which triggers only after its own wait: without it they
//     would read the cache while the caller's update of it still runs.)
//   * it calls ptx::grid_launch_dependents() only after that wait.  So once a kernel's successor runs at all, everything in
//     front of the kernel itself, the caller's work included, has completed.
// What overlaps is the set-up (barriers, TMEM allocation, tensor-map fetches) and the launch latency.
// MOA_PDL=0 in the environment turns the attribute off (plain stream order).
bool pdl_enabled();
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster_as(bool dependent, void (*kernel)(KArgs...), unsigned cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dependent && pdl_enabled() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), unsigned cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    return launch_cluster_as(true, kernel, cluster, grid, block, smem, st, args...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    return launch_cluster(kernel, 1u, grid, block, smem, st, args...);
}

// Lets `Kernel` use `bytes` of dynamic shared memory (cudaFuncSetAttribute).  The driver call is made once per kernel and
// device and again only for more than any call before asked for; it took a tenth of a small call's host time.
template <auto Kernel>
cudaError_t allow_smem(size_t bytes)
{
    constexpr int kMaxDev = 64;
    static std::atomic<size_t> allowed[kMaxDev];
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < kMaxDev;
    if (known && allowed[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
    std::lock_guard<std::mutex> lk(mu);      // (so that two threads cannot leave the smaller of two sizes in force)
    if (known && allowed[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && known) allowed[dev].store(bytes, std::memory_order_release);
    return e;
}

// Whether two arrays share memory.  A caller may lay an output over an input that only earlier kernels of a call read (dx over dy, say); a
// rule that lets kernels of a call run side by side has to look.
inline bool arrays_meet(const void *a, size_t a_bytes, const void *b, size_t b_bytes)
{
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return x < y + b_bytes && y < x + a_bytes;
}

// Device address of the status word kernels write when a bounded wait expires.
unsigned int *device_status_ptr();

// MOA_OK when the current device is compute capability 10.x, MOA_ERR_ARCH otherwise (cached per device).
moa_status check_device_arch();

// ---- block pieces (block_norm.cu, tc_gemm.cu), bf16 ------------------------------------
size_t rmsnorm_workspace_bytes(int n, int d);          // per-CTA partial sums of dg
cudaError_t rmsnorm_fwd(int n, int d, float eps, const void *x, const void *g, void *y, float *r, cudaStream_t st);
// dx_add (may be null): dx = (RMSNorm backward) + dx_add
cudaError_t rmsnorm_bwd(int n, int d, float eps, const void *x, const void *g, const float *r, const void *dy,
                        const void *dx_add, void *dx, void *dg, void *ws, cudaStream_t st);
// gated MLP (tc_gemm.cu): x, y, dy, dx [n,d]; W1, W3 [d_ff,d]; W2 [d,d_ff]; a, u, h, da, du [n,d_ff]
// res (may be null): y = h W2^T + res
cudaError_t gated_mlp_fwd(int n, int d, int dff, const void *x, const void *W1, const void *W3, const void *W2,
                          const void *res, void *a, void *u, void *h, void *y, cudaStream_t st);
// C[M,N] = A B^T (+ R): A given as [M,K] (a_mn = 0) or [K,M] (a_mn = 1), B as [N,K] (b_mn = 0) or [K,N] (b_mn = 1); bf16
cudaError_t gemm_bf16(int a_mn, int b_mn, int M, int N, int K, const void *A, const void *B, const void *R, void *C,
                      cudaStream_t st);
struct GemmArgs {
    int a_mn, b_mn, M, N, K;
    const void *A, *B;
    void *C;
};
cudaError_t gemm_bf16_two(const GemmArgs &x, const GemmArgs &y, cudaStream_t st);      // one launch where both are small
cudaError_t gated_mlp_bwd(int n, int d, int dff, const void *x, const void *W1, const void *W3, const void *W2,
                          const void *a, const void *u, const void *h, const void *dy, void *da, void *du,
                          void *dx, void *dW1, void *dW3, void *dW2, cudaStream_t st);

template <typename T> __device__ __forceinline__ float to_float(T v);
template <> __device__ __forceinline__ float to_float<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_float(float v);
template <> __device__ __forceinline__ float from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---- tensor-core path (tc_fwd.cu), bf16 only ---------------------------------------------
// What the forward of a fused call does for its backward (all null for a plain forward): it clears the fp32
// dQ accumulator [B*H, n, kernel_d(d)], and writes the backward's per-row inputs -L log2 e and -D = -rowsum(dO o O)
// (from the fp32 O it holds), padded to n_pad rows per head with -inf / 0.
struct FwdForBwd {
    float *zero_acc = nullptr;
    const void *dO = nullptr;
    float *Lp = nullptr, *Dp = nullptr;
};
cudaError_t tc_fwd(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L,
                   const FwdForBwd &fb, cudaStream_t st);

// The same on pairs of query tiles (tc_fwd2.cu; d <= 128), and whether that is the faster form of a problem
cudaError_t tc_fwd_pairs(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb, cudaStream_t st);
bool fwd_pairs_pay(const Problem &p);

// Head dimensions 136..256 (tc_fwd_wide.cu)
cudaError_t tc_fwd_wide(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb, cudaStream_t st);

// Lp = -L*log2(e) and Dp = -rowsum(dO o O) (negated: fma/add operands), each padded per head to a
// multiple of 128 rows (-inf / 0 past n)
// (and, unless zero_acc is null, clears the fp32 accumulator [B*H, n, kernel_d(d)] the backward adds dQ into)
cudaError_t tc_bwd_preprocess(const Problem &p, const void *dO, const void *O, const float *L, float *Lp, float *Dp,
                              float *zero_acc, cudaStream_t st);
// dK, dV; UNSCALED dQ contributions (dS K, without the factor scale) red-added into dQacc
// (fp32 [B,H,n,kernel_d(d)], pre-zeroed); dQacc == nullptr skips the dQ contraction altogether
cudaError_t tc_bwd_kv(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                      const float *Lp, const float *Dp, void *dK, void *dV, float *dQacc, int dq_bulk,
                      bool share, cudaStream_t st);   // dq_bulk: TMA bulk add-reduce instead of red.global (d <= 128 only)
// share: several CTAs may share a key tile (bwd_split).  MOA_DQ_AUTO only: the dq_modes a caller names are for comparing the
// strategies, all on the same one-CTA-per-key-tile form (and its bits of dK, dV, which the paired form reproduces).

// The same on pairs of CTAs (tc_bwd_pair.cu; the 128-column kernel only), and whether tc_bwd_kv hands such
// problems to it (moa_bwd_pair_mode; environment variable MOA_BWD_PAIR=1 for the initial mode; default: no)
cudaError_t tc_bwd_kv_pair(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                           const float *Lp, const float *Dp, void *dK, void *dV, float *dQacc, int dq_bulk,
                           cudaStream_t st);
bool bwd_pair_enabled();
int bwd_pair_mode(int set);      // set < 0: query; returns the mode in force before the call

// Head dimensions 136..192 in one pass (tc_bwd_192.cu) and 200..256 in two passes over the halves of d (tc_bwd_wide.cu): tiles of 128
// keys x 64 queries; dQ by red.global into dQacc (fp32 [B,H,n,256], pre-zeroed)
cudaError_t tc_bwd_kv_192(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                          const float *Lp, const float *Dp, void *dK, void *dV, float *dQacc, bool share, cudaStream_t st);
cudaError_t tc_bwd_kv_wide(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                           const float *Lp, const float *Dp, void *dK, void *dV, float *dQacc, bool share, cudaStream_t st);

// atomic-free query-parallel dQ pass on the tensor cores (tc_dq.cu); writes dQ (bf16) directly
cudaError_t tc_bwd_dq(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                      const float *Lp, const float *Dp, void *dQ, cudaStream_t st);

// ---- n x n-materialising comparison variant (tc_materialize.cu), bf16 --------------------
// P^T and dS^T are [heads][n_pad][n_pad] bf16 arrays in the caller's workspace.
cudaError_t mat_fwd(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, void *PT,
                    cudaStream_t st);
cudaError_t mat_bwd(const Problem &p, const void *Q, const void *K, const void *V, const void *dO, const float *Dp,
                    const void *PT, void *GST, void *dQ, void *dK, void *dV, cudaStream_t st);

// ---- SIMT fp32 path (simt_kernels.cu) -------------------------------------------------
// dtype: MOA_BF16 or MOA_F32 storage; arithmetic is fp32 FMA throughout.
// What the forward of a fused call prepares for its backward (all null for a plain forward): D = rowsum(dO o O) [B*H, n]
// and the cleared dQ accumulator [B*H, n, d] (null: not wanted).
struct SimtPrep {
    const void *dO = nullptr;
    float *Dv = nullptr, *dQzero = nullptr;
};
cudaError_t simt_fwd(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                     void *O, float *L, const SimtPrep &pr, cudaStream_t st);
// D_i = sum_k dO_ik O_ik; dQzero (may be null): fp32 [B*H, n, d] to clear
cudaError_t row_dot(const Problem &p, int dtype, const void *dO, const void *O, float *Dv, float *dQzero, cudaStream_t st);
// dK, dV always; dQ contributions are atomically added into dQacc (fp32 [B,H,n,d], pre-zeroed)
// when dQacc != nullptr.
cudaError_t simt_bwd_kv(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                        const void *dO, const float *L, const float *Dv,
                        void *dK, void *dV, float *dQacc, cudaStream_t st);
// atomic-free query-parallel dQ pass
// Row-parallel fused forward+backward in one kernel with dK (sites = 1) or dK and dV (sites = 2)
// accumulated by fp32 atomics into dKacc / dVacc [B*H, n, d]; writes O, L, D, dQ.
cudaError_t simt_rowpar(const Problem &p, int dtype, const void *Q, const void *K, const void *V, const void *dO,
                        void *O, float *L, float *Dv, void *dQ, float *dKacc, float *dVacc, int sites, cudaStream_t st);
cudaError_t simt_bwd_dq(const Problem &p, int dtype, const void *Q, const void *K, const void *V,
                        const void *dO, const float *L, const float *Dv, void *dQ, cudaStream_t st);
// dst[i] = (bf16)(mul * src[i])
cudaError_t convert_f32_to_bf16(const float *src, void *dst, size_t count, float mul, cudaStream_t st);
// the same row by row: the accumulator is [B*H, n, src_ld] (src_ld >= d: the kernels' padded head
// dimension), the destination addressed through the strides `ds` of the caller's dQ
cudaError_t convert_f32_to_bf16_rows(const float *src, int src_ld, void *dst, int B, int H, int n, int d, Strides ds,
                                     float mul, cudaStream_t st);

}  // namespace moa
