// Decode attention for bf16 caches shared by groups of 4 to 16 query heads: the scores and the weighted sums of a group on
// warp-level tensor-core instructions (mma.sync m16n8k16, the queries of a group as the 16 rows), the cache streamed once.
//
// HBM-bound: 4 d bytes of cache per key against 4 d G flop; what matters is that every SM streams all the time.  The 128-row
// tiles of the tcgen05 forward kernel cost a job of that kernel about 3.5 tile times beside its tiles and the jobs go in
// whole rounds; here
//   * one CTA per SM takes an equal, contiguous share of all (K/V head, key tile) units, across heads, through one
//     ring of TMA loads (six stages of 32 KB: 64 keys at d = 128, 128 at d = 64) that never drains at a head's end;
//   * warp 8 requests the tiles; two groups of four warps take the tiles in turn, a warp 16 (d = 64: 32) keys of its group's tile:
//     S = q K^T with K rows by ldmatrix, online softmax per warp (rescaled only when a maximum grows by more than 8 in
//     the log2 domain), O += P V with V by ldmatrix.trans; about a hundred instructions per warp and 16 keys, a tenth of
//     what the SM can issue in the time HBM takes for them;
//   * when a CTA's share of a head ends, its eight warps' results are merged through shared memory.  A head that lies in one
//     CTA's share is written out at once; the others leave fp32 partial results in the workspace (at most two per CTA) for a
//     merge kernel, which is set up while this one streams;
//     (A wait, a softmax and an arrival per 16 KB were too much at d = 64: with 128 keys per tile there, and the merge in stripes, B1 H32/4
//     n16000 d64 went from 18.7 to 5.8 us, n32768 from 21.1 to 8.6, B2 H32/8 n8000 from 17.4 to 8.7, B1 H16/4 n3000 from 5.5 to 4.5.)
//   * few heads: a cluster of up to eight CTAs per head, merged through distributed shared memory, and no second kernel.
// Every wait is bounded; no CTA waits for another outside its cluster.
#include "common.cuh"
#include "ptx.cuh"
#include "tensormap.cuh"

namespace moa {
namespace {

using namespace ptx;

constexpr int kConsumers = 8, kMmaThreads = 32 * (kConsumers + 1);
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
constexpr float kRescale = 8.f;
enum : uint32_t { MERR_EMPTY = 0x311, MERR_FULL = 0x312 };

template <int D>
struct MmaSmem {
    static constexpr int kKeys = D == 128 ? 64 : 128;            // keys per tile: 16 or 32 per warp of a group
    static constexpr int kBox = kKeys * 128;                     // kKeys keys x 64 columns, 128-byte swizzle
    static constexpr int kTile = D / 64 * kBox;
    static constexpr int kStages = 6;                            // even: a stage belongs to one group of warps for good
    static constexpr int offMerge = kStages * 2 * kTile;         // [8 warps][8 queries][D + 2] floats
    static constexpr int offBar = offMerge + kConsumers * 8 * (D + 2) * 4;
    static constexpr int kTotal = offBar + 2 * kStages * 8 + 16;
};

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Units of CTA c: [first_unit(c), first_unit(c + 1)); the CTA that holds unit u.
__device__ __forceinline__ int first_unit(int units, int c, int ctas) { return (int)((long long)units * c / ctas); }
__device__ __forceinline__ int cta_of_unit(int units, int u, int ctas)
{
    int c = (int)(((long long)u * ctas) / units);
    while (first_unit(units, c + 1, ctas) <= u) ++c;
    return c;
}

// kHi: groups of 9 to 16 (the upper eight rows of the tiles are queries too)
template <int D, bool kHi>
__global__ void __launch_bounds__(kMmaThreads, 1)
decode_mma_kernel(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV,
                  const __nv_bfloat16 *__restrict__ q, __nv_bfloat16 *__restrict__ out, float *__restrict__ lse,
                  float *__restrict__ part_o, float *__restrict__ part_ml, int n, int Hkv, int G, int nt, int units, int cl,
                  float scale_log2, unsigned int *status)
{
    using S = MmaSmem<D>;
    constexpr int kRowsLane = kHi ? 2 : 1, kKS = D / 16, kNT = D / 8, kKeys = S::kKeys, kW = kKeys / 64;      // kW: 16-key steps of a warp
    extern __shared__ __align__(1024) uint8_t smem[];
    float *merge = reinterpret_cast<float *>(smem + S::offMerge);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + S::offBar), *empty = full + S::kStages;
    volatile uint32_t *abortp = reinterpret_cast<uint32_t *>(empty + S::kStages);
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    // cl > 0: the CTA of rank r of a cluster takes the r-th part of the cluster's head; otherwise an equal share of all units
    const int rank = cl ? (int)cluster_ctarank() : 0, ctas = (int)gridDim.x;
    const int u0 = cl ? (int)blockIdx.x / cl * nt + nt * rank / cl : first_unit(units, blockIdx.x, ctas);
    const int u1 = cl ? (int)blockIdx.x / cl * nt + nt * (rank + 1) / cl : first_unit(units, blockIdx.x + 1, ctas);
    if (tid == 0) {
        for (int s = 0; s < S::kStages; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, kConsumers / 2); }
        *abortp = (smem_u32(smem) & 1023u) ? 1u : 0u;
        if (*abortp && status) atomicCAS(status, 0u, (unsigned int)MERR_FULL);
        fence_mbar_init();
        prefetch_tensormap(&mapK);
        prefetch_tensormap(&mapV);
    }
    __syncthreads();
    grid_dependency_wait();
    grid_launch_dependents();
    const bool sound = *abortp == 0;

    if (warp == kConsumers) {
        // ------------------------------------------------------------------ producer
        if (lane == 0 && sound) {
            ArmCounts<S::kStages> armed;
            int head = u0 / nt, t = u0 - head * nt;
            for (int u = u0; u < u1; ++u) {
                const int i = u - u0, s = i % S::kStages;
                if (i >= S::kStages && !mbar_wait(empty + s, (i / S::kStages - 1) & 1, abortp, status, MERR_EMPTY)) break;
                const int b = head / Hkv, hk = head - b * Hkv;
                mbar_arm(full, s, 2 * S::kTile, armed);
                uint8_t *dst = smem + s * 2 * S::kTile;
                for (int x = 0; x < D / 64; ++x) {
                    tma_load_4d(dst + x * S::kBox, &mapK, full + s, 64 * x, t * kKeys, hk, b);
                    tma_load_4d(dst + S::kTile + x * S::kBox, &mapV, full + s, 64 * x, t * kKeys, hk, b);
                }
                if (++t == nt) { t = 0; ++head; }
            }
            mbar_drain(full, armed);      // copies still on their way land before the CTA leaves (bounded)
        }
        __syncwarp();
        if (cl > 1) {
            cluster_sync_all();
            cluster_sync_all();
        }
        return;
    }

    // ---------------------------------------------------------------------- consumers
    q = after_wait(q);
    const int grp = warp / 4, w4 = warp % 4, r0 = lane / 4, c0 = (lane % 4) * 2;
    // lane addresses of ldmatrix inside a tile: K rows as [keys][d], V transposed
    const uint32_t base = smem_u32(smem);
    const int krow = 16 * kW * w4 + (lane / 16) * 8 + lane % 8, kch = (lane / 8) & 1;
    const int vrow = 16 * kW * w4 + ((lane / 8) & 1) * 8 + lane % 8, vch = lane / 16;
    auto addr = [&](int row, int chunk) {       // 16-byte chunk `chunk` of a row of the tile
        return (uint32_t)((chunk >> 3) * S::kBox + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
    };
    int u = u0;
    bool ok = sound;
    while (u < u1) {
        const int head = u / nt, t_first = u - head * nt, seg_end = min(u1, (head + 1) * nt);
        uint32_t qa[kKS][4];
#pragma unroll
        for (int ks = 0; ks < kKS; ++ks)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = r0 + 8 * (e & 1);
                qa[ks][e] = ((e & 1) == 0 || kHi) && row < G
                                ? *reinterpret_cast<const uint32_t *>(q + ((size_t)head * G + row) * D + 16 * ks + c0 + 8 * (e >> 1)) : 0u;
            }
        float o[kNT][4], m[kRowsLane], l[kRowsLane];
#pragma unroll
        for (int i = 0; i < kNT; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[i][e] = 0.f;
#pragma unroll
        for (int i = 0; i < kRowsLane; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
        for (; u < seg_end; ++u) {
            const int i = u - u0, s = i % S::kStages;
            if ((i & 1) != grp) continue;                           // the other group's tile (and, kStages being even, stage)
            if (ok && !mbar_wait(full + s, (i / S::kStages) & 1, abortp, status, MERR_FULL)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) continue;
            const uint32_t tk = base + s * 2 * S::kTile, tv = tk + S::kTile;
            float sc[2 * kW][4];
#pragma unroll
            for (int j = 0; j < 2 * kW; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) sc[j][e] = 0.f;
#pragma unroll
            for (int ks = 0; ks < kKS; ++ks)
#pragma unroll
                for (int w = 0; w < kW; ++w) {
                    uint32_t kb[4];
                    ldmatrix4(kb, tk + addr(krow + 16 * w, 2 * ks + kch));
                    mma16816(sc[2 * w], qa[ks], kb[0], kb[1]);
                    mma16816(sc[2 * w + 1], qa[ks], kb[2], kb[3]);
                }
            const int key0 = (u - head * nt) * kKeys + 16 * kW * w4 + c0;
            if ((u - head * nt + 1) * kKeys > n)
#pragma unroll
                for (int j = 0; j < 2 * kW; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (key0 + 8 * j + (e & 1) >= n) sc[j][e] = -INFINITY;
            float mx[kRowsLane];
            bool grow = false;
#pragma unroll
            for (int h = 0; h < kRowsLane; ++h) {
                mx[h] = fmaxf(sc[0][2 * h], sc[0][2 * h + 1]);
#pragma unroll
                for (int j = 1; j < 2 * kW; ++j) mx[h] = fmaxf(mx[h], fmaxf(sc[j][2 * h], sc[j][2 * h + 1]));
                mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
                mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2)) * scale_log2;
                grow = grow || mx[h] > m[h] + kRescale;
            }
            if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
                for (int h = 0; h < kRowsLane; ++h) {
                    const float mn = fmaxf(m[h], mx[h]);
                    const float a = mn == -INFINITY ? 1.f : ex2(m[h] - mn);
                    m[h] = mn;
                    l[h] *= a;
#pragma unroll
                    for (int i2 = 0; i2 < kNT; ++i2) { o[i2][2 * h] *= a; o[i2][2 * h + 1] *= a; }
                }
            }
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                uint32_t pa[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int j = 0; j < 2; ++j)
#pragma unroll
                    for (int h = 0; h < kRowsLane; ++h) {
                        const float ref = m[h] == -INFINITY ? 0.f : m[h];      // (no key visible yet)
                        const float p0 = ex2(fmaf(sc[2 * w + j][2 * h], scale_log2, -ref)), p1 = ex2(fmaf(sc[2 * w + j][2 * h + 1], scale_log2, -ref));
                        l[h] += p0 + p1;
                        pa[2 * j + h] = pack_bf16(p0, p1);
                    }
#pragma unroll
                for (int nn = 0; nn < kNT / 2; ++nn) {
                    uint32_t vb[4];
                    ldmatrix4_trans(vb, tv + addr(vrow + 16 * w, 2 * nn + vch));
                    mma16816(o[2 * nn], pa, vb[0], vb[1]);
                    mma16816(o[2 * nn + 1], pa, vb[2], vb[3]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + s);
        }
        // ---- the segment's end: merge the warps, eight queries at a time
        const bool whole = t_first == 0 && seg_end == (head + 1) * nt;
        const int slot = 2 * (int)blockIdx.x + (t_first == 0 ? 1 : 0);
        constexpr int kLd = D + 2;
        float *seg = reinterpret_cast<float *>(smem);      // cluster: this CTA's part, [G][D + 2], over the ring, which is done
#pragma unroll
        for (int h = 0; h < kRowsLane; ++h) {
            float lt = l[h];
            lt += __shfl_xor_sync(0xffffffffu, lt, 1);
            lt += __shfl_xor_sync(0xffffffffu, lt, 2);
            named_barrier(1, 256);          // (the merge before has been read)
            float *row = merge + (warp * 8 + r0) * kLd;
#pragma unroll
            for (int i2 = 0; i2 < kNT; ++i2) *reinterpret_cast<float2 *>(row + 8 * i2 + c0) = make_float2(o[i2][2 * h], o[i2][2 * h + 1]);
            if (lane % 4 == 0) { row[D] = m[h]; row[D + 1] = lt; }
            named_barrier(1, 256);
            for (int idx = tid; idx < min(8, G - 8 * h) * D; idx += 256) {
                const int r = idx / D, c = idx - r * D, g = 8 * h + r;
                float mt = -INFINITY, ot = 0.f, ls = 0.f;
#pragma unroll
                for (int w = 0; w < kConsumers; ++w) mt = fmaxf(mt, merge[(w * 8 + r) * kLd + D]);
                const float ref = mt == -INFINITY ? 0.f : mt;
#pragma unroll
                for (int w = 0; w < kConsumers; ++w) {
                    const float *src = merge + (w * 8 + r) * kLd;
                    const float a = ex2(src[D] - ref);
                    ot = fmaf(src[c], a, ot);
                    ls = fmaf(src[D + 1], a, ls);
                }
                if (cl > 1) {
                    seg[g * kLd + c] = ot;
                    if (c == 0) { seg[g * kLd + D] = mt; seg[g * kLd + D + 1] = ls; }
                } else if (whole) {
                    out[((size_t)head * G + g) * D + c] = __float2bfloat16_rn(ot / ls);
                    if (lse && c == 0) lse[(size_t)head * G + g] = (mt + log2f(ls)) * kLn2;
                } else {
                    part_o[((size_t)slot * G + g) * D + c] = ot;
                    if (c == 0) { part_ml[((size_t)slot * G + g) * 2] = mt; part_ml[((size_t)slot * G + g) * 2 + 1] = ls; }
                }
            }
        }
        if (cl > 1) {       // (the only segment)
            cluster_sync_all();
            auto peer = [&](const float *mine, int k) {
                float v;
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(mapa_u32(smem_u32(mine), (uint32_t)k)) : "memory");
                return v;
            };
            for (int idx = rank * 256 + tid; idx < G * D; idx += cl * 256) {
                const int g = idx / D, c = idx - g * D;
                const float *at = seg + g * kLd;
                float mt = -INFINITY, ot = 0.f, ls = 0.f;
                for (int k = 0; k < cl; ++k) mt = fmaxf(mt, peer(at + D, k));
                for (int k = 0; k < cl; ++k) {
                    const float a = ex2(peer(at + D, k) - mt);
                    ot = fmaf(peer(at + c, k), a, ot);
                    ls = fmaf(peer(at + D + 1, k), a, ls);
                }
                out[((size_t)head * G + g) * D + c] = __float2bfloat16_rn(ot / ls);
                if (lse && c == 0) lse[(size_t)head * G + g] = (mt + log2f(ls)) * kLn2;
            }
            cluster_sync_all();       // nobody leaves while another CTA may still read its shared memory
        }
    }
}

// Heads shared by several CTAs of the kernel above: a block per query head adds their partial results, its 128 threads in stripes of D / 4
// over the CTAs, so that a head of 37 CTAs (four heads on 148 SMs) is one or two rounds of loads and not ten.
template <int D>
__global__ void __launch_bounds__(128)
decode_mma_merge_kernel(const float *__restrict__ part_o, const float *__restrict__ part_ml, __nv_bfloat16 *__restrict__ out,
                        float *__restrict__ lse, int G, int nt, int units, int ctas)
{
    constexpr int kLanes = D / 4, kStripes = 128 / kLanes, kBatch = 8;
    __shared__ float4 so[kStripes][kLanes];
    __shared__ float2 sml[kStripes];
    const int head = (int)blockIdx.x / G, g = (int)blockIdx.x - head * G;
    const int ca = cta_of_unit(units, head * nt, ctas), cb = cta_of_unit(units, (head + 1) * nt - 1, ctas);
    grid_dependency_wait();
    grid_launch_dependents();
    if (ca == cb) return;
    part_o = after_wait(part_o);
    part_ml = after_wait(part_ml);
    const int stripe = (int)threadIdx.x / kLanes, lane = (int)threadIdx.x % kLanes, c = 4 * lane;
    float mt = -INFINITY, ls = 0.f;
    float4 ot = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = ca + stripe; k0 <= cb; k0 += kStripes * kBatch) {
        float2 ml[kBatch];
        float4 v[kBatch];
        float mn = mt;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int k = k0 + u * kStripes;
            const size_t at = (size_t)(2 * k + (k == ca ? 1 : 0)) * G + g;
            const bool there = k <= cb;
            ml[u] = there ? *reinterpret_cast<const float2 *>(part_ml + at * 2) : make_float2(-INFINITY, 0.f);
            v[u] = there ? *reinterpret_cast<const float4 *>(part_o + at * D + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) mn = fmaxf(mn, ml[u].x);
        const float ref = mn == -INFINITY ? 0.f : mn, b = ex2(mt - ref);
        mt = mn;
        ls *= b;
        ot.x *= b; ot.y *= b; ot.z *= b; ot.w *= b;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float a = ex2(ml[u].x - ref);
            ls = fmaf(ml[u].y, a, ls);
            ot.x = fmaf(v[u].x, a, ot.x); ot.y = fmaf(v[u].y, a, ot.y); ot.z = fmaf(v[u].z, a, ot.z); ot.w = fmaf(v[u].w, a, ot.w);
        }
    }
    so[stripe][lane] = ot;
    if (lane == 0) sml[stripe] = make_float2(mt, ls);
    __syncthreads();
    if (stripe == 0) {
        float mx = -INFINITY;
#pragma unroll
        for (int k = 0; k < kStripes; ++k) mx = fmaxf(mx, sml[k].x);
        ls = 0.f;
        ot = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kStripes; ++k) {
            const float a = ex2(sml[k].x - mx);
            const float4 v = so[k][lane];
            ls = fmaf(sml[k].y, a, ls);
            ot.x = fmaf(v.x, a, ot.x); ot.y = fmaf(v.y, a, ot.y); ot.z = fmaf(v.z, a, ot.z); ot.w = fmaf(v.w, a, ot.w);
        }
        const float inv = 1.f / ls;
        *reinterpret_cast<uint2 *>(out + ((size_t)head * G + g) * D + c) =
            make_uint2(pack_bf16(ot.x * inv, ot.y * inv), pack_bf16(ot.z * inv, ot.w * inv));
        if (lse && c == 0) lse[(size_t)head * G + g] = (mx + log2f(ls)) * kLn2;
    }
}

template <int D, bool kHi>
cudaError_t launch(const DecodeProblem &p, const void *q, const void *K, const void *V, void *out, float *lse, void *ws, cudaStream_t st)
{
    using S = MmaSmem<D>;
    CUtensorMap mk, mv;
    const auto bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    if (!make_tensor_map_4d(&mk, K, bf, 2, p.B, p.Hkv, p.n, D, false, S::kKeys, 64) ||
        !make_tensor_map_4d(&mv, V, bf, 2, p.B, p.Hkv, p.n, D, false, S::kKeys, 64))
        return cudaErrorInvalidValue;
    const int G = p.H / p.Hkv, nt = (p.n + S::kKeys - 1) / S::kKeys, heads = p.B * p.Hkv, units = nt * heads, sms = device_info().sms;
    const cudaError_t e = allow_smem<decode_mma_kernel<D, kHi>>(S::kTotal);
    if (e != cudaSuccess) return e;
    // A cluster per head while all of them fit at once (clusters of 4 and 8 leave SMs of a GPC over: a sixteenth cluster of 8 waits for the
    // others, 24.7 us for B16 H8/1 n12595 d64, 13.4 without clusters), unless its CTAs would stream more than 192 KB beyond an equal share: the merge
    // kernel costs about what an SM streams in that time.
    int cl = 0;
    for (int c = 1; c <= 8 && c <= nt && heads * c * 100 <= sms * (c == 8 ? 85 : c == 4 ? 90 : 100); c *= 2) cl = c;
    if (cl && (long long)((nt + cl - 1) / cl - (units + sms - 1) / sms) * 2 * S::kTile > 192 * 1024) cl = 0;
    const int ctas = cl ? heads * cl : units < sms ? units : sms;
    float *part_o = (float *)ws, *part_ml = part_o + (size_t)2 * sms * G * D;
    {
        LaunchScope scope(MOA_KERNEL_OTHER, st);
        const cudaError_t le = launch_cluster(decode_mma_kernel<D, kHi>, cl > 1 ? (unsigned)cl : 1u, dim3((unsigned)ctas), dim3(kMmaThreads),
                                              (size_t)S::kTotal, st, mk, mv, (const __nv_bfloat16 *)q, (__nv_bfloat16 *)out, lse, part_o,
                                              part_ml, p.n, p.Hkv, G, nt, units, cl, p.scale * kLog2e, device_status_ptr());
        if (le != cudaSuccess || cl) return le;
    }
    LaunchScope scope(MOA_KERNEL_OTHER, st);
    return launch_dependent(decode_mma_merge_kernel<D>, dim3((unsigned)(heads * G)), dim3(128), (size_t)0, st, (const float *)part_o,
                            (const float *)part_ml, (__nv_bfloat16 *)out, lse, G, nt, units, ctas);
}

}  // namespace

// Groups of 4 to 16 (below, the CUDA-core kernels keep their fp32 weights; above, the group fills the rows of a tcgen05 tile
// better); the units have to be countable in an int.
bool decode_uses_mma(const DecodeProblem &p, int dtype)
{
    const int G = p.H / p.Hkv;
    return dtype == MOA_BF16 && G >= 4 && G <= 16 && p.scale > 0.f && ((long long)p.n + 63) / 64 * p.B * p.Hkv < (1LL << 31);
}

size_t decode_mma_workspace_bytes(const DecodeProblem &p)
{
    return (size_t)2 * device_info().sms * (p.H / p.Hkv) * (p.d + 2) * sizeof(float);
}

cudaError_t decode_mma(const DecodeProblem &p, const void *q, const void *K, const void *V, void *out, float *lse, void *ws, cudaStream_t st)
{
    const bool hi = p.H / p.Hkv > 8;
    if (p.d == 64) return hi ? launch<64, true>(p, q, K, V, out, lse, ws, st) : launch<64, false>(p, q, K, V, out, lse, ws, st);
    if (p.d == 128) return hi ? launch<128, true>(p, q, K, V, out, lse, ws, st) : launch<128, false>(p, q, K, V, out, lse, ws, st);
    return cudaErrorInvalidValue;
}

}  // namespace moa
