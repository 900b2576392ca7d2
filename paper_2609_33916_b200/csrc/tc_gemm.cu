// bf16 GEMMs of the gated MLP on the tensor cores (tcgen05, fp32 accumulators in TMEM, operands
// staged by TMA), with the gate arithmetic fused into the epilogues.
//
//   C[M,N] = sum over operand pairs p of  A_p[M,K] * B_p[N,K]^T
//
// One persistent CTA per SM walks output tiles of 128 x kN, kN = 256, 128 or 64.  Warp 0 is the TMA producer (a ring of
// stages of 64 K-elements: 16 KB of A, 128 kN bytes of B), warp 1 allocates TMEM and issues the
// UMMAs (M = 128, N = kN, K = 16 each, four per stage), warps 2-9 are the epilogue (two warps per
// 32-lane group of TMEM, one column half each).  Two
// kN-column accumulators in TMEM alternate between tiles, so the epilogue of a tile runs under the main
// loop of the next one.  Every wait is bounded (ptx::mbar_wait).
//
// kPair: the same roles in each of the two CTAs of a cluster, on tiles of 256 x 256: the CTA of rank 0
// issues UMMAs of M = 256 (tcgen05.mma.cta_group::2) that read 128 rows of A and HALF of the B rows
// from each CTA's shared memory and write 128 x 256 accumulators in each CTA's TMEM.  Per SM and
// unit of work the B traffic (L2 -> shared memory, shared memory -> tensor core) halves; a stage holds
// two 64-element K blocks (64 KB) and the ring has three.  Both producers' copies complete on the full barrier of rank 0; its
// commits arrive on the empty and accumulator-full barriers of both CTAs; both epilogues hand the
// accumulator back on the barrier of rank 0; a cluster-wide barrier at both ends keeps either CTA
// from touching the other before it is set up or after it has left.  Measured: products of every
// operand layout 1240-1340 -> 1350-1530 TFLOP/s; launches of a few tiles, and shapes whose M is so
// small that pairs would need more waves, stay on single CTAs.
//
// A small product is bound by what a launch does once: in a chain of dependent launches of 512 x 64 x 64 the first load went out 0.9 us
// after the kernel in front was done and the CTA left 1.3 us after its last store was issued.  The place of the first tile is worked out in
// front of the wait for that kernel, K blocks past K are not loaded, the residual (and the gate's stored a, u) are requested
// while the main loop runs, and copies are only waited for at the end if a wait has expired (in every other case each of them has been waited
// for): 5.4 -> 3.3 us per launch, and 8192 x 2048 x 2048 53.6 -> 49.7 us.
//
// Operand storage is a template choice per operand, because the backward's GEMMs read the same
// arrays transposed:
//   K-major  : the array is [rows = M or N, K] row-major; one TMA box of 64 K-elements x rows.
//   MN-major : the array is [K, cols = M or N] row-major; boxes of 64 columns x 64 K-rows.
// Tails in M, N and K are handled by the TMA zero fill on loads and by guards on stores.
//
// Epilogues:
//   EPI_STORE       C -> bf16; with a residual R (map C2) C + R -> bf16 (residual connections, sums of products)
//   EPI_SWIGLU_FWD  the tile's B rows are 128 rows of W1 and the same 128 rows of W3 (two maps), so
//                   its accumulator holds a | u for 128 hidden units; writes a, u and
//                   h = silu(a) * u (all from the fp32 values).
//   EPI_SWIGLU_BWD  C = dh; reads the stored a, u; writes da = dh u s (1 + a (1 - s)) and
//                   du = dh a s, s = sigmoid(a).  dh itself never reaches memory.
#include "common.cuh"
#include "gemm_rule.cuh"
#include "ptx.cuh"
#include "tensormap.cuh"
#include "moa_block.h"

namespace moa {
namespace {

using namespace ptx;

constexpr int GM = 128, GK = 64;                       // (gemm_rule.cuh counts in these)
constexpr int kGemmThreads = 320;                      // producer, issuer, eight epilogue warps
constexpr int kABytes = GM * GK * 2;
// A CTA on its own stages 16 KB of A and 32 KB of B per 64 K-elements, four stages (three measured 7-16 % slower: the
// ring has to cover the L2 latency).  A CTA of a pair stages 16 KB of A and its half of B, 16 KB: six stages.
// In a pair a stage holds two such blocks (128 K-elements, 64 KB) and the ring has three: one wait and one commit of
// the issuing thread per eight UMMAs instead of per four (six stages of one block: 4096^3 94.9 / 97.5 us, 8192 x 2048 x 8192
// 187 / 191).
// Narrower tiles are for launches whose 256-column tiles would leave SMs idle: less work per SM and a shorter epilogue, at more operand
// traffic per unit of work.  Their stages hold two K blocks as well: with one (six stages at 128 columns, eight at 64) operands stored by
// columns, whose copies are many, fall behind (512 x 512 x 2048 (1,1) 7.8 / 9.7 us, 1024 x 1024 x 1613 (1,1) 7.7 / 9.1; others level).
constexpr int kMaxStages = 6;
__host__ __device__ constexpr int gemm_sub(bool pair, int n) { return pair || n < 256 ? 2 : 1; }       // 64-element K blocks per stage
__host__ __device__ constexpr int gemm_stages(bool pair, int n) { return pair ? 3 : n == 256 ? 4 : n == 128 ? 3 : 4; }
__host__ __device__ constexpr int gemm_b_bytes(int n) { return n * GK * 2; }
__host__ __device__ constexpr int gemm_sub_bytes(bool pair, int n) { return kABytes + (pair ? gemm_b_bytes(n) / 2 : gemm_b_bytes(n)); }
__host__ __device__ constexpr int gemm_stage_bytes(bool pair, int n) { return gemm_sub(pair, n) * gemm_sub_bytes(pair, n); }
constexpr int kMnBox = 64 * GK * 2;                    // one MN-major box: 64 columns x 64 K-rows
constexpr int kOutBox = 128 * 64 * 2;                  // one staged output chunk: 128 rows x 64 columns, bf16
__host__ __device__ constexpr int gemm_smem(bool pair, int n)
{
    return gemm_stages(pair, n) * gemm_stage_bytes(pair, n) + 2 * kOutBox + 1024 /* alignment */ + 256 /* barriers */;
}
constexpr int kStages = kMaxStages;                    // barrier slots (the ring uses gemm_stages() of them)

enum { EPI_STORE = 0, EPI_SWIGLU_FWD = 1, EPI_SWIGLU_BWD = 2 };
enum { G_FULL = 0, G_EMPTY = kStages, G_ACCFULL = 2 * kStages, G_ACCEMPTY = 2 * kStages + 2, G_EPI = 2 * kStages + 4,
       G_IN = 2 * kStages + 5, G_RES = 2 * kStages + 6 /* two */, G_COUNT = 2 * kStages + 8 };
enum { GERR_EMPTY = 0x301, GERR_FULL = 0x302, GERR_ACCFULL = 0x303, GERR_ACCEMPTY = 0x304, GERR_EPI = 0x305, GERR_IN = 0x306, GERR_RES = 0x307 };

// Outputs leave through TMA stores (tensor maps C0..C3: STORE: C (and the second product's C); FWD gate: a, u, h;
// BWD gate: da, du, and the stored a, u as C2, C3, which its epilogue brings in by TMA loads).

__device__ __forceinline__ void unpack8(const uint4 &v, float *f)
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[i]));
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}
// 1 / (1 + exp(-a)) on the two fast special-function instructions (ex2.approx, rcp.approx).  (__frcp_rn, the
// correctly rounded reciprocal, is a multi-instruction sequence: with it the backward gate epilogue took 17,000
// cycles per tile instead of 6,800 and held its GEMM 25 % below the others.)
__device__ __forceinline__ float sigmoidf_fast(float a)
{
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(-1.4426950408889634f * a));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
    return r;
}

// Tile order: groups of `kGroup` tile rows, column-major inside a group, so that the CTAs running at the same time
// share a few A row blocks and a few B column blocks.  B is swept once per group: the launcher picks taller groups
// when B is too large to survive in L2 between sweeps (with groups of 8 a [8192 x 2048] x [16384 x 2048]^T product
// read its 67 MB of B eight times from DRAM: the outputs streaming through L2 evict it in between).
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int kGroup, int &tm, int &tn)
{
    const int per_group = kGroup * tiles_n;
    const int g = t / per_group, r = t - g * per_group;
    const int rows = min(kGroup, tiles_m - g * kGroup);
    tn = r / rows;
    tm = g * kGroup + (r - tn * rows);
}

template <bool kAMn, bool kBMn, int kEpi, bool kPair, int kN>
__global__ void __launch_bounds__(kGemmThreads, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap mapA0, const __grid_constant__ CUtensorMap mapB0,
               const __grid_constant__ CUtensorMap mapA1, const __grid_constant__ CUtensorMap mapB1,
               const __grid_constant__ CUtensorMap mapC0, const __grid_constant__ CUtensorMap mapC1,
               const __grid_constant__ CUtensorMap mapC2, const __grid_constant__ CUtensorMap mapC3, int M, int N, int K, int nparts, int nbatch, int a_blocked, int b_blocked, int has_res, int group_rows, unsigned int *status)
{
    static_assert(kN == 256 || (!kPair && (kN == 128 || (kN == 64 && kEpi != EPI_SWIGLU_FWD))), "tile widths");
    constexpr bool kDualN = kEpi == EPI_SWIGLU_FWD;         // B tile = kN / 2 rows of map B0 + kN / 2 rows of map B1
    constexpr int kTileN = kDualN ? kN / 2 : kN;             // output columns a tile covers
    constexpr int kBBytes = gemm_b_bytes(kN);
    // Epilogue warps: two per 32-lane group of TMEM; together they fill one 64-column output chunk at a time
    constexpr int kEpiWarps = 8;
    // kPair: the two CTAs of a cluster share tiles of 256 rows: UMMAs of M = 256 issued by the CTA of rank 0 read the
    // A rows and the B half staged in each CTA (this CTA: rows rank*128.. of the tile, B rows rank*128.. of its 256)
    // and write each CTA's accumulator; every CTA runs its own producer and epilogue.
    constexpr int kSt = gemm_stages(kPair, kN), kStageBytes = gemm_stage_bytes(kPair, kN), kTileM = kPair ? 2 * GM : GM;
    constexpr int kSub = gemm_sub(kPair, kN), kSubBytes = gemm_sub_bytes(kPair, kN);
    const uint32_t rank = kPair ? cluster_ctarank() : 0u;
    const int cta = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, ncta = kPair ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sout = sm + kSt * kStageBytes;               // two staged output chunks (128-byte swizzle)
    uint64_t *bars = reinterpret_cast<uint64_t *>(sout + 2 * kOutBox);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + G_COUNT);
    volatile uint32_t *abortp = tmem_slot + 1;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;

    const int tiles_m = (M + kTileM - 1) / kTileM, tiles_n = (N + kTileN - 1) / kTileN;
    // nbatch = 2: two independent products of one shape in one launch (A1 B1^T -> map C1 after A0 B0^T ->
    // map C0), so that their tiles share the waves of the persistent grid
    const int tiles_one = tiles_m * tiles_n, tiles = tiles_one * nbatch;
    const int nk = (K + GK * kSub - 1) / (GK * kSub), nk_total = nk * nparts;     // stages per operand pair
    const int tail = (K + GK - 1) / GK - (nk - 1) * kSub;                         // K blocks of a pair's last stage
    int armed = 0;       // loads this thread armed a barrier for: stages (the producer), staging buffers (the epilogue's leader)

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + G_FULL + i, 1);
            mbar_init(bars + G_EMPTY + i, 1);
        }
        mbar_init(bars + G_ACCFULL + 0, 1);
        mbar_init(bars + G_ACCFULL + 1, 1);
        mbar_init(bars + G_ACCEMPTY + 0, (kPair ? 2 : 1) * 32 * kEpiWarps);   // a pair: the epilogue threads of both CTAs
        mbar_init(bars + G_ACCEMPTY + 1, (kPair ? 2 : 1) * 32 * kEpiWarps);
        mbar_init(bars + G_EPI, 32 * kEpiWarps);
        mbar_init(bars + G_IN, 1);
        mbar_init(bars + G_RES + 0, 1);
        mbar_init(bars + G_RES + 1, 1);
        *abortp = 0;
        fence_mbar_init();
        prefetch_tensormap(&mapA0);      // (kernel parameters: nothing to wait for)
        prefetch_tensormap(&mapB0);
        prefetch_tensormap(&mapC0);
    }
    if (warp == 1) {
        if (kPair) {
            tmem_alloc_pair(tmem_slot, 512);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(tmem_slot, 2 * kN);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (kPair) cluster_sync_all();       // the other CTA's barriers are initialised before anything arrives on them
    tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    if (warp != 0) {
        grid_dependency_wait();
        grid_launch_dependents();
    }

    bool producer = false;
    if (warp == 0 && elect_one()) {
        producer = true;
        // ------------------------------------------------------------------ TMA producer
        int it = 0, tm = 0, tn = 0, second = 0;
        bool ok = true;
        auto place = [&](int t) {
            second = t >= tiles_one ? 1 : 0;
            tile_coords(t - second * tiles_one, tiles_m, tiles_n, group_rows, tm, tn);
        };
        // (the divisions of the first tile's place run in front of the wait: behind it they were 0.6 us of a small product's 5)
        if (cta < tiles) place(cta);
        grid_dependency_wait();
        grid_launch_dependents();
        for (int t = cta; ok && t < tiles; t += ncta) {
            if (t != cta) place(t);
            const int m0 = tm * kTileM + (int)rank * GM, n0 = tn * kTileN;
            const int nb0 = n0 + ((kPair && !kDualN) ? (int)rank * (kN / 2) : 0);    // first B row this CTA stages
            int part = 0, kstage = 0;
            for (int ks = 0; ks < nk_total; ++ks, ++it) {
                const int s = it % kSt;
                if (it >= kSt && !mbar_wait(bars + G_EMPTY + s, ((it / kSt) & 1) ^ 1, abortp, status, GERR_EMPTY)) { ok = false; break; }
                const int nsub = kstage == nk - 1 ? tail : kSub, kbase = kstage * kSub * GK;
                const CUtensorMap *ma = (part || second) ? &mapA1 : &mapA0;
                const CUtensorMap *mb = ((part || second) && !kDualN) ? &mapB1 : &mapB0;
                uint64_t *full = bars + G_FULL + s;
                // a pair: the copies of both CTAs complete on the barrier of rank 0, which its producer arms for both
                const uint32_t full_pair = kPair ? mapa_u32(smem_u32(full), 0) : 0u;
                if (!kPair || rank == 0) {
                    mbar_arrive_expect_tx(full, (uint32_t)((kPair ? 2 : 1) * nsub * kSubBytes));
                    ++armed;
                }
                auto load = [&](void *dst, const CUtensorMap *m, int x, int y, int z) {
                    if (kPair) tma_load_3d_pair(dst, m, full_pair, x, y, z);
                    else tma_load_3d(dst, m, full, x, y, z);
                };
#pragma unroll
              for (int sub = 0; sub < kSub; ++sub) {          // (what lies past K in a block is filled with zeros by the copy)
                if (sub >= nsub) break;
                const int k0 = kbase + sub * GK;
                uint8_t *sa = sm + s * kStageBytes + sub * kSubBytes, *sb = sa + kABytes;
                if (kAMn) {
                    if (a_blocked) {                          // one copy: (64 columns, K rows, column blocks)
                        load(sa, ma, 0, k0, m0 / 64);
                    } else {
                        load(sa, ma, m0, k0, 0);
                        load(sa + kMnBox, ma, m0 + 64, k0, 0);
                    }
                } else {
                    load(sa, ma, k0, m0, 0);
                }
                if (kBMn) {
                    if (b_blocked) {
                        load(sb, mb, 0, k0, nb0 / 64);
                    } else {
#pragma unroll
                        for (int b = 0; b < (kPair ? 2 : kN / 64); ++b) load(sb + b * kMnBox, mb, nb0 + 64 * b, k0, 0);
                    }
                } else if (kDualN) {
                    if (kPair) {                              // rank 0 stages the W1 rows, rank 1 the W3 rows
                        load(sb, rank ? &mapB1 : &mapB0, k0, n0, 0);
                    } else {
                        load(sb, &mapB0, k0, n0, 0);
                        load(sb + kBBytes / 2, &mapB1, k0, n0, 0);
                    }
                } else {
                    load(sb, mb, k0, nb0, 0);
                }
              }
                if (++kstage == nk) { kstage = 0; ++part; }
            }
        }
    } else if (warp == 1 && rank == 0 && elect_one()) {
        // ------------------------------------------------------------------- UMMA issuer
        constexpr uint32_t idesc = idesc_bf16_f32(kTileM, kN, kAMn ? 1 : 0, kBMn ? 1 : 0);
        const uint64_t km_proto = smem_desc_sw128(0, 16, 1024), mn_proto = smem_desc_sw128(0, kMnBox, 1024);
        const uint32_t a_hi = (uint32_t)((kAMn ? mn_proto : km_proto) >> 32), b_hi = (uint32_t)((kBMn ? mn_proto : km_proto) >> 32);
        const uint32_t a_lo0 = (uint32_t)(kAMn ? mn_proto : km_proto), b_lo0 = (uint32_t)(kBMn ? mn_proto : km_proto);
        constexpr uint32_t a_step = (kAMn ? 2048 : 32) >> 4, b_step = (kBMn ? 2048 : 32) >> 4;   // per 16 K-elements
        int it = 0, ti = 0;
        bool ok = true;
        for (int t = cta; ok && t < tiles; t += ncta, ++ti) {
            const int buf = ti & 1;
            if (!mbar_wait(bars + G_ACCEMPTY + buf, ((ti >> 1) & 1) ^ 1, abortp, status, GERR_ACCEMPTY)) break;
            tc_fence_after();
            const uint32_t acc = tbase + (uint32_t)(buf * kN);
            int kstage = 0;
            for (int ks = 0; ks < nk_total; ++ks, ++it) {
                const int s = it % kSt;
                const bool last = ++kstage == nk;
                if (last) kstage = 0;
                if (!mbar_wait(bars + G_FULL + s, (it / kSt) & 1, abortp, status, GERR_FULL)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a_lo = a_lo0 + ((smem_u32(sm + s * kStageBytes) >> 4) & 0x3FFFu);
                const uint32_t b_lo = b_lo0 + ((smem_u32(sm + s * kStageBytes + kABytes) >> 4) & 0x3FFFu);
#pragma unroll
                for (int sub = 0; sub < kSub; ++sub) {
                    if (sub > 0 && last && sub >= tail) break;
                    const uint32_t a_s = a_lo + (uint32_t)(sub * (kSubBytes >> 4)), b_s = b_lo + (uint32_t)(sub * (kSubBytes >> 4));
                    if (ks == 0 && sub == 0) {
                        if (kPair) umma_ss2_pair<false>(acc, a_s, a_hi, b_s, b_hi, idesc);
                        else       umma_ss2<false>(acc, a_s, a_hi, b_s, b_hi, idesc);
                    } else {
                        if (kPair) umma_ss2_pair<true>(acc, a_s, a_hi, b_s, b_hi, idesc);
                        else       umma_ss2<true>(acc, a_s, a_hi, b_s, b_hi, idesc);
                    }
#pragma unroll
                    for (int q = 1; q < GK / 16; ++q) {
                        if (kPair) umma_ss2_pair<true>(acc, a_s + q * a_step, a_hi, b_s + q * b_step, b_hi, idesc);
                        else       umma_ss2<true>(acc, a_s + q * a_step, a_hi, b_s + q * b_step, b_hi, idesc);
                    }
                }
                // the stage is free (in both CTAs of a pair) once these UMMAs have read it
                if (kPair) umma_commit_pair(bars + G_EMPTY + s);
                else       umma_commit(bars + G_EMPTY + s);
            }
            if (ok) {
                if (kPair) umma_commit_pair(bars + G_ACCFULL + buf);
                else umma_commit(bars + G_ACCFULL + buf);
            }
        }
    } else if (warp >= 2 && warp < 2 + kEpiWarps) {
        // ---------------------------------------------------------------------- epilogue
        // A thread owns one row of the tile (its TMEM lane) and 32 of the 64 columns of the current chunk.  Results go
        // to a shared-memory chunk in the 128-byte-swizzle layout and leave as one TMA store per chunk (whole 128-byte
        // lines; rows and columns past the array are clipped by the tensor map): row-owner 16-byte stores to global
        // memory cost one L2 request each, and at 6000 requests per tile they slowed the operand loads of the next tile.
        const int lane_row = 32 * (warp % 4) + lane;               // TMEM lane = row of the tile
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        const int half = (warp - 2) / 4;                           // which 32 columns of a 64-column chunk
        const bool leader = tid == 64;
        uint32_t epi_phase = 0, chunk_q = 0, in_q = 0;
        bool ok = true;
        // hands an accumulator back to the issuer (a pair: to the issuer in the CTA of rank 0)
        const uint32_t accempty_pair = kPair ? mapa_u32(smem_u32(bars + G_ACCEMPTY), 0) : 0u;
        auto acc_release = [&](int b) {
            tc_fence_before();
            if (kPair) mbar_arrive_cluster(accempty_pair + 8u * (uint32_t)b);
            else mbar_arrive(bars + G_ACCEMPTY + b);
        };
        // all epilogue threads meet (bounded wait)
        auto epi_sync = [&]() -> bool {
            mbar_arrive(bars + G_EPI);
            const bool r = mbar_wait(bars + G_EPI, epi_phase & 1, abortp, status, GERR_EPI);
            ++epi_phase;
            return r;
        };
        // the 32 values of this thread (as 16 bf16 pairs) -> staged chunk -> TMA store at (row0, col0)
        auto stage_store = [&](const CUtensorMap *map, const uint32_t (&v)[16], int col0, int row0) -> bool {
            uint8_t *buf = sout + (chunk_q & 1) * kOutBox;
            if (leader) bulk_wait_read<1>();                       // the store issued two chunks ago has left this buffer
            if (!epi_sync()) return false;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<uint4 *>(buf + lane_row * 128 + (((half * 4 + j) ^ (lane_row & 7)) << 4)) =
                    make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            fence_proxy_async_smem();
            if (!epi_sync()) return false;
            if (leader) {
                if (row0 < M) tma_store_3d(map, buf, col0, row0, 0);   // (a pair's second half can lie past the last row)
                bulk_commit();
            }
            ++chunk_q;
            return true;
        };
        // the same with a residual: the chunk of R comes into the staging buffer by TMA (requested a chunk ahead, a tile's first
        // before its main loop has finished), every thread adds its 32 values in place, and the buffer leaves by a TMA store
        auto load_res = [&](uint32_t q, int col0, int row0) {          // (leader; the buffer's last store has been read)
            mbar_arrive_expect_tx(bars + G_RES + (q & 1), kOutBox);
            ++armed;
            tma_load_3d(sout + (q & 1) * kOutBox, &mapC2, bars + G_RES + (q & 1), col0, row0, 0);
        };
        auto stage_store_res = [&](const CUtensorMap *map, const uint32_t (&racc)[32], int col0, int row0, bool more) -> bool {
            const uint32_t b = chunk_q & 1;
            uint8_t *buf = sout + b * kOutBox;
            if (leader && more) {
                bulk_wait_read<0>();                                   // the store of the last chunk has left the other buffer
                load_res(chunk_q + 1, col0 + 64, row0);
            }
            if (!mbar_wait(bars + G_RES + b, (chunk_q >> 1) & 1, abortp, status, GERR_RES)) return false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint4 *pr = reinterpret_cast<uint4 *>(buf + lane_row * 128 + (((half * 4 + j) ^ (lane_row & 7)) << 4));
                float r8[8];
                unpack8(*pr, r8);
#pragma unroll
                for (int i = 0; i < 8; ++i) r8[i] += __uint_as_float(racc[8 * j + i]);
                *pr = make_uint4(pack_bf16(r8[0], r8[1]), pack_bf16(r8[2], r8[3]), pack_bf16(r8[4], r8[5]), pack_bf16(r8[6], r8[7]));
            }
            fence_proxy_async_smem();
            if (!epi_sync()) return false;
            if (leader) {
                if (row0 < M) tma_store_3d(map, buf, col0, row0, 0);   // (a pair's second half can lie past the last row)
                bulk_commit();
            }
            ++chunk_q;
            return true;
        };
        int ti = 0;
        for (int t = cta; ok && t < tiles; t += ncta, ++ti) {
            int tm, tn;
            const int second = t >= tiles_one ? 1 : 0;
            tile_coords(t - second * tiles_one, tiles_m, tiles_n, group_rows, tm, tn);
            const int buf = ti & 1;
            const int m0 = tm * kTileM + (int)rank * GM, n0 = tn * kTileN;
            if (kEpi == EPI_STORE && has_res && leader) {     // the tile's residual, while its main loop runs: the first chunk, the rest into L2
                bulk_wait_read<1>();
                load_res(chunk_q, n0, m0);
#pragma unroll
                for (int c0 = 64; c0 < kN; c0 += 64) tma_prefetch_3d(&mapC2, n0 + c0, m0, 0);
            }
            auto load_gate = [&](int c0) {                    // (leader)
                bulk_wait_read<0>();                          // the previous chunk's stores have left both buffers
                mbar_arrive_expect_tx(bars + G_IN, 2 * kOutBox);
                ++armed;
                tma_load_3d(sout, &mapC2, bars + G_IN, n0 + c0, m0, 0);
                tma_load_3d(sout + kOutBox, &mapC3, bars + G_IN, n0 + c0, m0, 0);
            };
            if (kEpi == EPI_SWIGLU_BWD && leader) {       // the tile's stored a, u, while its main loop runs: likewise
                load_gate(0);
#pragma unroll
                for (int c0 = 64; c0 < kN; c0 += 64) {
                    tma_prefetch_3d(&mapC2, n0 + c0, m0, 0);
                    tma_prefetch_3d(&mapC3, n0 + c0, m0, 0);
                }
            }
            if (!mbar_wait(bars + G_ACCFULL + buf, (ti >> 1) & 1, abortp, status, GERR_ACCFULL)) break;
            tc_fence_after();
            const uint32_t acc = lane_addr + (uint32_t)(buf * kN);
            const int cols = min(kTileN, (N - n0 + 63) / 64 * 64);      // chunks wholly past the last column are not worked on
            if (kEpi == EPI_SWIGLU_FWD) {
#pragma unroll 1
                for (int c0 = 0; ok && c0 < cols; c0 += 64) {
                    const int c = c0 + 32 * half;
                    uint32_t ra[32], ru[32];
                    tmem_ld(acc + c, ra);
                    tmem_ld(acc + kN / 2 + c, ru);
                    tc_wait_ld();
                    if (c0 == cols - 64) {                // last read of this accumulator: hand it back early
                        acc_release(buf);
                    }
                    uint32_t pa[16], pu[16], ph[16];
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float a0 = __uint_as_float(ra[e]), a1 = __uint_as_float(ra[e + 1]);
                        const float u0 = __uint_as_float(ru[e]), u1 = __uint_as_float(ru[e + 1]);
                        pa[e / 2] = pack_bf16(a0, a1);
                        pu[e / 2] = pack_bf16(u0, u1);
                        ph[e / 2] = pack_bf16(a0 * sigmoidf_fast(a0) * u0, a1 * sigmoidf_fast(a1) * u1);
                    }
                    ok = stage_store(&mapC0, pa, n0 + c0, m0) && stage_store(&mapC1, pu, n0 + c0, m0) &&
                         stage_store(&mapC2, ph, n0 + c0, m0);
                }
            } else if (kEpi == EPI_STORE) {
#pragma unroll 1
                for (int c0 = 0; ok && c0 < cols; c0 += 64) {
                    uint32_t r[32];
                    tmem_ld(acc + c0 + 32 * half, r);
                    tc_wait_ld();
                    if (c0 == cols - 64) {                // last read of this accumulator: hand it back early
                        acc_release(buf);
                    }
                    if (has_res) {
                        ok = stage_store_res(&mapC0, r, n0 + c0, m0, c0 + 64 < cols);
                    } else {
                        uint32_t pc[16];
#pragma unroll
                        for (int e = 0; e < 32; e += 2) pc[e / 2] = pack_bf16(__uint_as_float(r[e]), __uint_as_float(r[e + 1]));
                        ok = stage_store(second ? &mapC1 : &mapC0, pc, n0 + c0, m0);
                    }
                }
            } else {
                // Backward gate: per 64-column chunk the stored a and u come into the two staging buffers by TMA, every
                // thread turns its 32 + 32 values into da, du in place, and the buffers leave by TMA stores.
#pragma unroll 1
                for (int c0 = 0; ok && c0 < cols; c0 += 64, ++in_q) {
                    if (leader && c0 > 0) load_gate(c0);
                    uint32_t r[32];
                    tmem_ld(acc + c0 + 32 * half, r);
                    tc_wait_ld();
                    if (c0 == cols - 64) {
                        acc_release(buf);
                    }
                    if (!mbar_wait(bars + G_IN, in_q & 1, abortp, status, GERR_IN)) { ok = false; break; }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint32_t off = lane_row * 128 + (((half * 4 + q) ^ (lane_row & 7)) << 4);
                        uint4 *pa = reinterpret_cast<uint4 *>(sout + off), *pu = reinterpret_cast<uint4 *>(sout + kOutBox + off);
                        float fa[8], fu[8], da[8], du[8];
                        unpack8(*pa, fa);
                        unpack8(*pu, fu);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float f = __uint_as_float(r[8 * q + i]);
                            const float sg = sigmoidf_fast(fa[i]);
                            da[i] = f * fu[i] * sg * (1.f + fa[i] * (1.f - sg));
                            du[i] = f * fa[i] * sg;
                        }
                        *pa = make_uint4(pack_bf16(da[0], da[1]), pack_bf16(da[2], da[3]), pack_bf16(da[4], da[5]), pack_bf16(da[6], da[7]));
                        *pu = make_uint4(pack_bf16(du[0], du[1]), pack_bf16(du[2], du[3]), pack_bf16(du[4], du[5]), pack_bf16(du[6], du[7]));
                    }
                    fence_proxy_async_smem();
                    if (!epi_sync()) { ok = false; break; }
                    if (leader) {
                        if (m0 < M) {
                            tma_store_3d(&mapC0, sout, n0 + c0, m0, 0);
                            tma_store_3d(&mapC1, sout + kOutBox, n0 + c0, m0, 0);
                        }
                        bulk_commit();
                    }
                }
            }
        }
        if (leader) bulk_wait_read<0>();          // every store has read its buffer before the CTA gives up its shared memory
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (*abortp) {      // a wait expired somewhere: copies still on their way land before the CTA leaves (bounded)
        if (producer)
            for (int s = 0; s < kSt; ++s) mbar_drain_one(bars + G_FULL + s, armed > s ? (armed - s + kSt - 1) / kSt : 0);
        if (tid == 64 && kEpi == EPI_STORE)
            for (int b = 0; b < 2; ++b) mbar_drain_one(bars + G_RES + b, armed > b ? (armed - b + 1) / 2 : 0);
        if (tid == 64 && kEpi == EPI_SWIGLU_BWD) mbar_drain_one(bars + G_IN, armed);
    }
    if (kPair) {
        // neither CTA leaves, or frees its TMEM, while the other may still read its shared memory, write its
        // accumulator or arrive on its barriers
        cluster_sync_all();
        if (warp == 1) tmem_dealloc_pair(tbase, 512);
    } else if (warp == 1) {
        tmem_dealloc(tbase, 2 * kN);
    }
}

// Several products C = A B^T (one or two operand pairs, any storage order) as ONE launch of single CTAs: what the backward of a small block needs
// next to each other.  A launch costs such a product 3 us beside its K blocks and leaves most SMs idle; here the tiles of all of them are
// walked by one grid.  Same roles, ring and epilogue as tc_gemm_kernel, the operand layouts taken from the job at run time.
constexpr int kMaxJobs = 4;
struct GroupJob {
    CUtensorMap A[2], B[2], C;
    int M, N, K, nparts, a_mn, b_mn, a_blocked, b_blocked, tile0 /* number of the job's first tile */;
};
struct GroupJobs {
    GroupJob j[kMaxJobs];
    int count, tiles;
};

template <int kN>
__global__ void __launch_bounds__(kGemmThreads, 1)
tc_gemm_group_kernel(const __grid_constant__ GroupJobs jobs, unsigned int *status)
{
    constexpr int kEpiWarps = 8;
    constexpr int kSt = gemm_stages(false, kN), kStageBytes = gemm_stage_bytes(false, kN), kSub = gemm_sub(false, kN), kSubBytes = gemm_sub_bytes(false, kN);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sout = sm + kSt * kStageBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sout + 2 * kOutBox);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + G_COUNT);
    volatile uint32_t *abortp = tmem_slot + 1;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + G_FULL + i, 1);
            mbar_init(bars + G_EMPTY + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bars + G_ACCFULL + i, 1);
            mbar_init(bars + G_ACCEMPTY + i, 32 * kEpiWarps);
        }
        mbar_init(bars + G_EPI, 32 * kEpiWarps);
        *abortp = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 2 * kN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    const int cta = (int)blockIdx.x, ncta = (int)gridDim.x, tiles = jobs.tiles;
    // the job of a tile (tiles are walked in ascending order) and the tile's place in it
    auto job_of = [&](int t, int &jx, int &m0, int &n0) {
        while (jx + 1 < jobs.count && t >= jobs.j[jx + 1].tile0) ++jx;
        const GroupJob &J = jobs.j[jx];
        int tm, tn;
        tile_coords(t - J.tile0, (J.M + GM - 1) / GM, (J.N + kN - 1) / kN, 8, tm, tn);
        m0 = tm * GM;
        n0 = tn * kN;
    };
    auto stages_of = [&](const GroupJob &J) { return (J.K + GK * kSub - 1) / (GK * kSub); };      // per operand pair

    auto tail_of = [&](const GroupJob &J) { return (J.K + GK - 1) / GK - (stages_of(J) - 1) * kSub; };   // K blocks of a pair's last stage
    int armed = 0;       // stages the producer armed
    if (warp != 0) {
        grid_dependency_wait();
        grid_launch_dependents();
    }

    bool producer = false;
    if (warp == 0 && elect_one()) {
        producer = true;
        // ------------------------------------------------------------------ TMA producer
        int it = 0, jx = 0, m0 = 0, n0 = 0;
        bool ok = true;
        if (cta < tiles) {                // in front of the wait: where the first tile is, and its maps
            job_of(cta, jx, m0, n0);
            prefetch_tensormap(&jobs.j[jx].A[0]);
            prefetch_tensormap(&jobs.j[jx].B[0]);
            prefetch_tensormap(&jobs.j[jx].C);
        }
        grid_dependency_wait();
        grid_launch_dependents();
        for (int t = cta; ok && t < tiles; t += ncta) {
            if (t != cta) job_of(t, jx, m0, n0);
            const GroupJob &J = jobs.j[jx];
            const int nk = stages_of(J), tail = tail_of(J);
            int part = 0, kstage = 0;
            for (int ks = 0; ks < nk * J.nparts; ++ks, ++it) {
                const int s = it % kSt;
                if (it >= kSt && !mbar_wait(bars + G_EMPTY + s, ((it / kSt) & 1) ^ 1, abortp, status, GERR_EMPTY)) { ok = false; break; }
                uint64_t *full = bars + G_FULL + s;
                const int nsub = kstage == nk - 1 ? tail : kSub, kbase = kstage * kSub * GK;
                mbar_arrive_expect_tx(full, (uint32_t)(nsub * kSubBytes));
                ++armed;
                const CUtensorMap *ma = &J.A[part], *mb = &J.B[part];
#pragma unroll
                for (int sub = 0; sub < kSub; ++sub) {
                    if (sub >= nsub) break;
                    const int k0 = kbase + sub * GK;
                    uint8_t *sa = sm + s * kStageBytes + sub * kSubBytes, *sb = sa + kABytes;
                    if (!J.a_mn) {
                        tma_load_3d(sa, ma, full, k0, m0, 0);
                    } else if (J.a_blocked) {
                        tma_load_3d(sa, ma, full, 0, k0, m0 / 64);
                    } else {
                        tma_load_3d(sa, ma, full, m0, k0, 0);
                        tma_load_3d(sa + kMnBox, ma, full, m0 + 64, k0, 0);
                    }
                    if (!J.b_mn) {
                        tma_load_3d(sb, mb, full, k0, n0, 0);
                    } else if (J.b_blocked) {
                        tma_load_3d(sb, mb, full, 0, k0, n0 / 64);
                    } else {
#pragma unroll
                        for (int b = 0; b < kN / 64; ++b) tma_load_3d(sb + b * kMnBox, mb, full, n0 + 64 * b, k0, 0);
                    }
                }
                if (++kstage == nk) { kstage = 0; ++part; }
            }
        }
    } else if (warp == 1 && elect_one()) {
        // ------------------------------------------------------------------- UMMA issuer
        const uint64_t km_proto = smem_desc_sw128(0, 16, 1024), mn_proto = smem_desc_sw128(0, kMnBox, 1024);
        int it = 0, ti = 0, jx = 0;
        bool ok = true;
        for (int t = cta; ok && t < tiles; t += ncta, ++ti) {
            int m0, n0;
            job_of(t, jx, m0, n0);
            const GroupJob &J = jobs.j[jx];
            const uint64_t ap = J.a_mn ? mn_proto : km_proto, bp = J.b_mn ? mn_proto : km_proto;
            const uint32_t a_hi = (uint32_t)(ap >> 32), b_hi = (uint32_t)(bp >> 32), a_lo0 = (uint32_t)ap, b_lo0 = (uint32_t)bp;
            const uint32_t a_step = (J.a_mn ? 2048 : 32) >> 4, b_step = (J.b_mn ? 2048 : 32) >> 4, idesc = idesc_bf16_f32(GM, kN, J.a_mn, J.b_mn);
            const int nk = stages_of(J), nk_total = nk * J.nparts, tail = tail_of(J), buf = ti & 1;
            if (!mbar_wait(bars + G_ACCEMPTY + buf, ((ti >> 1) & 1) ^ 1, abortp, status, GERR_ACCEMPTY)) break;
            tc_fence_after();
            const uint32_t acc = tbase + (uint32_t)(buf * kN);
            int kstage = 0;
            for (int ks = 0; ks < nk_total; ++ks, ++it) {
                const int s = it % kSt;
                const bool last = ++kstage == nk;
                if (last) kstage = 0;
                if (!mbar_wait(bars + G_FULL + s, (it / kSt) & 1, abortp, status, GERR_FULL)) { ok = false; break; }
                tc_fence_after();
                const uint32_t a_lo = a_lo0 + ((smem_u32(sm + s * kStageBytes) >> 4) & 0x3FFFu);
                const uint32_t b_lo = b_lo0 + ((smem_u32(sm + s * kStageBytes + kABytes) >> 4) & 0x3FFFu);
#pragma unroll
                for (int sub = 0; sub < kSub; ++sub) {
                    if (sub > 0 && last && sub >= tail) break;
                    const uint32_t a_s = a_lo + (uint32_t)(sub * (kSubBytes >> 4)), b_s = b_lo + (uint32_t)(sub * (kSubBytes >> 4));
                    if (ks == 0 && sub == 0) umma_ss2<false>(acc, a_s, a_hi, b_s, b_hi, idesc);
                    else                     umma_ss2<true>(acc, a_s, a_hi, b_s, b_hi, idesc);
#pragma unroll
                    for (int q = 1; q < GK / 16; ++q) umma_ss2<true>(acc, a_s + q * a_step, a_hi, b_s + q * b_step, b_hi, idesc);
                }
                umma_commit(bars + G_EMPTY + s);
            }
            if (ok) umma_commit(bars + G_ACCFULL + buf);
        }
    } else if (warp >= 2 && warp < 2 + kEpiWarps) {
        // ---------------------------------------------------------------------- epilogue (as in tc_gemm_kernel, EPI_STORE)
        const int lane_row = 32 * (warp % 4) + lane, half = (warp - 2) / 4;
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        const bool leader = tid == 64;
        uint32_t epi_phase = 0, chunk_q = 0;
        auto epi_sync = [&]() -> bool {
            mbar_arrive(bars + G_EPI);
            const bool r = mbar_wait(bars + G_EPI, epi_phase & 1, abortp, status, GERR_EPI);
            ++epi_phase;
            return r;
        };
        bool ok = true;
        int ti = 0, jx = 0;
        for (int t = cta; ok && t < tiles; t += ncta, ++ti) {
            int m0, n0;
            job_of(t, jx, m0, n0);
            const GroupJob &J = jobs.j[jx];
            const int buf = ti & 1, cols = min(kN, (J.N - n0 + 63) / 64 * 64);
            if (!mbar_wait(bars + G_ACCFULL + buf, (ti >> 1) & 1, abortp, status, GERR_ACCFULL)) break;
            tc_fence_after();
            const uint32_t acc = lane_addr + (uint32_t)(buf * kN);
#pragma unroll 1
            for (int c0 = 0; ok && c0 < cols; c0 += 64, ++chunk_q) {
                uint32_t r[32];
                tmem_ld(acc + c0 + 32 * half, r);
                tc_wait_ld();
                if (c0 == cols - 64) {                    // last read of this accumulator: hand it back early
                    tc_fence_before();
                    mbar_arrive(bars + G_ACCEMPTY + buf);
                }
                uint8_t *out = sout + (chunk_q & 1) * kOutBox;
                if (leader) bulk_wait_read<1>();          // the store issued two chunks ago has left this buffer
                if (!epi_sync()) { ok = false; break; }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) w[e] = pack_bf16(__uint_as_float(r[8 * j + 2 * e]), __uint_as_float(r[8 * j + 2 * e + 1]));
                    *reinterpret_cast<uint4 *>(out + lane_row * 128 + (((half * 4 + j) ^ (lane_row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                fence_proxy_async_smem();
                if (!epi_sync()) { ok = false; break; }
                if (leader) {
                    tma_store_3d(&J.C, out, n0 + c0, m0, 0);
                    bulk_commit();
                }
            }
        }
        if (leader) bulk_wait_read<0>();
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    if (*abortp && producer)      // (as in tc_gemm_kernel)
        for (int s = 0; s < kSt; ++s) mbar_drain_one(bars + G_FULL + s, armed > s ? (armed - s + kSt - 1) / kSt : 0);
    if (warp == 1) tmem_dealloc(tbase, 2 * kN);
}

struct Operand {
    const void *p;
    int rows, cols;          // the array as stored: [rows, cols] row-major
};

// K-major: stored [MN, K], box of `box_rows` rows x 64 K-elements.  MN-major: stored [K, MN]: one blocked box of
// box_rows / 64 column blocks x 64 K-rows when `blocked`, else boxes of 64 x 64.
bool operand_map(CUtensorMap *m, const Operand &o, bool mn_major, int box_rows, bool blocked = false)
{
    if (mn_major && blocked)
        return make_tensor_map_blocked(m, o.p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)o.rows, (uint64_t)o.cols, 64,
                                       (uint32_t)box_rows / 64);
    return make_tensor_map_3d(m, o.p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 1, (uint64_t)o.rows, (uint64_t)o.cols,
                              mn_major ? 64 : (uint32_t)box_rows, 64);
}

// Clusters of two CTAs of `kernel` that can be resident at once (cudaOccupancyMaxActiveClusters; cached per kernel
// and device); half the SM count if the query fails.
template <typename K>
int max_active_pairs(K kernel, int smem)
{
    constexpr int kMaxDev = 64;
    static int cache[kMaxDev] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return device_info().sms / 2;
    if (cache[dev] > 0) return cache[dev];
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)device_info().sms / 2 * 2);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n <= 0) {
        (void)cudaGetLastError();
        n = device_info().sms / 2;
    }
    if (n > device_info().sms / 2) n = device_info().sms / 2;
    return cache[dev] = n;
}

template <bool kAMn, bool kBMn, int kEpi, bool kPair, int kN>
// C0..C2: output arrays (row length ldc); unused ones may repeat C0.
cudaError_t launch_gemm_as(const Operand &A0, const Operand &B0, const Operand *A1, const Operand *B1, void *C0, void *C1,
                        const void *C2, const void *C3, int c_rows, int ldc, int M, int N, int K, cudaStream_t st,
                        int nbatch = 1, bool has_res = false)
{
    constexpr bool kDualN = kEpi == EPI_SWIGLU_FWD;
    CUtensorMap ma0, mb0, ma1, mb1;
    const int b_rows = (kDualN || kPair) ? kN / 2 : kN;     // B rows one CTA stages per copy
    // MN-major operands whose width is a multiple of 64 come in by one blocked copy per stage (try the encode; if the
    // driver refuses the map, or a width has a tail, use one copy per 64-column block)
    const Operand &a1 = A1 ? *A1 : A0, &b1 = B1 ? *B1 : B0;
    // (maps that repeat another one are copied, not looked up again: a launch of a small product is host time)
    bool a_blocked = kAMn && A0.cols % 64 == 0 && a1.cols % 64 == 0;
    bool b_blocked = kBMn && B0.cols % 64 == 0 && b1.cols % 64 == 0;
    auto pair_of = [](CUtensorMap &m0, CUtensorMap &m1, const Operand &o0, const Operand *o1, bool mn, int rows, bool blocked) {
        if (!operand_map(&m0, o0, mn, rows, blocked)) return false;
        if (o1) return operand_map(&m1, *o1, mn, rows, blocked);
        m1 = m0;
        return true;
    };
    if (a_blocked && !pair_of(ma0, ma1, A0, A1, true, GM, true)) a_blocked = false;
    if (b_blocked && !pair_of(mb0, mb1, B0, B1, true, b_rows, true)) b_blocked = false;
    if (!a_blocked && !pair_of(ma0, ma1, A0, A1, kAMn, GM, false)) return cudaErrorInvalidValue;
    if (!b_blocked && !pair_of(mb0, mb1, B0, B1, kBMn, b_rows, false)) return cudaErrorInvalidValue;
    CUtensorMap mc[4];
    const void *cs[4] = {C0, C1, C2, C3};
    for (int i = 0; i < 4; ++i) {     // [c_rows, ldc] bf16, boxes of 128 rows x 64 columns, 128-byte swizzle
        if (i > 0 && !cs[i]) mc[i] = mc[0];
        else if (!make_tensor_map_3d(&mc[i], cs[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 1, (uint64_t)c_rows, (uint64_t)ldc, 128, 64))
            return cudaErrorInvalidValue;
    }
    auto kernel = tc_gemm_kernel<kAMn, kBMn, kEpi, kPair, kN>;
    constexpr int kSmem = gemm_smem(kPair, kN), kTileN = kDualN ? kN / 2 : kN, kTileM = kPair ? 2 * GM : GM;
    cudaError_t e = allow_smem<tc_gemm_kernel<kAMn, kBMn, kEpi, kPair, kN>>(kSmem);
    if (e != cudaSuccess) return e;
    const int tiles = ((M + kTileM - 1) / kTileM) * ((N + kTileN - 1) / kTileN) * nbatch;
    const int nparts = (A1 && !kDualN && nbatch == 1) ? 2 : 1;
    // Groups of 8 tile rows, unless B is too large to stay in L2 between groups (above 48 MB): then groups as tall as
    // keeps their A rows within 32 MB, so that B is swept fewer times (measured: taller groups cost the products with
    // a small B 2-5 %, and save the forward gate GEMM, whose B is W1 and W3 together, 3 % and 70 % of its DRAM reads)
    const long long b_bytes = (long long)B0.rows * B0.cols * 2 * ((kDualN || nparts == 2) ? 2 : 1);
    long long group_rows = 8;
    if (b_bytes > (48LL << 20)) {
        group_rows = (32LL << 20) / ((long long)GM * K * nparts * 2);
        group_rows = group_rows < 8 ? 8 : group_rows > 64 ? 64 : group_rows;
    }
    if (kPair) group_rows = group_rows / 2 < 2 ? 2 : group_rows / 2;     // tile rows of 256
    LaunchScope scope(MOA_KERNEL_OTHER, st);
    // persistent grid: one CTA per SM, or as many clusters of two as the device can hold at once
    const int sms = device_info().sms, pairs = kPair ? max_active_pairs(kernel, kSmem) : 0;
    const int ctas = kPair ? 2 * (tiles < pairs ? tiles : pairs) : (tiles < sms ? tiles : sms);
    return launch_cluster(kernel, kPair ? 2u : 1u, dim3((unsigned)ctas), dim3(kGemmThreads), (size_t)kSmem, st, ma0, mb0, ma1, mb1, mc[0],
                          mc[1], mc[2], mc[3], M, N, K, nparts, nbatch, a_blocked ? 1 : 0, b_blocked ? 1 : 0, has_res ? 1 : 0,
                          (int)group_rows, device_status_ptr());
}

// Pairs of CTAs (tiles of 256 rows, half the B traffic per SM) by default; single CTAs where pairs would need more
// waves.  MOA_GEMM_PAIR (read once): 0 never pairs, 2 always.
int gemm_pair_mode()
{
    static int mode = -1;
    if (mode < 0) {
        const char *e = getenv("MOA_GEMM_PAIR");
        mode = e ? atoi(e) : 1;
    }
    return mode;
}
template <bool kAMn, bool kBMn, int kEpi>
cudaError_t launch_gemm(const Operand &A0, const Operand &B0, const Operand *A1, const Operand *B1, void *C0, void *C1,
                        const void *C2, const void *C3, int c_rows, int ldc, int M, int N, int K, cudaStream_t st,
                        int nbatch = 1, bool has_res = false)
{
    constexpr bool kDualN = kEpi == EPI_SWIGLU_FWD;
    const GemmTile tile = gemm_tile(M, N, K, kAMn, kBMn, kEpi == EPI_STORE, kDualN, A1 && !kDualN && nbatch == 1, nbatch, device_info().sms, gemm_pair_mode());
    if (tile.pair) return launch_gemm_as<kAMn, kBMn, kEpi, true, 256>(A0, B0, A1, B1, C0, C1, C2, C3, c_rows, ldc, M, N, K, st, nbatch, has_res);
    if constexpr (!kDualN)
        if (tile.columns == 64) return launch_gemm_as<kAMn, kBMn, kEpi, false, 64>(A0, B0, A1, B1, C0, C1, C2, C3, c_rows, ldc, M, N, K, st, nbatch, has_res);
    if (tile.columns == 128) return launch_gemm_as<kAMn, kBMn, kEpi, false, 128>(A0, B0, A1, B1, C0, C1, C2, C3, c_rows, ldc, M, N, K, st, nbatch, has_res);
    return launch_gemm_as<kAMn, kBMn, kEpi, false, 256>(A0, B0, A1, B1, C0, C1, C2, C3, c_rows, ldc, M, N, K, st, nbatch, has_res);
}

// One product of a group
struct Product {
    Operand A0, B0;
    const Operand *A1, *B1;      // second operand pair (null: none)
    void *C;                     // [M, N]
    int M, N, K, a_mn, b_mn;
    long long tiles(int n) const { return (long long)((M + GM - 1) / GM) * ((N + n - 1) / n); }
    bool writes_into(const void *p, long long rows, long long cols) const { return arrays_meet(C, (size_t)M * N * 2, p, (size_t)(rows * cols) * 2); }
    bool disturbs(const Product &o) const       // writes what `o` reads or writes
    {
        for (const Operand *r : {&o.A0, &o.B0, o.A1, o.B1})
            if (r && writes_into(r->p, r->rows, r->cols)) return true;
        return writes_into(o.C, o.M, o.N);
    }
};

template <int kN>
cudaError_t launch_group_n(const Product *p, int count, cudaStream_t st)
{
    GroupJobs g;
    int tiles = 0;
    for (int i = 0; i < count; ++i) {
        GroupJob &j = g.j[i];
        const Operand &a1 = p[i].A1 ? *p[i].A1 : p[i].A0, &b1 = p[i].B1 ? *p[i].B1 : p[i].B0;
        j.M = p[i].M; j.N = p[i].N; j.K = p[i].K; j.nparts = p[i].A1 ? 2 : 1; j.a_mn = p[i].a_mn; j.b_mn = p[i].b_mn;
        j.tile0 = tiles;
        tiles += (int)p[i].tiles(kN);
        auto maps = [](CUtensorMap *m, const Operand &o0, const Operand &o1, bool two, int mn, int rows, int &blocked) {
            blocked = mn && o0.cols % 64 == 0 && o1.cols % 64 == 0;
            for (int tries = 0; tries < 2; ++tries, blocked = 0) {
                if (operand_map(m, o0, mn != 0, rows, blocked != 0) && (!two || operand_map(m + 1, o1, mn != 0, rows, blocked != 0))) return true;
                if (!blocked) return false;
            }
            return false;
        };
        if (!maps(j.A, p[i].A0, a1, p[i].A1 != nullptr, j.a_mn, GM, j.a_blocked) || !maps(j.B, p[i].B0, b1, p[i].A1 != nullptr, j.b_mn, kN, j.b_blocked) ||
            !make_tensor_map_3d(&j.C, p[i].C, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 1, (uint64_t)p[i].M, (uint64_t)p[i].N, 128, 64))
            return cudaErrorInvalidValue;
        if (!p[i].A1) { j.A[1] = j.A[0]; j.B[1] = j.B[0]; }
    }
    for (int i = count; i < kMaxJobs; ++i) g.j[i] = g.j[0];
    g.count = count;
    g.tiles = tiles;
    constexpr int kSmem = gemm_smem(false, kN);
    const cudaError_t e = allow_smem<tc_gemm_group_kernel<kN>>(kSmem);
    if (e != cudaSuccess) return e;
    const int sms = device_info().sms;
    LaunchScope scope(MOA_KERNEL_OTHER, st);
    return launch_dependent(tc_gemm_group_kernel<kN>, dim3((unsigned)(tiles < sms ? tiles : sms)), dim3(kGemmThreads), (size_t)kSmem, st, g,
                            device_status_ptr());
}

// Whether `count` products go out as one launch: while their 128-column tiles fit on the SMs at once (then no wider tile and no pair
// would have been faster for any of them), none writes what another one reads (one after the other they may: dx over dy or x), and
// MOA_GEMM_PAIR does not ask for pairs.
bool group_fits(const Product *p, int count)
{
    long long t = 0;
    for (int i = 0; i < count; ++i) {
        t += p[i].tiles(128);
        for (int j = 0; j < count; ++j)
            if (i != j && p[i].disturbs(p[j])) return false;
    }
    return gemm_pair_mode() != 2 && t <= device_info().sms;
}
cudaError_t launch_group(const Product *p, int count, cudaStream_t st)
{
    long long t = 0;
    for (int i = 0; i < count; ++i) t += p[i].tiles(64);
    return t <= device_info().sms ? launch_group_n<64>(p, count, st) : launch_group_n<128>(p, count, st);
}

}  // namespace

// Two products of gemm_bf16 that do not depend on each other
cudaError_t gemm_bf16_two(const GemmArgs &x, const GemmArgs &y, cudaStream_t st)
{
    auto product = [](const GemmArgs &g) {
        return Product{Operand{g.A, g.a_mn ? g.K : g.M, g.a_mn ? g.M : g.K}, Operand{g.B, g.b_mn ? g.K : g.N, g.b_mn ? g.N : g.K}, nullptr, nullptr, g.C,
                       g.M, g.N, g.K, g.a_mn, g.b_mn};
    };
    const Product two[2] = {product(x), product(y)};
    if (group_fits(two, 2)) return launch_group(two, 2, st);
    const cudaError_t e = gemm_bf16(x.a_mn, x.b_mn, x.M, x.N, x.K, x.A, x.B, nullptr, x.C, st);
    return e != cudaSuccess ? e : gemm_bf16(y.a_mn, y.b_mn, y.M, y.N, y.K, y.A, y.B, nullptr, y.C, st);
}

// C[M,N] = A B^T (+ R): A given as [M,K] (a_mn = 0) or [K,M] (a_mn = 1), B as [N,K] (b_mn = 0) or [K,N] (b_mn = 1)
cudaError_t gemm_bf16(int a_mn, int b_mn, int M, int N, int K, const void *A, const void *B, const void *R, void *C,
                      cudaStream_t st)
{
    const Operand a{A, a_mn ? K : M, a_mn ? M : K}, b{B, b_mn ? K : N, b_mn ? N : K};
    const bool res = R != nullptr;
    if (!a_mn && !b_mn) return launch_gemm<false, false, EPI_STORE>(a, b, nullptr, nullptr, C, nullptr, R, nullptr, M, N, M, N, K, st, 1, res);
    if (!a_mn && b_mn) return launch_gemm<false, true, EPI_STORE>(a, b, nullptr, nullptr, C, nullptr, R, nullptr, M, N, M, N, K, st, 1, res);
    if (a_mn && b_mn) return launch_gemm<true, true, EPI_STORE>(a, b, nullptr, nullptr, C, nullptr, R, nullptr, M, N, M, N, K, st, 1, res);
    return launch_gemm<true, false, EPI_STORE>(a, b, nullptr, nullptr, C, nullptr, R, nullptr, M, N, M, N, K, st, 1, res);
}

cudaError_t gated_mlp_fwd(int n, int d, int dff, const void *x, const void *W1, const void *W3, const void *W2,
                          const void *res, void *a, void *u, void *h, void *y, cudaStream_t st)
{
    // a | u = x [W1; W3]^T with the gate in the epilogue, then y = h W2^T
    const Operand X{x, n, d}, w1{W1, dff, d}, w3{W3, dff, d}, Hh{h, n, dff}, w2{W2, d, dff};
    cudaError_t e = launch_gemm<false, false, EPI_SWIGLU_FWD>(X, w1, nullptr, &w3, a, u, h, nullptr, n, dff, n, dff, d, st);
    if (e != cudaSuccess) return e;
    return launch_gemm<false, false, EPI_STORE>(Hh, w2, nullptr, nullptr, y, nullptr, res, nullptr, n, d, n, d, dff, st, 1, res != nullptr);
}

cudaError_t gated_mlp_bwd(int n, int d, int dff, const void *x, const void *W1, const void *W3, const void *W2,
                          const void *a, const void *u, const void *h, const void *dy, void *da, void *du,
                          void *dx, void *dW1, void *dW3, void *dW2, cudaStream_t st)
{
    const Operand X{x, n, d}, w1{W1, dff, d}, w3{W3, dff, d}, w2{W2, d, dff}, Hh{h, n, dff}, DY{dy, n, d};
    const Operand DA{da, n, dff}, DU{du, n, dff};
    // dh = dy W2 (W2 [d,d_ff] read as the MN-major B operand), gate backward in the epilogue -> da, du
    cudaError_t e = launch_gemm<false, true, EPI_SWIGLU_BWD>(DY, w2, nullptr, nullptr, da, du, a, u, n, dff, n, dff, d, st);
    if (e != cudaSuccess) return e;
    // small: the four products that follow as one launch
    const Product rest[4] = {{DY, Hh, nullptr, nullptr, dW2, d, dff, n, 1, 1}, {DA, X, nullptr, nullptr, dW1, dff, d, n, 1, 1},
                             {DU, X, nullptr, nullptr, dW3, dff, d, n, 1, 1}, {DA, w1, &DU, &w3, dx, n, d, dff, 0, 1}};
    if (group_fits(rest, 4)) return launch_group(rest, 4, st);
    // dW2 [d,d_ff] = dy^T h: both operands read transposed (K = tokens)
    if ((e = launch_gemm<true, true, EPI_STORE>(DY, Hh, nullptr, nullptr, dW2, nullptr, nullptr, nullptr, d, dff, d, dff, n, st)) !=
        cudaSuccess)
        return e;
    // dW1 = da^T x, dW3 = du^T x   [d_ff,d]: one launch, so that the two tile sets fill the waves together
    if ((e = launch_gemm<true, true, EPI_STORE>(DA, X, &DU, &X, dW1, dW3, nullptr, nullptr, dff, d, dff, d, n, st, 2)) != cudaSuccess)
        return e;
    // dx = da W1 + du W3: two operand pairs accumulate into one tile (W1, W3 [d_ff,d] as MN-major B)
    return launch_gemm<false, true, EPI_STORE>(DA, w1, &DU, &w3, dx, nullptr, nullptr, nullptr, n, d, n, d, dff, st);
}

}  // namespace moa
