// Backward attention for head dimensions 136..192 on the sm_100a tensor cores, bf16 in, fp32 accumulate: the whole head dimension in
// ONE pass.  (tc_bwd_wide.cu, which runs 200..256, computes the scores and dP in each of two passes over the halves of d; run on 192
// columns, 40 UMMAs per pass and 64-query tile against 56 here for both, and its loop is bound by the chain of hand-offs, which
// is paid once here: B1 H16 H_kv4 n3001 causal backward 385 -> 279 us, B1 H8 n8192 2108 -> 1420 us; with elected producers and
// issuers 253, and 1285 in runs of 40 ms under the power cap, 1452 before, or 1162 in short ones.)
//
// Same mathematics, the same key-tile-parallel structure and the same one-writer rule for dK and dV as tc_bwd.cu.  CTA = 128 keys of one
// K/V head (or, kSplit, its part of their query tiles); query tiles of 64 rows.
// TMEM (512 columns, all of them): S^T [0,64), dP^T [64,128), dV [128,320), dK [320,512).  dQ^T, 192 x 64, has no columns of its own: its
// rows 0..127 of d go over S^T, rows 64..191 (of which 128..191 are used; a UMMA has 128 rows) over dP^T.  So S^T and dP^T of the next
// tile wait until dQ has been read out; what runs under the elementwise phases is dP^T under P, dV under dS, and dK under the read-out.
// Per query tile i: S(i), dP(i) | P -> dV(i) | dS -> dQ(i), dK(i) | dQ read out.  P^T (bf16) overwrites the front of its S^T columns; dS^T
// goes to shared memory only, read from there as the K-major operand of dK and the MN-major one of dQ.
// Shared memory: K 48 KB + V 48 KB + two Q slots 48 KB + two dO slots 48 KB + dS^T 16 KB = 208 KB; dQ leaves as red.global.add.f32 from
// registers (one warp-wide instruction = 32 consecutive floats of one dQ row).
// Head dimensions below 192 run with the missing columns zero-filled by the loads and dropped by the stores.
#include "common.cuh"
#include "ptx.cuh"
#include "tensormap.cuh"

namespace moa {
namespace {

using namespace ptx;

constexpr int kThreads = 512;   // warps 0-7 elementwise, 8-11 dQ read-out and reds, 12 TMA, 13 UMMA, 14-15 idle
constexpr int kReduceWarp0 = 8, kLoadWarp = 12, kMmaWarp = 13;
constexpr int kTmemCols = 512;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int BQ = 64;          // query rows per tile
constexpr int NB = 3;           // 64-column boxes of the head dimension
constexpr int ACC = 256;        // row length of the dQ accumulator

enum : uint32_t {
    XERR_KV = 0x261, XERR_FULL = 0x262, XERR_EMPTY = 0x263, XERR_SDP = 0x264, XERR_PDS = 0x265, XERR_DQ = 0x266,
    XERR_DQR = 0x267, XERR_ALIGN = 0x268
};

struct Smem {
    static constexpr int kBoxK = 128 * 128;          // [128 keys][64 columns] bf16, 128-byte rows
    static constexpr int kBoxQ = 64 * 128;           // [64 queries][64 columns]
    static constexpr int kTile = NB * kBoxQ;         // a query tile
    static constexpr int offK = 0;
    static constexpr int offV = offK + NB * kBoxK;
    static constexpr int offQ = offV + NB * kBoxK;   // 2 slots
    static constexpr int offdO = offQ + 2 * kTile;   // 2 slots
    static constexpr int offdS = offdO + 2 * kTile;  // dS^T tile, [128 keys][64 queries]
    static constexpr int offL = offdS + 128 * 128;   // 2 x 64 floats, travels with the Q slot
    static constexpr int offDd = offL + 2 * 256;
    static constexpr int offBar = offDd + 2 * 256;
    static constexpr int kTotal = offBar + 256;
    static constexpr int kPart = 128 * NB * 64 * 4;  // kSplit: partial dV (and dK), fp32, over K, V, Q and dO
};
static_assert(Smem::kTotal <= 232448, "shared memory of one CTA");
static_assert(2 * Smem::kPart <= Smem::offdS, "the partial dV, dK are staged over K, V, Q and dO");

enum {
    X_KV = 0, X_Q = 1 /*2*/, X_QEMPTY = 3 /*2*/, X_DO = 5 /*2*/, X_DOEMPTY = 7 /*2*/, X_S = 9, X_P = 10, X_DP = 11, X_DS = 12, X_DQ = 13,
    X_DQR = 14, X_EPI = 15, X_COUNT = 16
};

__device__ __forceinline__ void red_add_f32(float *addr, float a)
{
    asm volatile("red.global.add.f32 [%0], %1;" ::"l"(addr), "f"(a) : "memory");
}

template <bool kGrouped, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
tc_bwd192_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                   const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapdO,
                   const __grid_constant__ CUtensorMap mapdK, const __grid_constant__ CUtensorMap mapdV,
                   const float *__restrict__ Lp, const float *__restrict__ Dp, float *__restrict__ dQacc,
                   int n, int n_pad, int d, int causal, float scale, float scale_log2, int nkt, int nqt /*tiles of 64 rows*/, int hpg, int group,
                   int Hkv, unsigned int *status, int split, __nv_bfloat16 *__restrict__ dK, __nv_bfloat16 *__restrict__ dV,
                   Strides skv)
{
    using SM = Smem;
    constexpr uint32_t colS = 0, colDP = 64, colDV = 128, colDK = 320;
    extern __shared__ __align__(1024) uint8_t sm[];
    uint8_t *sK = sm + SM::offK, *sV = sm + SM::offV, *sQ = sm + SM::offQ, *sdO = sm + SM::offdO, *sdS = sm + SM::offdS;
    float *sL = reinterpret_cast<float *>(sm + SM::offL);
    float *sD = reinterpret_cast<float *>(sm + SM::offDd);
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + SM::offBar);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(bars + X_COUNT);
    volatile uint32_t *abortp = reinterpret_cast<uint32_t *>(bars + X_COUNT + 1);

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    // kSplit: the `split` CTAs of a cluster share a key tile, each takes a contiguous part of its query tiles
    const int rank = kSplit ? (int)cluster_ctarank() : 0, blk = kSplit ? (int)blockIdx.x / split : (int)blockIdx.x;
    int bh, kt;                                           // causal: key tile 0 has the most query tiles and goes first
    job_from_block(blk, nkt, (int)gridDim.x / (kSplit ? split : 1) / nkt, hpg, bh, kt);
    const int k0 = kt * 128;
    const int i_begin = causal ? 2 * kt : 0;
    const int bb = bh / Hkv, hk = bh - bb * Hkv;
    const int hq0 = hk * (kGrouped ? group : 1) - bh * (kGrouped ? group : 1);   // query head in batch = flat index + hq0
    const int niter_tile = (kGrouped ? group : 1) * (nqt - i_begin);
    const int it0 = kSplit ? niter_tile * rank / split : 0;                 // this CTA's first query tile of the job
    const int niter_all = kSplit ? niter_tile * (rank + 1) / split - it0 : niter_tile;
    struct TileWalk {
        int qh, qi, first, end;
        __device__ void next()
        {
            ++qi;
            if (kGrouped && qi == end) { qi = first; ++qh; }
        }
    };
    const int head0 = kGrouped && kSplit ? it0 / (nqt - i_begin) : 0;       // query heads of the group in front of it
    const TileWalk walk0{(kGrouped ? bh * group : bh) + head0, i_begin + it0 - head0 * (nqt - i_begin), i_begin, nqt};

    // the first loads go out before the rest of the set-up (K, V, Q and dO are the call's inputs; -L, -D and the cleared accumulator
    // come from the kernel in front)
    if (warp == kLoadWarp && elect_one()) {
        mbar_init(bars + X_KV, 1u);
        for (int s = 0; s < 2; ++s) { mbar_init(bars + X_Q + s, 1u); mbar_init(bars + X_DO + s, 1u); }
        fence_mbar_init();
        if ((smem_u32(sm) & 1023u) == 0 && niter_all > 0) {
            mbar_arrive_expect_tx(bars + X_KV, 2 * NB * SM::kBoxK);
            mbar_arrive_expect_tx(bars + X_Q, SM::kTile + 512);            // (with its L and D, requested later)
            mbar_arrive_expect_tx(bars + X_DO, SM::kTile);
            for (int b = 0; b < NB; ++b) {
                tma_load_4d(sK + b * SM::kBoxK, &mapK, bars + X_KV, 64 * b, k0, hk, bb);
                tma_load_4d(sQ + b * SM::kBoxQ, &mapQ, bars + X_Q, 64 * b, walk0.qi * BQ, walk0.qh + hq0, bb);
            }
            for (int b = 0; b < NB; ++b) {
                tma_load_4d(sV + b * SM::kBoxK, &mapV, bars + X_KV, 64 * b, k0, hk, bb);
                tma_load_4d(sdO + b * SM::kBoxQ, &mapdO, bars + X_DO, 64 * b, walk0.qi * BQ, walk0.qh + hq0, bb);
            }
        }
    }
    if (tid == 0) {
        for (int b = 0; b < X_COUNT; ++b)
            if (b > X_Q + 1 && b != X_DO && b != X_DO + 1) mbar_init(bars + b, (b == X_P || b == X_DS || b == X_EPI) ? 256u : (b == X_DQR) ? 128u : 1u);
        *abortp = (smem_u32(sm) & 1023u) ? 1u : 0u;
        if (*abortp && status) atomicCAS(status, 0u, (unsigned)XERR_ALIGN);
        fence_mbar_init();
        prefetch_tensormap(&mapQ); prefetch_tensormap(&mapK); prefetch_tensormap(&mapV); prefetch_tensormap(&mapdO);
        prefetch_tensormap(&mapdK); prefetch_tensormap(&mapdV);
    }
    if (warp == kMmaWarp) { tmem_alloc(tmem_base_s, kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *tmem_base_s;
    const int niter = (*abortp == 0) ? niter_all : 0;

    if (warp >= kLoadWarp) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
      if (warp == kLoadWarp && elect_one()) {
        // ------------------------------------------------------------------ TMA producer (one thread)
        const int nq_per = nqt - i_begin;
        auto tile_of = [&](int it, int &qh, int &q0) {
            const int at = it0 + it, hh = kGrouped ? at / nq_per : 0;
            qh = (kGrouped ? bh * group : bh) + hh;
            q0 = (i_begin + at - hh * nq_per) * BQ;
        };
        auto load_q = [&](int it) {           // Q_it with -L log2e and -D of its 64 queries
            int qh, q0;
            tile_of(it, qh, q0);
            const int s = it & 1;
            if (it > 0) {
                mbar_arrive_expect_tx(bars + X_Q + s, SM::kTile + 512);
                for (int b = 0; b < NB; ++b) tma_load_4d(sQ + s * SM::kTile + b * SM::kBoxQ, &mapQ, bars + X_Q + s, 64 * b, q0, qh + hq0, bb);
            }
            bulk_load_1d(sL + s * 64, Lp + (size_t)qh * n_pad + q0, 256, bars + X_Q + s);
            bulk_load_1d(sD + s * 64, Dp + (size_t)qh * n_pad + q0, 256, bars + X_Q + s);
        };
        auto load_do = [&](int it) {
            int qh, q0;
            tile_of(it, qh, q0);
            const int s = it & 1;
            mbar_arrive_expect_tx(bars + X_DO + s, SM::kTile);
            for (int b = 0; b < NB; ++b) tma_load_4d(sdO + s * SM::kTile + b * SM::kBoxQ, &mapdO, bars + X_DO + s, 64 * b, q0, qh + hq0, bb);
        };
        if (niter > 1) load_do(1);
        grid_dependency_wait();
        grid_launch_dependents();
        if (niter > 0) {
            load_q(0);
            if (niter > 1) load_q(1);
        }
        for (int it = 0; it + 2 < niter; ++it) {      // the slots of tile `it` are free once its dV (dK) has completed
            if (!mbar_wait(bars + X_DOEMPTY + (it & 1), (it >> 1) & 1, abortp, status, XERR_EMPTY)) break;
            load_do(it + 2);
            if (!mbar_wait(bars + X_QEMPTY + (it & 1), (it >> 1) & 1, abortp, status, XERR_EMPTY)) break;
            load_q(it + 2);
        }
      } else if (warp == kMmaWarp && elect_one()) {
        // ------------------------------------------------------------------- UMMA issuer (one thread)
        constexpr uint32_t idesc_st = idesc_bf16_f32(128, 64, 0, 0);          // S^T, dP^T: 128 keys x 64 queries
        constexpr uint32_t idesc_acc = idesc_bf16_f32(128, 64 * NB, 0, 1);    // dV, dK: B MN-major, all columns of d
        constexpr uint32_t idesc_dq = idesc_bf16_f32(128, 64, 1, 1);          // dQ^T: 128 rows of d x 64 queries
        const uint64_t km_proto = smem_desc_sw128(0, 16, 1024);
        const uint64_t mnq_proto = smem_desc_sw128(0, SM::kBoxQ, 1024);  // MN-major over boxes of 64 rows (Q, dO, dS^T)
        const uint64_t mnk_proto = smem_desc_sw128(0, SM::kBoxK, 1024);  // MN-major over boxes of 128 rows (K)
        const uint32_t km_hi = (uint32_t)(km_proto >> 32), mnq_hi = (uint32_t)(mnq_proto >> 32), mnk_hi = (uint32_t)(mnk_proto >> 32);
        const uint32_t km_lo = (uint32_t)km_proto, mnq_lo = (uint32_t)mnq_proto, mnk_lo = (uint32_t)mnk_proto;
        auto field = [](const void *ptr) { return (smem_u32(ptr) >> 4) & 0x3FFFu; };
        const uint32_t k_km = km_lo + field(sK), v_km = km_lo + field(sV), ds_km = km_lo + field(sdS);
        const uint32_t q_km0 = km_lo + field(sQ), q_mn0 = mnq_lo + field(sQ), do_km0 = km_lo + field(sdO), do_mn0 = mnq_lo + field(sdO);
        const uint32_t k_mn = mnk_lo + field(sK), ds_mn = mnq_lo + field(sdS);
        constexpr uint32_t kSlot = (uint32_t)(SM::kTile >> 4);
        auto moff = [](int ks) { return (uint32_t)((ks * 2048) >> 4); };
        // A[128 keys] (boxes of 128 rows) times B[64 queries] over the whole head dimension: twelve k-steps
        auto over_d = [&](uint32_t col, uint32_t a0, uint32_t b0) {
#pragma unroll
            for (int bx = 0; bx < NB; ++bx) {
                const uint32_t a = a0 + (uint32_t)((bx * SM::kBoxK) >> 4), b = b0 + (uint32_t)((bx * SM::kBoxQ) >> 4);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (bx == 0 && q == 0) umma_ss2<false>(tbase + col, a, km_hi, b, km_hi, idesc_st);
                    else umma_ss2<true>(tbase + col, a + (uint32_t)((q * 32) >> 4), km_hi, b + (uint32_t)((q * 32) >> 4), km_hi, idesc_st);
                }
            }
        };
        bool ok = niter > 0 && mbar_wait(bars + X_KV, 0, abortp, status, XERR_KV);
        for (int it = 0; ok && it < niter; ++it) {
            const int s = it & 1;
            if (!mbar_wait(bars + X_Q + s, (it >> 1) & 1, abortp, status, XERR_FULL)) break;
            if (!mbar_wait(bars + X_DO + s, (it >> 1) & 1, abortp, status, XERR_FULL)) break;
            if (it > 0 && !mbar_wait(bars + X_DQR, (it - 1) & 1, abortp, status, XERR_DQR)) break;   // dQ(it-1) is out of both column ranges
            tc_fence_after();
            over_d(colS, k_km, q_km0 + s * kSlot);          // S^T(it) = K Q_it^T
            umma_commit(bars + X_S);
            over_d(colDP, v_km, do_km0 + s * kSlot);        // dP^T(it) = V dO_it^T
            umma_commit(bars + X_DP);
            if (!mbar_wait(bars + X_P, it & 1, abortp, status, XERR_PDS)) break;
            tc_fence_after();
            // dV += P^T dO_it: 64 queries = four k-steps; P^T bf16 at columns 0-15 (queries 0-31) and 32-47 (queries 32-63) of S^T
            const uint32_t do_mn = do_mn0 + s * kSlot, q_mn = q_mn0 + s * kSlot;
            if (it > 0) umma_ts2<true>(tbase + colDV, tbase + colS, do_mn, mnq_hi, idesc_acc);
            else        umma_ts2<false>(tbase + colDV, tbase + colS, do_mn, mnq_hi, idesc_acc);
#pragma unroll
            for (int ks = 1; ks < 4; ++ks)
                umma_ts2<true>(tbase + colDV, tbase + colS + 32 * (ks >> 1) + 8 * (ks & 1), do_mn + moff(ks), mnq_hi, idesc_acc);
            umma_commit(bars + X_DOEMPTY + s);
            if (!mbar_wait(bars + X_DS, it & 1, abortp, status, XERR_PDS)) break;
            tc_fence_after();
            // dQ_it^T = K^T dS^T: 128 keys = eight k-steps; rows 0..127 of d over S^T (dV, issued before, has read P there), 64..191 over dP^T
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t kk = k_mn + (uint32_t)((h * SM::kBoxK) >> 4), col = tbase + (h ? colDP : colS);
                umma_ss2<false>(col, kk, mnk_hi, ds_mn, mnq_hi, idesc_dq);
#pragma unroll
                for (int ks = 1; ks < 8; ++ks) umma_ss2<true>(col, kk + moff(ks), mnk_hi, ds_mn + moff(ks), mnq_hi, idesc_dq);
            }
            umma_commit(bars + X_DQ);
            // dK += dS^T Q_it, dS^T from the shared-memory tile (K-major): runs under the read-out of dQ
            if (it > 0) umma_ss2<true>(tbase + colDK, ds_km, km_hi, q_mn, mnq_hi, idesc_acc);
            else        umma_ss2<false>(tbase + colDK, ds_km, km_hi, q_mn, mnq_hi, idesc_acc);
#pragma unroll
            for (int ks = 1; ks < 4; ++ks)
                umma_ss2<true>(tbase + colDK, ds_km + (uint32_t)((ks * 32) >> 4), km_hi, q_mn + moff(ks), mnq_hi, idesc_acc);
            umma_commit(bars + X_QEMPTY + s);
        }
      }
    } else if (warp >= kReduceWarp0) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
        // ------------------------------------------------- dQ warps: lanes are columns of d
        grid_dependency_wait();      // the accumulator these warps add into was cleared by the kernel in front
        const int lane_row = 32 * (warp % 4) + lane;
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        const bool upper = warp % 4 >= 2, up_exists = upper && 64 + lane_row < d;      // (the accumulator's columns past d stay zero)
        TileWalk wr = walk0;
        for (int it = 0; it < niter; ++it) {
            const int q0 = wr.qi * BQ, qh = wr.qh;
            wr.next();
            if (!mbar_wait(bars + X_DQ, it & 1, abortp, status, XERR_DQ)) break;
            tc_fence_after();
            uint32_t lo[2][32], up[2][32];
            tmem_ld(lane_addr + colS, lo[0]);
            tmem_ld(lane_addr + colS + 32, lo[1]);
            if (upper) {            // (warp-uniform)
                tmem_ld(lane_addr + colDP, up[0]);
                tmem_ld(lane_addr + colDP + 32, up[1]);
            }
            tc_wait_ld();
            tc_fence_before();
            mbar_arrive(bars + X_DQR);      // the columns are free again; the reds go out from registers
            float *dst = dQacc + ((size_t)qh * n + q0) * ACC + lane_row;
            const int valid = min(BQ, n - q0);
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (32 * t + e < valid) red_add_f32(dst + (size_t)(32 * t + e) * ACC, __uint_as_float(lo[t][e]));
            if (up_exists) {
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (32 * t + e < valid) red_add_f32(dst + 64 + (size_t)(32 * t + e) * ACC, __uint_as_float(up[t][e]));
            }
        }
    } else {
        // ----------------------------------------------------------- elementwise warps 0-7
        asm volatile("setmaxnreg.inc.sync.aligned.u32 144;");
        const int wg = warp / 4;                          // query columns [32 wg, 32 wg + 32) of the 64-query tile
        const int lane_row = 32 * (warp % 4) + lane;      // TMEM lane of this thread = key index in the tile
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        uint64_t p2[16];                                  // this thread's 32 probabilities of the current tile, as fp32 pairs
        const uint64_t sl2 = pack_f32x2(scale_log2, scale_log2);
        const int qc0 = 32 * wg;
        bool ok = true;

        TileWalk wp = walk0;
        auto p_phase = [&](int it) -> bool {
            const int s = it & 1;
            // causal: query (tile qi of 64, column q) sees key (tile kt of 128, row lane_row) iff qi*64 + q >= kt*128 + lane_row
            const int rel = wp.qi * BQ - k0;
            const bool masked = causal && rel < 128;        // p_phase runs for it = 0, 1, 2, ... in order
            wp.next();
            if (!mbar_wait(bars + X_S, it & 1, abortp, status, XERR_SDP)) return false;
            tc_fence_after();
            const float *Ls = sL + s * 64;     // -L log2e
            uint32_t rs[32];
            tmem_ld(lane_addr + colS + qc0, rs);
            tc_wait_ld();
            score_exponents<32>(rs, Ls + qc0, sl2, masked, lane_row - qc0 - rel);
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
                const float a0 = ex2(__uint_as_float(rs[e])), a1 = ex2(__uint_as_float(rs[e + 1]));
                p2[e / 2] = pack_f32x2(a0, a1);
                pk[e / 2] = pack_bf16(a0, a1);
            }
            tmem_st(lane_addr + colS + qc0, pk);          // over the first 16 of the 32 columns just read
            tc_wait_st();
            tc_fence_before();
            mbar_arrive(bars + X_P);
            return true;
        };

        // (one loop, entered a step early, so that the P phase is inlined once: the roles' hot code is what the
        // schedulers keep fetching, and the kernel measurably runs faster the smaller it is)
        ok = niter > 0;
        for (int it = -1; ok && it < niter; ++it) {
          if (it >= 0) {
            const int s = it & 1;
            // dS-phase: dS^T = P^T o (dP^T - D)   (the factor `scale` is applied to dK and dQ at the end).
            // dP(it) complete also means that dQ(it-1) and dK(it-1), issued before it, have read the dS^T tile.
            if (!mbar_wait(bars + X_DP, it & 1, abortp, status, XERR_SDP)) { ok = false; break; }
            tc_fence_after();
            const float *Ds = sD + s * 64;     // -D
            uint32_t rd[32];
            tmem_ld(lane_addr + colDP + qc0, rd);
            tc_wait_ld();
            uint32_t gk[16];
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
                const ulonglong2 d4 = *reinterpret_cast<const ulonglong2 *>(Ds + qc0 + e);
                const uint64_t u0 = add_f32x2(pack_f32x2(__uint_as_float(rd[e]), __uint_as_float(rd[e + 1])), d4.x);
                const uint64_t u1 = add_f32x2(pack_f32x2(__uint_as_float(rd[e + 2]), __uint_as_float(rd[e + 3])), d4.y);
                float g0, g1, g2, g3;
                unpack_f32x2(mul_f32x2(p2[e / 2], u0), g0, g1);
                unpack_f32x2(mul_f32x2(p2[e / 2 + 1], u1), g2, g3);
                gk[e / 2] = pack_bf16(g0, g1);
                gk[e / 2 + 1] = pack_bf16(g2, g3);
            }
            // dS^T row (this key) into the MN-major tile: 128-byte row of 64 queries, 16-byte chunks 4 wg .. 4 wg + 3, swizzled
            uint8_t *rowp = sdS + lane_row * 128;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const int chunk = (4 * wg + jj) ^ (lane_row & 7);
                *reinterpret_cast<uint4 *>(rowp + chunk * 16) = make_uint4(gk[4 * jj], gk[4 * jj + 1], gk[4 * jj + 2], gk[4 * jj + 3]);
            }
            tc_fence_before();
            fence_proxy_async_smem();
            mbar_arrive(bars + X_DS);
          }
            if (it + 1 < niter) ok = p_phase(it + 1);
        }
        // every UMMA has completed once dK of the last tile has (one issuing thread; its phase before is known complete: dP of the last tile is)
        auto all_done = [&]() { return mbar_wait(bars + X_QEMPTY + ((niter - 1) & 1), ((niter - 1) >> 1) & 1, abortp, status, XERR_DQ); };
        if (kSplit) {
            const bool done = ok && all_done();
            tc_fence_after();
            // partial dV, dK as floats over K, V, Q and dO, which are no longer read: rows of 192 floats, 16-byte chunks swizzled by the row
#pragma unroll 1
            for (int which = 0; which < 2; ++which) {
                uint8_t *row = sm + which * SM::kPart + lane_row * (64 * NB * 4);
#pragma unroll 1
                for (int c = 0; c < 32 * NB; c += 32) {
                    const int c0 = 32 * NB * wg + c;
                    uint32_t r[32];
                    if (__all_sync(0xffffffffu, done)) {
                        tmem_ld(lane_addr + (which == 0 ? colDV : colDK) + c0, r);
                        tc_wait_ld();
                    } else {              // (a CTA without query tiles adds nothing)
#pragma unroll
                        for (int e = 0; e < 32; ++e) r[e] = 0u;
                    }
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<uint4 *>(row + ((((c0 + e) / 4) ^ (lane_row & 7)) << 4)) = make_uint4(r[e], r[e + 1], r[e + 2], r[e + 3]);
                }
            }
        } else if (ok) {
            // dV and scale*dK go out as bf16 through the V and K tiles (no longer read) and TMA stores; rows past n and columns past d are
            // clipped by the tensor map.  dV first, under the last dQ and dK: it is complete once the last dO slot is free.
#pragma unroll 1
            for (int which = 0; which < 2; ++which) {
                const bool there = which == 0 ? mbar_wait(bars + X_DOEMPTY + ((niter - 1) & 1), ((niter - 1) >> 1) & 1, abortp, status, XERR_DQ) : all_done();
                if (!there) break;
                tc_fence_after();
                const float mul = which == 0 ? 1.f : scale;
                uint8_t *stage = which == 0 ? sV : sK;
#pragma unroll 1
                for (int c = 0; c < 32 * NB; c += 32) {
                    const int c0 = 32 * NB * wg + c;
                    uint32_t r[32];
                    tmem_ld(lane_addr + (which == 0 ? colDV : colDK) + c0, r);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; e += 8) {
                        uint4 v;
                        v.x = pack_bf16(__uint_as_float(r[e + 0]) * mul, __uint_as_float(r[e + 1]) * mul);
                        v.y = pack_bf16(__uint_as_float(r[e + 2]) * mul, __uint_as_float(r[e + 3]) * mul);
                        v.z = pack_bf16(__uint_as_float(r[e + 4]) * mul, __uint_as_float(r[e + 5]) * mul);
                        v.w = pack_bf16(__uint_as_float(r[e + 6]) * mul, __uint_as_float(r[e + 7]) * mul);
                        const int cabs = c0 + e;          // first of 8 columns
                        const int chunk = ((cabs & 63) >> 3) ^ (lane_row & 7);   // 128-byte swizzle, as the maps expect
                        *reinterpret_cast<uint4 *>(stage + (cabs >> 6) * SM::kBoxK + lane_row * 128 + chunk * 16) = v;
                    }
                }
                fence_proxy_async_smem();
                mbar_arrive(bars + X_EPI);
                if (tid == 0 && mbar_wait(bars + X_EPI, which, abortp, status, XERR_DQ)) {
                    for (int b = 0; b < NB; ++b)
                        if (64 * b < d) tma_store_4d(which == 0 ? &mapdV : &mapdK, stage + b * SM::kBoxK, 64 * b, k0, hk, bb);     // (a box wholly past the head dimension has nothing to store)
                    bulk_commit();
                }
            }
            if (tid == 0) bulk_wait_read<0>();      // shared memory is read before the CTA may exit
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tbase, kTmemCols);
    if (kSplit) {
        // the ranks add up the partial results, 128 / split rows each, and write them out
        cluster_sync_all();
        if (warp < kLoadWarp) {
            const int per = 128 / split;
            for (int i = tid; i < 2 * per * 8 * NB; i += 32 * kLoadWarp) {
                const int c8 = i % (8 * NB), r = rank * per + (i / (8 * NB)) % per, which = i / (8 * NB) / per;
                const uint32_t row = smem_u32(sm) + which * SM::kPart + r * (64 * NB * 4);
                float v[8];
                sum_split(row + (((2 * c8) ^ (r & 7)) << 4), row + (((2 * c8 + 1) ^ (r & 7)) << 4), rank, split, which == 0 ? 1.f : scale, v);
                if (k0 + r < n && 8 * c8 < d)
                    *reinterpret_cast<uint4 *>((which == 0 ? dV : dK) + skv.at(bb, hk, k0 + r) + 8 * c8) =
                        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
            }
        }
        cluster_sync_all();       // nobody leaves while another rank may still read its shared memory
    }
    if (*abortp && tid == kLoadWarp * 32) {
        // A wait expired: copies the producer asked for may still be on their way into the CTA's shared memory.  It
        // stays for a fixed 400,000 cycles (hundreds of times a copy's latency) (any one thread keeps it) before the CTA can leave.
        const long long t0 = clock64();
        while (clock64() - t0 < 400000LL) { }
    }
}

template <bool kGrouped, bool kSplit>
cudaError_t launch_192(const Problem &p, const void *Q, const void *K, const void *V, const void *dO, const float *Lp,
                        const float *Dp, void *dK, void *dV, float *dQacc, int split, cudaStream_t st)
{
    CUtensorMap mq, mk, mv, mdo, mdk, mdv;
    const auto bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const int hkv = p.kv_heads();
    // p.d <= 192 columns exist in memory: loads fill the rest of a box with zeros, stores drop it
    if (!make_tensor_map_4d_strided(&mq, Q, bf, 2, p.B, p.H, p.n, p.d, p.sq.row, p.sq.head, p.sq.batch, 64, 64) ||
        !make_tensor_map_4d_strided(&mdo, dO, bf, 2, p.B, p.H, p.n, p.d, p.so.row, p.so.head, p.so.batch, 64, 64) ||
        !make_tensor_map_4d_strided(&mk, K, bf, 2, p.B, hkv, p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mv, V, bf, 2, p.B, hkv, p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mdk, dK, bf, 2, p.B, hkv, p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mdv, dV, bf, 2, p.B, hkv, p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64))
        return cudaErrorInvalidValue;
    constexpr int kSmem = Smem::kTotal;
    cudaError_t e = allow_smem<tc_bwd192_kernel<kGrouped, kSplit>>(kSmem);
    if (e != cudaSuccess) return e;
    const int nkt = (p.n + 127) / 128;
    LaunchScope scope(MOA_KERNEL_BWD_KV, st);
    Problem pkv = p;
    pkv.H = hkv;
    pkv.Hkv = 0;
    return launch_cluster(tc_bwd192_kernel<kGrouped, kSplit>, (unsigned)split, dim3((unsigned)(nkt * p.BHkv() * split)), dim3(kThreads),
                          (size_t)kSmem, st,
        mq, mk, mv, mdo, mdk, mdv, Lp, Dp, dQacc, p.n, nkt * 128, p.d, p.causal, p.scale, p.scale * kLog2e, nkt, (p.n + BQ - 1) / BQ,
        heads_per_group(pkv, nkt), p.group(), hkv, device_status_ptr(), split, (__nv_bfloat16 *)dK, (__nv_bfloat16 *)dV, p.skv);
}

}  // namespace

cudaError_t tc_bwd_kv_192(const Problem &p, const void *Q, const void *K, const void *V, const void *dO,
                          const float *Lp, const float *Dp, void *dK, void *dV, float *dQacc, bool share, cudaStream_t st)
{
    if (p.d <= 128 || p.d > 192 || p.d % 8 || dQacc == nullptr) return cudaErrorInvalidValue;
    const long long nkt = (p.n + 127) / 128, nqt = (p.n + BQ - 1) / BQ, jobs = nkt * p.BHkv(), longest = nqt * p.group();     // query tiles of 64
    const long long total = p.causal ? (nkt * nqt - nkt * (nkt - 1)) * p.BHkv() * p.group() : jobs * longest;
    const int split = !share ? 1 : bwd_split(jobs, longest, total, p.causal, 2.5, 3.0);
    // (both sides, alone / pairs: 64 jobs of 16 tiles 50.1 / 40.6 us, of 8 tiles 32.4 / 31.5.  24 jobs of 6 tiles 24.5 / 25.3, of 5 tiles 21.8 / 25.0, where
    // the estimate, whose constants are older than the elected issuers, takes fours: 28.5 and 28.3)
    if (split > 1)
        return p.group() > 1 ? launch_192<true, true>(p, Q, K, V, dO, Lp, Dp, dK, dV, dQacc, split, st)
                             : launch_192<false, true>(p, Q, K, V, dO, Lp, Dp, dK, dV, dQacc, split, st);
    return p.group() > 1 ? launch_192<true, false>(p, Q, K, V, dO, Lp, Dp, dK, dV, dQacc, 1, st)
                         : launch_192<false, false>(p, Q, K, V, dO, Lp, Dp, dK, dV, dQacc, 1, st);
}

}  // namespace moa
