// Forward attention for head dimensions 136..256 on the sm_100a tensor cores, bf16 in, fp32 accumulate: the whole head dimension in one
// CTA.  (Two CTAs per query tile, each with half of the output columns, compute every score and every exponential twice: B1 H16
// H_kv4 n3001 d192 causal 110 us, here 57; B1 H8 n8192 d192 637, here 350; B1 H8 n8192 d256 638, here 460 (in turn, runs of 20 ms under the power cap).  From 200
// columns on that form is still the faster one where there are few query tiles: the rule is in tc_fwd.cu.)
//
// CTA = 128 query rows of one (batch, head); roles, barriers and the order of the products as in tc_fwd.cu: two softmax warpgroups take
// the key tiles in turn, one score buffer, K and V rings with a producer thread each, one issuing thread, which queues
// S(j + 2), P V(j), S(j + 3), ...  What differs: TMEM has room for ONE accumulator of 192 or 256 columns beside the scores
// and the two P buffers, so both warpgroups' products go into it, and their weights have to be relative to one maximum per row:
//   * the reference m of a row lives in shared memory and passes from the warpgroup of tile j - 1 to that of tile j through a barrier: the
//     warpgroup takes its own tile's maximum, waits for the reference, raises it if the maximum is more than 8 (log2 domain) above,
//     and hands it on -- long before the other warpgroup needs it, which still waits for the scores of tile j + 1;
//   * raising it means rescaling O, once P V of all tiles before has completed (rare: every few tiles at most);
//   * a warpgroup rescales its own row sum when it next sees the reference changed.
// TMEM (512 columns): scores [0,128), P of even / odd tiles [128,192) / [192,256), O [256, 256 + 64 NB).
// What bounds it: per 128 x 128 tile the UMMAs need 1536 (NB = 3) or 2048 cycles and the exponentials 1024 of the MUFU unit; a tile takes
// about 2000 cycles at d = 192 -- the softmax warpgroups' chain, as in tc_fwd.cu, plus the hand-over of the reference -- and 2650 at d = 256, where
// the rings hold less than a tile of V ahead of the products.
// Shared memory: Q 16 NB KB; K ring of whole tiles (NB = 3: two slots of 48 KB) or half tiles of 128 columns (NB = 4: three of 32 KB);
// V ring of half tiles of 64 keys (NB = 3: three of 24 KB; NB = 4: two of 32 KB).  NB: 64-column boxes of the head dimension (3 for 136..192, 4).
#include "common.cuh"
#include "ptx.cuh"
#include "tensormap.cuh"

namespace moa {
namespace {

using namespace ptx;

constexpr int BM = 128, BN = 128;
constexpr int kThreads = 384;      // warps 0-7 softmax, 8 TMA of Q and K, 9 UMMA issuer, 11 TMA of V
constexpr int kTmemCols = 512;
constexpr uint32_t kColS = 0, kColP = 128, kColO = 256;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.f;

enum : uint32_t { ERRW_Q = 0x141, ERRW_K = 0x142, ERRW_V = 0x143, ERRW_S = 0x144, ERRW_P = 0x145, ERRW_O = 0x146, ERRW_M = 0x147, ERRW_ALIGN = 0x148,
                ERRW_DO = 0x149 };

enum { FW_Q = 0, FW_KFULL = 1 /*3*/, FW_KEMPTY = 4 /*3*/, FW_VFULL = 7 /*3*/, FW_VEMPTY = 10 /*3*/, FW_P = 13 /*2: by tile parity*/,
       FW_SFREE = 15 /*2*/, FW_OB = 17 /*2: P V of the tile has completed*/, FW_M = 19 /*2: the row references of the tile are posted*/,
       FW_S = 21 /*[parity][tile / 2 & 1]: 4*/, FW_X = 25 /*epilogue exchange*/, FW_E = 26 /*O staged*/, FW_DONE = 27 /*last P V*/,
       FW_DO = 28 /*the dO tile (fused call)*/, FW_COUNT = 29 };

template <int NB>
struct WideFwd {
    static constexpr int kBox = 128 * 128;                        // 128 rows x 64 columns
    static constexpr int kQ = NB * kBox;
    static constexpr int kChunkBoxes = NB == 3 ? 3 : 2;           // K columns per ring slot, in boxes
    static constexpr int kChunks = NB / kChunkBoxes;              // slots a key tile passes through
    static constexpr int kKSlots = NB == 3 ? 2 : 3, kKSlot = kChunkBoxes * kBox;
    static constexpr int kVBox = 64 * 128;                        // 64 keys x 64 columns
    static constexpr int kVSlots = NB == 3 ? 3 : 2, kVSlot = NB * kVBox;
    static constexpr int offK = kQ, offV = offK + kKSlots * kKSlot, offM = offV + kVSlots * kVSlot;     // row references, 128 floats
    static constexpr int offX = offM + 512;                       // exchange (m, l): 2 x 128 float2
    static constexpr int offBar = offX + 2048;
    static constexpr int kTotal = offBar + 8 * FW_COUNT + 16;
};
static_assert(WideFwd<3>::kTotal <= 232448 && WideFwd<4>::kTotal <= 232448, "shared memory of one CTA");

struct WidePrep {
    int with_bwd;        // fused call: mapdO, Lp and Dp are there (what the forward prepares: tc_fwd.cu)
    float *Lp, *Dp, *zero_acc;
    int n_pad;
};

template <int NB>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd_wide_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                   const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapdO, float *__restrict__ L, int n, int d,
                   int causal, float scale_log2, int nqt, int hpg, int group, int H, WidePrep prep,
                   unsigned int *status)
{
    using S = WideFwd<NB>;
    extern __shared__ __align__(1024) uint8_t sm[];
    uint8_t *sQ = sm, *sK = sm + S::offK, *sV = sm + S::offV;
    float *mref = reinterpret_cast<float *>(sm + S::offM);
    float2 *xch = reinterpret_cast<float2 *>(sm + S::offX);
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + S::offBar);
    uint32_t *tmem_base_p = reinterpret_cast<uint32_t *>(bars + FW_COUNT);
    volatile uint32_t *abortp = tmem_base_p + 1;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    int bh, t0;
    job_from_block((int)blockIdx.x, nqt, (int)gridDim.x / nqt, hpg, bh, t0);
    const int bb = bh / H, hq = bh - bb * H, hk = hq / group;
    const int qt = causal ? nqt - 1 - t0 : t0;   // causal: longest rows first
    const int q0 = qt * BM;
    const int nkt_want = causal ? qt + 1 : (n + BN - 1) / BN;
    const bool aligned = (smem_u32(sm) & 1023u) == 0;

    auto load_k = [&](int g) {         // chunk g: columns of chunk g % kChunks of key tile g / kChunks
        const int s = g % S::kKSlots, j = g / S::kChunks, c = g % S::kChunks;
        mbar_arrive_expect_tx(bars + FW_KFULL + s, S::kKSlot);
        for (int b = 0; b < S::kChunkBoxes; ++b)
            tma_load_4d(sK + s * S::kKSlot + b * S::kBox, &mapK, bars + FW_KFULL + s, 64 * (c * S::kChunkBoxes + b), j * BN, hk, bb);
    };
    auto load_v = [&](int g) {         // half g: keys 64 g .. 64 g + 63
        const int s = g % S::kVSlots;
        mbar_arrive_expect_tx(bars + FW_VFULL + s, S::kVSlot);
        for (int b = 0; b < NB; ++b) tma_load_4d(sV + s * S::kVSlot + b * S::kVBox, &mapV, bars + FW_VFULL + s, 64 * b, g * 64, hk, bb);
    };
    const int nk_all = aligned ? nkt_want * S::kChunks : 0, nv_all = aligned ? nkt_want * 2 : 0;
    const int early_k = min(nk_all, S::kKSlots), early_v = min(nv_all, S::kVSlots);
    // the first loads go out before the rest of the set-up
    if (warp == 8 && elect_one()) {
        mbar_init(bars + FW_Q, 1u);
        for (int s = 0; s < 3; ++s) mbar_init(bars + FW_KFULL + s, 1u);
        fence_mbar_init();
        grid_dependency_wait();
        if (early_k > 0) {
            mbar_arrive_expect_tx(bars + FW_Q, S::kQ);
            for (int b = 0; b < NB; ++b) tma_load_4d(sQ + b * S::kBox, &mapQ, bars + FW_Q, 64 * b, q0, hq, bb);
            for (int g = 0; g < early_k; ++g) load_k(g);
            if (prep.with_bwd)      // (what the end of the job reads: into L2)
                for (int b = 0; b < NB; ++b) tma_prefetch_4d(&mapdO, 64 * b, q0, hq, bb);
        }
    }
    if (warp == 11 && elect_one()) {
        for (int s = 0; s < 3; ++s) mbar_init(bars + FW_VFULL + s, 1u);
        fence_mbar_init();
        grid_dependency_wait();
        for (int g = 0; g < early_v; ++g) load_v(g);
    }
    if (tid == 0) {
        for (int b = 0; b < FW_COUNT; ++b) {
            if (b < FW_KEMPTY || (b >= FW_VFULL && b < FW_VEMPTY)) continue;   // (the producers' own)
            const bool of_group = (b >= FW_P && b < FW_OB) || (b >= FW_M && b < FW_S);
            mbar_init(bars + b, of_group ? 128u : (b == FW_X || b == FW_E) ? 256u : 1u);
        }
        *abortp = aligned ? 0u : 1u;
        if (!aligned && status) atomicCAS(status, 0u, (unsigned int)ERRW_ALIGN);
        fence_mbar_init();
        prefetch_tensormap(&mapO);
    }
    if (warp == 9) { tmem_alloc(tmem_base_p, kTmemCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_wait();
    if (gridDim.x <= 512) grid_launch_dependents();      // (short launches only: see tc_fwd.cu)
    const uint32_t tbase = *tmem_base_p;
    const int nkt = (*abortp == 0) ? nkt_want : 0;       // misaligned shared memory: every role is a no-op
    const int dslot = NB == 3 ? nkt & 1 : 0;             // first K slot of the dO tile: that of the last tile but one, or the first two

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");      // (128 x 88 + 256 x 208 = 384 x 168, the launch's registers)
      if (warp == 8) {
        // ------------------------------------------------------------------ TMA producer of K
        int nk = early_k;
        if (prep.zero_acc != nullptr) {      // this CTA's rows of the dQ accumulator ([B*H, n, 256]), under the first loads
            float4 *dst = reinterpret_cast<float4 *>(prep.zero_acc + ((size_t)bh * n + q0) * 256);
            for (int i = lane; i < min(BM, n - q0) * 64; i += 32) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (elect_one()) {      // (one thread from here on)
            for (int g = early_k; g < nkt * S::kChunks; ++g) {
                if (!mbar_wait(bars + FW_KEMPTY + g % S::kKSlots, (g / S::kKSlots - 1) & 1, abortp, status, ERRW_K)) break;
                load_k(g);
                ++nk;
            }
            // fused call: the dO tile, which the epilogue multiplies its rows with, goes over K slots that have come free (see tc_fwd2.cu)
            int armed_do = 0;
            if (prep.with_bwd && nkt > 0) {
                bool free = true;
                for (int s = dslot; free && s < dslot + (NB == 3 ? 1 : 2); ++s) {
                    const int uses = (nkt * S::kChunks - s + S::kKSlots - 1) / S::kKSlots;
                    free = uses <= 0 || mbar_wait(bars + FW_KEMPTY + s, (uses - 1) & 1, abortp, status, ERRW_K);
                }
                if (free) {
                    mbar_arrive_expect_tx(bars + FW_DO, NB * S::kBox);
                    armed_do = 1;
                    for (int b = 0; b < NB; ++b) tma_load_4d(sK + dslot * S::kKSlot + b * S::kBox, &mapdO, bars + FW_DO, 64 * b, q0, hq, bb);
                }
            }
            if (*abortp) {
                mbar_drain_one(bars + FW_DO, armed_do);
                mbar_drain_one(bars + FW_Q, early_k > 0 ? 1 : 0);
                for (int s = 0; s < S::kKSlots; ++s) mbar_drain_one(bars + FW_KFULL + s, nk > s ? (nk - s + S::kKSlots - 1) / S::kKSlots : 0);
            }
        }
      } else if (warp == 11 && elect_one()) {
        // ------------------------------------------------------------------ TMA producer of V
        int nv = early_v;
        for (int g = early_v; g < nkt * 2; ++g) {
            if (!mbar_wait(bars + FW_VEMPTY + g % S::kVSlots, (g / S::kVSlots - 1) & 1, abortp, status, ERRW_V)) break;
            load_v(g);
            ++nv;
        }
        if (*abortp)
            for (int s = 0; s < S::kVSlots; ++s) mbar_drain_one(bars + FW_VFULL + s, nv > s ? (nv - s + S::kVSlots - 1) / S::kVSlots : 0);
      } else if (warp == 9 && elect_one()) {
        // ------------------------------------------- UMMA issuer (one thread): S(j + 2), P V(j), S(j + 3), ... (why: tc_fwd2.cu)
        // Two threads / one, forward alone, in turn: runs of 40 ms under the power cap B1 H16/4 n3001 d192 causal 60.1 / 57.0 us, B1 H8 n8192 d192 360 / 346,
        // B2 H16 n4096 d256 causal 268 / 261; at 1965 MHz B1 H8 n1500 d256 24.6 / 22.3.
        constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0), idesc_pv = idesc_bf16_f32(128, 64 * NB, 0, 1);
        const uint64_t km_proto = smem_desc_sw128(0, 16, 1024), mn_proto = smem_desc_sw128(0, S::kVBox, 1024);
        const uint32_t km_hi = (uint32_t)(km_proto >> 32), mn_hi = (uint32_t)(mn_proto >> 32);
        auto field = [](const void *ptr) { return (smem_u32(ptr) >> 4) & 0x3FFFu; };
        const uint32_t q_lo = (uint32_t)km_proto + field(sQ);
        bool ok = nkt > 0 && mbar_wait(bars + FW_Q, 0, abortp, status, ERRW_Q);
        for (int step = 0; ok && step < nkt + 2; ++step) {
            if (step < nkt) {
                const int j = step;
#pragma unroll
                for (int c = 0; c < S::kChunks; ++c) {
                    const int g = j * S::kChunks + c, sl = g % S::kKSlots;
                    const uint32_t k_lo = (uint32_t)km_proto + field(sK + sl * S::kKSlot);
                    if (!mbar_wait(bars + FW_KFULL + sl, (g / S::kKSlots) & 1, abortp, status, ERRW_K)) { ok = false; break; }
                    // the one score buffer is free once the warpgroup of tile j-1 holds that tile's scores in registers
                    if (c == 0 && j >= 1 && !mbar_wait(bars + FW_SFREE + ((j - 1) & 1), ((j - 1) >> 1) & 1, abortp, status, ERRW_O)) { ok = false; break; }
                    tc_fence_after();
#pragma unroll
                    for (int ks = 0; ks < 4 * S::kChunkBoxes; ++ks) {
                        const uint32_t koff = (uint32_t)(((ks / 4) * S::kBox + (ks % 4) * 32) >> 4), qoff = koff + (uint32_t)((c * S::kKSlot) >> 4);
                        if (c == 0 && ks == 0) umma_ss2<false>(tbase + kColS, q_lo, km_hi, k_lo, km_hi, idesc_s);
                        else                   umma_ss2<true>(tbase + kColS, q_lo + qoff, km_hi, k_lo + koff, km_hi, idesc_s);
                    }
                    umma_commit(bars + FW_KEMPTY + sl);
                }
                if (!ok) break;
                umma_commit(bars + FW_S + 2 * (j & 1) + ((j >> 1) & 1));
            }
            if (step >= 2) {
                const int j = step - 2, b = j & 1, g = 2 * j, s0 = g % S::kVSlots, s1 = (g + 1) % S::kVSlots;
                if (!mbar_wait(bars + FW_VFULL + s0, (g / S::kVSlots) & 1, abortp, status, ERRW_V)) break;
                if (!mbar_wait(bars + FW_VFULL + s1, ((g + 1) / S::kVSlots) & 1, abortp, status, ERRW_V)) break;
                if (!mbar_wait(bars + FW_P + b, (j >> 1) & 1, abortp, status, ERRW_P)) break;
                tc_fence_after();
                const uint32_t acol = tbase + kColP + 64 * b, ocol = tbase + kColO;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {          // 16 keys each; P (bf16) is 64 TMEM columns
                    const uint32_t v_lo = (uint32_t)mn_proto + field(sV + (ks < 4 ? s0 : s1) * S::kVSlot) + (uint32_t)(((ks & 3) * 2048) >> 4);
                    if (ks == 0 && j == 0) umma_ts2<false>(ocol, acol, v_lo, mn_hi, idesc_pv);
                    else                   umma_ts2<true>(ocol, acol + ks * 8, v_lo, mn_hi, idesc_pv);
                    if (ks == 3) umma_commit(bars + FW_VEMPTY + s0);
                }
                umma_commit(bars + FW_VEMPTY + s1);
                umma_commit(bars + FW_OB + b);
                if (j == nkt - 1) umma_commit(bars + FW_DONE);
            }
        }
      }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
        // ---------------------------------------------------------------- softmax warps: thread = query row (TMEM lane)
        const int h = warp / 4;
        const int lane_row = 32 * (warp % 4) + lane;
        const int row = q0 + lane_row;
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        const uint32_t pcol = kColP + 64 * h;
        float m_used = -1e30f, l = 0.f;      // (a warpgroup without tiles contributes nothing)
        bool ok = nkt > 0;
        for (int j = h; ok && j < nkt; j += 2) {
            const int t = j >> 1;
            if (!mbar_wait(bars + FW_S + 2 * h + (t & 1), (t >> 1) & 1, abortp, status, ERRW_S)) { ok = false; break; }
            tc_fence_after();
            const int k0 = j * BN;
            const bool need_mask = (k0 + BN > n) || (causal && k0 + BN - 1 > q0);
            uint32_t r[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld(lane_addr + kColS + 32 * c, r[c]);
            tc_wait_ld();
            tc_fence_before();
            mbar_arrive(bars + FW_SFREE + h);      // the score columns are free: S(j+1) runs under this tile's exponentials
            if (need_mask) {
                const int lim = min(n, causal ? row + 1 : n) - k0;      // columns of this tile the row may see
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (32 * c + i >= lim) r[c][i] = 0xff800000u;   // -inf
            }
            float mx16[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int c = q >> 2, i0 = 8 * (q & 3);
                float a = fmax3(__uint_as_float(r[c][i0]), __uint_as_float(r[c][i0 + 1]), __uint_as_float(r[c][i0 + 2]));
                a = fmax3(a, __uint_as_float(r[c][i0 + 3]), __uint_as_float(r[c][i0 + 4]));
                a = fmax3(a, __uint_as_float(r[c][i0 + 5]), __uint_as_float(r[c][i0 + 6]));
                mx16[q] = fmaxf(a, __uint_as_float(r[c][i0 + 7]));
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) mx16[q] = fmaxf(mx16[q], mx16[q + 8]);
            const float mx = fmax3(fmax3(mx16[0], mx16[1], mx16[2]), fmax3(mx16[3], mx16[4], mx16[5]), fmaxf(mx16[6], mx16[7])) * scale_log2;
            // the row's reference: taken over from tile j-1, raised if this tile needs it, handed on
            float m_new;
            if (j == 0) {
                m_new = (mx == -INFINITY) ? -1e30f : mx;     // (a row past n)
                mref[lane_row] = m_new;
                mbar_arrive(bars + FW_M + 0);
            } else {
                if (!mbar_wait(bars + FW_M + (h ^ 1), ((j - 1) >> 1) & 1, abortp, status, ERRW_M)) { ok = false; break; }
                const float m_old = mref[lane_row];
                const bool grow = mx > m_old + kRescaleThreshold;
                m_new = grow ? mx : m_old;
                if (grow) mref[lane_row] = m_new;
                mbar_arrive(bars + FW_M + h);
                if (__any_sync(0xffffffffu, grow)) {
                    // O must hold every tile before this one and be still: P V(j-2) (the phase before on that barrier), then P V(j-1)
                    if (j >= 2 && !mbar_wait(bars + FW_OB + h, (t - 1) & 1, abortp, status, ERRW_O)) { ok = false; break; }
                    if (!mbar_wait(bars + FW_OB + (h ^ 1), ((j - 1) >> 1) & 1, abortp, status, ERRW_O)) { ok = false; break; }
                    tc_fence_after();
                    const float alpha = grow ? ex2(m_old - m_new) : 1.f;
#pragma unroll 1
                    for (int c = 0; c < 64 * NB; c += 16) {   // rare path
                        uint32_t o[16];
                        tmem_ld(lane_addr + kColO + c, o);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st(lane_addr + kColO + c, o);
                    }
                }
            }
            if (m_new != m_used) {           // (raised here or, since this warpgroup's last tile, by the other one)
                l *= ex2(m_used - m_new);
                m_used = m_new;
            }
            const uint64_t sl2 = pack_f32x2(scale_log2, scale_log2);
            const uint64_t negm2 = pack_f32x2(-m_used, -m_used);
            uint64_t ls2[2] = {0ull, 0ull};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    const uint64_t tt = fma_f32x2(pack_f32x2(__uint_as_float(r[c][i]), __uint_as_float(r[c][i + 1])), sl2, negm2);
                    float p0, p1;
                    unpack_f32x2(tt, p0, p1);
                    p0 = ex2(p0);
                    p1 = ex2(p1);
                    ls2[(i >> 1) & 1] = add_f32x2(ls2[(i >> 1) & 1], pack_f32x2(p0, p1));
                    pk[i / 2] = pack_bf16(p0, p1);
                }
                // P(j) goes where P(j-2) was: that product has read it by now
                if (c == 0 && t > 0 && !mbar_wait(bars + FW_OB + h, (t - 1) & 1, abortp, status, ERRW_O)) { ok = false; break; }
                tmem_st(lane_addr + pcol + 16 * c, pk);
            }
            {
                float s0, s1, s2, s3;
                unpack_f32x2(ls2[0], s0, s1);
                unpack_f32x2(ls2[1], s2, s3);
                l += (s0 + s1) + (s2 + s3);
            }
            tc_wait_st();
            tc_fence_before();
            mbar_arrive(bars + FW_P + h);
        }
        // ---- epilogue: the two row sums on the final reference (the larger of the two last seen), O / l as bf16 through the Q tile and a
        // TMA store, half of the columns per warpgroup
        float dpart = 0.f;
        const bool want_d = prep.with_bwd != 0;
        const uint8_t *drow = sK + dslot * S::kKSlot + lane_row * 128;       // this row of the dO tile
        xch[h * 128 + lane_row] = make_float2(m_used, l);
        mbar_arrive(bars + FW_X);
        if (ok && mbar_wait(bars + FW_X, 0, abortp, status, ERRW_P) && mbar_wait(bars + FW_DONE, 0, abortp, status, ERRW_O) &&
            (!want_d || mbar_wait(bars + FW_DO, 0, abortp, status, ERRW_DO))) {
            tc_fence_after();
            const float2 other = xch[(h ^ 1) * 128 + lane_row];
            const float m_all = fmaxf(m_used, other.x);
            const float l_all = l * ex2(m_used - m_all) + other.y * ex2(other.x - m_all);
            const float inv = 1.f / l_all;
#pragma unroll 1
            for (int c = 0; c < 32 * NB; c += 32) {
                const int c0 = 32 * NB * h + c;
                uint32_t o[32];
                tmem_ld(lane_addr + kColO + c0, o);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; i += 8) {
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __uint_as_float(o[i + u]) * inv;
                    const int cabs = c0 + i, chunk = ((cabs & 63) >> 3) ^ (lane_row & 7);       // 128-byte swizzle, as the maps expect
                    if (want_d) {      // (columns past the head dimension and rows past n are zeros)
                        const uint4 g = *reinterpret_cast<const uint4 *>(drow + (cabs >> 6) * S::kBox + chunk * 16);
                        const uint32_t gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 gg = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gw[u]));
                            dpart = fmaf(v[2 * u], gg.x, dpart);
                            dpart = fmaf(v[2 * u + 1], gg.y, dpart);
                        }
                    }
                    *reinterpret_cast<uint4 *>(sQ + (cabs >> 6) * S::kBox + lane_row * 128 + chunk * 16) =
                        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                }
            }
            if (h == 1) mref[lane_row] = dpart;      // (no tile needs the reference any more)
            fence_proxy_async_smem();
            mbar_arrive(bars + FW_E);
            if (want_d && h == 0 && mbar_wait(bars + FW_E, 0, abortp, status, ERRW_O)) {
                // both halves of the row are in: the backward's per-row inputs, in its padded layout
                const size_t prow = (size_t)bh * prep.n_pad + row;
                prep.Dp[prow] = row < n ? -(dpart + mref[lane_row]) : 0.f;
                prep.Lp[prow] = row < n ? -(m_all + log2f(l_all)) : -INFINITY;
            }
            if (tid == 0 && mbar_wait(bars + FW_E, 0, abortp, status, ERRW_O)) {
                for (int b = 0; b < NB; ++b)
                    if (64 * b < d) tma_store_4d(&mapO, sQ + b * S::kBox, 64 * b, q0, hq, bb);
                bulk_commit();
                bulk_wait_read<0>();      // shared memory is read before the CTA may exit
            }
            if (row < n && h == 0) L[(size_t)bh * n + row] = m_all * kLn2 + logf(l_all);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) tmem_dealloc(tbase, kTmemCols);
}

template <int NB>
cudaError_t launch(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb,
                   cudaStream_t st)
{
    using S = WideFwd<NB>;
    CUtensorMap mq, mk, mv, mo, mdo;
    const auto bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    // p.d <= 64 NB columns exist in memory: loads fill the rest of a box with zeros, the store drops it
    if (!make_tensor_map_4d_strided(&mq, Q, bf, 2, p.B, p.H, p.n, p.d, p.sq.row, p.sq.head, p.sq.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mk, K, bf, 2, p.B, p.kv_heads(), p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mv, V, bf, 2, p.B, p.kv_heads(), p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 64, 64) ||
        !make_tensor_map_4d_strided(&mo, O, bf, 2, p.B, p.H, p.n, p.d, p.so.row, p.so.head, p.so.batch, 128, 64))
        return cudaErrorInvalidValue;
    mdo = mo;
    if (fb.dO && !make_tensor_map_4d_strided(&mdo, fb.dO, bf, 2, p.B, p.H, p.n, p.d, p.so.row, p.so.head, p.so.batch, 128, 64)) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem<tc_fwd_wide_kernel<NB>>(S::kTotal);
    if (e != cudaSuccess) return e;
    const int nqt = (p.n + BM - 1) / BM;
    LaunchScope scope(MOA_KERNEL_FWD, st);
    return launch_dependent(tc_fwd_wide_kernel<NB>, dim3((unsigned)(nqt * p.BH())), dim3(kThreads), (size_t)S::kTotal, st, mq, mk, mv, mo, mdo, L,
                            p.n, p.d, p.causal, p.scale * kLog2e, nqt, heads_per_group(p, nqt), p.group(), p.H,
                            WidePrep{fb.dO != nullptr, fb.Lp, fb.Dp, fb.zero_acc, nqt * BM}, device_status_ptr());
}

}  // namespace

cudaError_t tc_fwd_wide(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb, cudaStream_t st)
{
    if (p.d <= 128 || p.d > 256 || p.d % 8) return cudaErrorInvalidValue;
    return p.d <= 192 ? launch<3>(p, Q, K, V, O, L, fb, st) : launch<4>(p, Q, K, V, O, L, fb, st);
}

}  // namespace moa
