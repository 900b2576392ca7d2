// Forward attention, two query tiles per CTA (head dimensions up to 128): the form of tc_fwd.cu for launches with enough of them.
//
// tc_fwd.cu gives its two softmax streams the even and the odd key tiles of ONE query tile; here stream h takes ALL key tiles of
// query tile h of a pair, so that
//   * a K or V tile fetched once serves two score (P V) products: half the operand traffic L2 -> shared memory per unit of work;
//   * what a job costs beside its tiles (set-up, first loads, epilogue: 7.5 us of tc_fwd.cu) is paid once per 256 rows;
//   * the streams share nothing, so the epilogue merges nothing: a stream that has finished writes its rows while the other still works.
// The order of the products is that of tc_fwd.cu with its tile number j read as (key tile j / 2, query tile j % 2), and so are the roles, the
// barriers, the one score buffer used in turn, the order of the products and the TMEM plan.  With the causal mask the
// longer query tile of a pair (one key tile more) is stream 0; a query tile without a partner (odd count: the last one, causal the
// first, which is the shortest) runs alone in stream 0.
// Shared memory: two Q tiles, two K and two V slots (192 KB at D = 128).  A stream's O leaves through its own Q tile.
#include "common.cuh"
#include "ptx.cuh"
#include "tensormap.cuh"

namespace moa {
namespace {

using namespace ptx;

constexpr int BM = 128, BN = 128;
constexpr int kThreads = 384;      // warps 0-7 softmax, 8 TMA of Q and K, 9 UMMA issuer (D = 64: for S, and 10 for P V), 11 TMA of V
constexpr int kTmemCols = 512;     // scores [0,128); bf16 P of the two streams [128,192), [192,256); two O accumulators from 256
constexpr uint32_t kColS = 0, kColP = 128, kColO = 256;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.f;

enum : uint32_t { ERR2_Q = 0x121, ERR2_K = 0x122, ERR2_V = 0x123, ERR2_S = 0x124, ERR2_P = 0x125, ERR2_O = 0x126, ERR2_DO = 0x127, ERR2_ALIGN = 0x128 };

enum { F2_Q = 0, F2_KFULL = 1 /*2*/, F2_KEMPTY = 3 /*2*/, F2_VFULL = 5 /*2*/, F2_VEMPTY = 7 /*2*/, F2_P = 9 /*2: per stream*/,
       F2_SFREE = 11 /*2: per stream, the tile's scores are in registers*/, F2_OB = 13 /*2: per stream, P V of the stream's tile has completed*/,
       F2_E = 15 /*2: per stream, O staged*/, F2_S = 17 /*[stream][key tile & 1]: 4, as in tc_fwd.cu*/,
       F2_DO = 21 /*2: per stream, its dO tile (fused call)*/, F2_COUNT = 23 };

struct FwdPrep2 {
    int with_bwd;        // fused call: mapdO, Lp and Dp are there
    float *Lp, *Dp;
    int n_pad;
    int d;               // columns of a row in memory (<= D)
};

// KL: 16-column steps of the head dimension that hold anything (D / 16, or 6 for 72..96 columns at D = 128)
template <int D, int KL>
__global__ void __launch_bounds__(kThreads, 1)
tc_fwd2_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
               const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO, const __grid_constant__ CUtensorMap mapdO, float *__restrict__ L, int n,
               int causal, float scale_log2, int npairs, int hpg, int group, int H, float *__restrict__ zero_acc, FwdPrep2 prep,
               unsigned int *status)
{
    constexpr int kTileBytes = 128 * D * 2, kBoxes = D / 64, kBoxBytes = 128 * 128;
    constexpr bool kOneIssuer = D == 128;
    extern __shared__ __align__(1024) uint8_t sm[];
    uint8_t *sQ = sm /*2 tiles: stream 0, 1*/, *sK = sm + 2 * kTileBytes, *sV = sm + 4 * kTileBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + 6 * kTileBytes);
    uint32_t *tmem_base_p = reinterpret_cast<uint32_t *>(bars + F2_COUNT);
    volatile uint32_t *abortp = tmem_base_p + 1;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    int bh, t;
    job_from_block((int)blockIdx.x, npairs, (int)gridDim.x / npairs, hpg, bh, t);
    const int bb = bh / H, hq = bh - bb * H, hk = hq / group;
    const int nqt = (n + BM - 1) / BM, nkt_all = (n + BN - 1) / BN;
    // query tiles of the two streams (-1: none) and their numbers of key tiles; n0 >= n1, n0 - n1 <= 1 or n1 = 0
    const int pair = causal ? npairs - 1 - t : t;      // causal: longest rows first
    int qt0, qt1;
    if (causal) {
        qt0 = nqt % 2 ? 2 * pair : 2 * pair + 1;
        qt1 = qt0 - 1;
    } else {
        qt0 = 2 * pair;
        qt1 = 2 * pair + 1 < nqt ? 2 * pair + 1 : -1;
    }
    const int want0 = causal ? qt0 + 1 : nkt_all, want1 = qt1 < 0 ? 0 : causal ? qt1 + 1 : nkt_all;
    const int q00 = qt0 * BM, q01 = qt1 * BM;

    const bool aligned = (smem_u32(sm) & 1023u) == 0;
    const int early = aligned ? min(want0, 2) : 0;
    auto load_k = [&](int j) {
        const int s = j & 1;
        mbar_arrive_expect_tx(bars + F2_KFULL + s, kTileBytes);
        for (int b = 0; b < kBoxes; ++b) tma_load_4d(sK + s * kTileBytes + b * kBoxBytes, &mapK, bars + F2_KFULL + s, 64 * b, j * BN, hk, bb);
    };
    auto load_v = [&](int j) {
        const int s = j & 1;
        mbar_arrive_expect_tx(bars + F2_VFULL + s, kTileBytes);
        for (int b = 0; b < kBoxes; ++b) tma_load_4d(sV + s * kTileBytes + b * kBoxBytes, &mapV, bars + F2_VFULL + s, 64 * b, j * BN, hk, bb);
    };
    // the first loads go out before the rest of the set-up
    if (warp == 8 && elect_one()) {
        mbar_init(bars + F2_Q, 1u);
        mbar_init(bars + F2_KFULL, 1u);
        mbar_init(bars + F2_KFULL + 1, 1u);
        fence_mbar_init();
        grid_dependency_wait();
        if (early > 0) {
            mbar_arrive_expect_tx(bars + F2_Q, (want1 > 0 ? 2 : 1) * kTileBytes);
            for (int b = 0; b < kBoxes; ++b) tma_load_4d(sQ + b * kBoxBytes, &mapQ, bars + F2_Q, 64 * b, q00, hq, bb);
            if (early > 0) load_k(0);
            if (want1 > 0)
                for (int b = 0; b < kBoxes; ++b) tma_load_4d(sQ + kTileBytes + b * kBoxBytes, &mapQ, bars + F2_Q, 64 * b, q01, hq, bb);
            if (early > 1) load_k(1);
            if (prep.with_bwd)      // (what the end of the job reads: into L2)
                for (int b = 0; b < kBoxes; ++b) {
                    if (want1 > 0) tma_prefetch_4d(&mapdO, 64 * b, q01, hq, bb);
                    tma_prefetch_4d(&mapdO, 64 * b, q00, hq, bb);
                }
        }
    }
    if (warp == 11 && elect_one()) {
        mbar_init(bars + F2_VFULL, 1u);
        mbar_init(bars + F2_VFULL + 1, 1u);
        fence_mbar_init();
        grid_dependency_wait();
        for (int j = 0; j < early; ++j) load_v(j);
    }
    if (tid == 0) {
        for (int b = 0; b < F2_COUNT; ++b) {
            if (b == F2_Q || b == F2_KFULL || b == F2_KFULL + 1 || b == F2_VFULL || b == F2_VFULL + 1) continue;   // (the producers' own)
            const bool of_stream = (b >= F2_P && b < F2_P + 2) || (b >= F2_SFREE && b < F2_SFREE + 2) || (b >= F2_E && b < F2_E + 2);
            mbar_init(bars + b, of_stream ? 128u : 1u);
        }
        *abortp = aligned ? 0u : 1u;
        if (!aligned && status) atomicCAS(status, 0u, (unsigned int)ERR2_ALIGN);
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
    const bool sound = *abortp == 0;      // misaligned shared memory: every role is a no-op
    const int n0 = sound ? want0 : 0, n1 = sound ? want1 : 0;

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");      // (128 x 88 + 256 x 208 = 384 x 168, the launch's registers)
      if (warp == 8) {
        // ------------------------------------------------------------------ TMA producer of K
        if (zero_acc != nullptr) {
            // fused forward+backward: this CTA's rows of the fp32 dQ accumulator ([B*H, n, D]) are cleared while the first loads are in flight
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const int q0 = h ? q01 : q00, rows = (h ? qt1 : qt0) < 0 ? 0 : min(BM, n - q0);
                float4 *dst = reinterpret_cast<float4 *>(zero_acc + ((size_t)bh * n + (rows > 0 ? q0 : 0)) * D);
                for (int i = lane; i < rows * (D / 4); i += 32) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        if (elect_one()) {      // (one thread from here on)
            int nk = early;
            for (int j = early; j < n0; ++j) {
                if (!mbar_wait(bars + F2_KEMPTY + (j & 1), ((j >> 1) - 1) & 1, abortp, status, ERR2_K)) break;
                load_k(j);
                ++nk;
            }
            // Fused call: the streams' dO tiles, which the epilogues multiply their rows with, go into the K slots as these come free: stream 1's
            // into that of the last tile but one (stream 1 ends first), stream 0's into the last tile's.  (Read by the row's owner straight from
            // global memory, 16 bytes of 32 rows at a time, the two tiles were 2 us of LSU work at the end of a job.)
            int armed_do = 0;       // bit h
            if (prep.with_bwd)
#pragma unroll 1
                for (int h = 1; h >= 0; --h) {
                    const int s = (n0 - 1 + h) & 1, uses = (n0 - s + 1) / 2;
                    if ((h ? n1 : n0) == 0) continue;
                    if (uses > 0 && !mbar_wait(bars + F2_KEMPTY + s, (uses - 1) & 1, abortp, status, ERR2_K)) break;
                    mbar_arrive_expect_tx(bars + F2_DO + h, kTileBytes);
                    armed_do |= 1 << h;
                    for (int b = 0; b < kBoxes; ++b) tma_load_4d(sK + s * kTileBytes + b * kBoxBytes, &mapdO, bars + F2_DO + h, 64 * b, h ? q01 : q00, hq, bb);
                }
            if (*abortp) {
                for (int h = 0; h < 2; ++h) mbar_drain_one(bars + F2_DO + h, (armed_do >> h) & 1);
                mbar_drain_one(bars + F2_Q, early > 0 ? 1 : 0);
                for (int s = 0; s < 2; ++s) mbar_drain_one(bars + F2_KFULL + s, nk > s ? (nk - s + 1) / 2 : 0);
            }
        }
      } else if (warp == 11 && elect_one()) {
        // ------------------------------------------------------------------ TMA producer of V
        int nv = early;
        for (int j = early; j < n0; ++j) {
            if (!mbar_wait(bars + F2_VEMPTY + (j & 1), ((j >> 1) - 1) & 1, abortp, status, ERR2_V)) break;
            load_v(j);
            ++nv;
        }
        if (*abortp)
            for (int s = 0; s < 2; ++s) mbar_drain_one(bars + F2_VFULL + s, nv > s ? (nv - s + 1) / 2 : 0);
      } else if ((warp == 9 || (!kOneIssuer && warp == 10)) && elect_one()) {
        // ------------------------------------------- UMMA issuer: scores and O += P V
        // 128 columns: one thread, and the products go through the pipe in the order S(q + 2), P V(q), S(q + 3), ... with q counting the tiles of both streams:
        // what S(q + 2) waits for (the scores of tile q + 1 in registers) comes before P(q), which its warpgroup writes before it loads tile q + 2, which is
        // what S(q + 3) waits for.  A P V is queued behind its S instead of being issued once that has been seen to complete.  Two / one, forward alone, in
        // turn: under the power cap (runs of 40 ms) B1 H16 n16384 1806 / 1784 us at 1567 MHz, B1 H8 n8192 245 / 242, B2 H16 n4096 causal 139.3 / 138.1; at
        // 1965 MHz the last one 125.6 / 122.9.  A query tile that is alone (n1 == 0: the last one of an odd count) is the exception to the order's reason: tile
        // q + 1 is the same warpgroup's, which writes P(q) first, so that P V(q) could go before S(q + 2).  It costs nothing there but in one of the shapes timed
        // (B1 H30 n640 13.28 / 13.02, H74 n384 10.53 / 10.39, H32 n1152 25.4 / 25.4; H64 n640 23.85 / 24.24).  64 columns: two threads, warp 10 for P V, whose
        // products are short and should not wait for a late K tile (B1 H8 n8192 causal 96.9 / 98.9 us, not causal 194.4 / 198.7).
        const bool scores = kOneIssuer || warp == 9, values = kOneIssuer || warp == 10;
        constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, 0, 0), idesc_pv = idesc_bf16_f32(128, 16 * KL, 0, 1);
        const uint64_t km_proto = smem_desc_sw128(0, 16, 1024), mn_proto = smem_desc_sw128(0, kBoxBytes, 1024);
        const uint32_t km_hi = (uint32_t)(km_proto >> 32), mn_hi = (uint32_t)(mn_proto >> 32);
        auto field = [](const void *ptr) { return (smem_u32(ptr) >> 4) & 0x3FFFu; };
        const uint32_t q_lo0 = (uint32_t)km_proto + field(sQ), k_lo0 = (uint32_t)km_proto + field(sK), v_lo0 = (uint32_t)mn_proto + field(sV);
        constexpr uint32_t kSlot = (uint32_t)(kTileBytes >> 4);
        bool ok = n0 > 0 && (!scores || mbar_wait(bars + F2_Q, 0, abortp, status, ERR2_Q));
        int kt = 0, h = 0, pk = 0, ph = 0;      // the tile (key tile, stream) whose scores come next, and whose P V
        int bk = -1, bh0 = 0;                   // the tile of the scores issued last
        const int total = n0 + n1;
        for (int step = 0; ok && step < total + 2; ++step) {
            if (scores && step < total) {
                if (h == 0 && !mbar_wait(bars + F2_KFULL + (kt & 1), (kt >> 1) & 1, abortp, status, ERR2_K)) break;
                // the one score buffer: the tile before is in registers
                if (bk >= 0 && !mbar_wait(bars + F2_SFREE + bh0, bk & 1, abortp, status, ERR2_O)) break;
                tc_fence_after();
                const uint32_t k_lo = k_lo0 + (kt & 1) * kSlot, q_lo = q_lo0 + h * kSlot;
                umma_ss2<false>(tbase + kColS, q_lo, km_hi, k_lo, km_hi, idesc_s);
#pragma unroll
                for (int ks = 1; ks < KL; ++ks) {
                    const uint32_t off = (uint32_t)(((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4);
                    umma_ss2<true>(tbase + kColS, q_lo + off, km_hi, k_lo + off, km_hi, idesc_s);
                }
                if (h == 1 || kt >= n1) umma_commit(bars + F2_KEMPTY + (kt & 1));       // the K tile's last product
                umma_commit(bars + F2_S + 2 * h + (kt & 1));
                bk = kt;
                bh0 = h;
                if (h == 0 && kt < n1) h = 1;
                else { h = 0; ++kt; }
            }
            if (values && step >= 2) {
                if (ph == 0 && !mbar_wait(bars + F2_VFULL + (pk & 1), (pk >> 1) & 1, abortp, status, ERR2_V)) break;
                if (!mbar_wait(bars + F2_P + ph, pk & 1, abortp, status, ERR2_P)) break;
                // (two threads: the scores come first, their UMMAs and these would interleave and both take twice as long)
                if (!kOneIssuer && pk + 1 < (ph ? n1 : n0) && !mbar_wait(bars + F2_S + 2 * ph + ((pk + 1) & 1), ((pk + 1) >> 1) & 1, abortp, status, ERR2_S)) break;
                tc_fence_after();
                const uint32_t v_lo = v_lo0 + (pk & 1) * kSlot, ocol = tbase + kColO + ph * D, acol = tbase + kColP + 64 * ph;
                if (pk > 0) umma_ts2<true>(ocol, acol, v_lo, mn_hi, idesc_pv);
                else        umma_ts2<false>(ocol, acol, v_lo, mn_hi, idesc_pv);
#pragma unroll
                for (int ks = 1; ks < 8; ++ks)
                    umma_ts2<true>(ocol, acol + ks * 8, v_lo + (uint32_t)((ks * 2048) >> 4), mn_hi, idesc_pv);
                umma_commit(bars + F2_OB + ph);
                if (ph == 1 || pk >= n1) umma_commit(bars + F2_VEMPTY + (pk & 1));       // the V tile's last product
                if (ph == 0 && pk < n1) ph = 1;
                else { ph = 0; ++pk; }
            }
        }
      }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
        // ---------------------------------------------------------------- softmax warps: thread = query row (TMEM lane)
        const int h = warp / 4;
        const int lane_row = 32 * (warp % 4) + lane;
        const int q0 = h ? q01 : q00, nk = h ? n1 : n0;
        const int row = q0 + lane_row;
        const uint32_t lane_addr = tbase + ((uint32_t)(32 * (warp % 4)) << 16);
        const uint32_t ocol = kColO + h * D, pcol = kColP + 64 * h;
        float m_used = -1e30f, l = 0.f;
        bool ok = nk > 0;
        for (int t = 0; ok && t < nk; ++t) {
            if (!mbar_wait(bars + F2_S + 2 * h + (t & 1), (t >> 1) & 1, abortp, status, ERR2_S)) { ok = false; break; }
            tc_fence_after();
            const int k0 = t * BN;
            const bool need_mask = (k0 + BN > n) || (causal && k0 + BN - 1 > q0);
            uint32_t r[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld(lane_addr + kColS + 32 * c, r[c]);
            tc_wait_ld();
            tc_fence_before();
            mbar_arrive(bars + F2_SFREE + h);      // the score columns are free: the next product runs under this tile's exponentials
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
            if (t == 0) {
                m_used = (mx == -INFINITY) ? -1e30f : mx;     // (a row past n)
            } else {
                const bool grow = mx > m_used + kRescaleThreshold;
                if (__any_sync(0xffffffffu, grow)) {
                    if (!mbar_wait(bars + F2_OB + h, (t - 1) & 1, abortp, status, ERR2_O)) { ok = false; break; }
                    tc_fence_after();
                    const float alpha = grow ? ex2(m_used - mx) : 1.f;
                    if (grow) m_used = mx;
                    l *= alpha;
#pragma unroll 1
                    for (int c = 0; c < D; c += 16) {   // rare path
                        uint32_t o[16];
                        tmem_ld(lane_addr + ocol + c, o);
                        tc_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st(lane_addr + ocol + c, o);
                    }
                }
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
                // P goes where the stream's P before was: that product has read it by now
                if (c == 0 && t > 0 && !mbar_wait(bars + F2_OB + h, (t - 1) & 1, abortp, status, ERR2_O)) { ok = false; break; }
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
            mbar_arrive(bars + F2_P + h);
        }
        // ---- epilogue of this stream: O / l as bf16 through the stream's Q tile and a TMA store; the row's logsumexp and, in a fused
        // call, the backward's per-row inputs.  (The barrier's phase before is known complete: the loop has waited for it.)
        const bool want_d = prep.with_bwd != 0;
        const uint8_t *drow = sK + ((n0 - 1 + h) & 1) * kTileBytes + lane_row * 128;       // this row of the dO tile
        if (ok && mbar_wait(bars + F2_OB + h, (nk - 1) & 1, abortp, status, ERR2_O) && (!want_d || mbar_wait(bars + F2_DO + h, 0, abortp, status, ERR2_DO))) {
            tc_fence_after();
            const float inv = 1.f / l;
            float dsum = 0.f;
            uint8_t *stage = sQ + h * kTileBytes;
#pragma unroll 1
            for (int c = 0; c < D; c += 32) {
                uint32_t o[32];
                tmem_ld(lane_addr + ocol + c, o);
                tc_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; i += 8) {
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __uint_as_float(o[i + u]) * inv;
                    if (KL < D / 16 && c + i >= 16 * KL)      // columns no product wrote
#pragma unroll
                        for (int u = 0; u < 8; ++u) v[u] = 0.f;
                    const int cabs = c + i, chunk = ((cabs & 63) >> 3) ^ (lane_row & 7);       // 128-byte swizzle, as the maps expect
                    if (want_d) {      // (columns past the head dimension and rows past n are zeros)
                        const uint4 g = *reinterpret_cast<const uint4 *>(drow + (cabs >> 6) * kBoxBytes + chunk * 16);
                        const uint32_t gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float2 gg = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gw[u]));
                            dsum = fmaf(v[2 * u], gg.x, dsum);
                            dsum = fmaf(v[2 * u + 1], gg.y, dsum);
                        }
                    }
                    *reinterpret_cast<uint4 *>(stage + (cabs >> 6) * kBoxBytes + lane_row * 128 + chunk * 16) =
                        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                }
            }
            fence_proxy_async_smem();
            mbar_arrive(bars + F2_E + h);
            if (want_d && row < prep.n_pad) {
                const size_t prow = (size_t)bh * prep.n_pad + row;
                prep.Dp[prow] = row < n ? -dsum : 0.f;
                prep.Lp[prow] = row < n ? -(m_used + log2f(l)) : -INFINITY;
            }
            if (row < n) L[(size_t)bh * n + row] = m_used * kLn2 + logf(l);
            if (tid == 128 * h && mbar_wait(bars + F2_E + h, 0, abortp, status, ERR2_O)) {
                for (int b = 0; b < kBoxes; ++b)
                    if (64 * b < prep.d) tma_store_4d(&mapO, stage + b * kBoxBytes, 64 * b, q0, hq, bb);
                bulk_commit();
                bulk_wait_read<0>();      // shared memory is read before the CTA may exit
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) tmem_dealloc(tbase, kTmemCols);
}

template <int D, int KL>
cudaError_t launch(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb, cudaStream_t st)
{
    constexpr int kSmem = 6 * 128 * D * 2 + 8 * F2_COUNT + 16;
    CUtensorMap mq, mk, mv, mo, mdo;
    const auto bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    // p.d <= D columns exist in memory: loads fill the rest of a box with zeros, the store drops it
    if (!make_tensor_map_4d_strided(&mq, Q, bf, 2, p.B, p.H, p.n, p.d, p.sq.row, p.sq.head, p.sq.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mk, K, bf, 2, p.B, p.kv_heads(), p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mv, V, bf, 2, p.B, p.kv_heads(), p.n, p.d, p.skv.row, p.skv.head, p.skv.batch, 128, 64) ||
        !make_tensor_map_4d_strided(&mo, O, bf, 2, p.B, p.H, p.n, p.d, p.so.row, p.so.head, p.so.batch, 128, 64))
        return cudaErrorInvalidValue;
    mdo = mo;
    if (fb.dO && !make_tensor_map_4d_strided(&mdo, fb.dO, bf, 2, p.B, p.H, p.n, p.d, p.so.row, p.so.head, p.so.batch, 128, 64)) return cudaErrorInvalidValue;
    const cudaError_t e = allow_smem<tc_fwd2_kernel<D, KL>>(kSmem);
    if (e != cudaSuccess) return e;
    const int nqt = (p.n + BM - 1) / BM, npairs = (nqt + 1) / 2;
    LaunchScope scope(MOA_KERNEL_FWD, st);
    return launch_dependent(tc_fwd2_kernel<D, KL>, dim3((unsigned)(npairs * p.BH())), dim3(kThreads), (size_t)kSmem, st, mq, mk, mv, mo, mdo, L,
                            p.n, p.causal, p.scale * kLog2e, npairs, heads_per_group(p, npairs), p.group(), p.H, fb.zero_acc,
                            FwdPrep2{fb.dO != nullptr, fb.Lp, fb.Dp, nqt * BM, p.d}, device_status_ptr());
}

}  // namespace

// Whether pairs of query tiles finish before single ones (tc_fwd.cu), in units of one key tile of one query tile: a job costs about 8
// (9 for a pair) beside its tiles; equal jobs go in rounds over the SMs, causal ones longest first.  Forward alone, single / pairs:
// B2 H16 n4096 d128 causal 145 / 128 us, B1 H16 n16384 1795 / 1780, B4 H8 n1024 d64 20.6 / 16.1, B4 H32 n200 causal 13.4 / 8.2, but
// B1 H8 n2048 18.4 / 30.1 (64 pairs on 148 SMs) and B1 H32 n512 causal 9.1 / 10.8; close to the line B1 H32 n1024 causal 17.6 / 17.9, H8 n4096 62.5 / 61.5.
bool fwd_pairs_pay(const Problem &p)
{
    const long long sms = device_info().sms, nqt = (p.n + BM - 1) / BM, np = (nqt + 1) / 2, bh = p.BH();
    auto cost = [&](long long jobs, double longest, double total, double fixed) {
        const double even = (double)((jobs + sms - 1) / sms) * (longest + fixed), avg = (total + (double)jobs * fixed) / (double)sms;
        const double packed = avg + 0.2 * (total / (double)jobs + fixed), last = longest + fixed;
        return !p.causal ? even : last > packed ? last : packed < even ? packed : even;
    };
    const double total = (double)bh * (p.causal ? nqt * (nqt + 1) / 2 : nqt * nqt);
    const double one = cost(bh * nqt, (double)nqt, total, 8.0);
    const double two = cost(bh * np, (double)(nqt == 1 ? 1 : p.causal ? 2 * nqt - 1 : 2 * nqt), total, 9.0);
    return two < 0.98 * one;
}

cudaError_t tc_fwd_pairs(const Problem &p, const void *Q, const void *K, const void *V, void *O, float *L, const FwdForBwd &fb, cudaStream_t st)
{
    if (p.d < 8 || p.d > 128 || p.d % 8) return cudaErrorInvalidValue;
    if (p.d <= 64) return launch<64, 4>(p, Q, K, V, O, L, fb, st);
    return p.d <= 96 ? launch<128, 6>(p, Q, K, V, O, L, fb, st) : launch<128, 8>(p, Q, K, V, O, L, fb, st);
}

}  // namespace moa
