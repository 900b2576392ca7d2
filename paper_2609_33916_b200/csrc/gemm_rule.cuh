// Which tile a product of tc_gemm.cu is cut into: plain arithmetic on the host, without CUDA, so that it can be looked at on any machine.
#pragma once

namespace moa {

struct GemmTile {
    int columns;       // 256, 128 or 64
    bool pair;         // on pairs of CTAs (256 columns only)
};

// M, N, K: the product (N: columns of each weight where two are read side by side, `dual`).  a_mn, b_mn: the operand is stored by columns.  plain: nothing
// in the epilogue but an addition; dual: gate forward.  two_pairs: a second operand pair is added into the same tile; nbatch: products in the
// launch.  mode: MOA_GEMM_PAIR (0 never pairs, 2 always pairs, 1 by this rule).
inline GemmTile gemm_tile(long long M, long long N, long long K, bool a_mn, bool b_mn, bool plain, bool dual, bool two_pairs, int nbatch, long long sms, int mode)
{
    // Pairs unless they would need more waves than single CTAs (tiny M); the two gate GEMMs only when the main loop outlasts
    // their epilogue.
    const long long pairs = sms / 2, rows = (M + 127) / 128, K64 = (K + 63) / 64;
    auto tiles = [&](int n) { return rows * ((N + (dual ? n / 2 : n) - 1) / (dual ? n / 2 : n)) * nbatch; };
    const long long pair_tiles = (M + 255) / 256 * (tiles(256) / rows);
    const bool fits = pair_tiles >= 8 && (pair_tiles + pairs - 1) / pairs <= (tiles(256) + sms - 1) / sms;   // (a few tiles: launch-bound)
    // A plain product whose single tiles all run at once, and whose K loop is not long, is over before the pairs' cluster start is paid: pairs / single
    // 4096 x 1024 x 1024 11.1 / 10.0 us, 1300 x 3072 x 1024 11.2 / 10.0, 4096 x 1024 x 3072 (0,1) 21.2 / 20.6, 3072 x 1024 x 1300 (1,1) 12.7 / 12.2; but
    // not where an operand stored by columns comes in by many copies (1024 x 2728 x 1300 (1,1) 13.0 / 14.8), and not where rows of 2 K bytes start off the
    // 32-byte sectors or 64-byte halves of a line: a tile's row then takes one more of them, and a single CTA, which loads all of B's columns instead of half
    // of them, waits for it (4192 x 720 x 1976 18.0 / 22.8, 4080 x 1024 x 1032 12.8 / 14.9, 5312 x 768 x 1800 (1,0) 15.4 / 18.7, 4096 x 1024 x 2064 106 : 100;
    // with B by columns level or better at every K).  Over a short K they stay ahead all the same (pairs : single at K 568 100 : 91, at 784 100 : 98).
    const long long parts = two_pairs ? 2 : 1;
    const bool few_copies = (!a_mn || M % 64 == 0) && (!b_mn || N % 64 == 0);
    const bool whole_rows = b_mn || K % 32 == 0 || (K % 16 == 0 && (a_mn || K64 <= 13)) || K64 <= 9;
    const bool one_wave = plain && tiles(256) <= sms && K64 * parts <= 48 && few_copies && whole_rows;
    const bool pair_ok = mode && fits && !one_wave && (plain || K >= 1024);
    // Where the 256-column tiles leave SMs idle, the narrower ones compete: cycles of a K block (UMMAs at 256 columns, its
    // operands' way from L2 below that), of a chunk of the epilogue, and the rounds the grid takes.  The cycles are of issuers that were not elected; as
    // slopes over K (1024 to 3072, 128 tiles at once, 1965 MHz) a block now takes 287 at 64 columns, 387 to 395 at 128 in every storage order, 690 at 256
    // columns and 655 in pairs (615 and 590 at 64 tiles at once).  The choice holds up: over 70 products of random sizes and storage each width forced is
    // at most 4.5 % faster from K 512 on (368 x 3600 x 2104 (0,1) 14.6 us, 14.0 at 128 columns), up to 14 % below (408 x 3840 x 136 5.7, 5.0 at 128), and
    // for operands that come in by blocks of columns a long K loop at 128 columns loses to pairs (1208 x 5048 x 1664 (1,1) 35.0 us, 27.5 in pairs).
    const double chunk = plain ? 1100 : dual ? 2500 : 3500;
    const double blocks = (double)(K64 * parts);
    auto cost = [&](long long t, long long slots, double block, int n) {
        const double epi = chunk * (dual ? n / 128 : n / 64), main = blocks * block;
        return (double)((t + slots - 1) / slots) * (main > epi ? main : epi) + epi;
    };
    GemmTile g{256, mode == 2 || pair_ok};
    if (mode != 2 && tiles(256) < 2 * sms) {
        double best = g.pair ? cost(pair_tiles, pairs, 530, 256) : cost(tiles(256), sms, 520, 256);
        const double c128 = cost(tiles(128), sms, K64 < 12 ? 360 : a_mn ? 430 : b_mn ? 390 : 360, 128);
        if (c128 < 0.95 * best) { best = c128; g = GemmTile{128, false}; }
        const double c64 = dual ? 1e30 : cost(tiles(64), sms, 290, 64);
        if (c64 < 0.95 * best) g = GemmTile{64, false};
    }
    return g;
}

}  // namespace moa
