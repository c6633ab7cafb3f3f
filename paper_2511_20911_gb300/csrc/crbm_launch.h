// Launch shapes by sizes: what the launchers and the context take before a
// call chooses otherwise.  Host code without CUDA calls.
#pragma once

#include <algorithm>
#include <cmath>

#include "crbm_internal.h"

namespace crbm {

// ---- warps per CTA of the SMEM sweeps
// Bit-plane sweep: with less than three words per SM one round of node groups, up
// to 16 warps, finishes a word's half-step soonest; with more, smaller CTAs, of
// which more are resident, fill each other's barriers; the smallest lattices
// take so few warps that every word is resident, else the words queue at the
// scheduler (us per sweep with 4, 3, 1 warps,
// 1600 words: L = 4 9.1 4.4 4.4, L = 6 9.6 5.8 6.0, L = 8 10.4 7.0 7.4, L = 12 13.8
// 14.0 14.4; 3000 words: 12.3 10.8 7.5, 14.0 12.4 10.2, 15.6 14.0 12.5, 23.9
// 23.1 24.0).
// Generic sweep (us per sweep with 4, 8, 16 warps, 48 words of 18 x 12
// spins: 8.8 6.2 5.4, 304 words: 11.7 9.8 10.7, 600 words: 18.7 19.1 21.1, of 9 x 9
// spins 9.1 10.0 11.5): fewer warps the more words an SM has.  The canonical sweep, by whether every SM has two
// words or more (us per sweep of 384 words with 4, 8, 12, 16 warps: L = 6 2.65
// 2.81, L = 12 6.07 6.07 5.42 5.50, L = 18 11.5 10.6 11.0 11.4, L = 24 21.1 18.7 -
// 18.5, L = 30 32.6 29.1 28.8 28.4; of 152 words with 8, 16, 32: L = 18 5.1 4.6
// 4.7, L = 48 30.1 26.6 26.4, L = 64 74.4 50.2 47.6; L = 6, every sweep measured:
// 1.29 with 9 warps, 1.20 with 12, one of them free to finish the measurements).
// Between L = 12 and 18 the 8 and 12 warps are close (304 words of L = 14, 49 cells:
// 6.10, 5.97; 600 words of L = 16, 64 cells: 12.9, 13.1; in paper precision 4.24,
// 4.23; 8.98, 9.43), which is where the line lies; paper precision keeps the order.
// With correlations beyond L = 34, 32 warps: a sample takes as long as 20 to 40
// sweeps there, waiting for its popcounts, and the sweep itself loses nothing (us
// per sweep with a sample each, 16 -> 32 warps: L = 36, 1 word 228 -> 156, L = 48,
// 384 words 1730 -> 1133; a sample every 100: 16.9 -> 16.6, 84.8 -> 79.3).
inline int sweep_warps(const Geometry& g, int n_words, int sms, bool correlations) {
    if (g.bitplane) {
        const int groups = (g.n_cells * 10 + 31) / 32;
        const int round = (groups + 3) & ~3;  // one round of hidden groups
        const int per = (n_words + sms - 1) / sms;  // words of the fullest SM; 36 warps of 56 registers a thread fit
        const int w = n_words >= 5 * sms   ? (groups > 12 ? 8 : groups > 8 || per <= 9 ? 4 : per <= 12 || groups > 5 ? 3 : 1)
                      : n_words >= 3 * sms ? (groups <= 12 ? std::min(8, round) : 12)
                      : groups <= 16       ? std::min(12, round)
                                           : std::min(16, (g.n_cells + 5) / 6);
        return std::max(1, std::min(kMaxSweepWarps, w));
    }
    if (!g.canonical)
        return std::max(1, std::min(std::min(n_words <= sms ? 16 : n_words < 3 * sms || g.n_cells >= 64 ? 8 : 4, kMaxSweepWarps),
                                    g.n_cells));
    if (correlations && g.L > 34) return std::min(kMaxSweepWarps, 32);
    if (n_words >= 2 * sms && g.n_cells <= 400)  // (larger ones hold one CTA per SM)
        return std::min(kMaxSweepWarps, g.n_cells < 16 ? 4 : g.n_cells < 30 || (g.n_cells >= 50 && g.n_cells <= 144) ? 8 : 12);
    return std::min(kMaxSweepWarps, g.n_cells < 8 ? 8 : g.n_cells <= 16 ? 12 : g.n_cells <= 600 || 2 * n_words <= sms ? 16 : 32);
}

// ---- batched launch: warps per CTA of members at their rules' shapes
// With a CTA per SM at most, the largest member's (`warps`).  With more, so many
// that registers (128 a thread) let as many CTAs share an SM as shared memory
// does, up to four and to the CTAs per SM: a CTA alone on its SM waits at its
// barriers, and CTAs wait for SMs (us per sweep, 16 or 12 warps -> by this rule:
// 600 words of L = 12 37.9 -> 14.9, 150 of L = 18 and 100 of L = 12 31.2 -> 13.7,
// 300 of L = 6 and 300 of L = 8 4.3 -> 3.3, 200 of L = 30 39.7 -> 23.7, 400 of
// 9 x 9 7.9 -> 7.3, 300 of L = 18 in paper precision 5.8 -> 5.7).
inline int batch_warps(int warps, int n_ctas, size_t smem, int sms) {
    const int per = (n_ctas + sms - 1) / sms, fit = static_cast<int>(228 * 1024 / (smem + kReservedSmem));
    const int share = std::min(std::min(per, fit), 4);
    return share <= 1 ? warps : std::min(warps, share == 2 ? 8 : 4);
}

// ---- streamed lane-uniform sweep: tiles of `rows` rows of cells by `seg`
// segments of three, rows in {4, 8, 16}, seg in {4, 5, 6}
constexpr int kTileRows = 16, kMaxTileSeg = 6;
struct RowCut {
    int seg, rows;
    int64_t tiles(const Geometry& g, int n_words) const {
        return static_cast<int64_t>((g.W + rows - 1) / rows) * ((g.Wc + 3 * seg - 1) / (3 * seg)) * n_words;
    }
};
// The half-steps' cut: the width that pads the lattice least, then the rows
// with the least time of the fullest SM: the staging and cells of its k CTAs, and
// the latency of one CTA, which grows less than its cells.  The constants (us)
// are fits to both half-steps timed with every cut, 64 x 64 .. 512 x 512 and
// 34 x 2048 spins in 2 .. 64 words; of the rows their choice is within 1.2 % of
// the one of fewest CTAs from four per SM up, and up to 20 % faster.  us per
// sweep with 16, 8 and 4 rows: 384 x 384, 2 words: 39 43 45; 96 x 96, 24 words:
// 31 31 37; 100 x 100, 16 words: 41 33 29.
inline RowCut row_cut(const Geometry& g, int n_words, int sms) {
    RowCut c{5, kTileRows};
    int waste = 1 << 30;
    for (int s = 4; s <= kMaxTileSeg; ++s) {
        const int pad = (g.Wc + 3 * s - 1) / (3 * s) * (3 * s) - g.Wc;
        if (pad < waste || (pad == waste && s == 5)) {
            c.seg = s;
            waste = pad;
        }
    }
    double best = 0.0;
    int rows = kTileRows;
    for (c.rows = kTileRows; c.rows >= 4; c.rows /= 2) {
        const int64_t n = c.tiles(g, n_words), k = (n + sms - 1) / sms;
        const double mean = static_cast<double>(g.n_cells) * n_words / static_cast<double>(n);
        const double most = static_cast<double>(std::min(c.rows, g.W)) * std::min(3 * c.seg, g.Wc);
        const double cost = static_cast<double>(k) * (1.1 + 0.023 * mean + 0.016 * most) + 0.6 * std::sqrt(most);
        if (c.rows == kTileRows || cost <= best) {
            best = cost;
            rows = c.rows;
        }
    }
    c.rows = rows;
    return c;
}
// The count's cut: the half-steps', in taller tiles while a word has more than 64.
// Every tile adds 96 sums to its word's counts, so many small ones queue at the
// same addresses (us per sweep, every sweep counted, with 16, 8 and 4 rows: 256 x
// 256, 2 words: 37 39 43; 512 x 512, 2 words: 87 97 115; with 21 tiles of 8 rows
// a word, 100 x 100 in 32 words: 65 63 65).
inline RowCut count_cut(const Geometry& g, int n_words, int sms) {
    RowCut c = row_cut(g, n_words, sms);
    while (c.rows < kTileRows && c.tiles(g, 1) > 64) c.rows *= 2;
    return c;
}

// ---- canonical SMEM sweep: how a launch with more words than resident CTAs
// runs.  `all`: a CTA per word for the whole launch, placed by the hardware;
// else a persistent grid over (word, chunk of sweeps) items.
struct CanonSchedule {
    bool all;
    int chunk;  // sweeps per item
};
// Persistent: the chunk with the least (rounds of items over the grid of per_sm
// CTAs per SM) x (sweeps + the staging of a word, 0.7 sweeps on the L=18 grid:
// 5.79 ms per 500 sweeps in chunks of 8, 5.56 in chunks of 16).  It balances the
// SMs, at a staging and a claim (a scan of every word's state) per item.
// All: where one chunk per word is the best anyway (265 sweeps of 600 words of
// L = 14 on 304 CTAs, us per sweep: claimed 14.5, placed 11.7), and for short
// launches, of up to eight stagings a word, where the fullest SM's words and their
// staging, once for every `resident` of them, cost less.  By estimates (us): a
// word's sweep takes an SM 0.7 + 0.042 a cell, its staging 5 + 0.009 a cell.  us
// per launch of one sweep, persistent -> all, 1600 words: L = 4 191 -> 19, L = 6
// 186 -> 21, L = 12 246 -> 43; 384 words of L = 18 34 -> 21.
inline CanonSchedule canon_schedule(int n_sweeps, int n_words, int n_cells, int sms, int per_sm, int resident) {
    const int64_t grid = static_cast<int64_t>(per_sm) * sms;
    CanonSchedule best{false, n_sweeps};
    int64_t rounds = 0;
    double best_cost = 0.0;
    for (int n_chunks = 1; n_chunks <= 64 && n_chunks <= n_sweeps; ++n_chunks) {
        const int chunk = (n_sweeps + n_chunks - 1) / n_chunks;
        const int64_t items = static_cast<int64_t>(n_words) * ((n_sweeps + chunk - 1) / chunk);
        const double cost = static_cast<double>((items + grid - 1) / grid) * (chunk + 0.7);
        if (n_chunks == 1 || cost < best_cost) {
            best.chunk = chunk;
            best_cost = cost;
            rounds = (items + grid - 1) / grid;
        }
    }
    if (best.chunk >= n_sweeps) return {true, n_sweeps};
    const double sweep = 0.7 + 0.042 * n_cells, stage = 5.0 + 0.009 * n_cells;
    if (sweep * n_sweeps > 8.0 * stage) return best;
    const int most = (n_words + sms - 1) / sms;  // words of the fullest SM
    const double all = most * sweep * n_sweeps + (most + resident - 1) / resident * stage;
    return all <= static_cast<double>(rounds) * (best.chunk * per_sm * sweep + stage) ? CanonSchedule{true, n_sweeps} : best;
}

}  // namespace crbm
