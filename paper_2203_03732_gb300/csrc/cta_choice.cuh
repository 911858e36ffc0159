// cta_choice.cuh -- which part of a single solve one CTA runs (k_solo): plain
// C++, so that the rule can be tested without a GPU.
#pragma once

#include <string.h>

#include <algorithm>

#ifdef __CUDACC__
#define PR_HD __host__ __device__
#else
#define PR_HD
#endif

namespace prot {

constexpr long long kNearMaxK = 20;  // floor(1/eps) up to which most of a solve is one phase of many rounds
constexpr int kBatch = 256;  // items a CTA of k_phases turns into scan jobs at a time

// Every next-phase row goes to the pool: no CTA of k_phases takes more than
// kBatch rows in a round, so its donations of a round fit its buffer and the
// barrier places them.  (Otherwise CTAs with short rows keep some of theirs.)
PR_HD inline bool all_to_pool(int n_rows, int ctas) { return n_rows <= kBatch * ctas; }

// Small problems.  A round of the grid costs about 4.3 us whatever it does (a
// grid barrier and four or five dependent L2 trips); on one CTA with its
// state in shared memory a round of a few rows costs about 1.5 us, and more
// with more rows, since one SM scans them all.  So one CTA runs small problems
// from the start (solo_fits), and for larger ones the grid runs the first,
// crowded phases and one CTA the rest, from the first phase with at most
// kHandRows free rows (fewer with long rows: kHandBytes of rounded costs in
// all).  Where T is not below that, the grid runs alone.  Solve time, ms, eps =
// 0.01 / 0.003, one CTA / take-over / grid: n = 300: 0.93 / 0.96 / 3.0, 7.0 /
// 7.1 / 25; n = 1000: 1.61 / 1.60 / 3.93, 8.8 / 8.6 / 24.7; n = 2000: 1.70 /
// 1.44 / 2.23, 16.4 / 14.3 / 30.6; n = 4000: 3.85 / 2.53 / 2.79, 36 / 24.0 /
// 27.4; 1000 x 1500: 0.23 / 0.13 / 0.17, 0.72 / 0.41 / 0.63.  Half or twice the
// rows or bytes was slower; rows past kHandRowBytes as well (n = 6000 in 16
// bits: 43.0 against 41.8).
constexpr int kSoloMaxRows = 384;
constexpr int kHandRows = 64, kHandBytes = 256 * 1024, kHandRowBytes = 8192;

// Whether one CTA is the fastest from the start: few rows, or few phases (at
// larger eps), or about as many columns as rows (long solves of small rounds).
// With columns to spare most rows match in the first phases, which scan whole
// rows: the grid's work.  Time, us, one CTA / take-over / grid:
//   64 rows x 8000 0.01 22 / 31 / 29, 0.003 (16 bits) 51 / 37 / 37; 32 x 8000 0.003 35 / 46 / 46
//   384 x 8000 0.1 54 / 75 / 76, 0.05 49 / 54 / 55, 0.02 59 / 46 / 44, 0.003 253 / 56 / 56
//   200 x 3000 0.02 36 / 35 / 37, 0.01 51 / 37 / 39; 300 x 3000 0.02 42 / 39 / 40
//   384 x 441 (22 K) 0.01 380 / 410, 300 x 450 (45 K) 110 / 119, 300 x 600 (90 K) 71 / 64
inline bool solo_fits(int n_rows, int n_cols, int row_bytes, long long K) {
    if (n_rows > kSoloMaxRows) return false;
    if (n_rows <= 64) return n_rows * row_bytes <= 512 * 1024;
    return K <= kNearMaxK || (K <= 50 && n_rows <= 200) || n_rows * (n_cols - n_rows) <= 48 * 1024;
}

// At floor(1/eps) <= kNearMaxK most of a solve can be one phase of a hundred
// rounds in which hundreds of rows lose the same columns (squared distances, n
// = 1000, eps = 0.1: 131 rounds of 464 rows).  The grid's rounds cost 4 us, one
// CTA's 2 us at 512 to 1024 rows, so one CTA takes over inside a phase that has
// lasted kMidRounds rounds: that solve 534 -> 320 us, n = 1500 835 -> 547 us,
// Euclidean costs, eps = 0.3 497 -> 300 us.  (Problems of 20 to 30 rounds gain
// little: Euclidean, eps = 0.1, grid / take-over / one CTA n = 1000 119 / 109 / 118
// us, n = 1536 164 / 155 / 215.)
constexpr int kMidRows = 1536;

// Whether one CTA runs the problem from the start (solo), takes over from the
// grid once at most `hand` rows are free (0: never), or inside a long phase
// (mid).
struct CtaChoice {
    bool solo = false;
    int hand = 0;
    bool mid = false;
};

// seq: the sequential rule; row_bytes: of a row of rounded costs; T: the free
// rows at which a solve stops; K: floor(1/eps); ctas: the grid that the phase
// loop would run on; mode: PR_PHASE_MODE or null.
inline CtaChoice choose_cta(bool seq, int n_rows, int n_cols, int row_bytes, int T, long long K, int ctas,
                            const char *mode) {
    CtaChoice c;
    if (mode && (strcmp(mode, "grid") == 0 || strcmp(mode, "cluster") == 0)) return c;
    if (!seq && (mode ? strcmp(mode, "solo") == 0 : solo_fits(n_rows, n_cols, row_bytes, K))) {
        c.solo = true;
        return c;
    }
    // the rows that k_solo goes on with are read from the pool (the sequential
    // rule's from its ring, which holds every one)
    if (!seq && !all_to_pool(n_rows, ctas)) return c;
    // the sequential rule: half the bytes, and never from the start (ms, grid /
    // take-over: n = 200, eps = 0.01 2.28 / 0.63, n = 1000, eps = 0.003 24.1 /
    // 9.0, n = 2000, eps = 0.01 1.85 / 1.43; n = 4000, eps = 0.01 with 64 rows of
    // 4 KB 2.10 / 2.26; n = 384, eps = 0.1 on one CTA alone 0.07 / 0.17)
    const int rows = std::min(kHandRows, (seq ? kHandBytes / 2 : kHandBytes) / row_bytes);
    if (row_bytes <= kHandRowBytes && rows > T) c.hand = rows;
    c.mid = !seq && K <= kNearMaxK && n_rows <= kMidRows;
    return c;
}

}  // namespace prot
