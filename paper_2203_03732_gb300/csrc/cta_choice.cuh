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

constexpr int kBatch = 256;  // items a CTA of k_phases turns into scan jobs at a time

// Every next-phase row goes to the pool: no CTA of k_phases takes more than
// kBatch rows in a round, so its donations of a round fit its buffer and the
// barrier places them.  (Otherwise CTAs with short rows keep some of theirs.)
PR_HD inline bool all_to_pool(int n_rows, int ctas) { return n_rows <= kBatch * ctas; }

// Small problems.  A round of the grid costs about 4.3 us whatever it does (a
// grid barrier and four or five dependent L2 trips); on one CTA with its
// state in shared memory it costs 0.9 us with a few rows, and grows with the
// rows, since one SM scans them all.  So one CTA runs problems of up to
// kSoloMaxRows rows from the start, and for larger ones the grid runs the
// first, crowded phases and one CTA the rest, from the first phase with at
// most kHandRows free rows (fewer with long rows: kHandBytes of rounded costs
// in all).  Where T is not below that, the grid runs alone.  Solve time, ms,
// eps = 0.01 / 0.003, one CTA / take-over / grid: n = 300: 0.46 / 0.47 / 1.44,
// 12.6 / 12.9 / 54; n = 1000: 1.61 / 1.60 / 3.93, 8.8 / 8.6 / 24.7; n = 2000:
// 1.70 / 1.44 / 2.23, 16.4 / 14.3 / 30.6; n = 4000: 3.85 / 2.53 / 2.79, 36 /
// 24.0 / 27.4; 1000 x 1500: 0.23 / 0.13 / 0.17, 0.72 / 0.41 / 0.63.  Half or
// twice the rows or bytes was slower; rows past kHandRowBytes as well (n =
// 6000 in 16 bits: 43.0 against 41.8).
constexpr int kSoloMaxRows = 384;
constexpr int kHandRows = 64, kHandBytes = 256 * 1024, kHandRowBytes = 8192;
// At floor(1/eps) <= kNearMaxK most of a solve can be one phase of a hundred
// rounds in which hundreds of rows lose the same columns (squared distances, n
// = 1000, eps = 0.1: 131 rounds of 464 rows).  The grid's rounds cost 4.3 us,
// one CTA's 2.3 us at 512 to 1024 rows, so one CTA takes over inside a phase
// that has lasted kMidRounds rounds: that solve 574 -> 347 us, n = 1500 855 -> 552
// us, n = 1000 at eps = 0.3 1545 -> 701 us.  (A problem of 20 rounds is faster on
// the grid: n = 1000, Euclidean, 122 us against 153 us on one CTA; at n = 2000
// such a problem is 8 % slower with the take-over, 228 against 210 us.)
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
// rows at which a solve stops; coarse: floor(1/eps) <= 20; ctas: the grid that
// the phase loop would run on; mode: PR_PHASE_MODE or null.
inline CtaChoice choose_cta(bool seq, int n_rows, int row_bytes, int T, bool coarse, int ctas, const char *mode) {
    CtaChoice c;
    if (mode && (strcmp(mode, "grid") == 0 || strcmp(mode, "cluster") == 0)) return c;
    if (mode ? strcmp(mode, "solo") == 0 : n_rows <= kSoloMaxRows && !seq) {
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
    c.mid = !seq && coarse && n_rows <= kMidRows;
    return c;
}

}  // namespace prot
