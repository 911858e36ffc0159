// cta_solve.cuh -- the whole main routine of Sec. 2.2 on one problem by one
// CTA, with every piece of state in shared memory.  Used by the batched
// solver (one problem per CTA at a time) and by pr_assign for small problems.
//
// What bounds it: the chain of a round (row load from L2, byte test, shared-
// memory atomics, two CTA barriers), not bandwidth, so everything that a
// round touches except the rounded rows is in shared memory, and a round has
// two barriers and no pass over a list of past proposals:
//   - The word of a column is 32 bits, (round << 16) | (0xFFFF - row), so a
//     proposal is one native shared-memory atomicMax (64-bit ones are not
//     native).  Rounds are renumbered before they reach 2^16.
//   - Every atomicMax that finds the current round's tag names one loser, the
//     higher of the two rows, and queues it with its resume column at once:
//     the next round's rows are exactly that list.
//   - Columns taken in earlier rounds of the phase are a bitmap, so a scan
//     drops all of them with one AND instead of one word lookup each.
//   - Rounds with more than kLaneMin rows per warp give each row to one lane
//     first (up to kLaneSteps steps of one 32-byte load), until at most
//     kLaneFew of a warp's rows are left: where many edges are admissible, and
//     for losers, which resume right after the column they lost, the next
//     candidate is near.  The rows left are scanned by the whole warp.  First
//     rounds of phases stop trying it once most rows turn out to end further.
//   - The first row of a warp's next round is loaded before the round's last
//     barrier (KEEP: one problem alone; with several problems per SM their
//     other warps hide that latency, and it measured 3 % slower).
//
// The 512-problem batch (64 to 2048 rows, eps = 0.01) took 2.59 ms in the
// solver with 64-bit words, past-proposal lists and a word lookup per taken
// candidate; it takes 1.23 ms.  64 problems of 4096 points: 7.0 ms -> 1.19 ms.
// A round of few rows (n = 1000) takes about 1.5 us, of which the scan of a
// row is 0.9 us: instructions of one warp, not its loads.  Measured and left
// out: 4 or 8 lanes per row (the lanes' shared-memory and L1 accesses cost
// less, their instructions more: 14 % slower on the batch), unrolled lane
// steps (instruction-cache misses: 40 % slower).
#pragma once

#include "prot_internal.cuh"
#include "scan_common.cuh"

namespace prot {
namespace {

constexpr int kCtaRowBits = 13;  // a list entry: row | resume column << 13
constexpr int kCtaRowMask = (1 << kCtaRowBits) - 1;
static_assert(kCtaMaxCols < (1 << kCtaRowBits), "rows and resume columns must fit 13 bits (and row words 16)");
// Swept on the 512-problem batch, the 64 point clouds and n = 1000 / 2000 alone:
// 8 steps 3-5 % slower, 32 the same; 2 or 4 rows left over 1-6 % slower; 2 or 8
// rows per warp the same to 10 % slower.
constexpr int kLaneSteps = 16;
constexpr int kLaneFew = 1;
constexpr int kLaneSure = 2;  // steps that run while any row is left
constexpr int kLaneMin = 4;

struct CtaShared {
    int nfl[2];    // rows of this / the next phase
    int nlose[2];  // losers of a round, by round parity
    int nwon[2];   // columns won in this / the previous phase
    int far;       // first rounds: some warp's rows mostly end beyond the lane window
    int total;
    int warp_tot[32];
    unsigned long long bytes, rows, cells;
};

// Dynamic shared memory of one problem: column words, three row lists (this
// phase, next phase, losers), the won columns and the row duals (16 bits
// each), the keys in the stored type, the taken bitmap.  Row counts are
// rounded up to 16 and column counts to kRowAlign, so every region starts
// 16-byte aligned.
struct CtaLayout {
    int rows, cols;  // rounded capacities
    __host__ __device__ CtaLayout(int nB, int nA) : rows((nB + 15) & ~15), cols((nA + kRowAlign - 1) & ~(kRowAlign - 1)) {}
    __host__ __device__ size_t words() const { return 0; }
    __host__ __device__ size_t list(int i) const { return (size_t)cols * 4 + (size_t)i * rows * 4; }
    __host__ __device__ size_t won() const { return list(3); }
    __host__ __device__ size_t y() const { return won() + (size_t)rows * 2; }
    __host__ __device__ size_t keys() const { return y() + (size_t)rows * 2; }
    __host__ __device__ size_t taken(int key_bytes) const { return keys() + (size_t)cols * key_bytes; }
    __host__ __device__ size_t total(int key_bytes) const {
        return (taken(key_bytes) + (size_t)((cols + 31) / 32) * 4 + 15) & ~(size_t)15;
    }
};

// Shared memory a kernel of this solver holds besides the problem's state, at
// most: CtaShared and up to 1024 partial sums of the cost.
constexpr size_t kCtaStaticSmem = 12 * 1024;

struct CtaCounts {
    long long phases, rounds, barriers;
    int free_at_stop;
    bool failed;  // the phase cap was reached
};

// 16-byte load of a rounded row: KEEP leaves it in L1 (one problem whose rows
// come back again and again), otherwise it is streamed.
template <bool KEEP>
__device__ __forceinline__ uint4 cta_ld(const void *p) {
    return KEEP ? ld_nc_v4(p) : ld_nc_na_v4(p);
}

// Target of a row in every lane of a packed word.
template <class CB>
__device__ __forceinline__ uint32_t cta_target(int y) {
    const uint32_t t = (uint32_t)(y - 1);
    return sizeof(CB) == 2 ? (t | (t << 16)) : t * 0x01010101u;
}

// The warp's loads of one chunk: UNROLL 16-byte vectors per lane from column c0.
template <int UNROLL, class CB, bool KEEP>
__device__ __forceinline__ void cta_load(const CB *__restrict__ row, int c0, int ldq, int lane, uint4 (&cv)[UNROLL],
                                         unsigned &bytes) {
    constexpr int W = 16 / (int)sizeof(CB);
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
        const int idx = c0 + (u * 32 + lane) * W;
        if (idx < ldq) cv[u] = cta_ld<KEEP>(row + idx);
    }
    bytes += sizeof(CB) * (unsigned)min(32 * W * UNROLL, ldq - c0);
}

// Lowest candidate (cbar + k == tgt, not before `start`, not taken earlier in
// the phase) of a loaded chunk, or -1.  The vectors are pre-tested two at a
// time, with one ballot for a pair without a candidate.
template <int UNROLL, class CB, bool F7>
__device__ __forceinline__ int cta_test(const uint4 (&cv)[UNROLL], const CB *ks, const unsigned *tk, int c0, int start,
                                        int ldq, uint32_t t, int lane) {
    constexpr int W = 16 / (int)sizeof(CB);
#pragma unroll
    for (int u0 = 0; u0 < UNROLL; u0 += 2) {
        if (u0 && c0 + u0 * 32 * W >= ldq) break;  // the row ends before these vectors
        unsigned flags = 0;
#pragma unroll
        for (int u = u0; u < u0 + 2; ++u) {
            const int idx = c0 + (u * 32 + lane) * W;
            const uint4 kv = *reinterpret_cast<const uint4 *>(ks + (idx < ldq ? idx : 0));
            if (idx < ldq && vec_may_match<CB, F7>(cv[u], kv, t)) flags |= 1u << u;
        }
        if (!__any_sync(0xFFFFFFFFu, flags != 0)) continue;
#pragma unroll
        for (int u = u0; u < u0 + 2; ++u) {
            const int idx = c0 + (u * 32 + lane) * W;
            unsigned m = 0;
            if (flags & (1u << u)) {
                m = vec_marks<CB, F7>(cv[u], *reinterpret_cast<const uint4 *>(ks + idx), t);
                const int lo = start - idx;
                if (lo > 0) m &= lo >= W ? 0u : ~0u << lo;
                m &= ~(tk[idx >> 5] >> (idx & 31));
            }
            const unsigned any = __ballot_sync(0xFFFFFFFFu, m != 0);
            if (any) return __shfl_sync(0xFFFFFFFFu, idx + __ffs(m) - 1, __ffs(any) - 1);
        }
    }
    return -1;
}

// Lowest candidate of the row from column `from` on, by the whole warp; -1 if none.
template <int UNROLL, class CB, bool F7, bool KEEP>
__device__ __forceinline__ int cta_scan_row(const CB *__restrict__ row, const CB *ks, const unsigned *tk, int from,
                                            int ldq, uint32_t t, int lane, unsigned &bytes) {
    constexpr int W = 16 / (int)sizeof(CB);
#pragma unroll 1
    for (int c0 = from; c0 < ldq; c0 += 32 * W * UNROLL) {
        uint4 cv[UNROLL];
        cta_load<UNROLL, CB, KEEP>(row, c0, ldq, lane, cv, bytes);
        const int a = cta_test<UNROLL, CB, F7>(cv, ks, tk, c0, from, ldq, t, lane);
        if (a >= 0) return a;
    }
    return -1;
}

// The views of the shared-memory regions.
template <class CB>
struct CtaState {
    unsigned *pw;   // column words
    int *la, *lb, *lq;  // this phase's rows (then losers), the next phase's rows, losers
    uint16_t *won, *y;
    CB *ks;
    unsigned *tk;
    __device__ CtaState(unsigned char *dyn, const CtaLayout &L)
        : pw(reinterpret_cast<unsigned *>(dyn + L.words())),
          la(reinterpret_cast<int *>(dyn + L.list(0))),
          lb(reinterpret_cast<int *>(dyn + L.list(1))),
          lq(reinterpret_cast<int *>(dyn + L.list(2))),
          won(reinterpret_cast<uint16_t *>(dyn + L.won())),
          y(reinterpret_cast<uint16_t *>(dyn + L.y())),
          ks(reinterpret_cast<CB *>(dyn + L.keys())),
          tk(reinterpret_cast<unsigned *>(dyn + L.taken((int)sizeof(CB)))) {}
};

// Counters at the start of cta_phases or cta_seq_phases, the first list
// holding nf rows; the taken set empty.  Barrier before and after by the
// caller.
template <class CB>
__device__ __forceinline__ void cta_begin(CtaShared &s, const CtaState<CB> &c, int ldq, int nf) {
    for (int w = threadIdx.x; w < (ldq + 31) / 32; w += blockDim.x) c.tk[w] = 0;
    if (threadIdx.x == 0) {
        s.nfl[0] = nf;
        s.nfl[1] = s.nlose[0] = s.nlose[1] = s.nwon[0] = s.nwon[1] = 0;
        s.far = 0;
        s.bytes = s.rows = s.cells = 0;
    }
}

// Initialisation of a solve (Sec. 2.2): y(b) = eps, y(a) = 0, M empty, B' = B.
template <class CB>
__device__ __forceinline__ void cta_init(CtaShared &s, const CtaState<CB> &c, int nB, int nA, int ldq) {
    cta_begin(s, c, ldq, nB);
    for (int a = threadIdx.x; a < ldq; a += blockDim.x) c.ks[a] = a < nA ? (CB)0 : (CB)(sizeof(CB) == 1 ? 0xFF : kPadKey);
    for (int a = threadIdx.x; a < nA; a += blockDim.x) c.pw[a] = 0;  // round 0: never won
    for (int b = threadIdx.x; b < nB; b += blockDim.x) {
        c.y[b] = 1;
        c.la[b] = b;
    }
}

// Runs the phases from `nf` rows in the first list and round tags up to
// `R`; `out` carries the counts on.  With mid > 0 it goes on inside a phase
// whose next round has the `mid` rows of the first list: the taken set, the
// won columns and the next phase's list (and their counters) hold that
// phase's so far.  On return the words, row duals and keys hold the result.
// Every thread of the CTA calls it, after a barrier.
template <int UNROLL, class CB, bool F7, bool KEEP>
__device__ __forceinline__ void cta_phases(CtaShared &s, const CtaState<CB> &st, const CB *__restrict__ cb, int nB,
                                           int nA, int ldq, int T, long long cap, unsigned R, int nf, int mid, CtaCounts &out) {
    constexpr int W = 16 / (int)sizeof(CB);
    unsigned *const pw = st.pw, *const tk = st.tk;
    int *la = st.la, *lb = st.lb, *const lq = st.lq;
    uint16_t *const won = st.won, *const y = st.y;
    CB *const ks = st.ks;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;

    int cur = 0;
    bool near = true;  // the same in every thread: read between a round's two barriers
    bool loaded = false;  // cv holds the first chunk of entry e0, this warp's first row of the round
    int e0 = 0;
    uint4 cv[UNROLL];
    unsigned long long my_cells = 0, my_rows = 0, my_bytes = 0;
    while (mid > 0 || nf > T) {
        if (mid == 0 && out.phases >= cap) {
            out.failed = true;
            break;
        }
        ++out.phases;
        if (R + (unsigned)nB + 2u > 0xFFFFu) {  // a phase has at most nB + 1 rounds
#pragma unroll 1
            for (int a = tid; a < nA; a += nthr)
                if (pw[a]) pw[a] = 0x10000u | (pw[a] & 0xFFFFu);
            R = 1;
            __syncthreads();
        }
        const unsigned Rps = mid ? R : R + 1;
        const int pp = (int)(out.phases & 1), nxt = cur ^ 1;
        int items = mid ? mid : nf, nwon_seen = mid ? s.nwon[pp] : 0, q = 0;
        if (mid) {
            mid = 0;
            __syncthreads();  // every thread has read the won count
        }
        const int *in = la;
        int *lose = lq;
        for (;;) {
            ++R;
            const bool later = R > Rps;
            const unsigned Rhi = R << 16;
            const bool by_lanes = items > kLaneMin * nwarps && (later || near);
            // one column's proposal by one lane; returns the row that lost it, or -1
            auto propose = [&](int b, int a) -> int {
                const unsigned old = atomicMax(pw + a, Rhi | (0xFFFFu - (unsigned)b));
                const unsigned t = old >> 16;
                const int orow = 0xFFFF - (int)(old & 0xFFFFu);
                if (t == R) return max(b, orow);
                // first proposal: a is won this round (step III a at the phase
                // end).  Its partner is evicted (step II) and resumes after
                // a: every column <= a is above its unchanged target for good.
                won[atomicAdd(&s.nwon[pp], 1)] = (uint16_t)a;
                if (t) lb[atomicAdd(&s.nfl[nxt], 1)] = orow | ((a + 1) << kCtaRowBits);
                return -1;
            };
            unsigned bytes = 0, cells = 0;
            if (by_lanes) {
#pragma unroll 1
                for (int i0 = warp * 32; i0 < items; i0 += nthr) {
                    const int it = i0 + lane;
                    const bool act = it < items;
                    const int e = act ? in[it] : 0;
                    const int b = e & kCtaRowMask, start = e >> kCtaRowBits;
                    const uint32_t t = cta_target<CB>(y[b]);
                    const CB *row = cb + (size_t)b * ldq;
                    int a = -1, c = start & ~(2 * W - 1);
                    unsigned from = ~0u << (start - c);
                    bool go = act && c < ldq;
#pragma unroll 1
                    for (int k = 0; k < kLaneSteps; ++k) {
                        if (go) {
                            uint4 v0, v1;
                            ld_nc_v8(row + c, v0, v1);
                            bytes += 32;
                            const uint4 *kv = reinterpret_cast<const uint4 *>(ks + c);
                            unsigned m = vec_marks<CB, F7>(v0, kv[0], t) | (vec_marks<CB, F7>(v1, kv[1], t) << W);
                            m &= from & ~(tk[c >> 5] >> (c & 31));
                            from = ~0u;
                            if (m) a = c + __ffs(m) - 1;
                            c += 2 * W;
                            go = a < 0 && c < ldq;
                        }
                        const int n = __popc(__ballot_sync(0xFFFFFFFFu, go));
                        if (n == 0 || (n <= kLaneFew && k >= kLaneSure)) break;
                    }
                    if (!later && __popc(__ballot_sync(0xFFFFFFFFu, act && a >= 0)) < 8 && lane == 0) s.far = 1;
                    // rows not settled: the whole warp scans each from where its lane stopped
                    unsigned left = __ballot_sync(0xFFFFFFFFu, go);
#pragma unroll 1
                    while (left) {
                        const int l = __ffs(left) - 1;
                        left &= left - 1;
                        const int bl = __shfl_sync(0xFFFFFFFFu, b, l), cl = __shfl_sync(0xFFFFFFFFu, c, l);
                        const uint32_t tl = __shfl_sync(0xFFFFFFFFu, t, l);
                        unsigned by = 0;
                        const int al =
                            cta_scan_row<UNROLL, CB, F7, KEEP>(cb + (size_t)bl * ldq, ks, tk, cl, ldq, tl, lane, by);
                        if (lane == l) {
                            a = al;
                            bytes += by;
                        }
                    }
                    if (act) cells += a >= 0 ? (unsigned)(a - start + 1) : (start < nA ? (unsigned)(nA - start) : 0u);
                    // proposals, all lanes together: lanes that share the first
                    // lane's column (losers of one column often do) send their
                    // lowest row only
                    int loser = -1, won_a = -1, next_e = -1;
                    const unsigned has = __ballot_sync(0xFFFFFFFFu, a >= 0);
                    if (has) {
                        const int af = __shfl_sync(0xFFFFFFFFu, a, __ffs(has) - 1);
                        const unsigned low =
                            __reduce_min_sync(0xFFFFFFFFu, a == af ? (unsigned)b : 0xFFFFFFFFu);
                        if (a >= 0) {
                            if (a == af && (unsigned)b != low) {
                                loser = b;
                            } else {
                                const unsigned old = atomicMax(pw + a, Rhi | (0xFFFFu - (unsigned)b));
                                const unsigned tag = old >> 16;
                                const int orow = 0xFFFF - (int)(old & 0xFFFFu);
                                if (tag == R) {
                                    loser = max(b, orow);
                                } else {
                                    won_a = a;
                                    if (tag) next_e = orow | ((a + 1) << kCtaRowBits);
                                }
                            }
                        }
                        __syncwarp();
                    }
                    if (act && a < 0) {  // step (III b): relabel
                        y[b] += 1;
                        next_e = b;
                    }
                    // the three lists' places in one shared-memory trip: lane 0
                    // takes the losers', lane 1 the won columns', lane 2 the
                    // next phase's
                    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, loser >= 0);
                    const unsigned m1 = __ballot_sync(0xFFFFFFFFu, won_a >= 0);
                    const unsigned m2 = __ballot_sync(0xFFFFFFFFu, next_e >= 0);
                    int base = 0;
                    if (lane < 3) {
                        int *cnt = lane == 0 ? &s.nlose[q ^ 1] : lane == 1 ? &s.nwon[pp] : &s.nfl[nxt];
                        base = atomicAdd(cnt, __popc(lane == 0 ? m0 : lane == 1 ? m1 : m2));
                    }
                    const unsigned below = (1u << lane) - 1u;
                    const int b0 = __shfl_sync(0xFFFFFFFFu, base, 0), b1 = __shfl_sync(0xFFFFFFFFu, base, 1),
                              b2 = __shfl_sync(0xFFFFFFFFu, base, 2);
                    if (loser >= 0) lose[b0 + __popc(m0 & below)] = loser | ((a + 1) << kCtaRowBits);
                    if (won_a >= 0) won[b1 + __popc(m1 & below)] = (uint16_t)won_a;
                    if (next_e >= 0) lb[b2 + __popc(m2 & below)] = next_e;
                }
            } else {
#pragma unroll 1
                for (int it = warp; it < items; it += nwarps) {
                    if (it != warp || !loaded) {
                        e0 = in[it];
                        cta_load<UNROLL, CB, KEEP>(cb + (size_t)(e0 & kCtaRowMask) * ldq, (e0 >> kCtaRowBits) & ~(W - 1),
                                                   ldq, lane, cv, bytes);
                    }
                    const int b = e0 & kCtaRowMask, start = e0 >> kCtaRowBits;
                    const uint32_t t = cta_target<CB>(y[b]);
                    int a = -1;
#pragma unroll 1
                    for (int c0 = start & ~(W - 1); c0 < ldq;) {
                        a = cta_test<UNROLL, CB, F7>(cv, ks, tk, c0, start, ldq, t, lane);
                        c0 += 32 * W * UNROLL;
                        if (a >= 0 || c0 >= ldq) break;
                        cta_load<UNROLL, CB, KEEP>(cb + (size_t)b * ldq, c0, ldq, lane, cv, bytes);
                    }
                    if (lane == 0) {
                        cells += a >= 0 ? (unsigned)(a - start + 1) : (start < nA ? (unsigned)(nA - start) : 0u);
                        if (a >= 0) {
                            const int loser = propose(b, a);
                            if (loser >= 0) lose[atomicAdd(&s.nlose[q ^ 1], 1)] = loser | ((a + 1) << kCtaRowBits);
                        } else {
                            y[b] += 1;  // step (III b): relabel
                            lb[atomicAdd(&s.nfl[nxt], 1)] = b;
                        }
                    }
                }
                if (lane != 0) bytes = 0;  // counted once a warp
            }
            my_cells += cells;
            my_bytes += bytes;
            if (tid == 0) my_rows += (unsigned)items;
            ++out.barriers;
            __syncthreads();
            const int nwon = s.nwon[pp], nlose = s.nlose[q ^ 1];
            if (s.far) near = false;
            // the next round's rows are known (the losers, or the next phase's
            // list): each warp issues its first row's loads here, so their
            // latency runs beside the key update and the second barrier
            nf = s.nfl[nxt];
            {
                const int *next = nlose ? lose : lb;
                const int count = nlose ? nlose : nf;
                loaded = KEEP && warp < count && !(count > kLaneMin * nwarps && (nlose || near));
                if (loaded) {
                    unsigned by = 0;
                    e0 = next[warp];
                    cta_load<UNROLL, CB, KEEP>(cb + (size_t)(e0 & kCtaRowMask) * ldq, (e0 >> kCtaRowBits) & ~(W - 1), ldq,
                                               lane, cv, by);
                    if (lane == 0) my_bytes += by;
                }
            }
            if (nwon > nwon_seen) ++out.rounds;  // a proposal was made: some column was won
            if (nlose == 0) {
                // the phase is over: step (III a), y(a) -= eps for the columns
                // won in it; the taken set (columns won before this round) empties
#pragma unroll 1
                for (int i = tid; i < nwon; i += nthr) {
                    const int a = won[i];
                    ks[a] += (CB)1;
                    if (i < nwon_seen) tk[a >> 5] = 0;
                }
                if (tid == 0) {
                    s.nfl[cur] = 0;       // read at the phase start, filled next phase
                    s.nwon[pp ^ 1] = 0;   // the previous phase's
                    s.nlose[q] = 0;
                }
                __syncthreads();
                break;
            }
#pragma unroll 1
            for (int i = nwon_seen + tid; i < nwon; i += nthr) atomicOr(tk + (won[i] >> 5), 1u << (won[i] & 31));
            if (tid == 0) s.nlose[q] = 0;  // this round's list has been read
            nwon_seen = nwon;
            items = nlose;
            int *t = const_cast<int *>(in);  // the list just read takes the next losers
            in = lose;
            lose = t;
            q ^= 1;
            __syncthreads();
        }
        int *t = la;
        la = lb;
        lb = t;
        cur = nxt;
    }
    out.free_at_stop = nf;
    warp_count(&s.cells, my_cells);
    warp_count(&s.bytes, my_bytes);
    warp_count(&s.rows, my_rows);
    __syncthreads();
}

// The same with the sequential greedy as step (I) (rule_seq.cuh: chains on
// phase-tagged words; the result does not depend on their order).  A warp per
// row; `ph` is the tag of the last phase run.
template <int UNROLL, class CB, bool F7>
__device__ __forceinline__ void cta_seq_phases(CtaShared &s, const CtaState<CB> &st, const CB *__restrict__ cb, int nA,
                                               int ldq, int T, long long cap, unsigned ph, int nf, CtaCounts &out) {
    constexpr int W = 16 / (int)sizeof(CB);
    unsigned *const pw = st.pw, *const tk = st.tk;
    int *la = st.la, *lb = st.lb;
    uint16_t *const won = st.won, *const y = st.y;
    CB *const ks = st.ks;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
    int cur = 0;
    unsigned long long my_cells = 0, my_bytes = 0;  // lane 0's
    while (nf > T) {
        if (out.phases >= cap) {
            out.failed = true;
            break;
        }
        ++out.phases;
        if (ph == 0xFFFFu) {  // tags are 16 bits: earlier phases' become 1
#pragma unroll 1
            for (int a = tid; a < nA; a += nthr)
                if (pw[a]) pw[a] = 0x10000u | (pw[a] & 0xFFFFu);
            ph = 1;
            __syncthreads();
        }
        ++ph;
        const int pp = (int)(out.phases & 1), nxt = cur ^ 1;
#pragma unroll 1
        for (int it = warp; it < nf; it += nwarps) {
            int b = la[it] & kCtaRowMask, start = la[it] >> kCtaRowBits;
#pragma unroll 1
            for (;;) {  // one chain: row b from column start, then any row it displaces
                const CB *row = cb + (size_t)b * ldq;
                const uint32_t t = cta_target<CB>(y[b]);
                const int first = start;
                int found = -1;
                unsigned old = 0, bytes = 0;
                uint4 cv[UNROLL];
#pragma unroll 1
                for (int c0 = start & ~(W - 1); c0 < ldq && found < 0; c0 += 32 * W * UNROLL) {
                    cta_load<UNROLL, CB, true>(row, c0, ldq, lane, cv, bytes);
                    int a;
#pragma unroll 1
                    while ((a = cta_test<UNROLL, CB, F7>(cv, ks, tk, c0, start, ldq, t, lane)) >= 0) {
                        if (lane == 0) old = atomicMax(pw + a, (ph << 16) | (0xFFFFu - (unsigned)b));
                        old = __shfl_sync(0xFFFFFFFFu, old, 0);
                        if (old >> 16 != ph || 0xFFFF - (int)(old & 0xFFFFu) > b) {
                            found = a;
                            break;
                        }
                        start = a + 1;  // a lower row holds it
                    }
                }
                if (lane == 0) {
                    my_cells += found >= 0 ? (unsigned)(found - first + 1) : (first < nA ? (unsigned)(nA - first) : 0u);
                    my_bytes += bytes;
                }
                const int other = 0xFFFF - (int)(old & 0xFFFFu);
                if (found >= 0 && old >> 16 == ph) {  // a higher row is displaced: its columns before found are settled
                    b = other;
                    start = found + 1;
                    continue;
                }
                if (lane == 0) {
                    if (found >= 0) {  // found enters M' now; its partner in M, if any, leaves M
                        won[atomicAdd(&s.nwon[pp], 1)] = (uint16_t)found;
                        if (old >> 16) lb[atomicAdd(&s.nfl[nxt], 1)] = other | ((found + 1) << kCtaRowBits);
                    } else {  // y(b) += eps, next phase from column 0
                        y[b] += 1;
                        lb[atomicAdd(&s.nfl[nxt], 1)] = b;
                    }
                }
                break;
            }
        }
        ++out.barriers;
        __syncthreads();
        const int nwon = s.nwon[pp];
        nf = s.nfl[nxt];
#pragma unroll 1
        for (int i = tid; i < nwon; i += nthr) ks[won[i]] += (CB)1;
        if (tid == 0) {
            s.nfl[cur] = 0;      // read at the phase start, filled next phase
            s.nwon[pp ^ 1] = 0;  // the previous phase's
        }
        __syncthreads();
        int *t = la;
        la = lb;
        lb = t;
        cur = nxt;
    }
    out.rounds = out.phases;
    out.free_at_stop = nf;
    warp_count(&s.cells, my_cells);
    warp_count(&s.bytes, my_bytes);
    __syncthreads();
}

__device__ __forceinline__ int cta_scan_excl(int flag, CtaShared &s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, flag);
    const int within = __popc(bal & ((1u << lane) - 1));
    if (lane == 0) s.warp_tot[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
        const int v = lane < nw ? s.warp_tot[lane] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane < nw) s.warp_tot[lane] = x - v;
        if (lane == 31) s.total = x;
    }
    __syncthreads();
    const int r = s.warp_tot[warp] + within;
    __syncthreads();
    return r;
}

// After cta_phases: matching out of the words, completion (the k-th free row
// takes the k-th free column, Sec. 2.1), duals and the FP64 cost, each to
// global memory.  The cost is summed as `sums` strided partial sums (a power
// of two; threads past it idle) and a halving tree over them, in `part`
// (shared memory, `sums` doubles), so its order depends on `sums` alone.
template <class CB, class Cost>
__device__ __forceinline__ void cta_finish(CtaShared &s, unsigned char *dyn, const CtaLayout &L, int nB, int nA,
                                           double *part, int sums, const Cost &cost_of, int *row_to_col,
                                           int *col_to_row, int *y_row, int *y_col, double *cost) {
    int *ma = reinterpret_cast<int *>(dyn + L.words());  // in place of the words
    int *mb = reinterpret_cast<int *>(dyn + L.list(0));
    int *free_b = reinterpret_cast<int *>(dyn + L.list(1));
    int *free_a = reinterpret_cast<int *>(dyn + L.list(2));
    const uint16_t *y = reinterpret_cast<const uint16_t *>(dyn + L.y());
    const CB *ks = reinterpret_cast<const CB *>(dyn + L.keys());
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int b = tid; b < nB; b += nthr) mb[b] = -1;
    __syncthreads();
    for (int a = tid; a < nA; a += nthr) {
        const unsigned w = (unsigned)ma[a];
        const int b = w >> 16 ? 0xFFFF - (int)(w & 0xFFFFu) : -1;
        ma[a] = b;
        if (b >= 0) mb[b] = a;
    }
    __syncthreads();
    int nfb = 0;
    for (int base = 0; base < nB; base += nthr) {
        const int b = base + tid;
        const int f = (b < nB && mb[b] < 0) ? 1 : 0;
        const int pos = cta_scan_excl(f, s);
        if (f) free_b[nfb + pos] = b;
        nfb += s.total;
        __syncthreads();
    }
    int nfa = 0;
    for (int base = 0; base < nA && nfa < nfb; base += nthr) {
        const int a = base + tid;
        const int f = (a < nA && ma[a] < 0) ? 1 : 0;
        const int pos = cta_scan_excl(f, s);
        if (f && nfa + pos < nfb) free_a[nfa + pos] = a;
        nfa += s.total;
        __syncthreads();
    }
    for (int k = tid; k < nfb; k += nthr) {
        mb[free_b[k]] = free_a[k];
        ma[free_a[k]] = free_b[k];
    }
    __syncthreads();
    for (int v = tid; v < sums; v += nthr) {
        double acc = 0.0;
        for (int b = v; b < nB; b += sums) {
            row_to_col[b] = mb[b];
            y_row[b] = y[b];
            acc = __dadd_rn(acc, cost_of(b, mb[b]));
        }
        part[v] = acc;
    }
    for (int a = tid; a < nA; a += nthr) {
        col_to_row[a] = ma[a];
        y_col[a] = -(int)ks[a];
    }
    __syncthreads();
    for (int w = sums / 2; w > 0; w >>= 1) {
        for (int v = tid; v < w; v += nthr) part[v] = __dadd_rn(part[v], part[v + w]);
        __syncthreads();
    }
    if (tid == 0) *cost = part[0];
}

}  // namespace
}  // namespace prot
