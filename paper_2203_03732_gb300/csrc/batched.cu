// batched.cu -- many independent assignment problems in one persistent launch.
//
// Each CTA pulls problems from a queue in longest-first order (LPT on n) and
// runs the whole main routine of Sec. 2.2 on one problem (cta_solve.cuh) with
// every piece of per-problem state in shared memory.  Rounds are separated by
// __syncthreads() instead of a grid barrier.  Only the rounded cost rows are
// read from global memory (HBM / L2).
//
// Problem i is square (n_i rows and columns).  Packed layouts:
//   costs   C[c_off_i + b * n_i + a], c_off_i = sum_{j<i} n_j^2 (rows = B)
//   points  XA[(v_off_i + a) * dim + k], XB[(v_off_i + b) * dim + k]
//   vectors row_to_col[v_off_i + b] (a column of problem i), v_off_i = sum_{j<i} n_j
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <numeric>
#include <type_traits>
#include <vector>

#include "prot_internal.cuh"
#include "scan_common.cuh"
#include "quantise.cuh"
#include "points.cuh"
#include "cta_solve.cuh"

namespace prot {
namespace {

constexpr int kMaxN = 5000;               // largest problem whose state fits shared memory
static_assert(kMaxN <= kCtaMaxCols, "rows and resume columns must fit the CTA solver's list entries");
constexpr int kCostSums = 256;            // partial sums of a problem's cost at the default launch shape
constexpr int kMaxCbarByte = 252;         // byte storage when floor(1/eps) <= 252 (as pr_assign)

struct BDesc {
    long long cb_off;  // element offset of the rounded costs (row stride ldq)
    long long c_off;   // element offset of the cost matrix (matrix source)
    long long cap;     // phase cap
    int n;
    int ldq;
    int v_off;
    int T;
};

struct BCtl {
    WsHead head;
    unsigned queue;
    unsigned pad;
    long long phases;
    long long rounds;
    unsigned long long bytes;
    unsigned long long rows;
};

struct BLayout {
    size_t ctl, desc, order, maxbits, cb, total;
};

BLayout make_blayout(int P, long long cb_elems) {
    BLayout L;
    Carver c;
    L.ctl = c.take<BCtl>(1);
    L.desc = c.take<BDesc>(P);
    L.order = c.take<int>(P);
    L.maxbits = c.take<unsigned>(P);
    L.cb = c.take<uint16_t>((size_t)cb_elems);
    L.total = c.total();
    return L;
}

struct BParams {
    BCtl *ctl;
    const BDesc *desc;
    const int *order;
    const void *cb;  // uint8_t or uint16_t, as k_bsolve is instantiated
    int nprob;
    int n_max;
    int cost_sums;  // strided partial sums of a problem's cost
    // cost source for the reported costs
    const void *C;
    int dt;  // PR_F32 / PR_F64 (matrix source)
    const float *XA, *XB;
    int dim, squared, points;
    // outputs
    int *row_to_col, *col_to_row, *y_row, *y_col;
    double *costs;
    int64_t *phases;
};

// ---------------------------------------------------------------------------
// Rounding of the packed matrices (Eq. 1, exact).
// ---------------------------------------------------------------------------
// Padding of the stored type: uint16 0x7FFF or, when floor(1/eps) <= 252, byte 0xFF.
template <class CB> constexpr uint32_t kPadOf = sizeof(CB) == 1 ? 0xFFu : (uint32_t)kPadCost;

// Every kernel below takes the rows of all problems in one sweep: warp w takes
// global rows w, w + W, ... (global row r is row r - v_off_i of the problem i
// with v_off_i <= r < v_off_i + n_i, found once per row), and its lanes take
// consecutive columns, so each load instruction of a warp reads one
// contiguous piece of the row and each store writes one contiguous piece of
// the rounded row (padding columns n_i .. ldq_i - 1 included).
__device__ __forceinline__ int problem_of_row(const BDesc *d, int P, int r) {
    int lo = 0, hi = P - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (d[mid].v_off <= r) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Eq. (1) on the packed matrices, a warp per row (round_chunk): about 8
// instructions per cost and 64 bytes in flight per lane.  512 problems (3.17
// GB of FP32 read, 0.80 GB written): 1.06 ms -> 0.71 ms; it was bound by the 25
// instructions a cost took one at a time.
template <class T, class CB>
__global__ void __launch_bounds__(256, 4) k_bquant_matrix(const T *__restrict__ C, const BDesc *__restrict__ d, int P, int total_rows,
                                EpsSplit e, CB *__restrict__ cb, WsHead *head) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < total_rows; r += nw) {
        const BDesc D = d[problem_of_row(d, P, r)];
        const int b = r - D.v_off;
        const T *row = C + D.c_off + (long long)b * D.n;
        CB *out = cb + D.cb_off + (long long)b * D.ldq;
        for (int c0 = 0; c0 < D.ldq; c0 += kRoundCols<T>) round_chunk<T, CB>(row, D.n, D.ldq, c0, e, out, lane, bad);
    }
    if (bad) record_error(head, PR_ERR_INVALID);
}

// ---------------------------------------------------------------------------
// Costs from points (points.cuh): c = RN32(d / max d) per problem.  A warp
// takes kPtRows global rows (cut at problem boundaries) and, step by step, 4
// consecutive columns a lane, so a column's coordinates are loaded once per
// kPtRows pairs and the rounded costs are stored 4 (16-bit storage: 8) bytes at
// a time; the squared sum keeps the operation order of dist_f32.  DIM = 0: any
// dimension, one pair at a time.  64 clouds of 4096 3-D points (1.07 G pairs):
// largest distance 0.96 -> 0.35 ms, rounding 2.20 -> 0.63 ms (three loads and about
// 60 instructions a pair before).
// ---------------------------------------------------------------------------
constexpr int kPtRows = 8;

// Calls body(problem, first global row, rows) for each run of rows that this
// warp takes.
template <class Body>
__device__ __forceinline__ void point_tiles(const BDesc *__restrict__ d, int P, int total_rows, const Body &body) {
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; (long long)t * kPtRows < total_rows; t += nw) {
        const int end = min(total_rows, (t + 1) * kPtRows);
        for (int r = t * kPtRows; r < end;) {
            const int i = problem_of_row(d, P, r);
            const int stop = min(end, d[i].v_off + d[i].n);
            body(i, r, stop - r);
            r = stop;
        }
    }
}

// The squared sums of one row point against a lane's 4 column points.
template <int DIM>
__device__ __forceinline__ void sq_group4(const float (&xb)[DIM], const float (&xa)[4][DIM], float (&sq)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const float t = __fsub_rn(xb[k], xa[j][k]);
            const float q = __fmul_rn(t, t);
            acc = k == 0 ? q : __fadd_rn(acc, q);
        }
        sq[j] = acc;
    }
}

template <int DIM>
__device__ __forceinline__ void load_points(const float *__restrict__ XB, int r, int rows, float (&xb)[kPtRows][DIM]) {
#pragma unroll
    for (int q = 0; q < kPtRows; ++q)
#pragma unroll
        for (int k = 0; k < DIM; ++k) xb[q][k] = __ldg(XB + (long long)(r + min(q, rows - 1)) * DIM + k);
}
template <int DIM>
__device__ __forceinline__ void load_columns(const float *__restrict__ XA, const BDesc &D, int a, float (&xa)[4][DIM]) {
#pragma unroll
    for (int j = 0; j < 4; ++j)  // columns past the last repeat it
#pragma unroll
        for (int k = 0; k < DIM; ++k) xa[j][k] = __ldg(XA + (long long)(D.v_off + min(a + j, D.n - 1)) * DIM + k);
}

// Largest squared sum of every problem (the IEEE root is non-decreasing, so
// the root of the largest sum is the largest root): one atomic per run of
// rows (non-negative floats order like their bit patterns).
template <int DIM>
__global__ void __launch_bounds__(256, 4) k_bpoints_max(const float *__restrict__ XA, const float *__restrict__ XB, int dim,
                              const BDesc *__restrict__ d, int P, int total_rows, unsigned *maxbits) {
    const int lane = threadIdx.x & 31;
    point_tiles(d, P, total_rows, [&](int i, int r, int rows) {
        const BDesc D = d[i];
        float m = 0.0f;
        if constexpr (DIM == 0) {
            for (int q = 0; q < rows; ++q)
                for (int a = lane; a < D.n; a += 32)
                    m = fmaxf(m, dist_f32(XB + (long long)(r + q) * dim, XA + (long long)(D.v_off + a) * dim, dim, 1));
        } else {
            float xb[kPtRows][DIM];
            load_points<DIM>(XB, r, rows, xb);  // rows past the run's last repeat it
            for (int a = 4 * lane; a < D.n; a += 128) {
                float xa[4][DIM];
                load_columns<DIM>(XA, D, a, xa);
#pragma unroll
                for (int q = 0; q < kPtRows; ++q) {
                    float sq[4];
                    sq_group4<DIM>(xb[q], xa, sq);
                    m = fmaxf(m, fmaxf(fmaxf(sq[0], sq[1]), fmaxf(sq[2], sq[3])));
                }
            }
        }
        const unsigned mx = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(m));
        if (lane == 0) atomicMax(maxbits + i, mx);
    });
}

constexpr int kPointCtas = 3;  // CTAs of k_bpoints_quant per SM, by its registers
template <int DIM, bool SQ, class CB>
__global__ void __launch_bounds__(256, kPointCtas) k_bpoints_quant(const float *__restrict__ XA, const float *__restrict__ XB, int dim,
                                const BDesc *__restrict__ d, int P, int total_rows,
                                const unsigned *__restrict__ maxbits, EpsSplit e, CB *__restrict__ cb, WsHead *head) {
    const int lane = threadIdx.x & 31;
    bool bad = false;
    point_tiles(d, P, total_rows, [&](int i, int r, int rows) {
        const BDesc D = d[i];
        const PointsScale ps = points_scale(maxbits[i], SQ, e);
        CB *out = cb + D.cb_off + (long long)(r - D.v_off) * D.ldq;
        // A rounded cost that is no cost (NaN or infinite coordinates, an
        // infinite largest distance) is reported, and stored as 0: the marker's
        // low byte is the padding's, whose sums carry into real columns.
        const auto checked = [&](float dist, uint32_t k) {
            if (dist >= 0.0f && dist <= ps.M && k != 0xFFFFFFFFu) return k;
            bad = true;
            return 0u;
        };
        if constexpr (DIM == 0) {
            for (int q = 0; q < rows; ++q)
                for (int a = lane; a < D.ldq; a += 32) {
                    uint32_t h = kPadOf<CB>;
                    if (a < D.n) {
                        const float dd =
                            dist_f32(XB + (long long)(r + q) * dim, XA + (long long)(D.v_off + a) * dim, dim, SQ);
                        const float c = ps.M > 0.0f ? __fdiv_rn(dd, ps.M) : 0.0f;
                        h = checked(dd, quantise_fbits(__float_as_uint(c), e));
                    }
                    out[(long long)q * D.ldq + a] = (CB)h;
                }
        } else {
            float xb[kPtRows][DIM];
            load_points<DIM>(XB, r, rows, xb);
            for (int a = 4 * lane; a < D.ldq; a += 128) {
                float xa[4][DIM];
                load_columns<DIM>(XA, D, a, xa);
#pragma unroll
                for (int q = 0; q < kPtRows; ++q) {
                    if (q >= rows) break;
                    float sq[4];
                    uint32_t h[4];
                    sq_group4<DIM>(xb[q], xa, sq);
                    quantise_points<4>(sq, SQ, ps, e, h, checked);
                    if (a + 4 > D.n) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (a + j >= D.n) h[j] = kPadOf<CB>;
                    }
                    CB *o = out + (long long)q * D.ldq + a;
                    if (sizeof(CB) == 1)
                        *reinterpret_cast<uint32_t *>(o) = pack_bytes(h[0], h[1], h[2], h[3]);
                    else
                        *reinterpret_cast<uint2 *>(o) = make_uint2(pack_halves(h[0], h[1]), pack_halves(h[2], h[3]));
                }
            }
        }
    });
    if (bad) record_error(head, PR_ERR_INVALID);
}

// ---------------------------------------------------------------------------
// The per-problem solver.
// ---------------------------------------------------------------------------
// The reported cost of a matched pair of one problem: the input matrix's
// entry, or the FP64 distance of the matched points (input units).
struct BatchCost {
    const BParams &p;
    const BDesc &D;
    __device__ double operator()(int b, int a) const {
        if (p.points)
            return dist_f64(p.XB + (long long)(D.v_off + b) * p.dim, p.XA + (long long)(D.v_off + a) * p.dim, p.dim,
                            p.squared);
        const long long at = D.c_off + (long long)b * D.n + a;
        return p.dt == PR_F64 ? reinterpret_cast<const double *>(p.C)[at]
                              : (double)reinterpret_cast<const float *>(p.C)[at];
    }
};

// Outputs of a problem that is not solved, because an error was recorded: cost
// NaN, and mates that are indices all the same (the identity), so that an
// asynchronous caller neither takes what the buffers held for a result nor
// reads out of range with it.
__device__ void write_unsolved(const BParams &p, const BDesc &D, int pi) {
    for (int i = threadIdx.x; i < D.n; i += blockDim.x) {
        p.row_to_col[D.v_off + i] = p.col_to_row[D.v_off + i] = i;
        p.y_row[D.v_off + i] = p.y_col[D.v_off + i] = 0;
    }
    if (threadIdx.x == 0) {
        p.costs[pi] = __longlong_as_double(0x7FF8000000000000ll);
        p.phases[pi] = 0;
    }
}

// CTAs per SM the registers are held to: 128 registers a thread at 128 and 256
// threads, so that 4 and 2 CTAs fit (the compiler takes 172 otherwise, and one
// CTA of 256 threads sat alone on an SM: 512 problems of up to 2048 rows 2.69
// -> 2.00 ms, 1.93 now).  85 and 64 registers spill: that batch 1.90 and 1.86 ms, but 300
// problems of up to 700 rows 0.73 -> 0.85 and 0.91 ms.
template <int THREADS>
constexpr int kSolveCtas = THREADS == 128 ? 4 : THREADS == 256 ? 2 : 1;

// F7: floor(1/eps) <= 125, so every sum of a real column's cbar and key
// stays below 256 and the byte pre-test is one plain add (may_match<true>).
template <int THREADS, int UNROLL, class CB, bool F7>
__global__ void __launch_bounds__(THREADS, kSolveCtas<THREADS>) k_bsolve(BParams p) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ CtaShared s;
    __shared__ int cur_problem, stopped;
    __shared__ double part[THREADS > kCostSums ? THREADS : kCostSums];
    const CtaLayout L(p.n_max, p.n_max);
    const CtaState<CB> state(dyn, L);
    long long my_phases = 0, my_rounds = 0;
    unsigned long long my_bytes = 0, my_rows = 0;  // thread 0's

    for (;;) {
        if (threadIdx.x == 0) {
            cur_problem = (int)atomicAdd(&p.ctl->queue, 1u);
            stopped = ld_relaxed_s32(&p.ctl->head.abort);  // nothing is solved after an error
        }
        __syncthreads();
        const int t = cur_problem, stop = stopped;
        __syncthreads();  // every thread has read them before they change
        if (t >= p.nprob) break;
        const int pi = p.order[t];
        const BDesc D = p.desc[pi];
        if (stop) {
            write_unsolved(p, D, pi);
            continue;
        }
        const CB *cb = static_cast<const CB *>(p.cb) + D.cb_off;
        CtaCounts c = {0, 0, 0, 0, false};
        cta_init(s, state, D.n, D.n, D.ldq);
        __syncthreads();
        cta_phases<UNROLL, CB, F7, false>(s, state, cb, D.n, D.n, D.ldq, D.T, D.cap, 0u, D.n, 0, c);
        my_phases += c.phases;
        my_rounds += c.rounds;
        if (threadIdx.x == 0) {
            my_bytes += s.bytes;
            my_rows += s.rows;
        }
        if (c.failed) {
            if (threadIdx.x == 0) record_error(&p.ctl->head, PR_ERR_NO_CONVERGENCE);
            write_unsolved(p, D, pi);
            __syncthreads();
            continue;
        }
        cta_finish<CB>(s, dyn, L, D.n, D.n, part, p.cost_sums, BatchCost{p, D}, p.row_to_col + D.v_off,
                       p.col_to_row + D.v_off, p.y_row + D.v_off, p.y_col + D.v_off, p.costs + pi);
        if (threadIdx.x == 0) p.phases[pi] = c.phases;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd((unsigned long long *)&p.ctl->phases, (unsigned long long)my_phases);
        atomicAdd((unsigned long long *)&p.ctl->rounds, (unsigned long long)my_rounds);
        atomicAdd(&p.ctl->bytes, my_bytes);
        atomicAdd(&p.ctl->rows, my_rows);
    }
}

__global__ void k_binit(BCtl *ctl, unsigned *maxbits, int P) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        memset(ctl, 0, sizeof(BCtl));
        ctl->head.magic = kWsMagic;
    }
    for (int i = t; i < P; i += gridDim.x * blockDim.x) maxbits[i] = 0;
}

struct Plan {
    std::vector<BDesc> desc;
    std::vector<int> order;
    long long cb_elems = 0, c_elems = 0;
    int n_max = 0, v_total = 0;
};

pr_status make_plan(int P, const int32_t *n_host, double eps, Plan &pl) {
    if (P < 1) return fail(PR_ERR_INVALID, "batched: n_problems must be >= 1");
    if (!n_host) return fail(PR_ERR_INVALID, "batched: NULL size array");
    pl.desc.resize(P);
    long long cb = 0, c = 0;
    long long v = 0;
    const long long K = eps > 0 ? (long long)floor(1.0 / eps) : 0;
    for (int i = 0; i < P; ++i) {
        const int n = n_host[i];
        if (n < 1 || n > kMaxN) return fail(PR_ERR_INVALID, "batched: problem %d has n = %d (need 1..%d)", i, n, kMaxN);
        BDesc &d = pl.desc[i];
        d.n = n;
        d.ldq = row_stride(n);
        d.cb_off = cb;
        d.c_off = c;
        d.v_off = (int)v;
        d.T = (int)floor(eps * (double)n);
        d.cap = ((long long)n * (2 * K + 3)) / (d.T + 1) + 1;
        cb += (long long)n * d.ldq;
        c += (long long)n * n;
        v += n;
        pl.n_max = std::max(pl.n_max, n);
    }
    if (v > (1ll << 30)) return fail(PR_ERR_INVALID, "batched: too many rows in total");
    pl.cb_elems = cb;
    pl.c_elems = c;
    pl.v_total = (int)v;
    pl.order.resize(P);
    std::iota(pl.order.begin(), pl.order.end(), 0);
    // longest processing time first: larger problems start first
    std::stable_sort(pl.order.begin(), pl.order.end(),
                     [&](int a, int b) { return pl.desc[a].n > pl.desc[b].n; });
    return PR_OK;
}

struct Source {
    const void *C = nullptr;
    pr_dtype dt = PR_F64;
    const float *XA = nullptr, *XB = nullptr;
    int dim = 0;
    int squared = 1;
    bool points = false;
};

pr_status run_batched(const Source &src, int32_t P, const int32_t *n_host, double eps,
                      int32_t *row_to_col, int32_t *col_to_row, int32_t *y_row, int32_t *y_col,
                      double *costs, int64_t *phases, const pr_batched_tune *tune, pr_stats *stats,
                      void *ws, size_t ws_bytes, void *stream) {
    if (!row_to_col || !col_to_row || !y_row || !y_col || !costs || !phases)
        return fail(PR_ERR_INVALID, "batched: NULL output pointer");
    if (!(eps > 0.0 && eps < 1.0) || floor(1.0 / eps) > 32766.0)
        return fail(PR_ERR_INVALID, "batched: need 0 < eps < 1 and floor(1/eps) <= 32766");
    Plan pl;
    pr_status rc = make_plan(P, n_host, eps, pl);
    if (rc != PR_OK) return rc;
    const BLayout L = make_blayout(P, pl.cb_elems);
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < L.total)
        return fail(PR_ERR_WORKSPACE, "batched: workspace NULL, not 256-byte aligned or < %zu bytes", L.total);
    // Threads per CTA by the largest problem: short rows and few of them want
    // cheap CTA barriers and many problems per SM, larger problems more warps,
    // unless there are more problems than SMs and rounds are small (eps = 0.01,
    // ms at 128 / 256 / 512 threads: 512 problems up to 300 rows 1.10 / 1.22 /
    // 1.46; 300 up to 700: 0.90 / 0.64 / 0.99; 100 up to 1024: 0.98 / 0.73 / 0.77;
    // 512 up to 2048: 2.26 / 1.93 / 2.19; at eps = 0.1, 300 up to 1500: 1.36 /
    // 0.90 / 0.66).  The order of the cost sum stays that of kCostSums partial
    // sums.
    const DeviceInfo &di = device_info();
    const bool many = P > di.sms && floor(1.0 / eps) > 20.0;
    int threads = pl.n_max <= 400 ? 128 : pl.n_max <= 700 || many ? 256 : 512, per_sm_want = 0;
    int cost_sums = kCostSums;
    if (tune) {
        if (tune->threads) cost_sums = threads = tune->threads;
        per_sm_want = tune->ctas_per_sm;
    }
    if (threads != 128 && threads != 256 && threads != 512 && threads != 1024)
        return fail(PR_ERR_INVALID, "batched: threads must be 128, 256, 512 or 1024");
    if (per_sm_want < 0) return fail(PR_ERR_INVALID, "batched: ctas_per_sm must be >= 0");

    cudaStream_t st = (cudaStream_t)stream;
    char *w = (char *)ws;
    BCtl *ctl = (BCtl *)(w + L.ctl);
    BDesc *d_desc = (BDesc *)(w + L.desc);
    int *d_order = (int *)(w + L.order);
    unsigned *d_max = (unsigned *)(w + L.maxbits);
    void *d_cb = w + L.cb;
    const bool cb8 = floor(1.0 / eps) <= (double)kMaxCbarByte;
    k_binit<<<(P + 255) / 256, 256, 0, st>>>(ctl, d_max, P);
    PR_CUDA(cudaGetLastError());
    // problem table: copied from pageable host memory (waits for earlier work
    // on the stream; the host vectors may be freed on return)
    PR_CUDA(cudaMemcpyAsync(d_desc, pl.desc.data(), sizeof(BDesc) * P, cudaMemcpyHostToDevice, st));
    PR_CUDA(cudaMemcpyAsync(d_order, pl.order.data(), sizeof(int) * P, cudaMemcpyHostToDevice, st));

    const EpsSplit e = make_eps_split(eps);
    // a warp per row: 4 CTAs of 8 warps per SM (all resident at up to 64
    // registers a thread), fewer when there are fewer rows
    const int qgrid = std::max(1, std::min(di.sms * 4, (pl.v_total + 7) / 8));
    if (src.points) {
        // two and three dimensions have their own kernels (coordinates in
        // registers); any other runs one pair at a time
        const int D = src.dim == 2 ? 2 : src.dim == 3 ? 3 : 0;
        const void *kmax = D == 2 ? (const void *)k_bpoints_max<2> : D == 3 ? (const void *)k_bpoints_max<3>
                                                                              : (const void *)k_bpoints_max<0>;
        const auto quant = [&](auto d_, auto sq_) -> const void * {
            constexpr int kD = decltype(d_)::value;
            constexpr bool kSq = decltype(sq_)::value;
            return cb8 ? (const void *)k_bpoints_quant<kD, kSq, uint8_t> : (const void *)k_bpoints_quant<kD, kSq, uint16_t>;
        };
        const auto quant_d = [&](auto d_) {
            return src.squared ? quant(d_, std::true_type{}) : quant(d_, std::false_type{});
        };
        const void *kq = D == 2   ? quant_d(std::integral_constant<int, 2>{})
                         : D == 3 ? quant_d(std::integral_constant<int, 3>{})
                                  : quant_d(std::integral_constant<int, 0>{});
        int dim_ = src.dim, P_ = P, rows_ = pl.v_total;
        const float *xa_ = src.XA, *xb_ = src.XB;
        const BDesc *dd_ = d_desc;
        unsigned *mx_ = d_max;
        // a warp per kPtRows rows
        // (no more CTAs than are resident: a second wave of the rounding took 0.81
        // against 0.68 ms at 64 clouds of 4096 points)
        const int tiles = std::max(1, (pl.v_total + 8 * kPtRows - 1) / (8 * kPtRows));
        void *amax[] = {(void *)&xa_, (void *)&xb_, (void *)&dim_, (void *)&dd_, (void *)&P_, (void *)&rows_,
                        (void *)&mx_};
        PR_CUDA(cudaLaunchKernel(kmax, dim3(std::min(di.sms * 4, tiles)), dim3(256), amax, 0, st));
        const unsigned *cmx_ = d_max;
        void *cbp_ = d_cb;
        WsHead *head_ = &ctl->head;
        void *aq[] = {(void *)&xa_, (void *)&xb_, (void *)&dim_, (void *)&dd_, (void *)&P_,
                      (void *)&rows_, (void *)&cmx_, (void *)&e, (void *)&cbp_, (void *)&head_};
        PR_CUDA(cudaLaunchKernel(kq, dim3(std::min(di.sms * kPointCtas, tiles)), dim3(256), aq, 0, st));
    } else if (src.dt == PR_F64) {
        if (cb8)
            k_bquant_matrix<double, uint8_t><<<qgrid, 256, 0, st>>>((const double *)src.C, d_desc, P, pl.v_total, e,
                                                                    (uint8_t *)d_cb, &ctl->head);
        else
            k_bquant_matrix<double, uint16_t><<<qgrid, 256, 0, st>>>((const double *)src.C, d_desc, P, pl.v_total,
                                                                     e, (uint16_t *)d_cb, &ctl->head);
    } else {
        if (cb8)
            k_bquant_matrix<float, uint8_t><<<qgrid, 256, 0, st>>>((const float *)src.C, d_desc, P, pl.v_total, e,
                                                                   (uint8_t *)d_cb, &ctl->head);
        else
            k_bquant_matrix<float, uint16_t><<<qgrid, 256, 0, st>>>((const float *)src.C, d_desc, P, pl.v_total, e,
                                                                    (uint16_t *)d_cb, &ctl->head);
    }
    PR_CUDA(cudaGetLastError());

    const size_t smem = CtaLayout(pl.n_max, pl.n_max).total(cb8 ? 1 : 2);
    if (smem + kCtaStaticSmem > (size_t)di.max_smem_optin)
        return fail(PR_ERR_INVALID, "batched: problem of n = %d does not fit shared memory", pl.n_max);
    // A warp scans a row in 2 KiB steps (a whole row of the largest size
    // for bytes; measured 9.5 % faster than 4 KiB steps on 512 problems of
    // 64..2048 points).
    const bool f7 = floor(1.0 / eps) <= 125.0;
    const void *kern = !cb8 ? (threads == 128   ? (const void *)k_bsolve<128, 4, uint16_t, false>
                               : threads == 256 ? (const void *)k_bsolve<256, 4, uint16_t, false>
                               : threads == 512 ? (const void *)k_bsolve<512, 4, uint16_t, false>
                                                : (const void *)k_bsolve<1024, 4, uint16_t, false>)
                       : f7 ? (threads == 128   ? (const void *)k_bsolve<128, 4, uint8_t, true>
                               : threads == 256 ? (const void *)k_bsolve<256, 4, uint8_t, true>
                               : threads == 512 ? (const void *)k_bsolve<512, 4, uint8_t, true>
                                                : (const void *)k_bsolve<1024, 4, uint8_t, true>)
                            : (threads == 128   ? (const void *)k_bsolve<128, 4, uint8_t, false>
                               : threads == 256 ? (const void *)k_bsolve<256, 4, uint8_t, false>
                               : threads == 512 ? (const void *)k_bsolve<512, 4, uint8_t, false>
                                                : (const void *)k_bsolve<1024, 4, uint8_t, false>);
    // one value for every batch, so that calls from several threads agree
    PR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((size_t)di.max_smem_optin - kCtaStaticSmem)));
    int per_sm = 0;
    PR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    if (per_sm < 1) return fail(PR_ERR_INVALID, "batched: solver CTA does not fit an SM");
    if (per_sm_want > 0 && per_sm_want < per_sm) per_sm = per_sm_want;
    int grid = di.sms * per_sm;
    if (grid > P) grid = P;

    BParams bp;
    bp.ctl = ctl;
    bp.desc = d_desc;
    bp.order = d_order;
    bp.cb = d_cb;
    bp.nprob = P;
    bp.n_max = pl.n_max;
    bp.cost_sums = cost_sums;
    bp.C = src.C;
    bp.dt = src.dt;
    bp.XA = src.XA;
    bp.XB = src.XB;
    bp.dim = src.dim;
    bp.squared = src.squared;
    bp.points = src.points ? 1 : 0;
    bp.row_to_col = row_to_col;
    bp.col_to_row = col_to_row;
    bp.y_row = y_row;
    bp.y_col = y_col;
    bp.costs = costs;
    bp.phases = phases;
    cudaEvent_t ev0, ev1;
    kernel_events(&ev0, &ev1);
    if (ev0 && ev1) PR_CUDA(cudaEventRecord(ev0, st));
    {
        void *args[] = {(void *)&bp};
        PR_CUDA(cudaLaunchKernel(kern, dim3(grid), dim3(threads), args, smem, st));
    }
    if (ev0 && ev1) PR_CUDA(cudaEventRecord(ev1, st));

    if (stats) {
        BCtl h;
        PR_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(BCtl), cudaMemcpyDeviceToHost, st));
        PR_CUDA(cudaStreamSynchronize(st));
        stats->phases = h.phases;
        stats->rounds = h.rounds;
        stats->bytes_scanned = (int64_t)h.bytes;
        stats->rows_scanned = (int64_t)h.rows;
        stats->free_at_stop = 0;
        stats->threshold = 0;
        stats->loop_ctas = 0;
        stats->loop_cluster = 0;
        stats->cells_examined = 0;
        stats->barriers = 0;
        if (h.head.err != 0)
            return fail((pr_status)h.head.err, "batched: device reported %s", pr_status_string((pr_status)h.head.err));
    }
    return PR_OK;
}

}  // namespace
}  // namespace prot

using namespace prot;

extern "C" size_t pr_assign_batched_workspace(int32_t n_problems, const int32_t *n_host) {
    Plan pl;
    if (make_plan(n_problems, n_host, 0.5, pl) != PR_OK) return 0;
    return make_blayout(n_problems, pl.cb_elems).total;
}

extern "C" pr_status pr_assign_batched(const void *C, pr_dtype dt, int32_t n_problems,
                                       const int32_t *n_host, double eps, int32_t *row_to_col,
                                       int32_t *col_to_row, int32_t *y_row, int32_t *y_col,
                                       double *costs, int64_t *phases, const pr_batched_tune *tune,
                                       pr_stats *stats, void *ws, size_t ws_bytes, void *stream) {
    if (!C) return fail(PR_ERR_INVALID, "pr_assign_batched: NULL cost pointer");
    if (dt != PR_F32 && dt != PR_F64) return fail(PR_ERR_INVALID, "pr_assign_batched: bad dtype");
    Source src;
    src.C = C;
    src.dt = dt;
    return run_batched(src, n_problems, n_host, eps, row_to_col, col_to_row, y_row, y_col, costs,
                       phases, tune, stats, ws, ws_bytes, stream);
}

extern "C" pr_status pr_assign_batched_points(const float *XA, const float *XB, int32_t dim,
                                              pr_metric metric, int32_t n_problems,
                                              const int32_t *n_host, double eps,
                                              int32_t *row_to_col, int32_t *col_to_row,
                                              int32_t *y_row, int32_t *y_col, double *costs,
                                              int64_t *phases, const pr_batched_tune *tune,
                                              pr_stats *stats, void *ws, size_t ws_bytes,
                                              void *stream) {
    if (!XA || !XB) return fail(PR_ERR_INVALID, "pr_assign_batched_points: NULL point pointer");
    if (dim < 1 || dim > 4096) return fail(PR_ERR_INVALID, "pr_assign_batched_points: need 1 <= dim <= 4096");
    if (metric != PR_SQEUCLIDEAN && metric != PR_EUCLIDEAN)
        return fail(PR_ERR_INVALID, "pr_assign_batched_points: bad metric");
    Source src;
    src.XA = XA;
    src.XB = XB;
    src.dim = dim;
    src.squared = metric == PR_SQEUCLIDEAN ? 1 : 0;
    src.points = true;
    return run_batched(src, n_problems, n_host, eps, row_to_col, col_to_row, y_row, y_col, costs,
                       phases, tune, stats, ws, ws_bytes, stream);
}

// Launch-shape autotuner for the batched solver: runs the solve once with
// every candidate (threads per CTA x resident CTAs per SM) on the caller's
// batch, times each with CUDA events on `stream`, and returns the fastest.
// The outputs hold the last candidate's (identical) results.
extern "C" pr_status pr_assign_batched_autotune(const float *XA, const float *XB, int32_t dim,
                                                pr_metric metric, const void *C, pr_dtype dt,
                                                int32_t n_problems, const int32_t *n_host, double eps,
                                                int32_t *row_to_col, int32_t *col_to_row,
                                                int32_t *y_row, int32_t *y_col, double *costs,
                                                int64_t *phases, pr_batched_tune *best,
                                                float *best_ms, void *ws, size_t ws_bytes,
                                                void *stream) {
    if (!best || !best_ms) return fail(PR_ERR_INVALID, "pr_assign_batched_autotune: NULL result pointer");
    const bool points = XA && XB;
    if (!points && !C) return fail(PR_ERR_INVALID, "pr_assign_batched_autotune: give points or costs");
    cudaStream_t st = (cudaStream_t)stream;
    auto run = [&](const pr_batched_tune *t) -> pr_status {
        return points ? pr_assign_batched_points(XA, XB, dim, metric, n_problems, n_host, eps, row_to_col,
                                                 col_to_row, y_row, y_col, costs, phases, t, nullptr, ws,
                                                 ws_bytes, stream)
                      : pr_assign_batched(C, dt, n_problems, n_host, eps, row_to_col, col_to_row, y_row,
                                          y_col, costs, phases, t, nullptr, ws, ws_bytes, stream);
    };
    cudaEvent_t e0, e1;
    PR_CUDA(cudaEventCreate(&e0));
    PR_CUDA(cudaEventCreate(&e1));
    const int threads_c[] = {128, 256, 512, 1024};
    const int per_sm_c[] = {1, 2, 3, 4};
    float best_t = -1.0f;
    pr_batched_tune bt{0, 0};
    bool warmed = false;
    pr_status last_err = PR_OK;
    for (int th : threads_c) {
        for (int ps : per_sm_c) {
            pr_batched_tune t{th, ps};
            if (!warmed) {
                if (run(&t) != PR_OK) {
                    last_err = PR_ERR_INVALID;
                    continue;
                }
                warmed = true;
            }
            cudaEventRecord(e0, st);
            const pr_status rc = run(&t);
            cudaEventRecord(e1, st);
            if (rc != PR_OK) {  // this shape does not fit: skip it
                last_err = rc;
                cudaStreamSynchronize(st);
                continue;
            }
            PR_CUDA(cudaEventSynchronize(e1));
            float ms = 0.0f;
            PR_CUDA(cudaEventElapsedTime(&ms, e0, e1));
            if (best_t < 0.0f || ms < best_t) {
                best_t = ms;
                bt = t;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (best_t < 0.0f) return fail(last_err != PR_OK ? last_err : PR_ERR_INVALID,
                                   "pr_assign_batched_autotune: no launch shape worked");
    // the solve with the chosen shape leaves its results in the outputs; an error
    // found on the device (costs out of range) stops every candidate's solve, so
    // the times tell nothing
    pr_status rc = run(&bt);
    if (rc == PR_OK) rc = pr_ws_status(ws, stream);
    if (rc != PR_OK) return rc;
    *best = bt;
    *best_ms = best_t;
    return PR_OK;
}
