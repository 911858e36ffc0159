// quantise.cuh -- the rounding kernel of Eq. (1), shared by the single-
// problem and the optimal-transport paths.
#pragma once

#include "prot_internal.cuh"
#include "scan_common.cuh"

namespace prot {
namespace {

// ---------------------------------------------------------------------------
// One warp rounds columns [c0, c0 + 128 U) of a row: U groups of 4 consecutive
// columns a lane, all loads issued first, one 4-byte (16-bit storage: 8-byte)
// store per group; padding columns n .. ldq - 1 included.  Rows that start on
// 16 bytes take vector loads, others 4 scalar loads per group, whose lines the
// other lanes' loads bring to L1 as well.
// ---------------------------------------------------------------------------
template <class T> constexpr int kRoundGroups = sizeof(T) == 8 ? 2 : 4;  // 64 bytes in flight per lane
template <class T> constexpr int kRoundCols = 128 * kRoundGroups<T>;

template <class T, class CB>
__device__ __forceinline__ void round_chunk(const T *__restrict__ row, int n, int ldq, int c0, const EpsSplit &e,
                                            CB *__restrict__ out, int lane, bool &bad) {
    constexpr int U = kRoundGroups<T>;
    constexpr uint32_t kPad = sizeof(CB) == 1 ? 0xFFu : (uint32_t)kPadCost;
    const bool vec = ((uintptr_t)row & 15) == 0;
    T x[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int a = c0 + 128 * u + 4 * lane;
        if (vec && a + 4 <= n) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(row + a));
            if (sizeof(T) == 8) {
                const uint4 w = __ldg(reinterpret_cast<const uint4 *>(row + a) + 1);
                x[u][0] = (T)__hiloint2double((int)v.y, (int)v.x);
                x[u][1] = (T)__hiloint2double((int)v.w, (int)v.z);
                x[u][2] = (T)__hiloint2double((int)w.y, (int)w.x);
                x[u][3] = (T)__hiloint2double((int)w.w, (int)w.z);
            } else {
                x[u][0] = (T)__uint_as_float(v.x);
                x[u][1] = (T)__uint_as_float(v.y);
                x[u][2] = (T)__uint_as_float(v.z);
                x[u][3] = (T)__uint_as_float(v.w);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[u][j] = a + j < n ? __ldg(row + a + j) : (T)0;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int a = c0 + 128 * u + 4 * lane;
        if (a >= ldq) break;
        uint32_t h[4];
        quantise_group<4>(x[u], e, h, bad);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (a + j >= n) h[j] = kPad;
        if (sizeof(CB) == 1)
            *reinterpret_cast<uint32_t *>(out + a) = pack_bytes(h[0], h[1], h[2], h[3]);
        else
            *reinterpret_cast<uint2 *>(out + a) = make_uint2(pack_halves(h[0], h[1]), pack_halves(h[2], h[3]));
    }
}

// ---------------------------------------------------------------------------
// k_quantise: Eq. (1) exactly.  With VEC (rows 16-byte aligned) a thread takes
// 8 columns with 16-byte loads; otherwise a warp takes a chunk of a row.
// Bound by HBM: n = 10,000 FP64 to bytes (0.9 GB) 129 us (7.0 TB/s; 147 one cost
// at a time), FP32 (0.5 GB) 77 us (92), 9999 x 9999 (rows off 16 bytes) FP64 137
// us (194), FP32 77 us (105).
// ---------------------------------------------------------------------------
// CTAs per SM of the grid.  With VEC those that are resident at once, 5 (the
// launch bound holds the registers to 48): n = 10,000 FP64 131 us, FP32 77 us;
// 16 per SM, a last wave of one fifth, 136 and 83 us.  The other form, 6
// resident, runs four waves (n = 9999 FP64 137 us; one wave 139, 5 per SM 156).
constexpr int kRoundCtas = 5, kRoundCtasUnaligned = 24;
// CB is the stored type: uint16_t, or uint8_t when every cbar <= 252 (the
// caller checks floor(1/eps) <= 252); padding columns get 0x7FFF / 0xFF.
template <class T, bool VEC, class CB>
__global__ void __launch_bounds__(256, VEC ? 5 : 6) k_quantise(const T *__restrict__ C, long long ldc, int nB, int nA, int ldq,
                           EpsSplit e, CB *__restrict__ cb, WsHead *head) {
    constexpr uint32_t kPad = sizeof(CB) == 1 ? 0xFFu : (uint32_t)kPadCost;
    bool bad = false;
    if (!VEC) {
        const int chunks = (ldq + kRoundCols<T> - 1) / kRoundCols<T>, lane = threadIdx.x & 31;
        const long long items = (long long)nB * chunks, nw = ((long long)gridDim.x * blockDim.x) >> 5;
        for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < items; i += nw) {
            const int b = (int)(i / chunks), c0 = (int)(i % chunks) * kRoundCols<T>;
            round_chunk<T, CB>(C + (long long)b * ldc, nA, ldq, c0, e, cb + (long long)b * ldq, lane, bad);
        }
        if (bad) record_error(head, PR_ERR_INVALID);
        return;
    }
    // Grid-stride over (row, group of 8 columns); the row and group indices
    // advance by the stride's quotient and remainder (no division per step).
    const int groups = ldq >> 3;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long g0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int step_b = (int)(stride / groups), step_g = (int)(stride % groups);
    int b = (int)(g0 / groups), gi = (int)(g0 % groups);
    for (; b < nB; b += step_b, gi += step_g) {
        if (gi >= groups) {
            gi -= groups;
            ++b;
            if (b >= nB) break;
        }
        const int a0 = gi << 3;
        const T *row = C + (long long)b * ldc;
        T x[8];
        if (a0 + 8 <= nA) {
            // 8 consecutive costs: 4 x 16 B (FP64) or 2 x 16 B (FP32)
            const uint4 *v = reinterpret_cast<const uint4 *>(row + a0);
#pragma unroll
            for (int j = 0; j < (int)sizeof(T) / 2; ++j) {
                const uint4 w = __ldg(v + j);
                if (sizeof(T) == 8) {
                    x[(2 * j) & 7] = (T)__hiloint2double((int)w.y, (int)w.x);
                    x[(2 * j + 1) & 7] = (T)__hiloint2double((int)w.w, (int)w.z);
                } else {
                    x[(4 * j) & 7] = (T)__uint_as_float(w.x);
                    x[(4 * j + 1) & 7] = (T)__uint_as_float(w.y);
                    x[(4 * j + 2) & 7] = (T)__uint_as_float(w.z);
                    x[(4 * j + 3) & 7] = (T)__uint_as_float(w.w);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = a0 + j < nA ? row[a0 + j] : (T)0;
        }
        uint32_t h[8];
        quantise_group<8>(x, e, h, bad);
        if (a0 + 8 > nA) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (a0 + j >= nA) h[j] = kPad;
        }
        if (sizeof(CB) == 1) {
            *reinterpret_cast<uint2 *>(cb + (long long)b * ldq + a0) =
                make_uint2(pack_bytes(h[0], h[1], h[2], h[3]), pack_bytes(h[4], h[5], h[6], h[7]));
        } else {
            *reinterpret_cast<uint4 *>(cb + (long long)b * ldq + a0) =
                make_uint4(pack_halves(h[0], h[1]), pack_halves(h[2], h[3]), pack_halves(h[4], h[5]),
                           pack_halves(h[6], h[7]));
        }
    }
    if (bad) record_error(head, PR_ERR_INVALID);
}

// Launch k_quantise with 16-byte loads when every row starts 16-byte aligned.
template <class T, class CB = uint16_t>
void launch_quantise(const T *C, long long ldc, int nB, int nA, int ldq, double eps, CB *cb,
                     WsHead *head, int sms, cudaStream_t st) {
    const EpsSplit e = make_eps_split(eps);
    const bool vec = ((uintptr_t)C % 16 == 0) && ((ldc * (long long)sizeof(T)) % 16 == 0);
    const long long want = (long long)nB * (ldq >> 3) / 256 + 1, most = (long long)sms * (vec ? kRoundCtas : kRoundCtasUnaligned);
    const int grid = (int)(want < most ? want : most);
    if (vec) k_quantise<T, true, CB><<<grid, 256, 0, st>>>(C, ldc, nB, nA, ldq, e, cb, head);
    else k_quantise<T, false, CB><<<grid, 256, 0, st>>>(C, ldc, nB, nA, ldq, e, cb, head);
}

}  // namespace
}  // namespace prot
