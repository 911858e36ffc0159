// scan_common.cuh -- device primitives shared by the single-problem and the
// batched solvers: exact rounding of Eq. (1), the packed 16-bit admissibility
// test, the per-column proposal word and a few load forms.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace prot {

// Row stride of the rounded costs: rows start on 32 bytes in either storage
// type where the CTA solver may read them (its 32-byte loads), otherwise on 16.
constexpr int kRowAlign = 32;
constexpr int kCtaMaxCols = 8000;  // cta_solve.cuh
constexpr int row_stride(int cols) {
    return cols <= kCtaMaxCols ? (cols + kRowAlign - 1) & ~(kRowAlign - 1) : (cols + 15) & ~15;
}
constexpr uint16_t kPadCost = 0x7FFF;  // cbar of padding columns
constexpr uint16_t kPadKey = 0x8000;   // k of padding columns: pad sum 0xFFFF never matches

// eps split exactly as me * 2^ee (me < 2^53, an integer), plus the FP32
// reciprocal used for the estimate and the estimate's margin.  Built on the
// host by make_eps_split.
struct EpsSplit {
    unsigned long long me;
    int ee;
    float inv;
    float win;  // an estimate within win of an integer takes the exact test
    float low;  // 0.25 eps: costs below it round to 0
};

// The FP32 estimate q of c / eps (c truncated to 24 significant bits:
// relative error < 2^-23; RN32(1/eps) and the rounded product: 2^-24 each)
// is within c / eps * 2^-22 (1 + 2^-24) < (floor(1/eps) + 1) * 2^-22 of the
// exact quotient, as c <= 1.  The margin is twice that, at most 1/64: at
// eps = 0.01 it is 5e-5, so about one cost in 10^4 takes the exact test.
inline EpsSplit make_eps_split(double eps) {  // eps normal, in (0, 1)
    unsigned long long bits;
    memcpy(&bits, &eps, sizeof bits);
    EpsSplit e;
    e.me = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    e.ee = (int)((bits >> 52) & 0x7FF) - 1075;
    e.inv = (float)(1.0 / eps);
    const double w = (floor(1.0 / eps) + 1.0) * ldexp(1.0, -21);
    e.win = (float)(w < 0.015625 ? w : 0.015625);
    e.low = (float)(0.25 * eps);
    return e;
}

// Exact test c >= m * eps for c = mc * 2^ec (2^23 <= mc < 2^53), 1 <= m < 2^16
// and |c / eps - m| <= 1/16: the sign of 2 (mc 2^(ec - ee) - m me) in 64-bit
// arithmetic mod 2^64.  As c is that near m eps, 2^(ec - ee) is between 1/2 and
// 2^47 and the difference is below 2 me / 16 < 2^50.  About 12 instructions;
// comparing two 128-bit numbers took 50, and in 16 copies per thread they thrashed
// the instruction cache (n = 9999 FP32, 1 % ones at eps = 0.1, whole solve: 238 ->
// 155 us; all costs multiples of eps, n = 10,000 FP64: 322 -> 207 us).
__device__ __forceinline__ bool ge_multiple(unsigned long long mc, int ec, uint32_t m, const EpsSplit &e) {
    return (long long)((mc << (ec - e.ee + 1)) - ((e.me * m) << 1)) >= 0;
}

// Eq. (1) exactly: cbar = the largest k with k * eps <= c, for 0 <= c <= 1.
// An FP32 estimate q of c/eps is within (floor(1/eps) + 1) * 2^-22 of the
// exact quotient (see make_eps_split), so floor(q) is exact whenever q is at
// least e.win (twice that bound, at most 1/64) away from an integer.
// Otherwise the exact quotient lies within 1/32 of the integer m nearest q,
// so the floor is m or m - 1, settled by the exact integer test c >= m * eps.
// No floating-point division and no FP64 instruction runs (GB300 runs FP64
// at a small fraction of its FP32 rate).
//
// For an FP64 cost given by its bit pattern.  Range test on the bits:
// 0 <= c <= 1 (or -0.0), which also rejects NaN and infinities.  The FP32
// estimate truncates the mantissa (relative error < 2^-23) before the two
// roundings of the product.
// Returns 0xFFFFFFFF for a cost outside [0, 1].
__device__ __forceinline__ uint32_t quantise_bits(uint32_t hi, uint32_t lo, const EpsSplit &e) {
    if (hi >= 0x80000000u) {  // sign bit: only -0.0 is valid
        return (hi == 0x80000000u && lo == 0u) ? 0u : 0xFFFFFFFFu;
    }
    if (hi > 0x3FF00000u || (hi == 0x3FF00000u && lo != 0u)) return 0xFFFFFFFFu;  // > 1, NaN, inf
    const uint32_t ex = hi >> 20;
    if (ex <= 896u) {
        // c < 2^-126 (zero or tiny): floor(c / eps) is 0 unless eps is tinier,
        // which eps >= 1/32767 rules out
        return 0u;
    }
    const uint32_t fbits = ((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
    const float q = __fmul_rn(__uint_as_float(fbits), e.inv);
    const float kf = floorf(q);
    const float fr = q - kf;
    uint32_t k = (uint32_t)kf;
    if (!(fr >= e.win && fr <= 1.0f - e.win)) {
        const uint32_t m = k + (fr > 0.5f ? 1u : 0u);
        if (m == 0u) return 0u;
        const unsigned long long mc = (((unsigned long long)(hi & 0xFFFFFu) << 32) | lo) | (1ull << 52);
        k = ge_multiple(mc, (int)ex - 1075, m, e) ? m : m - 1u;
    }
    return k;
}

// The same for an FP32 cost: range test on the bits, exact FP32 estimate,
// the same integer test near a multiple of eps.
__device__ __forceinline__ uint32_t quantise_fbits(uint32_t fb, const EpsSplit &e) {
    if (fb >= 0x80000000u) return fb == 0x80000000u ? 0u : 0xFFFFFFFFu;
    if (fb > 0x3F800000u) return 0xFFFFFFFFu;
    const uint32_t ex = fb >> 23;
    if (ex == 0u) return 0u;  // zero or subnormal: below eps >= 1/32767
    const float q = __fmul_rn(__uint_as_float(fb), e.inv);
    const float kf = floorf(q);
    const float fr = q - kf;
    uint32_t k = (uint32_t)kf;
    if (!(fr >= e.win && fr <= 1.0f - e.win)) {
        const uint32_t m = k + (fr > 0.5f ? 1u : 0u);
        if (m == 0u) return 0u;
        const unsigned long long mc = (unsigned long long)((fb & 0x7FFFFFu) | 0x800000u);
        k = ge_multiple(mc, (int)ex - 150, m, e) ? m : m - 1u;
    }
    return k;
}

// ---------------------------------------------------------------------------
// Eq. (1) for a group of N values: 8 (FP32) to 13 (FP64) instructions each on
// the way that nearly all take, against about 25 for quantise_bits one value
// at a time, which bound the rounding kernels by instructions, not memory.
//
// t = 2^23 + v * scale rounded down has floor(v * scale) in its low bits (the
// sum's unit is 1, and the product is not rounded first); d = v * scale -
// floor - 1/2 tells how near an integer the estimate is.  A value whose |d|
// is within `near` of 1/2 is settled by `settle(j, m)`, m >= 1 the integer
// nearest the estimate; a group with a value outside the range that the
// estimate covers goes to `exact(j)` value by value; one test covers both.
// Values below low (scale * low = 1/4) are taken as low: their floor is 0,
// and exact zeros, common in real costs, stay on the short way.
// Only the low 8 or 16 bits of h[j] are the result.
// ---------------------------------------------------------------------------
// ONE (costs from points, where a value takes a square root and a division
// again): `exact(j)` settles everything, low is not used.
template <int N, bool ONE, class Exact, class Settle>
__device__ __forceinline__ void floor_group(const float (&v)[N], float scale, float low, float near, bool out_of_range,
                                            uint32_t (&h)[N], const Exact &exact, const Settle &settle) {
    float d[N], far = 0.0f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float x = ONE ? v[j] : fmaxf(v[j], low);
        const float t = __fmaf_rd(x, scale, 8388608.0f);
        d[j] = __fmaf_rn(x, scale, __fsub_rn(8388607.5f, t));  // 2^23 - 1/2 - t is exact
        far = fmaxf(far, fabsf(d[j]));
        h[j] = __float_as_uint(t);
    }
    if (out_of_range || !(far <= 0.5f - near)) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const bool close = !(fabsf(d[j]) <= 0.5f - near);
            if (ONE ? out_of_range || close : out_of_range) h[j] = exact(j);
            else if (!ONE && close) h[j] = settle(j, (h[j] & 0xFFFFu) + (d[j] > 0.0f ? 1u : 0u));
        }
    }
}

// The estimate's operand of each cost, and whether the group has a cost
// outside the range that it covers.
// FP32: the cost itself.  The estimate's error is below (floor(1/eps) + 1) *
// 2^-23 (the rounding of 1/eps), inside e.win.
template <int N>
__device__ __forceinline__ bool group_operands(const float (&c)[N], float (&f)[N]) {
    uint32_t top = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        f[j] = c[j];
        top = max(top, __float_as_uint(c[j]));
    }
    return top > 0x3F800000u;
}
// FP64: for 2^-126 <= c < 2 the exponent's low 7 bits and the mantissa's
// leading 23 are those of c truncated to FP32 (relative error below 2^-23), so
// with the rounding of 1/eps the error is below (floor(1/eps) + 1) * 1.5 *
// 2^-23, inside e.win.  The high word of a smaller cost is raised to 2^-127's,
// which gives a value below e.low.  Out of range: c > 1 (the bits less one,
// compared from the high word down, reach 1's), NaN among it, or a sign bit.
// (With 0 and 1 out of range, as at first, one of them sent all 8 values of a
// group the long way: n = 10,000, 1 % ones at eps = 0.3, whole solve 191 ->
// 241 us.)
template <int N>
__device__ __forceinline__ bool group_operands(const double (&c)[N], float (&f)[N]) {
    int top = 0;
    uint32_t signs = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(c[j]);
        const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
        f[j] = __uint_as_float(__funnelshift_l(lo, (uint32_t)max((int)hi, 0x38000000), 3) & 0x3FFFFFFFu);
        top = max(top, (int)((b - 1ull) >> 32));
        signs |= hi;
    }
    return top >= 0x3FF00000 || (int)signs < 0;
}

// One cost the long way; 0 and `bad` for one outside [0, 1].
__device__ __forceinline__ uint32_t quantise_exact(float c, const EpsSplit &e, bool &bad) {
    const uint32_t q = quantise_fbits(__float_as_uint(c), e);
    if (q == 0xFFFFFFFFu) bad = true;
    return q == 0xFFFFFFFFu ? 0u : q;
}
__device__ __forceinline__ uint32_t quantise_exact(double c, const EpsSplit &e, bool &bad) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(c);
    const uint32_t q = quantise_bits((uint32_t)(b >> 32), (uint32_t)b, e);
    if (q == 0xFFFFFFFFu) bad = true;
    return q == 0xFFFFFFFFu ? 0u : q;
}
// A cost in [e.low, 1] whose estimate is near the integer m >= 1.
__device__ __forceinline__ uint32_t quantise_near(float c, uint32_t m, const EpsSplit &e) {
    const uint32_t b = __float_as_uint(c);
    return ge_multiple((b & 0x7FFFFFu) | 0x800000u, (int)(b >> 23) - 150, m, e) ? m : m - 1u;
}
__device__ __forceinline__ uint32_t quantise_near(double c, uint32_t m, const EpsSplit &e) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(c);
    return ge_multiple((b & 0xFFFFFFFFFFFFFull) | (1ull << 52), (int)(b >> 52) - 1075, m, e) ? m : m - 1u;
}

template <int N, class T>
__device__ __forceinline__ void quantise_group(const T (&c)[N], const EpsSplit &e, uint32_t (&h)[N], bool &bad) {
    float f[N];
    const bool out_of_range = group_operands<N>(c, f);
    floor_group<N, false>(
        f, e.inv, e.low, e.win, out_of_range, h, [&](int j) { return quantise_exact(c[j], e, bad); },
        [&](int j, uint32_t m) { return quantise_near(c[j], m, e); });
}

// Costs from points: c = RN32(dist / M), dist the squared sum sq or its IEEE
// root, M the largest.  scale = RN32(e.inv / M).  Against the exact c / eps
// the estimate is off by at most 6 * 2^-24 of it (the two roundings of c, the
// approximate root's 2^-23, the two of the scale), 0.75 e.win; the test takes
// twice e.win.  Out of range: an M whose scale could overflow or lose bits
// (all values then, M is the same for all), and NaN.  exact_cost(dist, q) is
// called with the exact way's distance and result and returns what to store.
struct PointsScale {
    float M, scale;
    bool wide;
};
__device__ __forceinline__ PointsScale points_scale(uint32_t max_sq_bits, int squared, const EpsSplit &e) {
    PointsScale p;
    p.M = squared ? __uint_as_float(max_sq_bits) : __fsqrt_rn(__uint_as_float(max_sq_bits));
    p.wide = !(p.M >= 1e-18f && p.M <= 1e18f);
    p.scale = p.wide ? 0.0f : __fdiv_rn(e.inv, p.M);
    return p;
}
template <int N, class Cost>
__device__ __forceinline__ void quantise_points(const float (&sq)[N], int squared, const PointsScale &p,
                                                const EpsSplit &e, uint32_t (&h)[N], const Cost &exact_cost) {
    float v[N];
    uint32_t top = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        v[j] = sq[j];
        if (!squared) asm("sqrt.approx.f32 %0, %1;" : "=f"(v[j]) : "f"(sq[j]));
        top = max(top, __float_as_uint(sq[j]));
    }
    floor_group<N, true>(
        v, p.scale, 0.0f, 2.0f * e.win, p.wide || top >= 0x7F800000u, h,
        [&](int j) {
            const float d = squared ? sq[j] : __fsqrt_rn(sq[j]);
            const float c = p.M > 0.0f ? __fdiv_rn(d, p.M) : 0.0f;
            return exact_cost(d, quantise_fbits(__float_as_uint(c), e));
        },
        [](int, uint32_t) { return 0u; });
}

// Low bytes (16-bit halves) of four values as one stored word (pair).
__device__ __forceinline__ uint32_t pack_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}
__device__ __forceinline__ uint32_t pack_halves(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5410); }

// Bit j of the result: 16-bit lane j of the 8-lane vector s equals t (t2 =
// t in both halves).
__device__ __forceinline__ unsigned eq_mask(uint4 s, uint32_t t2) {
    const uint32_t w0 = s.x ^ t2, w1 = s.y ^ t2, w2 = s.z ^ t2, w3 = s.w ^ t2;
    unsigned m = 0;
    m |= (w0 & 0xFFFFu) == 0 ? 1u : 0u;
    m |= (w0 >> 16) == 0 ? 2u : 0u;
    m |= (w1 & 0xFFFFu) == 0 ? 4u : 0u;
    m |= (w1 >> 16) == 0 ? 8u : 0u;
    m |= (w2 & 0xFFFFu) == 0 ? 16u : 0u;
    m |= (w2 >> 16) == 0 ? 32u : 0u;
    m |= (w3 & 0xFFFFu) == 0 ? 64u : 0u;
    m |= (w3 >> 16) == 0 ? 128u : 0u;
    return m;
}

// Byte form of the test on four packed bytes: 0x80 in each byte i with
// c_i + k_i == t (t4 = t in all four bytes), else 0.  The low seven bits of
// each byte are added with no carry into the next byte and bit 7 by
// exclusive or, which gives every byte's sum mod 256; a byte whose true sum
// reaches 256 (carry out of its bit 7) is masked out, since such a sum never
// equals a target <= 253.  The zero test of z = sum ^ t4 is exact per byte:
// (z & 0x7F) + 0x7F sets bit 7 iff the low seven bits are not all zero.
__device__ __forceinline__ uint32_t byte_marks(uint32_t c, uint32_t k, uint32_t t4) {
    const uint32_t s7 = (c & 0x7F7F7F7Fu) + (k & 0x7F7F7F7Fu);  // bit 7: carry out of bits 0..6
    const uint32_t s = s7 ^ ((c ^ k) & 0x80808080u);             // sum mod 256
    const uint32_t z = s ^ t4;
    const uint32_t zero = ~(((z & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | z | 0x7F7F7F7Fu);
    const uint32_t ovf = (c & k) | ((c | k) & s7);  // bit 7: carry out of bit 7
    return zero & ~ovf;
}
// A first test that most loads settle: nonzero iff some byte of the four
// words may match.  (z - 0x01..) & ~z & 0x80.. is nonzero iff some byte of
// z is zero (exact as an existence test).  F7 (floor(1/eps) <= 125: cbar <=
// 125, keys <= 127): a plain add has no carry between the bytes of real
// columns (padding bytes 0xFF + 0xFF sit above them and never equal a
// target), so z = (c + k) ^ t4.  Otherwise z is formed from the per-byte sum
// mod 256, and a sum that reached 256 can pass; the exact marks settle it.
__device__ __forceinline__ uint32_t zero_byte(uint32_t z) { return (z - 0x01010101u) & ~z & 0x80808080u; }
template <bool F7>
__device__ __forceinline__ uint32_t may_match(uint32_t c, uint32_t k, uint32_t t4) {
    if (F7) return zero_byte((c + k) ^ t4);
    return zero_byte((((c & 0x7F7F7F7Fu) + (k & 0x7F7F7F7Fu)) ^ ((c ^ k) & 0x80808080u)) ^ t4);
}
// The exact test without a branch, for scans that find a candidate in most
// vectors: bit j of the result is set iff column j of the vector has cbar + k
// == target.  Per word 5 operations mark the zero bytes (halves) of z = (c +
// k) ^ t at their top bit, and one dp4a gathers a word's marks into bits
// (0x80 per marked byte times a power of two, summed), 27 instructions per
// 16 bytes against about 70 for four multiplications that gather byte by byte.
// 16-bit values: cbar + k <= 65534 never carries between halves (padding
// 0x7FFF + 0x8000).  Bytes with F7: real columns' sums stay below 256 and
// padding bytes sit above them; otherwise byte_marks masks the carries.
__device__ __forceinline__ uint32_t half_marks(uint32_t s, uint32_t t2) {
    const uint32_t z = s ^ t2;
    return ~(((z & 0x7FFF7FFFu) + 0x7FFF7FFFu) | z) & 0x80008000u;
}
template <bool F7>
__device__ __forceinline__ uint32_t byte_marks_of(uint32_t c, uint32_t k, uint32_t t4) {
    if (!F7) return byte_marks(c, k, t4);
    const uint32_t z = (c + k) ^ t4;
    return ~(((z & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | z) & 0x80808080u;
}
template <class CB, bool F7>
__device__ __forceinline__ unsigned vec_marks(uint4 c, uint4 k, uint32_t t) {
    if (sizeof(CB) == 1) {
        uint32_t lo = __dp4a(byte_marks_of<F7>(c.x, k.x, t), 0x08040201u, 0u);
        lo = __dp4a(byte_marks_of<F7>(c.y, k.y, t), 0x80402010u, lo);
        uint32_t hi = __dp4a(byte_marks_of<F7>(c.z, k.z, t), 0x08040201u, 0u);
        hi = __dp4a(byte_marks_of<F7>(c.w, k.w, t), 0x80402010u, hi);
        return (lo >> 7) | (hi << 1);
    }
    uint32_t m = __dp4a(half_marks(c.x + k.x, t), 0x02000100u, 0u);
    m = __dp4a(half_marks(c.y + k.y, t), 0x08000400u, m);
    m = __dp4a(half_marks(c.z + k.z, t), 0x20001000u, m);
    m = __dp4a(half_marks(c.w + k.w, t), 0x80004000u, m);
    return m >> 7;
}
// Bytes: the pre-test, then the exact marks for the loads that pass it.
template <bool F7 = false>
__device__ __forceinline__ unsigned eq_mask8(uint4 c, uint4 k, uint32_t t4) {
    if ((may_match<F7>(c.x, k.x, t4) | may_match<F7>(c.y, k.y, t4) | may_match<F7>(c.z, k.z, t4) |
         may_match<F7>(c.w, k.w, t4)) == 0u)
        return 0u;
    return vec_marks<uint8_t, F7>(c, k, t4);
}
// A test that never misses a candidate: nonzero if some column of the vector
// may match (16-bit values and F7: exactly if one does).
__device__ __forceinline__ uint32_t zero_half(uint32_t z) { return (z - 0x00010001u) & ~z & 0x80008000u; }
template <class CB, bool F7>
__device__ __forceinline__ uint32_t vec_may_match(uint4 c, uint4 k, uint32_t t) {
    if (sizeof(CB) == 1)
        return may_match<F7>(c.x, k.x, t) | may_match<F7>(c.y, k.y, t) | may_match<F7>(c.z, k.z, t) |
               may_match<F7>(c.w, k.w, t);
    return zero_half((c.x + k.x) ^ t) | zero_half((c.y + k.y) ^ t) | zero_half((c.z + k.z) ^ t) |
           zero_half((c.w + k.w) ^ t);
}

// Adds every thread's v to a counter in shared memory, one atomic per warp (all
// lanes call it).  A 64-bit shared-memory add is a compare-and-swap loop, and
// 512 threads on one word took 12 us at the end of every phase loop (65 x 8000,
// eps = 0.01, one round: k_phases 22.7 -> 8.2 us; 384 x 768, eps = 0.05, on one
// CTA: k_solo 62 -> 44 us).
__device__ __forceinline__ void warp_count(unsigned long long *counter, unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(counter, v);
}

// Read-only 32-byte load (32-byte aligned).
__device__ __forceinline__ void ld_nc_v8(const void *p, uint4 &a, uint4 &b) {
    asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(p));
}

// Read-only 16-byte load that does not allocate in L1 (streamed rows).
__device__ __forceinline__ uint4 ld_nc_na_v4(const void *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Proposal word of a column: (round << 32) | (0xFFFFFFFF - row).  An
// atomicMax keeps the lowest row among same-round proposals and lets a later
// round overwrite an earlier one.  Round 0 with row -1 means "never won".
__device__ __forceinline__ unsigned tag_of(unsigned long long w) { return (unsigned)(w >> 32); }
__device__ __forceinline__ int row_of(unsigned long long w) { return (int)(0xFFFFFFFFu - (unsigned)w); }
__device__ __forceinline__ unsigned long long word_of(unsigned R, int b) {
    return ((unsigned long long)R << 32) | (0xFFFFFFFFu - (unsigned)b);
}

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

}  // namespace prot
