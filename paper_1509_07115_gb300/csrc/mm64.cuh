// mm64.cuh -- FP64 products on the FP16 tensor cores through exact digits.
//
// The FP64 units of this part do 1.7 multiply-adds per clock and SM (measured;
// 1.04 TFLOP/s over 152 SMs, the FP64 matrix instruction the same), the FP16
// matrix instruction mma.sync m16n8k16 does 1024.  So an FP64 operand is
// written as a fixed-point number of 64 bits relative to a power of two above
// its largest magnitude, and that as eight balanced base-256 digits
// D_0 .. D_7 in [-128, 127], each exact in FP16.  A product of two digits is at
// most 2^14, so a sum of 2^10 of them is an integer of at most 2^24 and exact
// in the FP32 accumulator (checked on the hardware for random and extreme
// digits).  The 36 digit products D_i D_j with i + j <= 7 give
//     sum_k a_k x_k = sum_s 2^(-8 s) sum_{i + j = s} sum_k D_i(a_k) D_j(x_k),
// the sums of each s added up as integers (the results' rounding: to_double,
// to_double_once).  36 matrix instructions of two clocks replace 2048
// multiply-adds: 28 per clock and SM.
//
// What is left out, with 2 the scale of A and 2^E that of a line x: the bits of an
// operand below 2^-62 of its scale, and the products with i + j >= 8, which for
// each k are seven terms of up to 2^-62 of the scales' product (i + j = 8; the next
// ones 2^-8 of that).  At random digits that is sqrt(K) 2^-61 of 2^E in a sum over K
// columns.  FP64 multiply-adds round at 2^-53 of each product and partial sum instead: more
// where a line's entries are alike in size, less where dense factors meet a line with
// one large entry among small ones (error of the inverse over the norm, a unit entry among
// entries of 1e-5, here and with multiply-adds: dense N = 1024 5e-16 and 4e-16,
// N = 2048 8e-16 and 5e-16, N = 4096 1.6e-15 and 6e-16; through the interval scheme, whose
// sums are short, no difference).
//
// K runs in blocks of 16.  Lane (g = lane / 4, t = lane % 4) of a warp holds
// columns 4t .. 4t+3 of rows g and g + 8 of the A operand (one 32-byte piece of
// each row), as the instruction's k indices 2t, 2t+1, 2t+8, 2t+9; the B operand
// is read with the same permutation of k.
#pragma once

#include <math.h>
#include <stdint.h>

#include <cuda_fp16.h>

namespace dsbt {
namespace mm64 {

constexpr int ND = 8;                    // digits
constexpr uint32_t kBias = 0x80808080u;  // every digit plus 128

// 64-bit fixed point of v, m = v 2^(62 - E) truncated, plus the digit bias; shift
// = 1 + (E's exponent field) - (v's), see exponent_of.
__device__ __forceinline__ void fixed_point(uint32_t vl, uint32_t mh, int shift, int sign, uint32_t& lo, uint32_t& hi) {
    const uint32_t s = min((uint32_t)shift, 63u);
    unsigned long long m = ((unsigned long long)mh << 32 | (vl << 10)) >> s;
    const unsigned long long sg = (unsigned long long)(long long)sign;   // 0 or all ones
    m = (m ^ sg) + (((unsigned long long)kBias << 32 | kBias) - sg);
    lo = (uint32_t)m;
    hi = (uint32_t)(m >> 32);
}

// A operand: entries of orthogonal factors, |a| < 2, at the fixed scale 2^-61.
__device__ __forceinline__ void fixed_a(double v, uint32_t& lo, uint32_t& hi) {
    const uint32_t vl = (uint32_t)__double2loint(v), vh = (uint32_t)__double2hiint(v);
    const uint32_t mh = (__funnelshift_l(vl, vh, 10) & 0x3fffffffu) | 0x40000000u;
    fixed_point(vl, mh, 1024 - (int)((vh >> 20) & 0x7ffu), (int)vh >> 31, lo, hi);
}

// The words of fixed_a for a small host table.
inline uint2 fixed_a_host(double v) {
    const long long m = (long long)ldexp(v, 61);   // |v| < 2; truncates toward zero as the device does
    const unsigned long long b = (unsigned long long)m + ((unsigned long long)kBias << 32 | kBias);
    return make_uint2((uint32_t)b, (uint32_t)(b >> 32));
}

// Exponent field of v (0 .. 2047); the largest over a line is its scale ef:
// |v| < 2^(ef - 1022) = 2^E.
__device__ __forceinline__ int exponent_of(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// B operand: v relative to its line's scale ef >= 64.  Zero and subnormals (field
// 0) are shifted out.
__device__ __forceinline__ void fixed_b(double v, int ef, uint32_t& lo, uint32_t& hi) {
    const uint32_t vl = (uint32_t)__double2loint(v), vh = (uint32_t)__double2hiint(v);
    const uint32_t mh = (__funnelshift_l(vl, vh, 10) & 0x3fffffffu) | 0x40000000u;
    fixed_point(vl, mh, 1 + ef - (int)((vh >> 20) & 0x7ffu), (int)vh >> 31, lo, hi);
}

// The smallest scale taken: the unit of to_double is then the smallest number 2^-1074,
// and every such number a multiple of 2^(E - 62).  (With the scale of 2^-1020 and below
// that unit underflowed, and the line's results were zeros.)
constexpr int kMinScale = 3;

// The same for any scale: a line whose largest magnitude is below 2^-958.
static __device__ __noinline__ void fixed_b_tiny(double v, int ef, uint32_t& lo, uint32_t& hi) {
    const uint32_t vl = (uint32_t)__double2loint(v), vh = (uint32_t)__double2hiint(v);
    const int e = (int)((vh >> 20) & 0x7ffu);
    const uint32_t mh = (__funnelshift_l(vl, vh, 10) & 0x3fffffffu) | (e ? 0x40000000u : 0u);
    fixed_point(vl, mh, 1 + max(ef, kMinScale) - max(e, 1), (int)vh >> 31, lo, hi);
}

// Digit d of two fixed-point words as a pair of FP16 integers: byte b becomes
// 1024 + b (0x6400 | b), minus 1152.
template <int d>
__device__ __forceinline__ uint32_t digit_pair(uint32_t lo0, uint32_t hi0, uint32_t lo1, uint32_t hi1) {
    constexpr uint32_t b = 3 - (d & 3);
    const uint32_t p = d < 4 ? __byte_perm(hi0, hi1, b | ((4 + b) << 8)) : __byte_perm(lo0, lo1, b | ((4 + b) << 8));
    const uint32_t q = (p & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&q), __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// The eight digits of a thread's four consecutive k of one row: [d][pair].
struct Digits4 {
    uint32_t d[ND][2];
    __device__ __forceinline__ void set(const uint32_t* lo, const uint32_t* hi) {
#define DSBT_DIGIT(k)                                              \
    d[k][0] = digit_pair<k>(lo[0], hi[0], lo[1], hi[1]);           \
    d[k][1] = digit_pair<k>(lo[2], hi[2], lo[3], hi[3]);
        DSBT_DIGIT(0) DSBT_DIGIT(1) DSBT_DIGIT(2) DSBT_DIGIT(3) DSBT_DIGIT(4) DSBT_DIGIT(5) DSBT_DIGIT(6) DSBT_DIGIT(7)
#undef DSBT_DIGIT
    }
};

__device__ __forceinline__ void mma16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// FP32 sums of the digit products of one n8 tile, by i + j, added to 64-bit sums:
// hi takes i + j <= 3 in units of 2^24, lo the rest.
__device__ __forceinline__ void drain8(const float (*acc)[4], long long* hi, long long* lo) {
#pragma unroll
    for (int s = 0; s < ND; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const long long v = __float2int_rn(acc[s][c]);
            if (s < 4) hi[c] += v * (1ll << (8 * (3 - s)));
            else lo[c] += v * (1ll << (8 * (7 - s)));
        }
}

// All 36 digit products of one unit (16 rows x 16 k) with one n8 tile.  b: the
// thread's columns (lane row g of digit 0); rows of one digit are dstride halfs apart.
__device__ __forceinline__ void unit8(float (*acc)[4], const Digits4& d0, const Digits4& d1, const __half* b, int dstride) {
#pragma unroll
    for (int j = 0; j < ND; ++j) {
        const uint2 v = *reinterpret_cast<const uint2*>(b + (size_t)j * dstride);
#pragma unroll
        for (int i = 0; i + j < ND; ++i)
            mma16816(acc[i + j], d0.d[i][0], d1.d[i][0], d0.d[i][1], d1.d[i][1], v.x, v.y);
    }
}

// Product of a 16-row block of fixed-point words (row stride lda, K = 16 units) with
// NT n8 tiles of digits [ND][8 NT][bs] in shared memory; K at most 128.  Results:
// hi, lo[n][c] with c = 0, 1: row g, columns 2t, 2t + 1 of tile n; c = 2, 3: row g + 8.
template <int NT>
__device__ __forceinline__ void block_product(const uint2* A, int lda, int units, const __half* dig, int bs, int lane,
                                              long long (*hi)[4], long long (*lo)[4]) {
    const int g = lane >> 2, t = lane & 3;
    float acc[NT][ND][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int s = 0; s < ND; ++s)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[n][s][c] = 0.f;
    const uint4* r0 = reinterpret_cast<const uint4*>(A + (size_t)g * lda + 4 * t);
    const uint4* r1 = reinterpret_cast<const uint4*>(A + (size_t)(g + 8) * lda + 4 * t);
    uint4 w[4] = {__ldg(r0), __ldg(r0 + 1), __ldg(r1), __ldg(r1 + 1)};
    for (int u = 0; u < units; ++u) {
        uint32_t l0[4] = {w[0].x, w[0].z, w[1].x, w[1].z}, h0[4] = {w[0].y, w[0].w, w[1].y, w[1].w};
        uint32_t l1[4] = {w[2].x, w[2].z, w[3].x, w[3].z}, h1[4] = {w[2].y, w[2].w, w[3].y, w[3].w};
        if (u + 1 < units) {
            r0 += 8;
            r1 += 8;
            w[0] = __ldg(r0); w[1] = __ldg(r0 + 1); w[2] = __ldg(r1); w[3] = __ldg(r1 + 1);
        }
        Digits4 d0, d1;
        d0.set(l0, h0);
        d1.set(l1, h1);
#pragma unroll
        for (int n = 0; n < NT; ++n) unit8(acc[n], d0, d1, dig + (size_t)(n * 8 + g) * bs + u * 16 + 4 * t, 8 * NT * bs);
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
#pragma unroll
        for (int c = 0; c < 4; ++c) hi[n][c] = lo[n][c] = 0;
        drain8(acc[n], hi[n], lo[n]);
    }
}

// Digits of four consecutive k of one column to its place in [ND][ncols][bs] (dst:
// the column's first of the four, digit 0).
__device__ __forceinline__ void put_digits4(__half* dst, int dstride, const double* v, int ef) {
    uint32_t wl[4], wh[4];
    if (ef >= 64) {
#pragma unroll
        for (int c = 0; c < 4; ++c) fixed_b(v[c], ef, wl[c], wh[c]);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) fixed_b_tiny(v[c], ef, wl[c], wh[c]);
    }
    Digits4 d;
    d.set(wl, wh);
#pragma unroll
    for (int q = 0; q < ND; ++q) *reinterpret_cast<uint2*>(dst + (size_t)q * dstride) = make_uint2(d.d[q][0], d.d[q][1]);
}

__device__ __forceinline__ int exponent4(const double* v) {
    return max(max(exponent_of(v[0]), exponent_of(v[1])), max(exponent_of(v[2]), exponent_of(v[3])));
}

// A result: sum = 2^(E - 67) (hi 2^32 + lo).  |sum| <= ||a|| ||x|| < 2^(E + 6.5)
// for K <= 8192, so hi 2^20 stays below 2^62 and one 64-bit integer with the
// unit 2^(E - 55) holds it: an error of 2^-56 of the line's scale in every result.
__device__ __forceinline__ double to_double(long long hi, long long lo, int ef) {
    if (ef == 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);   // a line with an infinity or NaN
    const long long v = hi * (1ll << 20) + ((lo + 2048) >> 12);
    const int e = max(ef, kMinScale) - 1022 - 55;
    const double s = e > -1022 ? __hiloint2double((e + 1023) << 20, 0) : ldexp(1.0, e);
    return (double)v * s;
}

// v 2^e for e <= -1022, where 2^e may be no FP64 number (a line whose largest magnitude is
// below 2^-955): in two steps, of which only the second rounds.
static __device__ __noinline__ double times_small_power(double v, int e) {
    return v * __hiloint2double((e + 1223) << 20, 0) * 0x1p-200;
}

// The same rounded to FP64 once, for long lines: with lo's carry in it hi has at most 42
// bits, and the whole, shifted down by the s of them above 31 that it has, fills a 64-bit
// integer.  (The unit above, in the N results of a line with one large entry, is
// sqrt(N / 3) 2^-56 of it: 1.5e-15 at N = 8192, three times the sine transform's error.
// The columns of the angular products have 64 entries, 6e-17, and keep it.)
__device__ __forceinline__ double to_double_once(long long hi, long long lo, int ef) {
    if (ef == 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);
    hi += lo >> 32;
    const int top = (int)(hi >> 31), s = 32 - __clz(top ^ (top >> 31));
    const long long v = (long long)((unsigned long long)hi << (32 - s)) + (long long)((uint32_t)lo >> s);
    const int e = max(ef, kMinScale) - 1022 - 67 + s;
    if (e <= -1022) return times_small_power((double)v, e);
    return (double)v * __hiloint2double((e + 1023) << 20, 0);
}

}  // namespace mm64
}  // namespace dsbt
