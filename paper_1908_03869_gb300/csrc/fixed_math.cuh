// Sine, cosine, logarithm and square root of the FP64 path in 64-bit fixed
// point on the integer pipes.
//
// An SM of this GPU retires 1.68 FP64 instructions per clock (any FP64 add,
// multiply, fma or conversion) against 22 wide 32 x 32 -> 64 multiplies or 64
// integer adds or shifts.  CUDA's double sincos, log and sqrt are sequences
// on that one pipe: they were 59 of the 65.6 FP64 instructions per
// oscillator-step of the Kuramoto kernel.  Here they are integer sequences
// whose error is below 2^-56 of full scale before the one rounding to
// double.
//
//   angle reduction  |x| / 2 pi modulo 1 as the product of x's 53-bit
//                    mantissa and the window of the bits of 1/(2 pi) that its
//                    exponent selects (M. H. Payne, R. N. Hanek, 1983)
//   sine, cosine     the fraction of a quarter turn in radians, split as
//                    a_j + d with a_j = j 2^-8; (cos a_j, sin a_j) from a
//                    table, turned by d in three shears (x -= t y, y += s x,
//                    x -= t y with t = tan(d/2), s = sin d; A. W. Paeth,
//                    1986), t and s by their Taylor polynomials
//   logarithm        u = 2^-n m, m in [1/2, 1): -ln m = ln c_j - ln(1 - r),
//                    r = 1 - m c_j exact, c_j near 1/m from a table of 256
//                    (P. T. P. Tang, 1990), -ln(1 - r) by its series
//   square root      a reciprocal square root y of 22 bits from the SFU, then
//                    sqrt(a) = a y (1 + e/2 + 3 e^2/8), e = 1 - a y^2
//
// All magnitudes are unsigned; signs are carried beside them.
// Qk below: the integer v stands for v 2^-k.
#pragma once

#ifndef __CUDACC_RTC__
#include <cstdint>
#include <cuda_runtime.h>

#include "sdeb_fixed_tables.inc"  // written by build.py; the run-time compiled path gets it ahead of this header
#endif

namespace sdeb {

__device__ __forceinline__ ulonglong2 fixed_trig_table(uint32_t j) {
    return __ldg(reinterpret_cast<const ulonglong2 *>(kFixedTrig) + j);
}

struct FixedLogEntry {
    uint64_t lnc;  // ln c in Q58
    uint32_t c;    // Q15
};
__device__ __forceinline__ FixedLogEntry fixed_log_table(uint32_t j) {
    const ulonglong2 e = __ldg(reinterpret_cast<const ulonglong2 *>(kFixedLog) + j);
    return FixedLogEntry{e.x, (uint32_t)e.y};
}

__device__ __forceinline__ uint32_t hi32(uint64_t v) { return (uint32_t)(v >> 32); }

// v or, with `sign` (0 or 1 << 31), -v.
__device__ __forceinline__ int64_t with_sign(uint64_t v, uint32_t sign) {
    const int64_t m = (int64_t)((uint64_t)sign << 32) >> 63;
    return ((int64_t)v ^ m) - m;
}

// (a b) >> 64, too small by at most 3, for a, b <= 2^63: the low product is
// left out and the two cross products add without a carry.  Three wide
// multiply-adds.
__device__ __forceinline__ uint64_t mul_top(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = hi32(a), bl = (uint32_t)b, bh = hi32(b);
    const uint64_t cross = (uint64_t)al * bh + (uint64_t)ah * bl;
    return (uint64_t)ah * bh + hi32(cross);
}

// v 2^-q as a double, rounded to nearest (ties up), `sign` (0 or 1 << 31) its
// sign bit.  v = 0 gives a magnitude below 2^-100.  The shift comes from the
// exponent of a truncating float conversion (64 a clock; a count of leading
// zeros runs at 16).
__device__ __forceinline__ double fixed_to_double(uint64_t v, int q, uint32_t sign) {
    const bool low = hi32(v) == 0;
    const uint32_t h = low ? (uint32_t)v : hi32(v), l = low ? 0u : (uint32_t)v;
    const int top = (int)(__float_as_uint(__uint2float_rz(h)) >> 23) - 127;  // leading bit of h
    const uint64_t m = (((uint64_t)h << 32) | l) << ((31 - top) & 63);         // leading bit at 63
    const uint64_t mant = ((m >> 10) + 1) >> 1;  // 53 bits; their leading 1 adds 1 to the exponent field
    const uint32_t e = (uint32_t)(1022 + (low ? 0 : 32) + top - q);
    return __hiloint2double((int)((sign | (e << 20)) + hi32(mant)), (int)(uint32_t)mant);
}

// cos and sin (Q62) of f quarter turns, f in Q63 (< 2^63): rho = f pi/2 in
// Q61, j = rho's multiple of 2^-8, d the rest (Q64).
__device__ __forceinline__ void sincos_quarter(uint64_t f, uint64_t &c, uint64_t &s) {
    const uint64_t rho = mul_top(f, 0x6487ED5110B4611AULL);  // pi/2 in Q62
    const uint32_t j = (uint32_t)(rho >> 53);
    const uint64_t d = (rho << 3) & 0x00FFFFFFFFFFFFFFULL;
    // d 2^39, rounded, kept below 2^31 (d just under a table step rounds up to it, and z would be 2^32)
    const uint32_t dh = min((uint32_t)((d + 0x1000000u) >> 25), 0x7FFFFFFFu);
    const uint32_t z = (uint32_t)(((uint64_t)dh * dh) >> 30);       // d^2 2^48 (< 2^32: d < 2^-8)
    const uint32_t a = __umulhi(z, 0xAAAAAAABu);                    // d^2/6 2^50
    const uint32_t b = __umulhi(__umulhi(a, z), 0x0CCCCCCDu) >> 16;  // d^4/120 2^50
    // sin d = d - d (d^2/6 - d^4/120); tan(d/2) = d/2 + d/2 (d^2/12 + d^4/120)
    const uint64_t sn = d - (((uint64_t)dh * (a - b)) >> 25);
    const uint64_t tn = (d >> 1) + (((uint64_t)dh * (a + 2 * b)) >> 27);
    const ulonglong2 t = fixed_trig_table(j);
    uint64_t x = t.x, y = t.y;
    x -= mul_top(tn, y);
    y += mul_top(sn, x);
    x -= mul_top(tn, y);
    c = x;
    s = y;
}

// cos and sin of `turn` (Q64 fraction of a full turn) as Q62 magnitudes and
// sign bits (0 or 1 << 31).
__device__ __forceinline__ void sincos_turn(uint64_t turn, uint64_t &c, uint32_t &c_sign, uint64_t &s,
                                            uint32_t &s_sign) {
    uint64_t cq, sq;
    sincos_quarter((turn << 1) & 0x7FFFFFFFFFFFFFFFULL, cq, sq);
    const uint32_t th = hi32(turn);
    const bool odd = (th & 0x40000000u) != 0;  // quadrants 1 and 3: (cos, sin)(a + pi/2) = (-sin a, cos a)
    c = odd ? sq : cq;
    s = odd ? cq : sq;
    c_sign = (th + 0x40000000u) & 0x80000000u;  // quadrants 1 and 2
    s_sign = th & 0x80000000u;                  // quadrants 2 and 3
}

// Phases whose sine and cosine are taken here: 2^-11 <= |x| < 2^21.  Smaller
// ones (whose sine would lose relative precision in fixed point), larger and
// non-finite ones go to CUDA's sincos, out of line.
constexpr uint32_t kPhaseMinHi = 0x3F400000u;                 // high word of 2^-11
constexpr uint32_t kPhaseSpanHi = 0x41400000u - kPhaseMinHi;  // to 2^21

__device__ __forceinline__ bool phase_fixed(uint32_t hi) { return (hi & 0x7fffffffu) - kPhaseMinHi < kPhaseSpanHi; }

// |x| / (2 pi) modulo 1 in Q64 (hi, lo: the words of a phase in the range
// above).  |x| = m 2^-s with s in [32, 63], so the fraction is m times the 96
// bits of 1/(2 pi) from the one that weighs 2^(s - 64) on, modulo 2^64.  (Any
// other phase gives some value.)
__device__ __forceinline__ uint64_t turn_fraction(uint32_t hi, uint32_t lo) {
    const uint32_t sh = 1043u - ((hi >> 20) & 0x7ffu);  // s - 32
    const uint32_t w2 = __funnelshift_r(0x28BE60DBu, 0u, sh);
    const uint32_t w1 = __funnelshift_r(0x9391054Au, 0x28BE60DBu, sh);
    const uint32_t w0 = __funnelshift_r(0x7F09D5F4u, 0x9391054Au, sh);
    const uint32_t m0 = lo, m1 = (hi & 0xfffffu) | 0x100000u;
    uint64_t r = (uint64_t)m0 * w2 + __umulhi(m0, w1);
    r += (uint64_t)m1 * w1;
    r += __umulhi(m1, w0);
    return r + ((uint64_t)(m1 * w2) << 32);
}

static __device__ __noinline__ double2 sincos_general(double x) {
    double2 r;
    sincos(x, &r.y, &r.x);
    return r;
}

__device__ __forceinline__ void sincos_fixed(double x, double &s, double &c) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    if (phase_fixed(hi)) {
        uint64_t cv, sv;
        uint32_t cs, ss;
        sincos_turn(turn_fraction(hi, lo), cv, cs, sv, ss);
        c = fixed_to_double(cv, 62, cs);
        s = fixed_to_double(sv, 62, ss ^ (hi & 0x80000000u));
    } else {
        const double2 r = sincos_general(x);
        c = r.x;
        s = r.y;
    }
}

// The SFU's reciprocal square root (2^-22.9 relative).
__device__ __forceinline__ float rsqrt_seed_f32(float y) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

// sqrt(-2 ln u), u = (w + 1/2) 2^-32, as r 2^-63 2^h with r in [2^62, 2^63].
__device__ __forceinline__ uint64_t normal_radius(uint32_t w, int &h) {
    // u = m 2^-n, m in [1/2, 1) in Q64
    const int n = __clz((int)w);
    const uint64_t m = (((uint64_t)w << 32) | 0x80000000u) << n;
    const FixedLogEntry t = fixed_log_table((hi32(m) >> 23) & 255u);
    // r = 1 - m c: m has 33 leading bits at most, c is in Q15, so r is exact
    // in Q48 and below 2^-7.9
    const uint64_t r48 = (1ULL << 48) - ((uint64_t)hi32(m) * (2u * t.c) + ((uint32_t)m != 0 ? t.c : 0u));
    const uint64_t r = r48 << 22;                // Q70
    const uint32_t rr = (uint32_t)(r48 >> 9);    // Q39
    // -ln(1 - r) = r (1 + r (1/2 + r (1/3 + r (1/4 + r (1/5 + r (1/6 + r/7))))))
    uint32_t i = 0x2AAAAAABu + (__umulhi(rr, 0x24924925u) >> 7);   // Q32
    i = 0x33333333u + (__umulhi(rr, i) >> 7);                      // Q32
    i = 0x80000000u + (__umulhi(rr, i) >> 6);                      // Q33
    uint64_t q = 0x2AAAAAAAAAAAAAABULL + (((uint64_t)rr * i) >> 9);  // Q63
    q = (1ULL << 62) + (mul_top(r, q) >> 6);                       // Q63
    q = (1ULL << 62) + (mul_top(r, q) >> 7);                       // Q62
    const uint64_t p = mul_top(r, q);                              // Q68
    const uint64_t base = (uint64_t)(uint32_t)n * 0x02C5C85FDF473DE7ULL + t.lnc;  // n ln 2 + ln c in Q58
    // u within 2^-9 of 1: the series alone, kept at its full resolution
    const uint64_t v = base == 0 ? p : base + (p >> 10);
    const int ex = base == 0 ? 68 : 58;
    // 2 L = a 2^(64 - ex - up), a = A 2^-63 in [1/4, 1), up even
    const int top = (int)(__float_as_uint(__uint2float_rz(hi32(v))) >> 23) - 127;
    const int up = (30 - top) & ~1;
    const uint64_t A = v << up;
    h = (64 - ex - up) >> 1;
    // y below 1/sqrt(a) by 2^-23 to 2^-20.7 (so e > 0): the seed's 2^-22.9 and
    // three float roundings against a bias of 2^-21.4
    const float y0 = rsqrt_seed_f32(__uint2float_rn(hi32(A)) * 0x1p-31f);
    const uint32_t Y = __float2uint_rz(y0 * 1073741440.0f);        // Q30, bias 384 / 2^30
    const uint64_t e = (1ULL << 59) - mul_top(A, (uint64_t)Y * Y);  // Q59, < 2^40
    const uint32_t e51 = (uint32_t)(e >> 8);
    const uint64_t c = e + (((__umulhi(e51, e51) >> 1) * 3u) >> 12);  // e/2 + 3 e^2/8 in Q60
    const uint64_t r0 = (uint64_t)hi32(A) * Y + __umulhi((uint32_t)A, Y);  // a y in Q61
    return (r0 << 2) + (mul_top(r0, c << 23) >> 17);
}

// Eq. 3 for the word pair (w_first, w_second): radius sqrt(-2 ln u1), angle u2
// turns.
__device__ __forceinline__ void box_muller_fixed(uint32_t w_first, uint32_t w_second, double &n_cos, double &n_sin) {
    int h;
    const uint64_t r = normal_radius(w_first, h);
    uint64_t cv, sv;
    uint32_t cs, ss;
    sincos_turn(((uint64_t)w_second << 32) | 0x80000000u, cv, cs, sv, ss);
    n_cos = fixed_to_double(mul_top(r, cv), 61 - h, cs);
    n_sin = fixed_to_double(mul_top(r, sv), 61 - h, ss);
}

}  // namespace sdeb
