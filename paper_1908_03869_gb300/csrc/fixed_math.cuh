// Sine, cosine, logarithm and square root of the FP64 path in 64-bit fixed
// point on the integer pipes.
//
// An SM of this GPU retires 1.68 FP64 instructions per clock (any FP64 add,
// multiply, fma or conversion) against 22 wide 32 x 32 -> 64 multiplies or 64
// integer adds or shifts.  CUDA's double sincos, log and sqrt are sequences
// on that one pipe: they were 59 of the 65.6 FP64 instructions per
// oscillator-step of the Kuramoto kernel.  Here they are integer sequences,
// each result rounded to double once and right relative to itself, however
// small it is (the largest errors on the host against 64-bit mantissas, in
// units of 2^-53: sine and cosine 2.0, the radius before its rounding 0.3,
// normals 2.0, 2.8 next to a multiple of a quarter turn):
//
//   angle reduction  |x| / 2 pi modulo 1 as the product of x's 53-bit
//                    mantissa and the window of the bits of 1/(2 pi) that its
//                    exponent selects (M. H. Payne, R. N. Hanek, 1983), to 96
//                    bits, folded to an eighth of a turn
//   sine, cosine     of a_j + d, a_j = j pi/4096: (cos a_j, sin a_j) from a
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

// (cos, sin)(j pi/4096) in Q63 and Q64, j = 0 .. 1023 (an eighth of a turn).
__device__ __forceinline__ ulonglong2 fixed_trig_table(uint32_t j) {
    return __ldg(reinterpret_cast<const ulonglong2 *>(kFixedTrig) + j);
}

struct FixedLogEntry {
    uint64_t lnc;  // ln c in Q64, 2 units up (the bits that normal_radius shifts out then round)
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

// (a b) >> 64, too small by at most 3: the low product is left out and the two
// cross products add without a carry, so a's and b's high words may take 32
// bits between them less than their number (a, b <= 2^63, or a < 2^62 and any
// b < 2^63.5).  Three wide multiply-adds.
__device__ __forceinline__ uint64_t mul_top(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = hi32(a), bl = (uint32_t)b, bh = hi32(b);
    const uint64_t cross = (uint64_t)al * bh + (uint64_t)ah * bl;
    return (uint64_t)ah * bh + hi32(cross);
}

// The position of the leading bit of h > 0, from the exponent of a truncating
// float conversion (64 a clock; a count of leading zeros runs at 16).
__device__ __forceinline__ int leading_bit(uint32_t h) { return (int)(__float_as_uint(__uint2float_rz(h)) >> 23) - 127; }

// m 2^-q as a double, rounded to nearest (ties up), for m in [2^62, 2^63];
// `sign` (0 or 1 << 31) its sign bit.
__device__ __forceinline__ double normal_to_double(uint64_t m, int q, uint32_t sign) {
    const uint64_t mant = (m + 512u) >> 10;  // 53 bits; their leading 1 adds 1 to the exponent field
    return __hiloint2double((int)(sign + ((uint32_t)(1084 - q) << 20) + hi32(mant)), (int)(uint32_t)mant);
}

// (v + rest 2^-32) 2^-q as a double, rounded to nearest (ties up); v in two's
// complement, |v| < 2^63.  JUMP: the rare leading zero words are skipped in a
// loop (fewer instructions), else by selections (shorter chain).  (An early
// return with FP64 instructions would be turned into selections that every call
// pays for.)
template <bool JUMP>
__device__ __forceinline__ double sum_to_double(int64_t v, uint32_t rest, int q) {
    const uint32_t sign = hi32((uint64_t)v) & 0x80000000u, flip = (uint32_t)((int32_t)sign >> 31);
    uint32_t c = (rest ^ flip) - flip;  // -(v + rest) = ~v + (1 - rest), or -v
    const uint64_t m = ((uint64_t)v ^ (((uint64_t)flip << 32) | flip)) + (c == 0 ? flip & 1u : 0u);
    uint32_t a = hi32(m), b = (uint32_t)m;
    int e = 1085 - q;
    if constexpr (JUMP) {
#pragma unroll 1
        for (; a == 0 && (b | c) != 0; e -= 32) {
            a = b;
            b = c;
            c = 0;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const bool shift = a == 0;
            a = shift ? b : a;
            b = shift ? c : b;
            c = shift ? 0u : c;
            e -= shift ? 32 : 0;
        }
    }
    const int up = 31 - leading_bit(a | (a == 0));
    const uint32_t mh = __funnelshift_l(b, a, up), ml = __funnelshift_l(c, b, up);
    // 53 bits of the 64 from the leading one on, which adds 1 to the exponent field
    const uint64_t mant = ((((uint64_t)mh << 32) | ml) >> 11) + ((ml >> 10) & 1u);
    const uint32_t hi = sign + ((uint32_t)(e - up) << 20) + hi32(mant);
    return __hiloint2double(a == 0 ? 0 : (int)hi, (int)(uint32_t)mant);
}

// |v| <= 1, in Q60, rounded down; hi, lo: its words.
__device__ __forceinline__ uint64_t to_q60(uint32_t hi, uint32_t lo) {
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    return (m << 8) >> min(1023u - ((hi >> 20) & 0x7ffu), 63u);
}

// Cosine and sine of an angle of a quadrant, with their distance from an axis
// folded to an eighth of a turn: `c` (Q63, at least 0.7) is the larger one,
// `s` (Q64) the smaller one, `m` 2^-q the smaller one with its leading bit at
// 62 and 62 bits of its own; swap: the sine is the larger one.
struct Octant {
    uint64_t c, s, m;
    int q;
    bool swap;
    bool tiny;  // the smaller one is below 2^-15: m has lost bits, take the general functions
};

// turn (Q64) and turn_lo (its next 32 bits): the angle as a fraction of a turn.
// d is exact to 2^-70, so the smaller one keeps its 54 bits from 2^-15 on, and
// comes from the table's S_j (up to 2^-65 off) only where that is above 2^-10.4.
__device__ __forceinline__ Octant sincos_octant(uint64_t turn, uint32_t turn_lo) {
    Octant o;
    uint64_t f = (turn << 2) | (turn_lo >> 30);  // quarter turns, Q64
    uint32_t f_lo = turn_lo << 2;
    const uint32_t fold = (uint32_t)((int32_t)hi32(f) >> 31);
    f ^= ((uint64_t)fold << 32) | fold;  // f' = 1 - f
    f_lo ^= fold;
    o.swap = (((hi32(turn) >> 30) ^ fold) & 1u) != 0;  // quadrants 1 and 3: (cos, sin)(a + pi/2) = (-sin a, cos a)
    const uint32_t j = hi32(f) >> 21;
    const uint64_t rest = ((f << 10) | (f_lo >> 22)) & 0x7FFFFFFFFFFFFFFFULL;  // Q74, below 2^-11
    const uint64_t d = mul_top(rest, 0x6487ED5110B4611AULL);                  // times pi/2 (Q62): Q72, below 2^-10.3
    const uint32_t dh = (uint32_t)((d + 0x20000000u) >> 30);                  // Q42, below 2^31.7
    const uint32_t z = hi32((uint64_t)dh * dh + 0x80000000u);                 // d^2, Q52
    const uint32_t a = hi32((uint64_t)z * 0xAAAAAAABu + 0x80000000u);         // d^2/6, Q54
    const uint32_t b = __umulhi(__umulhi(a, z), 0x0CCCCCCDu) >> 20;           // d^4/120, Q54
    // sin d = d - d (d^2/6 - d^4/120), Q72; tan(d/2) = d/2 + d/2 (d^2/12 + d^4/120), Q63
    const uint64_t sn = d - (((uint64_t)dh * (a - b)) >> 24);
    const uint64_t tn = (d >> 10) + (((uint64_t)dh * (a + 2 * b)) >> 35);
    const ulonglong2 t = fixed_trig_table(j);
    uint64_t x = t.x - mul_top(tn, t.y);
    const uint64_t y = t.y + (mul_top(sn, x) >> 7);
    x -= mul_top(tn, y);
    o.c = x;
    o.s = y;
    const uint64_t own = j == 0 ? sn : y;  // S_0 = 0: the sine is sn itself, at its full resolution
    const int up = 31 - leading_bit(hi32(own) | 1u);
    o.m = (own << up) >> 1;
    o.q = (j == 0 ? 71 : 63) + up;
    o.tiny = j == 0 && hi32(own) < 0x02000000u;
    return o;
}

// Signs (0 or 1 << 31) of the cosine and the sine of `turn`.
__device__ __forceinline__ uint32_t cos_sign(uint64_t turn) { return (hi32(turn) + 0x40000000u) & 0x80000000u; }
__device__ __forceinline__ uint32_t sin_sign(uint64_t turn) { return hi32(turn) & 0x80000000u; }

// (cos, sin) of an octant's angle.
__device__ __forceinline__ void octant_to_double(const Octant &o, uint32_t c_sign, uint32_t s_sign, double &c,
                                                 double &s) {
    const double large = normal_to_double(o.c, 63, o.swap ? s_sign : c_sign);
    const double small = normal_to_double(o.m, o.q, o.swap ? c_sign : s_sign);
    c = o.swap ? small : large;
    s = o.swap ? large : small;
}

// Phases whose sine and cosine are taken here, in line: 2^-11 <= |x| < 2^21.
// Smaller ones are their own reduced angle (sincos_small); larger ones, and
// those within 2^-15 of a multiple of a quarter turn, go out of line.
constexpr uint32_t kPhaseMinHi = 0x3F400000u;                 // high word of 2^-11
constexpr uint32_t kPhaseSpanHi = 0x41400000u - kPhaseMinHi;  // to 2^21

__device__ __forceinline__ bool phase_fixed(uint32_t hi) { return (hi & 0x7fffffffu) - kPhaseMinHi < kPhaseSpanHi; }
__device__ __forceinline__ bool phase_small(uint32_t hi) { return (hi & 0x7fffffffu) < kPhaseMinHi; }

// |x| / (2 pi) modulo 1 in Q64 and the next 32 bits (hi, lo: the words of a
// phase in the range above; BIG: of one from 2^21 to 2^53), less than 2^-74 too
// small.  |x| = m 2^-s with s in [32, 63], so the fraction is m times the bits
// of 1/(2 pi) from the one that weighs 2^(s - 64) on, modulo 2^64; BIG, s in
// [0, 31], from one word further on.  (Any other phase gives some value.)
template <bool BIG = false>
__device__ __forceinline__ uint64_t turn_fraction(uint32_t hi, uint32_t lo, uint32_t &next) {
    constexpr uint32_t kBits[5] = {0u, 0x28BE60DBu, 0x9391054Au, 0x7F09D5F4u, 0x7D4D3770u};
    constexpr int o = BIG ? 1 : 0;
    const uint32_t sh = 1043u - ((hi >> 20) & 0x7ffu);  // s - 32; a funnel shift takes it modulo 32
    const uint32_t w2 = __funnelshift_r(kBits[o + 1], kBits[o], sh);
    const uint32_t w1 = __funnelshift_r(kBits[o + 2], kBits[o + 1], sh);
    const uint32_t w0 = __funnelshift_r(kBits[o + 3], kBits[o + 2], sh);
    const uint32_t m0 = lo, m1 = (hi & 0xfffffu) | 0x100000u;
    const uint64_t t = (uint64_t)m0 * w1 + __umulhi(m0, w0);
    const uint64_t u = (uint64_t)m1 * w0 + (uint32_t)t;
    uint64_t r = (uint64_t)m0 * w2 + hi32(t);
    r += (uint64_t)m1 * w1;
    r += hi32(u);
    next = (uint32_t)u;
    uint32_t top = m1 * w2;
    if constexpr (BIG) top += m0 * __funnelshift_r(kBits[1], kBits[0], sh);  // whole turns but for m0's bits below them
    return r + ((uint64_t)top << 32);
}

// (cos, sin) of |x| < 2^-11 by their Taylor polynomials (the terms left out
// are below 2^-77 and 2^-75).
__device__ __forceinline__ double2 sincos_small(double x) {
    const double x2 = x * x;
    return make_double2(fma(x2, fma(x2, 1.0 / 24.0, -0.5), 1.0), fma(x * x2, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x));
}

// (cos, sin) of any phase: from 2^21 to 2^53 as in line, else by CUDA's sincos.
static __device__ __noinline__ double2 sincos_general(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    double2 r;
    if ((hi & 0x7fffffffu) - (kPhaseMinHi + kPhaseSpanHi) < 0x43400000u - (kPhaseMinHi + kPhaseSpanHi)) {
        uint32_t next;
        const uint64_t turn = turn_fraction<true>(hi, (uint32_t)__double2loint(x), next);
        const Octant o = sincos_octant(turn, next);
        octant_to_double(o, cos_sign(turn), sin_sign(turn) ^ (hi & 0x80000000u), r.x, r.y);
        if (!o.tiny) return r;
    }
    sincos(x, &r.y, &r.x);
    return r;
}

__device__ __forceinline__ void sincos_fixed(double x, double &s, double &c) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    uint32_t next;
    const uint64_t turn = turn_fraction(hi, lo, next);
    const Octant o = sincos_octant(turn, next);
    octant_to_double(o, cos_sign(turn), sin_sign(turn) ^ (hi & 0x80000000u), c, s);
    if (!phase_fixed(hi) || o.tiny) {
        const double2 r = phase_small(hi) ? sincos_small(x) : sincos_general(x);
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
    const uint32_t j = (hi32(m) >> 23) & 255u;
    const FixedLogEntry t = fixed_log_table(j);
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
    // -ln u = n ln 2 + ln c - ln(1 - r): in Q58, for u past 1/2 in Q62; for u
    // past 1 - 2^-9, where ln c = 0, as r (Q70) times q below
    const bool near_one = n == 0 && j == 255u;
    uint64_t v = r;
    int ex = 70;
    if (!near_one) {
        const uint64_t frac = t.lnc + (mul_top(r, q) >> 4);  // Q64
        v = (uint64_t)(uint32_t)n * 0x02C5C85FDF473DE7ULL + (frac >> (n == 0 ? 2 : 6));
        ex = n == 0 ? 62 : 58;
    }
    // 2 L = a 2^(64 - ex - up), a = A 2^-63 in [1/4, 1), up even
    const int up = (30 - leading_bit(hi32(v))) & ~1;
    uint64_t A = v << up;
    h = (64 - ex - up) >> 1;
    if (near_one) {
        A = mul_top(A, q) << 2;
        if ((A >> 63) != 0) {
            A >>= 2;
            ++h;
        }
    }
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

static __device__ __noinline__ double2 cospi_sinpi_general(double x) {
    double2 r;
    sincospi(x, &r.y, &r.x);
    return r;
}

// p 2^-q as a double for p in [2^60, 2^62]: a product of two numbers in
// [2^62, 2^63].
__device__ __forceinline__ double product_to_double(uint64_t p, int q, uint32_t sign) {
    const int up = hi32(p) < 0x20000000u ? 2 : 1;
    return normal_to_double(p << up, q + up, sign);
}

// Eq. 3 for the word pair (w_first, w_second): radius sqrt(-2 ln u1), angle u2
// turns.  Angles within 2^-15 of a multiple of a quarter turn take the product
// of the rounded radius and CUDA's sincospi.
__device__ __forceinline__ void box_muller_fixed(uint32_t w_first, uint32_t w_second, double &n_cos, double &n_sin) {
    int h;
    const uint64_t r = normal_radius(w_first, h);
    const uint64_t turn = ((uint64_t)w_second << 32) | 0x80000000u;
    const Octant o = sincos_octant(turn, 0);
    const uint32_t cs = cos_sign(turn), ss = sin_sign(turn);
    const double large = product_to_double(mul_top(r, o.c), 62 - h, o.swap ? ss : cs);
    const double small = product_to_double(mul_top(r, o.m), o.q - 1 - h, o.swap ? cs : ss);
    n_cos = o.swap ? small : large;
    n_sin = o.swap ? large : small;
    if (o.tiny) {
        const double2 t = cospi_sinpi_general(__uint2double_rn(w_second) * 0x1p-31 + 0x1p-32);
        const double radius = normal_to_double(r, 63 - h, 0u);
        n_cos = radius * t.x;
        n_sin = radius * t.y;
    }
}

}  // namespace sdeb
