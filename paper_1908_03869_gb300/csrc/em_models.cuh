// Drift / diffusion functors of Eq. 1 for the lane-group layout.
//
// An orbit is integrated by G consecutive lanes; lane g owns the P "units"
// u0 = g P .. u0 + P - 1.  A unit is one Wiener channel with its U state
// components (U = 1 for the phase / scalar models, U = 2 for a
// FitzHugh-Nagumo unit (v, w)).  Units at or past `units` are padding: they
// hold zeros, add nothing to the coupling sums and are never stored.
//
// Each functor provides
//   load(p, u0, units, dt, sqdt)      parameters of the orbit into registers
//   prepare(x, cp, u0, units, red)    per-lane partial coupling sums (and any
//                                     per-unit value reused by incr); cp is
//                                     the Kahan compensation (zero in FP64)
//   prepare_stage(z, u0, units, red)  prepare for a stage state of the ODE
//                                     schemes, built on stage_base (no
//                                     compensation word; a phase within a
//                                     step of [-pi, pi] is not reduced again)
//   incr(i, x, red, N, inc)           the Eq. 2 increment f dt + g sqrt(dt) N
//                                     of unit i's components, after red has
//                                     been summed over the G lanes.
//   drift_incr(i, x, red, inc)        f dt alone (the ODE schemes' stages)
//   newton_solve(z, red, r, theta,    r <- (I - theta dt J(z))^-1 r for the
//                u0, units, reduce)   implicit ODE schemes, J the drift's
//                                     Jacobian, after prepare(z) and the sums
//                                     red; padding units do not enter its
//                                     sums.
// State component c of unit j lives at x[c * units + j] in the orbit's row.
#pragma once

#include "em_device.cuh"

namespace sdeb {

// Two sums of terms of magnitude at most 1 as exact integers in Q60: the upper
// bits in Q54 (of at most 256 terms: 2^62), the last 6 bits in the 16-bit halves
// of `low`.
struct FixedSums {
    static constexpr int kUnits = 4;             // terms added up before they are split: 2^62
    static constexpr uint32_t kLarge = 1u << 22;  // high word of 2^-6 in Q60
    // of `seen`: a non-finite phase; sum q has a term of at least 2^-6: kSeen << q
    static constexpr uint32_t kBad = 1u, kSeen = 2u, kAllSeen = 6u;
    int64_t top[2] = {0, 0};
    uint32_t low = 0, seen = 0;

    __device__ __forceinline__ void take(int64_t (&part)[2]) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            top[q] += part[q] >> 6;
            low += ((uint32_t)part[q] & 63u) << (16 * q);
            part[q] = 0;
        }
    }
    __device__ __forceinline__ void take_unit(double2 r, uint32_t (&large)[2]) {
        const uint32_t hc = (uint32_t)__double2hiint(r.x), hs = (uint32_t)__double2hiint(r.y);
        const uint64_t c = to_q60(hc, (uint32_t)__double2loint(r.x)), s = to_q60(hs, (uint32_t)__double2loint(r.y));
        int64_t part[2] = {with_sign(c, hc & 0x80000000u), with_sign(s, hs & 0x80000000u)};
        large[0] |= hi32(c);
        large[1] |= hi32(s);
        take(part);
    }
    template <bool JUMP>
    __device__ __forceinline__ double value(int q) const {
        const uint32_t l = low >> (16 * q) & 0xffffu;
        return sum_to_double<JUMP>((q != 0 ? top[1] : top[0]) + (l >> 6), l << 26, 54);
    }
};

// Kuramoto, Eq. 5/6, drift in its mean-field form: with C = sum_j cos x_j and
// S = sum_j sin x_j, sum_j sin(x_j - x_i) = S cos x_i - C sin x_i.
// PAPER = false: p = (K, sigma, omega_1..omega_n); true: p = (K, omega, p_1..p_n).
template <typename Real, int P, bool PAPER>
struct KuramotoLane {
    static constexpr int U = 1;
    static constexpr int NR = 2;
    static constexpr bool kFixedSums = sizeof(Real) == 8;  // fixed_sums: exact sums in 64-bit integers
    static constexpr bool kNoise = true;
    static constexpr bool kSplitNoise = !PAPER;  // one noise strength for every unit
    // FP32: compensation folded into x every kCompPeriod steps (the phase
    // the drift reads is x - c, formed anyway by the phase reduction)
    static constexpr bool kDelayedComp = sizeof(Real) == 4;
    static constexpr bool kPacked = false;
    Real omega_dt[P];         // omega_i dt
    Real live[P];             // 1 for the orbit's units, 0 for padding
    Real gsq[PAPER ? P : 1];  // noise strength times sqrt(dt)
    Real gsq_bm;              // g sqrt(dt) times the factor box_muller_polar leaves out
    Real kn;                  // K / n
    Real kn_dt;               // (K / n) dt
    Real sn[P], cs[P];

    __device__ __forceinline__ void load(const Real *p, int u0, int units, Real dt, Real sqdt) {
        kn = p[0] / (Real)units;
        kn_dt = mul_r(kn, dt);
        if (!PAPER) {
            gsq[0] = p[1] * sqdt;
            gsq_bm = mul_r(gsq[0], bm_amp_unit<Real>());
        }
#pragma unroll
        for (int i = 0; i < P; ++i) {
            int j = u0 + i;
            bool ok = j < units;
            omega_dt[i] = ok ? mul_r(p[(PAPER ? 1 : 2) + j], dt) : Real(0);
            live[i] = ok ? Real(1) : Real(0);
            if (PAPER) gsq[i] = ok ? p[1 + units + j] * sqdt : Real(0);
        }
    }

    // Base of the ODE schemes' stage states: the compensated phase reduced
    // to [-pi, pi] (sin and cos are 2 pi periodic; the stages see the phase
    // with the rounding of a number below pi).
    __device__ __forceinline__ void stage_base(const Real (&x)[U][P], const Real (&cp)[U][P],
                                               Real (&base)[U][P]) const {
#pragma unroll
        for (int i = 0; i < P; ++i) base[0][i] = reduce_phase(x[0][i], cp[0][i]);
    }

    // Padding units enter the sums with weight 0: fma(1, v, s) == s + v.
    // rph: the phases x - c reduced to [-pi, pi] (FP32) that sin and cos were
    // taken of, kept for the adjoint's replay record.
    Real rph[P];

    __device__ __forceinline__ void prepare(const Real (&x)[U][P], const Real (&cp)[U][P], int, int,
                                            Real (&red)[NR]) {
        Real C = 0, S = 0;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            rph[i] = reduce_phase(x[0][i], cp[0][i]);
            sincos_reduced(rph[i], sn[i], cs[i]);
            C = fma_r(live[i], cs[i], C);
            S = fma_r(live[i], sn[i], S);
        }
        red[0] = C;
        red[1] = S;
    }

    __device__ __forceinline__ void prepare_stage(const Real (&z)[U][P], int, int, Real (&red)[NR]) {
        Real C = 0, S = 0;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            sincos_reduced(z[0][i], sn[i], cs[i]);
            C = fma_r(live[i], cs[i], C);
            S = fma_r(live[i], sn[i], S);
        }
        red[0] = C;
        red[1] = S;
    }

    // FP64: sines, cosines and the orbit's sums over the lanes of `reduce`, the
    // sums as exact integers in Q60, so that every layout gets the same bits
    // (FixedSums).  A term is off by 2^-60 at most, which is below what an FP64
    // sum rounds by unless all the orbit's terms are small; small_sum then takes
    // the sum again at their scale.
    // All units go through the fixed-point sequences, in one straight block
    // with the step's noise for the scheduler; the units outside their range
    // (whose values there mean nothing) are then taken again.
    template <class RED>
    __device__ __forceinline__ void fixed_sums(const double (&z)[P], int u0, int units, RED &reduce,
                                               double (&red)[NR]) {
        FixedSums t;
        uint32_t again = 0, large[NR] = {0, 0};
        int64_t part[NR] = {0, 0};
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const uint32_t hi = (uint32_t)__double2hiint(z[i]);
            uint32_t next;
            const uint64_t turn = turn_fraction(hi, (uint32_t)__double2loint(z[i]), next);
            const Octant o = sincos_octant(turn, next);
            const uint32_t c_sign = cos_sign(turn), s_sign = sin_sign(turn) ^ (hi & 0x80000000u);
            octant_to_double(o, c_sign, s_sign, cs[i], sn[i]);
            const bool in_range = phase_fixed(hi) && !o.tiny, mine = u0 + i < units;
            again |= mine && !in_range ? 1u << i : 0u;
            const uint64_t keep = mine && in_range ? ~0ULL : 0ULL, lg = o.c >> 3, sm = o.s >> 4;
            const uint64_t c = (o.swap ? sm : lg) & keep, s = (o.swap ? lg : sm) & keep;
            part[0] += with_sign(c, c_sign);
            part[1] += with_sign(s, s_sign);
            large[0] |= hi32(c);
            large[1] |= hi32(s);
            if (i % FixedSums::kUnits == FixedSums::kUnits - 1 || i == P - 1) t.take(part);
        }
        // rolled: the instruction cache holds little more than the block above
#pragma unroll 1
        for (; again != 0; again &= again - 1) {
            const int i = __ffs((int)again) - 1;
            double zi = 0.0;  // selected, not indexed: the units stay in registers
#pragma unroll
            for (int j = 0; j < P; ++j) zi = j == i ? z[j] : zi;
            const double2 r = phase_small((uint32_t)__double2hiint(zi)) ? sincos_small(zi) : sincos_general(zi);
#pragma unroll
            for (int j = 0; j < P; ++j) {
                cs[j] = j == i ? r.x : cs[j];
                sn[j] = j == i ? r.y : sn[j];
            }
            if (isfinite(zi)) t.take_unit(r, large);
            else t.seen |= FixedSums::kBad;
        }
#pragma unroll
        for (int q = 0; q < NR; ++q) t.seen |= large[q] >= FixedSums::kLarge ? FixedSums::kSeen << q : 0u;
        const bool some_small = reduce.template fixed<(P >= 4)>(t, u0 < units);
        reduce.template values<(P >= 4)>(t, red);
        if (some_small) {
#pragma unroll 1
            for (int q = 0; q < NR; ++q) {
                const bool own = (t.seen & FixedSums::kSeen << q) == 0;
                if (!reduce.any(own)) continue;
                double v[P];
#pragma unroll
                for (int i = 0; i < P; ++i) v[i] = q == 0 ? cs[i] : sn[i];
                const double sum = small_sum(v, u0, units, reduce);
                red[0] = own && q == 0 ? sum : red[0];
                red[1] = own && q == 1 ? sum : red[1];
            }
            if ((t.seen & FixedSums::kBad) != 0) red[0] = red[1] = __longlong_as_double(0x7ff8000000000000LL);
        }
    }

    // The sum of an orbit's terms v, again as an exact integer: of the terms
    // times the power of two that takes their largest to 62 bits less
    // log2(units).  (The warp's other orbits come along.)
    template <class RED>
    static __device__ __forceinline__ double small_sum(const double (&v)[P], int u0, int units, RED &reduce) {
        uint32_t top = 1u << 20;  // high word of the largest term, or of the least normal number
#pragma unroll
        for (int i = 0; i < P; ++i)
            if (u0 + i < units) top = max(top, (uint32_t)__double2hiint(v[i]) & 0x7fffffffu);
        const int e_top = (int)(reduce.largest(top) >> 20);  // terms are below 2^(e_top - 1022)
        const int q = 30 + __clz(units - 1);
        FixedSums t;
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const uint32_t hi = (uint32_t)__double2hiint(v[i]);
            const int e = (int)(hi >> 20 & 0x7ffu);
            const uint64_t m = ((uint64_t)((hi & 0xfffffu) | (e != 0 ? 0x100000u : 0u)) << 32) | (uint32_t)__double2loint(v[i]);
            if (u0 + i < units) t.top[0] += with_sign(m << (q - 53) >> min(e_top - max(e, 1), 63), hi & 0x80000000u);
        }
        (void)reduce.template fixed<false>(t, true);
        return sum_to_double<true>(t.top[0], 0u, q) * __hiloint2double((e_top + 1) << 20, 0);
    }

    // f dt = (K/n) dt (S cos x_i - C sin x_i) + omega_i dt, with (K/n) dt S
    // and (K/n) dt C formed once per step (the same products for every unit).
    __device__ __forceinline__ Real drift_dt(int i, const Real (&red)[NR]) const {
        const Real kS = mul_r(kn_dt, red[1]), kC = mul_r(kn_dt, red[0]);
        return fma_r(kS, cs[i], fma_r(-kC, sn[i], omega_dt[i]));
    }

    // f dt + g sqrt(dt) N
    __device__ __forceinline__ void incr(int i, const Real (&x)[U][P], const Real (&red)[NR], Real N,
                                         Real (&inc)[U]) const {
        (void)x;
        const Real kS = mul_r(kn_dt, red[1]), kC = mul_r(kn_dt, red[0]);
        inc[0] = fma_r(kS, cs[i], fma_r(-kC, sn[i], fma_r(gsq[PAPER ? i : 0], N, omega_dt[i])));
    }

    // The scalar noise strength g sqrt(dt) times a Box-Muller amplitude (and
    // the factor the polar form leaves out), once per pair; the increment is
    // then f dt + (g sqrt(dt) amp) trig.
    __device__ __forceinline__ Real noise_scaled(Real amp) const {
        if constexpr (sizeof(Real) == 8) return gsq_bm;  // FP64: amp is 1
        else return mul_r(gsq_bm, amp);
    }

    __device__ __forceinline__ void incr_split(int i, const Real (&red)[NR], Real amp_scaled, Real trig,
                                               Real (&inc)[U]) const {
        inc[0] = fma_r(amp_scaled, trig, drift_dt(i, red));
    }

    __device__ __forceinline__ void drift_incr(int i, const Real (&)[U][P], const Real (&red)[NR],
                                               Real (&inc)[U]) const {
        inc[0] = drift_dt(i, red);
    }

    // With c_i = cos z_i, s_i = sin z_i the drift's Jacobian is
    // (K/n) (c c^T + s s^T) - diag((K/n) (C c_i + S s_i)), so
    // I - theta dt J = D - beta U U^T with U = [c s], beta = theta (K/n) dt,
    // D = diag(1 + beta (C c_i + S s_i)): solved by the Woodbury identity,
    // w = D^-1 r, m = U^T D^-1 U and q = U^T w summed over the orbit's units,
    // r <- w + beta D^-1 U (I - beta m)^-1 q.  m22 = sum s^2 / a is taken as
    // sum 1 / a - m11 (c^2 + s^2 = 1).  D is nonsingular while theta K dt < 1.
    // Padding units get a zero correction.
    template <class RED>
    __device__ __forceinline__ void newton_solve(const Real (&)[U][P], const Real (&red)[NR], Real (&r)[U][P],
                                                 Real theta, int, int, RED &reduce) const {
        const Real C = red[0], S = red[1], beta = theta * kn_dt;
        Real inv_a[P], m[2] = {Real(0), Real(0)}, q[2] = {Real(0), Real(0)}, ia[1] = {Real(0)};
#pragma unroll
        for (int i = 0; i < P; ++i) {
            inv_a[i] = live[i] * recip_fast(fma_r(beta, fma_r(C, cs[i], mul_r(S, sn[i])), Real(1)));
            const Real w = r[0][i] * inv_a[i];
            const Real tc = cs[i] * inv_a[i];
            r[0][i] = w;
            m[0] = fma_r(cs[i], tc, m[0]);
            m[1] = fma_r(sn[i], tc, m[1]);
            ia[0] += inv_a[i];
            q[0] = fma_r(cs[i], w, q[0]);
            q[1] = fma_r(sn[i], w, q[1]);
        }
        reduce(m);
        reduce(q);
        reduce(ia);
        const Real e11 = Real(1) - beta * m[0], e22 = Real(1) - beta * (ia[0] - m[0]), e12 = -beta * m[1];
        const Real b_det = beta * recip_fast(e11 * e22 - e12 * e12);
        const Real z1 = (e22 * q[0] - e12 * q[1]) * b_det, z2 = (e11 * q[1] - e12 * q[0]) * b_det;
#pragma unroll
        for (int i = 0; i < P; ++i) r[0][i] = fma_r(inv_a[i], fma_r(cs[i], z1, sn[i] * z2), r[0][i]);
    }
};

// Milstein correction for diagonal noise whose channel drives one component
// with g = s x (multiplicative): 1/2 g g' (dW^2 - dt) = 1/2 (s sqrt(dt))^2 x (N^2 - 1).
// (The Milstein scheme, named by the paper as the next integrator in
// Sec. 2.1 and Sec. 3; Kloeden and Platen's form for diagonal noise.)
template <typename Real>
__device__ __forceinline__ Real milstein_multiplicative(Real half_gsq2, Real x, Real N) {
    return half_gsq2 * x * (N * N - Real(1));
}

// FitzHugh-Nagumo network: unit j has v_j = x[j], w_j = x[units + j];
// p = (a, b, eps, I, c, sigma); multiplicative noise sigma v_j dW_j on v only.
// MIL: Milstein step (adds 1/2 g g' (dW^2 - dt) to v) instead of Euler-Maruyama.
template <typename Real, int P, bool MIL>
struct FhnLane {
    static constexpr int U = 2;
    static constexpr int NR = 1;
    static constexpr bool kFixedSums = false;
    static constexpr bool kNoise = true;
    static constexpr bool kSplitNoise = false;
    static constexpr bool kDelayedComp = false;
    // FP32: two units an instruction (pairs of em_device.cuh), the drift and the
    // noise apart until the last fused multiply-add:
    //   dv = v (sigma sqrt(dt) N) + dt (v (-c - v^2 / 3) + v - w + I + c mean)
    //   dw = dt (eps (v + a - b w))
    // (Milstein: n + n^2 / 2 - sigma^2 dt / 2 for n = sigma sqrt(dt) N).  Twelve
    // packed operations a pair of units.  Ten do with the noise inside the
    // bracket that dt multiplies and one constant eps dt; but the bracket then
    // rounds by the noise over dt (and leaves the range for a small dt), and v
    // and w run on clocks rounded differently: 2 to 6 % further from the 64-bit
    // result than the scalar step at dt = 0.01.  (Polynomials with dt inside every
    // coefficient take seven and are half as far off again.)
    static constexpr bool kPacked = sizeof(Real) == 4 && P > 1;
    Real kgsq;
    Real a, b, eps, I, c, gsq, dt, inv_units;
    Real half_gsq2;  // (sigma sqrt(dt))^2 / 2, the Milstein coefficient

    // Base of the ODE schemes' stage states: the state itself.
    __device__ __forceinline__ void stage_base(const Real (&x)[U][P], const Real (&)[U][P],
                                               Real (&base)[U][P]) const {
#pragma unroll
        for (int c = 0; c < U; ++c)
#pragma unroll
            for (int i = 0; i < P; ++i) base[c][i] = x[c][i];
    }

    __device__ __forceinline__ void load(const Real *p, int, int units, double dt64, double sqdt64) {
        const Real dt_ = (Real)dt64, sqdt = (Real)sqdt64;
        if constexpr (kPacked) kgsq = (Real)((double)p[5] * sqdt64 * (double)bm_amp_unit<float>());
        a = p[0];
        b = p[1];
        eps = p[2];
        I = p[3];
        c = p[4];
        gsq = p[5] * sqdt;
        dt = dt_;
        inv_units = Real(1) / (Real)units;
        half_gsq2 = Real(0.5) * gsq * gsq;
    }

    __device__ __forceinline__ void prepare(const Real (&x)[U][P], const Real (&)[U][P], int u0, int units,
                                            Real (&red)[NR]) {
        if constexpr (kPacked) {
            if (u0 + P <= units) {
                F2 s2 = pair_of<P>(x[0], 0);
#pragma unroll
                for (int p = 1; p < P / 2; ++p) s2 = add2(s2, pair_of<P>(x[0], p));
                float lo, hi;
                unpack2(s2, lo, hi);
                red[0] = lo + hi;
                return;
            }
        }
        Real sv = 0;
#pragma unroll
        for (int i = 0; i < P; ++i)
            if (u0 + i < units) sv += x[0][i];
        red[0] = sv;
    }

    __device__ __forceinline__ void prepare_stage(const Real (&z)[U][P], int u0, int units, Real (&red)[NR]) {
        prepare(z, z, u0, units, red);
    }

    __device__ __forceinline__ void incr(int i, const Real (&x)[U][P], const Real (&red)[NR], Real N,
                                         Real (&inc)[U]) const {
        Real v = x[0][i], w = x[1][i];
        Real mean_v = red[0] * inv_units;
        Real fv = v - v * v * v * Real(1.0 / 3.0) - w + I + c * mean_v - c * v;
        Real fw = eps * (v + a - b * w);
        inc[0] = fv * dt + gsq * v * N;
        if constexpr (MIL) inc[0] += milstein_multiplicative(half_gsq2, v, N);
        inc[1] = fw * dt;
    }

    struct Step2 {
        F2 k0;
    };
    __device__ __forceinline__ Step2 step2(const Real (&red)[NR]) const { return Step2{dup2(fma_r(c, mul_r(red[0], inv_units), I))}; }
    __device__ __forceinline__ F2 noise_scaled2(F2 amp) const { return mul2(dup2(kgsq), amp); }
    __device__ __forceinline__ void incr2(int p, const Step2 &st, const Real (&x)[U][P], F2 amp_scaled, F2 trig,
                                          F2 (&inc)[U]) const {
        const F2 v = pair_of<P>(x[0], p), w = pair_of<P>(x[1], p);
        const F2 m = fma2(dup2(Real(-1.0 / 3.0)), mul2(v, v), dup2(-c));
        F2 n = mul2(amp_scaled, trig);
        if constexpr (MIL) n = fma2(n, fma2(n, dup2(Real(0.5)), dup2(Real(1))), dup2(-half_gsq2));
        inc[0] = fma2(n, v, mul2(dup2(dt), fma2(v, m, add2(sub2(st.k0, w), v))));
        inc[1] = mul2(dup2(dt), mul2(dup2(eps), fma2(dup2(-b), w, add2(v, dup2(a)))));
    }

    __device__ __forceinline__ void drift_incr(int i, const Real (&x)[U][P], const Real (&red)[NR],
                                               Real (&inc)[U]) const {
        Real v = x[0][i], w = x[1][i];
        Real mean_v = red[0] * inv_units;
        inc[0] = (v - v * v * v * Real(1.0 / 3.0) - w + I + c * mean_v - c * v) * dt;
        inc[1] = eps * (v + a - b * w) * dt;
    }

    // I - theta dt J is block diagonal, E_i = [[1 - th (1 - v_i^2 - c), th],
    // [-th eps, 1 + th eps b]] with th = theta dt, minus the mean-field
    // coupling's rank-1 term gamma e e^T (e: 1 on every v, gamma = th c / u):
    // by Sherman-Morrison, p = E^-1 r and q = E^-1 e unit by unit, P and Q
    // the sums of their v parts over the orbit's units,
    // r <- p + gamma P / (1 - gamma Q) q.
    template <class RED>
    __device__ __forceinline__ void newton_solve(const Real (&z)[U][P], const Real (&)[NR], Real (&r)[U][P],
                                                 Real theta, int u0, int units, RED &reduce) const {
        const Real th = theta * dt, gamma = th * c * inv_units;
        const Real e12 = th, e21 = -th * eps, e22 = Real(1) + th * eps * b;
        Real qv[P], qw[P], sums[2] = {Real(0), Real(0)};
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const Real v = z[0][i];
            const Real e11 = Real(1) - th * (Real(1) - v * v - c);
            const Real inv_det = Real(1) / (e11 * e22 - e12 * e21);
            const Real pv = (e22 * r[0][i] - e12 * r[1][i]) * inv_det;
            const Real pw = (e11 * r[1][i] - e21 * r[0][i]) * inv_det;
            r[0][i] = pv;
            r[1][i] = pw;
            qv[i] = e22 * inv_det;
            qw[i] = -e21 * inv_det;
            if (u0 + i < units) {
                sums[0] += pv;
                sums[1] += qv[i];
            }
        }
        reduce(sums);
        const Real coef = gamma * sums[0] / (Real(1) - gamma * sums[1]);
#pragma unroll
        for (int i = 0; i < P; ++i) {
            r[0][i] = fma_r(coef, qv[i], r[0][i]);
            r[1][i] = fma_r(coef, qw[i], r[1][i]);
        }
    }
};

// Ornstein-Uhlenbeck (KIND 0), geometric Brownian motion (KIND 1) and the
// linear ODE (KIND 2, no noise): componentwise, no coupling.  MIL: Milstein
// step; only GBM's multiplicative noise has a correction (OU's noise is
// additive, where Milstein equals Euler-Maruyama).
template <typename Real, int P, int KIND, bool MIL = false>
struct ScalarLane {
    static constexpr int U = 1;
    static constexpr int NR = 0;
    static constexpr bool kFixedSums = false;
    static constexpr bool kNoise = KIND != 2;
    static constexpr bool kSplitNoise = false;
    static constexpr bool kDelayedComp = false;
    static constexpr bool kPacked = false;
    Real rate, gsq, dt, half_gsq2;

    // Base of the ODE schemes' stage states: the state itself.
    __device__ __forceinline__ void stage_base(const Real (&x)[U][P], const Real (&)[U][P],
                                               Real (&base)[U][P]) const {
#pragma unroll
        for (int i = 0; i < P; ++i) base[0][i] = x[0][i];
    }

    __device__ __forceinline__ void load(const Real *p, int, int, Real dt_, Real sqdt) {
        rate = p[0];
        gsq = KIND == 2 ? Real(0) : p[1] * sqdt;
        dt = dt_;
        half_gsq2 = Real(0.5) * gsq * gsq;
    }

    __device__ __forceinline__ void prepare(const Real (&)[U][P], const Real (&)[U][P], int, int,
                                            Real (&)[NR > 0 ? NR : 1]) {}
    __device__ __forceinline__ void prepare_stage(const Real (&)[U][P], int, int, Real (&)[NR > 0 ? NR : 1]) {}

    __device__ __forceinline__ void incr(int i, const Real (&x)[U][P], const Real (&)[NR > 0 ? NR : 1],
                                         Real N, Real (&inc)[U]) const {
        Real xi = x[0][i];
        if (KIND == 0) inc[0] = -rate * xi * dt + gsq * N;
        if (KIND == 1) {
            inc[0] = rate * xi * dt + gsq * xi * N;
            if constexpr (MIL) inc[0] += milstein_multiplicative(half_gsq2, xi, N);
        }
        if (KIND == 2) inc[0] = -rate * xi * dt;
    }

    __device__ __forceinline__ void drift_incr(int i, const Real (&x)[U][P], const Real (&)[NR > 0 ? NR : 1],
                                               Real (&inc)[U]) const {
        inc[0] = (KIND == 1 ? rate : -rate) * x[0][i] * dt;
    }

    // The drift is lambda x (lambda = rate for GBM, -rate otherwise):
    // I - theta dt J = 1 - theta dt lambda.
    template <class RED>
    __device__ __forceinline__ void newton_solve(const Real (&)[U][P], const Real (&)[NR > 0 ? NR : 1],
                                                 Real (&r)[U][P], Real theta, int, int, RED &) const {
        const Real lambda = KIND == 1 ? rate : -rate;
        const Real inv = Real(1) / (Real(1) - theta * dt * lambda);
#pragma unroll
        for (int i = 0; i < P; ++i) r[0][i] *= inv;
    }
};

}  // namespace sdeb
