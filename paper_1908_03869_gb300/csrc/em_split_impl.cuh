// Forward Euler-Maruyama kernel for few orbits of the phase models: the
// noise on warps of its own.
//
// With fewer lanes than the GPU has issue slots to hide latency with, a
// launch takes steps x (latency of one step).  A step's normals do not depend
// on the state, so here the block's last warps (producers) draw them ahead,
// kSplitSteps steps at a time into one half of a double buffer in shared
// memory, while its first warps (consumers), one unit a lane, run the chain
// that is left -- sines, coupling sums, update -- on the other half.  One
// block barrier per kSplitSteps steps hands the halves over.  The results are
// the bits of the other kernels: FP64 sums are exact, FP32 ones are added in
// the default layout's order.
// Measured, whole passes (before: the whole step on every lane): 1024 orbits of
// n = 4, FP64, 1000 steps 1.30 -> 0.65 ms; 64 orbits of n = 100, FP64, 1000 steps
// with moments 1.43 -> 0.97 ms; 256 orbits of n = 8, FP32, 200 steps 77 -> 55 us
// (45 to 47 with the start state set by one kernel).
#pragma once

#include "em_forward_impl.cuh"
#include "split_chunks.h"

namespace sdeb {

constexpr int kSplitSteps = (int)SplitChunks::kSteps;

// Lanes, warps and orbits of a block, and the producers' share: two noise
// blocks of four normals per producer lane and buffer half keeps them ahead.
template <int G, int P>
struct SplitShape {
    static constexpr int kConsumerWarps = G > 32 ? G / 32 : 1;
    static constexpr int kOrbits = G > 32 ? 1 : 32 / G;
    static constexpr int kSlots = kOrbits * G * P;  // normals of a step
    static constexpr int kBlocksMax = kOrbits * ((G * P + 3) / 4);
    static constexpr int kProducerWarps = (kBlocksMax * kSplitSteps + 63) / 64;
    static constexpr int kThreads = 32 * (kConsumerWarps + kProducerWarps);
};

// FP32 coupling sums with the bits of the default layout, which has eight
// units a lane (all of them up to eight): the eight in order, then a butterfly
// over the eights.  Every lane fetches the terms of its eight; their shuffles
// do not depend on one another.
template <class M, int G, int P>
struct EightsSum {
    const M &model;
    template <int NR>
    __device__ __forceinline__ void operator()(float (&r)[NR]) const {
        static_assert(NR == 2 && G <= 32, "two sums over the lanes of a warp");
        constexpr int kEight = G * P < 8 ? G * P : 8;  // units summed in order
        constexpr int kLanes = kEight / P;             // on this many lanes
        const int first = (int)(threadIdx.x & 31u & ~(unsigned)(kLanes - 1));
        float C = 0.0f, S = 0.0f;
#pragma unroll
        for (int u = 0; u < kEight; ++u) {
            const float c = mul_r(model.live[u % P], model.cs[u % P]), s = mul_r(model.live[u % P], model.sn[u % P]);
            C = __fadd_rn(C, kLanes > 1 ? __shfl_sync(0xffffffffu, c, first + u / P) : c);
            S = __fadd_rn(S, kLanes > 1 ? __shfl_sync(0xffffffffu, s, first + u / P) : s);
        }
#pragma unroll
        for (int off = kLanes; off < G; off <<= 1) {
            C = __fadd_rn(C, __shfl_xor_sync(0xffffffffu, C, off));
            S = __fadd_rn(S, __shfl_xor_sync(0xffffffffu, S, off));
        }
        r[0] = C;
        r[1] = S;
    }
};

template <class M, typename Real, int G, int P>
__global__ void __launch_bounds__(SplitShape<G, P>::kThreads) em_split_kernel(const ForwardArgs a) {
    using Shape = SplitShape<G, P>;
    constexpr int kConsumers = 32 * Shape::kConsumerWarps, kProducers = 32 * Shape::kProducerWarps;
    constexpr bool kKahan = std::is_same<Real, float>::value;
    static_assert(M::U == 1, "phase models");
    __shared__ __align__(16) Real ring[2][kSplitSteps][Shape::kSlots];  // the normals; FP32: their sines and cosines
    __shared__ Real amps[2][kSplitSteps][kKahan ? (G * P > 1 ? Shape::kSlots / 2 : Shape::kSlots) : 1];  // FP32: a pair's amplitude
    __shared__ int s_bad[Shape::kOrbits];
    const int64_t orbit0 = (int64_t)blockIdx.x * Shape::kOrbits;
    const int units = a.units, nb = (units + 3) / 4;
    const uint32_t steps = a.k_end - a.k_begin;
    const bool producer = threadIdx.x >= kConsumers;
    if (threadIdx.x < Shape::kOrbits) s_bad[threadIdx.x] = 0;

    // Steps [from, from + kSplitSteps) of the run into ring[half] (those past
    // the run's end as well: nothing reads them).
    auto produce = [&](uint32_t from, int half) {
        const int per_step = Shape::kOrbits * nb;
        for (int i = (int)threadIdx.x - kConsumers; i < per_step * kSplitSteps; i += kProducers) {
            const int s = i / per_step, r = i - s * per_step, ob = r / nb, blk = r - ob * nb;
            const int64_t o = orbit0 + ob < a.orbits ? orbit0 + ob : a.orbits - 1;
            const U32x4 w = philox4x32_10(a.k_begin + from + (uint32_t)s, (uint32_t)blk, a.orbit_offset + (uint32_t)o,
                                          0u, a.keys);
            Real amp[2], z[4];
            box_muller_polar<Real>(w.x, w.y, amp[0], z[0], z[1]);
            box_muller_polar<Real>(w.z, w.w, amp[1], z[2], z[3]);
            Real *dst = &ring[half][s][ob * (G * P) + 4 * blk];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (G * P < 4 && j >= G * P) break;
                dst[j] = z[j];
                if (kKahan && j % 2 == 0) amps[half][s][(ob * (G * P) + 4 * blk + j) / (G * P > 1 ? 2 : 1)] = amp[j / 2];
            }
        }
    };

    if (producer) {
        produce(0, 0);
        __syncthreads();
        int half = 1;
        for (SplitChunks c(steps); !c.done(); c.next(), half ^= 1) {
            if (!c.last()) produce(c.from + kSplitSteps, half);
            __syncthreads();
        }
        __syncthreads();
        return;
    }

    const int ob = threadIdx.x / G, lig = threadIdx.x & (G - 1), u0 = lig * P;
    const bool active = orbit0 + ob < a.orbits;
    const int64_t o = active ? orbit0 + ob : a.orbits - 1;
    const int64_t n = a.n;
    (void)SDEB_CHECK(a.check, o >= 0 && o < a.orbits, kChkForwardState, o);
    M model;
    model.load(static_cast<const Real *>(a.params) + o * a.param_stride, u0, units, a.dt, sqrt(a.dt));
    Real *xrow = static_cast<Real *>(a.x) + o * n;
    Real x[1][P], cp[1][P];
    load_units<Real, 1, P>(xrow, units, u0, x);
    if constexpr (kKahan) {
        load_units<float, 1, P>(a.comp + o * n, units, u0, cp);
    } else {
#pragma unroll
        for (int i = 0; i < P; ++i) cp[0][i] = Real(0);
    }
    Real *frames = static_cast<Real *>(a.frames);
    uint32_t to_frame = a.stride - (a.k_begin % a.stride);
    auto make_reduce = [&]() {
        if constexpr (kKahan) {
            return EightsSum<M, G, P>{model};
        } else if constexpr (G > 32) {
            __shared__ TeamPartial team[2 * (G / 32)];
            return TeamFixedSum<Shape::kConsumerWarps, 1>{team, 0};
        } else {
            return WarpGroupSum<G>();
        }
    };
    auto reduce = make_reduce();
    // A step's normals, read one step ahead; padding units get zeros.
    const int slot = ob * (G * P) + u0;
    auto read = [&](int half, int s, Real(&amp)[kNoisePairs<P>], Real(&z)[P]) {
#pragma unroll
        for (int i = 0; i < P; ++i) z[i] = u0 + i < units ? ring[half][s][slot + i] : Real(0);
#pragma unroll
        for (int j = 0; j < kNoisePairs<P>; ++j)
            amp[j] = !kKahan ? Real(1) : u0 + 2 * j < units ? amps[half][s][slot / (G * P > 1 ? 2 : 1) + j] : Real(0);
    };
    __syncthreads();  // the first half is full
    int half = 0;
    for (SplitChunks c(steps); !c.done(); c.next(), half ^= 1) {
        const int count = (int)c.count();
        Real amp_next[kNoisePairs<P>], z_next[P];
        read(half, 0, amp_next, z_next);
#pragma unroll 1
        for (int s = 0; s < count; ++s) {
            Real amp[kNoisePairs<P>], z[P];
#pragma unroll
            for (int j = 0; j < kNoisePairs<P>; ++j) amp[j] = amp_next[j];
#pragma unroll
            for (int i = 0; i < P; ++i) z[i] = z_next[i];
            read(half, min(s + 1, kSplitSteps - 1), amp_next, z_next);
            em_step_noise<M, Real, P>(model, x, cp, amp, z, u0, units, reduce);
            const uint32_t k = a.k_begin + c.from + (uint32_t)s + 1;
            if constexpr (M::kDelayedComp) {
                if ((k & (kCompPeriod - 1u)) == 0) renormalize_units(x, cp);
            }
            if (--to_frame == 0) {
                to_frame = a.stride;
                const int64_t f = (int64_t)(k / a.stride);
                if (frames != nullptr && active && SDEB_CHECK(a.check, f < a.nframes, kChkForwardFrame, f)) {
                    Real v[1][P];
                    unit_values(x, cp, v);
                    store_units<Real, 1, P>(frames + (f * a.orbits + o) * n, units, u0, v);
                }
            }
        }
        __syncthreads();
    }
    if constexpr (M::kDelayedComp) {
        if (a.final_value) {
            Real v[1][P];
            unit_values(x, cp, v);
#pragma unroll
            for (int i = 0; i < P; ++i) {
                x[0][i] = v[0][i];
                cp[0][i] = Real(0);
            }
        }
    }
    bool bad = false;
#pragma unroll
    for (int i = 0; i < P; ++i)
        if (u0 + i < units && !isfinite(state_value(x[0][i], cp[0][i]))) bad = true;
    if (bad) s_bad[ob] = 1;
    if (active) {
        store_units<Real, 1, P>(xrow, units, u0, x);
        if constexpr (kKahan) store_units<float, 1, P>(a.comp + o * n, units, u0, cp);
    }
    __syncthreads();
    if (active && lig == 0) a.flags[o] = s_bad[ob] ? 1u : 0u;
}

template <class M, typename Real, int G, int P>
cudaError_t launch_split_layout(const ForwardArgs &a, cudaStream_t s) {
    using Shape = SplitShape<G, P>;
    const int64_t grid = (a.orbits + Shape::kOrbits - 1) / Shape::kOrbits;
    em_split_kernel<M, Real, G, P><<<(unsigned)grid, Shape::kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <template <typename, int> class MF, typename Real>
cudaError_t launch_split(const ForwardArgs &a, cudaStream_t s) {
#define SDEB_SPLIT(G_, P_) \
    if (a.units <= (G_) * (P_)) return launch_split_layout<MF<Real, P_>, Real, G_, P_>(a, s);
    SDEB_SPLIT(1, 1)
    SDEB_SPLIT(2, 1)
    SDEB_SPLIT(4, 1)
    SDEB_SPLIT(8, 1)
    SDEB_SPLIT(16, 1)
    SDEB_SPLIT(32, 1)
    if constexpr (sizeof(Real) == 8) {
        SDEB_SPLIT(64, 1)
        SDEB_SPLIT(128, 1)
        SDEB_SPLIT(256, 1)
    } else {
        SDEB_SPLIT(32, 2)
        SDEB_SPLIT(32, 4)
    }
#undef SDEB_SPLIT
    return cudaErrorNotSupported;
}

// Where the line lies, measured for n = 2 to 256 and 2^8 to 2^17 units in all,
// 300 steps, this kernel against the others (us):
//   FP64, n = 8   4864 units 202 / 446, 9728 202 / 446, 19456 235 / 443, 38912
//                 (the line) 381 / 446; n = 2, 64, 256 there 313 / 431, 365 / 459,
//                 435 / 492; past it, before its sums kept small phases' bits,
//                 2^16 502 / 500, 2^17 928 / 814
//   FP32, n = 8   2^13 units  48 /  89, 2^14  56 /  89, 2^15  74 /  89, 2^16 122 /  89
// (n = 2 in FP32 crosses between 2^14, 44 / 52, and 2^15, 64 / 52).  So: two
// warps of consumers for every sub-partition of the GPU in FP64, one in FP32,
// and in FP32 not past 128 units, where a lane has its eight units in either
// kernel (n = 256: 99 / 95).  A layout that was asked for runs as asked.
inline bool use_split(const ForwardArgs &a, bool fp64) {
    if (a.asked || a.ckpt != nullptr || a.nckpt > 0 || (!fp64 && a.units > 128)) return false;
    int64_t lanes = 1;
    while (lanes < a.units && (fp64 || lanes < 32)) lanes *= 2;
    return a.orbits <= (int64_t)kNumSms * 4 * 32 * (fp64 ? 2 : 1) / lanes;
}

}  // namespace sdeb
