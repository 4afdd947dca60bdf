// Ensemble moments of the stored frames, accumulated in FP64 on the GPU.
//
// The paper's accuracy experiment (Sec. 2.3) reports, over realisations, the
// mean and the standard deviation of the Kuramoto order parameter r(t) of
// Eq. 7; an SDE user generally wants the mean and variance over orbits of
// every state component at every output time.  Both are computed here from
// the frames in HBM, whatever the context precision, with FP64 accumulators
// and in a fixed order (the same bits on every call):
//
//   1. a block takes one frame and one chunk of kMomChunk orbits; each thread
//      accumulates its share of one state component (or, for r, one orbit
//      after another) as shifted sums -- shift K = the first value it reads,
//      s1 = sum (x - K), s2 = sum (x - K)^2, so mean = K + s1 / c and
//      M2 = s2 - s1^2 / c without cancellation against a large mean;
//   2. the threads' (count, mean, M2) triples of a component are combined
//      by halving with the pairwise update of Chan, Golub and LeVeque
//      (1979): mean_ab = mean_a + d n_b / n, M2_ab = M2_a + M2_b +
//      d^2 n_a n_b / n, d = mean_b - mean_a;
//   3. a second kernel combines the chunks of a frame in a fixed order and
//      writes (mean, M2 / count): the mean and the population variance.
//
// The chunk size is fixed, so a frame's result does not depend on which
// frame range a call asks for.  Reading every frame element once is the HBM
// cost (the forward kernel that wrote them runs ~100x longer).
#include <algorithm>

#include "em_internal.h"

namespace sdeb {

namespace {

constexpr int kMomBlock = 256;

struct Acc {
    double cnt, mean, m2;
};

__device__ __forceinline__ void chan_merge(Acc &a, const Acc &b) {
    if (b.cnt == 0.0) return;
    if (a.cnt == 0.0) {
        a = b;
        return;
    }
    const double n = a.cnt + b.cnt;
    const double d = b.mean - a.mean;
    a.mean = fma(d, b.cnt / n, a.mean);
    a.m2 = a.m2 + b.m2 + d * d * (a.cnt * b.cnt / n);
    a.cnt = n;
}

__device__ __forceinline__ Acc acc_from_shifted(double cnt, double K, double s1, double s2) {
    Acc a{0.0, 0.0, 0.0};
    if (cnt > 0.0) {
        a.cnt = cnt;
        a.mean = K + s1 / cnt;
        a.m2 = fmax(s2 - s1 * (s1 / cnt), 0.0);
    }
    return a;
}

// s += a, and the error of that sum exactly (D. E. Knuth's two-sum).
__device__ __forceinline__ float two_sum_add(float &s, float a) {
    const float t = __fadd_rn(s, a);
    const float z = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(a, z));
    s = t;
    return e;
}

// A sum of FP32 terms as three FP32 numbers: the value, the errors of its sums
// and the errors of theirs.
struct TripleSum {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) { add_low(two_sum_add(a, x)); }
    __device__ __forceinline__ void add_low(float x) { c = __fadd_rn(c, two_sum_add(b, x)); }  // of 2^-24 of the terms' size
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

// Elements whose shifted sums are carried in FP32 before they go to the FP64
// accumulators.
constexpr int kMomGroup = 16;

// s1 += sum (x - K), s2 += sum (x - K)^2 over the elements x[0], x[step], ...
// (count of them) of one thread.  An SM takes 128 FP32 operations a clock and
// 1.68 FP64 ones, so FP32 elements are summed as FP32 triples, kMomGroup at a
// time: x - K is split exactly into dh + dl, and (dh + dl)^2 into terms that
// drop less than 2^-70 of it.  A group's sums are off by some 2^-66, so the
// FP64 sums round once a group instead of once an element: at or below the error of
// adding the elements one by one in FP64.  (With FP32 pairs, 25 operations an
// element instead of 62, a group is off by 2^-47, and the variance of 64 or
// 300 orbits was 4 to 20 times further off than with FP64 sums.)  Half an FP64
// operation an element instead of 5.  Elements so far from K (2^60), or all so
// near it (2^-40), that a product or its error leaves the FP32 range, and
// non-finite ones, are taken again in FP64.
__device__ __forceinline__ void shifted_sums_f64(const float *x, int64_t step, int count, double K, double &s1,
                                                 double &s2) {
    s1 = s2 = 0.0;
    for (int i = 0; i < count; ++i) {
        const double d = (double)x[i * step] - K;
        s1 += d;
        s2 = fma(d, d, s2);
    }
}

__device__ __forceinline__ void shifted_sums(const float *x, int64_t step, int count, double &K, double &s1,
                                             double &s2) {
    const float Kf = x[0];
    K = (double)Kf;
    float far = 0.0f;
    for (int i0 = 0; i0 < count; i0 += kMomGroup) {
        float v[kMomGroup];
#pragma unroll
        for (int i = 0; i < kMomGroup; ++i) v[i] = i0 + i < count ? x[(i0 + i) * step] : Kf;  // past the end: d = 0
        TripleSum sum, sq;
#pragma unroll
        for (int i = 0; i < kMomGroup; ++i) {
            const float dh = __fsub_rn(v[i], Kf);
            const float z = __fsub_rn(dh, v[i]);
            const float dl = __fsub_rn(__fsub_rn(v[i], __fsub_rn(dh, z)), __fadd_rn(Kf, z));
            far = fmaxf(far, fabsf(dh));
            sum.add(dh);
            sum.add_low(dl);
            // (dh + dl)^2 = p + e + c1 + c2: dh^2 and its error, 2 dh dl and its error with dl^2
            const float p = __fmul_rn(dh, dh), h2 = __fadd_rn(dh, dh);
            const float c1 = __fmul_rn(h2, dl);
            sq.add(p);
            sq.add_low(__fmaf_rn(dh, dh, -p));
            sq.add_low(c1);
            sq.c = __fadd_rn(sq.c, __fmaf_rn(dl, dl, __fmaf_rn(h2, dl, -c1)));
        }
        s1 += sum.value();
        s2 += sq.value();
    }
    const bool in_range = far == 0.0f || (far >= 0x1p-40f && far <= 0x1p60f);
    if (!in_range || !isfinite(s1) || !isfinite(s2)) shifted_sums_f64(x, step, count, K, s1, s2);
}

__device__ __forceinline__ void shifted_sums(const double *x, int64_t step, int count, double &K, double &s1,
                                             double &s2) {
    K = x[0];
    for (int i = 0; i < count; ++i) {
        const double d = x[i * step] - K;
        s1 += d;
        s2 = fma(d, d, s2);
    }
}

// Per (frame, chunk) block: the moments of every state component over the
// chunk's orbits.  Components cb .. cb + ncomp - 1 are taken 256 at a time;
// thread t reads component comp = t mod ncomp of the orbits row, row + R,
// ... (R = 256 / ncomp rows), so consecutive threads read consecutive
// addresses.  The rows are merged by halving.
template <typename Real>
__global__ void __launch_bounds__(kMomBlock) state_moments_partial(const Real *frames, int64_t orbits, int n,
                                                                   int64_t f0, int64_t nframes, int C, Acc *part,
                                                                   unsigned long long *check) {
    __shared__ Acc sh[kMomBlock];
    const int c = (int)(blockIdx.x % (unsigned)C);
    const int64_t fr = blockIdx.x / (unsigned)C;
    if (!SDEB_CHECK(check, f0 + fr < nframes, kChkMomentFrame, f0 + fr)) return;  // uniform over the block
    const int64_t o0 = (int64_t)c * kMomChunk;
    const int in_chunk = (int)min(orbits - o0, kMomChunk);
    const Real *base = frames + ((f0 + fr) * orbits + o0) * (int64_t)n;
    const int t = threadIdx.x;
    for (int cb = 0; cb < n; cb += kMomBlock) {
        const int ncomp = min(n - cb, kMomBlock);
        const int R = kMomBlock / ncomp;
        const int row = t / ncomp, comp = cb + (t - row * ncomp);
        double K = 0.0, s1 = 0.0, s2 = 0.0;
        int count = 0;
        if (row < R && row < in_chunk) {
            count = (in_chunk - row + R - 1) / R;
            shifted_sums(base + (int64_t)row * n + comp, (int64_t)R * n, count, K, s1, s2);
        }
        sh[t] = acc_from_shifted((double)count, K, s1, s2);
        __syncthreads();
        for (int live = R; live > 1;) {
            const int half = (live + 1) / 2;
            if (row < half && row + half < live) chan_merge(sh[t], sh[t + half * ncomp]);
            live = half;
            __syncthreads();
        }
        if (t < ncomp) part[(fr * C + c) * (int64_t)n + cb + t] = sh[t];
        __syncthreads();
    }
}

// Per (frame, chunk) block: the moments of the order parameter of Eq. 7,
// r = |(1/n) sum_j exp(i theta_j)|, over the chunk's orbits.  A group of G
// lanes takes one orbit at a time: each lane sums cos and sin of components
// lig, lig + G, ... in the frame's precision (FP32: the phase reduced to
// [-pi, pi] and the special-function unit; FP64: fixed point) and the group
// adds them by a butterfly.  After J orbits (at most G) each lane has the
// sums of one of them, forms its r in FP64 and accumulates it: the FP64
// sequence (a root, nine more operations) runs once a lane and orbit, not
// once a group of lanes and orbit with one lane of them at work.  Every group
// runs the same number of iterations, so the shuffles always have the whole
// warp.
template <typename Real, int G>
__global__ void __launch_bounds__(kMomBlock) r_moments_partial(const Real *frames, int64_t orbits, int n,
                                                               int64_t f0, int64_t nframes, int C, Acc *part,
                                                               unsigned long long *check) {
    constexpr int kGroups = kMomBlock / G;
    __shared__ Acc sh[kMomBlock];
    const int c = (int)(blockIdx.x % (unsigned)C);
    const int64_t fr = blockIdx.x / (unsigned)C;
    if (!SDEB_CHECK(check, f0 + fr < nframes, kChkMomentFrame, f0 + fr)) return;  // uniform over the block
    const int64_t o0 = (int64_t)c * kMomChunk;
    const int in_chunk = (int)min(orbits - o0, kMomChunk);
    const Real *base = frames + ((f0 + fr) * orbits + o0) * (int64_t)n;
    const int g = threadIdx.x / G, lig = threadIdx.x & (G - 1);
    const int J = min(G, (in_chunk + kGroups - 1) / kGroups);
    const double inv_n = 1.0 / (double)n;
    double K = 0.0, s1 = 0.0, s2 = 0.0;
    int count = 0;
    for (int first = 0; first < in_chunk; first += J * kGroups) {
        Real Cm = Real(0), Sm = Real(0);
        for (int j = 0; j < J; ++j) {
            const int o = first + j * kGroups + g;
            Real Cs = Real(0), Ss = Real(0);
            if (o < in_chunk) {
                const Real *row = base + (int64_t)o * n;
#pragma unroll 4
                for (int i = lig; i < n; i += G) {
                    Real s, co;
                    sincos_phase(row[i], s, co);
                    Cs += co;
                    Ss += s;
                }
            }
            Cs = group_sum<G>(Cs);
            Ss = group_sum<G>(Ss);
            if (j == lig) {
                Cm = Cs;
                Sm = Ss;
            }
        }
        if (lig < J && first + lig * kGroups + g < in_chunk) {
            const double Cd = (double)Cm, Sd = (double)Sm;
            const double r = sqrt(fma(Cd, Cd, Sd * Sd)) * inv_n;
            if (count == 0) K = r;
            const double d = r - K;
            s1 += d;
            s2 = fma(d, d, s2);
            ++count;
        }
    }
    const int t = threadIdx.x;
    sh[t] = acc_from_shifted((double)count, K, s1, s2);
    __syncthreads();
    for (int half = kMomBlock / 2; half > 0; half /= 2) {
        if (t < half) chan_merge(sh[t], sh[t + half]);
        __syncthreads();
    }
    if (t == 0) part[fr * C + c] = sh[0];
}

// out[i][0..1] = (mean, population variance) of the chunks of item i (an
// item is a (frame, component) pair or a frame).  W lanes an item (1 or 32):
// lane l merges chunks l, l + W, ... in order, the lanes' results are merged
// by halving.
template <int W>
__global__ void merge_chunks(const Acc *part, int64_t items, int per_frame, int C, double *out) {
    const int lane = threadIdx.x & (W - 1);
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / W; i < items;
         i += (int64_t)gridDim.x * blockDim.x / W) {
        const int64_t fr = i / per_frame;
        const int q = (int)(i - fr * per_frame);
        Acc m{0.0, 0.0, 0.0};
        for (int c = lane; c < C; c += W) chan_merge(m, part[(fr * C + c) * per_frame + q]);
#pragma unroll
        for (int half = W / 2; half > 0; half /= 2) {
            const Acc b{__shfl_down_sync(0xffffffffu, m.cnt, half), __shfl_down_sync(0xffffffffu, m.mean, half),
                        __shfl_down_sync(0xffffffffu, m.m2, half)};
            if (lane < half) chan_merge(m, b);
        }
        if (lane == 0) {
            out[2 * i] = m.mean;
            out[2 * i + 1] = m.cnt > 0.0 ? m.m2 / m.cnt : 0.0;
        }
    }
}

template <typename Real>
cudaError_t launch_r_partial(const Real *frames, int64_t orbits, int n, int64_t f0, int64_t nframes, int C,
                             int64_t blocks, Acc *part, cudaStream_t s) {
    unsigned long long *ck = check_word();
    // Lanes an orbit: eight components a lane when the chunks are long (fewer
    // shuffles an orbit), one when they are short (64 orbits fill a block so).
    const int per_lane = orbits >= kMomChunk / 2 ? 8 : 1;
    const int lanes = (n + per_lane - 1) / per_lane;
#define SDEB_R_PARTIAL(G_) \
    r_moments_partial<Real, G_><<<(unsigned)blocks, kMomBlock, 0, s>>>(frames, orbits, n, f0, nframes, C, part, ck)
    if (lanes <= 1) SDEB_R_PARTIAL(1);
    else if (lanes <= 2) SDEB_R_PARTIAL(2);
    else if (lanes <= 4) SDEB_R_PARTIAL(4);
    else if (lanes <= 8) SDEB_R_PARTIAL(8);
    else if (lanes <= 16) SDEB_R_PARTIAL(16);
    else SDEB_R_PARTIAL(32);
#undef SDEB_R_PARTIAL
    return cudaGetLastError();
}

// The chunks of every item merged: a lane an item for few chunks, else a warp.
cudaError_t launch_merge(const Acc *part, int64_t items, int per_frame, int C, double *out, cudaStream_t s) {
    const int lanes = C <= 2 ? 1 : 32;
    const int64_t blocks = std::min<int64_t>((items * lanes + 255) / 256, 152 * 32);  // grid-stride loops
    if (lanes == 1) merge_chunks<1><<<(unsigned)blocks, 256, 0, s>>>(part, items, per_frame, C, out);
    else merge_chunks<32><<<(unsigned)blocks, 256, 0, s>>>(part, items, per_frame, C, out);
    return cudaGetLastError();
}

}  // namespace

FrameMomentsPlan frame_moments_plan(int64_t orbits, int n, int64_t count) {
    FrameMomentsPlan p;
    p.chunks = (int)((orbits + kMomChunk - 1) / kMomChunk);
    // frames per pass: partials of at most ~64 MiB and at most 2^31 - 1 blocks
    const int64_t per_frame = (int64_t)p.chunks * (n + 1) * (int64_t)sizeof(Acc);
    int64_t fb = std::max<int64_t>(1, (64ll << 20) / per_frame);
    fb = std::min<int64_t>(fb, 0x7fffffffLL / p.chunks);
    p.frames_per_pass = std::max<int64_t>(1, std::min<int64_t>(fb, count));
    p.partial_bytes = (size_t)(p.frames_per_pass * per_frame);
    p.out_bytes = (size_t)p.frames_per_pass * (n + 1) * 2 * sizeof(double);
    return p;
}

cudaError_t launch_frame_moments_pass(const void *frames, bool fp64, int64_t orbits, int n, int64_t f0,
                                      int64_t count, int64_t nframes, const FrameMomentsPlan &plan, void *partial,
                                      double *state_out, double *r_out, cudaStream_t s) {
    unsigned long long *ck = check_word();
    if (count <= 0) return cudaSuccess;
    const int C = plan.chunks;
    const int64_t blocks = (int64_t)C * count;
    Acc *part_state = static_cast<Acc *>(partial);
    Acc *part_r = part_state + count * C * (int64_t)n;
    cudaError_t e = cudaSuccess;
    if (state_out != nullptr) {
        if (fp64)
            state_moments_partial<double><<<(unsigned)blocks, kMomBlock, 0, s>>>(
                static_cast<const double *>(frames), orbits, n, f0, nframes, C, part_state, ck);
        else
            state_moments_partial<float><<<(unsigned)blocks, kMomBlock, 0, s>>>(
                static_cast<const float *>(frames), orbits, n, f0, nframes, C, part_state, ck);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        e = launch_merge(part_state, count * n, n, C, state_out, s);
        if (e != cudaSuccess) return e;
    }
    if (r_out != nullptr) {
        e = fp64 ? launch_r_partial<double>(static_cast<const double *>(frames), orbits, n, f0, nframes, C, blocks,
                                            part_r, s)
                 : launch_r_partial<float>(static_cast<const float *>(frames), orbits, n, f0, nframes, C, blocks,
                                           part_r, s);
        if (e != cudaSuccess) return e;
        e = launch_merge(part_r, count, 1, C, r_out, s);
    }
    return e;
}

}  // namespace sdeb
