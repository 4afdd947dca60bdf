// The chunks of eight steps in which the few-orbit kernel hands the noise from
// its producer warps to its consumer warps.  Both sides walk the same chunks,
// by the steps that are left: a run may have up to 2^32 - 1 steps, so the
// first step of a chunk past its end does not fit its type.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SDEB_HD __host__ __device__ __forceinline__
#else
#define SDEB_HD inline
#endif

namespace sdeb {

struct SplitChunks {
    static constexpr uint32_t kSteps = 8;
    uint32_t from = 0;  // first step of the chunk
    uint32_t left;      // steps from there to the end
    SDEB_HD explicit SplitChunks(uint32_t steps) : left(steps) {}
    SDEB_HD bool done() const { return left == 0; }
    SDEB_HD bool last() const { return left <= kSteps; }
    SDEB_HD uint32_t count() const { return last() ? left : kSteps; }
    SDEB_HD void next() {
        left -= count();
        from += kSteps;
    }
};

}  // namespace sdeb
