// Few-orbit forward kernel instantiations: Kuramoto models, float.
#include "em_split_impl.cuh"

namespace sdeb {

cudaError_t launch_forward_split_f32(const ForwardArgs &a, cudaStream_t s) {
    if (!use_split(a, false)) return cudaErrorNotSupported;
    if (a.model == kKuramoto) return launch_split<KuramotoScalarLane, float>(a, s);
    return launch_split<KuramotoPaperLane, float>(a, s);
}

}  // namespace sdeb
