// Few-orbit forward kernel instantiations: Kuramoto models, double.
#include "em_split_impl.cuh"

namespace sdeb {

cudaError_t launch_forward_split_f64(const ForwardArgs &a, cudaStream_t s) {
    if (!use_split(a, true)) return cudaErrorNotSupported;
    if (a.model == kKuramoto) return launch_split<KuramotoScalarLane, double>(a, s);
    return launch_split<KuramotoPaperLane, double>(a, s);
}

}  // namespace sdeb
