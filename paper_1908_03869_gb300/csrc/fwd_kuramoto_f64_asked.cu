// Forward kernel instantiations: Kuramoto models, double, the layouts that only run when they are asked for.
#include "em_forward_impl.cuh"

namespace sdeb {

cudaError_t launch_forward_kuramoto_f64_asked(const ForwardArgs &a, Layout l, cudaStream_t s) {
    if (a.model == kKuramoto) return dispatch_asked_layouts_f64<KuramotoScalarLane>(a, l, s);
    if (a.model == kKuramotoPaper) return dispatch_asked_layouts_f64<KuramotoPaperLane>(a, l, s);
    return cudaErrorNotSupported;
}

}  // namespace sdeb
