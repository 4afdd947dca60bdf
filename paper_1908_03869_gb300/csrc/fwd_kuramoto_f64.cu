// Forward kernel instantiations: Kuramoto models, double.
#include "em_forward_impl.cuh"

namespace sdeb {

cudaError_t launch_forward_kuramoto_f64(const ForwardArgs &a, Layout l, cudaStream_t s) {
    if (a.asked) {
        const cudaError_t e = launch_forward_kuramoto_f64_asked(a, l, s);
        if (e != cudaErrorNotSupported) return e;
    }
    if (a.model == kKuramoto) return dispatch_phase_layouts_f64<KuramotoScalarLane>(a, l, s);
    if (a.model == kKuramotoPaper) return dispatch_phase_layouts_f64<KuramotoPaperLane>(a, l, s);
    return cudaErrorNotSupported;
}

}  // namespace sdeb
