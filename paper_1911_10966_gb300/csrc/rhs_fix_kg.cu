// Fixed-point residual kernels: SF-KG flux.
#include "rhs_fix.cuh"

namespace esdc {

cudaError_t prepare_fix_kg(const esdc_ctx* c) { return prepare_vf<kFluxKG, false>(c); }
cudaError_t launch_fix_kg(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    return launch_vf<kFluxKG, false>(c, q, dqdt, s);
}

}  // namespace esdc
