// Fixed-point residual kernels: SF-KG flux, with the optional interface terms.
#include "rhs_fix.cuh"

namespace esdc {

cudaError_t prepare_fix_kg_xf(const esdc_ctx* c) { return prepare_vf<kFluxKG, true>(c); }
cudaError_t launch_fix_kg_xf(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    return launch_vf<kFluxKG, true>(c, q, dqdt, s);
}

}  // namespace esdc
