// Fixed-point residual kernels: DC flux, with the optional interface terms.
#include "rhs_fix.cuh"

namespace esdc {

cudaError_t prepare_fix_dc_xf(const esdc_ctx* c) { return prepare_vf<kFluxDC, true>(c); }
cudaError_t launch_fix_dc_xf(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    return launch_vf<kFluxDC, true>(c, q, dqdt, s);
}

}  // namespace esdc
