// Fixed-point residual kernels: DC flux.
#include "rhs_fix.cuh"

namespace esdc {

cudaError_t prepare_fix_dc(const esdc_ctx* c) { return prepare_vf<kFluxDC, false>(c); }
cudaError_t launch_fix_dc(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    return launch_vf<kFluxDC, false>(c, q, dqdt, s);
}

}  // namespace esdc
