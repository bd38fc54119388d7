// Fixed-point residual kernels: ES-C flux.
#include "rhs_fix.cuh"

namespace esdc {

cudaError_t prepare_fix_esc(const esdc_ctx* c) { return prepare_vf<kFluxESC, false>(c); }
cudaError_t launch_fix_esc(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    return launch_vf<kFluxESC, false>(c, q, dqdt, s);
}

}  // namespace esdc
