// Float64 residual launchers: for p <= 7 the element kernel of the context's volume flux and interface options
// (rhs_fix.cuh), then visc_sat_kernel (visc_sat.cuh), which adds the BR1 interface term
// (E_ii/2)(Ftilde_nbr - Ftilde_own) / (w_i J) on face nodes once every element's traces exist; p = 15 in passes
// (rhs_large_f64.cu).
#include <cuda_runtime.h>

#include "esdc_internal.h"
#include "kernels.h"
#include "visc_sat.cuh"

namespace esdc {
namespace {

// matrix dissipation, interior penalty, boundary faces, source or surface metrics: compiled into kernel
// instances of their own, so that the default ones carry none of them
bool extra_face_terms(const esdc_ctx* c) {
    return c->phys.dissipation == 2 || c->phys.ip_coef > 0.0 || c->setup.bounded != 0 || c->d_src || c->d_nsurf;
}

cudaError_t prepare_element(const esdc_ctx* c) {
    const bool xf = extra_face_terms(c);
    switch (c->setup.volume_flux) {
        case ESDC_FLUX_ESC: return xf ? prepare_fix_esc_xf(c) : prepare_fix_esc(c);
        case ESDC_FLUX_KG: return xf ? prepare_fix_kg_xf(c) : prepare_fix_kg(c);
        case ESDC_FLUX_DC: return xf ? prepare_fix_dc_xf(c) : prepare_fix_dc(c);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_element(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s) {
    const bool xf = extra_face_terms(c);
    switch (c->setup.volume_flux) {
        case ESDC_FLUX_ESC: return xf ? launch_fix_esc_xf(c, q, dqdt, s) : launch_fix_esc(c, q, dqdt, s);
        case ESDC_FLUX_KG: return xf ? launch_fix_kg_xf(c, q, dqdt, s) : launch_fix_kg(c, q, dqdt, s);
        case ESDC_FLUX_DC: return xf ? launch_fix_dc_xf(c, q, dqdt, s) : launch_fix_dc(c, q, dqdt, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int N>
cudaError_t launch_rhs_n(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    if (ev) cudaEventRecord(ev[0], s);
    cudaError_t e = launch_element(c, q, dqdt, s);
    if (e != cudaSuccess) return e;
    if (ev) cudaEventRecord(ev[1], s);
    if (ev) cudaEventRecord(ev[2], s);
    if (c->phys.viscous) {
        e = launch_visc_sat<double, N, true>(dqdt, c->d_jinv, c->d_nbr, (const double*)c->d_trace, c->K,
                                             c->ops.winv[0], s);
        if (e != cudaSuccess) return e;
    }
    if (ev) cudaEventRecord(ev[3], s);
    return cudaGetLastError();
}

}  // namespace

// A CTA with one element out of range takes the float64 form after its share of phase 0, at about 1.05 times the
// float64 kernel's cost against 0.35 of a CTA that stays in fixed point.
bool float64_form(const esdc_ctx* c, const int32_t* kn) {
    const int N3 = c->N3, epb = N3 >= 96 ? 1 : (N3 >= 48 ? 2 : (N3 >= 24 ? 4 : 16));
    int64_t out = 0, blocks = (c->K + epb - 1) / epb;
    for (int64_t b = 0; b < blocks; ++b) {
        bool s = false;
        for (int64_t e = b * epb; e < c->K && e < (b + 1) * epb; ++e) s = s || kn[e] == kStretched;
        out += s;
    }
    return 8 * out > 7 * blocks;
}

// Opt the element kernel into more than 48 KB of dynamic shared memory (on the current device).
cudaError_t prepare_rhs_f64(const esdc_ctx* c) {
    return c->N == kLargeN ? cudaSuccess : prepare_element(c);
}

cudaError_t launch_rhs_f64(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    switch (c->N) {
        case 2: return launch_rhs_n<2>(c, q, dqdt, s, ev);
        case 3: return launch_rhs_n<3>(c, q, dqdt, s, ev);
        case 4: return launch_rhs_n<4>(c, q, dqdt, s, ev);
        case 5: return launch_rhs_n<5>(c, q, dqdt, s, ev);
        case 6: return launch_rhs_n<6>(c, q, dqdt, s, ev);
        case 7: return launch_rhs_n<7>(c, q, dqdt, s, ev);
        case 8: return launch_rhs_n<8>(c, q, dqdt, s, ev);
        case kLargeN: return launch_rhs_large(c, q, dqdt, s, ev);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace esdc
