// Float64 residual launchers for p <= 7.  The ES-C flux runs in block fixed point (rhs_fix_f64.cu); the
// SF-KG and DC fluxes run the float64 form (element_f64.cuh) as rhs_main_f64.
// visc_sat_kernel (visc_sat.cuh) then adds the BR1 interface term (E_ii/2)(Ftilde_nbr - Ftilde_own)
// / (w_i J) on face nodes once every element's traces exist.
#include <cuda_runtime.h>

#include "element_f64.cuh"
#include "esdc_internal.h"
#include "kernels.h"
#include "visc_sat.cuh"

namespace esdc {
namespace {

template <int N, int VF, bool XF>
__global__ void __launch_bounds__(Cfg<N>::THREADS, Cfg<N>::MINB)
rhs_main_f64(const double* __restrict__ q, double* __restrict__ dqdt, const double* __restrict__ geom,
             const int32_t* __restrict__ nbr, double* __restrict__ trace, int64_t K, const Ops ops,
             const Phys ph, const double* __restrict__ qext, const double* __restrict__ src,
             const double* __restrict__ nsurf, const double* __restrict__ fnorm) {
    extern __shared__ double smem[];
    element_f64<N, VF, XF>(smem, q, dqdt, geom, nbr, trace, K, ops, ph, qext, src, nsurf, fnorm);
}

// ---- host-side launchers

template <int N, int VF, bool XF>
cudaError_t launch_rhs_n(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s,
                         cudaEvent_t* ev) {
    using C = Cfg<N>;
    [[maybe_unused]] const size_t smem = (size_t)C::EPB * C::SM * sizeof(double);
    [[maybe_unused]] const unsigned grid = (unsigned)((c->K + C::EPB - 1) / C::EPB);
    if (ev) cudaEventRecord(ev[0], s);
    if constexpr (VF == kFluxESC) {
        const cudaError_t e = launch_rhs_fix(c, XF, q, dqdt, s);
        if (e != cudaSuccess) return e;
    } else {
        rhs_main_f64<N, VF, XF><<<grid, C::THREADS, smem, s>>>(q, dqdt, c->d_geom, c->d_nbr, (double*)c->d_trace, c->K,
                                                               c->ops, c->phys, c->d_qext, c->d_src, c->d_nsurf,
                                                               c->d_fnorm);
    }
    if (ev) cudaEventRecord(ev[1], s);
    if (ev) cudaEventRecord(ev[2], s);
    if (c->phys.viscous) {
        const cudaError_t e = launch_visc_sat<double, N, true>(dqdt, c->d_jinv, c->d_nbr, (const double*)c->d_trace,
                                                               c->K, c->ops.winv[0], s);
        if (e != cudaSuccess) return e;
    }
    if (ev) cudaEventRecord(ev[3], s);
    return cudaGetLastError();
}

template <int N, bool XF>
cudaError_t prepare_xf(int vf) {
    using C = Cfg<N>;
    const int smem = (int)(C::EPB * C::SM * sizeof(double));
    constexpr cudaFuncAttribute kAttr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    switch (vf) {
        case kFluxKG: return cudaFuncSetAttribute(rhs_main_f64<N, kFluxKG, XF>, kAttr, smem);
        case kFluxDC: return cudaFuncSetAttribute(rhs_main_f64<N, kFluxDC, XF>, kAttr, smem);
        default: return cudaErrorInvalidValue;
    }
}

bool extra_face_terms(const esdc_ctx* c) {
    return c->phys.dissipation == 2 || c->phys.ip_coef > 0.0 || c->setup.bounded != 0 || c->d_src || c->d_nsurf;
}

template <int N>
cudaError_t prepare_n(const esdc_ctx* c) {
    const int vf = c->setup.volume_flux;
    if (vf == kFluxESC) return prepare_rhs_fix(c, extra_face_terms(c));
    return extra_face_terms(c) ? prepare_xf<N, true>(vf) : prepare_xf<N, false>(vf);
}

template <int N, bool XF>
cudaError_t launch_vf_xf(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    switch (c->setup.volume_flux) {
        case kFluxESC: return launch_rhs_n<N, kFluxESC, XF>(c, q, dqdt, s, ev);
        case kFluxKG: return launch_rhs_n<N, kFluxKG, XF>(c, q, dqdt, s, ev);
        case kFluxDC: return launch_rhs_n<N, kFluxDC, XF>(c, q, dqdt, s, ev);
        default: return cudaErrorInvalidValue;
    }
}

template <int N>
cudaError_t launch_vf(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    return extra_face_terms(c) ? launch_vf_xf<N, true>(c, q, dqdt, s, ev) : launch_vf_xf<N, false>(c, q, dqdt, s, ev);
}

}  // namespace

// Opt the fused kernel into more than 48 KB of dynamic shared memory (on the current device).
cudaError_t prepare_rhs_f64(const esdc_ctx* c) {
    switch (c->N) {
        case 2: return prepare_n<2>(c);
        case 3: return prepare_n<3>(c);
        case 4: return prepare_n<4>(c);
        case 5: return prepare_n<5>(c);
        case 6: return prepare_n<6>(c);
        case 7: return prepare_n<7>(c);
        case 8: return prepare_n<8>(c);
        case kLargeN: return prepare_rhs_large(c);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_rhs_f64(const esdc_ctx* c, const double* q, double* dqdt, cudaStream_t s, cudaEvent_t* ev) {
    switch (c->N) {
        case 2: return launch_vf<2>(c, q, dqdt, s, ev);
        case 3: return launch_vf<3>(c, q, dqdt, s, ev);
        case 4: return launch_vf<4>(c, q, dqdt, s, ev);
        case 5: return launch_vf<5>(c, q, dqdt, s, ev);
        case 6: return launch_vf<6>(c, q, dqdt, s, ev);
        case 7: return launch_vf<7>(c, q, dqdt, s, ev);
        case 8: return launch_vf<8>(c, q, dqdt, s, ev);
        case kLargeN: return launch_rhs_large(c, q, dqdt, s, ev);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace esdc
