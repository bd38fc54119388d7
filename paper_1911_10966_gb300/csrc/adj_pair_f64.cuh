// Float64 reverse of the Chandrashekar two-point flux in pair form, shared by the adjoint's interface terms
// (adjoint_f64.cu) and, for elements outside the fixed-point range, its pair loop (adj_pairs_fix.cu).
#pragma once

#include <cuda_runtime.h>

#include "esdc_internal.h"
#include "rcp_f64.cuh"

namespace esdc {
namespace {

// Pair form of a node's primitives for the ES-C reverse: half velocities and a quarter of |u|^2, so
// that the averages of the two-point flux are single additions.
struct PrimH {
    double rho, h0, h1, h2, beta, qsq;
};
// Cotangent accumulators of the ES-C reverse in pair form: rho and beta as in PBar, u twice the
// velocity cotangent, c the sum of the cotangents of c5 (the |u|^2 cotangent is -c/4); raw_to_pbar
// converts.
struct PRaw {
    double rho, u0, u1, u2, beta, c;
};

// Reverse of the contracted Chandrashekar flux f(a, b; n) for the cotangent mu[5]: adds the pair-form
// cotangents of both states to ab, bb.  Two reciprocals, 1/(rho_a + rho_b) (one Newton step: it only
// forms f = (a - b)/(a + b)) and 1/(beta_a + beta_b), which serves p_t and the reciprocal of the beta
// log mean.  Logarithmic means (series branch, u = f^2 < 1e-4, F(u) = artanh(f)/f = 1 + u/3 + u^2/5 +
// u^3/7 + u^4/9, G = 1/F = 1 - u/3 - 4u^2/45 - 44u^3/945):
//   rho:  L = (a + b) G/2,  dL/da = G/2 - f F'(u) G^2 (1 - f),  dL/db = G/2 + f F'(u) G^2 (1 + f);
//   beta: only 1/L enters the flux, IL = 2 F/(a + b), dIL/da = 2 (2 f F'(u) (1 - f) - F)/(a + b)^2,
//         dIL/db = -2 (2 f F'(u) (1 + f) + F)/(a + b)^2;
// otherwise, with l = log(a/b): L = (a - b)/l, dL/da = (1 - L/a)/l, dL/db = (L/b - 1)/l, and
// IL = l/(a - b), dIL/da = (1/a - IL)/(a - b), dIL/db = (IL - 1/b)/(a - b).
__device__ __forceinline__ void ec_pair_vjp(const PrimH& a, const PrimH& b, double n0, double n1, double n2,
                                            const double mu[5], const Phys& ph, PRaw& ab, PRaw& bb) {
    const double sr = a.rho + b.rho, sb = a.beta + b.beta;
    const double rsb = rcp_cubic(sb);
    // rho log mean and its partial derivatives
    double Lr, Lra, Lrb;
    {
        const double d = a.rho - b.rho;
        const double f = d * rcp_newton1(sr);
        const double u = f * f;
        if (u < 1.0e-4) {
            const double hG = fma(u, fma(u, fma(u, -22.0 / 945.0, -2.0 / 45.0), -1.0 / 6.0), 0.5);          // G/2
            const double Fp4 = fma(u, fma(u, fma(u, 16.0 / 9.0, 12.0 / 7.0), 8.0 / 5.0), 4.0 / 3.0);     // 4 F'
            const double W = f * Fp4 * (hG * hG);                                                          // f F' G^2
            const double Y = W * f;
            Lr = sr * hG;
            Lra = hG - W + Y;
            Lrb = hG + W + Y;
        } else {
            const double ra = rcp_cubic(a.rho), rb = rcp_cubic(b.rho);
            const double rl = rcp_cubic(log(a.rho * rb));
            Lr = d * rl;
            Lra = fma(-Lr, ra, 1.0) * rl;
            Lrb = fma(Lr, rb, -1.0) * rl;
        }
    }
    // reciprocal of the beta log mean and its partial derivatives: dIL/da = sc Ab, dIL/db = sc Bb
    double IB, sc, Ab, Bb;
    {
        const double d = a.beta - b.beta;
        const double f = d * rsb;
        const double u = f * f;
        if (u < 1.0e-4) {
            const double F = fma(u, fma(u, fma(u, fma(u, 1.0 / 9.0, 1.0 / 7.0), 1.0 / 5.0), 1.0 / 3.0), 1.0);
            const double Fp2 = fma(u, fma(u, fma(u, 8.0 / 9.0, 6.0 / 7.0), 4.0 / 5.0), 2.0 / 3.0);      // 2 F'
            const double w = f * Fp2;
            const double X = w * f;
            IB = 2.0 * F * rsb;
            sc = 2.0 * rsb * rsb;
            Ab = w - X - F;
            Bb = -(w + X + F);
        } else {
            const double ra = rcp_cubic(a.beta), rb = rcp_cubic(b.beta);
            sc = rcp_cubic(d);
            IB = log(a.beta * rb) * sc;
            Ab = ra - IB;
            Bb = IB - rb;
        }
    }
    const double hig = 0.5 * ph.inv_gm1;
    const double ub0 = a.h0 + b.h0, ub1 = a.h1 + b.h1, ub2 = a.h2 + b.h2;
    const double un = ub0 * n0 + ub1 * n1 + ub2 * n2;
    const double pt = 0.5 * sr * rsb;
    const double f1 = Lr * un;
    const double c5 = fma(hig, IB, -(a.qsq + b.qsq));
    // reverse
    const double fmb0 = fma(mu[4], ub0, mu[1]), fmb1 = fma(mu[4], ub1, mu[2]), fmb2 = fma(mu[4], ub2, mu[3]);
    const double f1b = mu[0] + mu[4] * c5 + fmb0 * ub0 + fmb1 * ub1 + fmb2 * ub2;
    const double c5b = mu[4] * f1;
    const double ptb = fmb0 * n0 + fmb1 * n1 + fmb2 * n2;
    const double unb = f1b * Lr;
    const double Lrb_ = f1b * un;
    // pt = (rho_a + rho_b)/(2 (beta_a + beta_b)): d pt/d rho = 1/(2 sb), d pt/d beta = -pt/sb
    const double ptr = ptb * rsb;
    const double hp = 0.5 * ptr;
    const double bp = -pt * ptr;
    const double S = c5b * hig * sc;
    ab.rho += fma(Lrb_, Lra, hp);
    bb.rho += fma(Lrb_, Lrb, hp);
    ab.beta += fma(S, Ab, bp);
    bb.beta += fma(S, Bb, bp);
    ab.c += c5b;
    bb.c += c5b;
    // ubar cotangent mu_5 f_m + fmb f1 + unb n with f_m = f1 ubar + p_t n:
    // f1 (mu_5 ubar + fmb) + (mu_5 p_t + unb) n
    const double An = fma(mu[4], pt, unb);
    const double ubb0 = fma(f1, fma(mu[4], ub0, fmb0), An * n0);
    const double ubb1 = fma(f1, fma(mu[4], ub1, fmb1), An * n1);
    const double ubb2 = fma(f1, fma(mu[4], ub2, fmb2), An * n2);
    ab.u0 += ubb0;
    ab.u1 += ubb1;
    ab.u2 += ubb2;
    bb.u0 += ubb0;
    bb.u1 += ubb1;
    bb.u2 += ubb2;
}

}  // namespace
}  // namespace esdc
