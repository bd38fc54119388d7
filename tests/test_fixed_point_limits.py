"""The two-point fluxes of csrc/fix_f64.cuh and their reverse with every operand at or next to the largest value
that its exponent admits: no signed 64-bit sum may overflow (the program traps where one does), and each flux
agrees with extended precision.  Bound: a flux takes fewer than 40 products, each within 2.5 units of 2^-60 and
multiplied by less than 3/2 on its way into the result, so 256 units, 2^-52 of the block's unit."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "fix_f64.cuh"
using namespace esdc;
typedef long double Q;
static Q log_mean(Q a, Q b) {
    const Q f = (a - b) / (a + b), u = f * f;
    if (u > 1e-2L) return (a - b) / std::log(a / b);
    Q F = 0, t = 1;
    for (int k = 0; k < 16; ++k, t *= u) F += t / (2 * k + 1);
    return (a + b) / 2 / F;
}
struct NoMean {      // the corners stay within the series
    long long rho() const { __builtin_trap(); }
    long long inv_beta() const { __builtin_trap(); }
    void rho(LogMeansFx&) const { __builtin_trap(); }
    void beta(LogMeansFx&) const { __builtin_trap(); }
};
static const double kTop[4] = {1.0 - 0x1p-53, 1.0 - 1e-12, 0.5, 0.75};
static int wrong = 0;
static void check(const char* what, const long long* f, const Q* ref, const int* k) {
    for (int v = 0; v < 5; ++v) {
        const Q err = std::fabs((Q)f[v] * std::ldexp(1.0L, -60) - std::ldexp(ref[v], -k[v]));
        if (!(err <= 0x1p-52L) && wrong++ < 10) std::printf("%s component %d: error %Lg\n", what, v, err);
    }
}
int main() {
    const double gamma = 1.4, g1 = 1.0 / (gamma - 1.0);
    int kg;
    const Fx cg = fx_split(fx_from_double(std::frexp(g1, &kg), 0));
    for (int top = 0; top < 256; ++top)
        for (int eb = 0; eb <= 14; ++eb)
            for (int signs = 0; signs < 32; ++signs) {
                // densities, velocities, beta and metrics from kTop; beta down to 2^-14 (which part of the momentum
                // and energy flux is the larger), every sign pattern of the velocities, two of the metrics
                const double hr = kTop[top & 3], u = kTop[top >> 2 & 3], b = std::ldexp(kTop[top >> 4 & 3], -eb), m = kTop[top >> 6];
                const double S = (top + eb) & 1 ? 1.0 : 0.95;
                double h[3], n[3];
                for (int d = 0; d < 3; ++d) h[d] = (signs >> d & 1 ? -u : u), n[d] = (signs & 8 ? (signs >> d & 1 ? -m : m) : m);
                const double q = h[0] * h[0] + h[1] * h[1] + h[2] * h[2];
                const int Er = biased_exp(hr), Eu = biased_exp(u), Eb = biased_exp(b), En = biased_exp(m);
                if (!fix_range_ok(Er, Er, Eu, Eb, Eb, En)) return 2;
                // metric and flux in extended precision
                Q nn[3], un = 0;
                for (int d = 0; d < 3; ++d) nn[d] = 2 * (Q)S * n[d], un += 2 * (Q)h[d] * nn[d];
                const Fx Sf = fx_split(fx_from_double(S, 0));
                auto metric = [&](int kn, Fx* f) {
                    for (int d = 0; d < 3; ++d) {
                        const Fx a = fx_split(fx_from_double(n[d], kn));
                        f[d] = fx_split(fx_mul<2>(Sf, fx_add(a, a)));
                    }
                };
                auto inputs = [&](const FixScale& s, double q_, double p_) {
                    auto f = [](double x, int k) { return fx_split(fx_from_double(x, k)); };
                    return PrimFx{f(hr, s.kr), f(h[0], s.ku), f(h[1], s.ku), f(h[2], s.ku), f(b, s.kb), f(q_, s.kq), f(p_, s.kp)};
                };
                long long f[5];
                Q ref[5];
                Fx nf[3];
                auto forward = [&](Q pt, Q e) {      // e: specific energy coefficient beside ubar.f_m
                    ref[0] = 2 * (Q)hr * un;
                    Q w = 0;
                    for (int d = 0; d < 3; ++d) ref[1 + d] = ref[0] * 2 * h[d] + pt * nn[d], w += 2 * (Q)h[d] * ref[1 + d];
                    ref[4] = ref[0] * e + w;
                };
                {
                    const FixScale s = fix_scale(Er, Er, Eu, Eb, Eb, En, 1000, 1000, kg);
                    const PrimFx a = inputs(s, q, 0.0);
                    const int k[5] = {s.k0, s.km, s.km, s.km, s.k5};
                    metric(s.kn, nf);
                    ec_flux_fx(a, a, nf[0], nf[1], nf[2], cg, s, NoMean{}, f);
                    forward((Q)hr / b, 0.5L * g1 / b - 2 * (Q)q);
                    check("ES-C", f, ref, k);
                    // the reverse, for cotangents of every sign pattern and energy parts over six decades
                    const int h0 = double_hi(hr / b);
                    for (int l4 = -10; l4 <= 10; l4 += 5) {
                        const double x = std::ldexp(u, l4);
                        const AdjScale t = adj_scale(s, biased_exp(m), biased_exp(u), biased_exp(x), h0, h0);
                        const double c[5] = {m, u, u, u, x};
                        long long mu[5];
                        for (int v = 0; v < 5; ++v) {
                            const int kv = v == 0 ? t.l0 : (v == 4 ? t.l4 : t.l1);
                            mu[v] = 2 * fx_from_double((signs >> v & 1) ? -c[v] : c[v], kv);
                        }
                        PairBarFx o;
                        ec_pair_vjp_fx(a, a, nf[0], nf[1], nf[2], mu, cg, s, t, NoMean{}, o);
                    }
                }
                {
                    const double p = hr * (0.5 / b), e = 0.5 * g1 * (0.5 / b) + q;
                    const FixScale s = fix_scale_kg(Er, Eu, Eb, En, 1000, 1000, biased_exp(e), biased_exp(p));
                    const PrimFx a = inputs(s, e, p);
                    const int k[5] = {s.k0, s.km, s.km, s.km, s.k5};
                    metric(s.kn, nf);
                    kg_flux_fx(a, a, nf[0], nf[1], nf[2], s, f);
                    forward(2 * (Q)p, 0);
                    ref[4] = ref[0] * 2 * e + 2 * (Q)p * un;
                    check("SF-KG", f, ref, k);
                }
            }
    // SF-KG mass flux through a face that the flow is parallel to, its velocity and normal along
    // different axes: products of zeros, exactly zero in float64 whatever the density and pressure
    for (int d = 0; d < 3; ++d)
        for (int t = 0; t < 16; ++t) {
            const double hr = kTop[t & 3], u = kTop[t >> 2], e = 2.0 + 0.1 * t, p = 0.7 + 0.01 * t;
            const FixScale s = fix_scale_kg(biased_exp(hr), biased_exp(u), 1022, 1022, 1000, 1000, biased_exp(e), biased_exp(p));
            Fx h[3] = {}, n[3] = {};
            h[d] = fx_split(fx_from_double(u, s.ku));
            n[(d + 1) % 3] = fx_split(fx_from_double(0.7, s.kn));
            auto f = [](double x, int k) { return fx_split(fx_from_double(x, k)); };
            const PrimFx a = {f(hr, s.kr), h[0], h[1], h[2], f(0.5, s.kb), f(e, s.kq), f(p, s.kp)};
            long long F[5];
            kg_flux_fx(a, a, n[0], n[1], n[2], s, F);
            if (F[0] != 0) wrong++, std::printf("SF-KG mass flux of parallel flow: %lld units\\n", F[0]);
        }
    return wrong != 0;
}
"""


def test_fluxes_at_the_largest_operands(tmp_path):
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error",
                    "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "paper_1911_10966_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
