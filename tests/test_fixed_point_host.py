"""The fixed-point two-point flux (csrc/fix_f64.cuh) on the host against extended precision: conversions,
and the flux over smooth, jumpy, supersonic and nearly still elements.  Bound: the flux's largest value in
the element times 2^-52, two float64 roundings (its own errors are a few units of 2^-60 of the largest
products, the inputs' conversion 2^-59)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = r"""
#include <cmath>
#include "fix_f64.cuh"
using namespace esdc;
struct LM {
    const double *a, *b; const FixScale& s; double g1;
    static long double lg(const double* x, const double* y) { return std::log((long double)*x / *y); }
    long long rho() const { return fx_from_double((double)(2 * ((long double)a[0] - b[0]) / lg(a, b)), s.kr); }
    long long inv_beta() const { return fx_from_double((double)(0.5L * g1 * lg(a + 4, b + 4) / ((long double)a[4] - b[4])), s.kA); }
};
extern "C" double ln_of(double x) {
    const double T = 1.0 / (1.0 + (ln_index(x) + 0.5) / 128);
    const long double L = -std::log((long double)T);
    const double hi = (double)L;
    return fx_to_double(ln_fx(x, fx_split(fx_from_double(T, 0)), fx_from_double(hi, 0) + fx_from_double((double)(L - hi), 0)), 2);
}
extern "C" double roundtrip(double x, int k) { return fx_to_double(fx_from_double(x, k), k); }
// prim [n][6], metric [n][3] of one element: f_EC of every pair with the summed metric, as float64; 1 if out of range
extern "C" int fluxes(int n, const double* P, const double* M, double gamma, double* out) {
    int E[6] = {0, 4096, 0, 0, 4096, 0}, kg;
    for (int i = 0; i < n; ++i) {
        const double *p = P + 6 * i, *m = M + 3 * i;
        E[0] = fx_max(E[0], biased_exp(p[0])); E[1] = -fx_max(-E[1], -biased_exp(p[0]));
        E[3] = fx_max(E[3], biased_exp(p[4])); E[4] = -fx_max(-E[4], -biased_exp(p[4]));
        for (int d = 0; d < 3; ++d) { E[2] = fx_max(E[2], biased_exp(p[1 + d])); E[5] = fx_max(E[5], biased_exp(m[d])); }
    }
    if (!fix_range_ok(E[0], E[1], E[2], E[3], E[4], E[5])) return 1;
    const double g1 = 1.0 / (gamma - 1.0);
    const Fx cg = fx_split(fx_from_double(std::frexp(g1, &kg), 0));
    const FixScale s = fix_scale(E[0], E[1], E[2], E[3], E[4], E[5], 1000, 1000, kg);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            PrimFx x[2];
            const int ij[2] = {i, j};
            for (int q = 0; q < 2; ++q) {
                const double* p = P + 6 * ij[q];
                x[q] = {fx_split(fx_from_double(p[0], s.kr)), fx_split(fx_from_double(p[1], s.ku)), fx_split(fx_from_double(p[2], s.ku)),
                        fx_split(fx_from_double(p[3], s.ku)), fx_split(fx_from_double(p[4], s.kb)), fx_split(fx_from_double(p[5], s.kq))};
            }
            Fx m[3];
            for (int d = 0; d < 3; ++d) m[d] = fx_split(fx_from_double(M[3 * i + d], s.kn) + fx_from_double(M[3 * j + d], s.kn));
            const LM lm = {P + 6 * i, P + 6 * j, s, g1};
            long long f[5];
            ec_flux_fx(x[0], x[1], m[0], m[1], m[2], cg, s, lm, f);
            const int k[5] = {s.k0, s.km, s.km, s.km, s.k5};
            for (int v = 0; v < 5; ++v) out[(i * n + j) * 5 + v] = fx_to_double(f[v], k[v]);
        }
    return 0;
}
struct AM {
    const double *a, *b; const FixScale& s; int kd; double hig;
    void rho(LogMeansFx& m) const {
        const long double x = 2 * a[0], y = 2 * b[0], l = std::log(x / y), L = (x - y) / l;
        m.rl = fx_from_double((double)L, s.kr); m.La = fx_from_double((double)((1 - L / x) / l), 0); m.Lb = fx_from_double((double)((L / y - 1) / l), 0);
    }
    void beta(LogMeansFx& m) const {
        const long double x = a[4], y = b[4], d = x - y, I = std::log(x / y) / d;
        m.A = fx_from_double((double)(hig * I), s.kA); m.DA = fx_from_double((double)(hig * (1 / x - I) / d), kd); m.DB = fx_from_double((double)(hig * (I - 1 / y) / d), kd);
    }
};
// reverse of every pair i < j for the cotangents lw_j - lw_i: (xa, xb, ba, bb, u0, u1, u2, c), u doubled
extern "C" int reverses(int n, const double* P, const double* M, const double* LW, double gamma, double* out) {
    int E[9] = {0, 4096, 0, 0, 4096, 0, 0, 0, 0}, kg;
    for (int i = 0; i < n; ++i) {
        const double *p = P + 6 * i, *m = M + 3 * i, *w = LW + 5 * i;
        E[0] = fx_max(E[0], biased_exp(p[0])); E[1] = -fx_max(-E[1], -biased_exp(p[0]));
        E[3] = fx_max(E[3], biased_exp(p[4])); E[4] = -fx_max(-E[4], -biased_exp(p[4]));
        E[6] = fx_max(E[6], biased_exp(w[0])); E[8] = fx_max(E[8], biased_exp(w[4]));
        for (int d = 0; d < 3; ++d) { E[2] = fx_max(E[2], biased_exp(p[1 + d])); E[5] = fx_max(E[5], biased_exp(m[d])); E[7] = fx_max(E[7], biased_exp(w[1 + d])); }
    }
    if (!fix_range_ok(E[0], E[1], E[2], E[3], E[4], E[5])) return 1;
    const double g1 = 1.0 / (gamma - 1.0);
    const Fx cg = fx_split(fx_from_double(std::frexp(g1, &kg), 0));
    const FixScale s = fix_scale(E[0], E[1], E[2], E[3], E[4], E[5], 1000, 1000, kg);
    int plo = 0x7ff00000, phi = 0;
    for (int i = 0; i < n; ++i) {
        const int h = double_hi(P[6 * i] / P[6 * i + 4]);
        plo = -fx_max(-plo, -h); phi = fx_max(phi, h);
    }
    const AdjScale t = adj_scale(s, E[6], E[7], E[8], plo, phi);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
            PrimFx x[2];
            const int ij[2] = {i, j};
            for (int q = 0; q < 2; ++q) {
                const double* p = P + 6 * ij[q];
                x[q] = {fx_split(fx_from_double(p[0], s.kr)), fx_split(fx_from_double(p[1], s.ku)), fx_split(fx_from_double(p[2], s.ku)),
                        fx_split(fx_from_double(p[3], s.ku)), fx_split(fx_from_double(p[4], s.kb)), fx_split(fx_from_double(p[5], s.kq))};
            }
            Fx m[3];
            for (int d = 0; d < 3; ++d) m[d] = fx_split(fx_from_double(M[3 * i + d], s.kn) + fx_from_double(M[3 * j + d], s.kn));
            long long mu[5];
            for (int v = 0; v < 5; ++v) {
                const int k = v == 0 ? t.l0 : (v == 4 ? t.l4 : t.l1);
                mu[v] = fx_from_double(LW[5 * j + v], k) - fx_from_double(LW[5 * i + v], k);
            }
            const AM lm = {P + 6 * i, P + 6 * j, s, t.kd, 0.5 * g1};
            PairBarFx o;
            ec_pair_vjp_fx(x[0], x[1], m[0], m[1], m[2], mu, cg, s, t, lm, o);
            double* r = out + (i * n + j) * 8;
            r[0] = o.xa; r[1] = o.xb; r[2] = o.ba; r[3] = o.bb; r[7] = o.c;
            for (int d = 0; d < 3; ++d) r[4 + d] = o.u[d];
        }
    return 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), "-I",
                    os.path.join(ROOT, "paper_1911_10966_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.roundtrip.restype = ctypes.c_double
    L.roundtrip.argtypes = [ctypes.c_double, ctypes.c_int]
    L.ln_of.restype = ctypes.c_double
    L.ln_of.argtypes = [ctypes.c_double]
    L.reverses.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_double, ctypes.c_void_p]
    L.fluxes.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p]
    return L


def test_conversions(lib):
    rng = np.random.default_rng(0)
    for x in np.concatenate([rng.uniform(-1, 1, 200) * 2.0 ** rng.integers(-7, 0, 200), [0.0, 0.5, -0.5, 1.0 - 2.0 ** -53]]):
        assert lib.roundtrip(x, 0) == x                  # seven bits to spare below 1
    assert lib.roundtrip(1e-30, 0) == 0.0                # below the unit
    assert lib.roundtrip(5e-324, 0) == 0.0


def _log_mean(a, b):
    s = a + b
    u = ((a - b) / s) ** 2
    near = u < 1e-4
    un = np.where(near, u, 0)
    ser = sum(un ** k / np.longdouble(2 * k + 1) for k in range(8))
    f = np.where(near, np.longdouble(0.5), (a - b) / s)
    return 0.5 * s / np.where(near, ser, np.arctanh(f) / f)


@pytest.mark.parametrize("Ma,jump,u,n", [(0.1, 1e-5, 1.0, 1.0), (0.1, 1e-2, 1.0, 1e-3), (0.5, 0.1, 1.0, 30.0), (0.5, 0.3, 1.0, 1.0),
                                         (4.0, 0.1, 1.0, 1.0), (0.1, 1e-3, 1e-9, 1.0), (1e-3, 1e-6, 1.0, 1.0)])
def test_flux_against_extended_precision(lib, Ma, jump, u, n):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this machine")
    rng = np.random.default_rng(3)
    L = np.longdouble
    for el in range(40):
        rho, T = 1 + jump * rng.uniform(-1, 1, 8), 1 + jump * rng.uniform(-1, 1, 8)
        vel = u * rng.uniform(-1, 1, (8, 3))
        P = np.empty((8, 6))
        P[:, 0], P[:, 1:4], P[:, 4], P[:, 5] = rho / 2, vel / 2, 0.5 * 1.4 * Ma * Ma / T, 0.25 * (vel ** 2).sum(1)
        M = n * (rng.uniform(-1, 1, 3) + 0.1 * rng.uniform(-1, 1, (8, 3)))
        out = np.empty((8, 8, 5))
        assert lib.fluxes(8, P.ctypes.data, M.ctypes.data, 1.4, out.ctypes.data) == 0
        a, b = P[:, None].astype(L), P[None].astype(L)
        m = M[:, None].astype(L) + M[None].astype(L)
        ub = a[..., 1:4] + b[..., 1:4]
        f1 = _log_mean(2 * a[..., 0], 2 * b[..., 0]) * (ub * m).sum(-1)
        fm = f1[..., None] * ub + ((a[..., 0] + b[..., 0]) / (a[..., 4] + b[..., 4]))[..., None] * m
        g1 = 1.0 / (1.4 - 1.0)
        f5 = f1 * (0.5 * L(g1) / _log_mean(a[..., 4], b[..., 4]) - a[..., 5] - b[..., 5]) + (ub * fm).sum(-1)
        ref = np.concatenate([f1[..., None], fm, f5[..., None]], -1)
        for v in (slice(0, 1), slice(1, 4), slice(4, 5)):
            err = np.abs(out[..., v].astype(L) - ref[..., v]).max()
            assert err <= 2.0 ** -52 * np.abs(ref[..., v]).max(), (el, v, float(err))


def _mean_derivative(a, b):
    """(L, dL/da, dL/db) of the logarithmic mean in extended precision."""
    L = _log_mean(a, b)
    f = (a - b) / (a + b)
    u = f * f
    near = u < 1e-2
    un = np.where(near, u, 0)
    F = sum(un ** k / np.longdouble(2 * k + 1) for k in range(14))
    dF = sum(k * un ** (k - 1) / np.longdouble(2 * k + 1) for k in range(1, 14))
    W = f * dF / F ** 2
    l = np.where(near, 1, np.log(a / b))
    return L, np.where(near, 0.5 / F - W + W * f, (1 - L / a) / l), np.where(near, 0.5 / F + W + W * f, (L / b - 1) / l)


@pytest.mark.parametrize("Ma,jump,u,n,lam", [(0.1, 1e-5, 1.0, 1.0, 1.0), (0.1, 1e-2, 1.0, 1e-3, 1e-4), (0.5, 0.1, 1.0, 30.0, 1.0),
                                             (0.5, 0.3, 1.0, 1.0, 1e3), (4.0, 0.1, 1.0, 1.0, 1.0), (0.1, 1e-3, 1.0, 1.0, 0.0)])
def test_reverse_against_extended_precision(lib, Ma, jump, u, n, lam):
    """The reverse of the flux.  Bound: each result against the largest sum of magnitudes of its terms times
    2^-50 (the cotangents are differences of rounded float64 inputs; the terms are products of up to five
    factors, each a few 2^-60 of its largest possible value, eight bits above the typical one)."""
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this machine")
    rng = np.random.default_rng(5)
    L = np.longdouble
    for el in range(20):
        rho, T = 1 + jump * rng.uniform(-1, 1, 8), 1 + jump * rng.uniform(-1, 1, 8)
        vel = u * rng.uniform(-1, 1, (8, 3))
        P = np.empty((8, 6))
        P[:, 0], P[:, 1:4], P[:, 4], P[:, 5] = rho / 2, vel / 2, 0.5 * 1.4 * Ma * Ma / T, 0.25 * (vel ** 2).sum(1)
        M = n * (rng.uniform(-1, 1, 3) + 0.1 * rng.uniform(-1, 1, (8, 3)))
        W = rng.uniform(-1, 1, (8, 5))
        W[:, 4] *= lam
        out = np.empty((8, 8, 8))
        assert lib.reverses(8, P.ctypes.data, M.ctypes.data, W.ctypes.data, 1.4, out.ctypes.data) == 0
        a, b = P[:, None].astype(L), P[None].astype(L)
        m = M[:, None].astype(L) + M[None].astype(L)
        mu = W[None].astype(L) - W[:, None].astype(L)
        ub = a[..., 1:4] + b[..., 1:4]
        un = (ub * m).sum(-1)
        rl, La, Lb = _mean_derivative(2 * a[..., 0], 2 * b[..., 0])
        bl, Ba, Bb = _mean_derivative(a[..., 4], b[..., 4])
        g1 = L(1.0 / (1.4 - 1.0))
        sb = a[..., 4] + b[..., 4]
        pt = (a[..., 0] + b[..., 0]) / sb
        f1, c5 = rl * un, 0.5 * g1 / bl - a[..., 5] - b[..., 5]
        mu4 = mu[..., 4]
        fmb = mu4[..., None] * ub + mu[..., 1:4]
        f1b = mu[..., 0] + mu4 * c5 + (fmb * ub).sum(-1)
        c5b, ptb = mu4 * f1, (fmb * m).sum(-1)
        An = mu4 * pt + f1b * rl
        q = 0.5 * g1 / bl ** 2
        ra, rb, dp = 2 * a[..., 0], 2 * b[..., 0], ptb / sb * (a[..., 0] * b[..., 4] - b[..., 0] * a[..., 4]) / sb
        terms = [[f1b * un * La * ra, -c5b * q * Ba * a[..., 4], dp], [f1b * un * Lb * rb, -c5b * q * Bb * b[..., 4], -dp], [-c5b * q * Ba, -pt * ptb / sb], [-c5b * q * Bb, -pt * ptb / sb]]
        terms += [[f1 * (mu4 * ub[..., d] + fmb[..., d]), An * m[..., d]] for d in range(3)] + [[c5b]]
        mags = [np.abs(mu[..., 0]) + np.abs(mu4 * c5) + np.abs(fmb * ub).sum(-1), np.abs(fmb * m).sum(-1)]
        size = [(mags[0] * np.abs(un) * ra).max() + np.abs(c5b * q * Ba * a[..., 4]).max() + (mags[1] / sb * a[..., 0]).max()] * 2 + [(np.abs(c5b * q * Ba)).max() + (pt * mags[1] / sb).max()] * 2
        size += [(np.abs(f1) * np.abs(fmb).max(-1)).max() + ((np.abs(mu4 * pt) + mags[0] * rl) * np.abs(m).max(-1)).max()] * 3 + [np.abs(c5b).max()]
        for k in range(8):
            err = np.abs(out[..., k].astype(L) - sum(terms[k])).max()
            assert err <= 2.0 ** -50 * size[k], (el, k, float(err), float(size[k]))


def test_out_of_range_is_refused(lib):
    P = np.array([[0.5, 0, 0, 0, 1.0, 0.0]] * 8)
    M = np.ones((8, 3))
    out = np.empty((8, 8, 5))
    assert lib.fluxes(8, P.ctypes.data, M.ctypes.data, 1.4, out.ctypes.data) == 0
    for col, val in ((0, 100.0), (4, 1e-3), (0, float("nan")), (4, float("inf")), (1, float("inf")), (0, 0.0)):
        Q = P.copy()
        Q[3, col] = val
        assert lib.fluxes(8, Q.ctypes.data, M.ctypes.data, 1.4, out.ctypes.data) == 1


@pytest.mark.parametrize("lo,hi", [(-1e-9, 1e-9), (-0.01, 0.01), (-3.0, 3.0), (-30.0, 30.0)])
def test_logarithm(lib, lo, hi):
    """ln_fx over its range against extended precision: |e|/8 + 3 units of 2^-58 (its own bound) and the
    rounding of the returned double."""
    x = np.exp(np.random.default_rng(4).uniform(lo, hi, 20000))
    x = np.concatenate([x, 2.0 ** np.arange(-44, 45), np.nextafter(2.0 ** np.arange(-43, 46), 0), 1.0 + np.arange(128) / 128.0])
    y = np.array([lib.ln_of(float(v)) for v in x])
    ref = np.log(x.astype(np.longdouble))
    bound = (np.abs(np.frexp(x)[1] - 1) / 8.0 + 3.0) * 2.0 ** -58 + np.abs(ref) * 2.0 ** -53
    assert (np.abs(y - ref) <= bound).all(), float((np.abs(y - ref) / bound).max())
