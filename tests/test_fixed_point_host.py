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


def test_out_of_range_is_refused(lib):
    P = np.array([[0.5, 0, 0, 0, 1.0, 0.0]] * 8)
    M = np.ones((8, 3))
    out = np.empty((8, 8, 5))
    assert lib.fluxes(8, P.ctypes.data, M.ctypes.data, 1.4, out.ctypes.data) == 0
    for col, val in ((0, 100.0), (4, 1e-3), (0, float("nan")), (4, float("inf")), (1, float("inf")), (0, 0.0)):
        Q = P.copy()
        Q[3, col] = val
        assert lib.fluxes(8, Q.ctypes.data, M.ctypes.data, 1.4, out.ctypes.data) == 1
