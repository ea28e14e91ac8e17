"""The face flux's arithmetic (csrc/wave_math.cuh, plain functions that also
compile for the host): time coefficients on both sides of the switch between
series and closed form, and the reverse pass of each part against central
differences of its forward pass."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <cmath>
using std::erfc; using std::exp; using std::expm1; using std::fabs; using std::log; using std::sqrt;
#include "wave_math.cuh"
using namespace ugkwp::wm;
typedef const double (*G)[3];
extern "C" {
void coeffs(double dt, double tau, double* o) { QC1 c = time_coeffs(dt, tau); o[0] = c.q1; o[1] = c.q4; o[2] = c.a4; }
// x: W (5), rho^h, grad rho^h (3), grad W (15); o: H, G, S
void side(const double* x, const double* n, double sgn, int K, double* o) {
    Gas g = gas_of(K); Prim s = prim_of(x, g); PrimGrad pg = prim_grad(s, (G)(x + 9), 1.0, g);
    SideFlux f = side_flux<true>(s, pg, x[5], x + 6, n, sgn, g);
    for (int k = 0; k < 5; ++k) { o[k] = f.H[k]; o[5 + k] = f.G[k]; o[10 + k] = f.S[k]; }
}
void side_adj(const double* x, const double* n, double sgn, int K, const double* b, double* xb) {
    Gas g = gas_of(K); Prim s = prim_of(x, g); PrimGrad pg = prim_grad(s, (G)(x + 9), 1.0, g), pgb{};
    PrimAdj a = prim_adj_zero(); double gb[5][3] = {};
    for (int k = 0; k < 24; ++k) xb[k] = 0.0;
    side_flux_adj<true>(s, pg, x[5], x + 6, n, sgn, g, b, b + 5, b + 10, a, pgb, xb[5], xb + 6);
    prim_grad_adj(s, (G)(x + 9), 1.0, pg, pgb, g, gb, a);
    prim_adj(s, a, g, xb);
    for (int k = 0; k < 15; ++k) xb[9 + k] = gb[k / 3][k % 3];
}
// x: W (5), grad W (15), q1, q2, q3
void eq(const double* x, const double* n, double pr, int K, double* o) {
    Gas g = gas_of(K); Prim s = prim_of(x, g); QC c{}; c.q1 = x[20]; c.q2 = x[21]; c.q3 = x[22];
    for (int k = 0; k < 5; ++k) o[k] = 0.0;
    equilibrium_flux(x, s, (G)(x + 5), 0.5, n, c, pr, g, o);
}
void eq_adj(const double* x, const double* n, double pr, int K, const double* b, double* xb) {
    Gas g = gas_of(K); Prim s = prim_of(x, g); QC c{}; c.q1 = x[20]; c.q2 = x[21]; c.q3 = x[22];
    PrimAdj a = prim_adj_zero(); double Bb[5][3] = {}, Eb = 0.0;
    for (int k = 0; k < 23; ++k) xb[k] = 0.0;
    equilibrium_flux_adj(x, s, (G)(x + 5), 0.5, n, c, pr, g, b, a, Eb, Bb, xb + 20);
    prim_adj(s, a, g, xb);
    xb[4] += Eb;
    for (int k = 0; k < 15; ++k) xb[5 + k] = Bb[k / 3][k % 3];
}
// x: W_L (5), rho^h_L, W_R (5), rho^h_R
void o1(const double* x, const double* n, double dt, int ghost, double C2, int K, double* o) {
    FaceGas g{gas_of(K), 0.02, 0.81, 1.1, C2};
    flux_o1(prim_of(x, g.gas), x[5], prim_of(x + 6, g.gas), x[11], ghost, false, n, dt, g, o);
}
void o1_adj(const double* x, const double* n, double dt, int ghost, double C2, int K, const double* b, double* xb) {
    FaceGas g{gas_of(K), 0.02, 0.81, 1.1, C2};
    Prim L = prim_of(x, g.gas), R = prim_of(x + 6, g.gas); PrimAdj aL = prim_adj_zero(), aR = aL;
    for (int k = 0; k < 12; ++k) xb[k] = 0.0;
    flux_o1_adj(L, x[5], R, x[11], ghost, n, dt, g, b, aL, xb[5], aR, xb[11]);
    prim_adj(L, aL, g.gas, xb); prim_adj(R, aR, g.gas, xb + 6);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("wave_math")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                    f"-I{ROOT}/paper_2007_13091_gb300/csrc", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _call(f, x, n, extra, out, b=None):
    arr = lambda a: np.ascontiguousarray(a, dtype=np.float64).ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    keep = [np.ascontiguousarray(x, dtype=np.float64), np.ascontiguousarray(n, dtype=np.float64)]
    ex = [ctypes.c_int(e) if isinstance(e, int) else ctypes.c_double(e) for e in extra]
    o = np.zeros(out)
    f(arr(keep[0]), arr(keep[1]), *ex, *([arr(b)] if b is not None else []), o.ctypes.data_as(ctypes.c_void_p))
    return o


def _state(rng, mach, K):
    rho, p = np.exp(0.3 * rng.normal(size=2))
    U = mach * rng.normal(size=3)
    return np.concatenate([[rho], rho * U, [0.5 * rho * U @ U + (1.5 + 0.5 * K) * p]])


def _check(fwd, adj, x, nout, rng):
    # <b, J v> by central differences with h = 1e-5: truncation ~ 1e-10 and
    # rounding ~ 1e-11 of the largest term, against <J^T b, v>
    b, v, h = rng.normal(size=nout), rng.normal(size=x.size), 1e-5
    jv = (fwd(x + h * v) - fwd(x - h * v)) / (2 * h)
    xb = adj(x, b)
    scale = np.abs(b * jv).sum() + np.abs(xb * v).sum()
    assert abs(b @ jv - xb @ v) <= 1e-6 * scale


@pytest.mark.parametrize("x", [1e-9, 1e-4, 0.3, np.nextafter(1.0, 0.0), 1.0, 1.7, 40.0])
def test_time_coefficients(lib, x):
    import mpmath as mp
    mp.mp.dps = 50
    dt, o = 0.37, np.zeros(3)
    tau = dt / x
    lib.coeffs(ctypes.c_double(dt), ctypes.c_double(tau), o.ctypes.data_as(ctypes.c_void_p))
    X = mp.mpf(dt) / mp.mpf(tau)
    q4 = -mp.mpf(tau) * mp.expm1(-X)
    ref = [mp.mpf(dt) - q4, q4, q4 - mp.mpf(dt) * mp.exp(-X)]
    for k in range(3):
        # a few roundings, amplified at most ~4 times by the differences; x itself is rounded (relative error of a4, q1: 2 ulp)
        assert abs(o[k] - ref[k]) <= 2e-15 * abs(ref[k]) * 4, k


@pytest.mark.parametrize("K", [0, 2])
@pytest.mark.parametrize("mach", [0.3, 1.5])
def test_reverse_passes(lib, K, mach):
    rng = np.random.default_rng(7 + K)
    for i in range(20):
        n = rng.normal(size=3)
        n /= np.linalg.norm(n)
        W = _state(rng, mach, K)
        x = np.concatenate([W, [0.4 * W[0]], 0.2 * rng.normal(size=3), 0.3 * rng.normal(size=15)])
        s = 1.0 if i % 2 else -1.0
        _check(lambda y: _call(lib.side, y, n, (s, K), 15), lambda y, b: _call(lib.side_adj, y, n, (s, K), 24, b), x, 15, rng)
        x = np.concatenate([W, 0.3 * rng.normal(size=15), [0.3, -0.7, 0.9]])
        pr = 0.5 if i % 3 == 0 else 0.0
        _check(lambda y: _call(lib.eq, y, n, (pr, K), 5), lambda y, b: _call(lib.eq_adj, y, n, (pr, K), 23, b), x, 5, rng)
        x = np.concatenate([W, [0.4 * W[0]], _state(rng, mach, K), [0.3]])
        e = (0.02 * float(np.exp(rng.normal())), i % 2, 0.4 if i % 4 == 1 else 0.0, K)
        _check(lambda y: _call(lib.o1, y, n, e, 5), lambda y, b: _call(lib.o1_adj, y, n, e, 12, b), x, 5, rng)
