"""The second-order time coefficients and their derivative along tau
(csrc/wave_math.cuh) against 50 digits, from dt/tau = 1e-8, where all of their
leading terms cancel, to 40: absolute errors at the rounding level of the terms
that are subtracted."""
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
extern "C" void coeffs_all(double dt, double tau, double* o) {
    const QC c = time_coeffs_all(dt, tau);
    const double v[7] = {c.q1, c.q4, c.a4, c.q2, c.q3, c.a5, c.q5};
    for (int k = 0; k < 7; ++k) o[k] = v[k];
    for (int k = 0; k < 6; ++k) {
        double b[6] = {};
        b[k] = 1.0;
        o[7 + k] = time_coeffs_adj(c, dt, tau, b[0], b[3], b[4], b[1], b[2], b[5]);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("time_coeffs")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                    f"-I{ROOT}/paper_2007_13091_gb300/csrc", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("x", [1e-8, 1e-5, 1e-3, 0.3, 1.7, 40.0])
def test_second_order_time_coefficients(lib, x):
    import mpmath as mp
    mp.mp.dps = 50
    dt = 0.37
    tau = dt / x
    o = np.zeros(13)
    lib.coeffs_all(ctypes.c_double(dt), ctypes.c_double(tau), o.ctypes.data_as(ctypes.c_void_p))

    def ref(T):
        D = mp.mpf(dt)
        e = mp.exp(-D / T)
        q4 = T * (1 - e)
        q5 = T * D * e - T * q4
        return [D - q4, q4, q4 - D * e, 2 * T * q4 - T * D - T * D * e, D * D / 2 - T * D + T * q4, q5 + D * D * e / 2, q5]

    T, u = mp.mpf(tau), mp.mpf(2) ** -53
    X = mp.mpf(dt) / T
    want, diff = ref(T), [mp.diff(lambda t, k=k: ref(t)[k], T) for k in range(6)]
    # roundings of the formula, with expm1 to an ulp: at most 10 u of dt in q1, q4, a4 and
    # 20 u of the largest term, dt max(tau, dt), in q2, q3, q5, a5
    for k in range(7):
        tol = 10 * u * dt if k < 3 else 20 * u * dt * max(tau, dt)
        assert abs(o[k] - want[k]) <= tol, k
    # derivatives: at most 64 u of their largest terms, 1 + x^2 times dt/tau or dt
    for k in range(6):
        tol = 64 * u * (1 + X * X) * (X if k < 3 else dt)
        assert abs(o[7 + k] - diff[k]) <= tol, k
