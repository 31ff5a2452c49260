"""The point physics (csrc/qp_physics.cuh) far from the reference stretch: strong
compression, strongly different stretches and numbers beyond FP32, compiled for
the host by g++ in a test-only shim (no GPU). For austenite (F^t = I) and
F = R diag(s) with the axes of the cubic stiffness, everything is in closed form:
h = log s, T = L h, W = h . T / 2, dW/dF = R diag(T_i / s_i), and along two
directions R diag(s_i a_i), R diag(s_i b_i) the second derivative is
sum_ij (L_ij - delta_ij T_i) a_i b_j."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2011_08802_gb300 import abi, inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EPS = 2.0 ** -53

SHIM = r'''
#include "paper_2011_08802_gb300/csrc/params.h"
extern "C" void qp_host(const pfm_params* prm, const double* F, double* W, double* g, double* H) {
  pfm::DevParams P;
  pfm::make_dev_params(*prm, P);
  const double eta[6] = {0, 0, 0, 0, 0, 0};
  pfm::qp_local<double, true>(P, F, eta, eta, W, g, H);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("qp_stretch")
    src, so = d / "qp.cpp", d / "qp.so"
    src.write_text(SHIM)
    subprocess.check_call([cxx, "-O2", "-shared", "-fPIC", "-std=c++17", "-I", ROOT, "-o", str(so), str(src)])
    return C.CDLL(str(so))


@pytest.mark.parametrize("s", [(1.1, 1.0, 0.95), (0.3, 0.31, 0.29), (0.01, 0.011, 0.009), (1e-4, 1.1e-4, 9e-5),
                               (1e-8, 1.1e-8, 9e-9), (30.0, 1.0, 1.02), (100.0, 1.02, 1.0), (1.0, 1.02, 0.03),
                               (1e4, 1.1e4, 9e3), (2e19, 2.2e19, 1.8e19), (1e20, 1.1e20, 9e19), (1e40, 1e40, 1e40)])
def test_closed_form_at_large_stretches(lib, s):
    """Each stretch enters with a few relative roundings, so h is off by a few units
    of 2^-53, T by as many of the largest stiffness row sum, and the other operations
    add relative roundings: 64 units cover the gradient. The Hessian's quadratic form
    adds 81 products, each entry within 1e-12 of its row and column as in the test of
    the point physics."""
    prm = abi.params_from_material(inputs.config_random(2, 2, 2, seed=1).material, 0.1)
    L = np.array(list(prm.Lvoigt[0])).reshape(6, 6)[:3, :3]
    row = np.abs(L).sum(1).max()
    s = np.array(s)
    h = np.log(s)
    T = L @ h
    rng = np.random.default_rng(8)
    for _ in range(8):
        R, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        F = np.ascontiguousarray(R * s)
        W, g, H = np.zeros(1), np.zeros(15), np.zeros(120)

        def dp(a):
            return a.ctypes.data_as(C.POINTER(C.c_double))

        lib.qp_host(C.byref(prm), dp(F), dp(W), dp(g), dp(H))
        # chemical and obstacle energy vanish in austenite (F_0 = 0)
        assert abs(W[0] - 0.5 * h @ T) <= 64 * EPS * row * (np.abs(h).sum() + np.abs(h @ h))
        P = R * (T / s)
        scale = row * max(1.0, np.abs(h).max())
        assert (np.abs(g[:9].reshape(3, 3) - P) <= 64 * EPS * scale / s).all()
        A = np.zeros((15, 15))
        A[np.triu_indices(15)] = H
        A = A + np.triu(A, 1).T
        a, b = rng.standard_normal(3), rng.standard_normal(3)
        got = (R * (s * a)).reshape(9) @ A[:9, :9] @ (R * (s * b)).reshape(9)
        D = L - np.diag(T)
        assert abs(got - a @ D @ b) <= 1e-12 * (np.abs(a) @ np.abs(D) @ np.abs(b) + scale)


@pytest.mark.parametrize("k", [1e-8, 1e-3, 0.1, 10.0, 1e19, 1e20, 1e25, 1e40])
def test_uniform_scaling_of_a_general_state(lib, k):
    """F = k F0 adds c I to the Hencky strain (c = log k): with r = C11 + 2 C12,
    W = W0 + c P0 : F0 + 3/2 c^2 r and dW/dF = (P0 + c r F0^-T) / k."""
    prm = abi.params_from_material(inputs.config_random(2, 2, 2, seed=1).material, 0.1)
    L = np.array(list(prm.Lvoigt[0])).reshape(6, 6)[:3, :3]
    r = L.sum(1)[0]
    rng = np.random.default_rng(9)
    for _ in range(8):
        F0 = np.eye(3) + 0.1 * rng.standard_normal((3, 3))

        def dp(a):
            return a.ctypes.data_as(C.POINTER(C.c_double))

        def run(F):
            W, g, H = np.zeros(1), np.zeros(15), np.zeros(120)
            F = np.ascontiguousarray(F)
            lib.qp_host(C.byref(prm), dp(F), dp(W), dp(g), dp(H))
            assert np.isfinite(H).all()
            return W[0], g[:9].reshape(3, 3)

        W0, P0 = run(F0)
        W, P = run(k * F0)
        c = np.log(k)
        ref = W0 + c * (P0 * F0).sum() + 1.5 * c * c * r
        inv = c * r * np.linalg.inv(F0).T
        assert abs(W - ref) <= 64 * EPS * (abs(W0) + np.abs(c * P0 * F0).sum() + 1.5 * c * c * r)
        assert np.abs(P * k - (P0 + inv)).max() <= 64 * EPS * (np.abs(P0).max() + np.abs(inv).max())
