"""The fixed-point contraction (csrc/fixed_point.cuh) of the FP64 tangent
application and of the coarse inverse, compiled for the host by g++ in a
test-only shim and compared with exact rational arithmetic (no GPU): symmetric
15 x 15 products over the forms that the kernels accept (parts of very different
size, zeros, numbers below the normal range, the ends of the exponent range), the
largest sums of products, and the inputs that are left to FP64."""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r'''
#include "paper_2011_08802_gb300/csrc/fixed_point.cuh"
using namespace pfm;
// sigma = H x of n unknowns, the first nf of them in the first part; 0 if refused
extern "C" int contract(int n, int nf, const double* H, const double* x, double* out) {
  unsigned top[3] = {0, 0, 0}, t[2] = {0, 0};
  for (int r = 0; r < n; ++r) {
    for (int c = r; c < n; ++c) {
      const unsigned v = fx_top(H[r * n + c]);
      unsigned& m = top[c < nf ? 0 : (r < nf ? 1 : 2)];
      m = v > m ? v : m;
    }
    unsigned& m = t[r < nf ? 0 : 1];
    m = fx_top(x[r]) > m ? fx_top(x[r]) : m;
  }
  const int hx = fx_hess_scales(top);
  int Z;
  if (!fx_input_scale(hx, t[0], t[1], Z)) return 0;
  auto a = [&](int r) { return r < nf ? fx_scale_F(hx) : fx_scale_eta(hx); };
  for (int r = 0; r < n; ++r) {
    int64_t s1 = 0, s0 = 0;
    for (int c = 0; c < n; ++c) {
      int h1, h0, x1, x0;
      fx_limbs(H[r * n + c], 1027 + a(r) + a(c), h1, h0);
      fx_limbs(x[c], 1027 + Z - a(c), x1, x0);
      fx_mad(s1, s0, h1, h0, x1, x0);
    }
    out[r] = fx_value(s1, s0, 1027 + a(r) + Z);
  }
  return 1;
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fixed_point")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SHIM)
    subprocess.check_call([cxx, "-O2", "-shared", "-fPIC", "-std=c++17", "-I", ROOT, "-o", str(so), str(src)])
    return C.CDLL(str(so))


def _contract(lib, H, x, nf):
    n = len(x)
    out = np.zeros(n)

    def dp(a):
        return a.ctypes.data_as(C.POINTER(C.c_double))

    H, x = np.ascontiguousarray(H), np.ascontiguousarray(x)
    return lib.contract(n, nf, dp(H), dp(x), dp(out)), out


def _exact(H, x):
    return [sum(Fraction(float(h)) * Fraction(float(v)) for h, v in zip(row, x)) for row in H]


@pytest.mark.parametrize("sF,se,sx", [(1.0, 1.0, 1.0), (1e3, 1e-2, 1.0), (1e-30, 1e20, 1e-60), (2.0**180, 2.0**-170, 2.0**150)])
def test_contraction_within_its_bound(lib, sF, se, sx):
    """Per row: 15 products, each limb product and each truncated operand within
    2^-58 of 2^(a_r + Z) (three of them), the shift by 2^-59 and the final
    rounding by 2^-53 of the result: (46 2^-58) 2^(a_r + Z) + 2^-53 |sigma_r|.
    2^(a_r + Z) is at most 8 times the largest |H_rc'| |x_c| scale of the point
    (the exponents are rounded up: twice for a_r + a_c, once for Z)."""
    rng = np.random.default_rng(5)
    n, nf = 15, 9
    scale = np.where(np.arange(n) < nf, sF, se)
    for it in range(60):
        A = rng.standard_normal((n, n)) * scale[:, None] * scale[None, :]
        H = np.triu(A) + np.triu(A, 1).T
        x = rng.standard_normal(n) * sx / scale
        if it % 3 == 1:
            x[rng.integers(n)] = 0.0
            H[2, :] = H[:, 2] = 0.0
        if it % 3 == 2:
            x[3], H[4, 4] = 1e-310, -1e-310  # below the normal numbers: read as zero
        ok, out = _contract(lib, H, x, nf)
        assert ok == 1
        ex = _exact(H, x)
        # the exponents as the kernel takes them, from |v| < 2^(e + 1)
        def up(v):
            return int(np.floor(np.log2(v))) + 1
        F, e = slice(0, nf), slice(nf, n)
        aF = -(-up(np.abs(H[F, F]).max()) // 2)
        ae = max(-(-up(np.abs(H[e, e]).max()) // 2), up(np.abs(H[F, e]).max()) - aF)
        Z = max(up(np.abs(x[F]).max()) + aF, up(np.abs(x[e]).max()) + ae)
        for r in range(n):
            bound = Fraction(46, 2**58) * Fraction(2) ** ((aF if r < nf else ae) + Z) + abs(ex[r]) / 2**53
            assert abs(Fraction(float(out[r])) - ex[r]) <= bound


@pytest.mark.parametrize("n", [1, 15, 16])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_largest_sums_do_not_overflow(lib, n, sign):
    """Every number just below a power of two and all products of one sign: the
    integer sums of up to 16 terms stay below 2^63."""
    v = np.nextafter(1.0, 0.0)
    H, x = np.full((n, n), v), np.full(n, sign * v)
    ok, out = _contract(lib, H, x, n)
    assert ok == 1
    ex = _exact(H, x)
    for r in range(n):
        assert abs(Fraction(float(out[r])) - ex[r]) <= abs(ex[r]) / 2**52


def test_zero_input_and_refused_inputs(lib):
    H, x = np.eye(15), np.zeros(15)
    ok, out = _contract(lib, H, x, 9)
    assert ok == 1 and not out.any()
    ok, out = _contract(lib, np.zeros((15, 15)), np.ones(15), 9)
    assert ok == 1 and not out.any()
    for bad in (np.inf, np.nan, -np.inf):
        x = np.ones(15)
        x[4] = bad
        assert _contract(lib, H, x, 9)[0] == 0
        G = np.eye(15)
        G[3, 11] = G[11, 3] = bad
        assert _contract(lib, G, np.ones(15), 9)[0] == 0
    assert _contract(lib, H, np.full(15, 1e200), 9)[0] == 0
    assert _contract(lib, 1e-280 * np.eye(15), np.ones(15), 9)[0] == 0
