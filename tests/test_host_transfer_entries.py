"""The multigrid transfers as the kernels call them, one (node, field) at a time and
with the difference r - y formed in the restriction (csrc/mg_device.cuh:
prolong_entry_nested, restrict_entry_nested, restrict_entry_int, restrict_node),
compiled for the host by nvcc in a test-only shim and compared with the oracle's
definitions (oracle/transfer.py) on nested and non-nested grids (no GPU)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import transfer as T

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r'''
#include "paper_2011_08802_gb300/csrc/mg_device.cuh"
using namespace pfm;
static Grid grid(const int* n) {
  Grid g;
  g.nx = n[0]; g.ny = n[1]; g.nz = n[2];
  g.hx = g.hy = g.hz = 1.0;
  return g;
}
template <typename T>
static void prolong(const int* fn, const int* cn, const T* xc, const unsigned short* mf, T* xf) {
  const Grid f = grid(fn), c = grid(cn);
  if (nested(f, c)) {
    for (int fld = 0; fld < NF; ++fld)
      for (int k = 0; k <= f.nz; ++k)
        for (int j = 0; j <= f.ny; ++j)
          for (int i = 0; i <= f.nx; ++i) prolong_entry_nested<T>(f, c, xc, mf, xf, fld, i, j, k);
  } else if constexpr (sizeof(T) == 4) {
    for (int64_t i = 0; i < NF * f.nn(); ++i) prolong_entry_int(f, c, xc, mf, xf, i);
  } else {
    for (int64_t i = 0; i < f.nn(); ++i) prolong_node<T>(f, c, xc, mf, xf, i);
  }
}
template <typename T>
static void restrict_to(const int* fn, const int* cn, const T* rf, const T* y, const unsigned short* mc, T* rc) {
  const Grid f = grid(fn), c = grid(cn);
  if (nested(f, c)) {
    for (int fld = 0; fld < NF; ++fld)
      for (int k = 0; k <= c.nz; ++k)
        for (int j = 0; j <= c.ny; ++j)
          for (int i = 0; i <= c.nx; ++i) restrict_entry_nested<T>(f, c, rf, y, mc, rc, fld, i, j, k);
  } else if constexpr (sizeof(T) == 4) {
    for (int64_t i = 0; i < NF * c.nn(); ++i) restrict_entry_int(f, c, rf, mc, rc, i, y);
  } else {
    for (int64_t i = 0; i < c.nn(); ++i) restrict_node<T>(f, c, rf, mc, rc, i, y);
  }
}
extern "C" {
void prolong_f32(const int* f, const int* c, const float* x, const unsigned short* m, float* o) { prolong(f, c, x, m, o); }
void prolong_f64(const int* f, const int* c, const double* x, const unsigned short* m, double* o) { prolong(f, c, x, m, o); }
void restrict_f32(const int* f, const int* c, const float* r, const float* y, const unsigned short* m, float* o) {
  restrict_to(f, c, r, y, m, o);
}
void restrict_f64(const int* f, const int* c, const double* r, const double* y, const unsigned short* m, double* o) {
  restrict_to(f, c, r, y, m, o);
}
}
'''

PAIRS = [((8, 8, 8), (4, 4, 4)), ((24, 18, 10), (12, 9, 5)), ((2, 2, 2), (1, 1, 1)), ((2, 2, 300), (1, 1, 150)),
         ((3, 3, 3), (2, 2, 2)), ((9, 7, 6), (5, 4, 3)), ((19, 10, 5), (10, 5, 3)), ((1, 1, 7), (1, 1, 4))]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("transfer_entries")
    src, so = d / "t.cu", d / "t.so"
    src.write_text(SHIM)
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-I", ROOT, "-o", str(so), str(src)])
    return C.CDLL(str(so))


def _p(a, t=None):
    if a is None:
        return None
    return a.ctypes.data_as(C.c_void_p)


def _n3(n):
    return (C.c_int * 3)(*n)


def _axis(nf, nc):
    """Weights of one axis, exact numerators over nf: 1 - |i nc - I nf| / nf where positive."""
    i, I = np.arange(nf + 1)[:, None], np.arange(nc + 1)[None, :]
    return np.maximum(nf - np.abs(i * nc - I * nf), 0).astype(np.longdouble) / nf


def _setup(fine, coarse, seed):
    rng = np.random.default_rng(seed)
    nnf, nnc = (int(np.prod([n + 1 for n in g])) for g in (fine, coarse))
    x, y, z = (_axis(f, c) for f, c in zip(fine, coarse))
    P = np.einsum("kK,jJ,iI->kjiKJI", z, y, x).reshape(nnf, nnc)
    Q = T.prolongation(fine, coarse)  # the oracle's, from floating-point coordinates
    np.testing.assert_allclose(P.astype(float), Q.toarray() if hasattr(Q, "toarray") else Q, rtol=0, atol=1e-13)
    return rng, nnf, nnc, P, rng.integers(0, 8, nnf).astype(np.uint16), rng.integers(0, 8, nnc).astype(np.uint16)


@pytest.mark.parametrize("fine, coarse", PAIRS)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("difference", [False, True])
def test_entries_match_the_oracle(lib, fine, coarse, dtype, difference):
    """Bounds: FP32 in integer weights is exact to 1.5 roundings; the others add up to
    27 (nested) or 64 weighted terms, one rounding each beside those of the weights."""
    rng, nnf, nnc, P, mf, mc = _setup(fine, coarse, 6)
    eps = np.finfo(dtype).eps / 2
    tag = "f32" if dtype == np.float32 else "f64"
    xc, xf = (rng.standard_normal((9, n)).astype(dtype) for n in (nnc, nnf))
    r = rng.standard_normal((9, nnf)).astype(dtype)
    y = rng.standard_normal((9, nnf)).astype(dtype) if difference else None
    got_f, got_c = xf.copy(), np.empty((9, nnc), dtype=dtype)
    getattr(lib, "prolong_" + tag)(_n3(fine), _n3(coarse), _p(xc), _p(mf), _p(got_f))
    getattr(lib, "restrict_" + tag)(_n3(fine), _n3(coarse), _p(r), _p(y), _p(mc), _p(got_c))
    d = (r if y is None else r - y).astype(np.longdouble)  # the difference is rounded once in the vectors' type
    for f in range(9):
        free = ((mf >> f) & 1) == 0
        corr, size = P @ xc[f].astype(np.longdouble), P @ np.abs(xc[f].astype(np.longdouble))
        ref = np.where(free, xf[f] + corr, xf[f])
        assert (np.abs(got_f[f] - ref) <= np.where(free, 16 * eps * size + eps * np.abs(ref), 0)).all()
        keep = ((mc >> f) & 1) == 0
        ref, size = P.T @ d[f], P.T @ np.abs(d[f])
        assert (np.abs(got_c[f] - np.where(keep, ref, 0)) <= np.where(keep, 80 * eps * size, 0)).all()


@pytest.mark.parametrize("fine, coarse", PAIRS)
@pytest.mark.parametrize("power", [100, 108, 120, 126])
def test_large_fp32_values_do_not_overflow_in_the_sums(lib, fine, coarse, power):
    """The transfers are linear, and scaling by a power of two is exact: where the
    scaled result is a number of FP32, it is the unscaled one times the power."""
    rng, nnf, nnc, P, mf, mc = _setup(fine, coarse, 7)
    s = np.float32(2.0) ** power
    xc = rng.uniform(0.5, 1.9, (9, nnc)).astype(np.float32) * rng.choice([-1, 1], (9, nnc)).astype(np.float32)
    r = rng.uniform(0.5, 1.9, (9, nnf)).astype(np.float32) * rng.choice([-1, 1], (9, nnf)).astype(np.float32)
    zero = np.zeros(nnf, dtype=np.uint16)

    def run(k):
        of, oc = np.zeros((9, nnf), dtype=np.float32), np.empty((9, nnc), dtype=np.float32)
        lib.prolong_f32(_n3(fine), _n3(coarse), _p(np.ascontiguousarray(xc * k)), _p(zero), _p(of))
        lib.restrict_f32(_n3(fine), _n3(coarse), _p(np.ascontiguousarray(r * k)), None, _p(zero[:nnc].copy()), _p(oc))
        return of.astype(np.float64), oc.astype(np.float64)

    one, big = run(np.float32(1)), run(s)
    nested = all(a == 2 * b for a, b in zip(fine, coarse))
    # FP32 sums of up to 8 values on nested grids: at 2^126 only copies are in range
    i, j, k = np.meshgrid(*[np.arange(n + 1) for n in fine[::-1]], indexing="ij")
    copy = ((i % 2 == 0) & (j % 2 == 0) & (k % 2 == 0)).reshape(-1)
    for to_fine, a, b in zip((True, False), one, big):
        inside = np.abs(a) * float(s) < 2.0 ** 127.9
        if nested and power == 126:
            if not to_fine:
                continue
            inside &= copy
        assert inside.any()
        ulp = 2.0 ** -22 * np.maximum(np.abs(a), 2.0 ** -20) * float(s)  # the FP64 sums round differently
        assert (np.abs(a * float(s) - b)[inside] <= ulp[inside]).all()


def test_infinite_values_stay_infinite(lib):
    fine, coarse = (9, 7, 6), (5, 4, 3)
    rng, nnf, nnc, P, mf, mc = _setup(fine, coarse, 8)
    xc, r = np.ones((9, nnc), dtype=np.float32), np.ones((9, nnf), dtype=np.float32)
    xc[4, nnc // 2] = np.inf
    r[2, nnf // 2] = -np.inf
    of, oc = np.zeros((9, nnf), dtype=np.float32), np.empty((9, nnc), dtype=np.float32)
    z = np.zeros(nnf, dtype=np.uint16)
    lib.prolong_f32(_n3(fine), _n3(coarse), _p(xc), _p(z), _p(of))
    lib.restrict_f32(_n3(fine), _n3(coarse), _p(r), None, _p(z), _p(oc))
    assert (of[4] == np.where(P[:, nnc // 2] > 0, np.inf, of[4])).all() and np.isinf(of[4]).any()
    assert (oc[2] == np.where(P[nnf // 2] > 0, -np.inf, oc[2])).all() and np.isinf(oc[2]).any()
    assert np.isfinite(np.delete(of, 4, 0)).all() and np.isfinite(np.delete(oc, 2, 0)).all()
