"""The FP32 transfers between non-nested grids with integer weights and
compensated sums (csrc/mg_device.cuh: prolong_entry_int, restrict_entry_int),
compiled for the host by nvcc and compared with the oracle's definitions in
FP64 on the same FP32 inputs (no GPU): every result is the exact value rounded
to FP32 up to the last bit of a sum of two numbers (1.5 units of 2^-24 of the
sum of the terms' magnitudes is the bound for one rounding of the sum and one
of an accumulated value)."""
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
extern "C" int host_integer(const int* fn) { return transfer_integer(grid(fn)) ? 1 : 0; }
extern "C" void host_prolong(const int* fn, const int* cn, const float* xc, const unsigned short* mf, float* xf) {
  const Grid f = grid(fn), c = grid(cn);
  for (int64_t i = 0; i < NF * f.nn(); ++i) prolong_entry_int(f, c, xc, mf, xf, i);
}
extern "C" void host_restrict(const int* fn, const int* cn, const float* rf, const unsigned short* mc, float* rc) {
  const Grid f = grid(fn), c = grid(cn);
  for (int64_t i = 0; i < NF * c.nn(); ++i) restrict_entry_int(f, c, rf, mc, rc, i);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("transfers_int")
    src, so = d / "t.cu", d / "t.so"
    src.write_text(SHIM)
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-gencode", "arch=compute_103a,code=sm_103a", "-I", ROOT, "-o", str(so), str(src)])
    return C.CDLL(str(so))


def _p(a, t):
    return a.ctypes.data_as(C.POINTER(t))


def _n3(n):
    return (C.c_int * 3)(*n)


@pytest.mark.parametrize("fine", [(3, 3, 3), (5, 4, 3), (9, 7, 6), (19, 10, 5), (1, 1, 7), (75, 2, 3), (1, 1, 1)])
def test_integer_transfers_match_the_oracle(lib, fine):
    coarse = tuple((n + 1) // 2 for n in fine)
    rng = np.random.default_rng(5)
    nnf, nnc = np.prod([n + 1 for n in fine]), np.prod([n + 1 for n in coarse])
    Pm = T.prolongation(fine, coarse)
    P = Pm.toarray() if hasattr(Pm, "toarray") else np.asarray(Pm)
    mf = rng.integers(0, 8, nnf).astype(np.uint16)
    mc = rng.integers(0, 8, nnc).astype(np.uint16)
    # values over nine orders of magnitude, with cancellation
    xc = (rng.standard_normal((9, nnc)) * 10.0 ** rng.uniform(-6, 3, (9, nnc))).astype(np.float32)
    xf = rng.standard_normal((9, nnf)).astype(np.float32)
    rf = (rng.standard_normal((9, nnf)) * 10.0 ** rng.uniform(-6, 3, (9, nnf))).astype(np.float32)
    got_f, got_c = xf.copy(), np.empty((9, nnc), dtype=np.float32)
    lib.host_prolong(_n3(fine), _n3(coarse), _p(xc, C.c_float), _p(mf, C.c_ushort), _p(got_f, C.c_float))
    lib.host_restrict(_n3(fine), _n3(coarse), _p(rf, C.c_float), _p(mc, C.c_ushort), _p(got_c, C.c_float))
    eps = 2.0 ** -24
    for f in range(9):
        free = ((mf >> f) & 1) == 0
        corr = P @ xc[f].astype(np.float64)
        ref = np.where(free, xf[f] + corr, xf[f].astype(np.float64))
        bound = 1.5 * eps * (np.abs(corr) + np.abs(ref)) + 2.0 ** -40 * (P @ np.abs(xc[f].astype(np.float64)))
        assert np.all(np.abs(got_f[f] - ref) <= np.where(free, bound, 0.0))
        ref = np.where(((mc >> f) & 1) == 0, P.T @ rf[f].astype(np.float64), 0.0)
        bound = 1.5 * eps * np.abs(ref) + 2.0 ** -40 * (P.T @ np.abs(rf[f].astype(np.float64)))
        assert np.all(np.abs(got_c[f] - ref) <= bound)


def test_range_of_the_integer_form(lib):
    assert lib.host_integer(_n3((255, 255, 255))) == 1
    assert lib.host_integer(_n3((256, 256, 256))) == 0
