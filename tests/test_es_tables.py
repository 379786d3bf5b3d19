"""The FP64 kernel-weight tables against the kernel itself in extended
precision, over the shapes they serve (CPU only: the header that the library
builds and reads them with, compiled by the host compiler)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2406_18356_gb300", "csrc")
SOURCE = r"""
#include <algorithm>
#include "es_tables.h"
extern "C" int table_size() { return ms::kEsTable; }
extern "C" double max_beta() { return ms::kEsMaxBeta; }
extern "C" void tables(double beta, double* t) {
  const std::vector<double> v = ms::es_tables(beta);
  std::copy(v.begin(), v.end(), t);
}
extern "C" void weights(const double* t, int n, const double* f, double* w) {
  for (int i = 0; i < n; ++i) ms::es_weights_tab(f[i], t, w + 7 * i);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("es")
    src, so = d / "es.cpp", str(d / "es.so")
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.max_beta.restype = ctypes.c_double
    lib.tables.argtypes = [ctypes.c_double, ctypes.c_void_p]
    lib.weights.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return lib


def test_range(lib):
    assert lib.max_beta() == 32.0


# Roundings: a tap is a coefficient (half a unit of 2^-52 at most, the peak
# being 1), the last multiply-add and smaller terms: 2.5e-16.  The outer taps
# also carry 1 - z^2: the roundings of f + 3, of z^2 and of the difference, 5e-16
# together, through the square root and exp(beta (v - 1)).
@pytest.mark.parametrize("beta", [1e-6, 1e-2, 0.5, 1.0, 2.0, 4.0, 8.0, 12.0, 16.1, 24.0, 32.0])
def test_weights(lib, beta):
    rng = np.random.default_rng(0)
    edge = 10.0 ** -np.arange(1, 17)
    f = np.concatenate([rng.uniform(-0.5, 0.5, 100000), np.linspace(-0.5, 0.5, 64 * 64 + 1),
                        0.5 - edge, edge - 0.5])
    t, w = np.zeros(lib.table_size()), np.zeros((len(f), 7))
    lib.tables(beta, t.ctypes.data)
    lib.weights(t.ctypes.data, len(f), f.ctypes.data, w.ctypes.data)
    z = 2 * (f.astype(np.longdouble)[:, None] + (3 - np.arange(7))) / 7
    v = np.sqrt(np.maximum(1 - z * z, 0))
    want = np.exp(np.longdouble(beta) * (v - 1))
    err = np.abs(w - want)
    assert float(err[:, 1:6].max()) <= 2.5e-16
    ds = 5e-16
    dv = np.minimum(ds / np.maximum(2 * v, 1e-300), np.sqrt(ds))
    outer = [0, 6]
    assert float((err - beta * want * np.exp(beta * dv) * dv)[:, outer].max()) <= 2.5e-16
