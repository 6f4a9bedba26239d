"""Functions of the face integrals compiled for the host and compared with
numpy in extended precision (CPU only)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2103_16841_gb300 import _build

SRC = r"""
#include "stbem_quad.cuh"
extern "C" void sinh_cosh_of(int n, const double* v, double* sh, double* ch) {
  for (int k = 0; k < n; ++k) stbem::sinh_cosh(v[k], sh[k], ch[k]);
}
extern "C" void edge_of(int n, const double* p, double* out) {
  for (int k = 0; k < n; ++k) out[k] = stbem::edge_dE<double>(p[4 * k], p[4 * k + 1], p[4 * k + 2], p[4 * k + 3]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    include = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    d = tmp_path_factory.mktemp("host")
    (d / "host.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-shared", "-fPIC", "-D__noinline__=__attribute__((noinline))",
                    "-I", include, "-I", _build.CSRC, str(d / "host.cpp"), "-o", str(d / "host.so")], check=True)
    return ctypes.CDLL(str(d / "host.so"))


def test_sinh_and_cosh_of_the_nodes(lib):
    """Both signs up to the largest argument (28 next to a pole): the six
    roundings and expm1's of the two formulas, 8 x 2^-53."""
    a = np.concatenate((np.linspace(1e-3, 30, 3001), np.logspace(-18, 1.4, 400)))
    v = np.concatenate((-a, [0.0], a))
    sh, ch = np.zeros_like(v), np.zeros_like(v)
    p = [ctypes.c_void_p(x.ctypes.data) for x in (v, sh, ch)]
    lib.sinh_cosh_of(len(v), *p)
    w = v.astype(np.longdouble)
    assert np.all(np.abs(sh - np.sinh(w)) <= 8 * 2.0 ** -53 * np.abs(np.sinh(w)))
    assert np.all(np.abs(ch - np.cosh(w)) <= 8 * 2.0 ** -53 * np.cosh(w))


@pytest.mark.parametrize("power", [-240, -130, -110, 110, 130, 240])
def test_edge_integrals_in_any_unit(lib, power):
    """The integral of an edge is a length: with all lengths times a power of two it
    is the same number times that. Terms of at most the edge's length cancel, each
    within a few 2^-53: 32 x 2^-53 of the terms."""
    rng = np.random.default_rng(1)
    n = 2000
    q = np.stack((rng.normal(size=n), 10 ** rng.uniform(-2, 0.5, n), rng.normal(size=n), rng.normal(size=n)), 1)
    s = 2.0 ** power
    a, b = np.zeros(n), np.zeros(n)
    for v, out in ((q, a), (q * s, b)):
        v = np.ascontiguousarray(v)
        lib.edge_of(n, ctypes.c_void_p(v.ctypes.data), ctypes.c_void_p(out.ctypes.data))
    terms = np.abs(q[:, 2]) * np.arcsinh(np.abs(q[:, 0]) + q[:, 1] + 1.0) + np.pi * np.abs(q[:, 3])
    assert np.all(np.abs(b / s - a) <= 32 * 2.0 ** -53 * terms)
