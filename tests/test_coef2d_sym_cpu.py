"""The linear p0 by parity classes that the 2D kernels evaluate
(csrc/hweno2d_sym.cuh): the generated code itself, compiled for the host in
FP64, against the oracle's derivation of the same polynomial, and its
transposes against the maps."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2002_08816_gb300", "csrc")

HOST = r"""
#define __device__
#define __forceinline__ inline
#include "hweno2d_sym.cuh"
#define MAPS(ng)                                                              \
  extern "C" void map%ng%(const double* d, double* o) {                       \
    double s[19];                                                             \
    hw2::p0_classes(d, s);                                                    \
    hw2::p0s_xfaces_ng%ng%(s, o);                                             \
    hw2::p0s_yfaces_ng%ng%(s, o + 2 * %ng%);                                  \
    hw2::p0s_interior_ng%ng%(s, o + 4 * %ng%);                                \
  }                                                                           \
  extern "C" void map%ng%T(const double* l, double* d) {                      \
    double s[19] = {0.0};                                                     \
    hw2::p0s_xfaces_ng%ng%_T(l, s);                                           \
    hw2::p0s_yfaces_ng%ng%_T(l + 2 * %ng%, s);                                \
    hw2::p0s_interior_ng%ng%_T(l + 4 * %ng%, s);                              \
    hw2::p0_classes_T(s, d);                                                  \
  }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sym")
    head, body = HOST.split("#define MAPS(ng)")
    body = body.replace("\\\n", "\n")
    (d / "m.cpp").write_text(head + body.replace("%ng%", "2") + body.replace("%ng%", "3"))
    so = str(d / "m.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I" + CSRC, str(d / "m.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _call(f, x, n):
    x, out = np.ascontiguousarray(x, dtype=np.float64), np.zeros(n)
    f(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
    return out


@pytest.mark.parametrize("ng", [2, 3])
def test_parity_class_maps_match_the_oracle(lib, ng):
    """Coefficient by coefficient: the value at each point for unit data (exact
    rationals to 20 digits against an FP64 KKT solve: 1e-12)."""
    npt = 4 * ng + ng * ng
    M = np.zeros((npt, 19))
    for j in range(19):
        d = np.zeros(19)
        d[j] = 1.0
        vb, wb = np.zeros(9), np.zeros(9)
        vb[[1, 3, 4, 5, 7]], wb[[1, 3, 4, 5, 7]] = d[9:14], d[14:19]
        M[:, j] = _call(getattr(lib, "map%d" % ng), d, npt)
        np.testing.assert_allclose(M[:, j], O.recon_candidates2d(d[:9], vb, wb, ng)[0][0], atol=1e-12)
    for p in range(npt):  # the transposes: the same matrix, column by column
        l = np.zeros(npt)
        l[p] = 1.0
        np.testing.assert_allclose(_call(getattr(lib, "map%dT" % ng), l, 19), M[p], atol=1e-14)
