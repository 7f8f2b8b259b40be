"""The FP64 quotient of the 2D kernels from a correctly rounded reciprocal
(csrc/hweno2d_common.cuh: quotient): the function itself, compiled for the host,
against IEEE division (which is CUDA's too), bit for bit."""

import ctypes
import os
import re
import subprocess

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2002_08816_gb300", "csrc")


def test_quotient_is_the_correctly_rounded_one(tmp_path):
    txt = open(os.path.join(CSRC, "hweno2d_common.cuh")).read()
    body = re.search(r"__device__ __forceinline__ (double quotient\(double x, double rho, double ir\) \{.*?\n\})",
                     txt, re.S).group(1)
    (tmp_path / "q.cpp").write_text("#include <cmath>\nusing std::fma;\nstatic " + body + """
extern "C" long differ(const double* x, const double* r, long n, double* out) {
  long k = 0;
  for (long i = 0; i < n; ++i) {
    out[i] = quotient(x[i], r[i], 1.0 / r[i]);
    k += !(out[i] == x[i] / r[i]);
  }
  return k;
}
""")
    so = str(tmp_path / "q.so")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", str(tmp_path / "q.cpp"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.differ.restype = ctypes.c_long
    rng = np.random.default_rng(7)
    n = 1000000

    def differ(x, r):
        x, r = np.ascontiguousarray(x), np.ascontiguousarray(r)
        out = np.empty_like(x)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        return lib.differ(p(x), p(r), ctypes.c_long(x.size), p(out))
    m = 1.0 + rng.integers(0, 1 << 52, (2, n)) * 2.0 ** -52
    sign = rng.choice([-1.0, 1.0], n)
    # mantissas of every kind over exponents whose quotients and remainders stay normal
    assert differ(sign * np.ldexp(m[0], rng.integers(-300, 300, n)), np.ldexp(m[1], rng.integers(-300, 300, n))) == 0
    # quotients within an ulp of a representable number or of a midpoint
    q = 1.0 + rng.integers(0, 1 << 52, n) * 2.0 ** -52
    x = m[1] * q
    assert differ(x, m[1]) + differ(np.nextafter(x, 0.0), m[1]) + differ(np.nextafter(x, 9.0), m[1]) == 0
    # next to the powers of two, and zero
    e = 1.0 + np.arange(1, 1001) * 2.0 ** -52
    a, b = (v.reshape(-1) for v in np.meshgrid(np.concatenate([e, 2.0 - e + 1.0, [0.0, 1.0]]),
                                               np.concatenate([e, 2.0 - e + 1.0 - 2.0 ** -52])))
    assert differ(a, b) == 0
