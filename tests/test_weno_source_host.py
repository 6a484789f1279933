"""The kernels' reconstruction arithmetic, compiled for the host from its own source text, against
the textbook WENO5-JS and WENO3 face values and against central differences.

weno.cuh is compiled as it stands in double, with the two hardware reciprocals replaced by
divisions, and weno5_diff_grad of adjoint_tile.cuh with its types widened to double.  What is
checked is the algebra, so the tolerances are those of double rounding: 1e-13 for values; central
differences of step h ~ 1e-6 of a function with eps = 1e-6 in its weights reach 1e-7."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from tests.test_weno_reformulations import _stencils, textbook

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_07694_gb300", "csrc")

SHIM = """
#include <cmath>
#define __device__
#define __forceinline__ inline
inline float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
inline double fma_t(double a, double b, double c) { return fma(a, b, c); }
constexpr int kSchemeWeno3 = 1, kSchemeSignSplit = 2;
"""

WRAP = """
extern "C" {
double weno5(const double* v) { return lw::recon_value(lw::weno5_recon<double>(v[0], v[1], v[2], v[3], v[4]), v[2]); }
double weno3(const double* v) { return lw::recon_value(lw::weno3_recon<double>(v[0], v[1], v[2]), v[1]); }
double face(const double* p, const double* m, double kd, double cl, double cr) {
  return lw::face_flux_x<double>(p[0], p[1], p[2], p[3], p[4], m[0], m[1], m[2], m[3], m[4], kd, cl, cr);
}
void grad(const double* v, double* e) {
  const double d1 = v[1] - v[0], d2 = v[2] - v[1], d3 = v[3] - v[2], d4 = v[4] - v[3];
  double g[4];
  lw::weno5_diff_grad(d1, d2, d3, d4, d2 - d1, d3 - d2, d4 - d3, g);
  for (int k = 0; k < 4; ++k) e[k] = g[k];
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    text = open(os.path.join(CSRC, "weno.cuh")).read()
    text = re.sub(r"^#(include|pragma).*$", "", text, flags=re.M)
    text, n = re.subn(r'asm\("rcp\.[^;]*;', "r = 1 / x;", re.sub(r'f(32|64) %0, %1;"', r'f\1 %0, %1"', text))
    assert n == 2
    tile = open(os.path.join(CSRC, "adjoint_tile.cuh")).read()
    grad = re.search(r"^__device__ __forceinline__ void weno5_diff_grad.*?^}", tile, re.S | re.M).group(0)
    grad = re.sub(r"(?<=[\d.])f\b", "", grad).replace("float", "double").replace("fmaf", "fma")
    grad = grad.replace("rcp_approx", "1.0 / ")
    d = tmp_path_factory.mktemp("weno")
    (d / "w.cc").write_text(SHIM + text + "namespace lw {\n" + grad + "\n}\n" + WRAP)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-o", str(d / "w.so"),
                    str(d / "w.cc")], check=True)
    L = ctypes.CDLL(str(d / "w.so"))
    dp = ctypes.POINTER(ctypes.c_double)
    for f in (L.weno5, L.weno3):
        f.argtypes, f.restype = [dp], ctypes.c_double
    L.face.argtypes, L.face.restype = [dp, dp] + [ctypes.c_double] * 3, ctypes.c_double
    L.grad.argtypes, L.grad.restype = [dp, dp], None
    return L


def _p(a):
    return np.ascontiguousarray(a).ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def textbook3(v, eps=1e-6):
    """Candidates (b + c)/2 and (3b - a)/2, indicators (c - b)^2 and (b - a)^2, weights 2/3 and 1/3."""
    a, b, c = v
    al = [(2 / 3) / (eps + (c - b) ** 2) ** 2, (1 / 3) / (eps + (b - a) ** 2) ** 2]
    return (al[0] * (b + c) / 2 + al[1] * (3 * b - a) / 2) / sum(al)


def test_face_values_are_the_textbook_ones(lib):
    for v in _stencils(2000, 2):
        ref = textbook(v)
        assert abs(lib.weno5(_p(v)) - ref) <= 1e-13 * max(1.0, abs(ref))
        ref = textbook3(v[:3])
        assert abs(lib.weno3(_p(v[:3])) - ref) <= 1e-13 * max(1.0, abs(ref))


def test_face_flux_adds_both_halves_and_diffusion(lib):
    rng = np.random.default_rng(3)
    for _ in range(300):
        p, m, c = rng.normal(size=5), rng.normal(size=5), rng.normal(size=2)
        ref = textbook(p) + textbook(m) + 0.02 * (c[0] - c[1])
        assert abs(lib.face(_p(p), _p(m), 0.02, c[0], c[1]) - ref) <= 1e-13 * max(1.0, abs(ref))


def test_difference_gradient_matches_central_differences(lib):
    for v in _stencils(500, 4):
        e = np.empty(4)
        lib.grad(_p(v), _p(e))
        dv = np.array([-e[0], e[0] - e[1], 1 + e[1] - e[2], e[2] - e[3], e[3]])
        h = 1e-6 * max(1e-3, np.abs(v).max())
        fd = np.array([(lib.weno5(_p(v + h * k)) - lib.weno5(_p(v - h * k))) / (2 * h) for k in np.eye(5)])
        assert np.abs(fd - dv).max() <= 1e-7 * max(1.0, np.abs(dv).max())
