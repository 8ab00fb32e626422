"""The FP32 far tests on the CPU: a pair closer than the radius is never proven far, at any scale.

geometry.cuh is compiled as plain C++ (as in test_closest_hint) and pt_far_f32 and ee_far_f32 are given
the radius that the contact screen gives them, for a dhat a thousandth above the FP64 distance and
for half of it: nothing may be far in the first case, and at scales where no product overflows nearly
everything is in the second.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from test_closest_hint import ROOT, SHIM

SCREEN = SHIM.split('extern "C" int compare')[0] + r"""
extern "C" int far_count(long n, const int* type, const double* x, double scale) {
  int far = 0;
  for (long k = 0; k < n; ++k) {
    V3 X[4];
    F3 P[4];
    float M = 0.f;
    for (int a = 0; a < 4; ++a) {
      const double* p = x + 12 * k + 3 * a;
      X[a] = {p[0], p[1], p[2]};
      P[a] = {(float)p[0], (float)p[1], (float)p[2]};
      M = fmaxf(M, fmax_abs(P[a]));
    }
    const double d = sqrt(type[k] == 0 ? pt_distance<false>(X[0], X[1], X[2], X[3], nullptr)
                                       : ee_distance<false>(X[0], X[1], X[2], X[3], nullptr));
    const float r = __double2float_ru(scale * d) + 80.f * M * 5.9604645e-8f, r2m = r * r * 1.004f;
    far += type[k] == 0 ? pt_far_f32(P[0], P[1], P[2], P[3], r2m) : ee_far_f32(P[0], P[1], P[2], P[3], r2m);
  }
  return far;
}
"""


@pytest.fixture(scope="module")
def far_count(tmp_path_factory):
    d = tmp_path_factory.mktemp("far")
    (d / "far.cpp").write_text(SCREEN)
    so = d / "far.so"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-fPIC", "-shared",
                           "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "paper_2409_16385_gb300", "csrc"),
                           str(d / "far.cpp"), "-o", str(so)])
    lib = ctypes.CDLL(str(so))
    return lambda ty, X, s: lib.far_count(ctypes.c_long(len(ty)), ty.ctypes.data_as(ctypes.c_void_p),
                                          X.ctypes.data_as(ctypes.c_void_p), ctypes.c_double(s))


@pytest.mark.parametrize("edge", [1e-12, 1e-10, 1e-9, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3, 1.0, 1e4, 1e5, 1e6, 1e7, 1e8, 1e9, 1e10, 1e12, 1e19, 1e30])
def test_pairs_within_the_radius_are_never_far(far_count, edge):
    rng = np.random.default_rng(9)
    n = 100000
    X = rng.normal(size=(n, 4, 3)) * edge
    X[:, 2:] += rng.normal(size=(n, 1, 3)) * edge * rng.choice([0.1, 1.0, 3.0], size=(n, 1, 1))
    par = rng.random(n) < 0.4                  # nearly parallel second primitive
    X[par, 3] = X[par, 2] + (X[par, 1] - X[par, 0]) * rng.uniform(0.5, 2.0, (par.sum(), 1)) + rng.normal(size=(par.sum(), 3)) * edge * 0.05
    ty = rng.integers(0, 2, n).astype(np.int32)
    assert far_count(ty, np.ascontiguousarray(X), 1.001) == 0
    if 1e-4 < edge < 1e5:
        assert far_count(ty, np.ascontiguousarray(X), 0.5) > 0.8 * n
