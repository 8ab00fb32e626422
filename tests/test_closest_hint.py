"""The FP32 choice of the closest feature against the full evaluation, on the CPU.

geometry.cuh is compiled as plain C++ (its few device intrinsics replaced by their host
meaning) and closest_pair with closest_hint's features is compared with pt_distance and
ee_distance, which evaluate every feature: the squared distance, the weights and the free
parameters have to be the same bits, whatever the shape, the scale and the distance from
the origin, on generic stencils and on the ones where two features tie.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <cuda_runtime.h>
#include <cmath>
#include <cstring>
static inline long long __double_as_longlong(double x) { long long r; memcpy(&r, &x, 8); return r; }
static inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static inline int __double2loint(double x) { return (int)__double_as_longlong(x); }
static inline float __int_as_float(int x) { float r; memcpy(&r, &x, 4); return r; }
static inline float __double2float_rn(double x) { return (float)x; }
static inline float __double2float_rd(double x) { float f = (float)x; return f > x ? std::nextafter(f, -INFINITY) : f; }
static inline float __double2float_ru(double x) { float f = (float)x; return f < x ? std::nextafter(f, INFINITY) : f; }
static inline float __fdividef(float a, float b) { return a / b; }
template <class T> static inline T __ldg(const T* p) { return *p; }
static inline int __ffs(int x) { return __builtin_ffs(x); }
static inline unsigned atomicOr(int*, int) { return 0; }
static inline unsigned long long atomicMax(unsigned long long*, unsigned long long) { return 0; }
struct Dim { int x; };
static Dim gridDim, blockDim;
using std::fmaxf; using std::fminf; using std::isfinite;
#include "geometry.cuh"
using namespace eipc;
extern "C" void convert(long n, const double* x, float* rn, float* rd, float* ru) {
  for (long k = 0; k < n; ++k) {
    rn[k] = to_float<0>(x[k]);
    rd[k] = to_float<-1>(x[k]);
    ru[k] = to_float<1>(x[k]);
  }
}
extern "C" int compare(long n, const int* type, const double* x, int* features) {
  int bad = 0;
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
    Stencil A, B;
    const double full = type[k] == 0 ? pt_distance<true>(X[0], X[1], X[2], X[3], &A)
                                     : ee_distance<true>(X[0], X[1], X[2], X[3], &A);
    const int hint = closest_hint(type[k], P[0], P[1], P[2], P[3], M * 5.9604645e-8f);
    const double got = closest_pair<true>(type[k], X, hint, &B);
    const double plain = closest_pair<false>(type[k], X, hint, nullptr);
    features[k] = hint;
    bool same = full == got && plain == full && A.m == B.m;
    for (int a = 0; a < 4; ++a) same = same && A.c[a] == B.c[a] && A.a[0][a] == B.a[0][a] && A.a[1][a] == B.a[1][a];
    bad += !same;
  }
  return bad;
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    d = tmp_path_factory.mktemp("hint")
    (d / "hint.cpp").write_text(SHIM)
    so = d / "hint.so"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-fPIC", "-shared",
                           "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "paper_2409_16385_gb300", "csrc"),
                           str(d / "hint.cpp"), "-o", str(so)])
    lib = ctypes.CDLL(str(so))

    def convert(x):
        x = np.ascontiguousarray(x, np.float64)
        r = np.zeros((3, len(x)), np.float32)
        lib.convert(ctypes.c_long(len(x)), x.ctypes.data_as(ctypes.c_void_p), *(r[k].ctypes.data_as(ctypes.c_void_p) for k in range(3)))
        return r

    def run(ty, X):
        ty, X = np.ascontiguousarray(ty, np.int32), np.ascontiguousarray(X, np.float64)
        f = np.zeros(len(ty), np.int32)
        bad = lib.compare(ctypes.c_long(len(ty)), ty.ctypes.data_as(ctypes.c_void_p), X.ctypes.data_as(ctypes.c_void_p),
                          f.ctypes.data_as(ctypes.c_void_p))
        return bad, f

    run.convert = convert
    return run


def _stencils(rng, n, edge, gap, offset):
    X = rng.normal(size=(n, 4, 3)) * edge
    ty = rng.integers(0, 2, n)
    # the second primitive a seeded gap away, over the middle, an edge or a corner of the first
    X[:, 2:] += rng.normal(size=(n, 1, 3)) * gap
    return ty, X + rng.normal(size=(n, 1, 3)) * offset


@pytest.mark.parametrize("edge,gap", [(1e-3, 5e-4), (1e-2, 2e-4), (5e-5, 1e-3), (1.0, 1e-3), (1e-12, 1e-12), (1e4, 1.0)])
@pytest.mark.parametrize("offset", [0.0, 0.1, 3.0])
def test_generic_stencils_take_the_full_evaluations_feature(compare, edge, gap, offset):
    rng = np.random.default_rng(5)
    ty, X = _stencils(rng, 20000, edge, gap, offset)
    bad, f = compare(ty, X)
    assert bad == 0
    if edge == 1e-3 and offset == 0.1:         # and it does choose: one feature for most
        one = (f == 48) | ((f & 48 == 0) & (f & (f - 1) == 0))
        assert one.mean() > 0.8


@pytest.mark.parametrize("offset", [0.0, 0.25])
def test_ties_boundaries_and_degenerate_stencils(compare, offset):
    rng = np.random.default_rng(6)
    X, ty = [], []
    for _ in range(3000):
        p = rng.normal(size=(4, 3)) * 1e-3
        e, f = rng.normal(size=3) * 1e-3, rng.normal(size=3) * 1e-3
        s = rng.choice([0.0, 1.0, 0.5, 1e-9, 1 - 1e-9, -1e-9])
        t = rng.choice([0.0, 1.0, 0.5, 1e-9, 1 - 1e-9, 1 + 1e-9])
        h = np.cross(e, f) / np.linalg.norm(np.cross(e, f)) * 3e-4
        k = rng.integers(0, 8)
        if k == 0:                             # projection on a triangle's edge, corner or just beside
            X.append([p[0] + s * e + (1 - s) * t * f + h, p[0], p[0] + e, p[0] + f]); ty.append(0)
        elif k == 1:                           # closest to a corner: two edges tie
            X.append([p[0] - 0.3 * e - 0.3 * f + h, p[0], p[0] + e, p[0] + f]); ty.append(0)
        elif k == 2:                           # a degenerate triangle
            X.append([p[1], p[0], p[0] + e, p[0] + rng.choice([0.0, 0.5, 2.0]) * e]); ty.append(0)
        elif k == 3:                           # closest points at the ends of both segments
            X.append([p[0], p[0] + e, p[0] + h - t * f, p[0] + h + (1 - t) * f]); ty.append(1)
        elif k == 4:                           # parallel and nearly parallel edges
            X.append([p[0], p[0] + e, p[0] + h + s * e, p[0] + h + t * e + rng.choice([0, 1e-13, 1e-8]) * f]); ty.append(1)
        elif k == 5:                           # two edge ends against each other
            X.append([p[0], p[0] + e, p[0] + h - f, p[0] + h - 2 * f]); ty.append(1)
        elif k == 6:                           # a zero-length edge
            X.append([p[0], p[0], p[1], p[2]]); ty.append(1)
        else:                                  # crossing at parameters on the boundary
            X.append([p[0] - s * e, p[0] + (1 - s) * e, p[0] + h - t * f, p[0] + h + (1 - t) * f]); ty.append(1)
    X = np.array(X) + offset
    bad, _ = compare(np.array(ty), X)
    assert bad == 0


def test_integer_conversions_round_like_the_instructions(compare):
    """to_float's three roundings against numpy's conversion and its neighbours: exact values, ties,
    both sides of them, the ends of FP32's normal range, subnormals, zeros, infinities and NaN."""
    rng = np.random.default_rng(7)
    f = np.ldexp(rng.uniform(0.5, 1.0, 4000), rng.integers(-148, 128, 4000)).astype(np.float32)
    up = np.nextafter(f, np.float32(np.inf)).astype(np.float64)
    f = f.astype(np.float64)
    tie = 0.5 * (f + up)
    x = np.concatenate([f, tie, np.nextafter(tie, 0.0), np.nextafter(tie, np.inf), np.ldexp(rng.uniform(0.5, 1.0, 4000), -150),
                        np.ldexp(rng.uniform(0.5, 1.0, 4000), rng.integers(-300, 300, 4000)),
                        [0.0, np.inf, np.finfo(np.float32).max, 3.4028235677973366e38, 1e39, np.finfo(np.float32).tiny]])
    x = np.concatenate([x, -x, [np.nan]])
    with np.errstate(over="ignore"):
        rn = x.astype(np.float32)
    rd = np.where(rn.astype(np.float64) > x, np.nextafter(rn, np.float32(-np.inf)), rn)
    ru = np.where(rn.astype(np.float64) < x, np.nextafter(rn, np.float32(np.inf)), rn)
    got = compare.convert(x)
    for g, want in zip(got, (rn, rd, ru)):
        np.testing.assert_array_equal(g, want)


@pytest.mark.parametrize("edge,gap,offset", [(1e8, 1e7, 0.0), (1e9, 1e9, 0.0), (2e9, 1e8, 1e9), (1e10, 1e10, 0.0), (1e12, 1e11, 0.0),
                                             (1e19, 1e18, 0.0), (1e21, 1e21, 0.0), (1e36, 1e36, 0.0), (1e40, 1e40, 0.0),
                                             (1e-3, 1e20, 0.0), (1e-3, 1e-3, 1e25), (1e19, 1e-3, 0.0), (1e6, 1e18, 0.0)])
def test_stencils_beyond_fp32s_range_keep_every_feature(compare, edge, gap, offset):
    """Lengths whose products, squares or selves overflow FP32: nothing may be concluded from what did."""
    rng = np.random.default_rng(8)
    ty, X = _stencils(rng, 50000, edge, gap, offset)
    bad, _ = compare(ty, X)
    assert bad == 0
    X = X * 10.0 ** rng.uniform(-12, 0, (len(X), 4, 1))           # ... and mixed with short ones
    bad, _ = compare(ty, X)
    assert bad == 0
