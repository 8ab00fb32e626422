// Device-side unsigned distance of point-triangle (PT) and edge-edge (EE) stencils
// (Sec. III-B, d_k(x)) with the closest-feature stencil needed by the closed-form
// derivatives.
//
// A stencil's squared distance is a partial minimum s(x) = min_beta |r(x, beta)|^2 with
// r = sum_a c_a(beta) x_a affine in beta (beta: barycentric / segment parameters of the
// closest feature).  For each region we report
//   c[4]      the coefficients at the minimiser (r = sum c_a x_a),
//   m         the number of free parameters of that feature (0, 1 or 2),
//   a[j][4]   dc/dbeta_j (constant per region),
// from which eval.cu builds the exact gradient and Hessian of s by the Schur complement of
// the inner minimisation.  Region choice: PT -- projection inside the triangle, else the
// nearest of the three edges (t0t1, t1t2, t2t0); EE -- unconstrained segment-parameter
// minimiser inside [0,1]^2 (and the segments not parallel to within 1e-20 relative),
// else the nearest of (a0, seg b), (a1, seg b), (b0, seg a), (b1, seg a); ties keep the
// first in that order.
#pragma once
#include "common.cuh"

namespace eipc {

struct Stencil {
  double c[4];
  double a[2][4];
  int m;
  double d2;
};

// Comparisons of doubles as integers: an FP64 compare holds the FP64 pipe for nearly two
// instruction slots, an integer one costs next to nothing.  a > 0; and a < b, a >= b for
// non-negative operands (whose bit patterns are ordered like their values).
__device__ __forceinline__ bool is_pos(double a) { return __double_as_longlong(a) > 0; }
__device__ __forceinline__ bool lt_nonneg(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }

// x to FP32, rounded to nearest (mode 0), down (-1) or up (+1), by integer instructions: the
// conversion instruction holds the FP64 pipe like an FP64 operation.  Results of FP32's normal
// range and zeros; anything else takes the instruction.
template <int mode>
__device__ __forceinline__ float to_float(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  if (((hi << 1) | lo) == 0) return __int_as_float(hi);
  const int e = ((hi >> 20) & 0x7ff) - 896;            // biased FP32 exponent
  if (e >= 1 && e <= 253) {
    const unsigned mag = ((unsigned)e << 23) | ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)lo >> 29);
    const unsigned rest = (unsigned)lo & 0x1fffffffu;
    const bool up = mode == 0 ? (rest > 0x10000000u || (rest == 0x10000000u && (mag & 1u)))
                              : (rest != 0u && (mode < 0) == (hi < 0));
    return __int_as_float((int)((unsigned)(hi & 0x80000000) | (mag + (up ? 1u : 0u))));
  }
  return mode == 0 ? __double2float_rn(x) : (mode < 0 ? __double2float_rd(x) : __double2float_ru(x));
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Per-vertex FP32 box of [lo, hi], rounded outward from the FP64 positions, in rows of 8 floats (lo
// xyz, hi xyz).  Outward rounding is monotone, so the min / max over a primitive's vertices of
// these boxes is bit for bit the box made from the primitive's FP64 positions: the hierarchy
// and the traversal read these instead of recomputing FP64 minima per primitive.
__device__ __forceinline__ void store_box(float* row, const double lo[3], const double hi[3]) {
  float4* o = reinterpret_cast<float4*>(row);
  o[0] = make_float4(to_float<-1>(lo[0]), to_float<-1>(lo[1]), to_float<-1>(lo[2]), to_float<1>(hi[0]));
  o[1] = make_float4(to_float<1>(hi[1]), to_float<1>(hi[2]), 0.f, 0.f);
}

// |p - (e0 + t (e1 - e0))|^2 over t in [0,1].  t = clamp((w.e) / (e.e), 0, 1), with the
// quotient (one reciprocal and a product) taken only inside (0, 1): w.e <= 0 gives 0 and
// w.e >= e.e gives 1, also for e = 0.  A NaN gives a NaN distance either way.
__device__ __forceinline__ double seg_point_d2(V3 p, V3 e0, V3 e1, double* t_out) {
  V3 e = e1 - e0, w = p - e0;
  const double we = dot(w, e), ee = dot(e, e);
  double t;
  if (!is_pos(we)) t = 0.0;
  else if (!lt_nonneg(we, ee)) t = 1.0;
  else t = we * (1.0 / ee);
  V3 r = w - e * t;
  *t_out = t;
  return dot(r, r);
}

__device__ __forceinline__ void set_zero(Stencil& S) {
#pragma unroll
  for (int k = 0; k < 4; ++k) { S.c[k] = 0.0; S.a[0][k] = 0.0; S.a[1][k] = 0.0; }
}

// closest feature on segment (ia, ib) at parameter t, seen from a fixed point slot `ip`
// with sign +1 (point on side A) -- used for PT edges and EE endpoint cases
__device__ __forceinline__ void point_segment_stencil(Stencil& S, int ip, double sp, int ia, int ib,
                                                      double t) {
  const bool at_a = !is_pos(t), at_b = __double2hiint(t) >= 0x3ff00000;   // t <= 0, t >= 1
  const double ca = at_b ? 0.0 : (at_a ? -sp : -sp * (1.0 - t)), cb = at_a ? 0.0 : (at_b ? -sp : -sp * t);
  const bool inner = !at_a && !at_b;
#pragma unroll
  for (int k = 0; k < 4; ++k) {            // selects, so that the stencil stays in registers
    S.c[k] = k == ip ? sp : (k == ia ? ca : (k == ib ? cb : 0.0));
    S.a[0][k] = !inner ? 0.0 : (k == ia ? sp : (k == ib ? -sp : 0.0));
    S.a[1][k] = 0.0;
  }
  S.m = inner ? 1 : 0;
}

template <bool kStencil>
__device__ __forceinline__ double pt_distance(V3 p, V3 t0, V3 t1, V3 t2, Stencil* S) {
  V3 e1 = t1 - t0, e2 = t2 - t0, w = p - t0;
  V3 n = cross(e1, e2);
  double nn = dot(n, n);
  // barycentric coordinates of the projection: beta1 = ((w x e2) . n)/nn, etc., with one
  // reciprocal of nn for the three quotients (nn = 0 gives infinite or NaN barycentrics,
  // which fail the face test, as the quotients would)
  const double inv_nn = 1.0 / nn;
  double b1 = dot(cross(w, e2), n) * inv_nn;
  double b2 = dot(cross(e1, w), n) * inv_nn;
  if (b1 >= 0.0 && b2 >= 0.0 && b1 + b2 <= 1.0) {
    double h = dot(w, n);
    double d2 = h * h * inv_nn;
    if (kStencil) {
      set_zero(*S);
      S->c[0] = 1.0; S->c[1] = -(1.0 - b1 - b2); S->c[2] = -b1; S->c[3] = -b2;
      S->a[0][1] = 1.0; S->a[0][2] = -1.0;
      S->a[1][1] = 1.0; S->a[1][3] = -1.0;
      S->m = 2;
      S->d2 = d2;
    }
    return d2;
  }
  double ta, tb, tc;
  double da = seg_point_d2(p, t0, t1, &ta);
  double db = seg_point_d2(p, t1, t2, &tb);
  double dc = seg_point_d2(p, t2, t0, &tc);
  int k = 0;
  double best = da, tbest = ta;
  if (db < best) { best = db; tbest = tb; k = 1; }
  if (dc < best) { best = dc; tbest = tc; k = 2; }
  if (kStencil) {
    point_segment_stencil(*S, 0, 1.0, 1 + k, 1 + (k + 1) % 3, tbest);
    S->d2 = best;
  }
  return best;
}

template <bool kStencil>
__device__ __forceinline__ double ee_distance(V3 a0, V3 a1, V3 b0, V3 b1, Stencil* S) {
  V3 ea = a1 - a0, eb = b1 - b0, w = a0 - b0;
  double A = dot(ea, ea), B = dot(ea, eb), C = dot(eb, eb);
  double D = dot(ea, w), E = dot(eb, w);
  V3 n = cross(ea, eb);
  double nn = dot(n, n);
  if (nn > 1e-20 * A * C) {
    const double inv_nn = 1.0 / nn;
    double s = (B * E - C * D) * inv_nn;
    double t = (A * E - B * D) * inv_nn;
    if (s >= 0.0 && s <= 1.0 && t >= 0.0 && t <= 1.0) {
      double h = dot(w, n);
      double d2 = h * h * inv_nn;
      if (kStencil) {
        set_zero(*S);
        S->c[0] = 1.0 - s; S->c[1] = s; S->c[2] = -(1.0 - t); S->c[3] = -t;
        S->a[0][0] = -1.0; S->a[0][1] = 1.0;
        S->a[1][2] = 1.0; S->a[1][3] = -1.0;
        S->m = 2;
        S->d2 = d2;
      }
      return d2;
    }
  }
  double t0, t1, t2, t3;
  double d0 = seg_point_d2(a0, b0, b1, &t0);
  double d1 = seg_point_d2(a1, b0, b1, &t1);
  double d2 = seg_point_d2(b0, a0, a1, &t2);
  double d3 = seg_point_d2(b1, a0, a1, &t3);
  int k = 0;
  double best = d0, tb = t0;
  if (d1 < best) { best = d1; tb = t1; k = 1; }
  if (d2 < best) { best = d2; tb = t2; k = 2; }
  if (d3 < best) { best = d3; tb = t3; k = 3; }
  if (kStencil) {
    if (k < 2) point_segment_stencil(*S, k, 1.0, 2, 3, tb);      // a_k - point on b
    else point_segment_stencil(*S, k, -1.0, 0, 1, tb);          // point on a - b_{k-2}
    S->d2 = best;
  }
  return best;
}

// ---------------------------------------------------------------- FP32 screen
// "Certainly farther than r" tests in FP32 only (62x the FP64 rate on GB300), on FP32 copies
// of the positions.  With M the largest coordinate of the candidate's points, each FP32
// coordinate is off by <= M 2^-24 and the FP32 distance by a small multiple of that (taken
// as 40 M 2^-24).  The callers prove far with a radius grown by twice that, 80 M 2^-24, and
// declare a pair far only if its FP32 squared distance also exceeds r^2 (1 + 4e-3), i.e.
// d > r (1 + 2e-3): the margin holds at any scene size.  Misclassifying the closest
// region can only (a) report a lower bound (plane / line distance when the projection is
// wrongly found inside), or (b) report a boundary value whose excess is bounded by the
// curvature times the squared parameter error.  Stencils whose parameter solve is not
// well conditioned (|n|^2 <= 0.1 |e1|^2 |e2|^2) are screened by a bound that needs no
// parameter solve: edges within 18 degrees of parallel by their segment-to-line distances
// (seg_line_far_f32); skinny triangles not at all.  Nor is a stencil whose products leave FP32's range
// (with dhat as large as the edges, at 1e5 units and more and at 1e-6 and less): an infinite, NaN or
// subnormal one proves nothing.  Every pair not screened goes through the exact FP64 test, so the
// kept set is unchanged.
struct F3 {
  float x, y, z;
};
__device__ __forceinline__ F3 load_xf(const float* __restrict__ x4f, int32_t v) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(x4f) + v);
  return {a.x, a.y, a.z};
}
__device__ __forceinline__ F3 operator-(F3 a, F3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ F3 operator*(F3 a, float s) { return {a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ float fdot(F3 a, F3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ F3 fcross(F3 a, F3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
// |w - t e|^2 over t in [0,1] (w relative to the segment start)
__device__ __forceinline__ float fseg_d2(F3 w, F3 e) {
  float t = fdot(w, e) / fdot(e, e);
  t = fminf(fmaxf(t, 0.f), 1.f);
  const F3 r = w - e * t;
  return fdot(r, r);
}

// a product that neither overflowed nor lost more than 2^-12 of itself as a subnormal
__device__ __forceinline__ bool in_f32_range(float x) { return x > 1e-41f && x < INFINITY; }

__device__ __forceinline__ bool pt_far_f32(F3 p, F3 t0, F3 t1, F3 t2, float r2m) {
  const F3 e1 = t1 - t0, e2 = t2 - t0, w = p - t0;
  const F3 n = fcross(e1, e2);
  const float nn = fdot(n, n), A = fdot(e1, e1), C = fdot(e2, e2);
  if (!(nn > 0.1f * A * C && nn > 1e-38f && A + C < 1e38f)) return false;
  const float b1 = fdot(fcross(w, e2), n) / nn;
  const float b2 = fdot(fcross(e1, w), n) / nn;
  if (!(fabsf(b1) + fabsf(b2) < INFINITY)) return false;
  float d2;
  if (b1 >= 0.f && b2 >= 0.f && b1 + b2 <= 1.f) {
    const float h = fdot(w, n), hh = h * h;
    if (!in_f32_range(hh)) return false;
    d2 = hh / nn;
  } else {
    d2 = fminf(fseg_d2(w, e1), fminf(fseg_d2(w - e1, e2 - e1), fseg_d2(w, e2)));
  }
  return d2 > r2m;
}

// Segment-to-line lower bound for near-parallel edges: with U = (segment start - line
// point) x e_line and V = e_seg x e_line, the squared distance from the point at parameter
// s of the segment to the line is |U + s V|^2 / L (L = |e_line|^2).  Its minimum over
// s in [0, 1] is |U|^2 (U.V >= 0), |U + V|^2 (U.V <= -|V|^2), else |U x V|^2 / |V|^2
// (Lagrange's identity, free of the cancellation in |U|^2 - (U.V)^2 / |V|^2).  A case
// chosen wrongly through rounding of U.V overestimates by at most (err U.V)^2 / |V|^2,
// of order eps^2 |U|^2: negligible against the margin.  The segments' distance is at least
// this (the other segment lies on the line), so "far" here proves the pair far.  The
// interior case needs |V|^2 > 1e-12 |e_seg|^2 L (edges not parallel to within 1e-6 rad),
// else nothing is proven.
__device__ __forceinline__ bool seg_line_far_f32(F3 U, F3 V, float Lseg, float L, float r2m) {
  const float uv = fdot(U, V), vv = fdot(V, V);
  if (!(vv + fabsf(uv) < INFINITY)) return false;
  float g;
  if (uv >= 0.f) {
    g = fdot(U, U);
  } else if (uv <= -vv) {
    const F3 W = {U.x + V.x, U.y + V.y, U.z + V.z};
    g = fdot(W, W);
  } else {
    if (!(vv > 1e-12f * Lseg * L && vv > 1e-38f)) return false;
    const F3 X = fcross(U, V);
    const float xx = fdot(X, X);
    if (!in_f32_range(xx)) return false;
    g = xx / vv;
  }
  return g > r2m * L && g > 1e-41f;
}

__device__ __forceinline__ bool ee_far_f32(F3 a0, F3 a1, F3 b0, F3 b1, float r2m) {
  const F3 ea = a1 - a0, eb = b1 - b0, w = a0 - b0;
  const float A = fdot(ea, ea), C = fdot(eb, eb);
  const F3 n = fcross(ea, eb);
  const float nn = fdot(n, n);
  if (!(nn > 0.1f * A * C && nn > 1e-38f)) {
    // near-parallel: segment a against line b, segment b against line a
    const F3 wb = b0 - a0;
    return seg_line_far_f32(fcross(w, eb), n, A, C, r2m) || seg_line_far_f32(fcross(wb, ea), n * -1.f, C, A, r2m);
  }
  const float B = fdot(ea, eb), D = fdot(ea, w), E = fdot(eb, w);
  const float s = (B * E - C * D) / nn, t = (A * E - B * D) / nn;
  if (!(fabsf(s) + fabsf(t) < INFINITY)) return false;
  float d2;
  if (s >= 0.f && s <= 1.f && t >= 0.f && t <= 1.f) {
    const float h = fdot(w, n), hh = h * h;
    if (!in_f32_range(hh)) return false;
    d2 = hh / nn;
  } else {
    d2 = fminf(fminf(fseg_d2(w, eb), fseg_d2(a1 - b0, eb)), fminf(fseg_d2(b0 - a0, ea), fseg_d2(b1 - a0, ea)));
  }
  return d2 > r2m;
}

// ---------------------------------------------------------------- FP32 choice of feature
// On GB300 an FP64 warp instruction holds its sub-partition's pipe for 64 cycles however many
// lanes are active (one dependent chain already saturates it), an FP32 one for about 1.6.  The
// FP64 distance above spends most of its instructions on features that turn out not to be the
// closest: the interior solve and three or four segments.  closest_hint decides in FP32 which
// of them can be: bit k (k < 4) for segment k (PT: t0t1, t1t2, t2t0; EE: a0-b, a1-b, b0-a,
// b1-a), kHintInterior if the interior solution is possible, kHintCertain if nothing else is.
// closest_pair then runs the same FP64 formulas, in the same order and with the same ties, on
// the features left: a feature is dropped only if its FP32 value misses the smallest by more
// than the error of both, so the result is the full evaluation's.
//
// Errors (u = 2^-24): a coordinate read from its FP32 copy is off by ec = M u, M the largest
// coordinate.  With E, W the longest edge and the offset w, the numerators of the interior
// parameters (sizes up to W E^3) are off by at most (16 u W E + 8 ec (E + 3 W)) E^2 to first
// order, taken as 64 (u E + ec)(W + E) E^2; a segment's FP32 distance is off by 8 u (W + E) + 4 ec,
// taken as 32 u (W + E) + 8 ec (its parameter enters in second order).  Where |e1 x e2|^2 is
// below 1e-6 |e1|^2 |e2|^2 or close to FP32's smallest numbers nothing is concluded.  Where the bound
// 64 (u E + ec)(W + E) E^2 is not below 1e30 -- lengths whose products may overflow FP32, infinite
// and NaN coordinates -- every feature is left in; below it W E^3 and E^4 are under 3e35, and every
// product here is finite.
constexpr int kHintInterior = 16, kHintCertain = 32;

__device__ __forceinline__ float fmax_abs(F3 a) { return fmaxf(fabsf(a.x), fmaxf(fabsf(a.y), fabsf(a.z))); }

__device__ __forceinline__ float fseg_d2_fast(F3 w, F3 e) {
  const float t = fminf(fmaxf(__fdividef(fdot(w, e), fdot(e, e)), 0.f), 1.f);
  const F3 r = w - e * t;
  return fdot(r, r);
}

__device__ __forceinline__ int closest_hint(int type, F3 p0, F3 p1, F3 p2, F3 p3, float ec) {
  const bool pt = type == 0;
  const F3 e1 = pt ? p2 - p1 : p1 - p0, e2 = pt ? p3 - p1 : p3 - p2, w = pt ? p0 - p1 : p0 - p2;
  const F3 n = fcross(e1, e2);
  const float nn = fdot(n, n), A = fdot(e1, e1), C = fdot(e2, e2), ww = fdot(w, w);
  const float Em = sqrtf(fmaxf(A, C)), W = sqrtf(ww);
  const float u = 5.9604645e-8f;
  const float tol = 64.f * (u * Em + ec) * (W + Em) * Em * Em;
  if (!(tol < 1e30f)) return kHintInterior | (pt ? 7 : 15);
  float lo;                                    // signed room inside the parameter region (times nn)
  float d2[4];
  if (pt) {
    const float n1 = fdot(fcross(w, e2), n), n2 = fdot(fcross(e1, w), n);
    lo = fminf(fminf(n1, n2), nn - n1 - n2);
    d2[0] = fseg_d2_fast(w, e1);
    d2[1] = fseg_d2_fast(p0 - p2, p3 - p2);
    d2[2] = fseg_d2_fast(p0 - p3, p1 - p3);
    d2[3] = INFINITY;
  } else {
    const float B = fdot(e1, e2), D = fdot(e1, w), E = fdot(e2, w);
    const float n1 = B * E - C * D, n2 = A * E - B * D;
    lo = fminf(fminf(n1, n2), fminf(nn - n1, nn - n2));
    d2[0] = fseg_d2_fast(w, e2);
    d2[1] = fseg_d2_fast(p1 - p2, e2);
    d2[2] = fseg_d2_fast(p2 - p0, e1);
    d2[3] = fseg_d2_fast(p3 - p0, e1);
  }
  const bool sharp = nn > 1e-6f * A * C && nn > 1e-30f;
  if (sharp && lo > 2.f * tol) return kHintInterior | kHintCertain;
  int hint = (sharp && lo < -2.f * tol) ? 0 : kHintInterior;
  const float dm = fminf(fminf(d2[0], d2[1]), fminf(d2[2], d2[3]));
  const float r = sqrtf(dm) + 64.f * u * (W + Em) + 16.f * ec;
  const float thr = r * r + 1e-30f;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (!(d2[k] > thr)) hint |= 1 << k;
  return pt ? hint & ~8 : hint;
}

// closest_hint of a stencil from the FP32 copies of its positions
__device__ __forceinline__ int stencil_hint(int type, const float* __restrict__ x4f, const int32_t v[4]) {
  F3 P[4];
  float M = 0.f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    P[a] = load_xf(x4f, v[a]);
    M = fmaxf(M, fmax_abs(P[a]));
  }
  return closest_hint(type, P[0], P[1], P[2], P[3], M * 5.9604645e-8f);
}

// X[k] by selects (a run-time index would put X in local memory)
template <class T>
__device__ __forceinline__ T pick(const T X[4], int k) {
  T r = X[0];
  if (k == 1) r = X[1];
  if (k == 2) r = X[2];
  if (k == 3) r = X[3];
  return r;
}

// slots of the point and the segment ends of segment k of a stencil
__device__ __forceinline__ void segment_slots(int type, int k, int* ip, int* ia, int* ib) {
  if (type == 0) {
    *ip = 0; *ia = 1 + k; *ib = k == 2 ? 1 : 2 + k;
  } else {
    *ip = k; *ia = k < 2 ? 2 : 0; *ib = k < 2 ? 3 : 1;
  }
}

// pt_distance (type 0) / ee_distance (type 1) of X with the features of `hint`
template <bool kStencil>
__device__ __forceinline__ double closest_pair(int type, const V3 X[4], int hint, Stencil* S) {
  if (hint & kHintInterior) {
    const bool certain = (hint & kHintCertain) != 0;
    const V3 e1 = type == 0 ? X[2] - X[1] : X[1] - X[0];
    const V3 e2 = type == 0 ? X[3] - X[1] : X[3] - X[2];
    const V3 w = type == 0 ? X[0] - X[1] : X[0] - X[2];
    const V3 n = cross(e1, e2);
    const double nn = dot(n, n);
    const double inv_nn = 1.0 / nn;
    double s = 0.0, t = 0.0;
    bool in = certain;
    if (type == 0) {
      if (kStencil || !certain) {
        s = dot(cross(w, e2), n) * inv_nn;
        t = dot(cross(e1, w), n) * inv_nn;
        in = certain || (s >= 0.0 && t >= 0.0 && s + t <= 1.0);
      }
    } else if (kStencil || !certain) {
      const double A = dot(e1, e1), B = dot(e1, e2), C = dot(e2, e2), D = dot(e1, w), E = dot(e2, w);
      s = (B * E - C * D) * inv_nn;
      t = (A * E - B * D) * inv_nn;
      in = certain || (nn > 1e-20 * A * C && s >= 0.0 && s <= 1.0 && t >= 0.0 && t <= 1.0);
    }
    if (in) {
      const double h = dot(w, n);
      const double d2 = h * h * inv_nn;
      if (kStencil) {
        set_zero(*S);
        if (type == 0) {
          S->c[0] = 1.0; S->c[1] = -(1.0 - s - t); S->c[2] = -s; S->c[3] = -t;
          S->a[0][1] = 1.0; S->a[0][2] = -1.0;
          S->a[1][1] = 1.0; S->a[1][3] = -1.0;
        } else {
          S->c[0] = 1.0 - s; S->c[1] = s; S->c[2] = -(1.0 - t); S->c[3] = -t;
          S->a[0][0] = -1.0; S->a[0][1] = 1.0;
          S->a[1][2] = 1.0; S->a[1][3] = -1.0;
        }
        S->m = 2;
        S->d2 = d2;
      }
      return d2;
    }
  }
  int k = -1;
  double best = 0.0, tb = 0.0;
  int left = hint & 15;
  for (int step = 0; step < 4 && left; ++step) {
    const int q = __ffs(left) - 1;
    left &= left - 1;
    int ip, ia, ib;
    segment_slots(type, q, &ip, &ia, &ib);
    double t;
    const double d2 = seg_point_d2(pick(X, ip), pick(X, ia), pick(X, ib), &t);
    if (k < 0 || d2 < best) { best = d2; tb = t; k = q; }
  }
  if (kStencil) {
    int ip, ia, ib;
    segment_slots(type, k, &ip, &ia, &ib);
    point_segment_stencil(*S, ip, (type == 0 || k < 2) ? 1.0 : -1.0, ia, ib, tb);
    S->d2 = best;
  }
  return best;
}

}  // namespace eipc
