// Step bound for the straight full-space motion x + t dx (Sec. III-C: phi is linear, so a
// reduced step is a straight motion of every surface vertex and linear CCD is exact).
//
// Candidates: PT / EE pairs (not incident, not all kinematic) whose closed FP64 swept
// boxes over [x, x + dx] overlap -- found with an LBVH over FP32 swept boxes rounded
// outward, then confirmed with the exact FP64 box test.  Per candidate, conservative
// advancement: remove the stencil's mean displacement; L = (largest relative speed on side
// A) + (largest on side B) bounds how fast the distance can shrink, so advancing t by
// (1 - s) d(t) / L keeps d > 0 on the whole advance; stop once d(t) <= s d(0), at t >= 1
// (then t = 1) or after accd_max_iter advances (the t reached is still safe).
// alpha = min(1, min_k t_k): exact minimum via atomicMin on the IEEE bit pattern (t >= 0),
// so the result does not depend on thread order.  A pair's t is scaled by (1 - 2^-30)
// before the minimum: a deliberate margin that keeps alpha on the safe side of rounding
// differences between this FP64 arithmetic and any other evaluation of the same bound.
#include "geometry.cuh"
#include "scene.cuh"
#include "sort.cuh"

namespace eipc {
namespace {

constexpr int kAccdThreads = 128;
constexpr double kMargin = 1.0 - 9.313225746154785e-10;   // 1 - 2^-30

// First kernel of a step bound: padded copies of x and dx, their FP32 copies, the per-vertex
// swept boxes, the counters and the bounds reset to one -- one pass over the vertices.
__global__ void __launch_bounds__(kBlock) k_ccd_begin(const double* __restrict__ x, const double* __restrict__ dx,
                                                      int64_t nv, double* __restrict__ x4, double* __restrict__ dx4,
                                                      float* __restrict__ x4f, float* __restrict__ dx4f,
                                                      float* __restrict__ vbox, DevStatus* st, CounterList zero,
                                                      unsigned long long* bits, unsigned long long* group_bits, int32_t ng) {
  pdl_entry();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int c = 0; c < kCounterList; ++c)
      if (zero.p[c]) *zero.p[c] = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *bits = __double_as_longlong(1.0);
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ng; g += grid_stride())
    group_bits[g] = __double_as_longlong(1.0);
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += grid_stride()) {
    const double p[3] = {x[3 * v], x[3 * v + 1], x[3 * v + 2]};
    const double d[3] = {dx[3 * v], dx[3 * v + 1], dx[3 * v + 2]};
    bool fine = true;
    double lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
      fine &= finite_bits(p[k]) && finite_bits(d[k]);
      const double e = p[k] + d[k];
      lo[k] = fmin(p[k], e);
      hi[k] = fmax(p[k], e);
    }
    if (!fine) raise_flag(st, EIPC_FLAG_NONFINITE);
    reinterpret_cast<double2*>(x4)[2 * v] = make_double2(p[0], p[1]);
    reinterpret_cast<double2*>(x4)[2 * v + 1] = make_double2(p[2], 0.0);
    reinterpret_cast<double2*>(dx4)[2 * v] = make_double2(d[0], d[1]);
    reinterpret_cast<double2*>(dx4)[2 * v + 1] = make_double2(d[2], 0.0);
    reinterpret_cast<float4*>(x4f)[v] = make_float4(to_float<0>(p[0]), to_float<0>(p[1]), to_float<0>(p[2]), 0.f);
    reinterpret_cast<float4*>(dx4f)[v] = make_float4(to_float<0>(d[0]), to_float<0>(d[1]), to_float<0>(d[2]), 0.f);
    store_box(vbox + 8 * v, lo, hi);
  }
}

__device__ __forceinline__ void decode_pair(const Topo& T, uint64_t key, int* type, int32_t v[4]) {
  const int32_t j = (int32_t)(key & ((1ull << T.bits_j) - 1));
  const int32_t i = (int32_t)((key >> T.bits_j) & ((1ull << T.bits_i) - 1));
  *type = (int)(key >> (T.bits_i + T.bits_j));
  if (*type == 0) {
    v[0] = i;
    v[1] = T.tris[3 * (int64_t)j]; v[2] = T.tris[3 * (int64_t)j + 1]; v[3] = T.tris[3 * (int64_t)j + 2];
  } else {
    // by single words: eipc_accd_toi_static's edges are the caller's, of any alignment
    v[0] = T.edges[2 * (int64_t)i]; v[1] = T.edges[2 * (int64_t)i + 1];
    v[2] = T.edges[2 * (int64_t)j]; v[3] = T.edges[2 * (int64_t)j + 1];
  }
}

// the exact closed swept-box overlap in FP64
__device__ __noinline__ bool swept_overlap_f64(const double* __restrict__ x4, const double* __restrict__ dx4, int na,
                                               const int32_t* v) {
  double lo[2][3], hi[2][3];
  for (int sd = 0; sd < 2; ++sd)
    for (int c = 0; c < 3; ++c) { lo[sd][c] = INFINITY; hi[sd][c] = -INFINITY; }
  for (int a = 0; a < 4; ++a) {
    const int sd = a < na ? 0 : 1;
    const V3 X = load_x(x4, v[a]), D = load_x(dx4, v[a]);
    const double p0[3] = {X.x, X.y, X.z};
    const double p1[3] = {X.x + D.x, X.y + D.y, X.z + D.z};
    for (int c = 0; c < 3; ++c) {
      lo[sd][c] = fmin(lo[sd][c], fmin(p0[c], p1[c]));
      hi[sd][c] = fmax(hi[sd][c], fmax(p0[c], p1[c]));
    }
  }
  bool ov = true;
  for (int c = 0; c < 3; ++c) ov &= !(lo[0][c] > hi[1][c] || lo[1][c] > hi[0][c]);
  return ov;
}

// Settles in FP32 the candidates it can, which is almost all of them, and lists the rest for
// k_ccd_advance.  Nothing here is decided by FP32 alone that FP64 could decide otherwise:
//  - the swept boxes overlap, or do not, by more than 8 u M (u = 2^-24, M the candidate's
//    largest position plus largest displacement; each FP32 bound is off by at most 2 u M), else
//    the FP64 boxes decide;
//  - the first advancement reaches t = 1 exactly when d0 >= L / (1 - s).  An upper bound of the
//    speeds (each FP32 speed is low by at most 16 u times the largest displacement) and the
//    conservative FP32 far tests of the contact screen, their radius grown by 80 u M for the
//    positions' rounding, prove d0 > L / (1 - s) at any motion size; a pair not proven far takes
//    the FP64 path.
// The FP64 boxes and speeds of every candidate used to cost about 130 FP64 instructions each (the
// pipe takes 64 cycles for a warp's one): 572 us of the 256-scene batch's 1.9 M candidates.
__global__ void __launch_bounds__(kBlock) k_ccd_screen(Topo T, const double* __restrict__ x4, const double* __restrict__ dx4,
                                                       const float* __restrict__ x4f, const float* __restrict__ dx4f,
                                                       const uint64_t* __restrict__ cand, const int64_t* n_cand, int64_t cap,
                                                       double s, uint64_t* __restrict__ list, int64_t* n_list, int64_t* n_adv) {
  pdl_entry();
  const int64_t n = clamp_count(n_cand, cap);
  const int lane = threadIdx.x & 31;
  const float inv_1s = __fdiv_ru(1.000001f, __double2float_rd(1.0 - s));
  const float u = 5.9604645e-8f;
  int counted = 0;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < n; base += grid_stride()) {
    const int64_t k = base + threadIdx.x;
    bool open = false;
    uint64_t key = 0;
    if (k < n) {
      key = cand[k];
      int type;
      int32_t v[4];
      decode_pair(T, key, &type, v);
      const int na = type == 0 ? 1 : 2;
      F3 P[4], Q[4];
      float Mx = 0.f, Md = 0.f;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        P[a] = load_xf(x4f, v[a]);
        Q[a] = load_xf(dx4f, v[a]);
        Mx = fmaxf(Mx, fmax_abs(P[a]));
        Md = fmaxf(Md, fmax_abs(Q[a]));
      }
      // smallest room between the boxes of the two sides over the axes
      float room = INFINITY;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float lo[2] = {INFINITY, INFINITY}, hi[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float p = c == 0 ? P[a].x : (c == 1 ? P[a].y : P[a].z);
          const float e = p + (c == 0 ? Q[a].x : (c == 1 ? Q[a].y : Q[a].z));
          const int sd = a == 0 ? 0 : (a == 1 && na == 2 ? 0 : 1);
          if (sd == 0) { lo[0] = fminf(lo[0], fminf(p, e)); hi[0] = fmaxf(hi[0], fmaxf(p, e)); }
          else { lo[1] = fminf(lo[1], fminf(p, e)); hi[1] = fmaxf(hi[1], fmaxf(p, e)); }
        }
        room = fminf(room, fminf(hi[1] - lo[0], hi[0] - lo[1]));
      }
      const float tol = 8.f * u * (Mx + Md);
      bool ov = room >= tol;
      if (!ov && !(room < -tol)) ov = swept_overlap_f64(x4, dx4, na, v);
      if (ov) {
        ++counted;
        const F3 mean = F3{0.25f * (Q[0].x + Q[1].x + Q[2].x + Q[3].x), 0.25f * (Q[0].y + Q[1].y + Q[2].y + Q[3].y),
                           0.25f * (Q[0].z + Q[1].z + Q[2].z + Q[3].z)};
        float la = 0.f, lb = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const F3 R = Q[a] - mean;
          const float sp = sqrtf(fdot(R, R));
          if (a == 0 || (a == 1 && na == 2)) la = fmaxf(la, sp);
          else lb = fmaxf(lb, sp);
        }
        const float L = (la + lb) * 1.000002f + 64.f * u * Md;
        const float r = L * inv_1s + 80.f * Mx * u;
        const float r2m = r * r * 1.004f;
        open = !(type == 0 ? pt_far_f32(P[0], P[1], P[2], P[3], r2m) : ee_far_f32(P[0], P[1], P[2], P[3], r2m));
      }
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, open);
    if (mask) {
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(n_list), (unsigned long long)__popc(mask));
      b = __shfl_sync(0xffffffffu, b, 0);
      // listed candidates never outnumber the candidates, so the position is below the capacity
      if (open) list[(int64_t)b + __popc(mask & ((1u << lane) - 1u))] = key;
    }
  }
  counted = __reduce_add_sync(0xffffffffu, counted);
  if (lane == 0 && counted) atomicAdd(reinterpret_cast<unsigned long long*>(n_adv), (unsigned long long)counted);
}

// Conservative advancement of the listed candidates in FP64.  Each step costs about 50 FP64
// instructions: the closest feature is chosen in FP32 (closest_hint, from the FP32 positions at
// the same t) and only its distance is taken in FP64.  A warp claims `tile` candidates at a
// time from a queue -- the first claim is its own.  A list shorter than the warps' first claims is
// taken by items_per_warp.
__global__ void __launch_bounds__(kAccdThreads) k_ccd_advance(Topo T, const double* __restrict__ x4,
                                                              const double* __restrict__ dx4, const float* __restrict__ x4f,
                                                              const float* __restrict__ dx4f,
                                                              const uint64_t* __restrict__ list, const int64_t* n_list,
                                                              double s, int max_iter, unsigned long long* alpha_bits,
                                                              unsigned long long* group_bits, DevStatus* st, int64_t* queue,
                                                              int tile_req) {
  pdl_entry();
  const int64_t n = *n_list;
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int tile = tile_req >= 32 ? (tile_req & ~31) : 32;
  if (n < warps * tile) tile = items_per_warp(n, 4);
  int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * tile;
  // every claim takes `tile` candidates, so n / tile + 2 claims cover all a warp can make
  const int64_t max_rounds = n / tile + 2;
  for (int64_t round = 0; base < n; ++round) {
    if (round > max_rounds) {
      raise_flag(st, EIPC_FLAG_STACK_OVERFLOW);
      break;
    }
    for (int o = 0; o < tile; o += 32) {
      const int64_t k = base + o + lane;
      int iters = 0;
      if (k < n && lane < tile) {
        int type;
        int32_t v[4];
        decode_pair(T, list[k], &type, v);
        const int na = type == 0 ? 1 : 2;
        V3 X[4], R[4];
        F3 Xf[4], Rf[4];
        float M = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          X[a] = load_x(x4, v[a]);
          R[a] = load_x(dx4, v[a]);
          Xf[a] = load_xf(x4f, v[a]);
          Rf[a] = load_xf(dx4f, v[a]);
          M = fmaxf(M, fmax_abs(Xf[a]) + fmax_abs(Rf[a]));
        }
        const V3 mean = (R[0] + R[1] + R[2] + R[3]) * 0.25;
        const F3 mf = F3{0.25f * (Rf[0].x + Rf[1].x + Rf[2].x + Rf[3].x), 0.25f * (Rf[0].y + Rf[1].y + Rf[2].y + Rf[3].y),
                         0.25f * (Rf[0].z + Rf[1].z + Rf[2].z + Rf[3].z)};
        double la = 0.0, lb = 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          R[a] = R[a] - mean;
          Rf[a] = Rf[a] - mf;
          const double sp = dot(R[a], R[a]);
          if (a == 0 || (a == 1 && na == 2)) la = fmax(la, sp);
          else lb = fmax(lb, sp);
        }
        const double L = sqrt(la) + sqrt(lb);
        // FP32 positions at t: the copies' rounding (u M), the displacements' (8 u M) and the sum's
        const float ec = 12.f * 5.9604645e-8f * M;
        double t = 1.0;
        if (L > 0.0) {
          const double d20 = closest_pair<false>(type, X, closest_hint(type, Xf[0], Xf[1], Xf[2], Xf[3], ec), nullptr);
          if (!(d20 > 0.0)) {
            raise_flag(st, EIPC_FLAG_PENETRATION);
            t = 0.0;
          } else {
            const double cl = (1.0 - s) / L;
            double d = sqrt(d20);
            const double stop = s * d;
            t = 0.0;
            while (true) {
              const double tn = fma(d, cl, t);
              if (!lt_nonneg(tn, 1.0)) { t = 1.0; break; }
              t = tn;
              const float tf = to_float<0>(t);
              V3 Pt[4];
              F3 Pf[4];
#pragma unroll
              for (int a = 0; a < 4; ++a) {
                Pt[a] = X[a] + R[a] * t;
                Pf[a] = F3{Xf[a].x + Rf[a].x * tf, Xf[a].y + Rf[a].y * tf, Xf[a].z + Rf[a].z * tf};
              }
              d = sqrt(closest_pair<false>(type, Pt, closest_hint(type, Pf[0], Pf[1], Pf[2], Pf[3], ec), nullptr));
              ++iters;
              if (!lt_nonneg(stop, d)) break;
              if (iters >= max_iter) { raise_flag(st, EIPC_FLAG_ACCD_CAP); break; }
            }
          }
        }
        if (t < 1.0) {
          // exact minimum, scene (of a batch) and whole; the plain read only saves atomics
          const unsigned long long tb = (unsigned long long)__double_as_longlong(t * kMargin);
          if (group_bits) {
            unsigned long long* gb = group_bits + T.vgroup[v[0]];
            if (tb < __ldcg(gb)) atomicMin(gb, tb);
          }
          if (tb < __ldcg(alpha_bits)) atomicMin(alpha_bits, tb);
        }
      }
      const int tot = __reduce_add_sync(0xffffffffu, iters);
      if (lane == 0 && tot) atomicAdd(&st->accd_iters, (unsigned long long)tot);
    }
    unsigned long long b = 0;
    if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(queue), (unsigned long long)tile);
    base = (int64_t)__shfl_sync(0xffffffffu, b, 0) + warps * tile;
  }
}

__global__ void k_alpha_out(const unsigned long long* bits, double* alpha, const int64_t* n_adv, int64_t* n_out) {
  pdl_entry();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    *alpha = __longlong_as_double((long long)*bits);
    if (n_out) *n_out = *n_adv;
  }
}

}  // namespace

void ccd_bound_launch(const CcdBound& b, cudaStream_t s) {
  launch(k_ccd_screen, blocks_for(b.cap, 8), kBlock, 0, s, b.topo, b.x4, b.dx4, b.x4f, b.dx4f, b.cand, b.n_cand, b.cap, b.s, b.list,
         b.n_list, b.n_adv);
  launch(k_ccd_advance, blocks_for(b.cap, 8, kAccdThreads), kAccdThreads, 0, s, b.topo, b.x4, b.dx4, b.x4f, b.dx4f,
         static_cast<const uint64_t*>(b.list), static_cast<const int64_t*>(b.n_list), b.s, b.max_iter, b.alpha_bits, b.group_bits,
         b.status, b.queue, b.tile);
}

void accd_launch(eipc_scene* sc, const double* x, const double* dx, const eipc_params& p, double* alpha,
                 int64_t* n_candidates, cudaStream_t s) {
  int64_t* n_cand = sc->counters + kCntCand;
  int64_t* n_adv = sc->counters + kCntAccd;
  int64_t* n_list = sc->counters + kCntCcdList;
  unsigned long long* abits = reinterpret_cast<unsigned long long*>(sc->counters + 12);
  int64_t* queue = sc->counters + kCntCcdQueue;
  // swept per-vertex boxes over [x, x + dx]; the hierarchies of the last contact-set build
  // are refitted with them when they exist (the topology is reused; only the boxes change)
  EIPC_TIMED(sc, kKEmbed, s,
             (launch(k_ccd_begin, blocks_for(sc->nv > sc->n_groups ? sc->nv : sc->n_groups), kBlock, 0, s, x, dx, sc->nv, sc->x4,
                     sc->dx4, sc->x4f, sc->dx4f, sc->vbox, sc->status, CounterList{{n_cand, n_adv, queue, n_list}}, abits,
                     sc->group_alpha_bits, sc->n_groups)));
  if (sc->broad.built) EIPC_TIMED(sc, kKBvh, s, bvh_refit(sc->broad, sc->vbox, s));
  else EIPC_TIMED(sc, kKBvh, s, bvh_build(sc->broad, sc->topo, sc->vbox, sc->sort_hist, s));
  EIPC_TIMED(sc, kKQuery, s,
             bvh_query(sc->broad, sc->topo, sc->vbox, sc->cand, n_cand, sc->cand_cap, sc->status, s,
                       sc->tune.query_threads, sc->tune.query_bps));
  // cand2 is free here (the contact search's screened list)
  sc->timers->start(kKCa, s);
  ccd_bound_launch(CcdBound{sc->topo, sc->x4, sc->dx4, sc->x4f, sc->dx4f, sc->cand, n_cand, sc->cand_cap, sc->cand2, n_list, n_adv,
                            queue, p.accd_s, p.accd_max_iter, abits, sc->group_alpha_bits, sc->status, sc->tune.ccd_tile},
                   s);
  sc->timers->stop(kKCa, s);
  launch(k_alpha_out, 1, 32, 0, s, abits, alpha, n_adv, n_candidates);
}

}  // namespace eipc
