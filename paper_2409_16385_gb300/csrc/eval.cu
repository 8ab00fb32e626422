// Per-pair contact potentials and their reduction into the subspace.
//
// Barrier (Eq. 7): E_k = kappa b(d), b = -(d - dhat)^2 log(d / dhat).
// With s = d^2 the partial minimum min_beta |r(x,beta)|^2 (geometry.cuh):
//   grad s   = 2 c (x) r
//   hess s   = 2 (c c^T) (x) I3 - G M^-1 G^T,  G_j = 2 (c (x) v_j + a_j (x) r),
//              v_j = sum_a a_j[a] x_a, M = 2 [v_j . v_l]
// (Schur complement of the inner minimisation), so
//   hess E = kappa [(b'' - b'/d) (c c^T) (x) (r^ r^T) + (b'/d) (c c^T) (x) I3]
//            - (kappa b' / (2d)) G M^-1 G^T.
// Every term lies in the span of {c^ (x) e_x, c^ (x) e_y, c^ (x) e_z, a^_1 (x) r^, a^_2 (x) r^}
// (a^_j: a_j orthonormalised against c), an orthonormal basis of at most 5 columns, so projecting
// the 12x12 Hessian onto the PSD cone (projected Newton, Sec. III-C) is projecting a matrix of at
// most 5x5: P+ acts on eigenpairs and the complement of the span is the zero eigenspace.  That
// projection is closed form: its one or two negative eigenvectors are roots of small secular
// equations, and what is left has rank two or three, P+ = sum_k z_k z_k^T (see "pair factors").
//
// Reduction (Eq. 17): g_r = J^T g, H_r = J^T H J.  J restricted to a stencil maps the
// stencil's unique cage nodes I to the 4 vertices with weights w_aI, so an item leaves one row of
// factors per node, z_kI with the scalars omega_I = sum_a c_a w_aI, and block(I, J) = sum_k z_kI
// z_kJ^T.
// Friction (Sec. III-B, lagged): D = mu lambda f0(|u|), u = (I - n n^T)(sum gamma_a x_a - anchor),
//   grad = mu lambda f1(y)/y gamma (x) u,   hess = (gamma gamma^T) (x) F,
//   F = mu lambda [(f1/y)(I - n n^T) + (f1' - f1/y) u^ u^T]   (PSD as written).
// Records: items with the same nodes form a group, in the order of a stable sort by node set, and
// a group is cut into chunks of 16 items from its own start; a record is one upper block of one
// chunk, multiplied out of its items' rows in their order (k_chunk_sums).  The records are stably
// sorted by block (key: its position in the upper triangle), and a block is the sum of its records
// by three interleaved chains that start at its first one (k_segment_sums).  Groups, chunks and
// chains depend on the scene's own items alone, so a result is bitwise repeatable and the same for
// a scene alone or inside a batch.
#include "geometry.cuh"
#include "scene.cuh"
#include "sort.cuh"

namespace eipc {
namespace {

constexpr int kMaxNodes = 16;
constexpr int kEvalThreads = 128;
constexpr int kRecCheckThreads = 512;

// Key of the upper block (I, J), I <= J < ns: its row-major position in the upper triangle,
// I ns - I (I - 1) / 2 + (J - I).  Ordered like (I, J), and below ns (ns + 1) / 2, so the
// record sort covers fewer bits than with I ns + J (24 instead of 25 for 5,664 nodes).
__host__ __device__ __forceinline__ uint64_t upper_key(uint64_t I, uint64_t J, uint64_t ns) {
  return I * ns - I * (I - 1) / 2 + (J - I);
}

// (I, J) of an upper key: I is the last row whose first key is at most the key; an FP64
// estimate from the quadratic, then exact integer correction
__device__ __forceinline__ void upper_decode(uint64_t key, uint64_t ns, uint64_t* I, uint64_t* J) {
  const double b = 2.0 * (double)ns + 1.0;
  double r = 0.5 * (b - sqrt(fmax(b * b - 8.0 * (double)key, 0.0)));
  int64_t i = (int64_t)r;
  if (i < 0) i = 0;
  if (i > (int64_t)ns - 1) i = (int64_t)ns - 1;
  while (i > 0 && upper_key((uint64_t)i, (uint64_t)i, ns) > key) --i;
  while (i + 1 < (int64_t)ns && upper_key((uint64_t)(i + 1), (uint64_t)(i + 1), ns) <= key) ++i;
  *I = (uint64_t)i;
  *J = key - upper_key((uint64_t)i, (uint64_t)i, ns) + (uint64_t)i;
}

// node I of a diagonal key (I, I): I ns - I (I - 1) / 2 = key, by bisection
__device__ __forceinline__ int64_t diagonal_node(uint64_t key, uint64_t ns) {
  uint64_t lo = 0, hi = ns - 1;
  while (lo < hi) {
    const uint64_t mid = (lo + hi + 1) >> 1;
    if (upper_key(mid, mid, ns) <= key) lo = mid;
    else hi = mid - 1;
  }
  return (int64_t)lo;
}

// stencil vertex ids of pair (type, i, j)
__device__ __forceinline__ void stencil_vertices(const Topo& T, int type, int32_t i, int32_t j, int32_t v[4]) {
  if (type == 0) {
    v[0] = i;
    v[1] = T.tris[3 * (int64_t)j]; v[2] = T.tris[3 * (int64_t)j + 1]; v[3] = T.tris[3 * (int64_t)j + 2];
  } else {
    v[0] = T.edges[2 * (int64_t)i]; v[1] = T.edges[2 * (int64_t)i + 1];
    v[2] = T.edges[2 * (int64_t)j]; v[3] = T.edges[2 * (int64_t)j + 1];
  }
}

// item k < P: barrier pair k; P <= k < P + L: friction pair k - P
__device__ __forceinline__ bool item_vertices(const Topo& T, const eipc_pairs& pr, int64_t P, const int32_t* lag_v,
                                              int64_t L, int64_t k, int32_t v[4]) {
  if (k < P) {
    stencil_vertices(T, pr.type[k], pr.i[k], pr.j[k], v);
    return true;
  }
  if (k < P + L) {
    const int4 q = reinterpret_cast<const int4*>(lag_v)[k - P];
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    return true;
  }
  return false;
}

// Friction merged into contact pairs with the same stencil: for pair k,
// fric_of_pair[k] = INT32_MAX - f when lagged friction item f takes k's records (0: none);
// pair_of_fric[f] = that pair + 1 (0: none).  The claim holds only if both agree.
// friction item f rides on pair kp's records (both arrays as in EvalArgs)
__device__ __forceinline__ bool friction_merged(const int32_t* __restrict__ fric_of_pair,
                                                const int32_t* __restrict__ pair_of_fric, int64_t f) {
  if (!pair_of_fric) return false;
  const int32_t kp = pair_of_fric[f] - 1;
  return kp >= 0 && fric_of_pair[kp] == INT32_MAX - (int32_t)f;
}

// (type, i, j) of a pair as one ordered 64-bit key (i, j < 2^31)
__device__ __forceinline__ uint64_t lag_pair_key(int type, int32_t i, int32_t j) {
  return ((uint64_t)(type & 1) << 62) | ((uint64_t)(uint32_t)i << 31) | (uint64_t)(uint32_t)j;
}

// first pair position k in [0, P) with (type[k], i[k]) >= (type, i) (the pair list is in
// (type, i, j) order)
__device__ __forceinline__ int64_t pair_lower_bound(const eipc_pairs& pr, int64_t P, int type, int32_t i) {
  int64_t lo = 0, hi = P;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    const int t = pr.type[mid];
    if (t < type || (t == type && pr.i[mid] < i)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Friction items that ride on a contact pair: lagged item f and pair k share their records
// when their stencils have the same four vertices in the same order (then the same cage
// nodes in the same order, so the same record keys).  The candidates are the PT pairs of
// vertex v0 and the EE pairs of edge (v0, v1).  When several items find the same pair (a
// lag list with repeated stencils), the lowest f wins; the others keep their own records.
__global__ void __launch_bounds__(kBlock) k_fric_match(Topo T, eipc_pairs pr, eipc_lag lag, int64_t item_cap,
                                                       const uint64_t* __restrict__ ekey,
                                                       const int32_t* __restrict__ eid,
                                                       const uint64_t* __restrict__ lag_key,
                                                       int32_t* __restrict__ fric_of_pair,
                                                       int32_t* __restrict__ pair_of_fric) {
  pdl_entry();
  int64_t P = clamp_count(pr.count, pr.capacity);
  if (P > item_cap) P = item_cap;
  int64_t L = clamp_count(lag.count, lag.capacity);
  if (P + L > item_cap) L = item_cap - P;
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < L; f += grid_stride()) {
    const int4 q = reinterpret_cast<const int4*>(lag.v)[f];
    int64_t found = -1;
    if (lag_key) {
      // the item's own pair key (type, i, j), recorded when the scene built this lag state:
      // one search in the pair list's order, then the same check of the four vertices
      const uint64_t key = lag_key[f];
      int64_t lo = 0, hi = P;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (lag_pair_key(pr.type[mid], pr.i[mid], pr.j[mid]) < key) lo = mid + 1;
        else hi = mid;
      }
      if (lo < P && lag_pair_key(pr.type[lo], pr.i[lo], pr.j[lo]) == key) {
        int32_t v[4];
        stencil_vertices(T, pr.type[lo], pr.i[lo], pr.j[lo], v);
        if (v[0] == q.x && v[1] == q.y && v[2] == q.z && v[3] == q.w) found = lo;
      }
      pair_of_fric[f] = (int32_t)(found + 1);
      if (found >= 0) atomicMax(fric_of_pair + found, INT32_MAX - (int32_t)f);
      continue;
    }
    for (int64_t k = pair_lower_bound(pr, P, 0, q.x); k < P && found < 0; ++k) {
      if (pr.type[k] != 0 || pr.i[k] != q.x) break;
      const int64_t j = pr.j[k];
      if (T.tris[3 * j] == q.y && T.tris[3 * j + 1] == q.z && T.tris[3 * j + 2] == q.w) found = k;
    }
    if (found < 0) {
      const int32_t e = edge_id_of(q.x, q.y, T.nv, ekey, eid, T.ne);
      if (e >= 0 && T.edges[2 * (int64_t)e] == q.x) {
        for (int64_t k = pair_lower_bound(pr, P, 1, e); k < P && found < 0; ++k) {
          if (pr.type[k] != 1 || pr.i[k] != e) break;
          const int64_t j = pr.j[k];
          if (T.edges[2 * j] == q.z && T.edges[2 * j + 1] == q.w) found = k;
        }
      }
    }
    pair_of_fric[f] = (int32_t)(found + 1);
    if (found >= 0) atomicMax(fric_of_pair + found, INT32_MAX - (int32_t)f);
  }
}

// Unique cage nodes of each item in ascending order (kinematic vertices carry none), the node of
// every (vertex, slot), record counts, and the key that brings items with the same nodes together:
// the first node above a hash of the others' offsets from it.  Offsets, not ids, so that a
// scene's items order alike alone and inside a batch, where its ids are shifted.  Items without
// nodes get a key above all.
// Too few bits and different sets with one key take turns in the order, each turn a group; a bit more
// costs nothing until the sort takes a pass more.  The full grasp, with about ten sets per first
// node, takes 618 us an evaluation with 5 bits, 587 with 7, 583 with 10; the plate in rack 178, 181 and
// 180, the 256-scene batch's stage 4,642, 4,634 and 4,636.
constexpr int kHashBits = 7;

__global__ void __launch_bounds__(kBlock) k_item_nodes(Topo T, eipc_pairs pr, const int32_t* lag_v,
                                                       const int64_t* lag_count, int64_t lag_cap,
                                                       const int32_t* __restrict__ cage_idx, int64_t item_cap,
                                                       int32_t* __restrict__ item_nodes, int32_t* __restrict__ item_n,
                                                       int32_t* __restrict__ item_group, const int32_t* __restrict__ vgroup,
                                                       int64_t* __restrict__ rc_h, int64_t* __restrict__ rc_g,
                                                       int64_t* n_items, DevStatus* st,
                                                       const int32_t* __restrict__ fric_of_pair,
                                                       const int32_t* __restrict__ pair_of_fric,
                                                       uint64_t* __restrict__ item_map, int key_bits,
                                                       uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  pdl_entry();
  const int64_t P = clamp_count(pr.count, pr.capacity);
  const int64_t L = lag_v ? clamp_count(lag_count, lag_cap) : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int64_t n = P + L;
    if (n > item_cap) {
      raise_flag(st, EIPC_FLAG_REC_OVERFLOW);
      n = item_cap;
    }
    *n_items = n;
  }
  const int64_t n = (P + L) < item_cap ? (P + L) : item_cap;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += grid_stride()) {
    int32_t v[4];
    item_vertices(T, pr, P, lag_v, L, k, v);
    item_group[k] = vgroup[v[0]];
    vals[k] = (uint32_t)k;
    int32_t nodes[kMaxNodes];
    int cnt = 0;
    uint64_t map = 0;              // nibble 4a + s: which of the item's nodes is slot s of vertex a
    // a merged friction item is evaluated in its contact pair's records
    if (k < P || !friction_merged(fric_of_pair, pair_of_fric, k - P)) {
      for (int a = 0; a < 4; ++a) {
        const int4 id = __ldg(reinterpret_cast<const int4*>(cage_idx) + v[a]);
        if (id.x < 0) continue;
        const int32_t ids[4] = {id.x, id.y, id.z, id.w};
        for (int s = 0; s < 4; ++s) {
          int at = cnt;
          for (int u = 0; u < cnt; ++u)
            if (nodes[u] == ids[s]) at = u;
          if (at == cnt) nodes[cnt++] = ids[s];
          map |= (uint64_t)at << (4 * (4 * a + s));
        }
      }
    }
    item_n[k] = cnt;
    rc_h[k] = (int64_t)cnt * (cnt + 1) / 2;
    rc_g[k] = cnt;
    if (cnt == 0) {
      keys[k] = (1ull << key_bits) - 1;
      continue;
    }
    uint64_t rank = 0;             // nibble u: place of nodes[u] in ascending order
    int32_t first = nodes[0];
    for (int u = 0; u < cnt; ++u) {
      int r = 0;
      for (int w = 0; w < cnt; ++w) r += nodes[w] < nodes[u];
      rank |= (uint64_t)r << (4 * u);
      item_nodes[kMaxNodes * k + r] = nodes[u];
      first = min(first, nodes[u]);
    }
    uint32_t h = (uint32_t)cnt;    // order-free over the nodes: a sum of mixed offsets
    for (int u = 0; u < cnt; ++u) {
      uint32_t x = (uint32_t)(nodes[u] - first) * 0x9e3779b1u;
      x = (x ^ (x >> 15)) * 0x85ebca6bu;
      h += x ^ (x >> 13);
    }
    h = (h ^ (h >> 16)) * 0xc2b2ae35u;
    keys[k] = (uint64_t)(uint32_t)first << kHashBits | (h >> (32 - kHashBits));
    uint64_t sorted_map = 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) sorted_map |= (rank >> (4 * ((map >> (4 * q)) & 15u)) & 15ull) << (4 * q);
    item_map[k] = sorted_map;
  }
}

struct EvalArgs {
  Topo T;
  eipc_pairs pr;
  const int32_t* cage_idx;
  const double* w;
  const double* x4;
  int64_t ns;
  double dhat, kappa;
  const int32_t* item_nodes;
  const int32_t* item_n;
  const int64_t* ro_h;
  const int64_t* ro_g;
  const int64_t* n_items;
  int64_t rec_cap, gcap;
  double* hrec;            // explicit records (mollified pairs)
  double* frow;            // factor rows, kFRow doubles per (item, node) at ro_g[item] + node
  double* ihead;           // item headers, kIHead doubles per item
  const uint64_t* item_map;
  const float* x4f;
  double inv_dhat;
  double* item_E;
  DevStatus* st;
  bool project;            // PSD-project the barrier Hessians (projected Newton)
  const double* moll_r2;   // EE mollifier: rest squared edge lengths (null: off)
  double moll_factor;      // eps_x = moll_factor |e_i|^2 |e_j|^2
  uint32_t* moll_list;     // mollified pairs found by the factor kernel, their number
  int64_t* n_moll;
  uint32_t* rest;          // items k_eval_factors leaves to k_eval_rest: pairs from the front, friction
                           // items from the back of item_cap entries
  int64_t* n_rest;         // [2] their numbers
  int64_t item_cap;
  int64_t* queue;          // next unclaimed item (work queue)
  int tile;                // items a warp claims from the queue at a time (multiple of 32)
  // friction merged into contact pairs (friction_merged; null: no merging); lag, mu and
  // eps_f are the friction parameters
  const int32_t* fric_of_pair;
  const int32_t* pair_of_fric;
  eipc_lag lag;
  double mu, eps_f;
};

// Lagged friction of item f at the current positions (Sec. III-B, Eq. 8-9): energy
// mu lambda f0(|u|), the gradient scale mu lambda f1(y)/y along u, the symmetric 3 x 3
// F = mu lambda (f1(y)/y (I - n n^T) + (f1'(y) - f1(y)/y) u u^T / y^2), and the per-node
// weights of gamma for the item's cage nodes.
struct FrictionTerms {
  double E, gs;
  double u[3];
  double F[3][3];
};

__device__ __forceinline__ void friction_terms(const double* __restrict__ x4, const eipc_lag& lag, int64_t f,
                                               const int32_t v[4], double mu, double eps, FrictionTerms& R,
                                               double gam[4]) {
  for (int a = 0; a < 4; ++a) gam[a] = lag.gamma[4 * f + a];
  const V3 nrm = {lag.n[3 * f], lag.n[3 * f + 1], lag.n[3 * f + 2]};
  const V3 anc = {lag.anchor[3 * f], lag.anchor[3 * f + 1], lag.anchor[3 * f + 2]};
  const double ml = mu * lag.lambda[f];
  V3 vs = {0.0, 0.0, 0.0};
  for (int a = 0; a < 4; ++a) vs = vs + load_x(x4, v[a]) * gam[a];
  vs = vs - anc;
  const V3 u = vs - nrm * dot(nrm, vs);
  const double y2 = dot(u, u);
  // f0(y), f1(y)/y and (f1'(y) - f1(y)/y) / y^2, with one reciprocal square root
  const double ie = 1.0 / eps;
  double f0 = eps / 3.0, f1y = 2.0 * ie, c2 = 0.0;
  if (is_pos(y2)) {
    const double iy = rsqrt(y2), y = y2 * iy;
    if (lt_nonneg(y, eps)) {
      const double yie2 = y * ie * ie;
      f0 = fma(y2, ie - yie2 * (1.0 / 3.0), f0);  // -y^3 / (3 eps^2) + y^2 / eps + eps / 3
      f1y -= yie2;
      c2 = -ie * ie * iy;                         // ((2/eps - 2y/eps^2) - (2/eps - y/eps^2)) / y^2
    } else {
      f0 = y; f1y = iy; c2 = -iy * iy * iy;
    }
  }
  R.E = ml * f0;
  R.gs = ml * f1y;
  R.u[0] = u.x; R.u[1] = u.y; R.u[2] = u.z;
  const double nn[3] = {nrm.x, nrm.y, nrm.z};
  const double mc = ml * c2;
  double mn[3], mu_[3];
#pragma unroll
  for (int p = 0; p < 3; ++p) { mn[p] = R.gs * nn[p]; mu_[p] = mc * R.u[p]; }
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = p; q < 3; ++q) {
      const double s = fma(mu_[p], R.u[q], fma(-mn[p], nn[q], p == q ? R.gs : 0.0));
      R.F[p][q] = s;
      R.F[q][p] = s;
    }
}

// Explicit records (mollified pairs): record pos of the item holds its upper block, of nodes
// (min, max), as nine values in rows of kHRecStride; a diagonal one the block's upper entries
// B00 B01 B02 B11 B12 B22 and then the item's gradient at that node.
__device__ __forceinline__ void emit_upper(const EvalArgs& A, int64_t pos, int32_t Iu, int32_t Iv, const double B[3][3]) {
  const bool swap = Iu > Iv;
  double v[9];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) v[3 * a + b] = swap ? B[b][a] : B[a][b];
  double2* p = reinterpret_cast<double2*>(A.hrec + kHRecStride * pos);
#pragma unroll
  for (int c = 0; c < 4; ++c) p[c] = make_double2(v[2 * c], v[2 * c + 1]);
  A.hrec[kHRecStride * pos + 8] = v[8];
}

__device__ __forceinline__ void emit_diag(const EvalArgs& A, int64_t pos, const double B[3][3], double g0, double g1,
                                          double g2) {
  double2* p = reinterpret_cast<double2*>(A.hrec + kHRecStride * pos);
  p[0] = make_double2(B[0][0], B[0][1]);
  p[1] = make_double2(B[0][2], B[1][1]);
  p[2] = make_double2(B[1][2], B[2][2]);
  p[3] = make_double2(g0, g1);
  A.hrec[kHRecStride * pos + 8] = g2;
}

// The barrier Hessian of one active pair in its span (Sec. III-B, Eq. 7; the 12 x 12
// Hessian of kappa b(d(x)) lies in the span of c^ (x) e_xyz and a^_j (x) r^): the
// orthonormal 4-vectors basis[0] = c^, basis[1..2] = a^_1, a^_2, the unit direction r^
// between the closest points, and the 5 x 5 matrix K of the Hessian in that basis,
// unprojected and symmetric.  Also the energy kappa b(d) and b'(d).
struct BarrierSpan {
  double E, b1, cn;
  V3 rh;
  double basis[3][4];
  double K[5][5];
};

__device__ __forceinline__ void barrier_span(const V3 Y[4], const Stencil& S, double d, double dhat, double kappa,
                                             BarrierSpan& B) {
  const double lg = log(d / dhat);
  const double m = d - dhat;
  const double inv_d = 1.0 / d;
  const double md = m * inv_d;
  const double b = -m * m * lg;
  const double b1 = -2.0 * m * lg - m * md;
  const double b2 = -2.0 * lg - 4.0 * md + md * md;
  B.E = kappa * b;
  B.b1 = b1;
  // r and r^
  V3 r = {0.0, 0.0, 0.0};
  for (int a = 0; a < 4; ++a) r = r + Y[a] * S.c[a];
  B.rh = r * rsqrt(dot(r, r));
  const V3 rh = B.rh;
  // orthonormal 4-vectors c^, a^_1, a^_2
  const double cc = S.c[0] * S.c[0] + S.c[1] * S.c[1] + S.c[2] * S.c[2] + S.c[3] * S.c[3];
  const double inv_cn = rsqrt(cc);
  const double cn = cc * inv_cn;
  B.cn = cn;
  for (int a = 0; a < 4; ++a) B.basis[0][a] = S.c[a] * inv_cn;
  for (int j = 0; j < 2; ++j) {
    if (j < S.m) {
      double t[4];
      for (int a = 0; a < 4; ++a) t[a] = S.a[j][a];
      for (int i = 0; i <= j; ++i) {
        double pr = 0.0;
        for (int a = 0; a < 4; ++a) pr += B.basis[i][a] * t[a];
        for (int a = 0; a < 4; ++a) t[a] -= pr * B.basis[i][a];
      }
      const double inv_tn = rsqrt(t[0] * t[0] + t[1] * t[1] + t[2] * t[2] + t[3] * t[3]);
      for (int a = 0; a < 4; ++a) B.basis[1 + j][a] = t[a] * inv_tn;
    } else {
      for (int a = 0; a < 4; ++a) B.basis[1 + j][a] = 0.0;
    }
  }
  // v_j, M = 2 [v_j . v_l], g_j = Q^T G_j
  V3 vj[2];
  for (int j = 0; j < 2; ++j) {
    vj[j] = {0.0, 0.0, 0.0};
    for (int a = 0; a < 4; ++a) vj[j] = vj[j] + Y[a] * S.a[j][a];
  }
  double (&K)[5][5] = B.K;
  const double kb = kappa * cn * cn;
  const double rr = kappa * (b2 - b1 * inv_d);
  const double kd = kb * b1 * inv_d;
  const double rhv[3] = {rh.x, rh.y, rh.z};
  for (int p = 0; p < 3; ++p)
    for (int q = 0; q < 3; ++q) K[p][q] = cn * cn * (rr * rhv[p] * rhv[q]) + (p == q ? kd : 0.0);
  for (int p = 0; p < 5; ++p)
    for (int q = 3; q < 5; ++q) { K[p][q] = 0.0; K[q][p] = 0.0; }
  if (S.m > 0) {
    double g[2][5];
    for (int j = 0; j < S.m; ++j) {
      double ca = 0.0;
      for (int a = 0; a < 4; ++a) ca += B.basis[0][a] * S.a[j][a];
      const double vv[3] = {vj[j].x, vj[j].y, vj[j].z};
      for (int p = 0; p < 3; ++p) g[j][p] = 2.0 * cn * vv[p] + 2.0 * d * ca * rhv[p];
      for (int l = 0; l < 2; ++l) {
        double al = 0.0;
        for (int a = 0; a < 4; ++a) al += B.basis[1 + l][a] * S.a[j][a];
        g[j][3 + l] = 2.0 * d * al;
      }
    }
    double Mi[2][2];
    if (S.m == 1) {
      Mi[0][0] = 0.5 / dot(vj[0], vj[0]);
    } else {
      const double m00 = 2.0 * dot(vj[0], vj[0]), m01 = 2.0 * dot(vj[0], vj[1]), m11 = 2.0 * dot(vj[1], vj[1]);
      const double inv_det = 1.0 / (m00 * m11 - m01 * m01);
      Mi[0][0] = m11 * inv_det; Mi[1][1] = m00 * inv_det; Mi[0][1] = Mi[1][0] = -m01 * inv_det;
    }
    const double beta = -0.5 * kappa * b1 * inv_d;
    for (int p = 0; p < 5; ++p)
      for (int q = 0; q < 5; ++q) {
        double s2 = 0.0;
        for (int j = 0; j < S.m; ++j)
          for (int l = 0; l < S.m; ++l) s2 += g[j][p] * Mi[j][l] * g[l][q];
        K[p][q] += beta * s2;
      }
  }
  // symmetrise against rounding
  for (int p = 0; p < 5; ++p)
    for (int q = p + 1; q < 5; ++q) { const double t = 0.5 * (K[p][q] + K[q][p]); K[p][q] = t; K[q][p] = t; }
}

// ------------------------------------------------------------------ EE mollifier
// IPC-style variant (the paper applies none): an edge-edge pair whose edges are nearly
// parallel, c = |e_i x e_j|^2 < eps_x = factor |e_i^rest|^2 |e_j^rest|^2, carries
// kappa m(c) b(d) with m(c) = c (2 / eps - c / eps^2), which is C1 at c = eps and vanishes
// as the edges become parallel.  Its Hessian leaves the 5-dimensional span, so these rare
// pairs take a full 12 x 12 path (exact Hessian; Jacobi projection for projected Newton).

__device__ __forceinline__ bool ee_mollified(const EvalArgs& A, int type, int32_t i, int32_t j, const V3 Y[4],
                                             double* eps, double* c) {
  if (type != 1 || !A.moll_r2) return false;
  const V3 nn = cross(Y[1] - Y[0], Y[3] - Y[2]);
  *c = dot(nn, nn);
  *eps = A.moll_factor * A.moll_r2[i] * A.moll_r2[j];
  return *c < *eps;
}

// energy, gradient and exact Hessian (node-major 3a + k) of kappa m(c(x)) b(d(x))
__device__ __noinline__ void mollified_local(const V3* Y, const Stencil& S, double d, double dhat, double kappa,
                                             double eps, double c, double* E, double* g, double* H) {
  BarrierSpan B;
  barrier_span(Y, S, d, dhat, kappa, B);
  const double rhv[3] = {B.rh.x, B.rh.y, B.rh.z};
  double Q[12][5];
#pragma unroll 1
  for (int a = 0; a < 4; ++a)
    for (int k = 0; k < 3; ++k) {
      for (int p = 0; p < 3; ++p) Q[3 * a + k][p] = (k == p) ? B.basis[0][a] : 0.0;
      Q[3 * a + k][3] = B.basis[1][a] * rhv[k];
      Q[3 * a + k][4] = B.basis[2][a] * rhv[k];
    }
  double QK[12][5];
#pragma unroll 1
  for (int r = 0; r < 12; ++r)
    for (int p = 0; p < 5; ++p) {
      double acc = 0.0;
      for (int q = 0; q < 5; ++q) acc += Q[r][q] * B.K[q][p];
      QK[r][p] = acc;
    }
  // kappa grad b = kappa b' c_a r^ (c_a = |c| basis0_a)
  double gb[12];
  for (int a = 0; a < 4; ++a)
    for (int k = 0; k < 3; ++k) gb[3 * a + k] = kappa * B.b1 * B.cn * B.basis[0][a] * rhv[k];
  // c = |e0 x e1|^2: gradient and Hessian blocks in (e0, e1)
  const V3 e0 = Y[1] - Y[0], e1 = Y[3] - Y[2];
  const double s00 = dot(e0, e0), s11 = dot(e1, e1), s01 = dot(e0, e1);
  const double E0[3] = {e0.x, e0.y, e0.z}, E1[3] = {e1.x, e1.y, e1.z};
  double ge[2][3];
  for (int k = 0; k < 3; ++k) {
    ge[0][k] = 2.0 * (s11 * E0[k] - s01 * E1[k]);
    ge[1][k] = 2.0 * (s00 * E1[k] - s01 * E0[k]);
  }
  double gc[12];
  for (int k = 0; k < 3; ++k) {
    gc[k] = -ge[0][k]; gc[3 + k] = ge[0][k]; gc[6 + k] = -ge[1][k]; gc[9 + k] = ge[1][k];
  }
  const double m = c * (2.0 / eps - c / (eps * eps));
  const double m1 = 2.0 / eps - 2.0 * c / (eps * eps);
  const double m2 = -2.0 / (eps * eps);
  const double kb = B.E;                 // kappa b
  *E = m * kb;
  for (int r = 0; r < 12; ++r) g[r] = m * gb[r] + kb * m1 * gc[r];
  // the e-blocks of the Hessian of c
  auto hc = [&](int ea, int eb, int k, int l) -> double {
    const double dl = (k == l) ? 1.0 : 0.0;
    if (ea == 0 && eb == 0) return 2.0 * (s11 * dl - E1[k] * E1[l]);
    if (ea == 1 && eb == 1) return 2.0 * (s00 * dl - E0[k] * E0[l]);
    if (ea == 0) return 4.0 * E0[k] * E1[l] - 2.0 * E1[k] * E0[l] - 2.0 * s01 * dl;
    return 4.0 * E1[k] * E0[l] - 2.0 * E0[k] * E1[l] - 2.0 * s01 * dl;
  };
  const int edge_of[4] = {0, 0, 1, 1};
  const double sgn[4] = {-1.0, 1.0, -1.0, 1.0};
#pragma unroll 1
  for (int r = 0; r < 12; ++r) {
    const int a = r / 3, k = r % 3;
    for (int q = 0; q < 12; ++q) {
      const int b2 = q / 3, l = q % 3;
      double hb = 0.0;
      for (int p = 0; p < 5; ++p) hb += QK[r][p] * Q[q][p];
      const double hcv = sgn[a] * sgn[b2] * hc(edge_of[a], edge_of[b2], k, l);
      H[12 * r + q] = m * hb + kb * (m2 * gc[r] * gc[q] + m1 * hcv) + m1 * (gb[r] * gc[q] + gc[r] * gb[q]);
    }
  }
  for (int r = 0; r < 12; ++r)
    for (int q = r + 1; q < 12; ++q) {
      const double t = 0.5 * (H[12 * r + q] + H[12 * q + r]);
      H[12 * r + q] = t; H[12 * q + r] = t;
    }
}

// ------------------------------------------------------------------ pair factors
// The FP64 pipe bounds this stage (an FP64 warp instruction holds it for 64 cycles), so the
// blocks J^T (pair Hessian) J are never formed pair by pair.  Each item leaves one row per cage
// node u,
//   z_u1, z_u2 (z_u3): block(u, v) = sum_k z_uk z_vk^T + w_u w_v F + iso omega_u omega_v I,
// with omega_u = sum_a c_a w_au (the gradient at u is omega_u r' + w_u u') and the friction
// weight w_u, and a header (F, r', u', iso).  The segment sums below multiply rows straight into
// their accumulators: 10 FP64 instructions per record and third of a block, against about 47 to
// form a block here and 9 to add it, and no block goes through memory.
//
// At most one free closest-point parameter (a point p against the edge x_a x_b, or two
// points): with e = x_b - x_a, r = p - x_a - t e, v^ = -e/|e|, c = (1, t - 1, -t) on (p, a, b),
// a = (0, 1, -1), and the orthonormal span c^ (x) r^, c^ (x) v^, a^ (x) r^ (a^: a made
// orthogonal to c), the Hessian is
//   K = diag(A, -B, 0) + B p p^T,  A = kappa |c|^2 b'',  B = -kappa |c|^2 b'/d > 0,
//   p = (rho (c.a) / |c|^2, 1, rho |a - (a.c^) c^| / |c|),  rho = d / |e|,
// plus -B on the direction c^ (x) (r^ x v^), which the projection drops.  Its (v^, v^) entry is
// exactly zero.  D = diag(A, -B, 0) has one negative entry and the rest is rank one and
// positive, so K has one negative eigenvalue -B x; x in (0, 1) solves
//   x^2 (A + B x) = (1 - x) (p_2^2 (A + B x) + p_0^2 B x)
// (the secular equation cleared of its denominators: every term is positive, nothing
// cancels), found in FP32 and polished by two Newton steps in FP64.  Then
// q = (p_0 B/(A + B x), -1/(1 - x), p_2/x) spans its eigenvector, K+ = K + B x q q^T / |q|^2, and
// two steps of Cholesky give K+ = l l^T + m m^T.  Two points (no free parameter): K+ is A on
// c^ (x) r^ alone.  Against a 12 x 12 eigensolver the factors agree to 4e-15 of the norm over
// d/dhat from 1e-6 to 1 - 1e-14 and |e| from 10 um to 10 cm.

// flags of an item header
constexpr int kItemFriction = 1, kItemThird = 2, kItemIso = 4, kItemExplicit = 8;

__device__ __forceinline__ void store_header(double* h, const FrictionTerms* R, V3 g, double iso, int flags) {
  double2* p = reinterpret_cast<double2*>(h);
  if (R) {
    p[0] = make_double2(R->F[0][0], R->F[0][1]);
    p[1] = make_double2(R->F[0][2], R->F[1][1]);
    p[2] = make_double2(R->F[1][2], R->F[2][2]);
    p[4] = make_double2(g.z, R->gs * R->u[0]);
    p[5] = make_double2(R->gs * R->u[1], R->gs * R->u[2]);
  } else {
    p[4] = make_double2(g.z, 0.0);
    p[5] = make_double2(0.0, 0.0);
  }
  p[3] = make_double2(g.x, g.y);
  p[6] = make_double2(iso, __longlong_as_double((long long)flags));
}

__device__ __forceinline__ void store_row(double* row, V3 z1, V3 z2, double om, double wf) {
  double2* p = reinterpret_cast<double2*>(row);
  p[0] = make_double2(z1.x, z1.y);
  p[1] = make_double2(z1.z, z2.x);
  p[2] = make_double2(z2.y, z2.z);
  p[3] = make_double2(om, wf);
}

// a mollified pair: its records come from k_mollified_eval
__device__ __forceinline__ void list_mollified(const EvalArgs& A, int64_t k) {
  store_header(A.ihead + kIHead * k, nullptr, V3{0.0, 0.0, 0.0}, 0.0, kItemExplicit);
  A.moll_list[atomicAdd(reinterpret_cast<unsigned long long*>(A.n_moll), 1ull)] = (uint32_t)k;
}

// out[u] += coef * w over the four cage slots of vertex v (slot nodes in the nibbles of map);
// nothing for a kinematic vertex
__device__ __forceinline__ void add_slots(const EvalArgs& A, int32_t v, uint32_t map, double coef, double* out) {
  if (A.T.vkin[v]) return;
  const double2 w01 = __ldg(reinterpret_cast<const double2*>(A.w) + 2 * (int64_t)v);
  const double2 w23 = __ldg(reinterpret_cast<const double2*>(A.w) + 2 * (int64_t)v + 1);
  const double ws[4] = {w01.x, w01.y, w23.x, w23.y};
#pragma unroll
  for (int s = 0; s < 4; ++s) out[(map >> (4 * s)) & 15u] += coef * ws[s];
}

// ... and of two coefficients at once
__device__ __forceinline__ void add_slots2(const EvalArgs& A, int32_t v, uint32_t map, double c1, double* o1, double c2,
                                           double* o2) {
  if (A.T.vkin[v]) return;
  const double2 w01 = __ldg(reinterpret_cast<const double2*>(A.w) + 2 * (int64_t)v);
  const double2 w23 = __ldg(reinterpret_cast<const double2*>(A.w) + 2 * (int64_t)v + 1);
  const double ws[4] = {w01.x, w01.y, w23.x, w23.y};
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int u = (map >> (4 * s)) & 15u;
    o1[u] += c1 * ws[s];
    o2[u] += c2 * ws[s];
  }
}

__device__ __forceinline__ void zero_nodes(double* x, int n) {
  for (int u = 0; u < n; ++u) x[u] = 0.0;
}

// b, b', b'' of the barrier at distance d < dhat (Eq. 7 without kappa)
__device__ __forceinline__ void barrier_scalars(double d, double inv_d, double dhat, double inv_dhat, double* b, double* b1,
                                                double* b2) {
  double q = d * inv_dhat;
  q = fma(fma(-q, dhat, d), inv_dhat, q);              // d / dhat, rounded as the quotient
  const double lg = log(q), m = d - dhat, md = m * inv_d;
  *b = -m * m * lg;
  *b1 = -2.0 * m * lg - m * md;
  *b2 = -2.0 * lg - 4.0 * md + md * md;
}

// x in (0, 1) with x^2 (A + B x) = (1 - x) (w2 (A + B x) + w0 B x); A, B > 0, w0 >= 0, w2 > 0
__device__ __forceinline__ double negative_root(double A, double B, double w0, double w2) {
  // scaled by a power of two so that A is near one (the equation is homogeneous in A, B)
  const int ea = (__double2hiint(A) >> 20) & 0x7ff;
  const double s = __hiloint2double((2046 - ea) << 20, 0);
  A *= s;
  B *= s;
  const float Af = (float)A, Bf = (float)B, w0f = (float)w0, w2f = (float)w2;
  // x^2 = (1 - x) w for w = w2 + w0 B x / (A + B x), w from the previous x
  float x = 0.f;
#pragma unroll
  for (int it = 0; it < 3; ++it) {
    const float w = fmaxf(w2f + w0f * __fdividef(Bf * x, Af + Bf * x), 1e-36f);
    x = 2.f * w / (w + sqrtf(w * w + 4.f * w));
  }
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const float G = Af + Bf * x, y = w2f * G + w0f * Bf * x;
    const float h = x * x * G - (1.f - x) * y, hp = 2.f * x * G + x * x * Bf + y - (1.f - x) * (w2f + w0f) * Bf;
    const float nx = x - __fdividef(h, hp);
    if (nx > 0.f && nx <= 1.f) x = nx;
  }
  double xd = (double)x;
  const double wb = w0 * B;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double G = fma(B, xd, A), y = fma(w2, G, wb * xd), h = fma(xd * xd, G, -(1.0 - xd) * y);
    const float Gf = Af + Bf * x, yf = w2f * Gf + w0f * Bf * x;
    const float hp = 2.f * x * Gf + x * x * Bf + yf - (1.f - x) * (w2f + w0f) * Bf;
    const float hf = (float)h;
    if (hp > 0.f) xd -= (double)__fdividef(hf, hp);
  }
  return xd;
}

// The closest segment of a pair among those of `hint` (closest_hint without kHintInterior): point
// slot ip against edge (ia, ib), e = x_b - x_a, parameter t in [0, 1] (inner: strictly inside),
// r = x_p - x_a - t e, rse = 1/|e| (inner only).
struct SegmentPair {
  int ip, ia, ib;
  bool inner;
  double t, rse;
  V3 e, r;
};

__device__ __forceinline__ SegmentPair closest_segment(int type, const V3 X[4], int hint) {
  // the only one left, or (ties, e.g. at a shared vertex) the closest in FP64
  int seg = __ffs(hint & 15) - 1;
  if (hint & (hint - 1) & 15) {
    double best = 0.0, t;
    int left = hint & 15;
    seg = -1;
    for (int step = 0; step < 4 && left; ++step) {
      const int q = __ffs(left) - 1;
      left &= left - 1;
      int qp, qa, qb;
      segment_slots(type, q, &qp, &qa, &qb);
      const double d2 = seg_point_d2(pick(X, qp), pick(X, qa), pick(X, qb), &t);
      if (seg < 0 || lt_nonneg(d2, best)) { best = d2; seg = q; }
    }
  }
  SegmentPair G;
  segment_slots(type, seg, &G.ip, &G.ia, &G.ib);
  const V3 xa = pick(X, G.ia), w = pick(X, G.ip) - xa;
  G.e = pick(X, G.ib) - xa;
  const double we = dot(w, G.e), ee = dot(G.e, G.e);
  G.t = 0.0;
  G.rse = 0.0;
  G.inner = is_pos(we) && lt_nonneg(we, ee);
  if (G.inner) {
    G.rse = rsqrt(ee);
    G.t = we * (G.rse * G.rse);
  } else if (is_pos(we)) {
    G.t = 1.0;
  }
  G.r = w - G.e * G.t;
  return G;
}

// Node rows and header of a pair whose closest features are one of the segments of `hint`
// (closest_hint without kHintInterior).
__device__ __forceinline__ void light_factors(const EvalArgs& A, int64_t k, int type, int32_t i, int32_t j, const int32_t v[4],
                                              int hint) {
  V3 X[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) X[a] = load_x(A.x4, v[a]);
  const SegmentPair Sg = closest_segment(type, X, hint);
  const int ip = Sg.ip, ia = Sg.ia, ib = Sg.ib;
  const bool inner = Sg.inner;
  const double t = Sg.t, rse = Sg.rse;
  const V3 e = Sg.e, r = Sg.r;
  const double d2 = dot(r, r);
  const bool apart = d2 > 0.0;
  if (!apart) raise_flag(A.st, EIPC_FLAG_PENETRATION);
  const double inv_d = apart ? rsqrt(d2) : 0.0;
  const double d = d2 * inv_d;
  const bool active = apart && lt_nonneg(d, A.dhat);
  if (active && A.moll_r2 && type == 1) {
    const V3 Y[4] = {{0.0, 0.0, 0.0}, X[1] - X[0], X[2] - X[0], X[3] - X[0]};
    double eps_m, c_m;
    if (ee_mollified(A, type, i, j, Y, &eps_m, &c_m)) {           // k_mollified_eval
      list_mollified(A, k);
      return;
    }
  }
  const int n = A.item_n[k];
  const uint64_t map = A.item_map[k];
  const V3 rh = r * inv_d;
  double E = 0.0, iso = 0.0, gs = 0.0;
  double k1 = 0.0, k2 = 0.0, k3 = 0.0, k4 = 0.0, k5 = 0.0, k6 = 0.0;
  double om[kMaxNodes], al[kMaxNodes], wf[kMaxNodes];
  zero_nodes(om, n);
  zero_nodes(al, n);
  zero_nodes(wf, n);
  V3 vh = {0.0, 0.0, 0.0};
  if (active) {
    double b, b1, b2;
    barrier_scalars(d, inv_d, A.dhat, A.inv_dhat, &b, &b1, &b2);
    E = A.kappa * b;
    gs = A.kappa * b1;
    const double bd = -A.kappa * (b1 * inv_d);                    // -kappa b'/d
    const double s1 = 1.0 - t;
    vh = e * -rse;
    if (A.project) {
      const double cc = 1.0 + s1 * s1 + t * t;
      const double Aq = A.kappa * cc * b2, B = cc * bd;
      const bool span = inner && is_pos(B);
      double K00 = Aq, K01 = 0.0, K02 = 0.0, K11 = 0.0, K12 = 0.0, K22 = 0.0, rcn = rsqrt(cc), ral = 0.0, cac = 0.0;
      if (span) {
        const double ca0 = 2.0 * t - 1.0;
        cac = ca0 * (rcn * rcn);                                  // c.a / |c|^2
        const double al2 = 2.0 - ca0 * cac;
        ral = rsqrt(al2);
        const double rho = d * rse;
        const double p0 = rho * cac, p2 = rho * (al2 * ral) * rcn;
        const double x = negative_root(Aq, B, p0 * p0, p2 * p2);
        const double G = fma(B, x, Aq), rc = 1.0 / (G * x);
        const double q0 = p0 * B * (rc * x), q2 = p2 * (rc * G), S = 1.0 + p0 * q0 + p2 * q2;
        const double f = x / (q0 * q0 + S * S + q2 * q2);
        const double fq0 = f * q0, fs = f * S;
        K00 += B * (p0 * p0 + fq0 * q0);
        K01 = B * (p0 - fq0 * S);
        K02 = B * (p0 * p2 + fq0 * q2);
        K11 = B * (fs * S);
        K12 = B * (p2 - fs * q2);
        K22 = B * (p2 * p2 + f * q2 * q2);
      }
      const double rk = rsqrt(K00);
      const double l0 = K00 * rk, l1 = K01 * rk, l2 = K02 * rk;
      double m1 = 0.0, m2 = 0.0;
      if (span) {
        const double s11 = K11 - l1 * l1, s12 = K12 - l1 * l2, s22 = K22 - l2 * l2;
        const bool first = __double_as_longlong(s11) >= __double_as_longlong(s22);
        const double piv = first ? s11 : s22;
        if (is_pos(piv)) {
          const double rp = rsqrt(piv), a = piv * rp, o = s12 * rp;
          m1 = first ? a : o;
          m2 = first ? o : a;
        }
      }
      k2 = l2 * ral;
      k1 = l0 * rcn - k2 * cac;
      k3 = l1 * rcn;
      k5 = m2 * ral;
      k4 = -k5 * cac;
      k6 = m1 * rcn;
    } else {
      // exact: kappa (b'' - b'/d) c c^T (x) r^ r^T + kappa (b'/d) c c^T (x) I - (kappa b'/(2d)) G M^-1 G^T
      const double h = fma(A.kappa, b2, bd);
      k1 = h * rsqrt(h);
      iso = -bd;
      if (inner) {
        const double sb = is_pos(bd) ? bd * rsqrt(bd) : 0.0;
        k5 = sb * rse * d;
        k6 = sb;
      }
    }
    // omega and alpha over the three used vertices (two where the closest point is a vertex)
    add_slots(A, pick(v, ip), (uint32_t)(map >> (16 * ip)) & 0xffffu, 1.0, om);
    if (inner) {
      add_slots2(A, pick(v, ia), (uint32_t)(map >> (16 * ia)) & 0xffffu, -s1, om, 1.0, al);
      add_slots2(A, pick(v, ib), (uint32_t)(map >> (16 * ib)) & 0xffffu, -t, om, -1.0, al);
    } else {
      const int iq = is_pos(t) ? ib : ia;
      add_slots(A, pick(v, iq), (uint32_t)(map >> (16 * iq)) & 0xffffu, -1.0, om);
    }
  }
  const int32_t fenc = A.fric_of_pair ? A.fric_of_pair[k] : 0;
  FrictionTerms R;
  if (fenc > 0) {
    double gam[4];
    friction_terms(A.x4, A.lag, (int64_t)(INT32_MAX - fenc), v, A.mu, A.eps_f, R, gam);
    E += R.E;
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (gam[a] != 0.0) add_slots(A, v[a], (uint32_t)(map >> (16 * a)) & 0xffffu, gam[a], wf);
  }
  A.item_E[k] = E;
  store_header(A.ihead + kIHead * k, fenc > 0 ? &R : nullptr, rh * gs, iso,
               (fenc > 0 ? kItemFriction : 0) | (iso != 0.0 ? kItemIso : 0));
  const int64_t base = A.ro_g[k];
  for (int u = 0; u < n; ++u) {
    if (base + u >= A.gcap) break;
    const double o = om[u], a = al[u];
    const V3 z1 = rh * (o * k1 + a * k2) + vh * (o * k3), z2 = rh * (o * k4 + a * k5) + vh * (o * k6);
    store_row(A.frow + kFRow * (base + u), z1, z2, o, wf[u]);
  }
}

// eigenvalues (big, small) of the symmetric [[a, b], [b, c]] and the unit eigenvector of the big one
template <class T>
__device__ __forceinline__ void eigen2(T a, T b, T c, T* big, T* small, T* y0, T* y1) {
  const T h = T(0.5) * (a + c), dl = T(0.5) * (a - c), r2 = dl * dl + b * b;
  const T r = r2 > T(0) ? r2 * rsqrt(r2) : T(0);
  const T p = r + (dl < T(0) ? -dl : dl), n = p * p + b * b;
  const T s = n > T(0) ? rsqrt(n) : T(0);
  const T u = n > T(0) ? p * s : T(1), v = b * s;
  *big = h + r;
  *small = h - r;
  *y0 = dl < T(0) ? v : u;
  *y1 = dl < T(0) ? u : v;
}

// Pairs whose closest points have two free parameters: a point over a triangle's interior, two
// edges' interiors.  n = e_1 x e_2 gives r^ = +-n/|n| and d = |w . n|/|n|.  With v_j = sum_a
// a_j[a] x_a = L (p_1, p_2) (Gram-Schmidt, in the plane normal to r^) and a_j made orthonormal
// against c and each other, the span c^ (x) r^, c^ (x) p_1, c^ (x) p_2, a^_1 (x) r^, a^_2 (x) r^ has
//   K = diag(A, -B, -B, 0, 0) + B U U^T,  U = [x^T; I; Y],
//   x = (d/|c|) L^-1 (c^.a_1, c^.a_2),  Y = (d/|c|) [a^_l . a_j] L^-T  (upper triangular),
// with A, B as for one parameter.  Two entries of the diagonal part are negative and the rest is
// positive, so K has exactly two negative eigenvalues -B mu: mu^2 = (1 - mu) N, where N is an
// eigenvalue of W(tau) = Y^T Y + tau x x^T at tau = B mu/(A + B mu) and y its eigenvector, and
// q = (tau/mu x.y, -y/(1 - mu), Y y/mu) spans K's eigenvector.  tau is found in FP32 and polished
// in FP64 (N moves by (x.y)^2 dtau, so each pass squares the error); mu and 1 - mu come from N
// without cancellation.  K+ = K + B sum mu q q^T/|q|^2 has rank three, taken by three steps of
// Cholesky with the largest pivot.  Against a 12 x 12 eigensolver: 8e-12 at d = 7e-6 dhat, 1e-13
// and below from 1e-3 dhat, near-parallel edges and slivers included.  About 700 FP64
// instructions, where a 5 x 5 Jacobi eigensolver and its set-up took over 4,000: 130 us for a
// warp of pairs before, 67 us after, 55 us with few pairs a warp.
//
// Two neighbouring lanes take a pair: each finds one of the two eigenvectors and writes every
// other row, and both do the rest alike, so that they stay together: 45 us for a
// short list where one lane a pair took 55, plate in rack 93 and 113 us.
__device__ __forceinline__ void heavy_factors(const EvalArgs& A, int64_t k) {
  const int half = threadIdx.x & 1;
  const unsigned both = 3u << (threadIdx.x & 30);
  int32_t v[4];
  const int type = A.pr.type[k];
  const int32_t i = A.pr.i[k], j = A.pr.j[k];
  stencil_vertices(A.T, type, i, j, v);
  const int hint = stencil_hint(type, A.x4f, v);
  V3 X[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) X[a] = load_x(A.x4, v[a]);
  const bool pt = type == 0;
  double c[4];
  V3 rh = {0.0, 0.0, 0.0};
  double d = 0.0, inv_d = 0.0;
  bool in, apart;
  {
    const V3 e1 = pt ? X[2] - X[1] : X[1] - X[0], e2 = pt ? X[3] - X[1] : X[3] - X[2], w = pt ? X[0] - X[1] : X[0] - X[2];
    const V3 n = cross(e1, e2);
    const double nn = dot(n, n), inv_nn = 1.0 / nn;
    double s, t;
    if (pt) {
      s = dot(cross(w, e2), n) * inv_nn;
      t = dot(cross(e1, w), n) * inv_nn;
      in = s >= 0.0 && t >= 0.0 && s + t <= 1.0;
      c[0] = 1.0; c[1] = -(1.0 - s - t); c[2] = -s; c[3] = -t;
    } else {
      const double a = dot(e1, e1), b = dot(e1, e2), cc = dot(e2, e2), dd = dot(e1, w), ee = dot(e2, w);
      s = (b * ee - cc * dd) * inv_nn;
      t = (a * ee - b * dd) * inv_nn;
      in = nn > 1e-20 * a * cc && s >= 0.0 && s <= 1.0 && t >= 0.0 && t <= 1.0;
      c[0] = 1.0 - s; c[1] = s; c[2] = -(1.0 - t); c[3] = -t;
    }
    in = in || (hint & kHintCertain);
    const double h = dot(w, n), rn = rsqrt(nn), hs = h < 0.0 ? -rn : rn;
    rh = n * hs;
    d = h * hs;
    apart = d > 0.0;
    if (apart) inv_d = 1.0 / d;
  }
  if (!in) {                                   // the region the FP32 test left open: a segment after all
    if (half == 0) light_factors(A, k, type, i, j, v, pt ? 7 : 15);
    return;
  }
  if (!apart) raise_flag(A.st, EIPC_FLAG_PENETRATION);
  const bool active = apart && lt_nonneg(d, A.dhat);
  if (active && A.moll_r2 && type == 1) {
    const V3 Y[4] = {{0.0, 0.0, 0.0}, X[1] - X[0], X[2] - X[0], X[3] - X[0]};
    double eps_m, c_m;
    if (ee_mollified(A, type, i, j, Y, &eps_m, &c_m)) {           // k_mollified_eval
      if (half == 0) list_mollified(A, k);
      return;
    }
  }
  const int n = A.item_n[k];
  const uint64_t map = A.item_map[k];
  double om[kMaxNodes], al[2][kMaxNodes], wf[kMaxNodes];
  zero_nodes(om, n);
  zero_nodes(al[0], n);
  zero_nodes(al[1], n);
  zero_nodes(wf, n);
  double E = 0.0, gs = 0.0, iso = 0.0;
  // z_k = (omega f[k][0] + alpha_1 f[k][1] + alpha_2 f[k][2]) r^ + omega P[k]
  double f[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  V3 P[3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  if (active) {
    double b, b1, b2;
    barrier_scalars(d, inv_d, A.dhat, A.inv_dhat, &b, &b1, &b2);
    E = A.kappa * b;
    gs = A.kappa * b1;
    const double bd = -A.kappa * (b1 * inv_d);
    // v_1, v_2 by Gram-Schmidt: v_1 = l11 p_1, v_2 = l21 p_1 + l22 p_2
    const V3 v1 = pt ? X[1] - X[2] : X[1] - X[0], v2 = pt ? X[1] - X[3] : X[2] - X[3];
    const double j11 = rsqrt(dot(v1, v1));
    const V3 p1 = v1 * j11;
    const double l21 = dot(v2, p1);
    const V3 u2 = v2 - p1 * l21;
    const double j22 = rsqrt(dot(u2, u2));
    const V3 p2 = u2 * j22;
    const double lj = l21 * j11;
    if (A.project && is_pos(bd)) {
      const double cc = c[0] * c[0] + c[1] * c[1] + c[2] * c[2] + c[3] * c[3], rcn = rsqrt(cc);
      const double Aq = A.kappa * cc * b2, B = cc * bd;
      const double k1 = (pt ? c[1] - c[2] : c[1] - c[0]) * rcn, k2 = (pt ? c[1] - c[3] : c[2] - c[3]) * rcn;
      const double t11 = 2.0 - k1 * k1, i11 = rsqrt(t11), al11 = t11 * i11;
      const double al12 = ((pt ? 1.0 : 0.0) - k1 * k2) * i11;
      const double t22 = 2.0 - k2 * k2 - al12 * al12, i22 = rsqrt(t22), al22 = t22 * i22;
      const double dc = d * rcn, d1 = dc * j11, d2 = dc * j22;
      const double x1 = k1 * d1, x2 = (k2 - k1 * lj) * d2;
      const double y11 = al11 * d1, y12 = (al12 - al11 * lj) * d2, y22 = al22 * d2;
      const double w11 = y11 * y11, w12 = y11 * y12, w22 = y12 * y12 + y22 * y22;
      const double s11 = x1 * x1, s12 = x1 * x2, s22 = x2 * x2;
      double K[5][5];                          // upper triangle, over B
      const double iB = 1.0 / B;
      K[0][0] = Aq * iB + s11 + s22;
      K[0][1] = x1; K[0][2] = x2; K[0][3] = x1 * y11 + x2 * y12; K[0][4] = x2 * y22;
      K[1][1] = 0.0; K[1][2] = 0.0; K[1][3] = y11; K[1][4] = 0.0;
      K[2][2] = 0.0; K[2][3] = y12; K[2][4] = y22;
      K[3][3] = w11 + y12 * y12; K[3][4] = y12 * y22; K[4][4] = y22 * y22;
      const double as = Aq * iB;               // A / B
      const float af = to_float<0>(as), w11f = to_float<0>(w11), w12f = to_float<0>(w12), w22f = to_float<0>(w22);
      const float s11f = to_float<0>(s11), s12f = to_float<0>(s12), s22f = to_float<0>(s22);
      const double dy = y11 * y22, det0 = dy * dy, g1 = y12 * x1 - y11 * x2, g2 = y22 * x1, det1 = g1 * g1 + g2 * g2;
      double mine[5], mu_mine;                 // this lane's eigenvector of K, times mu nu, and mu
      {
        const int e = half;
        float tf = 0.f;
#pragma unroll 1
        for (int it = 0; it < 4; ++it) {
          float big, sml, ya, yb;
          eigen2<float>(w11f + tf * s11f, w12f + tf * s12f, w22f + tf * s22f, &big, &sml, &ya, &yb);
          const float N = fmaxf(e == 0 ? big : sml, 1e-30f), mu = 2.f * N / (N + sqrtf(N * N + 4.f * N));
          tf = __fdividef(mu, af + mu);
        }
        double tau = tf >= 0.f && tf <= 1.f ? (double)tf : 0.5;
        double ya = 0.0, yb = 0.0, xy = 0.0, mu = 0.0, nu = 1.0;
#pragma unroll 1
        for (int it = 0; it < 8; ++it) {
          double big, sml;
          eigen2<double>(fma(tau, s11, w11), fma(tau, s12, w12), fma(tau, s22, w22), &big, &sml, &ya, &yb);
          double N = big;
          if (e == 1) {
            N = fma(tau, det1, det0) / big;    // the small eigenvalue without cancellation
            const double t = ya;
            ya = -yb;
            yb = t;
          }
          N = fmax(N, 1e-280);
          xy = x1 * ya + x2 * yb;
          // mu = 2N/(N + s), 1 - mu = 2/(N + 2 + s), s = sqrt(N^2 + 4N)
          double s2 = N * (N + 4.0), s = s2 * rsqrt(s2), a = N + s, g = a + 2.0, rc = 2.0 / (a * g);
          const double t1 = N * g * rc, tn = t1 / (as + t1), dt = tn - tau;
          N = fma(xy * xy, dt, N);
          N = fmax(N, 1e-280);
          s2 = N * (N + 4.0); s = s2 * rsqrt(s2); a = N + s; g = a + 2.0; rc = 2.0 / (a * g);
          mu = N * g * rc;
          nu = a * rc;
          tau = mu / (as + mu);
          if (lt_nonneg(fabs(dt), 1e-9)) break;
        }
        mine[0] = tau * xy * nu; mine[1] = -ya * mu; mine[2] = -yb * mu;
        mine[3] = (y11 * ya + y12 * yb) * nu; mine[4] = y22 * yb * nu;
        mu_mine = mu;
      }
      double q[2][5], mus[2];
#pragma unroll
      for (int p = 0; p < 5; ++p) {
        const double other = __shfl_xor_sync(both, mine[p], 1);
        q[0][p] = half ? other : mine[p];
        q[1][p] = half ? mine[p] : other;
      }
      {
        const double other = __shfl_xor_sync(both, mu_mine, 1);
        mus[0] = half ? other : mu_mine;
        mus[1] = half ? mu_mine : other;
      }
      double q0n = 0.0;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (e == 1) {                          // the second made orthogonal to the first
          double pr = 0.0;
#pragma unroll
          for (int p = 0; p < 5; ++p) pr += q[0][p] * q[1][p];
          pr *= q0n;
#pragma unroll
          for (int p = 0; p < 5; ++p) q[1][p] -= pr * q[0][p];
        }
        double qq = 0.0;
#pragma unroll
        for (int p = 0; p < 5; ++p) qq += q[e][p] * q[e][p];
        const double iq = 1.0 / qq, m = mus[e] * iq;
#pragma unroll
        for (int p = 0; p < 5; ++p) {
          const double mp = m * q[e][p];
#pragma unroll
          for (int r = p; r < 5; ++r) K[p][r] = fma(mp, q[e][r], K[p][r]);
        }
        if (e == 0) q0n = iq;
      }
      // three columns of Cholesky, times sqrt(B): r^ first, then the largest diagonal entries left
      const double sB = B * rsqrt(B);
      double S[4][4], l[3][5];
      {
        const double rk = rsqrt(K[0][0]);
#pragma unroll
        for (int p = 0; p < 5; ++p) l[0][p] = K[0][p] * rk;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int r = p; r < 4; ++r) {
            S[p][r] = fma(-l[0][1 + p], l[0][1 + r], K[1 + p][1 + r]);
            S[r][p] = S[p][r];
          }
      }
#pragma unroll
      for (int col = 1; col < 3; ++col) {
        int piv = 0;
        double best = S[0][0];
#pragma unroll
        for (int p = 1; p < 4; ++p)
          if (__double_as_longlong(S[p][p]) > __double_as_longlong(best)) { best = S[p][p]; piv = p; }
        const double rp = is_pos(best) ? rsqrt(best) : 0.0;
        double row[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          double x = S[0][r];
          if (piv == 1) x = S[1][r];
          if (piv == 2) x = S[2][r];
          if (piv == 3) x = S[3][r];
          row[r] = x * rp;
          l[col][1 + r] = row[r];
        }
        l[col][0] = 0.0;
        if (col == 1) {
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int r = p; r < 4; ++r) {
              S[p][r] = fma(-row[p], row[r], S[p][r]);
              S[r][p] = S[p][r];
            }
        }
      }
      // omega^ = omega/|c|, alpha^_1 = (alpha_1 - k1 omega^)/al11, alpha^_2 = (alpha_2 - k2 omega^ - al12 alpha^_1)/al22
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double m2 = l[q][4] * i22 * sB, m1 = (l[q][3] * sB - m2 * al12) * i11;
        f[q][1] = m1;
        f[q][2] = m2;
        f[q][0] = (l[q][0] * sB - m1 * k1 - m2 * k2) * rcn;
        P[q] = (p1 * l[q][1] + p2 * l[q][2]) * (sB * rcn);
      }
    } else {
      // exact: r^, isotropic and G M^-1 G^T terms (the last as y_1 = (omega v_1 + alpha_1 r)/l11, y_2
      // likewise less its share of y_1).  A projected pair whose b' has underflowed keeps r^ alone.
      const double h = A.project ? A.kappa * b2 : fma(A.kappa, b2, bd);
      f[0][0] = h * rsqrt(h);
      if (!A.project) {
        iso = -bd;
        const double sb = is_pos(bd) ? bd * rsqrt(bd) : 0.0, q1 = sb * d * j11, q2 = sb * d * j22;
        P[1] = p1 * sb;
        f[1][1] = q1;
        P[2] = p2 * sb;
        f[2][2] = q2;
        f[2][1] = -lj * q2;
      }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) add_slots(A, v[a], (uint32_t)(map >> (16 * a)) & 0xffffu, c[a], om);
    const int m1s = pt ? 2 : 0, p2s = pt ? 1 : 2;          // a_1 = +1 at 1, -1 at m1s; a_2 = +1 at p2s, -1 at 3
    add_slots(A, v[1], (uint32_t)(map >> 16) & 0xffffu, 1.0, al[0]);
    add_slots(A, pick(v, m1s), (uint32_t)(map >> (16 * m1s)) & 0xffffu, -1.0, al[0]);
    add_slots(A, pick(v, p2s), (uint32_t)(map >> (16 * p2s)) & 0xffffu, 1.0, al[1]);
    add_slots(A, v[3], (uint32_t)(map >> 48) & 0xffffu, -1.0, al[1]);
  }
  const int32_t fenc = A.fric_of_pair ? A.fric_of_pair[k] : 0;
  FrictionTerms R;
  if (fenc > 0) {
    double gam[4];
    friction_terms(A.x4, A.lag, (int64_t)(INT32_MAX - fenc), v, A.mu, A.eps_f, R, gam);
    E += R.E;
#pragma unroll
    for (int a = 0; a < 4; ++a) add_slots(A, v[a], (uint32_t)(map >> (16 * a)) & 0xffffu, gam[a], wf);
  }
  if (half == 0) {
    A.item_E[k] = E;
    store_header(A.ihead + kIHead * k, fenc > 0 ? &R : nullptr, rh * gs, iso,
                 (fenc > 0 ? kItemFriction : 0) | (iso != 0.0 ? kItemIso : 0) | kItemThird);
  }
  const int64_t base = A.ro_g[k];
  for (int u = half; u < n && base + u < A.gcap; u += 2) {
    const double o = om[u], a1 = al[0][u], a2 = al[1][u];
    V3 z[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) z[q] = P[q] * o + rh * (o * f[q][0] + a1 * f[q][1] + a2 * f[q][2]);
    double* row = A.frow + kFRow * (base + u);
    store_row(row, z[0], z[1], o, wf[u]);
    reinterpret_cast<double2*>(row)[4] = make_double2(z[2].x, z[2].y);
    row[10] = z[2].z;
  }
}

// ... of a lagged friction item without a contact pair
__device__ __forceinline__ void friction_factors(const EvalArgs& A, int64_t k, int64_t f) {
  const int4 q4 = reinterpret_cast<const int4*>(A.lag.v)[f];
  const int32_t v[4] = {q4.x, q4.y, q4.z, q4.w};
  const int n = A.item_n[k];
  const uint64_t map = A.item_map[k];
  FrictionTerms R;
  double gam[4], wf[kMaxNodes];
  friction_terms(A.x4, A.lag, f, v, A.mu, A.eps_f, R, gam);
  A.item_E[k] = R.E;
  zero_nodes(wf, n);
#pragma unroll
  for (int a = 0; a < 4; ++a)
    if (gam[a] != 0.0) add_slots(A, v[a], (uint32_t)(map >> (16 * a)) & 0xffffu, gam[a], wf);
  store_header(A.ihead + kIHead * k, &R, V3{0.0, 0.0, 0.0}, 0.0, kItemFriction);
  const int64_t base = A.ro_g[k];
  for (int u = 0; u < n && base + u < A.gcap; ++u)
    store_row(A.frow + kFRow * (base + u), V3{0.0, 0.0, 0.0}, V3{0.0, 0.0, 0.0}, 0.0, wf[u]);
}

// Factors of every item whose closest features are points and segments, by a work queue over the
// items, each warp claiming A.tile of them at a time (the first tile is the warp's own, so warps
// beyond a short list leave at once).  A divergent FP64 branch costs a warp its whole length, so
// pairs with an interior closest point and friction items without a pair are only listed here, for
// k_eval_rest to take in full warps: about one pair in a hundred of the bubble grasp, which used
// to hold up every third warp (459 us for factors and rest in one kernel, 126 us for these alone).
// The evaluation of the full bubble grasp (171k pairs, 163k friction items): 1194 -> 713 us.
__global__ void __launch_bounds__(kEvalThreads, 4) k_eval_factors(EvalArgs A) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  const int64_t P = clamp_count(A.pr.count, A.pr.capacity);
  const int64_t nit = *A.n_items;
  const int64_t np = P < nit ? P : nit;
  const int width = items_per_warp(nit);
  const int tile = width < 32 ? width : (A.tile >= 32 ? (A.tile & ~31) : 32);
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * tile;
  int left = tile;
  // a warp takes `width` items a round: nit / width + 2 rounds cover every claim it can make
  const int64_t max_rounds = nit / width + 2;
  for (int64_t round = 0;; ++round) {
    if (round > max_rounds) {
      raise_flag(A.st, EIPC_FLAG_STACK_OVERFLOW);
      break;
    }
    if (left == 0) {
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(A.queue), (unsigned long long)tile);
      base = (int64_t)__shfl_sync(0xffffffffu, b, 0) + warps * tile;
      left = tile;
    }
    if (base >= nit) break;
    const int64_t k = base + lane;
    int later = -1;
    const bool mine = lane < width;
    if (mine && k < np) {
      int32_t v[4];
      const int type = A.pr.type[k];
      const int32_t i = A.pr.i[k], j = A.pr.j[k];
      stencil_vertices(A.T, type, i, j, v);
      const int hint = stencil_hint(type, A.x4f, v);
      if (hint & kHintInterior) later = 0;
      else light_factors(A, k, type, i, j, v, hint);
    } else if (mine && k < nit) {
      if (friction_merged(A.fric_of_pair, A.pair_of_fric, k - P)) A.item_E[k] = 0.0;   // with its contact pair
      else later = 1;
    }
    const unsigned m = __ballot_sync(0xffffffffu, later >= 0);
    if (m) {
      // the interior pairs from the front, the friction items from the back (no more than items in all)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const unsigned mc = __ballot_sync(0xffffffffu, later == c);
        if (!mc) continue;
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(A.n_rest + c), (unsigned long long)__popc(mc));
        b = __shfl_sync(0xffffffffu, b, 0);
        if (later == c) {
          const int64_t at = (int64_t)b + __popc(mc & ((1u << lane) - 1u));
          A.rest[c == 0 ? at : A.item_cap - 1 - at] = (uint32_t)k;
        }
      }
    }
    base += width;
    left -= width;
  }
}

// ... of the items it listed: whole warps of one kind.
__global__ void __launch_bounds__(kEvalThreads, 2) k_eval_rest(EvalArgs A) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  const int64_t P = clamp_count(A.pr.count, A.pr.capacity);
  const int64_t n0 = A.n_rest[0], n1 = A.n_rest[1];
  const int width = items_per_warp(2 * n0 + n1), pairs = width > 1 ? width / 2 : 1;       // two lanes a pair
  const int64_t w0 = (n0 + pairs - 1) / pairs, w1 = (n1 + width - 1) / width;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < w0 + w1; w += nw) {
    if (w < w0) {
      const int64_t q = pairs * w + (lane >> 1);
      if (lane < 2 * pairs && q < n0) heavy_factors(A, A.rest[q]);
    } else if (lane < width) {
      const int64_t q = width * (w - w0) + lane;
      if (q < n1) {
        const int64_t k = A.rest[A.item_cap - 1 - q];
        friction_factors(A, k, k - P);
      }
    }
  }
}

// Mollified EE pairs in the evaluation (the factor kernel lists them): explicit records.
//
// Nine lanes per pair, three pairs per warp.  The pair's Hessian vanishes on translations, so it
// is taken in the nine directions u_i (x) e_k with the orthonormal u_1 = (1,-1,0,0)/sqrt 2,
// u_2 = (0,0,1,-1)/sqrt 2, u_3 = (1,1,-1,-1)/2; lane j holds column j.  The projection is a cyclic
// two-sided Jacobi in which each round's four disjoint rotations run at once (round r pairs i
// and j with i + j = r mod 9): a lane fetches its partner's column by shuffles and every lane
// applies the four row rotations to its own.  A rotation by any angle is exact, so the angle's
// tangent is taken in FP32 (the entry left is 1e-7 of the one removed) and only c = 1/sqrt(1 +
// t^2) in FP64.  One thread per pair, with its 12 x 12 matrices in local memory, kept 174 warps
// busy with 70,000 FP64 instructions each: 4.2 ms for the 2.5k mollified pairs of two
// 16 x 16-cell sheets.
constexpr int kMollWarps = 2;
struct MollShared {
  double H[81];                // the (projected) Hessian, column-major
  double HW[kMaxNodes][27];    // H times the node's weights: rows j, component k
  double W[3][kMaxNodes];      // the nodes' weights in the basis u_1, u_2, u_3
  double g[9];
};

__device__ __forceinline__ double shfl_d(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }

template <int N>
__device__ __forceinline__ double select_d(const double (&x)[N], int k) {
  double r = x[0];
#pragma unroll
  for (int i = 1; i < N; ++i)
    if (k == i) r = x[i];
  return r;
}

// one round of rotations on the columns T, V of lane `me` of the nine from lane `first` on; by no
// angle, which leaves the values as they are, where `on` (the same in all nine) is not set
template <int R>
__device__ __forceinline__ void jacobi9_round(double (&T)[9], double (&V)[9], int me, int first, bool on) {
  int other = R - me;
  if (other < 0) other += 9;
  const bool bye = other == me;
  const bool low = me < other;
  const int lp = first + (low ? me : other), lo = first + other;
  const double dg = select_d(T, me), off = shfl_d(select_d(T, other), lp), dgo = shfl_d(dg, lo);
  const double gap = low ? dgo - dg : dg - dgo;          // a_qq - a_pp
  const float gf = (float)gap, of = (float)off;
  float tf = 0.f;
  if (fabsf(of) > 0.f) {
    const float th = gf / (2.f * of), at = fabsf(th);
    tf = at > 1e18f ? 0.5f / at : 1.f / (at + sqrtf(at * at + 1.f));
    tf = th < 0.f ? -tf : tf;
  }
  if (bye || !on) tf = 0.f;
  const double t = (double)tf, c = rsqrt(fma(t, t, 1.0)), s = t * c, sg = low ? -s : s;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double a = shfl_d(T[k], lo), b = shfl_d(V[k], lo);
    T[k] = fma(c, T[k], bye ? 0.0 : sg * a);
    V[k] = fma(c, V[k], bye ? 0.0 : sg * b);
  }
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    const int q = (R - p + 9) % 9;
    if (q <= p) continue;
    const double cp = shfl_d(c, first + p), sp = shfl_d(s, first + p);
    const double tp = T[p], tq = T[q];
    T[p] = fma(cp, tp, -sp * tq);
    T[q] = fma(cp, tq, sp * tp);
  }
}

__global__ void __launch_bounds__(32 * kMollWarps) k_mollified_eval(EvalArgs A, const uint32_t* __restrict__ list,
                                                                    const int64_t* n_list) {
  pdl_entry();
  __shared__ MollShared shared[kMollWarps][3];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int grp = lane / 9 < 3 ? lane / 9 : 2, me = lane - 9 * (lane / 9), first = 9 * grp;
  const bool live_lane = lane < 27;
  MollShared& sh = shared[wib][grp];
  const int64_t n_list_v = *n_list;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w0 = 3 * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); w0 < n_list_v; w0 += 3 * nw) {
    // idle groups and lanes repeat the last pair's work without writing, so that the shuffles stay
    // whole
    const bool live = live_lane && w0 + grp < n_list_v;
    const int64_t k = list[w0 + grp < n_list_v ? w0 + grp : n_list_v - 1];
    const int m_e = me < 9 ? me : 8;
    int32_t v[4];
    const int32_t i = A.pr.i[k], j = A.pr.j[k];
    stencil_vertices(A.T, 1, i, j, v);
    V3 Y[4];
    const V3 X0 = load_x(A.x4, v[0]);
#pragma unroll
    for (int a = 0; a < 4; ++a) Y[a] = load_x(A.x4, v[a]) - X0;
    double eps, c;
    ee_mollified(A, 1, i, j, Y, &eps, &c);
    Stencil S;
    closest_pair<true>(1, Y, stencil_hint(1, A.x4f, v), &S);
    const double d = sqrt(S.d2);
    BarrierSpan B;
    barrier_span(Y, S, d, A.dhat, A.kappa, B);
    const double ie = 1.0 / eps;
    const double m = c * (2.0 * ie - c * ie * ie), m1 = 2.0 * ie - 2.0 * c * ie * ie, m2 = -2.0 * ie * ie;
    const double kb = B.E;                               // kappa b
    // the span's vectors in the basis u_1, u_2, u_3
    const double r2 = 0.70710678118654752440;
    double ub[3][3];                                     // [c^, a^_1, a^_2][u]
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      ub[q][0] = (B.basis[q][0] - B.basis[q][1]) * r2;
      ub[q][1] = (B.basis[q][2] - B.basis[q][3]) * r2;
      ub[q][2] = 0.5 * (B.basis[q][0] + B.basis[q][1] - B.basis[q][2] - B.basis[q][3]);
    }
    const V3 e0 = Y[1] - Y[0], e1 = Y[3] - Y[2];
    const double s00 = dot(e0, e0), s11 = dot(e1, e1), s01 = dot(e0, e1);
    const double E0[3] = {e0.x, e0.y, e0.z}, E1[3] = {e1.x, e1.y, e1.z};
    const double rh[3] = {B.rh.x, B.rh.y, B.rh.z};
    // gradients of c and of kappa b, component (u, k) at 3 u + k (e_0 = -sqrt 2 of the u_1 motion,
    // e_1 of u_2)
    double gc[9], gb[9];
    const double gs = A.kappa * B.b1 * B.cn;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      gc[q] = -4.0 * r2 * (s11 * E0[q] - s01 * E1[q]);
      gc[3 + q] = -4.0 * r2 * (s00 * E1[q] - s01 * E0[q]);
      gc[6 + q] = 0.0;
#pragma unroll
      for (int u = 0; u < 3; ++u) gb[3 * u + q] = gs * ub[0][u] * rh[q];
    }
    // column me of m H_b + kb (m2 gc gc^T + m1 H_c) + m1 (gb gc^T + gc gb^T)
    const int mu = m_e / 3, mk = m_e - 3 * mu;
    const double cu = mu == 0 ? ub[0][0] : (mu == 1 ? ub[0][1] : ub[0][2]);
    const double a1u = mu == 0 ? ub[1][0] : (mu == 1 ? ub[1][1] : ub[1][2]);
    const double a2u = mu == 0 ? ub[2][0] : (mu == 1 ? ub[2][1] : ub[2][2]);
    const double rk = select_d(rh, mk), gcm = select_d(gc, m_e), gbm = select_d(gb, m_e);
    const double E0m = select_d(E0, mk), E1m = select_d(E1, mk);
    double y[5];
#pragma unroll
    for (int p = 0; p < 5; ++p) {
      const double kp = mk == 0 ? B.K[p][0] : (mk == 1 ? B.K[p][1] : B.K[p][2]);
      y[p] = kp * cu + (B.K[p][3] * a1u + B.K[p][4] * a2u) * rk;
    }
    double T[9], V[9];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const double yr = ub[1][u] * y[3] + ub[2][u] * y[4];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        double hc = 0.0;                                 // second derivatives of c, in (e_0, e_1)
        const double dl = q == mk ? 1.0 : 0.0;
        if (u < 2 && mu < 2) {
          if (u == 0) hc = mu == 0 ? 2.0 * (s11 * dl - E1[q] * E1m) : 4.0 * E0[q] * E1m - 2.0 * E1[q] * E0m - 2.0 * s01 * dl;
          else hc = mu == 1 ? 2.0 * (s00 * dl - E0[q] * E0m) : 4.0 * E1[q] * E0m - 2.0 * E0[q] * E1m - 2.0 * s01 * dl;
          hc *= 2.0;
        }
        const int r = 3 * u + q;
        const double hb = ub[0][u] * y[q] + rh[q] * yr;
        T[r] = m * hb + kb * (m2 * gc[r] * gcm + m1 * hc) + m1 * (gb[r] * gcm + gc[r] * gbm);
        V[r] = r == m_e ? 1.0 : 0.0;
      }
    }
    if (A.project) {
      double fro = 0.0;
#pragma unroll
      for (int r = 0; r < 9; ++r) fro += T[r] * T[r];
      double tot = 0.0;
#pragma unroll
      for (int q = 0; q < 9; ++q) tot += shfl_d(fro, first + q);
      const double tol = 1e-28 * tot;
      for (int sweep = 0; sweep < 30; ++sweep) {
        double off = 0.0;
#pragma unroll
        for (int r = 0; r < 9; ++r) off += r == m_e ? 0.0 : T[r] * T[r];
        double all = 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) all += shfl_d(off, first + q);
        // each pair stops by itself: the list's order, and so its neighbours in the warp, differ from
        // call to call
        const bool on = 0.5 * all > tol;
        if (!__any_sync(0xffffffffu, on)) break;
        jacobi9_round<0>(T, V, m_e, first, on); jacobi9_round<1>(T, V, m_e, first, on); jacobi9_round<2>(T, V, m_e, first, on);
        jacobi9_round<3>(T, V, m_e, first, on); jacobi9_round<4>(T, V, m_e, first, on); jacobi9_round<5>(T, V, m_e, first, on);
        jacobi9_round<6>(T, V, m_e, first, on); jacobi9_round<7>(T, V, m_e, first, on); jacobi9_round<8>(T, V, m_e, first, on);
      }
      // column me of V max(Lambda, 0) V^T: sum over e of V[:, e] lambda_e V[me][e]
      const double lam = select_d(T, m_e), lp = lam > 0.0 ? lam : 0.0;
      __syncwarp();
      if (live_lane) {
#pragma unroll
        for (int r = 0; r < 9; ++r) sh.H[9 * m_e + r] = V[r];
        sh.g[m_e] = lp;
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < 9; ++r) T[r] = 0.0;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const double s = sh.g[q] * sh.H[9 * q + m_e];
#pragma unroll
        for (int r = 0; r < 9; ++r) T[r] = fma(s, sh.H[9 * q + r], T[r]);
      }
    }
    __syncwarp();
    const int n = A.item_n[k];
    const int32_t* nodes = A.item_nodes + kMaxNodes * k;
    const uint64_t map = A.item_map[k];
    if (live_lane) {
#pragma unroll
      for (int r = 0; r < 9; ++r) sh.H[9 * m_e + r] = T[r];
      sh.g[m_e] = m * gbm + kb * m1 * gcm;
      for (int u = m_e; u < n; u += 9) {
        double wa[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          wa[a] = 0.0;
          if (A.T.vkin[v[a]]) continue;
          for (int q = 0; q < 4; ++q)
            if ((int)((map >> (16 * a + 4 * q)) & 15u) == u) wa[a] += __ldg(A.w + 4 * (int64_t)v[a] + q);
        }
        sh.W[0][u] = (wa[0] - wa[1]) * r2;
        sh.W[1][u] = (wa[2] - wa[3]) * r2;
        sh.W[2][u] = 0.5 * (wa[0] + wa[1] - wa[2] - wa[3]);
      }
    }
    __syncwarp();
    if (live_lane) {
      for (int u = 0; u < n; ++u)                        // row me of H times node u's weights
#pragma unroll
        for (int q = 0; q < 3; ++q)
          sh.HW[u][3 * m_e + q] = sh.W[0][u] * sh.H[9 * q + m_e] + sh.W[1][u] * sh.H[9 * (3 + q) + m_e] +
                                  sh.W[2][u] * sh.H[9 * (6 + q) + m_e];
    }
    __syncwarp();
    if (live) {
      if (m_e == 0) A.item_E[k] = m * kb;
      const int64_t oh = A.ro_h[k];
      const int nrec = n * (n + 1) / 2;
      for (int l = m_e; l < nrec; l += 9) {
        int u = 0, before = 0;
        while (before + (n - u) <= l) { before += n - u; ++u; }
        const int w2 = u + (l - before);
        if (oh + l >= A.rec_cap) break;
        double Bk[3][3];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
          for (int q = 0; q < 3; ++q)
            Bk[p][q] = sh.W[0][u] * sh.HW[w2][3 * p + q] + sh.W[1][u] * sh.HW[w2][3 * (3 + p) + q] +
                       sh.W[2][u] * sh.HW[w2][3 * (6 + p) + q];
        if (w2 == u) {
          double gr[3];                                  // the diagonal record carries the gradient at node u
#pragma unroll
          for (int q = 0; q < 3; ++q) gr[q] = sh.W[0][u] * sh.g[q] + sh.W[1][u] * sh.g[3 + q] + sh.W[2][u] * sh.g[6 + q];
          emit_diag(A, oh + l, Bk, gr[0], gr[1], gr[2]);
        } else {
          emit_upper(A, oh + l, nodes[u], nodes[w2], Bk);
        }
      }
    }
    __syncwarp();
  }
}

// sums over a warp by a fixed shuffle tree (the result in lane 0)
template <int W>
__device__ __forceinline__ void warp_tree_sum(double acc[W]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < W; ++c) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], o);
}

// ------------------------------------------------------------------ Hessian-vector product
// out = J^T H u for the unprojected contact Hessian H and the full-space direction u = J v on the
// embedded vertices, u = kin_dir on the kinematic ones (Sec. III-D, Eq. 17).
//
// Each item's y = H_k u is twelve numbers on its four vertices, in closed form (no 12 x 12 matrix,
// no eigensolve, about 110 FP64 instructions); they are added per vertex, and J^T is applied once
// per vertex instead of once per item and cage node.  The sum over items has to be the same bits
// on every run without sorting records: every component of every vertex keeps the largest exponent
// E among its contributions (an integer maximum), and each contribution is added to it as a
// fixed-point number of 2 kFix = 68 bits below 2^(E+1), in two 64-bit integers of 34 bits each
// (headroom for 2^29 items, the most a scene takes).  Integer sums do not depend on their order, and
// a contribution loses less than 2^-67 of the component's largest, where an addition in FP64 loses up
// to 2^-53 of the sum.  Infinite and NaN contributions (whose sum has no order either) are added as
// they are.  The sums then become doubles where the static lists of each node's vertices gather them, a
// warp per node in a fixed order.  Before: 1.24 M keyed records of the bubble grasp written,
// radix-sorted and summed, 23 launches, 443 us; now 6 launches, 162 us.
constexpr int kKinSlots = 64;          // partial sums over the kinematic vertices
constexpr int kFix = 34;               // bits per fixed-point limb
static_assert(kFix + 29 <= 63, "2^29 contributions below 2^kFix fit a limb's sum");

__device__ __forceinline__ V3 load_dir(const double* __restrict__ v, int32_t node) {
  return {v[3 * (int64_t)node], v[3 * (int64_t)node + 1], v[3 * (int64_t)node + 2]};
}

// u = J v (kin on the kinematic vertices), padded, and the vertices' sums reset
__global__ void __launch_bounds__(kBlock) k_hvp_direction(int64_t nv, const int32_t* __restrict__ idx,
                                                          const double* __restrict__ w, const double* __restrict__ dir,
                                                          V3 kin, double* __restrict__ u4, int32_t* __restrict__ vexp,
                                                          unsigned long long* __restrict__ hi, unsigned long long* __restrict__ lo,
                                                          CounterList zero) {
  pdl_entry();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int c = 0; c < kCounterList; ++c)
      if (zero.p[c]) *zero.p[c] = 0;
  }
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += grid_stride()) {
    const int4 id = __ldg(reinterpret_cast<const int4*>(idx) + v);
    V3 r = kin;
    if (id.x >= 0) {
      const double2 w01 = __ldg(reinterpret_cast<const double2*>(w) + 2 * v);
      const double2 w23 = __ldg(reinterpret_cast<const double2*>(w) + 2 * v + 1);
      r = load_dir(dir, id.x) * w01.x + load_dir(dir, id.y) * w01.y + load_dir(dir, id.z) * w23.x + load_dir(dir, id.w) * w23.y;
    }
    reinterpret_cast<double2*>(u4)[2 * v] = make_double2(r.x, r.y);
    reinterpret_cast<double2*>(u4)[2 * v + 1] = make_double2(r.z, 0.0);
    reinterpret_cast<int4*>(vexp)[v] = make_int4(0, 0, 0, 0);
    reinterpret_cast<ulonglong2*>(hi)[2 * v] = make_ulonglong2(0, 0);
    reinterpret_cast<ulonglong2*>(hi)[2 * v + 1] = make_ulonglong2(0, 0);
    reinterpret_cast<ulonglong2*>(lo)[2 * v] = make_ulonglong2(0, 0);
    reinterpret_cast<ulonglong2*>(lo)[2 * v + 1] = make_ulonglong2(0, 0);
  }
}

struct HvpArgs {
  Topo T;
  eipc_pairs pr;
  eipc_lag lag;
  bool friction;
  const double* x4;
  const float* x4f;
  const double* u4;
  double dhat, inv_dhat, kappa, mu, eps_f;
  const double* moll_r2;
  double moll_factor;
  int64_t item_cap;
  double* y;                 // [12 * items]
  int32_t* vexp;             // [4 nv] largest exponent_of the contributions to each component of a vertex
  unsigned long long* hi;    // [4 nv] fixed-point sums, upper and lower limbs
  unsigned long long* lo;
  uint32_t* rest;            // pairs left to k_hvp_rest, mollified pairs left to k_hvp_mollified
  int64_t* n_rest;
  uint32_t* moll_list;
  int64_t* n_moll;
  DevStatus* st;
};

// biased exponent of x, 1 where x is subnormal, 0 for zeros, 0x7ff for infinities and NaN
__device__ __forceinline__ int32_t exponent_of(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  return (int32_t)max((hi >> 20) & 0x7ffu, min((hi << 1) | lo, 1u));
}

__device__ __forceinline__ void hvp_store(const HvpArgs& A, int64_t k, int slot, int32_t v, V3 y) {
  double* row = A.y + 12 * k + 3 * slot;
  row[0] = y.x; row[1] = y.y; row[2] = y.z;
  int32_t* held = A.vexp + 4 * (int64_t)v;
  const int4 h = __ldcg(reinterpret_cast<const int4*>(held));
  const int32_t ex = exponent_of(y.x), ey = exponent_of(y.y), ez = exponent_of(y.z);
  if (ex > h.x) atomicMax(held, ex);
  if (ey > h.y) atomicMax(held + 1, ey);
  if (ez > h.z) atomicMax(held + 2, ez);
}

// y of a pair whose closest feature is a segment of `hint`
__device__ __forceinline__ void hvp_light(const HvpArgs& A, int64_t k, int type, const int32_t v[4], int hint) {
  V3 X[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) X[a] = load_x(A.x4, v[a]);
  const SegmentPair G = closest_segment(type, X, hint);
  const double d2 = dot(G.r, G.r);
  const V3 zero = {0.0, 0.0, 0.0};
  V3 fc = zero, fa = zero;
  if (!(d2 > 0.0)) {
    raise_flag(A.st, EIPC_FLAG_PENETRATION);
  } else {
    const double inv_d = rsqrt(d2), d = d2 * inv_d;
    if (lt_nonneg(d, A.dhat)) {
      double b, b1, b2;
      barrier_scalars(d, inv_d, A.dhat, A.inv_dhat, &b, &b1, &b2);
      const double bd = -A.kappa * (b1 * inv_d);               // -kappa b'/d
      const V3 rh = G.r * inv_d;
      const V3 up = load_x(A.u4, pick(v, G.ip)), ua = load_x(A.u4, pick(v, G.ia)), ub = load_x(A.u4, pick(v, G.ib));
      const V3 ul = ua - ub, uc = up - ua + ul * G.t;          // sum alpha_a u_a, sum c_a u_a
      fc = rh * (fma(A.kappa, b2, bd) * dot(rh, uc)) - uc * bd;
      if (G.inner) {
        // -(kappa b'/(2d)) G M^-1 G^T with G = 2 (c (x) v + alpha (x) r), v = -e, M = 2 |e|^2
        const double s = bd * (G.rse * G.rse) * (dot(G.r, ul) - dot(G.e, uc));
        fc = fc - G.e * s;
        fa = G.r * s;
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    V3 y = zero;
    if (a == G.ip) y = fc;
    if (a == G.ia) y = fa - fc * (1.0 - G.t);
    if (a == G.ib) y = zero - fa - fc * G.t;
    hvp_store(A, k, a, v[a], y);
  }
}

// ... of any pair
__device__ __forceinline__ void hvp_heavy(const HvpArgs& A, int64_t k) {
  int32_t v[4];
  const int type = A.pr.type[k];
  stencil_vertices(A.T, type, A.pr.i[k], A.pr.j[k], v);
  V3 Y[4], u[4];
  const V3 X0 = load_x(A.x4, v[0]);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    Y[a] = load_x(A.x4, v[a]) - X0;
    u[a] = load_x(A.u4, v[a]);
  }
  Stencil S;
  closest_pair<true>(type, Y, stencil_hint(type, A.x4f, v), &S);
  const V3 zero = {0.0, 0.0, 0.0};
  V3 fc = zero, fa[2] = {zero, zero};
  if (!(S.d2 > 0.0)) {
    raise_flag(A.st, EIPC_FLAG_PENETRATION);
  } else {
    const double inv_d = rsqrt(S.d2), d = S.d2 * inv_d;
    if (lt_nonneg(d, A.dhat)) {
      double b, b1, b2;
      barrier_scalars(d, inv_d, A.dhat, A.inv_dhat, &b, &b1, &b2);
      const double bd = -A.kappa * (b1 * inv_d);
      V3 r = zero, uc = zero, ul[2] = {zero, zero}, vj[2] = {zero, zero};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        r = r + Y[a] * S.c[a];
        uc = uc + u[a] * S.c[a];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          ul[q] = ul[q] + u[a] * S.a[q][a];
          vj[q] = vj[q] + Y[a] * S.a[q][a];
        }
      }
      const V3 rh = r * inv_d;
      fc = rh * (fma(A.kappa, b2, bd) * dot(rh, uc)) - uc * bd;
      if (S.m > 0) {
        // s_j of bd M'^-1 g with M' = [v_j . v_l], g_j = v_j . u_c + r . u_j
        const double g0 = dot(vj[0], uc) + dot(r, ul[0]), g1 = dot(vj[1], uc) + dot(r, ul[1]);
        const double m00 = dot(vj[0], vj[0]);
        double s0 = 0.0, s1 = 0.0;
        if (S.m == 1) {
          s0 = bd * g0 / m00;
        } else {
          const double m01 = dot(vj[0], vj[1]), m11 = dot(vj[1], vj[1]);
          const double q = bd / (m00 * m11 - m01 * m01);
          s0 = q * (m11 * g0 - m01 * g1);
          s1 = q * (m00 * g1 - m01 * g0);
        }
        fc = fc + vj[0] * s0 + vj[1] * s1;
        fa[0] = r * s0;
        fa[1] = r * s1;
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) hvp_store(A, k, a, v[a], fc * S.c[a] + fa[0] * S.a[0][a] + fa[1] * S.a[1][a]);
}

__device__ __forceinline__ void hvp_friction(const HvpArgs& A, int64_t k, int64_t f) {
  const int4 q4 = reinterpret_cast<const int4*>(A.lag.v)[f];
  const int32_t v[4] = {q4.x, q4.y, q4.z, q4.w};
  FrictionTerms R;
  double gam[4];
  friction_terms(A.x4, A.lag, f, v, A.mu, A.eps_f, R, gam);
  V3 s = {0.0, 0.0, 0.0};
#pragma unroll
  for (int a = 0; a < 4; ++a) s = s + load_x(A.u4, v[a]) * gam[a];
  const V3 Fs = {R.F[0][0] * s.x + R.F[0][1] * s.y + R.F[0][2] * s.z, R.F[1][0] * s.x + R.F[1][1] * s.y + R.F[1][2] * s.z,
                 R.F[2][0] * s.x + R.F[2][1] * s.y + R.F[2][2] * s.z};
#pragma unroll
  for (int a = 0; a < 4; ++a) hvp_store(A, k, a, v[a], Fs * gam[a]);
}

// whether pair k is active and mollified (then Y, eps, c are its offsets and mollifier arguments)
__device__ __forceinline__ bool hvp_is_mollified(const HvpArgs& A, int type, int32_t i, int32_t j, const int32_t v[4], V3 Y[4],
                                                 double* eps, double* c) {
  if (!A.moll_r2 || type != 1) return false;
  const V3 X0 = load_x(A.x4, v[0]);
#pragma unroll
  for (int a = 0; a < 4; ++a) Y[a] = load_x(A.x4, v[a]) - X0;
  const V3 nn = cross(Y[1] - Y[0], Y[3] - Y[2]);
  *c = dot(nn, nn);
  *eps = A.moll_factor * A.moll_r2[i] * A.moll_r2[j];
  if (!(*c < *eps)) return false;
  const double d2 = closest_pair<false>(1, Y, stencil_hint(1, A.x4f, v), nullptr);
  return d2 > 0.0 && sqrt(d2) < A.dhat;
}

// a mollified EE pair: its full 12 x 12 Hessian
__device__ __forceinline__ void hvp_mollified(const HvpArgs& A, int64_t k) {
  int32_t v[4];
  const int32_t i = A.pr.i[k], j = A.pr.j[k];
  stencil_vertices(A.T, 1, i, j, v);
  V3 Y[4];
  double eps, c;
  if (!hvp_is_mollified(A, 1, i, j, v, Y, &eps, &c)) return;
  Stencil S;
  ee_distance<true>(Y[0], Y[1], Y[2], Y[3], &S);
  double g12[12], H12[144], E;
  mollified_local(Y, S, sqrt(S.d2), A.dhat, A.kappa, eps, c, &E, g12, H12);
  double u12[12];
  for (int a = 0; a < 4; ++a) {
    const V3 u = load_x(A.u4, v[a]);
    u12[3 * a] = u.x; u12[3 * a + 1] = u.y; u12[3 * a + 2] = u.z;
  }
  for (int a = 0; a < 4; ++a) {
    double y[3];
    for (int q = 0; q < 3; ++q) {
      double acc = 0.0;
      for (int p = 0; p < 12; ++p) acc += H12[12 * (3 * a + q) + p] * u12[p];
      y[q] = acc;
    }
    hvp_store(A, k, a, v[a], V3{y[0], y[1], y[2]});
  }
}

// appends k to a list (one atomic per warp)
__device__ __forceinline__ void list_append(bool mine, int64_t k, uint32_t* list, int64_t* n) {
  const unsigned m = __ballot_sync(0xffffffffu, mine);
  if (!m) return;
  const int lane = threadIdx.x & 31;
  unsigned long long b = 0;
  if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(n), (unsigned long long)__popc(m));
  b = __shfl_sync(0xffffffffu, b, 0);
  if (mine) list[(int64_t)b + __popc(m & ((1u << lane) - 1u))] = (uint32_t)k;
}

// y of every item but the pairs it lists: those with an interior closest point (as in
// k_eval_factors) and mollified ones
__global__ void __launch_bounds__(kEvalThreads, 4) k_hvp_items(HvpArgs A) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  const int64_t P = clamp_count(A.pr.count, A.pr.capacity);
  const int64_t L = A.friction ? clamp_count(A.lag.count, A.lag.capacity) : 0;
  const int64_t n = P + L < A.item_cap ? P + L : A.item_cap;
  if (P + L > A.item_cap && blockIdx.x == 0 && threadIdx.x == 0) raise_flag(A.st, EIPC_FLAG_REC_OVERFLOW);
  const int64_t np = P < n ? P : n;
  const int width = items_per_warp(n, 4);
  const int64_t stride = (int64_t)gridDim.x * (blockDim.x >> 5) * width;
  for (int64_t base = (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * width; base < n; base += stride) {
    const int64_t k = base + lane;
    bool rest = false, moll = false;
    const bool mine = lane < width;
    if (mine && k < np) {
      int32_t v[4];
      const int type = A.pr.type[k];
      const int32_t i = A.pr.i[k], j = A.pr.j[k];
      stencil_vertices(A.T, type, i, j, v);
      V3 Y[4];
      double eps, c;
      moll = hvp_is_mollified(A, type, i, j, v, Y, &eps, &c);
      if (!moll) {
        const int hint = stencil_hint(type, A.x4f, v);
        if (hint & kHintInterior) rest = true;
        else hvp_light(A, k, type, v, hint);
      }
    } else if (mine && k < n) {
      hvp_friction(A, k, k - P);
    }
    list_append(rest, k, A.rest, A.n_rest);
    if (A.n_moll) list_append(moll, k, A.moll_list, A.n_moll);
  }
}

__global__ void __launch_bounds__(kEvalThreads) k_hvp_rest(HvpArgs A) {
  pdl_entry();
  const int64_t n = *A.n_rest;
  const int lane = threadIdx.x & 31, width = items_per_warp(n);
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t w = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); w * width < n; w += nw) {
    const int64_t q = w * width + lane;
    if (lane < width && q < n) hvp_heavy(A, A.rest[q]);
  }
}

__global__ void __launch_bounds__(kEvalThreads) k_hvp_mollified(HvpArgs A) {
  pdl_entry();
  const int64_t n = *A.n_moll;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += grid_stride()) hvp_mollified(A, A.moll_list[q]);
}

// adds y / 2^(E - 1022) as a fixed-point number: kFix bits in hi, the next kFix in lo; where a
// contribution is not finite, those that are not as they are, in hi as a double
__device__ __forceinline__ void add_fixed(unsigned long long* hi, unsigned long long* lo, double y, int32_t E) {
  const long long b = __double_as_longlong(y);
  if (E == 0x7ff) {
    if (!finite_bits(y)) atomicAdd(reinterpret_cast<double*>(hi), y);
    return;
  }
  int32_t e = (int32_t)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (e > 0) m |= 1ull << 52;
  else e = 1;
  if (m == 0) return;
  const int sh = 2 * kFix - 53 - (E - e);      // value = m 2^sh in units of 2^(-2 kFix)
  const int down = kFix - sh;
  unsigned long long h = down < 64 ? m >> down : 0;
  unsigned long long l = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0);
  l &= (1ull << kFix) - 1;
  if (b < 0) { h = 0ull - h; l = 0ull - l; }
  if (h) atomicAdd(hi, h);
  if (l) atomicAdd(lo, l);
}

__global__ void __launch_bounds__(kBlock) k_hvp_accumulate(HvpArgs A) {
  pdl_entry();
  const int64_t P = clamp_count(A.pr.count, A.pr.capacity);
  const int64_t L = A.friction ? clamp_count(A.lag.count, A.lag.capacity) : 0;
  const int64_t n = P + L < A.item_cap ? P + L : A.item_cap;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 4 * n; t += grid_stride()) {
    const int64_t k = t >> 2;
    const int a = (int)(t & 3);
    int32_t v[4];
    item_vertices(A.T, A.pr, P, A.lag.v, L, k, v);
    const int32_t va = pick(v, a);
    const double* y = A.y + 3 * t;
    const double y0 = y[0], y1 = y[1], y2 = y[2];
    const int4 E = reinterpret_cast<const int4*>(A.vexp)[va];
    add_fixed(A.hi + 4 * (int64_t)va, A.lo + 4 * (int64_t)va, y0, E.x);
    add_fixed(A.hi + 4 * (int64_t)va + 1, A.lo + 4 * (int64_t)va + 1, y1, E.y);
    add_fixed(A.hi + 4 * (int64_t)va + 2, A.lo + 4 * (int64_t)va + 2, y2, E.z);
  }
}

// a fixed-point sum of contributions of largest exponent E as a double
__device__ __forceinline__ double from_fixed(long long hi, long long lo, int32_t E) {
  if (E == 0) return 0.0;
  if (E == 0x7ff) return __longlong_as_double(hi);
  // 2^(E - 1022 - kFix), subnormal below E = kFix
  const double scale = E >= kFix ? __hiloint2double((E - kFix + 1) << 20, 0) : __longlong_as_double(1ll << (E + 52 - kFix));
  const long long t = hi + (lo >> kFix), f = lo & ((1ll << kFix) - 1);
  return fma((double)f, 1.0 / (double)(1ll << kFix), (double)t) * scale;
}

// Rows of J^T: warp r < ns gathers node r's vertices, the next kKinSlots warps a share of the
// kinematic ones each (weight one); the last of these to finish adds the shares in order.
__global__ void __launch_bounds__(kBlock) k_hvp_gather(int64_t ns, const int64_t* __restrict__ inc_ptr,
                                                       const uint32_t* __restrict__ inc, const double* __restrict__ w,
                                                       const int32_t* __restrict__ vexp, const long long* __restrict__ hi,
                                                       const long long* __restrict__ lo, double* __restrict__ out_r,
                                                       double* __restrict__ out_kin, double* part, int64_t* ticket) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t rows = ns + (out_kin ? kKinSlots : 0);
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < rows; r += nw) {
    const bool kin = r >= ns;
    int64_t b = inc_ptr[kin ? ns : r], e = inc_ptr[(kin ? ns : r) + 1];
    if (kin) {
      const int64_t per = (e - b + kKinSlots - 1) / kKinSlots, b0 = b + per * (r - ns);
      e = b0 + per < e ? b0 + per : e;
      b = b0;
    }
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int64_t q = b + lane; q < e; q += 32) {
      const uint32_t t = inc[q];
      const int64_t v = t >> 2;
      const int4 E = reinterpret_cast<const int4*>(vexp)[v];
      if ((E.x | E.y | E.z) == 0) continue;
      const longlong2 h01 = *reinterpret_cast<const longlong2*>(hi + 4 * v), l01 = *reinterpret_cast<const longlong2*>(lo + 4 * v);
      const double ww = kin ? 1.0 : w[t];
      a0 = fma(ww, from_fixed(h01.x, l01.x, E.x), a0);
      a1 = fma(ww, from_fixed(h01.y, l01.y, E.y), a1);
      a2 = fma(ww, from_fixed(hi[4 * v + 2], lo[4 * v + 2], E.z), a2);
    }
    if (__any_sync(0xffffffffu, a0 != 0.0 || a1 != 0.0 || a2 != 0.0)) {
      double acc[3] = {a0, a1, a2};
      warp_tree_sum<3>(acc);
      a0 = acc[0]; a1 = acc[1]; a2 = acc[2];
    }
    if (!kin) {
      if (lane == 0) { out_r[3 * r] = a0; out_r[3 * r + 1] = a1; out_r[3 * r + 2] = a2; }
      continue;
    }
    int64_t done = 0;
    if (lane == 0) {
      double* p = part + 3 * (r - ns);
      p[0] = a0; p[1] = a1; p[2] = a2;
      __threadfence();
      done = (int64_t)atomicAdd(reinterpret_cast<unsigned long long*>(ticket), 1ull);
    }
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done == kKinSlots - 1) {
      __threadfence();
      double acc[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[c] = __ldcg(part + 3 * lane + c) + __ldcg(part + 3 * (lane + 32) + c);
      warp_tree_sum<3>(acc);
      if (lane == 0)
        for (int c = 0; c < 3; ++c) out_kin[c] = acc[c];
    }
  }
}

// Record totals -> overflow flags and clamped counts.  After an overflow the items whose factor rows
// end past gcap, or whose explicit records (mollifier) would end past rec_cap, are taken as items
// without nodes: no kernel writes rows or records for them and none sums any, so the flag and their
// missing shares are all that is left of them (their energies are still summed).  Decided here,
// before the items are read, rather than at each of k_chunk_sums' reads, which it would slow down.
__global__ void __launch_bounds__(kRecCheckThreads) k_rec_check(const int64_t* rh_total, const int64_t* rg_total,
                                                                int64_t rec_cap, int64_t gcap, int64_t* n_rh,
                                                                int64_t* n_rg, DevStatus* st, const int64_t* n_items,
                                                                const int64_t* __restrict__ ro_h,
                                                                const int64_t* __restrict__ ro_g,
                                                                int32_t* __restrict__ item_n, bool records) {
  pdl_entry();
  const int64_t a = *rh_total, b = *rg_total;
  if (threadIdx.x == 0) {
    if (a > rec_cap || b > gcap) {
      raise_flag(st, EIPC_FLAG_REC_OVERFLOW);
      raise_need(st, &st->need_rec, a > b ? a : b);
    }
    *n_rh = a < rec_cap ? a : rec_cap;
    *n_rg = b < gcap ? b : gcap;
  }
  if (b <= gcap && (!records || a <= rec_cap)) return;
  const int64_t n = *n_items;
  for (int64_t k = threadIdx.x; k < n; k += kRecCheckThreads) {
    const int64_t m = item_n[k];
    if (ro_g[k] + m > gcap || (records && ro_h[k] + m * (m + 1) / 2 > rec_cap)) item_n[k] = 0;
  }
}

// every upper block (I, J) becomes the full-pattern entry (I, J) and, off the diagonal,
// the transposed entry (J, I); diagonal blocks get a sentinel twin that sorts last.  Entry
// keys are row | col << br (br a whole number of radix digits): the upper blocks arrive in
// (I, J) order, so every transposed
// entry (r, I) of a row r (I < r) precedes the row's own upper entries, in increasing I;
// a stable sort on the row bits alone then leaves each row's columns increasing.
__global__ void __launch_bounds__(kBlock) k_full_entries(const uint64_t* __restrict__ ukey, const int64_t* n_seg,
                                                         int64_t ns, int br, int64_t cap,
                                                         uint64_t* __restrict__ fkey, uint32_t* __restrict__ fval,
                                                         int64_t* n_full_sort, int64_t* n_diag, DevStatus* st,
                                                         int32_t* __restrict__ dst) {
  pdl_entry();
  const int64_t S0 = *n_seg;
  const int64_t S = (2 * S0 <= cap) ? S0 : cap / 2;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *n_full_sort = 2 * S;
    if (S < S0) raise_flag(st, EIPC_FLAG_REC_OVERFLOW);
  }
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S; s += grid_stride()) {
    const uint64_t key = ukey[s];
    uint64_t I, J;
    upper_decode(key, (uint64_t)ns, &I, &J);
    fkey[2 * s] = I | (J << br);
    fval[2 * s] = (uint32_t)(s << 1);
    if (I != J) {
      fkey[2 * s + 1] = J | (I << br);
      fval[2 * s + 1] = (uint32_t)((s << 1) | 1);
    } else {
      fkey[2 * s + 1] = (1ull << br) - 1;           // row bits above every row: sorts last
      fval[2 * s + 1] = 0;
      dst[2 * s + 1] = -2;                          // marks a diagonal segment
      atomicAdd(reinterpret_cast<unsigned long long*>(n_diag), 1ull);
    }
  }
}

// ---- records.  Items with the same nodes -- 171k of the full bubble grasp have 9.7k node sets
// between them -- are summed together before anything is sorted by block: sorted by key, a run of
// items with equal nodes is a group, cut into chunks of kChunk items from its own start; a record is
// one upper block (u, v) of a chunk.  2.57 M item records become about 0.35 M.  Group and chunk
// borders depend only on the scene's own items, so sums are the same bits alone or in a batch.
constexpr int kChunk = 16;

// whether sorted item i starts a group (two sets with one key and hash part here as well)
__device__ __forceinline__ bool group_head(int64_t i, const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                           const int32_t* __restrict__ item_n, const int32_t* __restrict__ item_nodes) {
  if (i == 0 || keys[i] != keys[i - 1]) return true;
  const int64_t a = vals[i], b = vals[i - 1];
  const int n = item_n[a];
  if (n != item_n[b]) return true;
  const int4* p = reinterpret_cast<const int4*>(item_nodes + kMaxNodes * a);
  const int4* q = reinterpret_cast<const int4*>(item_nodes + kMaxNodes * b);
  for (int u = 0; u < n; u += 4) {
    const int4 x = p[u / 4], y = q[u / 4];
    if (x.x != y.x || (u + 1 < n && x.y != y.y) || (u + 2 < n && x.z != y.z) || (u + 3 < n && x.w != y.w)) return true;
  }
  return false;
}

__global__ void __launch_bounds__(256) k_group_count(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                                     const int64_t* n_items, const int32_t* __restrict__ item_n,
                                                     const int32_t* __restrict__ item_nodes, int64_t* __restrict__ partial) {
  pdl_entry();
  __shared__ int wsum[8];
  const int64_t n = *n_items, per = (n + gridDim.x - 1) / gridDim.x, b = blockIdx.x * per, e = b + per < n ? b + per : n;
  int c = 0;
  for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) c += group_head(i, keys, vals, item_n, item_nodes);
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < 8; ++w) t += wsum[w];
    partial[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(256) k_group_start(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                                                     const int64_t* n_items, const int32_t* __restrict__ item_n,
                                                     const int32_t* __restrict__ item_nodes,
                                                     const int64_t* __restrict__ partial, int64_t* n_groups,
                                                     int64_t* __restrict__ start) {
  pdl_entry();
  __shared__ int32_t wsum[8];
  const int64_t n = *n_items, per = (n + gridDim.x - 1) / gridDim.x, b = blockIdx.x * per, e = b + per < n ? b + per : n;
  int64_t all_groups;
  int64_t run = partials_before(partial, blockIdx.x, &all_groups);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (blockIdx.x == 0 && t == 0) *n_groups = all_groups;
  for (int64_t tile = b; tile < e; tile += 256) {
    const int64_t i = tile + t;
    const bool h = i < e && group_head(i, keys, vals, item_n, item_nodes);
    const unsigned m = __ballot_sync(0xffffffffu, h);
    if (lane == 0) wsum[warp] = __popc(m);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      before += w < warp ? wsum[w] : 0;
      all += wsum[w];
    }
    if (h) start[run + before + __popc(m & ((1u << lane) - 1u))] = i;
    __syncthreads();
    run += all;
  }
}

// records per group (none for the items without nodes, which end the order)
__global__ void __launch_bounds__(kBlock) k_group_records(const int64_t* __restrict__ start, const int64_t* n_groups,
                                                          const int64_t* n_items, const uint32_t* __restrict__ vals,
                                                          const int32_t* __restrict__ item_n, int64_t* __restrict__ count) {
  pdl_entry();
  const int64_t G = *n_groups, N = *n_items;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < G; g += grid_stride()) {
    const int64_t b = start[g], e = g + 1 < G ? start[g + 1] : N;
    const int n = item_n[vals[b]];
    count[g] = (e - b + kChunk - 1) / kChunk * (n * (n + 1) / 2);
  }
}

// Keys of the chunk records, and their source: first sorted item of the chunk, items - 1, local
// node of the row and of the column.  One warp per group.
__global__ void __launch_bounds__(kBlock) k_rec_keys(const int64_t* __restrict__ start, const int64_t* n_groups,
                                                     const int64_t* n_items, const uint32_t* __restrict__ vals,
                                                     const int32_t* __restrict__ item_n, const int32_t* __restrict__ item_nodes,
                                                     const int64_t* __restrict__ offset, int64_t rec_cap, int64_t ns,
                                                     uint64_t* __restrict__ hkeys, uint32_t* __restrict__ hvals,
                                                     uint64_t* __restrict__ rec_src) {
  pdl_entry();
  const int64_t G = *n_groups, N = *n_items;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < G; g += nw) {
    const int64_t b = start[g], e = g + 1 < G ? start[g + 1] : N, oh = offset[g];
    const int64_t item = vals[b];
    const int n = item_n[item];
    if (n == 0) continue;
    const int32_t* nodes = item_nodes + kMaxNodes * item;
    const int nrec = n * (n + 1) / 2;
    const int64_t all = (e - b + kChunk - 1) / kChunk * nrec;
    for (int64_t l = lane; l < all; l += 32) {
      const int64_t c = l / nrec;
      const int r = (int)(l - c * nrec);
      int u = 0, before = 0;                 // row u of the upper triangle holds n - u records
      while (before + (n - u) <= r) { before += n - u; ++u; }
      const int w2 = u + (r - before);
      const int64_t pos = oh + l;
      if (pos >= rec_cap) continue;
      const int64_t first = b + c * kChunk, left = e - first;
      hkeys[pos] = upper_key((uint64_t)nodes[u], (uint64_t)nodes[w2], (uint64_t)ns);
      hvals[pos] = (uint32_t)pos;
      rec_src[pos] = (uint64_t)first << 16 | (uint64_t)((left < kChunk ? left : kChunk) - 1) << 8 | (uint64_t)u << 4 | (uint64_t)w2;
    }
  }
}

// key of each segment (block) of the sorted records
__global__ void __launch_bounds__(kBlock) k_seg_keys(const int64_t* __restrict__ start, const int64_t* n_seg,
                                                     const uint64_t* __restrict__ keys, uint64_t* __restrict__ ukey) {
  pdl_entry();
  const int64_t S = *n_seg;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S; s += grid_stride()) ukey[s] = keys[start[s]];
}

// sorted full entries -> BSR columns, row counts, and for each upper segment s the BSR
// entry of its block (dst[2s]) and of its transpose (dst[2s+1]; -1 on the diagonal or
// beyond the capacity)
__global__ void __launch_bounds__(kBlock) k_bsr_pattern(const uint64_t* __restrict__ fkey, const uint32_t* __restrict__ fval,
                                                        const int64_t* n_full_sort, const int64_t* n_diag, int br,
                                                        int64_t ns, eipc_bsr H, int32_t* __restrict__ dst,
                                                        DevStatus* st, int64_t* __restrict__ n_gnodes) {
  pdl_entry();
  const int64_t nnzb = *n_full_sort - *n_diag;
  const uint64_t rmask = (1ull << br) - 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *H.nnzb = nnzb;
    *n_gnodes = *n_diag;           // nodes with a gradient: one diagonal block each
    if (nnzb > H.capacity) {
      raise_flag(st, EIPC_FLAG_BSR_OVERFLOW);
      raise_need(st, &st->need_bsr, nnzb);
    }
    if (nnzb == 0)
      for (int64_t r = 0; r <= ns; ++r) H.row_ptr[r] = 0;
  }
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnzb; e += grid_stride()) {
    const uint64_t key = fkey[e];
    const int64_t row = (int64_t)(key & rmask);
    // the entries are sorted by row: entry e starts every row after the previous entry's
    // row up to its own, and the last entry closes the rows after its own
    const int64_t prev = e > 0 ? (int64_t)(fkey[e - 1] & rmask) : -1;
    for (int64_t r = prev + 1; r <= row; ++r) H.row_ptr[r] = (int32_t)e;
    if (e == nnzb - 1)
      for (int64_t r = row + 1; r <= ns; ++r) H.row_ptr[r] = (int32_t)nnzb;
    const uint32_t v = fval[e];
    dst[2 * (int64_t)(v >> 1) + (v & 1u)] = e < H.capacity ? (int32_t)e : -1;
    if (e < H.capacity) H.col[e] = (int32_t)(key >> br);
  }
}

struct SumArgs {
  const uint64_t* src;        // sources of the records
  const int64_t* n_rec;
  int64_t cap;
  const uint32_t* items;      // items in group order
  const int64_t* ro_h;        // first explicit record of each item, its node count
  const int32_t* item_n;
  const int64_t* ro_g;
  const double* frow;
  const double* ihead;
  const double* hrec;
  double* piece;
};

__device__ __forceinline__ int sym_index(int p, int q) {   // (p, q) in B00 B01 B02 B11 B12 B22
  const int lo = p < q ? p : q, hi = p < q ? q : p;
  return lo * (5 - lo) / 2 + hi;
}

// The records' sums over their chunk's items, each block multiplied out of the item's factor rows
// (see "pair factors") into the accumulators.  Bound by the FP64 pipe: three lanes per record, lane
// i of them accumulating row i of the block -- 7 or 10 FP64 instructions per item (without or
// with friction), 30 of 32 lanes at work, neighbouring lanes on the same items.  In a diagonal
// record lane i takes entries (i, i) and (i, i + 1 mod 3) of the symmetric block and, in place of
// the third, component i of the gradient, with the same number of instructions.
__global__ void __launch_bounds__(128) k_chunk_sums(SumArgs A) {
  pdl_entry();
  const int64_t R = clamp_count(A.n_rec, A.cap);
  const int lane = threadIdx.x & 31, sub = lane / 3, i = lane - 3 * sub;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 10 < R; w += nw) {
    const int64_t r = w * 10 + sub;
    if (lane >= 30 || r >= R) continue;
    const uint64_t src = __ldg(A.src + r);
    const int lu = (int)((src >> 4) & 15), lv = (int)(src & 15), m = (int)((src >> 8) & 255) + 1;
    const uint32_t* items = A.items + (src >> 16);
    const bool diag = lu == lv;
    const int c0 = diag ? i : 0, c1 = diag ? (i == 2 ? 0 : i + 1) : 1;
    const int f0 = sym_index(i, c0), f1 = sym_index(i, c1), f2 = sym_index(i, 2);
    int64_t item = __ldg(items), base = __ldg(A.ro_g + item);
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int q = 0; q < m; ++q) {
      const double* ru = A.frow + kFRow * (base + lu);
      const double* rv = A.frow + kFRow * (base + lv);
      const double* hd = A.ihead + kIHead * item;
      const int64_t cur = item;
      if (q + 1 < m) {                       // the next item's rows are found while this one's arrive
        item = __ldg(items + q + 1);
        base = __ldg(A.ro_g + item);
      }
      const double2 hf = __ldg(reinterpret_cast<const double2*>(hd) + 6);
      const int flags = (int)__double_as_longlong(hf.y);
      if (flags & kItemExplicit) {
        const double* B = A.hrec + kHRecStride * (A.ro_h[cur] + lu * A.item_n[cur] - lu * (lu - 1) / 2 + lv - lu);
        a0 += diag ? B[f0] : B[3 * i];
        a1 += diag ? B[f1] : B[3 * i + 1];
        a2 += diag ? B[6 + i] : B[3 * i + 2];
        continue;
      }
      const double z1 = __ldg(ru + i), z2 = __ldg(ru + 3 + i);
      const double2 ou = __ldg(reinterpret_cast<const double2*>(ru) + 3);
      const double2 va = __ldg(reinterpret_cast<const double2*>(rv)), vb = __ldg(reinterpret_cast<const double2*>(rv) + 1);
      const double2 vc = __ldg(reinterpret_cast<const double2*>(rv) + 2), ov = __ldg(reinterpret_cast<const double2*>(rv) + 3);
      const double x0 = c0 == 0 ? va.x : (c0 == 1 ? va.y : vb.x), y0 = c0 == 0 ? vb.y : (c0 == 1 ? vc.x : vc.y);
      const double x1 = c1 == 0 ? va.x : (c1 == 1 ? va.y : vb.x), y1 = c1 == 0 ? vb.y : (c1 == 1 ? vc.x : vc.y);
      double p1 = z1, q1 = vb.x, p2 = z2, q2 = vc.y;
      if (diag) {
        p1 = ou.x; q1 = __ldg(hd + 6 + i);
        p2 = ou.y; q2 = __ldg(hd + 9 + i);
      }
      a0 = fma(z1, x0, a0); a1 = fma(z1, x1, a1); a2 = fma(p1, q1, a2);
      a0 = fma(z2, y0, a0); a1 = fma(z2, y1, a1); a2 = fma(p2, q2, a2);
      if (flags & kItemFriction) {
        const double ww = ou.y * ov.y;
        a0 = fma(ww, __ldg(hd + f0), a0);
        a1 = fma(ww, __ldg(hd + f1), a1);
        a2 = fma(ww, diag ? 0.0 : __ldg(hd + f2), a2);
      }
      if (flags & kItemThird) {
        const double z3 = __ldg(ru + 8 + i);
        a0 = fma(z3, __ldg(rv + 8 + c0), a0);
        a1 = fma(z3, __ldg(rv + 8 + c1), a1);
        a2 = fma(diag ? 0.0 : z3, __ldg(rv + 10), a2);
      }
      if (flags & kItemIso) {
        const double t = hf.x * (ou.x * ov.x);
        if (diag || i == 0) a0 += t;
        else if (i == 1) a1 += t;
        else a2 += t;
      }
    }
    double* p = A.piece + 9 * r + 3 * i;
    p[0] = a0; p[1] = a1; p[2] = a2;
  }
}

// The blocks, one warp per segment of the sorted records: lane 9 q + c adds component c of records
// q, q + 3, ... in order, then the three chains are added; the block goes into the BSR values at
// dst[2s] and, transposed, at dst[2s+1].  A diagonal segment (dst[2s+1] = -2) holds, per row i,
// entries (i, i) and (i, i + 1 mod 3) of its symmetric block and component i of the gradient at its
// node.
__global__ void __launch_bounds__(kBlock) k_segment_sums(const double* __restrict__ piece, const uint32_t* __restrict__ perm,
                                                         const int64_t* __restrict__ start, const int64_t* n_rec,
                                                         const int64_t* n_seg, int64_t cap,
                                                         const int32_t* __restrict__ dst, eipc_bsr H,
                                                         const uint64_t* __restrict__ ukey, int64_t ns,
                                                         double* __restrict__ g_r) {
  pdl_entry();
  const int64_t R = clamp_count(n_rec, cap);
  const int64_t S0 = *n_seg;
  const int64_t S = (2 * S0 <= cap) ? S0 : cap / 2;      // the segments k_full_entries kept
  const int64_t nnzb = *H.nnzb;
  const int lane = threadIdx.x & 31, q = lane / 9, c = lane - 9 * q;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < S; s += nw) {
    const int64_t b = start[s], e = (s + 1 < S0) ? start[s + 1] : R;
    double v = 0.0;
    if (q < 3) {
      int64_t k = b + q;
      for (; k + 9 < e; k += 12) {           // four gathers in flight
        const double x0 = __ldg(piece + 9 * (int64_t)__ldg(perm + k) + c), x1 = __ldg(piece + 9 * (int64_t)__ldg(perm + k + 3) + c);
        const double x2 = __ldg(piece + 9 * (int64_t)__ldg(perm + k + 6) + c), x3 = __ldg(piece + 9 * (int64_t)__ldg(perm + k + 9) + c);
        v += x0; v += x1; v += x2; v += x3;
      }
      for (; k < e; k += 3) v += __ldg(piece + 9 * (int64_t)__ldg(perm + k) + c);
    }
    const double v1 = __shfl_sync(0xffffffffu, v, c + 9), v2 = __shfl_sync(0xffffffffu, v, c + 18);
    if (e - b > 1) v += v1;
    if (e - b > 2) v += v2;
    if (q > 0) continue;
    const int32_t du = dst[2 * s], dl = dst[2 * s + 1];
    const int i = c / 3, k = c - 3 * i;
    if (dl != -2) {
      if (du >= 0 && du < nnzb) H.val[9 * (int64_t)du + c] = v;
      if (dl >= 0 && dl < nnzb) H.val[9 * (int64_t)dl + 3 * k + i] = v;
    } else if (k == 2) {
      g_r[3 * diagonal_node(ukey[s], (uint64_t)ns) + i] = v;
    } else if (du >= 0 && du < nnzb) {
      const int j = k == 0 ? i : (i == 2 ? 0 : i + 1);
      H.val[9 * (int64_t)du + 3 * i + j] = v;
      H.val[9 * (int64_t)du + 3 * j + i] = v;
    }
  }
}

// deterministic sum: fixed chunk per block, fixed in-block tree, partials summed in order
__global__ void __launch_bounds__(kBlock) k_sum_partial(const double* __restrict__ x, const int64_t* n_dev,
                                                        int64_t cap, double* __restrict__ partial) {
  pdl_entry();
  const int64_t n = clamp_count(n_dev, cap);
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t b = blockIdx.x * per, e = (b + per < n) ? b + per : n;
  double s = 0.0;
  for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) s += x[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  __shared__ double ws[kBlock / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) t += ws[w];
    partial[blockIdx.x] = t;
  }
}

// one warp: lane l adds partials l, l + 32, ... in order, then a fixed shuffle tree
__global__ void k_sum_final(const double* __restrict__ partial, int nb, double* out) {
  pdl_entry();
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  double t = 0.0;
  for (int b = lane; b < nb; b += 32) t += partial[b];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  if (lane == 0) *out = t;
}

// ------------------------------------------------------------------ friction lag
__global__ void __launch_bounds__(kEvalThreads) k_lag(Topo T, const double* __restrict__ x4,
                                                      const float* __restrict__ x4f, eipc_pairs pr,
                                                      double dhat, double kappa, eipc_lag out, DevStatus* st,
                                                      const double* __restrict__ moll_r2, double moll_factor,
                                                      uint64_t* __restrict__ key_out, int64_t key_cap) {
  pdl_entry();
  const int64_t P = clamp_count(pr.count, pr.capacity);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *out.count = P < out.capacity ? P : out.capacity;
    if (P > out.capacity) raise_flag(st, EIPC_FLAG_LAG_OVERFLOW);
  }
  const int64_t n = P < out.capacity ? P : out.capacity;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += grid_stride()) {
    int32_t v[4];
    const int type = pr.type[k];
    stencil_vertices(T, type, pr.i[k], pr.j[k], v);
    V3 X[4], Y[4];
    for (int a = 0; a < 4; ++a) X[a] = load_x(x4, v[a]);
    for (int a = 0; a < 4; ++a) Y[a] = X[a] - X[0];
    Stencil S;
    closest_pair<true>(type, Y, stencil_hint(type, x4f, v), &S);
    const double d = sqrt(S.d2);
    double b1 = 0.0;
    if (d > 0.0 && d < dhat) {
      const double lg = log(d / dhat), m = d - dhat;
      b1 = -2.0 * m * lg - m * m / d;
    }
    V3 rrel = {0.0, 0.0, 0.0};
    for (int a = 0; a < 4; ++a) rrel = rrel + Y[a] * S.c[a];
    const double rn = sqrt(dot(rrel, rrel));
    // anchor with the same arithmetic the evaluation uses for sum_a gamma_a x_a
    V3 anc = {0.0, 0.0, 0.0};
    for (int a = 0; a < 4; ++a) anc = anc + X[a] * S.c[a];
    reinterpret_cast<int4*>(out.v)[k] = make_int4(v[0], v[1], v[2], v[3]);
    if (k < key_cap) key_out[k] = lag_pair_key(type, pr.i[k], pr.j[k]);
    for (int a = 0; a < 4; ++a) out.gamma[4 * k + a] = S.c[a];
    out.n[3 * k] = rrel.x / rn; out.n[3 * k + 1] = rrel.y / rn; out.n[3 * k + 2] = rrel.z / rn;
    out.anchor[3 * k] = anc.x; out.anchor[3 * k + 1] = anc.y; out.anchor[3 * k + 2] = anc.z;
    // a mollified EE pair's lagged normal force is scaled by m(x^n)
    double mk = 1.0;
    if (type == 1 && moll_r2) {
      const V3 nn = cross(Y[1] - Y[0], Y[3] - Y[2]);
      const double c = dot(nn, nn);
      const double eps = moll_factor * moll_r2[pr.i[k]] * moll_r2[pr.j[k]];
      if (c < eps) mk = c * (2.0 / eps - c / (eps * eps));
    }
    out.lambda[k] = kappa * mk * fabs(b1);
  }
}

}  // namespace

int bits_for(uint64_t maxval) {
  int b = 1;
  while (b < 63 && (1ull << b) <= maxval) ++b;
  return b;
}

void lag_launch(eipc_scene* sc, const double* q_n, const eipc_pairs& pr, const eipc_params& p, const eipc_lag& out,
                cudaStream_t s) {
  EIPC_TIMED(sc, kKEmbed, s, embed_launch(sc, q_n, sc->x4, 1, 0, s));
  EIPC_TIMED(sc, kKLag, s,
             (launch(k_lag, blocks_for(pr.capacity, 8, kEvalThreads), kEvalThreads, 0, s, sc->topo, sc->x4,
                     static_cast<const float*>(sc->x4f), pr, p.dhat, p.kappa, out, sc->status, static_cast<const double*>(sc->moll_factor > 0.0 ? sc->moll_r2 : nullptr),
                     sc->moll_factor, sc->lag_key, sc->item_cap)));
  sc->lag_src = out.v;   // the lag state whose pair keys lag_key now holds
}

void eval_launch(eipc_scene* sc, const double* q, const eipc_pairs& pr, const eipc_lag* lag, const eipc_params& p,
                 double* E, double* g_r, const eipc_bsr& H, cudaStream_t s) {
  EIPC_TIMED(sc, kKEmbed, s, embed_launch(sc, q, sc->x4, 1, 0, s));
  const bool fr = lag && p.mu > 0.0;
  // friction items ride on the contact pairs with the same stencil (not with the EE
  // mollifier, whose pairs are evaluated by their own kernel)
  const bool merge = fr && !(sc->moll_factor > 0.0);
  int64_t* cnt = sc->counters;
  int64_t* n_full = cnt + 13;
  int64_t* n_diag = cnt + 14;
  const int64_t item_cap = sc->item_cap;
  const int64_t pcap = pr.capacity < item_cap ? pr.capacity : item_cap;
  int64_t* n_moll = sc->moll_factor > 0.0 ? cnt + kCntMollList : nullptr;
  // counters, the evaluation queue, g_r and the friction claims, all reset up front
  zero_ranges(s, {{cnt + kCntItems, 5 * sizeof(int64_t)}, {n_diag, sizeof(int64_t)},
                  {cnt + kCntEvalQueue, sizeof(int64_t)}, {cnt + kCntEvalRest, 2 * sizeof(int64_t)}, {n_moll, sizeof(int64_t)}, {g_r, sizeof(double) * 3 * sc->ns},
                  {merge ? sc->fric_of_pair : nullptr, sizeof(int32_t) * pcap}});
  // group keys: the first node above kHashBits of hash (a fixed number: a scene's items must fall
  // into the same groups whatever the size of the batch around it)
  const int key_bits = sc->bits_g + kHashBits;
  const int32_t* fop = merge ? sc->fric_of_pair : nullptr;
  const int32_t* pof = merge ? sc->pair_of_fric : nullptr;
  sc->timers->start(kKItems, s);
  if (merge)
    launch(k_fric_match, blocks_for(lag->capacity, 8), kBlock, 0, s, sc->topo, pr, *lag, item_cap,
           static_cast<const uint64_t*>(sc->edge_key), static_cast<const int32_t*>(sc->edge_id),
           static_cast<const uint64_t*>(lag->v == sc->lag_src ? sc->lag_key : nullptr), sc->fric_of_pair,
           sc->pair_of_fric);
  launch(k_item_nodes, blocks_for(item_cap, 8), kBlock, 0, s, sc->topo, pr, fr ? lag->v : nullptr, fr ? lag->count : nullptr,
                                                           fr ? lag->capacity : 0, sc->cage_idx, item_cap,
                                                           sc->item_nodes, sc->item_n, sc->item_group, sc->vgroup,
                                                           sc->rc_h, sc->rc_g,
                                                           cnt + kCntItems, sc->status, fop, pof, sc->item_map, key_bits,
                                                           sc->skeys, sc->svals);
  int64_t* tot_h = cnt + 9;
  int64_t* tot_g = cnt + 10;
  exclusive_scan2_i64(sc->rc_h, sc->ro_h, tot_h, sc->rc_g, sc->ro_g, tot_g, cnt + kCntItems, item_cap,
                      sc->scan_partial, s);
  launch(k_rec_check, 1, kRecCheckThreads, 0, s, tot_h, tot_g, sc->rec_cap, sc->gcap, cnt + kCntRecH, cnt + kCntRecG, sc->status,
         static_cast<const int64_t*>(cnt + kCntItems), static_cast<const int64_t*>(sc->ro_h),
         static_cast<const int64_t*>(sc->ro_g), sc->item_n, sc->moll_factor > 0.0);
  sc->timers->stop(kKItems, s);

  EvalArgs A{};
  A.T = sc->topo; A.pr = pr; A.cage_idx = sc->cage_idx; A.w = sc->w; A.x4 = sc->x4; A.x4f = sc->x4f; A.ns = sc->ns;
  A.dhat = p.dhat; A.inv_dhat = 1.0 / p.dhat; A.kappa = p.kappa; A.item_nodes = sc->item_nodes; A.item_n = sc->item_n;
  A.item_map = sc->item_map;
  A.ro_h = sc->ro_h; A.ro_g = sc->ro_g; A.n_items = cnt + kCntItems; A.rec_cap = sc->rec_cap; A.gcap = sc->gcap;
  A.frow = sc->frow; A.ihead = sc->ihead; A.hrec = sc->hrec; A.item_E = sc->item_E; A.st = sc->status;
  A.project = (p.flags & EIPC_PARAM_NO_PROJECTION) == 0;
  A.moll_r2 = sc->moll_factor > 0.0 ? sc->moll_r2 : nullptr;
  A.moll_factor = sc->moll_factor;
  A.fric_of_pair = fop; A.pair_of_fric = pof;
  A.lag = fr ? *lag : eipc_lag{};
  A.mu = p.mu; A.eps_f = p.eps_v * p.h;
  A.moll_list = reinterpret_cast<uint32_t*>(sc->rc_g);    // the record counts have been scanned
  A.n_moll = cnt + kCntMollList;
  A.rest = reinterpret_cast<uint32_t*>(sc->rc_h);
  A.n_rest = cnt + kCntEvalRest;
  A.item_cap = item_cap;
  A.queue = cnt + kCntEvalQueue;
  A.tile = sc->tune.eval_tile;
  // The factors and the pattern both follow from the items and are needed by the sums only:
  // the factors (bound by the FP64 pipe) run on the scene's second stream beside the pattern's
  // chain of sorts and scans (bound by latency and memory).
  cudaEventRecord(sc->ev_fork, s);
  cudaStreamWaitEvent(sc->aux, sc->ev_fork, 0);
  {
    const int64_t most = pr.capacity + (fr ? lag->capacity : 0);
    const int blocks = blocks_for(most < item_cap ? most : item_cap, sc->tune.eval_bps, sc->tune.eval_threads);
    sc->timers->start(kKEvalPair, sc->aux);
    EIPC_TIMED(sc, kKEvalBarrier, sc->aux,
               launch(k_eval_factors, blocks, sc->tune.eval_threads, 0, sc->aux, A);
               launch(k_eval_rest, 2 * kSMs, kEvalThreads, 0, sc->aux, A));
    if (A.moll_r2)
      EIPC_TIMED(sc, kKEvalBarrier, sc->aux,
                 (launch(k_mollified_eval, 8 * kSMs, 32 * kMollWarps, 0, sc->aux, A,
                         static_cast<const uint32_t*>(A.moll_list), static_cast<const int64_t*>(A.n_moll))));
    sc->timers->stop(kKEvalPair, sc->aux);
  }

  // groups of items with the same nodes, their chunks' records, and the records' sums (after the
  // factors, on their stream); beside those, the Hessian pattern: record keys (I, J), stable
  // sort, segments (one per BSR upper block), then the full symmetric pattern (every
  // off-diagonal upper block also at (J, I)), columns and row pointers
  sc->timers->start(kKHReduce, s);
  const int wi = radix_sort_u64(sc->skeys, sc->svals, sc->skeys_alt, sc->svals_alt, cnt + kCntItems, item_cap, key_bits,
                                sc->sort_hist, s);
  const uint64_t* ik = wi ? sc->skeys_alt : sc->skeys;
  const uint32_t* iv = wi ? sc->svals_alt : sc->svals;
  const int64_t* n_items = cnt + kCntItems;
  const int64_t* n_groups = cnt + kCntGroups;
  const int64_t* n_rec = cnt + kCntRecords;
  launch(k_group_count, kScanBlocks, 256, 0, s, ik, iv, n_items, static_cast<const int32_t*>(sc->item_n),
         static_cast<const int32_t*>(sc->item_nodes), sc->scan_partial);
  launch(k_group_start, kScanBlocks, 256, 0, s, ik, iv, n_items, static_cast<const int32_t*>(sc->item_n),
         static_cast<const int32_t*>(sc->item_nodes), static_cast<const int64_t*>(sc->scan_partial), cnt + kCntGroups, sc->group_start);
  int64_t* gcount = reinterpret_cast<int64_t*>(sc->gkeys);
  int64_t* goffset = reinterpret_cast<int64_t*>(sc->gkeys_alt);
  launch(k_group_records, blocks_for(item_cap, 8), kBlock, 0, s, static_cast<const int64_t*>(sc->group_start), n_groups, n_items,
         iv, static_cast<const int32_t*>(sc->item_n), gcount);
  exclusive_scan_i64(gcount, goffset, n_groups, item_cap, cnt + kCntRecords, sc->scan_partial, s);
  launch(k_rec_keys, blocks_for(32 * item_cap, 8), kBlock, 0, s, static_cast<const int64_t*>(sc->group_start), n_groups, n_items,
         iv, static_cast<const int32_t*>(sc->item_n), static_cast<const int32_t*>(sc->item_nodes),
         static_cast<const int64_t*>(goffset), sc->rec_cap, sc->ns, sc->hkeys, sc->hvals, sc->rec_src);
  cudaEventRecord(sc->ev_mid, s);
  cudaStreamWaitEvent(sc->aux, sc->ev_mid, 0);
  launch(k_chunk_sums, blocks_for(3 * sc->rec_cap, 32, 128), 128, 0, sc->aux,
         SumArgs{sc->rec_src, n_rec, sc->rec_cap, iv, sc->ro_h, sc->item_n, sc->ro_g, sc->frow, sc->ihead, sc->hrec, sc->piece});
  cudaEventRecord(sc->ev_join, sc->aux);
  const int wh = radix_sort_u64(sc->hkeys, sc->hvals, sc->hkeys_alt, sc->hvals_alt, n_rec, sc->rec_cap, sc->bits_h,
                                sc->sort_hist, s);
  const uint64_t* hk = wh ? sc->hkeys_alt : sc->hkeys;
  const uint32_t* hv = wh ? sc->hvals_alt : sc->hvals;
  segment_starts(hk, n_rec, sc->rec_cap, sc->seg_start, cnt + kCntSegH, sc->scan_partial, s);
  // seg_flag and seg_id hold the segment keys and the segments' BSR entries
  uint64_t* ukey = reinterpret_cast<uint64_t*>(sc->seg_flag);
  int32_t* dst = reinterpret_cast<int32_t*>(sc->seg_id);
  launch(k_seg_keys, blocks_for(sc->rec_cap), kBlock, 0, s, static_cast<const int64_t*>(sc->seg_start),
         static_cast<const int64_t*>(cnt + kCntSegH), hk, ukey);
  // row field: bits_g rounded up to whole radix digits (the sort passes cover whole bytes,
  // so the column must start on a byte); 2^bits_g > ns, so the all-ones row of the
  // diagonal twins is above every row.  The group buffers are free here.
  const int rb = ((sc->bits_g + 7) / 8) * 8;
  launch(k_full_entries, blocks_for(sc->rec_cap), kBlock, 0, s, static_cast<const uint64_t*>(ukey),
         static_cast<const int64_t*>(cnt + kCntSegH), sc->ns, rb, sc->rec_cap, sc->gkeys, sc->gvals, n_full, n_diag,
         sc->status, dst);
  const int wf = radix_sort_u64(sc->gkeys, sc->gvals, sc->gkeys_alt, sc->gvals_alt, n_full, sc->rec_cap, rb,
                                sc->sort_hist, s);
  const uint64_t* fk = wf ? sc->gkeys_alt : sc->gkeys;
  const uint32_t* fv = wf ? sc->gvals_alt : sc->gvals;
  launch(k_bsr_pattern, blocks_for(sc->rec_cap), kBlock, 0, s, fk, fv, static_cast<const int64_t*>(n_full),
         static_cast<const int64_t*>(n_diag), rb, sc->ns, H, dst, sc->status, cnt + kCntSegG);
  cudaStreamWaitEvent(s, sc->ev_join, 0);
  // blocks into the BSR values; the diagonal segments' gradients into g_r
  launch(k_segment_sums, blocks_for(32 * sc->rec_cap, 8), kBlock, 0, s, static_cast<const double*>(sc->piece), hv,
         static_cast<const int64_t*>(sc->seg_start), n_rec, static_cast<const int64_t*>(cnt + kCntSegH), sc->rec_cap,
         static_cast<const int32_t*>(dst), H, static_cast<const uint64_t*>(ukey), sc->ns, g_r);
  sc->timers->stop(kKHReduce, s);
  // energy
  sc->timers->start(kKEnergy, s);
  launch(k_sum_partial, kScanBlocks, kBlock, 0, s, sc->item_E, cnt + kCntItems, item_cap, sc->sum_partial);
  launch(k_sum_final, 1, 32, 0, s, sc->sum_partial, kScanBlocks, E);
  sc->timers->stop(kKEnergy, s);
}

void hvp_launch(eipc_scene* sc, const double* q, const eipc_pairs& pr, const eipc_lag* lag, const eipc_params& p,
                const double* v, const double* kin_dir, double* out_r, double* out_kin, cudaStream_t s) {
  const bool fr = lag && p.mu > 0.0;
  const V3 kin = kin_dir ? V3{kin_dir[0], kin_dir[1], kin_dir[2]} : V3{0.0, 0.0, 0.0};
  HvpArgs A{};
  A.T = sc->topo; A.pr = pr; A.friction = fr;
  if (fr) A.lag = *lag;
  A.x4 = sc->x4; A.x4f = sc->x4f; A.u4 = sc->dx4;
  A.dhat = p.dhat; A.inv_dhat = 1.0 / p.dhat; A.kappa = p.kappa; A.mu = p.mu; A.eps_f = p.eps_v * p.h;
  A.moll_r2 = sc->moll_factor > 0.0 ? sc->moll_r2 : nullptr;
  A.moll_factor = sc->moll_factor;
  A.item_cap = sc->item_cap;
  // scratch: the factor rows hold y, the search's per-vertex boxes the sums, the FP32
  // displacements the exponents (every other call writes them anew before it reads them)
  A.y = sc->frow;
  A.vexp = reinterpret_cast<int32_t*>(sc->dx4f);
  A.hi = reinterpret_cast<unsigned long long*>(sc->vbox);
  A.lo = reinterpret_cast<unsigned long long*>(sc->vbox_pad);
  A.st = sc->status;
  int64_t* ticket = sc->counters + kCntHvpTicket;
  EIPC_TIMED(sc, kKEmbed, s, embed_launch(sc, q, sc->x4, 1, 0, s);
             launch(k_hvp_direction, blocks_for(sc->nv), kBlock, 0, s, sc->nv, static_cast<const int32_t*>(sc->cage_idx),
                    static_cast<const double*>(sc->w), v, kin, sc->dx4, A.vexp, A.hi, A.lo,
                    CounterList{{ticket, sc->counters + kCntEvalRest, sc->counters + kCntMollList, nullptr}}));
  const int64_t want = pr.capacity + (fr ? lag->capacity : 0), most = want < sc->item_cap ? want : sc->item_cap;
  A.rest = sc->svals; A.n_rest = sc->counters + kCntEvalRest;
  A.moll_list = sc->svals_alt; A.n_moll = A.moll_r2 ? sc->counters + kCntMollList : nullptr;
  EIPC_TIMED(sc, kKEvalBarrier, s, launch(k_hvp_items, blocks_for(most, 8, kEvalThreads), kEvalThreads, 0, s, A);
             launch(k_hvp_rest, 2 * kSMs, kEvalThreads, 0, s, A));
  if (A.moll_r2)
    EIPC_TIMED(sc, kKEvalBarrier, s, (launch(k_hvp_mollified, 2 * kSMs, kEvalThreads, 0, s, A)));
  sc->timers->start(kKGReduce, s);
  launch(k_hvp_accumulate, blocks_for(4 * most, 8), kBlock, 0, s, A);
  launch(k_hvp_gather, blocks_for(32 * (sc->ns + kKinSlots), 8), kBlock, 0, s, sc->ns, static_cast<const int64_t*>(sc->inc_ptr),
         static_cast<const uint32_t*>(sc->inc), static_cast<const double*>(sc->w), static_cast<const int32_t*>(A.vexp),
         reinterpret_cast<const long long*>(A.hi), reinterpret_cast<const long long*>(A.lo), out_r, out_kin, sc->hvp_part, ticket);
  sc->timers->stop(kKGReduce, s);
}

// Static lists for J^T: the embedded vertices' (vertex, slot) entries by cage node, then the
// kinematic vertices; built once at scene creation on the default stream, by the stable radix
// sort.
namespace {
__global__ void __launch_bounds__(kBlock) k_incidence_keys(int64_t nv, int64_t ns, const int32_t* __restrict__ idx,
                                                           uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  pdl_entry();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 4 * nv; t += grid_stride()) {
    const int32_t id = idx[t];
    keys[t] = (uint64_t)(id >= 0 ? id : ((t & 3) == 0 ? ns : ns + 1));     // a kinematic vertex counts once
    vals[t] = (uint32_t)t;
  }
}

__global__ void __launch_bounds__(kBlock) k_incidence_rows(int64_t ns, int64_t n, const uint64_t* __restrict__ keys,
                                                           int64_t* __restrict__ ptr) {
  pdl_entry();
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < ns + 2; r += grid_stride()) {
    int64_t lo = 0, hi = n;                  // first entry of row r
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (keys[mid] < (uint64_t)r) lo = mid + 1;
      else hi = mid;
    }
    ptr[r] = lo;
  }
}
}  // namespace

cudaError_t incidence_build(eipc_scene* sc) {
  const int64_t n = 4 * sc->nv;
  uint64_t *k = nullptr, *ka = nullptr;
  uint32_t* va = nullptr;
  int64_t* nd = nullptr;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&k), 8 * n);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&ka), 8 * n);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&va), 4 * n);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&nd), 8);
  if (e == cudaSuccess) e = cudaMemcpy(nd, &n, 8, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    launch(k_incidence_keys, blocks_for(n), kBlock, 0, nullptr, sc->nv, sc->ns, static_cast<const int32_t*>(sc->cage_idx), k, sc->inc);
    const int which = radix_sort_u64(k, sc->inc, ka, va, nd, n, bits_for((uint64_t)sc->ns + 1), sc->sort_hist, nullptr);
    launch(k_incidence_rows, blocks_for(sc->ns + 2), kBlock, 0, nullptr, sc->ns, n, static_cast<const uint64_t*>(which ? ka : k),
           sc->inc_ptr);
    if (which) e = cudaMemcpyAsync(sc->inc, va, 4 * n, cudaMemcpyDeviceToDevice, nullptr);
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
  }
  if (k) cudaFree(k);
  if (ka) cudaFree(ka);
  if (va) cudaFree(va);
  if (nd) cudaFree(nd);
  return e;
}

}  // namespace eipc
