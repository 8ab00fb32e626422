// LBVH build (one Morton sort, Karras hierarchies, treelets), refit and traversal.
#include "bvh.cuh"
#include "sort.cuh"

namespace eipc {
namespace {

// order-preserving map float -> int for integer min / max
__device__ __forceinline__ int32_t f2ord(float f) {
  int32_t i = __float_as_int(f);
  return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ord2f(int32_t i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// min and max over the warp (no NaN reaches a primitive's box)
__device__ __forceinline__ float warp_min(float x) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}

__global__ void k_bounds_init(int32_t* b, int32_t* n_tri, int32_t* n_edge) {
  pdl_entry();
  if (threadIdx.x < 3) b[threadIdx.x] = 0x7fffffff;
  else if (threadIdx.x < 6) b[threadIdx.x] = (int32_t)0x80000000;
  else if (threadIdx.x < 9) n_tri[threadIdx.x - 6] = 0;
  else if (threadIdx.x < 12) n_edge[threadIdx.x - 9] = 0;
}

// scene box over all per-vertex boxes
__global__ void __launch_bounds__(kBlock) k_bounds(const float* __restrict__ vbox, int64_t nv, int32_t* __restrict__ b) {
  pdl_entry();
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += grid_stride()) {
    const float4 p = __ldg(reinterpret_cast<const float4*>(vbox + 8 * v));
    const float4 q = __ldg(reinterpret_cast<const float4*>(vbox + 8 * v) + 1);
    lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
    hi[0] = fmaxf(hi[0], p.w); hi[1] = fmaxf(hi[1], q.x); hi[2] = fmaxf(hi[2], q.y);
  }
  for (int k = 0; k < 3; ++k) {
    lo[k] = warp_min(lo[k]);
    hi[k] = warp_max(hi[k]);
  }
  if ((threadIdx.x & 31) == 0) {
    for (int k = 0; k < 3; ++k) {
      atomicMin(&b[k], f2ord(lo[k]));
      atomicMax(&b[3 + k], f2ord(hi[k]));
    }
  }
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000ffu;
  v = (v | (v << 8)) & 0x0300f00fu;
  v = (v | (v << 4)) & 0x030c30c3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// box of up to three vertices from the per-vertex boxes (ids < 0 are skipped)
__device__ __forceinline__ void verts_box(const float* __restrict__ vbox, int32_t a, int32_t b, int32_t c,
                                          float lo[3], float hi[3]) {
  for (int k = 0; k < 3; ++k) { lo[k] = INFINITY; hi[k] = -INFINITY; }
  const int32_t v[3] = {a, b, c};
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    if (v[s] < 0) continue;
    const float4 p = __ldg(reinterpret_cast<const float4*>(vbox + 8 * (int64_t)v[s]));
    const float4 q = __ldg(reinterpret_cast<const float4*>(vbox + 8 * (int64_t)v[s]) + 1);
    lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y); lo[2] = fminf(lo[2], p.z);
    hi[0] = fmaxf(hi[0], p.w); hi[1] = fmaxf(hi[1], q.x); hi[2] = fmaxf(hi[2], q.y);
  }
}

// Sort keys of every triangle, edge and vertex: kind (0, 1, 2) above the Morton code of the box
// centre, so that one sort orders all three.
__global__ void __launch_bounds__(kBlock) k_morton_keys(Topo T, const float* __restrict__ vbox, const int32_t* __restrict__ b,
                                                        uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  pdl_entry();
  float blo[3], bext[3];
  for (int k = 0; k < 3; ++k) {
    blo[k] = ord2f(b[k]);
    float e = ord2f(b[3 + k]) - blo[k];
    bext[k] = e > 0.f ? e : 1.f;
  }
  const int64_t n = T.nf + T.ne + T.nv;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += grid_stride()) {
    const int kind = g < T.nf ? 0 : (g < T.nf + T.ne ? 1 : 2);
    const int64_t i = kind == 0 ? g : (kind == 1 ? g - T.nf : g - T.nf - T.ne);
    float lo[3], hi[3];
    if (kind == 0) verts_box(vbox, T.tris[3 * i], T.tris[3 * i + 1], T.tris[3 * i + 2], lo, hi);
    else if (kind == 1) verts_box(vbox, T.edges[2 * i], T.edges[2 * i + 1], -1, lo, hi);
    else verts_box(vbox, (int32_t)i, -1, -1, lo, hi);
    uint32_t code = 0;
    for (int k = 0; k < 3; ++k) {
      float c = (0.5f * (lo[k] + hi[k]) - blo[k]) / bext[k];
      c = fminf(fmaxf(c, 0.f), 1.f);
      const uint32_t q = (uint32_t)fminf(c * 1024.f, 1023.f);
      code |= spread10(q) << (2 - k);
    }
    keys[g] = (uint64_t)kind << 30 | code;
    vals[g] = (uint32_t)i;
  }
}

__device__ __forceinline__ int delta(const uint64_t* __restrict__ k, int64_t n, int64_t i, int64_t j) {
  if (j < 0 || j >= n) return -1;
  uint64_t a = k[i], b = k[j];
  if (a == b) return 64 + __clzll((unsigned long long)(i ^ j));
  return __clzll((unsigned long long)(a ^ b));
}

// What building and refitting need of one tree; n = 0 marks an absent tree.
struct TreeView {
  int64_t n;
  const uint64_t* keys;      // this tree's sorted keys (build only)
  const uint32_t* prim;
  BvhNode* nodes;
  int32_t* parent;
  int4* leaf_info;
  float* leaf_box;
  int32_t* flag;
  int4* treelet;
  int4* cluster;
  float* part_box;
  int2* upper;
  int32_t* cluster_up;
  int32_t* top;
  int32_t* n_lists;
  // build only: per leaf, the leaves of the treelet that starts there (0: none) and that treelet's
  // parent << 1 | slot; in leaf_box, which the first refit overwrites
  __device__ int2* head() const { return reinterpret_cast<int2*>(leaf_box); }
};

// Karras 2012: internal node i covers a key range; its split is the highest differing bit.
__device__ __forceinline__ void internal_node(const TreeView& T, int64_t i) {
  const uint64_t* keys = T.keys;
  const int64_t n = T.n;
  int dir = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
  int dmin = delta(keys, n, i, i - dir);
  int64_t lmax = 2;
  while (delta(keys, n, i, i + lmax * dir) > dmin) lmax *= 2;
  int64_t l = 0;
  for (int64_t t = lmax / 2; t >= 1; t /= 2)
    if (delta(keys, n, i, i + (l + t) * dir) > dmin) l += t;
  int64_t j = i + l * dir;
  int dnode = delta(keys, n, i, j);
  int64_t s = 0;
  for (int64_t div = 2;; div *= 2) {
    int64_t t = (l + div - 1) / div;
    if (delta(keys, n, i, i + (s + t) * dir) > dnode) s += t;
    if (t == 1) break;
  }
  const int64_t split = i + s * dir + (dir < 0 ? -1 : 0);
  const int64_t lo = i < j ? i : j, hi = i < j ? j : i;
  int4* tail = reinterpret_cast<int4*>(&T.nodes[i].first);
  *tail = make_int4((int32_t)lo, (int32_t)hi, 0, (int32_t)split);
  T.flag[i] = 0;
  T.head()[i] = make_int2(0, 0);
  if (i == 0) T.head()[n - 1] = make_int2(0, 0);
  T.parent[lo == split ? n - 1 + split : split] = (int32_t)(i << 1);
  T.parent[hi == split + 1 ? n + split : split + 1] = (int32_t)(i << 1) | 1;
}

__global__ void __launch_bounds__(kBlock) k_internal(TreeView A, TreeView B) {
  pdl_entry();
  const int64_t nA = A.n > 1 ? A.n - 1 : 0, nB = B.n > 1 ? B.n - 1 : 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nA + nB; i += grid_stride()) {
    if (i < nA) internal_node(A, i);
    else internal_node(B, i - nA);
  }
}

// Leaf records, treelets and clusters: the largest subtrees of at most kTreelet and kCluster leaves
// (single leaves directly under a larger node among them).  The order of the clusters in their
// list has no meaning.  The nodes above the clusters are numbered, in any order; a node's flag
// holds twice its number (even: no arrival).
__device__ __forceinline__ void tree_parts(const TreeView& T, PrimKind kind, const Topo& topo, int64_t wbase) {
  const int lane = threadIdx.x & 31;
  const int64_t n = T.n, i = wbase + lane;
  int32_t first = 0, size = 0, ps = -1, above = 0;       // above: leaves of the parent
  auto size_of = [&](int32_t node) { return T.nodes[node].last - T.nodes[node].first + 1; };
  if (i < n) {                                    // leaf i
    const int64_t p = T.prim[i];
    if (kind == kTri) {
      const int32_t v0 = topo.tris[3 * p];
      T.leaf_info[i] = make_int4(v0, topo.tris[3 * p + 1], topo.tris[3 * p + 2], topo.fkin[p] | (topo.vgroup[v0] << 1));
    } else {
      const int32_t v0 = topo.edges[2 * p];
      T.leaf_info[i] = make_int4(v0, topo.edges[2 * p + 1], -1, topo.ekin[p] | (topo.vgroup[v0] << 1));
    }
    first = (int32_t)i;
    size = 1;
    if (n > 1) ps = T.parent[n - 1 + i];
  } else if (i < 2 * n - 1) {                     // internal node i - n
    const int32_t node = (int32_t)(i - n);
    first = T.nodes[node].first;
    size = size_of(node);
    if (node) ps = T.parent[node];
  }
  above = ps < 0 ? INT32_MAX : size_of(ps >> 1);
  if (size > 0 && size <= kTreelet && above > kTreelet) T.head()[first] = make_int2(size, ps);
  const bool is = size > 0 && size <= kCluster && above > kCluster;
  const unsigned m = __ballot_sync(0xffffffffu, is);
  if (m) {
    int base = 0;
    if (lane == 0) base = atomicAdd(T.n_lists + 1, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (is) T.cluster[base + __popc(m & ((1u << lane) - 1u))] = make_int4(first, size, ps, 0);
  }
  const unsigned u = __ballot_sync(0xffffffffu, size > kCluster);
  if (u) {
    int base = 0;
    if (lane == 0) base = atomicAdd(T.n_lists + 2, __popc(u));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (size > kCluster) {
      const int id = base + __popc(u & ((1u << lane) - 1u));
      T.flag[i - n] = 2 * id;
      if (id < kUpper) T.upper[id].x = (int32_t)(i - n);
    }
  }
}

__global__ void __launch_bounds__(kBlock) k_tree_parts(TreeView A, TreeView B, Topo topo) {
  pdl_entry();
  // whole warps per tree
  const int64_t nA = (2 * A.n + 30) / 32, nB = (2 * B.n + 30) / 32;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nA + nB; w += nw) {
    if (w < nA) tree_parts(A, kTri, topo, 32 * w);
    else tree_parts(B, kEdge, topo, 32 * (w - nA));
  }
}

// Each cluster's treelets, in leaf order, into consecutive entries of the treelet list; where the
// nodes above the clusters are few, the parents among them by number.  One warp per tree also finds
// the nodes that a walk starts from: from the root, four times every node whose children are both
// above the treelets is replaced by them.
__device__ __forceinline__ void walk_starts(const TreeView& T, int lane) {
  int count = T.n > kTreelet ? 1 : 0;
  int32_t node = 0;
  for (int level = 0; level < 4; ++level) {
    const bool mine = lane < count;
    const int4 tail = mine ? *reinterpret_cast<const int4*>(&T.nodes[node].first) : make_int4(0, 0, 0, 0);   // first, last, kin, split
    const bool open = mine && tail.w - tail.x + 1 > kTreelet && tail.y - tail.w > kTreelet;
    const unsigned m_open = __ballot_sync(0xffffffffu, open), below = (1u << lane) - 1u;
    const int at = lane + __popc(m_open & below);          // an opened node takes two places
    int32_t from = 0, next = 0;
    for (int l = 0; l < count; ++l) {
      const int32_t l_at = __shfl_sync(0xffffffffu, at, l), l_node = __shfl_sync(0xffffffffu, node, l);
      const int32_t l_split = __shfl_sync(0xffffffffu, tail.w, l);
      const bool l_open = m_open >> l & 1u;
      from = l_open ? l_split : l_node;
      if (lane == l_at) next = from;
      if (l_open && lane == l_at + 1) next = l_split + 1;
    }
    node = next;
    count += __popc(m_open);
  }
  if (lane < count) T.top[lane] = node;
  if (lane == 0) T.top[kWalkStarts] = count;
}

__global__ void __launch_bounds__(kBlock) k_cluster_treelets(TreeView A, TreeView B) {
  static_assert(kBlock * 2 == kCluster, "a thread takes two leaves");
  pdl_entry();
  __shared__ int32_t count[kCluster / 32], base;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t nA = A.n > 0 ? A.n_lists[1] : 0, nB = B.n > 0 ? B.n_lists[1] : 0;
  if (blockIdx.x == gridDim.x - 1 && warp < 2) walk_starts(warp == 0 ? A : B, lane);
  for (int64_t g = blockIdx.x * (int64_t)kBlock + t; g < 2 * (2 * kUpper + 1); g += grid_stride()) {
    const bool inA = g < 2 * kUpper + 1;
    const int32_t k = (int32_t)(inA ? g : g - (2 * kUpper + 1)), clusters = (int32_t)(inA ? nA : nB);
    const int32_t* flag = inA ? A.flag : B.flag;
    if (clusters > kUpper + 1) continue;
    auto numbered = [&](int32_t ps) { return ps < 0 ? -1 : (flag[ps >> 1] & ~1) | (ps & 1); };
    if (k < clusters) {
      (inA ? A.cluster_up : B.cluster_up)[k] = numbered((inA ? A.cluster : B.cluster)[k].z);
    } else if (k >= kUpper + 1 && k - (kUpper + 1) < clusters - 1) {
      int2* up = (inA ? A.upper : B.upper) + (k - (kUpper + 1));
      up->y = up->x ? numbered((inA ? A.parent : B.parent)[up->x]) : -1;
    }
  }
  for (int64_t c = blockIdx.x; c < nA + nB; c += gridDim.x) {
    const TreeView& T = c < nA ? A : B;
    int4* entry = T.cluster + (c < nA ? c : c - nA);
    const int32_t first = entry->x, leaves = entry->y;
    int2 h[2];
    unsigned m[2];
    for (int r = 0; r < 2; ++r) {
      const int l = r * kBlock + t;
      h[r] = l < leaves ? T.head()[first + l] : make_int2(0, 0);
      m[r] = __ballot_sync(0xffffffffu, h[r].x > 0);
      if (lane == 0) count[r * (kBlock / 32) + warp] = __popc(m[r]);
    }
    __syncthreads();
    if (t == 0) {
      int sum = 0;
      for (int k = 0; k < kCluster / 32; ++k) { const int v = count[k]; count[k] = sum; sum += v; }
      base = atomicAdd(T.n_lists, sum);
      entry->y = leaves | (sum << 16);
      entry->w = base;
    }
    __syncthreads();
    for (int r = 0; r < 2; ++r)
      if (h[r].x > 0)
        T.treelet[base + count[r * (kBlock / 32) + warp] + __popc(m[r] & ((1u << lane) - 1u))] =
            make_int4(first + r * kBlock + t, h[r].x, h[r].y, 0);
    __syncthreads();
  }
}

// Arrival counter of the bottom-up refit with release-acquire semantics at device scope:
// the child box a thread stored before its increment is visible to the thread whose
// increment comes second, which then reads the sibling's box.  A refit brings two arrivals
// to every node, so the counter's parity tells first from second and it is never reset.
__device__ __forceinline__ bool arrive_first(int32_t* f) {
  int32_t old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(f) : "memory");
  return (old & 1) == 0;
}

// Refit of both trees in two launches: leaves to subtree roots, then from there to the root.
// Nothing is kept below the treelets: the traversal reads their leaf boxes directly.  A climb goes
// up with a box; the second child to arrive at a node takes the union on, and no thread waits on
// another.  On a build (`first`) the kinematic bits climb with the boxes.  A level costs two
// device-scope round trips, 2 us, in L2 and about a twentieth of that in shared memory, so up to
// kClusterPrims primitives the subtrees are clusters, climbed in shared memory by a block each,
// and the nodes above them are climbed in shared memory by a block per tree (beyond kUpper
// nodes: in L2).  Sphere on pad 31.7 us with the treelets climbed in L2, 18.5 us so; bubble grasp
// (454,550 triangles and edges) 46.3 and 32.5 us.  On larger scenes the chip is full with a warp
// per treelet, and blocks that wait between a cluster's phases keep fewer reads in flight: the
// subtrees are the treelets and the climb is in L2.  256-scene batch (10.5 M) 129 + 99 us, by
// clusters 519 + 35 us; 211 + 150 us with shuffled integer reductions and 256-thread blocks.  Batches
// of 8 to 96 scenes, caches flushed, by clusters and by treelets: 0.32 M primitives 30 and 40 us, 0.55 M
// 39 and 46, 0.98 M 58 and 52, 1.31 M 105 and 59, 3.92 M 159 and 101: the two meet near 0.8 M, and the
// line costs up to 6 us between there and 2^20.
constexpr int64_t kClusterPrims = 1 << 20;

__global__ void __launch_bounds__(kBlock) k_refit_leaves(TreeView A, TreeView B, const float* __restrict__ vbox) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  const int64_t nA = A.n > 0 ? *A.n_lists : 0, nB = B.n > 0 ? *B.n_lists : 0;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nA + nB; w += nw) {
    const bool inA = w < nA;
    const int4 en = __ldg(inA ? A.treelet + w : B.treelet + (w - nA));
    const int64_t l = en.x + (int64_t)lane;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    int kin = 1;
    if (lane < en.y) {
      const int4 li = __ldg((inA ? A.leaf_info : B.leaf_info) + l);
      verts_box(vbox, li.x, li.y, li.z, lo, hi);
      kin = li.w & 1;
      float4* o = reinterpret_cast<float4*>((inA ? A.leaf_box : B.leaf_box) + 8 * l);
      o[0] = make_float4(lo[0], lo[1], lo[2], hi[0]);
      o[1] = make_float4(hi[1], hi[2], 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) { lo[k] = warp_min(lo[k]); hi[k] = warp_max(hi[k]); }
    kin = __all_sync(0xffffffffu, kin);
    if (lane == 0) {
      float4* o = reinterpret_cast<float4*>(inA ? A.part_box + 8 * w : B.part_box + 8 * (w - nA));
      o[0] = make_float4(lo[0], lo[1], lo[2], hi[0]);
      o[1] = make_float4(hi[1], hi[2], __int_as_float(kin), 0.f);
    }
  }
}

struct ClusterTree {
  float box[kCluster][2][6];           // of an internal node's children, by node - first leaf
  float treelet[kCluster][6];
  uint8_t kin[kCluster];               // treelet: all leaves kinematic
  int32_t parent[kCluster];
  int32_t flag[kCluster];              // arrivals | child 0, 1 kinematic << 8
};

template <bool first>
__global__ void __launch_bounds__(kBlock, 5) k_refit_clusters(TreeView A, TreeView B, const float* __restrict__ vbox) {
  pdl_entry();
  __shared__ ClusterTree S;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t nA = A.n > 0 ? A.n_lists[1] : 0, nB = B.n > 0 ? B.n_lists[1] : 0;
  for (int64_t c = blockIdx.x; c < nA + nB; c += gridDim.x) {
    const bool inA = c < nA;
    const int64_t cl = inA ? c : c - nA, n = inA ? A.n : B.n;
    const int4 entry = __ldg((inA ? A.cluster : B.cluster) + cl);
    const int32_t begin = entry.x, leaves = entry.y & 0xffff, treelets = entry.y >> 16;
    const int4* list = (inA ? A.treelet : B.treelet) + entry.w;
    const int4* leaf_info = inA ? A.leaf_info : B.leaf_info;
    float* leaf_box = inA ? A.leaf_box : B.leaf_box;
    const int32_t* parent = inA ? A.parent : B.parent;
    BvhNode* nodes = inA ? A.nodes : B.nodes;
    for (int l = t; l < leaves; l += kBlock) {
      const int64_t node = (int64_t)begin + l;
      S.parent[l] = node > 0 && node < n - 1 ? __ldg(parent + node) : -1;
      S.flag[l] = 0;
    }
    int4 en = make_int4(0, 0, 0, 0);
    if (warp < treelets) en = __ldg(list + warp);
    for (int k = warp; k < treelets; k += kBlock / 32) {
      const int64_t l = en.x + (int64_t)lane;
      const bool have = lane < en.y;
      if (k + kBlock / 32 < treelets) en = __ldg(list + k + kBlock / 32);
      float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
      int kin = 1;
      if (have) {
        const int4 li = __ldg(leaf_info + l);
        verts_box(vbox, li.x, li.y, li.z, lo, hi);
        kin = li.w & 1;
        float4* o = reinterpret_cast<float4*>(leaf_box + 8 * l);
        o[0] = make_float4(lo[0], lo[1], lo[2], hi[0]);
        o[1] = make_float4(hi[1], hi[2], 0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) { lo[q] = warp_min(lo[q]); hi[q] = warp_max(hi[q]); }
      if (first) kin = __all_sync(0xffffffffu, kin);
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) { S.treelet[k][q] = lo[q]; S.treelet[k][3 + q] = hi[q]; }
        if (first) S.kin[k] = (uint8_t)kin;
      }
    }
    __syncthreads();
    for (int k = t; k < treelets; k += kBlock) {
      float b[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) b[q] = S.treelet[k][q];
      int kin = first ? S.kin[k] : 0;
      int32_t ps = __ldg(&list[k].z);
      for (int step = 0; step < kCluster; ++step) {      // a path within the cluster has fewer nodes
        if (ps == entry.z) {                     // the cluster's root
          float4* o = reinterpret_cast<float4*>((inA ? A.part_box : B.part_box) + 8 * cl);
          o[0] = make_float4(b[0], b[1], b[2], b[3]);
          o[1] = make_float4(b[4], b[5], __int_as_float(kin), 0.f);
          break;
        }
        const int32_t node = ps >> 1, slot = ps & 1, at = node - begin;
        float2* mine = reinterpret_cast<float2*>(nodes[node].box[slot]);
        mine[0] = make_float2(b[0], b[1]);
        mine[1] = make_float2(b[2], b[3]);
        mine[2] = make_float2(b[4], b[5]);
#pragma unroll
        for (int q = 0; q < 6; ++q) S.box[at][slot][q] = b[q];
        __threadfence_block();
        const int old = atomicAdd(&S.flag[at], 1 + (kin << (8 + slot)));
        if ((old & 255) == 0) break;
        __threadfence_block();
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          b[q] = fminf(b[q], S.box[at][slot ^ 1][q]);
          b[3 + q] = fmaxf(b[3 + q], S.box[at][slot ^ 1][3 + q]);
        }
        if (first) {
          const int sib = (old >> (8 + (slot ^ 1))) & 1;
          nodes[node].kin = (kin << slot) | (sib << (slot ^ 1));
          kin &= sib;
        }
        ps = S.parent[at];
      }
    }
    __syncthreads();                             // before the next cluster takes the shared arrays
  }
}

struct TopTree {
  float box[kUpper][2][6];             // of the children of the nodes above the clusters, by number
  int32_t flag[kUpper];                // arrivals | child 0, 1 kinematic << 8
  int2 node[kUpper];                   // node, numbered parent << 1 | slot (-1: the root)
};

template <bool first>
__device__ __forceinline__ void climb_in_shared(const TreeView& T, int clusters, TopTree& S) {
  for (int k = threadIdx.x; k < clusters - 1; k += blockDim.x) {
    S.node[k] = T.upper[k];
    S.flag[k] = 0;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < clusters; c += blockDim.x) {
    int32_t ps = T.cluster_up[c];
    const float4* tb = reinterpret_cast<const float4*>(T.part_box + 8 * (int64_t)c);
    const float4 t0 = __ldg(tb), t1 = __ldg(tb + 1);
    float b[6] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y};
    int kin = first ? __float_as_int(t1.z) : 0;
    for (int step = 0; step < kUpper && ps >= 0; ++step) {     // a path has fewer nodes
      const int32_t at = ps >> 1, slot = ps & 1;
      const int2 node = S.node[at];
      float2* mine = reinterpret_cast<float2*>(T.nodes[node.x].box[slot]);
      mine[0] = make_float2(b[0], b[1]);
      mine[1] = make_float2(b[2], b[3]);
      mine[2] = make_float2(b[4], b[5]);
#pragma unroll
      for (int q = 0; q < 6; ++q) S.box[at][slot][q] = b[q];
      __threadfence_block();
      const int old = atomicAdd(&S.flag[at], 1 + (kin << (8 + slot)));
      if ((old & 255) == 0) break;
      __threadfence_block();
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        b[q] = fminf(b[q], S.box[at][slot ^ 1][q]);
        b[3 + q] = fmaxf(b[3 + q], S.box[at][slot ^ 1][3 + q]);
      }
      if (first) {
        const int sib = (old >> (8 + (slot ^ 1))) & 1;
        T.nodes[node.x].kin = (kin << slot) | (sib << (slot ^ 1));
        kin &= sib;
      }
      ps = node.y;
    }
  }
}

template <bool first>
__global__ void __launch_bounds__(kTopThreads) k_refit_climb(TreeView A, TreeView B, bool clusters) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char top_smem[];
  const int list = clusters ? 1 : 0;
  int64_t nA = A.n > 0 ? A.n_lists[list] : 0, nB = B.n > 0 ? B.n_lists[list] : 0;
  if (clusters) {                                    // blocks 0 and 1: a tree each in shared memory
    TopTree& S = *reinterpret_cast<TopTree*>(top_smem);
    const int64_t wA = nA, wB = nB;
    if (wA <= kUpper + 1) nA = 0;
    if (wB <= kUpper + 1) nB = 0;
    if (blockIdx.x == 0 && nA == 0) climb_in_shared<first>(A, (int)wA, S);
    if (blockIdx.x == 1 && nB == 0) climb_in_shared<first>(B, (int)wB, S);
  }
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nA + nB; k += grid_stride()) {
    const bool inA = k < nA;
    int32_t ps = (clusters ? (inA ? A.cluster + k : B.cluster + (k - nA)) : (inA ? A.treelet + k : B.treelet + (k - nA)))->z;
    if (ps < 0) continue;                            // the whole tree is this subtree
    const float4* tb = reinterpret_cast<const float4*>(inA ? A.part_box + 8 * k : B.part_box + 8 * (k - nA));
    const float4 t0 = __ldg(tb), t1 = __ldg(tb + 1);
    float lo[3] = {t0.x, t0.y, t0.z}, hi[3] = {t0.w, t1.x, t1.y};
    int kin = __float_as_int(t1.z);
    BvhNode* nodes = inA ? A.nodes : B.nodes;
    const int32_t* parent = inA ? A.parent : B.parent;
    int32_t* flag = inA ? A.flag : B.flag;
    const int64_t n = inA ? A.n : B.n;
    for (int64_t step = 0; step < n; ++step) {       // a root path has at most n-1 nodes
      const int32_t node = ps >> 1, slot = ps & 1;
      float2* mine = reinterpret_cast<float2*>(nodes[node].box[slot]);
      __stcg(mine, make_float2(lo[0], lo[1]));
      __stcg(mine + 1, make_float2(lo[2], hi[0]));
      __stcg(mine + 2, make_float2(hi[1], hi[2]));
      if (first && kin) atomicOr(&nodes[node].kin, 1 << slot);
      const int32_t up = node ? __ldg(parent + node) : 0;      // fetched before the arrival
      if (arrive_first(&flag[node])) break;
      const float2* sib = reinterpret_cast<const float2*>(nodes[node].box[slot ^ 1]);
      const float2 a = __ldcg(sib), b = __ldcg(sib + 1), c = __ldcg(sib + 2);
      lo[0] = fminf(lo[0], a.x); lo[1] = fminf(lo[1], a.y); lo[2] = fminf(lo[2], b.x);
      hi[0] = fmaxf(hi[0], b.y); hi[1] = fmaxf(hi[1], c.x); hi[2] = fmaxf(hi[2], c.y);
      if (first) kin = (__ldcg(&nodes[node].kin) & 3) == 3;
      if (node == 0) break;
      ps = up;
    }
  }
}

__device__ __forceinline__ bool box_overlap(const float* lo, const float* hi, const float qlo[3], const float qhi[3]) {
  return !((lo[0] > qhi[0]) | (qlo[0] > hi[0]) | (lo[1] > qhi[1]) | (qlo[1] > hi[1]) | (lo[2] > qhi[2]) |
           (qlo[2] > hi[2]));
}

// ---------------------------------------------------------------- traversal
// A warp answers up to 32 queries that are neighbours in Morton order.  Instructions bound it, then the
// chain of dependent node reads.  (1) It walks the nodes above the treelets with two boxes, the
// unions of its queries before and after their largest jump, sixteen waiting nodes at a time, a
// lane per child box: nearly always a level of the tree per step, from the (up to sixteen) nodes
// four levels below the root: 13 steps on the 256-scene batch.  The two meet 11 treelets there and the queries themselves 9, while tests of every node
// by every query (one node a step) took 33 steps of more instructions each.  (With one union a
// percent of the warps met hundreds of nodes and held up the kernel; queries so scattered that
// two do not do go on in the one-node form.)  (2) Each query tests the boxes of those treelets;
// the ballot is the set of queries that the treelet concerns.  (3) A treelet is tested a lane per
// leaf: its leaf boxes arrive in one coalesced read, fetched one treelet ahead, and each query
// that met the treelet is compared with all its leaves at once.  Candidates go to a buffer of
// the warp and out with one global atomic per flush.  With every query testing every node, with the
// unions, and with branch-free leaf tests, unions in shared memory and the start below the root:
// bubble grasp's contact set 181, 157 and 118 us, 256-scene batch 2,230, 2,036 and 1,581 us, sphere
// on pad 53, 41 and 20 us (with 8 queries a warp).  Four blocks of 256 an SM: with five, spilled
// registers and a smaller L1 cost 9 % of the contact set; with three, 2 %.
constexpr int kQueryBuf = 128;         // candidates; flushed when a treelet's 32 might not fit
constexpr int kNear = 64;              // treelets; handled when a step's 32 might not fit
constexpr int kWaiting = 128;          // nodes to visit
constexpr int kWaitingWide = 48;       // past this the queries are taken as scattered: one node at a time from then on

struct QueryWarp {
  float4 box[32][2];                   // lo xyz, hi x | hi yz, -, own leaf position
  float4 walk[3];                      // the two unions' lo xyz, hi xyz
  int4 info[32];                       // vertices a, b (PT: both the vertex), id, kin | group << 1
  float4 near[kNear][2];               // lo xyz, hi x | hi yz, first leaf, leaves | kin << 8
  uint64_t cand[kQueryBuf];
  int32_t waiting[kWaiting];
};

__device__ __forceinline__ void flush_candidates(QueryWarp& W, int count, uint64_t* cand, int64_t* n_cand, int64_t cap,
                                                 DevStatus* st, int lane) {
  __syncwarp();
  if (count > 0) {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(reinterpret_cast<unsigned long long*>(n_cand), (unsigned long long)count);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int k = lane; k < count; k += 32) {
      const int64_t pos = (int64_t)base + k;
      if (pos < cap) cand[pos] = W.cand[k];
    }
    if (lane == 0 && (int64_t)base + count > cap) {
      raise_flag(st, EIPC_FLAG_CAND_OVERFLOW);
      raise_need(st, &st->need_cand, (int64_t)base + count);
    }
  }
  __syncwarp();
}

__global__ void __launch_bounds__(256, 4) k_query(Bvh tt, Bvh te, Topo T, int per, const uint32_t* __restrict__ vertex_order,
                                               const float* __restrict__ vbox_q, uint64_t* cand, int64_t* n_cand,
                                               int64_t cap, DevStatus* st) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char query_smem[];
  QueryWarp& W = reinterpret_cast<QueryWarp*>(query_smem)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const int64_t pt_warps = tt.n > 0 ? (T.nv + per - 1) / per : 0, ee_warps = te.n > 0 ? (T.ne + per - 1) / per : 0;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < pt_warps + ee_warps; w += nw) {
    const bool pt = w < pt_warps;
    const BvhNode* nodes = pt ? tt.nodes : te.nodes;
    const float* leaf_box = pt ? tt.leaf_box : te.leaf_box;
    const int4* leaf_info = pt ? tt.leaf_info : te.leaf_info;
    const uint32_t* leaf_prim = pt ? tt.prim : te.prim;
    const int32_t n_leaves = (int32_t)(pt ? tt.n : te.n);
    const int64_t qi = per * (pt ? w : w - pt_warps) + lane;
    // the lane's query; a lane past the end has an empty box
    float qlo[3] = {INFINITY, INFINITY, INFINITY}, qhi[3] = {-INFINITY, -INFINITY, -INFINITY};
    int32_t qpos = INT32_MAX;
    bool kin = true;
    if (lane < per && qi < (pt ? T.nv : T.ne)) {
      const int32_t id = (int32_t)(pt ? vertex_order[qi] : leaf_prim[qi]);
      int32_t a = id, b = id;
      if (pt) {
        kin = T.vkin[id];
        qpos = -1;
      } else {
        const int2 e = reinterpret_cast<const int2*>(T.edges)[id];
        a = e.x; b = e.y;
        kin = T.ekin[id];
        qpos = (int32_t)qi;                // each EE pair is found once, from the edge earlier in Morton order
      }
      verts_box(vbox_q, a, pt ? -1 : b, -1, qlo, qhi);
      W.info[lane] = make_int4(a, b, id, (kin ? 1 : 0) | (T.vgroup[a] << 1));
      W.box[lane][0] = make_float4(qlo[0], qlo[1], qlo[2], qhi[0]);
      W.box[lane][1] = make_float4(qhi[1], qhi[2], 0.f, __int_as_float(qpos));
    }
    // the queries from `cut` on, whose box with its predecessor's is the longest, have a union of
    // their own
    float jump = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float plo = __shfl_up_sync(0xffffffffu, qlo[k], 1), phi = __shfl_up_sync(0xffffffffu, qhi[k], 1);
      jump = fmaxf(jump, fmaxf(qhi[k], phi) - fminf(qlo[k], plo));
    }
    if (lane == 0 || !(jump < INFINITY)) jump = 0.f;
    const int cut = __ffs(__ballot_sync(0xffffffffu, jump == warp_max(jump))) - 1;
    {
      float u[12];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        u[k] = warp_min(lane < cut ? qlo[k] : INFINITY);
        u[3 + k] = warp_max(lane < cut ? qhi[k] : -INFINITY);
        u[6 + k] = warp_min(lane < cut ? INFINITY : qlo[k]);
        u[9 + k] = warp_max(lane < cut ? -INFINITY : qhi[k]);
      }
      if (lane == 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) W.walk[k] = make_float4(u[4 * k], u[4 * k + 1], u[4 * k + 2], u[4 * k + 3]);
    }
    const int32_t upos = __reduce_min_sync(0xffffffffu, qpos);
    const bool ukin = __all_sync(0xffffffffu, kin);
    __syncwarp();
    int kept = 0, listed = 0;                // candidates and treelets in the buffers (the same in all lanes)
    auto handle = [&]() {
      for (int base = 0; base < listed; base += 32) {
        const int m = listed - base < 32 ? listed - base : 32;
        unsigned mask = 0;                   // lane t: the queries that meet treelet t
        for (int t = 0; t < m; ++t) {
          const float4 b0 = W.near[base + t][0], b1 = W.near[base + t][1];
          const float lo[3] = {b0.x, b0.y, b0.z}, hi[3] = {b0.w, b1.x, b1.y};
          const int tail = __float_as_int(b1.w), last = __float_as_int(b1.z) + (tail & 255) - 1;
          const unsigned meet = __ballot_sync(0xffffffffu, box_overlap(lo, hi, qlo, qhi) && last > qpos && !(kin && tail > 255));
          if (lane == t) mask = meet;
        }
        unsigned live = __ballot_sync(0xffffffffu, mask != 0);
        float4 nb0 = make_float4(0.f, 0.f, 0.f, 0.f), nb1 = nb0;
        int4 nli = make_int4(0, 0, 0, 0);
        int nfirst = 0, ncount = 0;
        auto fetch = [&](int t) {
          nfirst = __float_as_int(W.near[base + t][1].z);
          ncount = __float_as_int(W.near[base + t][1].w) & 255;
          if (lane < ncount) {
            const float4* p = reinterpret_cast<const float4*>(leaf_box + 8 * ((int64_t)nfirst + lane));
            nb0 = __ldg(p);
            nb1 = __ldg(p + 1);
            nli = __ldg(leaf_info + nfirst + lane);
          }
        };
        if (live) fetch(__ffs(live) - 1);
        while (live) {
          unsigned todo = __shfl_sync(0xffffffffu, mask, __ffs(live) - 1);
          live &= live - 1;
          const float llo[3] = {nb0.x, nb0.y, nb0.z}, lhi[3] = {nb0.w, nb1.x, nb1.y};
          const int4 li = nli;
          const int32_t lpos = lane < ncount ? nfirst + lane : -2;       // -2: below every query's position
          if (live) fetch(__ffs(live) - 1);
          // every query against the lane's leaf without a branch, then the lane's candidates one by
          // one, each lane at its own query
          unsigned hits = 0;
          while (todo) {
            const int q = __ffs(todo) - 1;
            const float4 q0 = W.box[q][0], q1 = W.box[q][1];
            const int4 qn = W.info[q];
            const float blo[3] = {q0.x, q0.y, q0.z}, bhi[3] = {q0.w, q1.x, q1.y};
            // not a candidate if the two share a vertex, are both kinematic or of different scenes
            const bool hit = (lpos > __float_as_int(q1.w)) & box_overlap(llo, lhi, blo, bhi) & (li.x != qn.x) & (li.y != qn.x) &
                             (li.z != qn.x) & (li.x != qn.y) & (li.y != qn.y) & ((unsigned)(li.w ^ qn.w) < 2u) & !(qn.w & li.w & 1);
            if (hit) hits |= todo & (0u - todo);
            todo &= todo - 1;
          }
          while (true) {
            const bool hit = hits != 0;
            const unsigned mh = __ballot_sync(0xffffffffu, hit);
            if (!mh) break;
            if (hit) {
              const uint32_t id = (uint32_t)W.info[__ffs(hits) - 1].z, prim = __ldg(leaf_prim + lpos);
              const uint32_t lo32 = pt ? id : (id < prim ? id : prim), hi32 = pt ? prim : (id < prim ? prim : id);
              W.cand[kept + __popc(mh & below)] = pair_key(pt ? 0 : 1, lo32, hi32, T.bits_i, T.bits_j);
            }
            hits &= hits - 1;
            kept += __popc(mh);
            if (kept > kQueryBuf - 32) {
              flush_candidates(W, kept, cand, n_cand, cap, st, lane);
              kept = 0;
            }
          }
        }
      }
      listed = 0;
      __syncwarp();
    };
    if (n_leaves <= kTreelet) {              // one treelet, met by every query
      if (lane == 0) {
        W.near[0][0] = make_float4(-INFINITY, -INFINITY, -INFINITY, INFINITY);
        W.near[0][1] = make_float4(INFINITY, INFINITY, __int_as_float(0), __int_as_float(n_leaves));
      }
      listed = 1;
    } else {
      const int32_t* top = pt ? tt.top : te.top;
      int held = __ldg(top + kWalkStarts);
      if (lane < held) W.waiting[lane] = __ldg(top + lane);
      bool wide = true;
      int visits = 0;                        // a tree of n leaves has n-1 internal nodes, each fetched at most once
      __syncwarp();
      while (held > 0) {
        wide = wide && held <= kWaitingWide;
        const int take = wide ? (held < 16 ? held : 16) : 1;
        const bool mine = (lane >> 1) < take;
        const int side = lane & 1;
        const int32_t node = mine ? W.waiting[held - 1 - (lane >> 1)] : 0;
        held -= take;
        visits += take;
        if (visits > n_leaves) {
          if (lane == 0) raise_flag(st, EIPC_FLAG_STACK_OVERFLOW);
          break;
        }
        __syncwarp();                        // the entries are read before new ones take their places
        const float2* bp = reinterpret_cast<const float2*>(nodes[node].box[side]);
        const float2 c0 = __ldg(bp), c1 = __ldg(bp + 1), c2 = __ldg(bp + 2);
        const int4 tail = __ldg(reinterpret_cast<const int4*>(&nodes[node].first));       // first, last, kin, split
        const float lo[3] = {c0.x, c0.y, c1.x}, hi[3] = {c1.y, c2.x, c2.y};
        const int32_t first = side ? tail.w + 1 : tail.x, last = side ? tail.y : tail.w;
        const int child_kin = (tail.z >> side) & 1;
        bool meet = mine && last > upos && !(ukin && child_kin);
        if (wide) {
          const float4 w0 = W.walk[0], w1 = W.walk[1], w2 = W.walk[2];
          const float ulo[2][3] = {{w0.x, w0.y, w0.z}, {w1.z, w1.w, w2.x}}, uhi[2][3] = {{w0.w, w1.x, w1.y}, {w2.y, w2.z, w2.w}};
          meet = meet & (box_overlap(lo, hi, ulo[0], uhi[0]) | box_overlap(lo, hi, ulo[1], uhi[1]));
        } else {                             // lanes 0 and 1 hold the two children
          unsigned met = 0;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            float clo[3], chi[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              clo[k] = __shfl_sync(0xffffffffu, lo[k], c);
              chi[k] = __shfl_sync(0xffffffffu, hi[k], c);
            }
            const int32_t clast = __shfl_sync(0xffffffffu, last, c);
            if (__any_sync(0xffffffffu, box_overlap(clo, chi, qlo, qhi) && clast > qpos)) met |= 1u << c;
          }
          meet = meet && (met >> side & 1u);
        }
        const bool leafy = last - first < kTreelet;
        const unsigned m_near = __ballot_sync(0xffffffffu, meet && leafy), m_next = __ballot_sync(0xffffffffu, meet && !leafy);
        if (meet && leafy) {
          const int k = listed + __popc(m_near & below);
          W.near[k][0] = make_float4(lo[0], lo[1], lo[2], hi[0]);
          W.near[k][1] = make_float4(hi[1], hi[2], __int_as_float(first), __int_as_float((last - first + 1) | (child_kin << 8)));
        } else if (meet) {
          const int k = held + __popc(m_next & below);
          if (k < kWaiting) W.waiting[k] = tail.w + side;
          else raise_flag(st, EIPC_FLAG_STACK_OVERFLOW);
        }
        listed += __popc(m_near);
        held += __popc(m_next);
        if (held > kWaiting) held = kWaiting;
        __syncwarp();
        if (listed > kNear - 32) handle();
      }
    }
    __syncwarp();
    handle();
    flush_candidates(W, kept, cand, n_cand, cap, st, lane);
  }
}

TreeView view(const Bvh& t, const uint64_t* keys) {
  return TreeView{t.n, keys, t.prim, t.nodes, t.parent, t.leaf_info, t.leaf_box, t.flag, t.treelet, t.cluster, t.part_box, t.upper,
                  t.cluster_up, t.top, t.n_lists};
}

template <bool first>
void refit(const TreeView& A, const TreeView& B, const float* vbox, cudaStream_t s) {
  const int64_t n = A.n + B.n;
  const bool clusters = n <= kClusterPrims;
  if (clusters) launch(k_refit_clusters<first>, blocks_for(n, 5), kBlock, 0, s, A, B, vbox);
  else launch(k_refit_leaves, blocks_for(n), kBlock, 0, s, A, B, vbox);
  const int blocks = blocks_for(n / (clusters ? 64 : 8), 4, kTopThreads);
  launch(k_refit_climb<first>, blocks < 2 ? 2 : blocks, kTopThreads, clusters ? sizeof(TopTree) : 0, s, A, B, clusters);
}

}  // namespace

cudaError_t bvh_prepare() {
  const cudaError_t e = cudaFuncSetAttribute(k_refit_climb<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(TopTree));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_refit_climb<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(TopTree));
}

void bvh_build(Broad& b, const Topo& topo, const float* vbox, uint32_t* sort_hist, cudaStream_t s) {
  const int64_t n = topo.nf + topo.ne + topo.nv;
  launch(k_bounds_init, 1, 32, 0, s, b.bounds, b.tri.n_lists, b.edge.n_lists);
  launch(k_bounds, blocks_for(topo.nv, 4), kBlock, 0, s, vbox, topo.nv, b.bounds);
  launch(k_morton_keys, blocks_for(n), kBlock, 0, s, topo, vbox, static_cast<const int32_t*>(b.bounds), b.keys, b.vals);
  const int which = radix_sort_u64(b.keys, b.vals, b.keys_alt, b.vals_alt, b.n_dev, n, 32, sort_hist, s);
  const uint64_t* sk = which ? b.keys_alt : b.keys;
  const uint32_t* sv = which ? b.vals_alt : b.vals;
  b.tri.prim = sv;
  b.edge.prim = sv + topo.nf;
  b.vertex_order = sv + topo.nf + topo.ne;
  const TreeView A = view(b.tri, sk), B = view(b.edge, sk + topo.nf);
  launch(k_internal, blocks_for(topo.nf + topo.ne), kBlock, 0, s, A, B);
  launch(k_tree_parts, blocks_for(2 * (topo.nf + topo.ne)), kBlock, 0, s, A, B, topo);
  launch(k_cluster_treelets, blocks_for(topo.nf + topo.ne), kBlock, 0, s, A, B);
  refit<true>(A, B, vbox, s);
  b.built = true;
}

void bvh_refit(Broad& b, const float* vbox, cudaStream_t s) {
  refit<false>(view(b.tri, nullptr), view(b.edge, nullptr), vbox, s);
}

void bvh_query(const Broad& b, const Topo& topo, const float* vbox_q, uint64_t* cand, int64_t* n_cand, int64_t cap,
               DevStatus* st, cudaStream_t s, int threads, int bps) {
  // queries per warp: 32, but 16 or 8 where that still leaves the warps room on the chip at once (4
  // blocks of 8 an SM): a small scene's time is its slowest warp's.  Sphere
  // on pad 41 us with 32, 25 us with 8
  const int64_t queries = (b.tri.n > 0 ? topo.nv : 0) + (b.edge.n > 0 ? topo.ne : 0);
  const int64_t room = (int64_t)kSMs * 32;
  const int per = queries <= 8 * room ? 8 : (queries <= 16 * room ? 16 : 32);
  const int64_t warps = queries / per + 2;
  if (queries <= 0) return;
  const size_t smem = (size_t)(threads / 32) * sizeof(QueryWarp);
  launch(k_query, blocks_for(32 * warps, bps, threads), threads, smem, s, b.tri, b.edge, topo, per, b.vertex_order, vbox_q, cand,
         n_cand, cap, st);
}

}  // namespace eipc
