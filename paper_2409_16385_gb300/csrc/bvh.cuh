// Linear BVH over the surface primitives (Karras 2012 construction on 30-bit Morton codes),
// cut into treelets of at most 32 consecutive leaves, and the traversal that produces
// candidate pairs for the contact set and for the CCD step bound.  Boxes are FP32 rounded
// outward from the FP64 positions, so a box test never rejects a pair that the exact FP64
// test would keep.
#pragma once
#include "common.cuh"

namespace eipc {

// One internal node holds the boxes of both children so a traversal step is one 64-byte
// fetch.  It covers the leaves [first, last]; child 0 the leaves up to `split`, child 1 the
// rest.  A child of several leaves is internal node `split` (child 0) or `split` + 1 (child 1).
// Only nodes of more than kTreelet leaves carry boxes.
struct alignas(16) BvhNode {
  float box[2][6];       // lo xyz, hi xyz of child 0, child 1
  int32_t first, last;
  int32_t kin;           // bit 0 / bit 1: every primitive under child 0 / 1 is kinematic
  int32_t split;
};

struct Bvh {
  int64_t n;             // primitives (static per scene)
  BvhNode* nodes;        // [n-1]
  int32_t* parent;       // [2n-1]: parent << 1 | slot (0: child 0, 1: child 1); internal i at i, leaf l at n-1+l
  const uint32_t* prim;  // [n] primitive of each leaf (Morton order): a part of the scene's sorted ids
  int4* leaf_info;       // [n] per leaf: vertex ids (-1 if unused), kinematic flag | scene group << 1
  float* leaf_box;       // [8n] per leaf: lo xyz, hi xyz, two unused
  int32_t* flag;         // [n] arrivals at each internal node (two per refit)
  int4* treelet;         // [n] first leaf, leaves, parent << 1 | slot (-1: none) of each treelet
  int4* cluster;         // [n] first leaf, leaves | treelets << 16, parent << 1 | slot (-1: none), first treelet
  float* part_box;       // [8n] of each cluster (large scenes: treelet): lo xyz, hi xyz, all kinematic, one unused
  int2* upper;           // [kUpper] the nodes above the clusters: node, numbered parent << 1 | slot (-1: none)
  int32_t* cluster_up;   // [kUpper + 1] each cluster's numbered parent << 1 | slot
  int32_t* top;          // [kWalkStarts + 1] the nodes a walk starts from, and their number
  int32_t* n_lists;      // [3] treelets, clusters, nodes above the clusters
};

// leaves per treelet: one warp refits one, and tests one against a query with a lane per leaf
constexpr int kTreelet = 32;
// leaves per cluster: one block refits one in shared memory
constexpr int kCluster = 512;
// nodes above the clusters that one block climbs in shared memory
constexpr int kUpper = 2048;
constexpr int kTopThreads = 512;
// nodes that a traversal's walk starts from, at most: one step of a warp
constexpr int kWalkStarts = 16;

enum PrimKind { kVertex = 0, kEdge = 1, kTri = 2 };

// Static topology needed by the broad and narrow phases.
struct Topo {
  int64_t nv, ne, nf;
  const int32_t* tris;   // [nf*3]
  const int32_t* edges;  // [ne*2]
  const uint8_t* vkin;   // [nv]
  const uint8_t* ekin;   // [ne] both ends kinematic
  const uint8_t* fkin;   // [nf] all three kinematic
  const int32_t* vgroup; // [nv] independent-scene id of each vertex (0 when not batched)
  int bits_i, bits_j;    // pair key packing
};

// Pair key: type << (bi+bj) | i << bj | j, ordered like (type, i, j).
__host__ __device__ __forceinline__ uint64_t pair_key(int type, uint32_t i, uint32_t j, int bi, int bj) {
  return ((uint64_t)type << (bi + bj)) | ((uint64_t)i << bj) | (uint64_t)j;
}

// Both hierarchies and the vertices' Morton order, with the scratch of their common sort.
struct Broad {
  Bvh tri, edge;
  const uint32_t* vertex_order;  // [nv] vertices in Morton order (of the last build)
  uint64_t* keys;                // [nf + ne + nv]
  uint64_t* keys_alt;
  uint32_t* vals;
  uint32_t* vals_alt;
  int64_t* n_dev;                // [1] nf + ne + nv
  int32_t* bounds;               // [6]
  bool built;
};

// Lets the refit's climb use its shared memory; once per scene, on the scene's device.
cudaError_t bvh_prepare();

// Builds both trees from the per-vertex boxes vbox (swept ones for CCD).
void bvh_build(Broad& b, const Topo& topo, const float* vbox, uint32_t* sort_hist, cudaStream_t s);

// Refits the hierarchies of the last bvh_build with new per-vertex boxes: any binary tree over
// the primitives with conservative boxes gives the same exact candidate set, so the Morton
// sort and the hierarchies can be reused while the topology stays.
void bvh_refit(Broad& b, const float* vbox, cudaStream_t s);

// Traverses both trees in one launch: every vertex box (from vbox_q: the per-vertex boxes
// grown by the contact distance, or swept for CCD) against the triangle tree -> PT
// candidates, every edge box against the edge tree -> EE candidates with j > i.  Incident
// pairs, all-kinematic pairs and pairs across groups are skipped; candidates are appended as
// pair keys to cand[0..cap) with the running count in *n_cand, and an overflow raises
// CAND_OVERFLOW.
void bvh_query(const Broad& b, const Topo& topo, const float* vbox_q, uint64_t* cand, int64_t* n_cand, int64_t cap,
               DevStatus* st, cudaStream_t s, int threads, int bps);

}  // namespace eipc
