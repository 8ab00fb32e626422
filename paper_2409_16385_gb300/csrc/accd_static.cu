// eipc_accd_toi_static: the CCD step bound over a caller-supplied candidate list, with
// its scratch memory in a fixed-size device array compiled into the library, so the call
// allocates no device memory at all.
//
// The caller's candidates are checked and packed into pair keys, kStaticChunk at a time, and go
// through the kernels of the scene-based eipc_accd_toi (ccd_bound_launch): one compiled arithmetic,
// hence the same bits.  (With kernels of its own, whose distances and advances were written
// differently, a third of the advances rounded differently.)  Incident candidates (sharing a vertex)
// are skipped here because the caller builds the list.
#include <mutex>

#include "geometry.cuh"
#include "scene.cuh"

namespace eipc {
namespace {

constexpr int64_t kStaticMaxVertices = 1 << 17;   // 131,072 vertices
constexpr int64_t kStaticChunk = 1 << 18;         // candidates taken at a time

// Layout: a header, then padded x and dx (32 B per vertex each), their FP32 copies (16 B each), and
// two lists of pair keys.
struct StaticHeader {
  DevStatus status;
  unsigned long long alpha_bits;
  int64_t n_adv, n_keys, n_list, queue;
};
constexpr size_t kStaticHeader = 256;
static_assert(sizeof(StaticHeader) <= kStaticHeader, "the header has its room");
constexpr size_t kStaticBytes = kStaticHeader + (size_t)kStaticMaxVertices * (2 * 32 + 2 * 16) + 2 * (size_t)kStaticChunk * 8;

static __device__ __align__(256) unsigned char g_accd_scratch[kStaticBytes];

struct StaticView {
  StaticHeader* head;
  double* x4;
  double* dx4;
  float* x4f;
  float* dx4f;
  uint64_t* keys;
  uint64_t* list;
};

StaticView view_of(unsigned char* base) {
  StaticView v;
  v.head = reinterpret_cast<StaticHeader*>(base);
  unsigned char* p = base + kStaticHeader;
  v.x4 = reinterpret_cast<double*>(p);
  v.dx4 = v.x4 + 4 * kStaticMaxVertices;
  v.x4f = reinterpret_cast<float*>(v.dx4 + 4 * kStaticMaxVertices);
  v.dx4f = v.x4f + 4 * kStaticMaxVertices;
  v.keys = reinterpret_cast<uint64_t*>(v.dx4f + 4 * kStaticMaxVertices);
  v.list = v.keys + kStaticChunk;
  return v;
}

// every call starts from alpha = 1, no flags, no advanced pairs; every chunk from empty lists
__global__ void k_static_init(StaticHeader* h, bool first) {
  pdl_entry();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (first) {
    h->status = DevStatus{};
    h->alpha_bits = (unsigned long long)__double_as_longlong(1.0);
    h->n_adv = 0;
  }
  h->n_keys = h->n_list = h->queue = 0;
}

__global__ void __launch_bounds__(256) k_static_pad(const double* __restrict__ x, const double* __restrict__ dx,
                                                    int64_t nv, StaticView sv) {
  pdl_entry();
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    const double a = x[3 * v], b = x[3 * v + 1], c = x[3 * v + 2];
    const double e = dx[3 * v], f = dx[3 * v + 1], g = dx[3 * v + 2];
    if (!(isfinite(a) && isfinite(b) && isfinite(c) && isfinite(e) && isfinite(f) && isfinite(g)))
      raise_flag(&sv.head->status, EIPC_FLAG_NONFINITE);
    reinterpret_cast<double2*>(sv.x4)[2 * v] = make_double2(a, b);
    reinterpret_cast<double2*>(sv.x4)[2 * v + 1] = make_double2(c, 0.0);
    reinterpret_cast<double2*>(sv.dx4)[2 * v] = make_double2(e, f);
    reinterpret_cast<double2*>(sv.dx4)[2 * v + 1] = make_double2(g, 0.0);
    reinterpret_cast<float4*>(sv.x4f)[v] = make_float4(to_float<0>(a), to_float<0>(b), to_float<0>(c), 0.f);
    reinterpret_cast<float4*>(sv.dx4f)[v] = make_float4(to_float<0>(e), to_float<0>(f), to_float<0>(g), 0.f);
  }
}

// candidates [0, nc) whose ids are in range and that share no vertex, as pair keys
__global__ void __launch_bounds__(kBlock) k_static_keys(Topo T, int64_t nc, const int32_t* __restrict__ ctype,
                                                        const int32_t* __restrict__ ci, const int32_t* __restrict__ cj,
                                                        StaticView sv) {
  pdl_entry();
  const int lane = threadIdx.x & 31;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < nc; base += grid_stride()) {
    const int64_t k = base + threadIdx.x;
    bool keep = false;
    uint64_t key = 0;
    if (k < nc) {
      const int type = ctype[k];
      const int32_t i = ci[k], j = cj[k];
      bool ids_ok = (type == 0) ? (i >= 0 && i < T.nv && j >= 0 && j < T.nf)
                                : (type == 1 && i >= 0 && i < T.ne && j >= 0 && j < T.ne);
      if (ids_ok) {
        int32_t v[4];
        if (type == 0) {
          v[0] = i;
          v[1] = T.tris[3 * (int64_t)j]; v[2] = T.tris[3 * (int64_t)j + 1]; v[3] = T.tris[3 * (int64_t)j + 2];
        } else {
          v[0] = T.edges[2 * (int64_t)i]; v[1] = T.edges[2 * (int64_t)i + 1];
          v[2] = T.edges[2 * (int64_t)j]; v[3] = T.edges[2 * (int64_t)j + 1];
        }
        for (int a = 0; a < 4; ++a) ids_ok = ids_ok && v[a] >= 0 && v[a] < T.nv;
        const int na = type == 0 ? 1 : 2;
        bool incident = false;
        for (int a = 0; a < na; ++a)
          for (int b = na; b < 4; ++b) incident |= (v[a] == v[b]);
        keep = ids_ok && !incident;
        key = pair_key(type, (uint32_t)i, (uint32_t)j, T.bits_i, T.bits_j);
      }
      if (!ids_ok) raise_flag(&sv.head->status, EIPC_FLAG_BAD_INDEX);
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, keep);
    if (mask) {
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(reinterpret_cast<unsigned long long*>(&sv.head->n_keys), (unsigned long long)__popc(mask));
      b = __shfl_sync(0xffffffffu, b, 0);
      // keys never outnumber the chunk's candidates
      if (keep) sv.keys[(int64_t)b + __popc(mask & ((1u << lane) - 1u))] = key;
    }
  }
}

__global__ void k_static_out(const StaticHeader* h, double* alpha, int32_t* flags, int64_t* n_adv) {
  pdl_entry();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    *alpha = __longlong_as_double((long long)h->alpha_bits);
    if (flags) *flags = h->status.flags;
    if (n_adv) *n_adv = h->n_adv;
  }
}

// Device address of g_accd_scratch, looked up once per device with that device current.
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_addr[kMaxDevices] = {};

cudaError_t scratch_address(unsigned char** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_accd_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_addr[dev] = p;
  }
  *out = static_cast<unsigned char*>(g_scratch_addr[dev]);
  return cudaSuccess;
}

}  // namespace
}  // namespace eipc

extern "C" int64_t eipc_accd_static_max_vertices(void) { return eipc::kStaticMaxVertices; }

extern "C" eipc_status eipc_accd_toi_static(int64_t Nv, int64_t F, int64_t E, const double* x, const double* dx,
                                            const int32_t* tris,
                                            const int32_t* edges, int64_t n_cand, const int32_t* cand_type,
                                            const int32_t* cand_i, const int32_t* cand_j, const eipc_params* p,
                                            double* alpha, int32_t* flags, int64_t* n_advanced,
                                            eipc_stream stream) {
  using namespace eipc;
  if (Nv <= 0 || Nv > kStaticMaxVertices) return EIPC_ERR_TOO_LARGE;
  if (!x || !dx || !alpha || !p || F < 0 || E < 0 || n_cand < 0 || n_cand >= (1ll << 31)) return EIPC_ERR_INVALID;
  if (n_cand > 0 && (!tris || !edges || !cand_type || !cand_i || !cand_j)) return EIPC_ERR_INVALID;
  if (!(p->accd_s > 0.0 && p->accd_s < 1.0 && p->accd_max_iter > 0)) return EIPC_ERR_INVALID;
  unsigned char* base = nullptr;
  if (scratch_address(&base) != cudaSuccess) return EIPC_ERR_CUDA;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const StaticView sv = view_of(base);
  launch(k_static_init, 1, 32, 0, s, sv.head, true);
  launch(k_static_pad, blocks_for(Nv, 4), kBlock, 0, s, x, dx, Nv, sv);
  Topo T{};
  T.nv = Nv; T.ne = E; T.nf = F;
  T.tris = tris; T.edges = edges;
  constexpr int64_t kMaxId = (1ll << 31) - 1;        // ids are 32 bits wide, whatever the counts
  const int64_t most_i = Nv > E ? Nv : E, most_j = F > E ? F : E;
  T.bits_i = bits_for((uint64_t)(most_i < kMaxId ? most_i : kMaxId));
  T.bits_j = bits_for((uint64_t)(most_j < kMaxId ? most_j : kMaxId));
  for (int64_t k = 0; k < n_cand; k += kStaticChunk) {
    const int64_t n = n_cand - k < kStaticChunk ? n_cand - k : kStaticChunk;
    if (k > 0) launch(k_static_init, 1, 32, 0, s, sv.head, false);
    launch(k_static_keys, blocks_for(n, 8), kBlock, 0, s, T, n, cand_type + k, cand_i + k, cand_j + k, sv);
    ccd_bound_launch(CcdBound{T, sv.x4, sv.dx4, sv.x4f, sv.dx4f, sv.keys, &sv.head->n_keys, n, sv.list, &sv.head->n_list,
                              &sv.head->n_adv, &sv.head->queue, p->accd_s, (int)p->accd_max_iter, &sv.head->alpha_bits, nullptr,
                              &sv.head->status, 32},
                     s);
  }
  launch(k_static_out, 1, 32, 0, s, static_cast<const StaticHeader*>(sv.head), alpha, flags, n_advanced);
  return cudaPeekAtLastError() == cudaSuccess ? EIPC_OK : EIPC_ERR_CUDA;
}
