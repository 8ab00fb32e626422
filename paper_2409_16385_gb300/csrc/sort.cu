// Stable LSD radix sort, exclusive scan and segment starts with device-resident element
// counts.
//
// A radix pass (8-bit digit) is one launch, a sort one more: one block per SM owns one contiguous
// chunk of the input.  (1) Before the first pass, per-block digit histograms.  (2) A pass: each
// block sums the histograms of the blocks before it and of all blocks (152 x 256 counters, four
// threads per digit), scans the 256 totals for its digit bases and scatters its chunk tile by
// tile: warp peers with equal digits are found with __match_any_sync and per-warp digit counts are
// prefix-summed across the block's 32 warps, so every element lands at a position that preserves
// input order among equal digits (stability is what makes the sort-and-reduce of the reduced
// Hessian deterministic).  The sorts of a step are short (a few thousand to a few hundred
// thousand elements), so a pass costs its launches:
// with 1,216 blocks a third one had to turn the counters into offsets.  An element's next digit is
// counted for the chunk that it is scattered to, so later passes need no histograms of their
// own (integer atomics: the counts do not depend on their order).  A block takes at least a
// whole tile, so that short inputs have few counters to sum.  Caches flushed, a
// pass of the sphere on pad (a few thousand) took 14.6 us in three launches, 11 us in two, 6.5 us
// and 5 us once a sort so; of the bubble grasp (2 x 10^5) 17.7, 19.5, and 15.8 us and 6.4 us once.
#include "common.cuh"
#include "sort.cuh"

namespace eipc {
namespace {

__device__ __forceinline__ uint32_t chunk_size(int64_t n) {
  const int64_t per = (n + kSortBlocks - 1) / kSortBlocks;
  return (uint32_t)(per > kSortThreads ? (per + 31) / 32 * 32 : kSortThreads);     // at least one whole tile: fewer counters to sum
}

__device__ __forceinline__ int chunk_range(int64_t n, int64_t* beg, int64_t* end) {
  const int64_t per = chunk_size(n);
  *beg = (int64_t)blockIdx.x * per;
  int64_t e = *beg + per;
  *end = e < n ? e : n;
  return (int)((n + per - 1) / per);           // blocks that have elements
}

__global__ void __launch_bounds__(kSortThreads) k_hist(const uint64_t* __restrict__ keys,
                                                       const int64_t* n_dev, int64_t cap, int shift,
                                                       uint32_t* __restrict__ hist, uint32_t* __restrict__ hist_next) {
  pdl_entry();
  __shared__ uint32_t h[256];
  if (threadIdx.x < 256) h[threadIdx.x] = 0;
  __syncthreads();
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  chunk_range(n, &beg, &end);
  if (beg >= end) return;                       // its counters are not read
  // one shared-memory atomic per distinct digit of a warp's 32 elements (keys can be heavily
  // skewed)
  const uint32_t lt_mask = (1u << (threadIdx.x & 31)) - 1u;
  for (int64_t i0 = beg; i0 < end; i0 += kSortThreads) {
    const int64_t i = i0 + threadIdx.x;
    const uint32_t d = i < end ? (uint32_t)((keys[i] >> shift) & 255u) : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    if (d < 256u && (peers & lt_mask) == 0u) atomicAdd(&h[d], (uint32_t)__popc(peers));
  }
  __syncthreads();
  if (threadIdx.x < 256) {
    hist[256 * blockIdx.x + threadIdx.x] = h[threadIdx.x];
    hist_next[256 * blockIdx.x + threadIdx.x] = 0;
  }
}

__global__ void __launch_bounds__(kSortThreads) k_scatter(const uint64_t* __restrict__ kin,
                                                          const uint32_t* __restrict__ vin,
                                                          uint64_t* __restrict__ kout,
                                                          uint32_t* __restrict__ vout,
                                                          const int64_t* n_dev, int64_t cap, int shift,
                                                          const uint32_t* __restrict__ hist,
                                                          uint32_t* hist_next, uint32_t* __restrict__ hist_clear,
                                                          bool more) {
  pdl_entry();
  constexpr int W = kSortThreads / 32;
  __shared__ uint32_t base[256];
  __shared__ uint32_t wcnt[W][257];
  __shared__ uint32_t part[4][256];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int d = t & 255, q = t >> 8;            // digit and quarter of this thread in the digit sums
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  const int blocks = chunk_range(n, &beg, &end);
  if (beg >= end) return;
  const uint32_t per = chunk_size(n);
  if (t < 256) hist_clear[256 * blockIdx.x + t] = 0;
  {
    uint32_t before = 0, all = 0;
#pragma unroll 8
    for (int b = q; b < blocks; b += 4) {
      const uint32_t c = __ldg(hist + 256 * b + d);
      all += c;
      before += b < (int)blockIdx.x ? c : 0u;
    }
    part[q][d] = before;
    wcnt[q][d] = all;
  }
  __syncthreads();
  uint32_t total = 0, incl = 0;
  if (t < 256) {                                // digit bases: exclusive scan of the 256 totals, plus this block's prefix
    total = wcnt[0][t] + wcnt[1][t] + wcnt[2][t] + wcnt[3][t];
    incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wcnt[4][warp] = incl;
  }
  __syncthreads();
  if (t < 256) {
    uint32_t run = incl - total + part[0][t] + part[1][t] + part[2][t] + part[3][t];
    for (int w = 0; w < warp; ++w) run += wcnt[4][w];
    base[t] = run;
  }
  __syncthreads();
  const uint32_t lt_mask = (1u << lane) - 1u;
  for (int64_t tile = beg; tile < end; tile += kSortThreads) {
    for (int e = lane; e < 257; e += 32) wcnt[warp][e] = 0;
    __syncwarp();
    const int64_t i = tile + t;
    const bool valid = i < end;
    const uint64_t key = valid ? kin[i] : 0;
    const uint32_t val = valid ? vin[i] : 0;
    const uint32_t digit = valid ? (uint32_t)((key >> shift) & 255u) : 256u;
    const uint32_t peers = __match_any_sync(0xffffffffu, digit);
    const uint32_t rank = __popc(peers & lt_mask);
    if (rank == 0) wcnt[warp][digit] = __popc(peers);
    __syncthreads();
    {                                           // eight warps' counts of digit d by each of its four threads
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < W / 4; ++w) {
        const uint32_t c = wcnt[q * (W / 4) + w][d];
        wcnt[q * (W / 4) + w][d] = run;
        run += c;
      }
      part[q][d] = run;
    }
    __syncthreads();
    if (valid) {
      uint32_t pos = base[digit] + wcnt[warp][digit] + rank;
      const int wq = warp / (W / 4);
      for (int p = 0; p < wq; ++p) pos += part[p][digit];
      kout[pos] = key;
      vout[pos] = val;
      if (more) atomicAdd(hist_next + 256 * (pos / per) + (uint32_t)((key >> (shift + 8)) & 255u), 1u);
    }
    __syncthreads();
    if (t < 256) base[t] += part[0][t] + part[1][t] + part[2][t] + part[3][t];
  }
}

// ---------------------------------------------------------------- exclusive scan
__device__ __forceinline__ void scan_range(int64_t n, int64_t* beg, int64_t* end) {
  int64_t per = (n + kScanBlocks - 1) / kScanBlocks;
  *beg = (int64_t)blockIdx.x * per;
  int64_t e = *beg + per;
  *end = e < n ? e : n;
}

__device__ int64_t block_sum_i64(int64_t v) {
  __shared__ int64_t ws[32];
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  int64_t r = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += ws[w];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(256) k_scan_partial(const int64_t* __restrict__ in, const int64_t* n_dev,
                                                      int64_t cap, int64_t* __restrict__ partial) {
  pdl_entry();
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t s = 0;
  for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) s += in[i];
  s = block_sum_i64(s);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void __launch_bounds__(256) k_scan_apply(const int64_t* __restrict__ in, int64_t* __restrict__ out,
                                                    const int64_t* n_dev, int64_t cap,
                                                    const int64_t* __restrict__ partial, int64_t* total) {
  pdl_entry();
  __shared__ int64_t tile_sum[256];
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t all;
  int64_t run = partials_before(partial, blockIdx.x, &all);
  const int t = threadIdx.x;
  if (total && blockIdx.x == 0 && t == 0) *total = all;
  for (int64_t tile = beg; tile < end; tile += 256) {
    int64_t i = tile + t;
    int64_t v = (i < end) ? in[i] : 0;
    tile_sum[t] = v;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {
      int64_t u = (t >= off) ? tile_sum[t - off] : 0;
      __syncthreads();
      tile_sum[t] += u;
      __syncthreads();
    }
    if (i < end) out[i] = run + tile_sum[t] - v;
    int64_t tot = tile_sum[255];
    __syncthreads();
    run += tot;
  }
}

// ---- two exclusive scans of the same length in the launches of one: partial holds
// 2 kScanBlocks entries, the first array's partials then the second's
__global__ void __launch_bounds__(256) k_scan2_partial(const int64_t* __restrict__ a, const int64_t* __restrict__ b,
                                                       const int64_t* n_dev, int64_t cap, int64_t* __restrict__ partial) {
  pdl_entry();
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t sa = 0, sb = 0;
  for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) {
    sa += a[i];
    sb += b[i];
  }
  sa = block_sum_i64(sa);
  sb = block_sum_i64(sb);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = sa;
    partial[kScanBlocks + blockIdx.x] = sb;
  }
}

// both arrays' tiles: one block-wide scan of (a, b) pairs per tile
__global__ void __launch_bounds__(256) k_scan2_apply(const int64_t* __restrict__ a, int64_t* __restrict__ out_a,
                                                     const int64_t* __restrict__ b, int64_t* __restrict__ out_b,
                                                     const int64_t* n_dev, int64_t cap,
                                                     const int64_t* __restrict__ partial, int64_t* total_a,
                                                     int64_t* total_b) {
  pdl_entry();
  __shared__ int64_t ta[256], tb[256];
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t all_a, all_b;
  int64_t run_a = partials_before(partial, blockIdx.x, &all_a), run_b = partials_before(partial + kScanBlocks, blockIdx.x, &all_b);
  const int t = threadIdx.x;
  if (blockIdx.x == 0 && t == 0) {
    *total_a = all_a;
    *total_b = all_b;
  }
  for (int64_t tile = beg; tile < end; tile += 256) {
    const int64_t i = tile + t;
    const int64_t va = (i < end) ? a[i] : 0, vb = (i < end) ? b[i] : 0;
    ta[t] = va;
    tb[t] = vb;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {
      const int64_t ua = (t >= off) ? ta[t - off] : 0, ub = (t >= off) ? tb[t - off] : 0;
      __syncthreads();
      ta[t] += ua;
      tb[t] += ub;
      __syncthreads();
    }
    if (i < end) {
      out_a[i] = run_a + ta[t] - va;
      out_b[i] = run_b + tb[t] - vb;
    }
    const int64_t sa = ta[255], sb = tb[255];
    __syncthreads();
    run_a += sa;
    run_b += sb;
  }
}

// ---- segment starts of a sorted key array (a segment = a run of equal keys)

__device__ __forceinline__ int64_t seg_head(const uint64_t* __restrict__ keys, int64_t i) {
  return (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

// per-chunk number of segment heads (chunks of scan_range)
__global__ void __launch_bounds__(256) k_seg_heads_partial(const uint64_t* __restrict__ keys, const int64_t* n_dev,
                                                           int64_t cap, int64_t* __restrict__ partial) {
  pdl_entry();
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t c = 0;
  for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) c += seg_head(keys, i);
  c = block_sum_i64(c);
  if (threadIdx.x == 0) partial[blockIdx.x] = c;
}

// start[s] = position of the s-th head: each chunk ranks its heads tile by tile from its
// exclusive partial
__global__ void __launch_bounds__(256) k_seg_heads_write(const uint64_t* __restrict__ keys, const int64_t* n_dev,
                                                         int64_t cap, const int64_t* __restrict__ partial, int64_t* n_seg,
                                                         int64_t* __restrict__ start) {
  pdl_entry();
  __shared__ int32_t wsum[8];
  int64_t n = *n_dev;
  if (n > cap) n = cap;
  int64_t beg, end;
  scan_range(n, &beg, &end);
  int64_t all_seg;
  int64_t run = partials_before(partial, blockIdx.x, &all_seg);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (blockIdx.x == 0 && t == 0) *n_seg = all_seg;
  for (int64_t tile = beg; tile < end; tile += 256) {
    const int64_t i = tile + t;
    const bool h = i < end && seg_head(keys, i);
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

struct ZeroArgs {
  uint32_t* p[kZeroRanges];
  int64_t n[kZeroRanges];
  int count;
};

__global__ void __launch_bounds__(kBlock) k_zero_ranges(ZeroArgs z) {
  pdl_entry();
  for (int r = 0; r < z.count; ++r)
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < z.n[r]; i += grid_stride()) z.p[r][i] = 0u;
}

}  // namespace

void zero_ranges(cudaStream_t s, std::initializer_list<ZeroRange> ranges) {
  ZeroArgs z{};
  int64_t most = 0;
  for (const ZeroRange& r : ranges) {
    if (r.ptr == nullptr || r.bytes == 0) continue;
    z.p[z.count] = static_cast<uint32_t*>(r.ptr);
    z.n[z.count] = (int64_t)(r.bytes / 4);
    if (z.n[z.count] > most) most = z.n[z.count];
    if (++z.count == kZeroRanges) {          // more ranges than one launch takes
      launch(k_zero_ranges, blocks_for(most, 4), kBlock, 0, s, z);
      z = ZeroArgs{};
      most = 0;
    }
  }
  if (z.count > 0) launch(k_zero_ranges, blocks_for(most, 4), kBlock, 0, s, z);
}

int radix_sort_u64(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt,
                   const int64_t* n, int64_t cap, int bits, uint32_t* hist, cudaStream_t s, int start_bit) {
  int which = 0, pass = 0;
  for (int shift = start_bit; shift < start_bit + bits; shift += 8) {
    uint64_t* ki = which ? keys_alt : keys;
    uint32_t* vi = which ? vals_alt : vals;
    uint64_t* ko = which ? keys : keys_alt;
    uint32_t* vo = which ? vals : vals_alt;
    // counters of this pass, of the next, and those that this pass clears for the one after it
    uint32_t* h[3];
    for (int k = 0; k < 3; ++k) h[k] = hist + (size_t)((pass + k) % 3) * (256u * kSortBlocks);
    if (pass == 0) launch(k_hist, kSortBlocks, kSortThreads, 0, s, ki, n, cap, shift, h[0], h[1]);
    launch(k_scatter, kSortBlocks, kSortThreads, 0, s, ki, vi, ko, vo, n, cap, shift, h[0], h[1], h[2],
           shift + 8 < start_bit + bits);
    which ^= 1;
    ++pass;
  }
  return which;
}

void exclusive_scan_i64(const int64_t* in, int64_t* out, const int64_t* n, int64_t cap, int64_t* total,
                        int64_t* partial, cudaStream_t s) {
  launch(k_scan_partial, kScanBlocks, 256, 0, s, in, n, cap, partial);
  launch(k_scan_apply, kScanBlocks, 256, 0, s, in, out, n, cap, partial, total);
}

void exclusive_scan2_i64(const int64_t* in_a, int64_t* out_a, int64_t* total_a, const int64_t* in_b, int64_t* out_b,
                         int64_t* total_b, const int64_t* n, int64_t cap, int64_t* partial, cudaStream_t s) {
  launch(k_scan2_partial, kScanBlocks, 256, 0, s, in_a, in_b, n, cap, partial);
  launch(k_scan2_apply, kScanBlocks, 256, 0, s, in_a, out_a, in_b, out_b, n, cap, static_cast<const int64_t*>(partial), total_a,
         total_b);
}

void segment_starts(const uint64_t* keys, const int64_t* n, int64_t cap, int64_t* start, int64_t* n_seg,
                    int64_t* partial, cudaStream_t s) {
  launch(k_seg_heads_partial, kScanBlocks, 256, 0, s, keys, n, cap, partial);
  launch(k_seg_heads_write, kScanBlocks, 256, 0, s, keys, n, cap, static_cast<const int64_t*>(partial), n_seg, start);
}

}  // namespace eipc
