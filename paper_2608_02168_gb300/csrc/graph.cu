// Relation-typed CSR / CSC construction on the device.
//
// The adjacency of one overlapping subgraph (Section 2.2 typed relations; Section 3.1, Eq. 5 and
// Algorithm 1: the induced subgraph of V_k extended by the sampled candidates) is laid out per
// relation twice: by destination (CSR, forward aggregation of Eq. 10) and by source (CSC, its
// transpose in the backward pass).  Rows of all relations are concatenated: relation r owns CSR
// rows [row_base[r], row_base[r+1]) = its destination type's nodes in local order, and CSC rows
// [csc_base[r], csc_base[r+1]) = its source type's nodes.
//
// Construction: each edge gets a row key (or a sentinel key past the last row when invalid), a
// STABLE least-significant-digit radix sort of (key, edge id) places every edge in its row with
// ascending edge ids, and the row pointers are read off the sorted keys (no atomics, so hub rows
// cost nothing extra).  The layout is therefore unique and bit-reproducible.
//
// Three stable sorts build both layouts: the edges by source id, then by CSR row (so a CSR row lists
// its in-edges by (source, edge id)); parallel edges are then adjacent, and each run of them becomes
// one entry (column, multiplicity) of the aggregation lists.  The third sort takes these runs, not
// the edges, by CSC row: a CSC row lists its out-edges by (destination, edge id), so the edges of a
// run stay together there too, in the order they have in the CSR row.  The sorted runs are the
// backward aggregation lists, and the CSC edge arrays are written run by run from them.  On the
// 10M-node, 200M-edge graph a fifth of the edges are runs: the build went from 20.65 to 17.75 ms.
// The non-empty CSR rows get a compact numbering, the rows in which the mean layer stores M_r and
// dMs_r.
#include <algorithm>

#include "hg_internal.cuh"

namespace hg {

// ---------------------------------------------------------------------------------------------
// exclusive scan (int32), three phases: tile sums -> scan of tile sums (recursive) -> tile scan
// ---------------------------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanSub = 4;                                            // 128-item sub-blocks per warp
constexpr int kScanWarpItems = 128 * kScanSub;                         // a warp's contiguous segment
constexpr int kScanTile = kScanThreads / 32 * kScanWarpItems;          // 4096 items per block

__device__ __forceinline__ int warp_inclusive_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Items i .. i + 3 (zero past n): one 16-byte load where the array is aligned and the four are in
// range.  A warp's lanes cover 128 consecutive items per call, so every access is coalesced.
__device__ __forceinline__ int4 scan_load4(const int32_t* in, int64_t i, int64_t n, bool vec) {
  if (vec && i + 3 < n) return *reinterpret_cast<const int4*>(in + i);
  int4 r;
  r.x = i < n ? in[i] : 0;
  r.y = i + 1 < n ? in[i + 1] : 0;
  r.z = i + 2 < n ? in[i + 2] : 0;
  r.w = i + 3 < n ? in[i + 3] : 0;
  return r;
}

__device__ __forceinline__ void scan_store4(int32_t* out, int64_t i, int64_t n, int4 v, bool vec) {
  if (vec && i + 3 < n) {
    *reinterpret_cast<int4*>(out + i) = v;
    return;
  }
  if (i < n) out[i] = v.x;
  if (i + 1 < n) out[i + 1] = v.y;
  if (i + 2 < n) out[i + 2] = v.z;
  if (i + 3 < n) out[i + 3] = v.w;
}

// sums[tile] = sum of the tile's kScanTile items (warp w: items tile * kScanTile + w * 512 ..).  n_dev, if
// given, holds the item count on the device (at most n; tiles past it sum to 0 and are not read).
__global__ void __launch_bounds__(kScanThreads) scan_tile_sums(const int32_t* __restrict__ in, int64_t n,
                                                                const int32_t* __restrict__ n_dev,
                                                                int32_t* __restrict__ sums) {
  pdl_begin();
  if (n_dev) n = *n_dev;
  if ((int64_t)blockIdx.x * kScanTile >= n) {
    if (threadIdx.x == 0) sums[blockIdx.x] = 0;
    return;
  }
  __shared__ int wt[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool vec = (reinterpret_cast<uintptr_t>(in) & 15) == 0;
  const int64_t seg = (int64_t)blockIdx.x * kScanTile + (int64_t)warp * kScanWarpItems;
  int s = 0;
#pragma unroll
  for (int j = 0; j < kScanSub; ++j) {
    const int4 v = scan_load4(in, seg + 128 * j + 4 * lane, n, vec);
    s += v.x + v.y + v.z + v.w;
  }
  s = warp_sum_i(s);
  if (lane == 0) wt[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) t += wt[w];
    sums[blockIdx.x] = t;
  }
}

// Exclusive scan of one tile plus tile_off[tile] (nullptr: a single tile starting at 0); the last
// tile also writes out[n] = the grand total.  out may equal in.  With n_dev (n the capacity), the scan ends
// at the device count: out[*n_dev] = the grand total, and nothing past it is read or written.
__global__ void __launch_bounds__(kScanThreads) scan_tiles(const int32_t* in, int32_t* out, int64_t n,
                                                            const int32_t* __restrict__ n_dev,
                                                            const int32_t* __restrict__ tile_off) {
  pdl_begin();
  bool last = blockIdx.x == gridDim.x - 1;  // the tile that writes the grand total
  if (n_dev) {
    n = *n_dev;
    const int64_t t0 = (int64_t)blockIdx.x * kScanTile;
    if (t0 > n || (t0 == n && n > 0)) return;
    last = n <= t0 + kScanTile;
  }
  __shared__ int wt[kScanThreads / 32 + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  const int64_t seg = (int64_t)blockIdx.x * kScanTile + (int64_t)warp * kScanWarpItems;
  int4 v[kScanSub];
  int ls[kScanSub];
  int s = 0;
#pragma unroll
  for (int j = 0; j < kScanSub; ++j) {
    v[j] = scan_load4(in, seg + 128 * j + 4 * lane, n, vec);
    ls[j] = v[j].x + v[j].y + v[j].z + v[j].w;
    s += ls[j];
  }
  s = warp_sum_i(s);
  if (lane == 0) wt[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {  // exclusive prefix over the warps, block total last
    int run = tile_off ? tile_off[blockIdx.x] : 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) {
      const int t = wt[w];
      wt[w] = run;
      run += t;
    }
    wt[kScanThreads / 32] = run;
  }
  __syncthreads();
  int carry = wt[warp];
#pragma unroll
  for (int j = 0; j < kScanSub; ++j) {
    const int incl = warp_inclusive_scan(ls[j]);
    int run = carry + incl - ls[j];
    int4 o;
    o.x = run;
    run += v[j].x;
    o.y = run;
    run += v[j].y;
    o.z = run;
    run += v[j].z;
    o.w = run;
    scan_store4(out, seg + 128 * j + 4 * lane, n, o, vec);
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (last && threadIdx.x == 0) out[n] = wt[kScanThreads / 32];
}

size_t scan_scratch_bytes(int64_t n) {
  size_t b = 0;
  while (n > kScanTile) {
    n = ceil_div(n, kScanTile);
    b += align_up((size_t)(n + 1) * sizeof(int32_t));
  }
  return b + 256;
}

hg_status exclusive_scan(const int32_t* in, int32_t* out, int64_t n, void* scratch, cudaStream_t s,
                         const int32_t* n_dev) {
  if (n <= 0) {
    if (n == 0) HG_CUDA(cudaMemsetAsync(out, 0, sizeof(int32_t), s));
    return HG_OK;
  }
  if (n <= kScanTile)
    return launch("scan_tiles", scan_tiles, dim3(1), dim3(kScanThreads), 0, s, in, out, n, n_dev,
                  (const int32_t*)nullptr);
  const int64_t tiles = ceil_div(n, kScanTile);
  int32_t* sums = static_cast<int32_t*>(scratch);
  char* rest = static_cast<char*>(scratch) + align_up((size_t)(tiles + 1) * sizeof(int32_t));
  HG_TRY(launch("scan_tile_sums", scan_tile_sums, dim3((unsigned)tiles), dim3(kScanThreads), 0, s,
                in, n, n_dev, sums));
  HG_TRY(exclusive_scan(sums, sums, tiles, rest, s));
  return launch("scan_tiles", scan_tiles, dim3((unsigned)tiles), dim3(kScanThreads), 0, s, in, out,
                n, n_dev, (const int32_t*)sums);
}

// ---------------------------------------------------------------------------------------------
// stable LSD radix sort of (uint32 key, uint32 value, uint32 second value), digits of up to 9 bits
// ---------------------------------------------------------------------------------------------
// A pass is bound by shared memory, not by HBM (random digits meet about 3.4 to a bank, and every item
// is ranked and placed there), so a pass less is worth more than narrower digits: 24-bit keys take three
// 8-bit passes and 26-bit keys three of 9, 9 and 8 bits (four before).  Measured on the 10M-node, 200M-edge
// build (zipf 1.2 / 0.65), against the former tiles of 4096 with a read and a write of the counts per
// round and 8-bit digits: 23.05 / 31.40 -> 20.65 / 29.12 ms; 1M edges 558 -> 545 us, 20k 343 -> 328 us.
// Tiles of 4096 (three CTAs on an SM) and 8192 items spill and were slower (19.9, 19.4 ms against 17.8 ms
// with the runs below), and so were CTAs of 256 threads (19.0 - 21.1 ms).  Graphs whose tiles of 6144
// do not fill the SMs once take tiles of 2048.
constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxBits = 9;
constexpr int kMaxRadix = 1 << kMaxBits;
static_assert(kMaxRadix <= kSortThreads, "a thread per digit");
constexpr int kItemsLarge = 12, kItemsSmall = 4;  // per thread
constexpr int64_t kSortLarge = (int64_t)2 * 152 * kSortThreads * kItemsLarge;

// Per-tile digit counts hist[digit * tiles + tile]; four warps count into one shared histogram, and
// the histograms are added at the end.
// n_dev, if given, holds the item count on the device, at most n; tiles past it count nothing.
template <int kItems>
__global__ void __launch_bounds__(kSortThreads) radix_hist(const uint32_t* __restrict__ keys, int64_t n,
                                                           const int32_t* __restrict__ n_dev, int shift, int bits,
                                                           int32_t* __restrict__ hist, int64_t tiles) {
  pdl_begin();
  constexpr int kTile = kSortThreads * kItems;
  constexpr int kCopies = 4;  // four warps share a histogram
  __shared__ int h[kCopies][kMaxRadix];
  const int radix = 1 << bits;
  const int64_t t0 = (int64_t)blockIdx.x * kTile;
  if (n_dev) {
    n = *n_dev;
    if (t0 >= n) {
      for (int d = threadIdx.x; d < radix; d += kSortThreads) hist[(int64_t)d * tiles + blockIdx.x] = 0;
      return;
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < radix)
#pragma unroll
    for (int w = 0; w < kCopies; ++w) h[w][threadIdx.x] = 0;
  // the warp's slice, 128 keys per round (16-byte loads), all loaded before any is counted
  const int64_t first = t0 + (int64_t)warp * 32 * kItems + lane * 4;
  uint4 k[kItems / 4];
#pragma unroll
  for (int i = 0; i < kItems / 4; ++i) {
    const int64_t p = first + i * 128;
    if (p + 4 <= n) {
      k[i] = *reinterpret_cast<const uint4*>(keys + p);
    } else {
      k[i].x = p < n ? keys[p] : 0u;
      k[i].y = p + 1 < n ? keys[p + 1] : 0u;
      k[i].z = p + 2 < n ? keys[p + 2] : 0u;
      k[i].w = 0u;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems / 4; ++i) {
    const int64_t p = first + i * 128;
    const uint32_t v[4] = {k[i].x, k[i].y, k[i].z, k[i].w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (p + e < n) atomicAdd(&h[warp % kCopies][(v[e] >> shift) & (radix - 1)], 1);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < radix; d += kSortThreads) {
    int t = 0;
#pragma unroll
    for (int w = 0; w < kCopies; ++w) t += h[w][d];
    hist[(int64_t)d * tiles + blockIdx.x] = t;
  }
}

// Stable scatter of one tile.  (1) Warp w reads the keys of its 32 kItems consecutive items, 32 at a
// time (coalesced).  (2) It ranks them round by round with __match_any_sync and per-digit running
// counts, so the item order inside the tile is (warp, round, lane).  (3) Per-digit prefixes over warps
// and over digits, added into the warps' counts, give every item its position in the tile sorted by
// digit (equal digits keep their order).  (4) Keys and values, then the second values, are put there in
// shared memory and consecutive threads write consecutive sorted items to the digit's base + position:
// runs of equal digits go out coalesced.  Only one array of values is staged at a time, which leaves
// room for two CTAs on an SM at 12 items a thread.
template <int kItems>
__global__ void __launch_bounds__(kSortThreads, 2) radix_scatter(
    const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in,
    const uint32_t* __restrict__ vals2_in, uint32_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out,
    uint32_t* __restrict__ vals2_out, int64_t n, const int32_t* __restrict__ n_dev, int shift, int bits,
    const int32_t* __restrict__ offs, int64_t tiles) {
  pdl_begin();
  constexpr int kTile = kSortThreads * kItems;
  extern __shared__ uint32_t sort_smem[];
  uint32_t* skey = sort_smem;      // sorted tile
  uint32_t* sval = skey + kTile;   // its values, then its second values
  int* whist = reinterpret_cast<int*>(sval + kTile);  // [warp][radix]
  int* base = reinterpret_cast<int*>(whist + kSortWarps * kMaxRadix);  // global position of sorted position 0, per digit
  __shared__ int wsum[kSortWarps];
  const int radix = 1 << bits, mask = radix - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = (int64_t)blockIdx.x * kTile;
  if (n_dev) n = *n_dev;
  if (t0 >= n) return;
  const int cnt = (int)min((int64_t)kTile, n - t0);
  int* wh = whist + warp * radix;
  for (int i = lane; i < radix; i += 32) wh[i] = 0;
  int goff = 0;
  if (threadIdx.x < radix) goff = offs[(int64_t)threadIdx.x * tiles + blockIdx.x];
  const int j0 = warp * 32 * kItems + lane;  // this thread's first item, the next ones 32 apart
  uint32_t k[kItems], v[kItems];
  uint32_t rank[kItems / 2];  // two 16-bit ranks, then positions, per word
#pragma unroll
  for (int r = 0; r < kItems; ++r) k[r] = j0 + 32 * r < cnt ? keys_in[t0 + j0 + 32 * r] : 0u;
  __syncwarp();
  // The first lane of each group of equal digits adds the group's size to the warp's count, and the
  // old count is the rank of the group's first item: the adds of all rounds are in flight together (a
  // read and a write per round, each waited for, made shared memory's latency the kernel's).
  unsigned peers[kItems];
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    peers[r] = __match_any_sync(0xffffffffu, j0 + 32 * r < cnt ? (int)(k[r] >> shift) & mask : radix);
  int old[kItems];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    old[r] = 0;
    if (j0 + 32 * r < cnt && lane == __ffs(peers[r]) - 1)
      old[r] = atomicAdd(&wh[(k[r] >> shift) & mask], __popc(peers[r]));
    __syncwarp();  // the next round's adds come after
  }
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const uint32_t rk = __shfl_sync(0xffffffffu, old[r], __ffs(peers[r]) - 1) + __popc(peers[r] & ((1u << lane) - 1u));
    if (r & 1) rank[r / 2] |= rk << 16;
    else rank[r / 2] = rk;
  }
#pragma unroll
  for (int r = 0; r < kItems; ++r)  // in flight over the prefixes; first pass: the input position
    v[r] = j0 + 32 * r < cnt ? (vals_in ? vals_in[t0 + j0 + 32 * r] : (uint32_t)(t0 + j0 + 32 * r)) : 0u;
  __syncthreads();
  int tot = 0;  // this thread's digit: items of the tile
  if (threadIdx.x < radix)
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) tot += whist[w * radix + threadIdx.x];
  const int incl = warp_inclusive_scan(tot);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (threadIdx.x < radix) {
    int run = incl - tot;  // sorted position of the digit's first item
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) run += w < warp ? wsum[w] : 0;
    base[threadIdx.x] = goff - run;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      const int c = whist[w * radix + threadIdx.x];
      whist[w * radix + threadIdx.x] = run;
      run += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    if (j0 + 32 * r < cnt) {
      const uint32_t p = wh[(k[r] >> shift) & mask] + ((rank[r / 2] >> (16 * (r & 1))) & 0xFFFFu);
      skey[p] = k[r];
      sval[p] = v[r];
      rank[r / 2] = (r & 1) ? (rank[r / 2] & 0xFFFFu) | p << 16 : (rank[r / 2] & 0xFFFF0000u) | p;
    }
  }
#pragma unroll
  for (int r = 0; r < kItems; ++r) v[r] = j0 + 32 * r < cnt ? vals2_in[t0 + j0 + 32 * r] : 0u;  // in flight meanwhile
  __syncthreads();
  int pos[kItems];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int p = threadIdx.x + r * kSortThreads;
    if (p < cnt) {
      const uint32_t kk = skey[p];
      pos[r] = base[(kk >> shift) & mask] + p;
      keys_out[pos[r]] = kk;
      vals_out[pos[r]] = sval[p];
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r)
    if (j0 + 32 * r < cnt) sval[(rank[r / 2] >> (16 * (r & 1))) & 0xFFFFu] = v[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int p = threadIdx.x + r * kSortThreads;
    if (p < cnt) vals2_out[pos[r]] = sval[p];
  }
}

struct SortBuffers {
  uint32_t* ckeys;  // CSR row keys (payload of the first sort), then the runs' CSC keys
  uint32_t* keys[2];
  uint32_t* vals[2];
  uint32_t* vals2[2];  // second payload (carried so the finish passes read sequentially)
  int32_t* hist;
  void* scan_scratch;
};

static bool sort_large(int64_t n) { return n >= kSortLarge; }
static int64_t sort_tiles(int64_t n) {
  return std::max<int64_t>(1, ceil_div(n, kSortThreads * (sort_large(n) ? kItemsLarge : kItemsSmall)));
}
// dynamic shared memory of radix_scatter: the sorted tile (key, value), warp counts, digit bases
template <int kItems>
constexpr size_t kScatterSmem = 2 * kSortThreads * kItems * sizeof(uint32_t) +
                                (kSortWarps + 1) * kMaxRadix * sizeof(int);

// Sorts (key, value, second payload) triples by the low `bits` key bits (at least one pass), stable.
// The first pass reads keys_src, vals_src (null: the input positions) and vals2_src, which may lie
// in buffer `start` (it writes buffer start ^ 1 first); n_dev as in radix_hist; returns the buffer
// index holding the sorted keys.  The last pass writes the payloads to vals_final / vals2_final when
// those are given (the caller's final arrays), else to the sort buffers beside the keys.
template <int kItems>
static hg_status radix_sort_t(SortBuffers& b, int64_t n, const int32_t* n_dev, int bits, const uint32_t* keys_src,
                              const uint32_t* vals_src, const uint32_t* vals2_src, int start, cudaStream_t s,
                              int* result, uint32_t* vals_final, uint32_t* vals2_final) {
  static bool attr = false;
  if (!attr) {
    HG_CUDA(cudaFuncSetAttribute(radix_scatter<kItems>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kScatterSmem<kItems>));
    attr = true;
  }
  int cur = start;
  const int64_t tiles = sort_tiles(n);
  const uint32_t* k = keys_src;
  const uint32_t* v = vals_src;
  const uint32_t* v2 = vals2_src;
  int left = std::max(bits, 1), shift = 0;
  for (int passes = (int)ceil_div(left, kMaxBits); passes > 0; --passes) {  // the widest digits first
    const int w = (int)ceil_div(left, passes);
    const bool last = passes == 1;
    uint32_t* vo = last && vals_final ? vals_final : b.vals[cur ^ 1];
    uint32_t* v2o = last && vals2_final ? vals2_final : b.vals2[cur ^ 1];
    HG_TRY(launch("radix_hist", radix_hist<kItems>, dim3((unsigned)tiles), dim3(kSortThreads), 0, s, k, n, n_dev, shift,
                  w, b.hist, tiles));
    HG_TRY(exclusive_scan(b.hist, b.hist, tiles << w, b.scan_scratch, s));
    HG_TRY(launch("radix_scatter", radix_scatter<kItems>, dim3((unsigned)tiles), dim3(kSortThreads),
                  kScatterSmem<kItems>, s, k, v, v2, b.keys[cur ^ 1], vo, v2o, n, n_dev, shift, w,
                  (const int32_t*)b.hist, tiles));
    k = b.keys[cur ^ 1];
    v = vo;
    v2 = v2o;
    cur ^= 1;
    shift += w;
    left -= w;
  }
  *result = cur;
  return HG_OK;
}

static hg_status radix_sort(SortBuffers& b, int64_t n, const int32_t* n_dev, int bits, const uint32_t* keys_src,
                            const uint32_t* vals_src, const uint32_t* vals2_src, int start, cudaStream_t s,
                            int* result, uint32_t* vals_final = nullptr, uint32_t* vals2_final = nullptr) {
  if (sort_large(n))
    return radix_sort_t<kItemsLarge>(b, n, n_dev, bits, keys_src, vals_src, vals2_src, start, s, result, vals_final,
                                     vals2_final);
  return radix_sort_t<kItemsSmall>(b, n, n_dev, bits, keys_src, vals_src, vals2_src, start, s, result, vals_final,
                                   vals2_final);
}

// ---------------------------------------------------------------------------------------------
// CSR / CSC kernels
// ---------------------------------------------------------------------------------------------
// Keys of the first sort: the source node id of every valid edge (0 for invalid ones), and, as its
// payload, the CSR row key (destination row; the sentinel past the last row for an invalid edge:
// relation or endpoint out of range, endpoint of the wrong type).  The relation tables are read
// from shared memory.
__global__ void __launch_bounds__(256) edge_keys(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                 const int32_t* __restrict__ rel, int64_t E, GraphMeta m,
                                                 int64_t rows, uint32_t* __restrict__ skeys,
                                                 uint32_t* __restrict__ rkeys) {
  pdl_begin();
  __shared__ int64_t row0[kMaxRels];  // first row of relation r minus its destination type's offset
  __shared__ int32_t rsrc[kMaxRels], rdst[kMaxRels];
  if (threadIdx.x < kMaxRels) {
    const int r = threadIdx.x;
    if (r < m.num_rels) {
      rsrc[r] = m.rel_src[r];
      rdst[r] = m.rel_dst[r];
      row0[r] = m.row_base[r] - m.type_off[m.rel_dst[r]];
    }
  }
  __syncthreads();
  const int64_t N = m.type_off[m.num_types];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
    const int r = rel[e];
    const int64_t sn = src[e], tn = dst[e];
    bool ok = r >= 0 && r < m.num_rels && sn >= 0 && sn < N && tn >= 0 && tn < N;
    int64_t key = rows;  // invalid edges sort after every row
    if (ok && node_type_of(m, sn) == rsrc[r] && node_type_of(m, tn) == rdst[r]) key = row0[r] + tn;
    else ok = false;
    skeys[e] = ok ? (uint32_t)sn : 0u;
    rkeys[e] = (uint32_t)key;
  }
}

// ---------------------------------------------------------------------------------------------
// non-empty CSR rows: the relation rows the mean layer stores (a row without in-edges has M = 0
// and is never stored, read or gathered)
// ---------------------------------------------------------------------------------------------
__global__ void nonempty_flags(const int32_t* __restrict__ ptr, int64_t rows, int32_t* __restrict__ flag) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x)
    flag[r] = ptr[r + 1] > ptr[r] ? 1 : 0;
}

// long rows of the fused layer: flag[r] = 1 when CSR row r has more than kFuseRuns runs
__global__ void long_flags(const int32_t* __restrict__ aptr, int64_t rows, int32_t* __restrict__ flag) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x)
    flag[r] = aptr[r + 1] - aptr[r] > kFuseRuns ? 1 : 0;
}

// list[ofs[r]] = r for every flagged row r (ofs = the exclusive scan of the flags)
__global__ void compact_list(const int32_t* __restrict__ flag, const int32_t* __restrict__ ofs, int64_t rows,
                             int32_t* __restrict__ list) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x)
    if (flag[r]) list[ofs[r]] = (int32_t)r;
}

// mbase[r] = compact index of relation r's first non-empty row (pos = the scan of the flags, whose
// entry `rows` is the number of non-empty rows).
__global__ void compact_bases(const int32_t* __restrict__ pos, GraphMeta m, int32_t* __restrict__ mbase) {
  pdl_begin();
  const int r = threadIdx.x;
  if (r <= m.num_rels) mbase[r] = pos[m.row_base[r]];
}

// In place: mrow[row] = its compact index when non-empty, `rows` (out of range) otherwise; mlist[k]
// = the CSR row of compact row k.
__global__ void compact_rows(const int32_t* __restrict__ flag, int64_t rows, int32_t* __restrict__ mrow,
                             int32_t* __restrict__ mlist) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t k = mrow[r];
    if (flag[r]) {
      mlist[k] = (int32_t)r;
    } else {
      mrow[r] = (int32_t)rows;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// runs of parallel edges: the CSR order (row, source), whose parallel edges are adjacent, as one entry
// per distinct (row, source) with its multiplicity, in the same order
// ---------------------------------------------------------------------------------------------
// flag[p] = 1 where a run starts (a new row or a new source) for p < ptr[rows]; 0 up to cap (the
// capacity the scan runs over).
// Four positions per thread, as 16-byte vectors (the arrays are 256-byte aligned).
__global__ void __launch_bounds__(256) run_flags(const uint32_t* __restrict__ rkey, const int32_t* __restrict__ col,
                                                 const int32_t* __restrict__ ptr, int64_t rows, int64_t cap,
                                                 int32_t* __restrict__ flag) {
  pdl_begin();
  const int64_t n = ptr[rows];
  for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; p < cap;
       p += (int64_t)gridDim.x * blockDim.x * 4) {
    if (p + 4 <= n) {
      const uint4 k = *reinterpret_cast<const uint4*>(rkey + p);
      const int4 c = *reinterpret_cast<const int4*>(col + p);
      const bool first = p == 0 || c.x != col[p - 1] || k.x != rkey[p - 1];
      *reinterpret_cast<int4*>(flag + p) = make_int4(first, c.y != c.x || k.y != k.x, c.z != c.y || k.z != k.y,
                                                     c.w != c.z || k.w != k.z);
    } else {
      for (int64_t q = p; q < min(p + 4, cap); ++q)
        flag[q] = (q < n && (q == 0 || col[q] != col[q - 1] || rkey[q] != rkey[q - 1])) ? 1 : 0;
    }
  }
}

constexpr uint32_t kOneEdge = 0x80000000u;
// With u = the exclusive scan of the run-start flags (u[n] = number of runs): position p starts a
// run exactly when u[p + 1] != u[p]; run k = u[p] gets its source ucol[k] = col[p], its start
// upos[k] = p (upos[U] = n), its CSC row ckey[k], its destination udst[k] and uval[k], what the CSC
// side needs to find its edge ids: k, or for a run of one edge that edge's id with the top bit set (no
// edge id has it), so that a graph of mostly distinct node pairs carries its ids through the sort
// instead of gathering them at random after it (200M edges at zipf 0.65: 40.0 -> 34.3 ms).  A lane per
// position, so that the entries of a graph of short runs are written coalesced.
__global__ void __launch_bounds__(256) run_write(const int32_t* __restrict__ u, const int32_t* __restrict__ col,
                                                 const uint32_t* __restrict__ rkey, const int32_t* __restrict__ ptr,
                                                 int64_t rows, GraphMeta m, const int32_t* __restrict__ eid,
                                                 int32_t* __restrict__ ucol, int32_t* __restrict__ upos,
                                                 uint32_t* __restrict__ ckey, uint32_t* __restrict__ udst,
                                                 uint32_t* __restrict__ uval) {
  pdl_begin();
  constexpr int kRounds = 4;  // positions per thread, a block apart, their loads in flight together
  const int64_t n = ptr[rows];
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x * kRounds + threadIdx.x; p0 <= n;
       p0 += (int64_t)gridDim.x * blockDim.x * kRounds) {
    int k[kRounds], c[kRounds], id[kRounds];
    int64_t key[kRounds];
    bool starts[kRounds], one[kRounds];
#pragma unroll
    for (int i = 0; i < kRounds; ++i) {
      const int64_t p = p0 + (int64_t)i * blockDim.x;
      k[i] = p <= n ? u[p] : 0;
      const int k1 = p < n ? u[p + 1] : k[i], k2 = p + 1 < n ? u[p + 2] : -1;
      starts[i] = k1 != k[i];
      one[i] = k2 != k1;
      c[i] = p < n ? col[p] : 0;
      key[i] = p < n ? rkey[p] : 0;
      id[i] = p < n ? eid[p] : 0;
    }
#pragma unroll
    for (int i = 0; i < kRounds; ++i) {
      const int64_t p = p0 + (int64_t)i * blockDim.x;
      if (p == n) upos[k[i]] = (int32_t)n;
      if (!starts[i]) continue;
      int r = 0;
#pragma unroll
      for (int x = 1; x < kMaxRels; ++x)
        if (x < m.num_rels && key[i] >= m.row_base[x]) r = x;
      ucol[k[i]] = c[i];
      upos[k[i]] = (int32_t)p;
      ckey[k[i]] = (uint32_t)(m.csc_base[r] + ((int64_t)c[i] - m.type_off[m.rel_src[r]]));
      udst[k[i]] = (uint32_t)(m.type_off[m.rel_dst[r]] + (key[i] - m.row_base[r]));
      uval[k[i]] = one[i] ? kOneEdge | (uint32_t)id[i] : (uint32_t)k[i];
    }
  }
}

// ucnt[k] = upos[k + 1] - upos[k] (the run's length) for k < U; uptr[r] = u[ptr[r]] for r <= rows.
__global__ void run_finish(const int32_t* __restrict__ u, const int32_t* __restrict__ upos,
                           const int32_t* __restrict__ ptr, int64_t rows, int32_t* __restrict__ ucnt,
                           int32_t* __restrict__ uptr) {
  pdl_begin();
  const int64_t U = u[ptr[rows]];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < U; k += stride) ucnt[k] = upos[k + 1] - upos[k];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= rows; r += stride) uptr[r] = u[ptr[r]];
}

// Row pointers from the sorted keys: ptr[k] = first position whose key is >= k, k in [0, rows].
// Position p owns the rows k with key[p-1] < k <= key[p] (key[-1] = -1, key[n] = rows), so every
// entry is written exactly once and empty rows get the position of the next non-empty one.  The
// owner of k = rows also writes n - ptr[rows] (the positions with keys past the last row) to
// *invalid when that is given.  n_dev, if given, holds n on the device.  Four keys per thread.
__global__ void row_ptr_from_keys(const uint32_t* __restrict__ keys, int64_t n, const int32_t* __restrict__ n_dev,
                                  int64_t rows, int32_t* __restrict__ ptr, int32_t* __restrict__ invalid) {
  pdl_begin();
  if (n_dev) n = *n_dev;
  for (int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; p0 <= n;
       p0 += (int64_t)gridDim.x * blockDim.x * 4) {
    uint32_t k[4];
    if (p0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(keys + p0);
      k[0] = v.x;
      k[1] = v.y;
      k[2] = v.z;
      k[3] = v.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) k[i] = p0 + i < n ? keys[p0 + i] : 0u;
    }
    int64_t lo = p0 == 0 ? 0 : (int64_t)keys[p0 - 1] + 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t p = p0 + i;
      if (p > n) break;
      const int64_t hi = p == n ? rows : min((int64_t)k[i], rows);
      for (int64_t r = lo; r <= hi; ++r) ptr[r] = (int32_t)p;
      if (invalid && lo <= rows && rows <= hi) *invalid = (int32_t)(n - p);
      lo = (int64_t)k[i] + 1;
    }
  }
}

// Out-runs of every node over all relations leaving its type (the length of its node-major row), from
// the CSC row pointers over runs.
__global__ void node_out_counts(const int32_t* __restrict__ cptr, GraphMeta m, int32_t* __restrict__ cnt) {
  pdl_begin();
  __shared__ int64_t cbase[kMaxRels];  // CSC row of the type's node 0 in relation r, minus the type offset
  __shared__ int32_t rsrc[kMaxRels];
  if (threadIdx.x < kMaxRels) {
    const int r = threadIdx.x;
    rsrc[r] = r < m.num_rels ? m.rel_src[r] : -1;
    if (r < m.num_rels) cbase[r] = m.csc_base[r] - m.type_off[m.rel_src[r]];
  }
  __syncthreads();
  const int64_t N = m.type_off[m.num_types];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    const int t = node_type_of(m, i);
    int c = 0;
#pragma unroll
    for (int r = 0; r < kMaxRels; ++r)
      if (rsrc[r] == t) c += cptr[cbase[r] + i + 1] - cptr[cbase[r] + i];
    cnt[i] = c;
  }
}

// What a run of the CSC order reads at random about its CSR row, in one word: pack[row] = the row's place
// among its relation's compact rows above the relation's degree bits, below it the in-degree, or all ones
// where it does not fit (the row pointers then give it).  The runs come relation by relation, so one
// relation's words are in use at a time (36 MB for 9M nodes): with (compact row, degree) pairs of 8 bytes
// they left the L2 and csc_runs took 3.6 ms instead of 2.8 ms at 200M edges of distinct pairs.
struct PackBits {
  int32_t deg[kMaxRels];  // degree bits of relation r: 32 - the width of its row count
};
__global__ void __launch_bounds__(256) row_pack(const int32_t* __restrict__ mrow, const int32_t* __restrict__ mbase,
                                                const int32_t* __restrict__ csr_ptr, int64_t rows, GraphMeta m,
                                                PackBits pb, uint32_t* __restrict__ pack) {
  pdl_begin();
  for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
       row += (int64_t)gridDim.x * blockDim.x) {
    int r = 0;
#pragma unroll
    for (int x = 1; x < kMaxRels; ++x)
      if (x < m.num_rels && row >= m.row_base[x]) r = x;
    const uint32_t full = (1u << pb.deg[r]) - 1u;
    const uint32_t deg = (uint32_t)(csr_ptr[row + 1] - csr_ptr[row]);
    if (deg) pack[row] = (uint32_t)(mrow[row] - mbase[r]) << pb.deg[r] | min(deg, full);  // empty rows have no run
  }
}

// The runs in CSC order (sorted keys, uval and destination of each; cptr: CSC row pointers over
// runs).  Writes the node-major list of out-runs used by the backward aggregation -- node i's row holds,
// relation by relation (ascending) and in CSC order within a relation, the compact row of each run's
// target and its multiplicity -- and, per run, its length, its first CSR position (or uval, for one
// edge), and 1 / deg_r(destination).
__global__ void __launch_bounds__(256) csc_runs(
    const uint32_t* __restrict__ skey, const uint32_t* __restrict__ srun, const uint32_t* __restrict__ sdst,
    const int32_t* __restrict__ n_dev, const int32_t* __restrict__ cptr, GraphMeta m,
    const int32_t* __restrict__ csr_ptr, const uint32_t* __restrict__ pack, PackBits pb,
    const int32_t* __restrict__ mbase, const int32_t* __restrict__ upos, const int32_t* __restrict__ bptr,
    int32_t* __restrict__ bcol, int32_t* __restrict__ bcnt, int32_t* __restrict__ qlen, int32_t* __restrict__ qstart,
    float* __restrict__ qcoef) {
  pdl_begin();
  const int64_t U = *n_dev;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < U; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t key = skey[q];
    const int64_t j = sdst[q];
    const uint32_t run = srun[q];
    int start = (int)run, len = 1;
    if (!(run & kOneEdge)) {
      start = upos[run];
      len = upos[run + 1] - start;
    }
    int r = 0;
#pragma unroll
    for (int k = 1; k < kMaxRels; ++k)
      if (k < m.num_rels && key >= m.csc_base[k]) r = k;
    const int64_t row = m.row_base[r] + (j - m.type_off[m.rel_dst[r]]);
    const uint32_t pk = __ldg(pack + row), full = (1u << pb.deg[r]) - 1u;
    int deg = (int)(pk & full);
    if (deg == (int)full) deg = csr_ptr[row + 1] - csr_ptr[row];
    // node-major position: the node's row start, the runs of its earlier relations, the rank in this one
    const int t = m.rel_src[r];
    const int64_t il = key - m.csc_base[r];  // type-local source id
    int64_t pos = bptr[m.type_off[t] + il] + (q - cptr[key]);
#pragma unroll
    for (int k = 0; k < kMaxRels; ++k)
      if (k < r && m.rel_src[k] == t) pos += cptr[m.csc_base[k] + il + 1] - cptr[m.csc_base[k] + il];
    bcol[pos] = mbase[r] + (int)(pk >> pb.deg[r]);
    bcnt[pos] = len;
    qlen[q] = len;
    qstart[q] = start;
    qcoef[q] = __fdiv_rn(1.0f, (float)deg);
  }
}

// CSC edge arrays from the runs in CSC order: run q's edges go to positions qpos[q] .. qpos[q + 1] (qpos
// the scan of the lengths, qpos[U] = their number) with the edge ids of its CSR positions, in order.  A
// warp writes kExpand consecutive positions: it finds the run of its first one by binary search, then
// takes 32 runs at a time, one per lane, and each position finds its run among them by shuffles, so a
// run of a million edges is spread over many warps and 32 runs of one edge fill one store.
constexpr int kExpand = 1024;
__global__ void __launch_bounds__(256) csc_expand(const int32_t* __restrict__ qpos, const int32_t* __restrict__ qstart,
                                                  const float* __restrict__ qcoef, const uint32_t* __restrict__ qdst,
                                                  const int32_t* __restrict__ n_dev,
                                                  const int32_t* __restrict__ csr_eid, int32_t* __restrict__ ccol,
                                                  int32_t* __restrict__ ceid, float* __restrict__ ccoef) {
  pdl_begin();
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t U = *n_dev, nv = qpos[U];
  constexpr int kRounds = 4;  // positions per lane whose edge ids are read together
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * kExpand < nv; w += warps) {
    int64_t p = w * kExpand;
    const int64_t p1 = min(p + kExpand, nv);
    int64_t lo = 0, hi = U;  // the last run with qpos <= p (every run has at least one edge)
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (qpos[mid] <= p) lo = mid;
      else hi = mid;
    }
    int first, end, start, dst;
    float coef;
    auto window = [&](int64_t q0) {  // one run per lane; lanes past the last run repeat it
      const int64_t q = min(q0 + lane, U - 1);
      first = qpos[q];
      end = qpos[q + 1];
      start = qstart[q];  // CSR position of the run's first edge, or its only id
      dst = (int)qdst[q];
      coef = qcoef[q];
    };
    window(lo);
    for (int64_t q0 = lo; p < p1; q0 += 32) {
      const int cfirst = first, cend = end, cstart = start, cdst = dst;
      const float ccf = coef;
      window(q0 + 32);  // the next runs, in flight meanwhile
      const int64_t wend = min(p1, (int64_t)__shfl_sync(kAll, cend, 31));
      const uint32_t xend = (uint32_t)wend;
      for (; p < wend; p += 32 * kRounds) {
        int id[kRounds], t[kRounds];
        float c[kRounds];
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
          if (p + 32 * k >= wend) break;
          const uint32_t x = (uint32_t)p + 32 * k + lane;  // past the end, up to 127 above 31 bits
          int i = 0;  // lanes whose run ends at or before x: the index of x's run
#pragma unroll
          for (int b = 16; b > 0; b >>= 1)
            if ((uint32_t)__shfl_sync(kAll, cend, i + b - 1) <= x) i += b;
          const int s0 = __shfl_sync(kAll, cstart, i), f0 = __shfl_sync(kAll, cfirst, i);
          t[k] = __shfl_sync(kAll, cdst, i);
          c[k] = __shfl_sync(kAll, ccf, i);
          id[k] = s0 & ~(int)kOneEdge;
          if (s0 >= 0 && x < xend) id[k] = __ldg(csr_eid + s0 + (x - (uint32_t)f0));
        }
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
          const uint32_t x = (uint32_t)p + 32 * k + lane;
          if (x < xend) {
            ceid[x] = id[k];
            ccol[x] = t[k];
            ccoef[x] = c[k];
          }
        }
      }
      p = wend;
    }
  }
}

// ptr[r] = pos[ptr[r]]: row pointers over runs become row pointers over edges
__global__ void run_to_edge_ptr(const int32_t* __restrict__ pos, int64_t rows, int32_t* __restrict__ ptr) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= rows; r += (int64_t)gridDim.x * blockDim.x)
    ptr[r] = pos[ptr[r]];
}

__global__ void chunk_counts(const int32_t* __restrict__ ptr, int64_t rows, int32_t* __restrict__ cnt) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int deg = ptr[r + 1] - ptr[r];
    cnt[r] = deg > kHubDegree ? (deg + kChunkEdges - 1) / kChunkEdges : 0;
  }
}

__global__ void chunk_fill(const int32_t* __restrict__ ofs, int64_t rows, int32_t* __restrict__ chunk_row) {
  pdl_begin();
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    for (int c = ofs[r]; c < ofs[r + 1]; ++c) chunk_row[c] = (int32_t)r;
  }
}

// ---- node order of the forward projection: a stable counting sort of each type's nodes by relation
// mask (at most kMaxRels relations into a type: 2^8 mask values).  Blocks own kOrderTile nodes.
constexpr int kOrderTile = 2048;
constexpr int kMaskValues = 1 << kMaxRels;

struct TypeRels {
  int n;                     // relations into the type
  int64_t row0[kMaxRels];    // CSR row of the type's local node 0 in each, by ascending relation id
};

__device__ __forceinline__ uint32_t node_mask(const int32_t* __restrict__ csr_ptr, const TypeRels& tr, int64_t j) {
  uint32_t m = 0;
  for (int k = 0; k < tr.n; ++k) {
    const int64_t row = tr.row0[k] + j;
    if (__ldg(csr_ptr + row + 1) > __ldg(csr_ptr + row)) m |= 1u << k;
  }
  return m;
}

// hist[v * nblk + block] = nodes of the block with mask v
__global__ void __launch_bounds__(256) order_hist(const int32_t* __restrict__ csr_ptr, TypeRels tr, int64_t n,
                                                  int nblk, int32_t* __restrict__ hist) {
  pdl_begin();
  __shared__ int32_t h[kMaskValues];
  const int V = 1 << tr.n;
  for (int v = threadIdx.x; v < V; v += blockDim.x) h[v] = 0;
  __syncthreads();
  const int64_t j0 = (int64_t)blockIdx.x * kOrderTile;
  for (int k = threadIdx.x; k < kOrderTile; k += blockDim.x) {
    const int64_t j = j0 + k;
    if (j < n) atomicAdd(&h[node_mask(csr_ptr, tr, j)], 1);
  }
  __syncthreads();
  for (int v = threadIdx.x; v < V; v += blockDim.x) hist[(int64_t)v * nblk + blockIdx.x] = h[v];
}

// perm[ofs[v * nblk + block] + rank] = j, rank = the node's place among the block's nodes with mask v
// in ascending id (rounds of 256 nodes; within a round, warp-level ranks plus earlier warps' counts)
__global__ void __launch_bounds__(256) order_scatter(const int32_t* __restrict__ csr_ptr, TypeRels tr, int64_t n,
                                                     int nblk, const int32_t* __restrict__ ofs,
                                                     int32_t* __restrict__ perm) {
  pdl_begin();
  __shared__ int32_t next[kMaskValues];
  __shared__ int32_t wcnt[8][kMaskValues];
  const int V = 1 << tr.n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int v = threadIdx.x; v < V; v += 256) next[v] = ofs[(int64_t)v * nblk + blockIdx.x];
  const int64_t j0 = (int64_t)blockIdx.x * kOrderTile;
  for (int k = 0; k < kOrderTile; k += 256) {
    for (int i = threadIdx.x; i < 8 * V; i += 256) wcnt[i / V][i % V] = 0;
    __syncthreads();
    const int64_t j = j0 + k + threadIdx.x;
    const bool live = j < n;
    const uint32_t mk = live ? node_mask(csr_ptr, tr, j) : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xffffffffu, mk);
    const int lrank = __popc(peers & ((1u << lane) - 1u));
    if (live && lrank == 0) wcnt[warp][mk] = __popc(peers);
    __syncthreads();
    if (live) {
      int pos = next[mk] + lrank;
      for (int w = 0; w < warp; ++w) pos += wcnt[w][mk];
      perm[pos] = (int32_t)j;
    }
    __syncthreads();
    for (int v = threadIdx.x; v < V; v += 256) {
      int c = 0;
      for (int w = 0; w < 8; ++w) c += wcnt[w][v];
      next[v] += c;
    }
    __syncthreads();
  }
}

// *nzero = nodes of the type with mask 0 (the scan's entry of mask 1, block 0);
// tmask[q] = OR of the masks at positions kProjTileRows q .. + kProjTileRows - 1 (one warp per tile)
__global__ void __launch_bounds__(256) order_tiles(const int32_t* __restrict__ csr_ptr, TypeRels tr, int64_t n,
                                                   const int32_t* __restrict__ perm, int64_t tiles,
                                                   int32_t* __restrict__ tmask, const int32_t* __restrict__ nz_src,
                                                   int32_t* __restrict__ nzero) {
  pdl_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) *nzero = *nz_src;
  const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (q >= tiles) return;
  uint32_t m = 0;
  for (int i = lane; i < kProjTileRows; i += 32) {
    const int64_t p = q * kProjTileRows + i;
    if (p < n) m |= node_mask(csr_ptr, tr, perm[p]);
  }
  m = __reduce_or_sync(0xffffffffu, m);
  if (lane == 0) tmask[q] = (int32_t)m;
}

static int64_t order_blocks(int64_t n) { return ceil_div(n, kOrderTile); }
// histogram entries over all types: sum_t 2^n_t ceil(n_t / kOrderTile) <= 2^8 (N / kOrderTile + kMaxTypes)
static int64_t order_hist_cap(int64_t N) { return (int64_t)kMaskValues * (N / kOrderTile + kMaxTypes); }
static int64_t order_tiles_cap(int64_t N) { return N / kProjTileRows + kMaxTypes; }

// Rows above kHubDegree hold sum ceil(deg / kChunkEdges) <= E / kChunkEdges + E / (kHubDegree + 1)
// chunks (each such row adds at most one partial chunk); +2 covers the integer floors.
// Chunks of `rows` rows with E runs in all: the whole ones, and one more per row above the hub degree.
static int64_t chunk_cap(int64_t E, int64_t rows) {
  return E / kChunkEdges + std::min(E / (kHubDegree + 1), rows) + 2;
}
// a long row has more than kFuseRuns runs, each of at least one edge
static int64_t long_cap(int64_t E) { return E / (kFuseRuns + 1) + 1; }

struct GraphLayout {
  int32_t *csr_ptr, *csr_col, *csr_eid, *csc_ptr, *csc_col, *csc_eid;
  float* csc_coef;
  int32_t* run_pos;  // first CSR position of each run of parallel edges
  uint32_t* row_pack;  // compact place and in-degree of each CSR row
  int32_t *invalid, *cnt;
  // parallel edges coalesced: CSR rows and node-major rows as (column, multiplicity) runs
  int32_t *agg_ptr, *agg_col, *agg_cnt, *agg_chunk_ofs, *agg_chunk_row;
  int32_t *bagg_ptr, *bagg_col, *bagg_cnt, *bagg_chunk_ofs, *bagg_chunk_row;
  int32_t *mrow, *mlist, *mbase;  // non-empty CSR rows: compact index per row, row per index, per relation
  int32_t *nperm, *tmask, *nzero, *ohist, *oofs;  // node order by relation mask, tile masks, the sort's counts
  int32_t *long_ofs, *long_list;          // the fused layer's long rows
  SortBuffers sort;
};

static size_t carve_graph(void* ws, int64_t E, int64_t rows, int64_t crows, int64_t N, GraphLayout* L) {
  Carve c(ws);
  const int64_t Ea = std::max<int64_t>(E, 1);
  L->csr_ptr = c.take<int32_t>(rows + 1);
  L->csr_col = c.take<int32_t>(Ea);
  L->csr_eid = c.take<int32_t>(Ea);
  L->csc_ptr = c.take<int32_t>(crows + 1);
  L->csc_col = c.take<int32_t>(Ea);
  L->csc_eid = c.take<int32_t>(Ea);
  L->csc_coef = c.take<float>(Ea);
  L->run_pos = c.take<int32_t>(Ea + 1);
  L->row_pack = c.take<uint32_t>(rows + 1);
  L->agg_ptr = c.take<int32_t>(rows + 1);
  L->agg_col = c.take<int32_t>(Ea);
  L->agg_cnt = c.take<int32_t>(Ea);
  L->agg_chunk_ofs = c.take<int32_t>(rows + 1);
  L->agg_chunk_row = c.take<int32_t>(chunk_cap(E, rows));
  L->bagg_ptr = c.take<int32_t>(N + 1);
  L->bagg_col = c.take<int32_t>(Ea);
  L->bagg_cnt = c.take<int32_t>(Ea);
  L->bagg_chunk_ofs = c.take<int32_t>(N + 1);
  L->bagg_chunk_row = c.take<int32_t>(chunk_cap(E, N));
  L->mrow = c.take<int32_t>(rows + 1);
  L->mlist = c.take<int32_t>(rows + 1);
  L->mbase = c.take<int32_t>(kMaxRels + 1);
  L->nperm = c.take<int32_t>(std::max<int64_t>(N, 1));
  L->tmask = c.take<int32_t>(order_tiles_cap(N));
  L->nzero = c.take<int32_t>(kMaxTypes);
  L->long_ofs = c.take<int32_t>(rows + 1);
  L->long_list = c.take<int32_t>(long_cap(E));
  L->ohist = c.take<int32_t>(order_hist_cap(N) + 1);
  L->oofs = c.take<int32_t>(order_hist_cap(N) + 1);
  L->invalid = c.take<int32_t>(1);
  L->cnt = c.take<int32_t>(std::max(std::max(rows, crows), N) + 1);
  L->sort.ckeys = c.take<uint32_t>(Ea + 1);
  for (int i = 0; i < 2; ++i) {  // one entry more than the edges: the coalescing scans reuse them
    L->sort.keys[i] = c.take<uint32_t>(Ea + 1);
    L->sort.vals[i] = c.take<uint32_t>(Ea + 1);
    L->sort.vals2[i] = c.take<uint32_t>(Ea + 1);
  }
  const int64_t hist_n = sort_tiles(E) * kMaxRadix;
  L->sort.hist = c.take<int32_t>(hist_n + 1);
  L->sort.scan_scratch =
      c.take<char>(scan_scratch_bytes(std::max(std::max(std::max(hist_n, rows), std::max(crows, N)),
                                               std::max(Ea, order_hist_cap(N)))));
  return c.used;
}

static hg_status make_meta(const int64_t* type_offsets, int32_t num_types, const hg_rel_desc* rels,
                           int32_t num_rels, GraphMeta* m) {
  HG_REQUIRE(type_offsets != nullptr && rels != nullptr, "type_offsets and rels must be non-null");
  if (num_types < 1 || num_types > kMaxTypes || num_rels < 1 || num_rels > kMaxRels) {
    set_error("need 1 <= num_types <= %d and 1 <= num_rels <= %d (got %d, %d)", kMaxTypes, kMaxRels,
              num_types, num_rels);
    return HG_ERR_UNSUPPORTED;
  }
  HG_REQUIRE(type_offsets[0] == 0, "type_offsets[0] must be 0");
  for (int t = 0; t < num_types; ++t)
    HG_REQUIRE(type_offsets[t + 1] >= type_offsets[t], "type_offsets must be non-decreasing");
  if (type_offsets[num_types] >= (int64_t(1) << 31)) {
    set_error("more than 2^31 - 1 nodes");
    return HG_ERR_UNSUPPORTED;
  }
  *m = GraphMeta{};
  m->num_types = num_types;
  m->num_rels = num_rels;
  for (int t = 0; t <= num_types; ++t) m->type_off[t] = type_offsets[t];
  for (int t = num_types + 1; t <= kMaxTypes; ++t) m->type_off[t] = type_offsets[num_types];
  m->row_base[0] = m->csc_base[0] = 0;
  for (int r = 0; r < num_rels; ++r) {
    const int s = rels[r].src_type, d = rels[r].dst_type;
    HG_REQUIRE(s >= 0 && s < num_types && d >= 0 && d < num_types,
               "relation %d has a node type out of range", r);
    m->rel_src[r] = s;
    m->rel_dst[r] = d;
    m->row_base[r + 1] = m->row_base[r] + (type_offsets[d + 1] - type_offsets[d]);
    m->csc_base[r + 1] = m->csc_base[r] + (type_offsets[s + 1] - type_offsets[s]);
  }
  if (m->row_base[num_rels] >= (int64_t(1) << 31) - 1 || m->csc_base[num_rels] >= (int64_t(1) << 31) - 1) {
    set_error("more than 2^31 - 2 relation rows");
    return HG_ERR_UNSUPPORTED;
  }
  return HG_OK;
}

static int bit_width(uint64_t x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

static unsigned grid_for(int64_t n, int threads = 256) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, threads), 152 * 16));
}

// ofs = exclusive scan of the chunk counts of the rows above the hub degree, row = the row of each chunk.
static hg_status chunk_table(const int32_t* ptr, int64_t rows, int32_t* ofs, int32_t* row, GraphLayout& L,
                             cudaStream_t s) {
  HG_TRY(launch("chunk_counts", chunk_counts, dim3(grid_for(rows)), dim3(256), 0, s, ptr, rows, L.cnt));
  HG_TRY(exclusive_scan(L.cnt, ofs, rows, L.sort.scan_scratch, s));
  return launch("chunk_fill", chunk_fill, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)ofs, rows, row);
}

}  // namespace hg

using namespace hg;

extern "C" hg_status hg_graph_workspace_size(int64_t num_edges, const int64_t* type_offsets,
                                             int32_t num_types, const hg_rel_desc* rels,
                                             int32_t num_rels, size_t* bytes) {
  clear_error();
  HG_REQUIRE(bytes != nullptr, "bytes must be non-null");
  HG_REQUIRE(num_edges >= 0, "num_edges must be >= 0");
  if (num_edges >= (int64_t(1) << 31)) {
    set_error("num_edges >= 2^31 is not supported");
    return HG_ERR_UNSUPPORTED;
  }
  GraphMeta m;
  HG_TRY(make_meta(type_offsets, num_types, rels, num_rels, &m));
  GraphLayout L;
  *bytes = carve_graph(nullptr, num_edges, m.row_base[num_rels], m.csc_base[num_rels], m.type_off[m.num_types], &L);
  return HG_OK;
}

extern "C" hg_status hg_build_csr(const int32_t* src, const int32_t* dst, const int32_t* rel,
                                  int64_t num_edges, const int64_t* type_offsets, int32_t num_types,
                                  const hg_rel_desc* rels, int32_t num_rels, void* workspace,
                                  size_t workspace_bytes, hg_stream stream, hg_graph** out) {
  clear_error();
  HG_TRY(device_guard());
  HG_REQUIRE(out != nullptr, "out must be non-null");
  *out = nullptr;
  HG_REQUIRE(num_edges >= 0, "num_edges must be >= 0");
  if (num_edges >= (int64_t(1) << 31)) {
    set_error("num_edges >= 2^31 is not supported");
    return HG_ERR_UNSUPPORTED;
  }
  HG_REQUIRE(num_edges == 0 || (src && dst && rel), "src, dst and rel must be non-null");
  HG_REQUIRE(workspace != nullptr, "workspace must be non-null");
  HG_REQUIRE(((uintptr_t)workspace & 255) == 0, "workspace must be 256-byte aligned");
  GraphMeta m;
  HG_TRY(make_meta(type_offsets, num_types, rels, num_rels, &m));
  const int64_t E = num_edges, rows = m.row_base[num_rels], crows = m.csc_base[num_rels];
  GraphLayout L;
  const int64_t N = m.type_off[num_types];
  const size_t need = carve_graph(nullptr, E, rows, crows, N, &L);
  if (workspace_bytes < need) {
    set_error("workspace has %zu bytes, %zu needed", workspace_bytes, need);
    return HG_ERR_WORKSPACE;
  }
  carve_graph(workspace, E, rows, crows, N, &L);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

  const unsigned g = grid_for(E + 1);
  int res = 0;
  if (E == 0) {
    HG_CUDA(cudaMemsetAsync(L.csr_ptr, 0, (rows + 1) * sizeof(int32_t), s));
    HG_CUDA(cudaMemsetAsync(L.csc_ptr, 0, (crows + 1) * sizeof(int32_t), s));
    HG_CUDA(cudaMemsetAsync(L.agg_ptr, 0, (rows + 1) * sizeof(int32_t), s));
    HG_CUDA(cudaMemsetAsync(L.bagg_ptr, 0, (N + 1) * sizeof(int32_t), s));
    HG_CUDA(cudaMemsetAsync(L.invalid, 0, sizeof(int32_t), s));
  } else {
    // CSR by (destination row, source, edge id): a stable sort by source, then by row
    HG_TRY(launch("edge_keys", edge_keys, dim3(g), dim3(256), 0, s, src, dst, rel, E, m, rows, L.sort.keys[0],
                  L.sort.ckeys));
    int r1 = 0;
    HG_TRY(radix_sort(L.sort, E, nullptr, bit_width((uint64_t)N), (const uint32_t*)L.sort.keys[0],
                      (const uint32_t*)nullptr, (const uint32_t*)L.sort.ckeys, 0, s, &r1));
    // the last pass writes the edge ids and source ids straight into csr_eid and csr_col
    HG_TRY(radix_sort(L.sort, E, nullptr, bit_width((uint64_t)rows), (const uint32_t*)L.sort.vals2[r1],
                      (const uint32_t*)L.sort.vals[r1], (const uint32_t*)L.sort.keys[r1], r1, s, &res,
                      (uint32_t*)L.csr_eid, (uint32_t*)L.csr_col));
    HG_TRY(launch("row_ptr_from_keys", row_ptr_from_keys, dim3(grid_for(E / 4 + 1)), dim3(256), 0, s,
                  (const uint32_t*)L.sort.keys[res], E, (const int32_t*)nullptr, rows, L.csr_ptr, L.invalid));
  }
  // non-empty CSR rows (the rows the mean layer stores) and their compact numbering
  HG_TRY(launch("nonempty_flags", nonempty_flags, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)L.csr_ptr,
                rows, L.cnt));
  HG_TRY(exclusive_scan(L.cnt, L.mrow, rows, L.sort.scan_scratch, s));
  HG_TRY(launch("compact_bases", compact_bases, dim3(1), dim3(32), 0, s, (const int32_t*)L.mrow, m, L.mbase));
  HG_TRY(launch("compact_rows", compact_rows, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)L.cnt, rows,
                L.mrow, L.mlist));
  if (E > 0) {
    // runs of parallel edges in CSR order: the forward aggregation lists, and the runs' CSC keys
    const int o = res ^ 1;
    int32_t* flag = reinterpret_cast<int32_t*>(L.sort.keys[o]);
    int32_t* u = reinterpret_cast<int32_t*>(L.sort.vals[o]);
    const uint32_t* rkey = L.sort.keys[res];
    HG_TRY(launch("run_flags", run_flags, dim3(grid_for(E / 4 + 1)), dim3(256), 0, s, rkey, (const int32_t*)L.csr_col,
                  (const int32_t*)L.csr_ptr, rows, E, flag));
    HG_TRY(exclusive_scan(flag, u, E, L.sort.scan_scratch, s));
    HG_TRY(launch("run_write", run_write, dim3(grid_for(E / 4 + 1)), dim3(256), 0, s, (const int32_t*)u,
                  (const int32_t*)L.csr_col, rkey, (const int32_t*)L.csr_ptr, rows, m, (const int32_t*)L.csr_eid,
                  L.agg_col, L.run_pos, L.sort.ckeys, L.sort.vals2[res], L.sort.vals[res]));
    HG_TRY(launch("run_finish", run_finish, dim3(grid_for(std::max(E, rows + 1))), dim3(256), 0, s, (const int32_t*)u,
                  (const int32_t*)L.run_pos, (const int32_t*)L.csr_ptr, rows, L.agg_cnt, L.agg_ptr));
    // the runs by CSC row
    const int32_t* nruns = L.agg_ptr + rows;
    int x = 0;
    HG_TRY(radix_sort(L.sort, E, nruns, bit_width((uint64_t)crows), (const uint32_t*)L.sort.ckeys,
                      (const uint32_t*)L.sort.vals[res], (const uint32_t*)L.sort.vals2[res], res, s, &x));
    const uint32_t *skey = L.sort.keys[x], *srun = L.sort.vals[x], *sdst = L.sort.vals2[x];
    HG_TRY(launch("row_ptr_from_keys", row_ptr_from_keys, dim3(grid_for(E / 4 + 1)), dim3(256), 0, s, skey, E, nruns,
                  crows, L.csc_ptr, (int32_t*)nullptr));
    // node-major rows: out-runs per node over its relations, their scan, then the runs
    HG_TRY(launch("node_out_counts", node_out_counts, dim3(grid_for(N)), dim3(256), 0, s, (const int32_t*)L.csc_ptr,
                  m, L.cnt));
    HG_TRY(exclusive_scan(L.cnt, L.bagg_ptr, N, L.sort.scan_scratch, s));
    int32_t* qpos = reinterpret_cast<int32_t*>(L.sort.keys[x ^ 1]);
    int32_t* qstart = reinterpret_cast<int32_t*>(L.sort.vals[x ^ 1]);
    float* qcoef = reinterpret_cast<float*>(L.sort.vals2[x ^ 1]);
    // each stored row's compact place and degree
    PackBits pb{};
    for (int r = 0; r < num_rels; ++r) pb.deg[r] = 32 - bit_width((uint64_t)(m.row_base[r + 1] - m.row_base[r]));
    HG_TRY(launch("row_pack", row_pack, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)L.mrow,
                  (const int32_t*)L.mbase, (const int32_t*)L.csr_ptr, rows, m, pb, L.row_pack));
    HG_TRY(launch("csc_runs", csc_runs, dim3(g), dim3(256), 0, s, skey, srun, sdst, nruns,
                  (const int32_t*)L.csc_ptr, m, (const int32_t*)L.csr_ptr, (const uint32_t*)L.row_pack, pb,
                  (const int32_t*)L.mbase, (const int32_t*)L.run_pos, (const int32_t*)L.bagg_ptr, L.bagg_col,
                  L.bagg_cnt, qpos, qstart, qcoef));
    HG_TRY(exclusive_scan(qpos, qpos, E, L.sort.scan_scratch, s, nruns));
    HG_TRY(launch("csc_expand", csc_expand, dim3((unsigned)std::min<int64_t>(ceil_div(E, kExpand * 8), 152 * 8)),
                  dim3(256), 0, s, (const int32_t*)qpos, (const int32_t*)qstart, (const float*)qcoef,
                  sdst, nruns,
                  (const int32_t*)L.csr_eid, L.csc_col, L.csc_eid, L.csc_coef));
    HG_TRY(launch("run_to_edge_ptr", run_to_edge_ptr, dim3(grid_for(crows + 1)), dim3(256), 0, s,
                  (const int32_t*)qpos, crows, L.csc_ptr));
  }
  // the fused layer's long rows (more than kFuseRuns runs) and their compact slots
  HG_TRY(launch("long_flags", long_flags, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)L.agg_ptr, rows,
                L.cnt));
  HG_TRY(exclusive_scan(L.cnt, L.long_ofs, rows, L.sort.scan_scratch, s));
  HG_TRY(launch("compact_list", compact_list, dim3(grid_for(rows)), dim3(256), 0, s, (const int32_t*)L.cnt,
                (const int32_t*)L.long_ofs, rows, L.long_list));
  // node order of the forward projection, per type: sorted by relation mask, and each tile's mask
  int64_t tile_base[kMaxTypes + 1] = {0};
  for (int t = 0; t < m.num_types; ++t) {
    const int64_t n = m.type_off[t + 1] - m.type_off[t];
    tile_base[t + 1] = tile_base[t] + ceil_div(n, kProjTileRows);
    if (n == 0) continue;
    TypeRels tr{};
    for (int r = 0; r < num_rels; ++r)
      if (m.rel_dst[r] == t) tr.row0[tr.n++] = m.row_base[r];
    const int nblk = (int)order_blocks(n);
    const int64_t nh = ((int64_t)1 << tr.n) * nblk;
    HG_TRY(launch("order_hist", order_hist, dim3(nblk), dim3(256), 0, s, (const int32_t*)L.csr_ptr, tr, n, nblk,
                  L.ohist));
    HG_TRY(exclusive_scan(L.ohist, L.oofs, nh, L.sort.scan_scratch, s));
    int32_t* perm = L.nperm + m.type_off[t];
    HG_TRY(launch("order_scatter", order_scatter, dim3(nblk), dim3(256), 0, s, (const int32_t*)L.csr_ptr, tr, n,
                  nblk, (const int32_t*)L.oofs, perm));
    const int64_t tiles = tile_base[t + 1] - tile_base[t];
    HG_TRY(launch("order_tiles", order_tiles, dim3((unsigned)ceil_div(tiles * 32, 256)), dim3(256), 0, s,
                  (const int32_t*)L.csr_ptr, tr, n, (const int32_t*)perm, tiles, L.tmask + tile_base[t],
                  (const int32_t*)L.oofs + nblk, L.nzero + t));
  }
  // chunk tables over runs for rows above the hub degree (mean and attention layers)
  HG_TRY(chunk_table(L.agg_ptr, rows, L.agg_chunk_ofs, L.agg_chunk_row, L, s));
  HG_TRY(chunk_table(L.bagg_ptr, N, L.bagg_chunk_ofs, L.bagg_chunk_row, L, s));

  hg_graph* gh = new hg_graph{};
  gh->meta = m;
  gh->num_edges = E;
  gh->csr_rows = rows;
  gh->csc_rows = crows;
  gh->chunk_cap_csr = chunk_cap(E, rows);
  gh->chunk_cap_node = chunk_cap(E, N);
  gh->stream = s;
  gh->csr_ptr = L.csr_ptr;
  gh->csr_col = L.csr_col;
  gh->csr_eid = L.csr_eid;
  gh->csc_ptr = L.csc_ptr;
  gh->csc_col = L.csc_col;
  gh->csc_eid = L.csc_eid;
  gh->csc_coef = L.csc_coef;
  gh->agg_ptr = L.agg_ptr;
  gh->agg_col = L.agg_col;
  gh->agg_cnt = L.agg_cnt;
  gh->agg_chunk_ofs = L.agg_chunk_ofs;
  gh->agg_chunk_row = L.agg_chunk_row;
  gh->bagg_ptr = L.bagg_ptr;
  gh->bagg_col = L.bagg_col;
  gh->bagg_cnt = L.bagg_cnt;
  gh->bagg_chunk_ofs = L.bagg_chunk_ofs;
  gh->bagg_chunk_row = L.bagg_chunk_row;
  gh->mrow = L.mrow;
  gh->mlist = L.mlist;
  gh->mbase = L.mbase;
  gh->nperm = L.nperm;
  gh->tmask = L.tmask;
  gh->nzero = L.nzero;
  gh->long_ofs = L.long_ofs;
  gh->long_list = L.long_list;
  gh->long_cap = long_cap(E);
  for (int t = 0; t <= kMaxTypes; ++t) gh->tile_base[t] = tile_base[std::min(t, m.num_types)];
  gh->invalid_count = L.invalid;
  *out = gh;
  return HG_OK;
}

extern "C" hg_status hg_graph_node_order(const hg_graph* graph, int32_t type, hg_node_order* out) {
  clear_error();
  HG_REQUIRE(graph != nullptr && out != nullptr, "graph and out must be non-null");
  const GraphMeta& m = graph->meta;
  HG_REQUIRE(type >= 0 && type < m.num_types, "type %d out of range", type);
  out->n = m.type_off[type + 1] - m.type_off[type];
  out->tiles = graph->tile_base[type + 1] - graph->tile_base[type];
  out->tile_rows = kProjTileRows;
  out->perm = graph->nperm + m.type_off[type];
  out->tile_mask = graph->tmask + graph->tile_base[type];
  return HG_OK;
}

extern "C" hg_status hg_graph_destroy(hg_graph* graph) {
  delete graph;
  return HG_OK;
}

extern "C" hg_status hg_graph_check(const hg_graph* graph, int64_t* num_invalid_edges) {
  clear_error();
  HG_TRY(device_guard());
  HG_REQUIRE(graph != nullptr, "graph must be non-null");
  int32_t bad = 0;
  HG_CUDA(cudaMemcpyAsync(&bad, graph->invalid_count, sizeof(int32_t), cudaMemcpyDeviceToHost,
                          graph->stream));
  HG_CUDA(cudaStreamSynchronize(graph->stream));
  if (num_invalid_edges) *num_invalid_edges = bad;
  if (bad != 0) {
    set_error("%d edges were dropped (id out of range, relation out of range, or endpoint types "
              "that do not match the relation)", bad);
    return HG_ERR_DEVICE_CHECK;
  }
  return HG_OK;
}

extern "C" hg_status hg_graph_view(const hg_graph* graph, int32_t rel, hg_graph_arrays* out) {
  clear_error();
  HG_REQUIRE(graph != nullptr && out != nullptr, "graph and out must be non-null");
  const GraphMeta& m = graph->meta;
  HG_REQUIRE(rel >= 0 && rel < m.num_rels, "relation %d out of range", rel);
  out->n_dst = m.row_base[rel + 1] - m.row_base[rel];
  out->n_src = m.csc_base[rel + 1] - m.csc_base[rel];
  out->num_edges = graph->num_edges;
  out->row_ptr = graph->csr_ptr + m.row_base[rel];
  out->col = graph->csr_col;
  out->eid = graph->csr_eid;
  out->csc_ptr = graph->csc_ptr + m.csc_base[rel];
  out->csc_col = graph->csc_col;
  out->csc_eid = graph->csc_eid;
  out->csc_coef = graph->csc_coef;
  return HG_OK;
}
