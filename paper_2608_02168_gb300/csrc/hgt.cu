// Attention layer (Heterogeneous Graph Transformer, Section 3.2, Eq. 6-11), forward and backward.
//
// With S heads of width d_h and c_r = mu[r] / sqrt(d_h), the layer is computed as
//   K, V = H W_K + b_K, H W_V + b_V (per source type; one N x 2d array, a node's K then V)
//   Q       = H W_Q + b_Q (per target type)
//   Q'_r(j) = c_r Q_j blockdiag(W_att[r])^T   (one row per non-empty (relation, target): the compact
//             rows of the mean layer; c_r applied in fp32)  so that score^s(e) = K^s(i) . Q'^s_r(j)
//   alpha   = softmax over every in-edge of j, per head (online: running maximum and sum)
//   S_r(j)  = sum over the r-edges into j of alpha V(i)    (per head; compact rows)
//   U       = sum_r S_r blockdiag(W_msg[r]) W_agg + b_agg, then activation, residual, LayerNorm:
//             the mean layer's projection with W_rel = blockdiag(W_msg[r]).
// Every product has a stored bf16 weight as one factor (W_K, W_Q, W_V, blockdiag(W_att[r]),
// blockdiag(W_msg[r]) paired with W_agg as the projection's hi / lo fused weights), so no product
// of two weights is ever rounded to bf16; the scalar c_r multiplies in the fp32 epilogue.
// The backward reuses that projection's backward (without the 1/deg scaling) for dS_r, then
//   target pass  D^s_j = sum_r <dS_r(j), S_r(j)>^s, de = alpha (<dS_r(j), V(i)>^s - D^s_j),
//                dQ'_r(j) = sum de K(i)
//   source pass  dK(i) = sum over out-edges de Q'_r(j), dV(i) = sum alpha dS_r(j)
//   (Q', S, dS, dQ' and the row statistics exist for the non-empty rows only: on the 1M-node, 20M-edge
//   graph those are 16 % of the rows, and forward + backward went from 13.2 to 11.05 ms with them)
//   and the dense products back to H (dQ = sum_r c_r dQ'_r blockdiag(W_att[r]), then dQ W_Q^T) and
//   to the weights.
// Edge work is warp per row (a lane holds d / 32 consecutive features, the 32 / S lanes of a head
// reduce by shuffles); rows above the hub degree are split into chunks whose partial results are
// merged in chunk order, so every reduction has a fixed order (the only atomics are the claim
// counters, which decide who computes a row and not the order of its terms).  The
// dense row products run on the tensor cores for bf16 (rows_gemm_tc.cu) and on CUDA cores for fp32.
#include <cuda_bf16.h>

#include <algorithm>

#include "hg_internal.cuh"
#include "layer_kernels.cuh"
#include "simt_tile.cuh"

namespace hg {

namespace {

// ---------------------------------------------------------------------------------------------
// per-lane slices: lane l owns features [l E, (l + 1) E), E = D / 32
// ---------------------------------------------------------------------------------------------
template <typename T, int E>
__device__ __forceinline__ void load_slice(const T* __restrict__ p, float (&f)[E]) {
  if constexpr (sizeof(T) == 4) {
    if constexpr (E == 2) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(p));
      f[0] = v.x;
      f[1] = v.y;
    } else {
#pragma unroll
      for (int e = 0; e < E; e += 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p + e));
        f[e] = v.x;
        f[e + 1] = v.y;
        f[e + 2] = v.z;
        f[e + 3] = v.w;
      }
    }
  } else {
    if constexpr (E == 2) {
      const uint32_t u = __ldg(reinterpret_cast<const unsigned int*>(p));
      f[0] = __uint_as_float(u << 16);
      f[1] = __uint_as_float(u & 0xFFFF0000u);
    } else if constexpr (E == 4) {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
      f[0] = __uint_as_float(u.x << 16);
      f[1] = __uint_as_float(u.x & 0xFFFF0000u);
      f[2] = __uint_as_float(u.y << 16);
      f[3] = __uint_as_float(u.y & 0xFFFF0000u);
    } else {
      unpack(ldg16(p), f, __nv_bfloat16());
    }
  }
}

// The same slice kept as loaded (bf16 pairs stay packed until they are used: half the registers of
// the rows in flight).
template <typename T, int E>
struct RawSlice {
  static constexpr int kWords = E * (int)sizeof(T) / 4;
  uint32_t w[kWords];
  __device__ __forceinline__ void load(const T* __restrict__ p) {
    if constexpr (kWords == 1) {
      w[0] = __ldg(reinterpret_cast<const unsigned int*>(p));
    } else if constexpr (kWords == 2) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
      w[0] = v.x;
      w[1] = v.y;
    } else {
#pragma unroll
      for (int i = 0; i < kWords; i += 4) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(p) + i / 4);
        w[i] = v.x;
        w[i + 1] = v.y;
        w[i + 2] = v.z;
        w[i + 3] = v.w;
      }
    }
  }
  __device__ __forceinline__ void get(float (&f)[E]) const {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int e = 0; e < E; ++e) f[e] = __uint_as_float(w[e]);
    } else {
#pragma unroll
      for (int e = 0; e < E; e += 2) {
        f[e] = __uint_as_float(w[e / 2] << 16);
        f[e + 1] = __uint_as_float(w[e / 2] & 0xFFFF0000u);
      }
    }
  }
};

template <typename T, int E>
__device__ __forceinline__ void store_slice(T* __restrict__ p, const float (&f)[E]) {
  if constexpr (sizeof(T) == 2 && E == 4) {
    *reinterpret_cast<uint2*>(p) = make_uint2(pack2_bf16(f[0], f[1]), pack2_bf16(f[2], f[3]));
  } else if constexpr (sizeof(T) == 2 && E == 2) {
    *reinterpret_cast<uint32_t*>(p) = pack2_bf16(f[0], f[1]);
  } else if constexpr (E * sizeof(T) % 16 == 0) {
#pragma unroll
    for (int e = 0; e < E; e += VecTraits<T>::kElems) st16(p + e, pack(f + e, T()));
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) p[e] = from_f32<T>(f[e]);
  }
}

// Sum over the lanes of this lane's head (lpw = 32 / S consecutive lanes).
__device__ __forceinline__ float head_sum(float x, int lph) {
  for (int o = 1; o < lph; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// ---------------------------------------------------------------------------------------------
// block-diagonal expansion of per-head weights (exact copies, no arithmetic)
// ---------------------------------------------------------------------------------------------
// out[r] = blockdiag(W[r]) (d x d, S blocks of d_h x d_h), or its transpose when transpose != 0.
template <typename T>
__global__ void hgt_blockdiag(const T* __restrict__ W, int R, int d, int S, int transpose, T* __restrict__ out) {
  pdl_begin();
  const int dh = d / S;
  const int64_t total = (int64_t)R * d * d;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(q / ((int64_t)d * d));
    int a = (int)((q / d) % d), b = (int)(q % d);
    if (transpose) {
      const int t = a;
      a = b;
      b = t;
    }
    const int s = a / dh;
    out[q] = b / dh == s ? W[((int64_t)r * S + s) * dh * dh + (a % dh) * dh + (b % dh)] : from_f32<T>(0.f);
  }
}

// out[i][j] = W[j][i] for one d x d matrix per block row.
template <typename T>
__global__ void hgt_transpose(const T* __restrict__ W, int count, int d, T* __restrict__ out) {
  pdl_begin();
  const int64_t total = (int64_t)count * d * d;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = q / ((int64_t)d * d);
    const int i = (int)((q / d) % d), j = (int)(q % d);
    out[q] = W[m * d * d + (int64_t)j * d + i];
  }
}

// ---------------------------------------------------------------------------------------------
// dense row products on CUDA cores: out[r][ocol0 + c] (=, or +=) scale sum_k A[r][k] B[k][c]
// (+ bias[c]), c < D, rows [0, n), K a multiple of 32; A row stride lda, out row stride ldo, B is
// K x D; scale = scale_mul * (*scale_ptr) (null scale_ptr: 1).  With a map, over the relation's
// stored rows (A or out indexed through their list).
// ---------------------------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(256) hgt_gemm_simt(const T* __restrict__ A, int64_t lda, const T* __restrict__ B,
                                                     const T* __restrict__ bias, int K, int64_t n, T* __restrict__ out,
                                                     int64_t ldo, int ocol0, int accumulate,
                                                     const float* __restrict__ scale_ptr, float scale_mul,
                                                     RowMap map) {
  pdl_begin();
  using Tl = Tile<float, D>;
  constexpr int CN = Tl::CN, RM = Tl::RM;
  __shared__ __align__(16) float As[kBM][kAPad];
  extern __shared__ __align__(16) float Bs[];  // [kKC][D]
  const int64_t r0 = (int64_t)blockIdx.x * kBM;
  int64_t base = 0;
  if (map.list) {
    base = map.base[map.rel];
    n = map.base[map.rel + 1] - base;
    if (r0 >= n) return;
  }
  auto in_row = [&](int64_t r) {
    return !map.list ? r : (map.scatter ? base + r : (int64_t)map.list[base + r] - map.row0);
  };
  auto out_row = [&](int64_t r) {
    return !map.list ? r : (map.scatter ? (int64_t)map.list[base + r] - map.row0 : base + r);
  };
  float acc[RM][CN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < CN; ++j) acc[i][j] = 0.f;
  for (int k0 = 0; k0 < K; k0 += kKC) {
    for (int idx = threadIdx.x; idx < kBM * kKC; idx += blockDim.x) {
      const int m = idx / kKC, k = idx % kKC;
      As[m][k] = r0 + m < n ? to_f32(A[in_row(r0 + m) * lda + k0 + k]) : 0.f;
    }
    for (int idx = threadIdx.x; idx < kKC * D; idx += blockDim.x) {
      const int k = idx / D, c = idx % D;
      Bs[k * D + b_pos<D>(c)] = to_f32(B[(int64_t)(k0 + k) * D + c]);
    }
    __syncthreads();
    mma_chunk<D, RM, CN>(&As[0][0], kAPad, 0, Bs, acc);
    __syncthreads();
  }
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  const float sc = scale_mul * (scale_ptr ? *scale_ptr : 1.f);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int64_t r = r0 + ty * RM + i;
    if (r >= n) continue;
    T* o = out + out_row(r) * ldo + ocol0 + tx * CN;
#pragma unroll
    for (int j = 0; j < CN; ++j) {
      float v = sc * acc[i][j];
      if (bias) v += to_f32(bias[tx * CN + j]);
      if (accumulate) v += to_f32(o[j]);
      o[j] = from_f32<T>(v);
    }
  }
}

// part[block][c] = sum over the block's rows of X[row][c], rows [0, n), row stride ldx.  A thread owns one
// 16-byte piece of a row and every kRows-th row of the block, eight in flight; the threads' sums are added
// in row order.  Bound by HBM; three sums of 1M rows, d = 128
// bf16: 512 -> 145 us (a column per thread and a row at a time before).
template <typename T, int D>
__global__ void __launch_bounds__(256) hgt_colsum(const T* __restrict__ X, int64_t ldx, int64_t n,
                                                  int64_t rows_per_block, float* __restrict__ part) {
  pdl_begin();
  constexpr int VEC = VecTraits<T>::kElems, TPR = D / VEC, kRows = 256 / TPR, U = 8;
  __shared__ float red[kRows][D];
  const int g = threadIdx.x % TPR, sub = threadIdx.x / TPR;
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_block, r1 = min(n, r0 + rows_per_block);
  float s[VEC];
#pragma unroll
  for (int i = 0; i < VEC; ++i) s[i] = 0.f;
  for (int64_t r = r0 + sub; r < r1; r += U * kRows) {
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      v[u] = r + u * kRows < r1 ? ldg16(X + (r + u * kRows) * ldx + g * VEC) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float f[VEC];
      unpack(v[u], f, T());
#pragma unroll
      for (int i = 0; i < VEC; ++i) s[i] += f[i];
    }
  }
#pragma unroll
  for (int i = 0; i < VEC; ++i) red[sub][g * VEC + i] = s[i];
  __syncthreads();
  for (int c = threadIdx.x; c < D; c += 256) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < kRows; ++k) t += red[k][c];
    part[(int64_t)blockIdx.x * D + c] = t;
  }
}

// ---------------------------------------------------------------------------------------------
// edge kernels
// ---------------------------------------------------------------------------------------------
struct HgtArgs {
  GraphMeta meta;
  int8_t rslot[kMaxTypes][kMaxRels];  // relations into each type in relation order, -1 past the last
  int64_t N, csr_rows;
  int S;
  // Edges as runs of parallel edges (column, multiplicity): a run's edges share their source, target
  // and relation, so their scores, weights and gradients are equal and the run is taken once times
  // its count.  Target side: each CSR row's runs by source (dptr / dcol / dcnt, hub chunks over
  // runs); source side: each node's out-runs (sptr / scol / scnt), scol naming the target's compact row.
  const int32_t* dptr;
  const int32_t* dcol;
  const int32_t* dcnt;
  const int32_t* dchunk_ofs;
  const int32_t* dchunk_row;
  const int32_t* sptr;
  const int32_t* scol;
  const int32_t* scnt;
  const int32_t* schunk_ofs;
  const int32_t* schunk_row;
  const int32_t* mrow;   // compact row of each CSR row (>= csr_rows: the row has no in-edge)
  const int32_t* mlist;  // CSR row of each compact row
  const int32_t* mcount; // device: number of compact rows
  // nodes by relation mask, per type: positions below nzero[t] have no in-edge at all
  const int32_t* nperm;
  const int32_t* nzero;
  int32_t* work;         // claim counters of the node and row kernels (zeroed before each pass)
  const void* KV;       // N x 2d: K then V of each node
  // compact rows
  const void* Qp;    // d: relation-scaled queries
  void* Srows;       // d: attention-weighted value sums (forward output, backward input)
  const void* dS;    // d
  float2* stats;     // N x S: running maximum and sum of each target's softmax
  float4* rstat;     // S: the target's (max, 1 / sum, D_j) on each of its rows, per head
  void* dQp;         // d
  void* dK;          // N x d
  void* dV;          // N x d
  float* part;       // chunk partials
};

// Edge passes.  All of them are bound by the latency of the row gathers (a run's two rows, 2 d bytes
// each, from L2 or HBM) and by the uneven rows, so
//  - warps claim work from a counter, a few nodes or rows at a time (a warp per node in grid order
//    left the SMs waiting for the blocks that held the longest rows);
//  - the bounds of everything claimed are loaded at once, one (node, relation) or row per lane;
//  - a row's run entries are loaded 32 at a time, one per lane, and handed out by shuffles, and the
//    first window is loaded together with the row's own slices;
//  - a hub chunk is a whole CTA, an even share of its runs per warp, merged in warp order.
// 1M nodes, 20M edges (3.2M runs), d = 128 bf16, against a warp per node and per chunk: forward nodes 1.98 ->
// 0.37 ms, target pass 2.28 -> 0.31 ms, source pass 1.73 -> 0.40 ms, the three chunk passes 1.28 -> 0.96 ms.
constexpr int kBatch = 4;        // runs of a row in flight per warp
constexpr int kEdgeWarps = 4;    // warps per CTA of the node and row kernels
constexpr int kChunkWarps = 8;   // warps per hub chunk
constexpr unsigned kAll = 0xffffffffu;

// One window of run entries: lane l holds entry base + l.
struct RunWindow {
  int col, cnt;
  __device__ __forceinline__ void load(const int32_t* __restrict__ c, const int32_t* __restrict__ n, int64_t base,
                                       int64_t end) {
    const int64_t e = base + (threadIdx.x & 31);
    col = e < end ? __ldg(c + e) : 0;
    cnt = e < end ? __ldg(n + e) : 0;
  }
};

// Runs per warp of a chunk of n runs: an even share in whole batches.  (With 64 runs per warp a chunk of
// 110 left six of eight warps idle: 50k nodes with 110 distinct in-neighbours each, d = 64 fp32, forward +
// backward 7.14 ms, with even shares 3.12 ms; the 1M-node graph above, 1.06 -> 0.96 ms for the chunk passes.)
__device__ __forceinline__ int64_t chunk_share(int64_t n) {
  return (n + kChunkWarps * kBatch - 1) / (kChunkWarps * kBatch) * kBatch;
}

// Rows of more runs than this go through the chunk kernels; nchunks = the chunks of all rows above kHubDegree
// runs.  Up to kManyChunks of them the hub rows are the exception that would hold a warp while the others are
// done.  From there on they are the work itself, enough of it to keep every warp busy, and a warp per row saves
// the CTA's barriers and the partials: degrees around 110 on 50k nodes, chunks / warps 2.96 / 2.13 ms; on
// 5k nodes of skewed degrees (zipf 0.8, 100 edges per node) 0.87 / 0.99 ms.  Rows of one chunk (at most
// kChunkEdges runs) can go either way.  With the line at 256 / 384 / 512 runs: degrees around 300 6.11 / 4.73 /
// 4.74 ms, around 450 8.10 / 8.56 / 6.96 ms, but 100k nodes of zipf 0.8, 100 edges per node, 5.31 / 5.44 / 5.70 ms (5.13
// with all in chunks): a late claim of long rows is that kernel's tail.
constexpr int kManyChunks = 16384, kHubMany = 384;
static_assert(kHubMany <= kChunkEdges, "rows of one chunk only");
__device__ __forceinline__ int hub_runs(int nchunks) { return nchunks < kManyChunks ? kHubDegree : kHubMany; }

// Calls f(c, row, beg, end) for this CTA's chunks of the rows above hub_runs runs, the whole CTA together.
template <typename F>
__device__ __forceinline__ void for_chunks(const int32_t* __restrict__ ptr, const int32_t* __restrict__ chunk_ofs,
                                           const int32_t* __restrict__ chunk_row, int nchunks, F f) {
  const int lane = threadIdx.x & 31, hub = hub_runs(nchunks);
  for (int64_t w0 = blockIdx.x; w0 < nchunks; w0 += 32 * (int64_t)gridDim.x) {
    const int64_t x = w0 + lane * (int64_t)gridDim.x;  // a chunk per lane
    int row = 0, beg = 0, end = 0;
    bool take = false;
    if (x < nchunks) {
      row = chunk_row[x];
      const int b = ptr[row], e = ptr[row + 1];
      take = e - b > hub;
      beg = b + (int)(x - chunk_ofs[row]) * kChunkEdges;
      end = e - beg < kChunkEdges ? e : beg + kChunkEdges;
    }
    for (unsigned todo = __ballot_sync(kAll, take); todo; todo &= todo - 1) {
      const int i = __ffs(todo) - 1;
      f((int)(w0 + i * (int64_t)gridDim.x), __shfl_sync(kAll, row, i), (int64_t)__shfl_sync(kAll, beg, i),
        (int64_t)__shfl_sync(kAll, end, i));
    }
  }
}

// Items per claim: `most`, or fewer when every warp would not get four claims of them (1000 nodes with 110
// in-neighbours each, d = 64 fp32: 629 -> 344 us; two claims instead of four cost 5 % at 50k nodes).
__device__ __forceinline__ int claim_size(int64_t total, int most) {
  const int64_t nwarps = (int64_t)gridDim.x * kEdgeWarps;
  while (most > 1 && total < 4 * nwarps * most) most >>= 1;
  return most;
}

// claims `n` consecutive items
__device__ __forceinline__ int64_t claim(int32_t* counter, int n) {
  int c = 0;
  if ((threadIdx.x & 31) == 0) c = atomicAdd(counter, n);
  return __shfl_sync(kAll, c, 0);
}

// What the exponents of a part with maximum m are taken from: a part whose scores are all -inf has sum and
// values 0 (exp(-inf - -inf) would make it, and every row merged from it, NaN).
__device__ __forceinline__ float exp_base(float m) { return m == -INFINITY ? 0.f : m; }

// Online softmax over a batch of nb runs of one row (per lane: its head's running maximum m and sum l;
// the value accumulators are rescaled when the maximum grows).
template <typename T, int E, int NACC>
__device__ __forceinline__ void online_batch(const float (&sc)[kBatch], const float (&w)[kBatch],
                                             const RawSlice<T, E> (&v)[kBatch], int nb, float& m, float& l,
                                             float (&acc)[NACC][E], int slot) {
  float mn = m;
#pragma unroll
  for (int u = 0; u < kBatch; ++u)
    if (u < nb) mn = fmaxf(mn, sc[u]);
  if (mn > m) {
    const float so = expf(m - mn);
    l *= so;
#pragma unroll
    for (int k = 0; k < NACC; ++k)
#pragma unroll
      for (int e = 0; e < E; ++e) acc[k][e] *= so;
    m = mn;
  }
  const float mb = exp_base(m);
#pragma unroll
  for (int u = 0; u < kBatch; ++u) {
    if (u >= nb) break;
    const float p = w[u] * expf(sc[u] - mb);  // w runs with this score
    l += p;
    float f[E];
    v[u].get(f);
#pragma unroll
    for (int k = 0; k < NACC; ++k)
      if (k == slot)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[k][e] = fmaf(p, f[e], acc[k][e]);
  }
}

// The runs [beg, end) of one CSR row against the query slice q, folded into (m, l, acc[slot]); `win`
// holds the first window.
template <typename T, int D, int NACC>
__device__ __forceinline__ void fwd_edges(const HgtArgs& a, int64_t beg, int64_t end, RunWindow win,
                                          const float (&q)[D / 32], int lph, float& m, float& l,
                                          float (&acc)[NACC][D / 32], int slot) {
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31;
  const T* KV = (const T*)a.KV + lane * E;
  for (int64_t w0 = beg; w0 < end; w0 += 32) {
    if (w0 > beg) win.load(a.dcol, a.dcnt, w0, end);
    const int n = (int)min((int64_t)32, end - w0);
    for (int b = 0; b < n; b += kBatch) {
      const int nb = min(kBatch, n - b);
      RawSlice<T, E> k[kBatch], v[kBatch];
      float w[kBatch], sc[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int64_t src = __shfl_sync(kAll, win.col, b + u);
        w[u] = (float)__shfl_sync(kAll, win.cnt, b + u);
        if (u < nb) {
          k[u].load(KV + src * 2 * D);
          v[u].load(KV + src * 2 * D + D);
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        sc[u] = 0.f;
        if (u >= nb) break;
        float f[E];
        k[u].get(f);
#pragma unroll
        for (int e = 0; e < E; ++e) sc[u] = fmaf(f[e], q[e], sc[u]);
        sc[u] = head_sum(sc[u], lph);
      }
      online_batch<T, E, NACC>(sc, w, v, nb, m, l, acc, slot);
    }
  }
}

// (m, l, acc) += (pm, pl, pv) of a later part of the same softmax
template <int E, int NACC>
__device__ __forceinline__ void merge_part(float pm, float pl, const float (&pv)[E], float& m, float& l,
                                           float (&acc)[NACC][E], int slot) {
  const float mn = fmaxf(m, pm);
  if (mn > m) {
    const float so = expf(m - mn);
    l *= so;
#pragma unroll
    for (int k = 0; k < NACC; ++k)
#pragma unroll
      for (int e = 0; e < E; ++e) acc[k][e] *= so;
    m = mn;
  }
  const float sp = expf(pm - exp_base(m));
  l = fmaf(pl, sp, l);
#pragma unroll
  for (int k = 0; k < NACC; ++k)
    if (k == slot)
#pragma unroll
      for (int e = 0; e < E; ++e) acc[k][e] = fmaf(sp, pv[e], acc[k][e]);
}

// One CTA per chunk of a hub row: (m, l, unnormalised value sum) of the chunk's runs, an even share per
// warp; warp 0 merges the warps' parts in order.
template <typename T, int D>
__global__ void __launch_bounds__(32 * kChunkWarps) hgt_fwd_chunks(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  __shared__ float part[kChunkWarps][32][E + 2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lph = 32 / a.S;
  const int nchunks = a.dchunk_ofs[a.csr_rows];
  const int stride = 2 * a.S + D;
  for_chunks(a.dptr, a.dchunk_ofs, a.dchunk_row, nchunks, [&](int c, int row, int64_t cb, int64_t ce) {
    const int64_t share = chunk_share(ce - cb), beg = cb + warp * share, end = min(ce, beg + share);
    float q[E], m = -INFINITY, l = 0.f, acc[1][E];
    load_slice<T, E>((const T*)a.Qp + (int64_t)a.mrow[row] * D + lane * E, q);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[0][e] = 0.f;
    RunWindow win;
    win.load(a.dcol, a.dcnt, beg, end);
    fwd_edges<T, D, 1>(a, beg, end, win, q, lph, m, l, acc, 0);
#pragma unroll
    for (int e = 0; e < E; ++e) part[warp][lane][e] = acc[0][e];
    part[warp][lane][E] = m;
    part[warp][lane][E + 1] = l;
    __syncthreads();
    if (warp == 0) {
      for (int w = 1; w < kChunkWarps && cb + w * share < ce; ++w) {
        float pv[E];
#pragma unroll
        for (int e = 0; e < E; ++e) pv[e] = part[w][lane][e];
        merge_part<E, 1>(part[w][lane][E], part[w][lane][E + 1], pv, m, l, acc, 0);
      }
      float* p = a.part + (int64_t)c * stride;
      if (lane % lph == 0) {
        p[2 * (lane / lph)] = m;
        p[2 * (lane / lph) + 1] = l;
      }
#pragma unroll
      for (int e = 0; e < E; ++e) p[2 * a.S + lane * E + e] = acc[0][e];
    }
    __syncthreads();
  });
}

// nodes with at least one in-edge
__device__ __forceinline__ int64_t live_nodes(const HgtArgs& a) {
  int64_t n = 0;
  for (int t = 0; t < a.meta.num_types; ++t) {
    const int64_t nt = a.meta.type_off[t + 1] - a.meta.type_off[t];
    if (nt > 0) n += nt - a.nzero[t];
  }
  return n;
}
// The x-th of them as (type, local id), the types in order and each type's masks descending (nodes
// with in-edges of every relation, which hold the most runs, come first); t = -1 past the last.
__device__ __forceinline__ void live_node(const HgtArgs& a, int64_t x, int& t, int64_t& jl) {
  for (t = 0; t < a.meta.num_types; ++t) {
    const int64_t nt = a.meta.type_off[t + 1] - a.meta.type_off[t];
    const int64_t live = nt > 0 ? nt - a.nzero[t] : 0;
    if (x < live) {
      jl = a.nperm[a.meta.type_off[t] + nt - 1 - x];
      return;
    }
    x -= live;
  }
  t = -1;
  jl = 0;
}

// A warp per node j: the softmax over all of j's in-edges (its rows of every relation into its
// type, hub rows through their chunk partials in order), S_r(j) = sum alpha V for each relation.
// Lane n KS + k holds the bounds of the claim's node n, relation slot k.
template <typename T, int D, int KS>
__global__ void __launch_bounds__(32 * kEdgeWarps, (D <= 128 && KS <= 4) ? 6 : 1) hgt_fwd_nodes(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32, NC = 32 / KS;
  const int lane = threadIdx.x & 31, lph = 32 / a.S;
  const int64_t total = live_nodes(a);
  const int stride = 2 * a.S + D;
  const int nc = claim_size(total, NC), hub = hub_runs(a.dchunk_ofs[a.csr_rows]);
  for (int64_t x0 = claim(a.work, nc); x0 < total; x0 = claim(a.work, nc)) {
    int t = -1, mrow = -1, eb = 0, ee = 0, cb = 0, ce = 0;
    int64_t jl = 0;
    if (lane / KS < nc && x0 + lane / KS < total) live_node(a, x0 + lane / KS, t, jl);
    const int r = t >= 0 ? a.rslot[t][lane % KS] : -1;
    if (r >= 0) {
      const int64_t cr = a.meta.row_base[r] + jl;
      const int mr = a.mrow[cr];
      if (mr < a.csr_rows) {
        mrow = mr;
        eb = a.dptr[cr];
        ee = a.dptr[cr + 1];
        cb = a.dchunk_ofs[cr];
        ce = a.dchunk_ofs[cr + 1];
      }
    }
    const int64_t node = t >= 0 ? a.meta.type_off[t] + jl : 0;
    const int nn = (int)min((int64_t)nc, total - x0);
    for (int n = 0; n < nn; ++n) {
      int row[KS];
      RawSlice<T, E> q[KS];
      RunWindow win[KS];
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        row[k] = __shfl_sync(kAll, mrow, n * KS + k);
        const int b = __shfl_sync(kAll, eb, n * KS + k), e = __shfl_sync(kAll, ee, n * KS + k);
        if (row[k] >= 0) {
          q[k].load((const T*)a.Qp + (int64_t)row[k] * D + lane * E);
          win[k].load(a.dcol, a.dcnt, b, e);
        }
      }
      float m = -INFINITY, l = 0.f, acc[KS][E];
#pragma unroll
      for (int k = 0; k < KS; ++k)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[k][e] = 0.f;
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        const int b = __shfl_sync(kAll, eb, n * KS + k), e = __shfl_sync(kAll, ee, n * KS + k);
        const int c0 = __shfl_sync(kAll, cb, n * KS + k), c1 = __shfl_sync(kAll, ce, n * KS + k);
        if (row[k] < 0) continue;
        if (e - b > hub) {
          for (int c = c0; c < c1; c += kBatch) {  // kBatch partials loaded before the first is merged
            float pm[kBatch], pl[kBatch], pv[kBatch][E];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
              if (c + u >= c1) break;
              const float* p = a.part + (int64_t)(c + u) * stride;
              pm[u] = p[2 * (lane / lph)];
              pl[u] = p[2 * (lane / lph) + 1];
#pragma unroll
              for (int i = 0; i < E; ++i) pv[u][i] = p[2 * a.S + lane * E + i];
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
              if (c + u >= c1) break;
              merge_part<E, KS>(pm[u], pl[u], pv[u], m, l, acc, k);
            }
          }
        } else {
          float qf[E];
          q[k].get(qf);
          fwd_edges<T, D, KS>(a, b, e, win[k], qf, lph, m, l, acc, k);
        }
      }
      const float inv = l > 0.f ? 1.f / l : NAN;  // (every node here has a run: 0 only if all its scores are -inf)
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        if (row[k] < 0) continue;
        float o[E];
#pragma unroll
        for (int e = 0; e < E; ++e) o[e] = acc[k][e] * inv;
        store_slice<T, E>((T*)a.Srows + (int64_t)row[k] * D + lane * E, o);
      }
      const int64_t j = __shfl_sync(kAll, node, n * KS);
      if (lane % lph == 0) a.stats[j * a.S + lane / lph] = make_float2(l > 0.f ? m : 0.f, l);
    }
  }
}

// D^s_j = sum over j's relation rows of <dS_r(j), S_r(j)> on head s, stored with the softmax statistics
// on every row of j (the target and source passes read them by row).  One warp per node with in-edges.
template <typename T, int D>
__global__ void __launch_bounds__(256) hgt_bwd_dstats(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31, lph = 32 / a.S;
  const int64_t total = live_nodes(a), nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < total; x += nw) {
    int t;
    int64_t jl;
    live_node(a, x, t, jl);
    int row = -1;  // lane k: the compact row of relation slot k
    if (lane < kMaxRels && a.rslot[t][lane] >= 0) {
      row = a.mrow[a.meta.row_base[a.rslot[t][lane]] + jl];
      if (row >= a.csr_rows) row = -1;
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxRels; ++k) {
      const int64_t rk = __shfl_sync(kAll, row, k);
      if (rk < 0) continue;
      float u[E], v[E];
      load_slice<T, E>((const T*)a.dS + rk * D + lane * E, u);
      load_slice<T, E>((const T*)a.Srows + rk * D + lane * E, v);
#pragma unroll
      for (int e = 0; e < E; ++e) s = fmaf(u[e], v[e], s);
    }
    s = head_sum(s, lph);
    const float2 st = a.stats[(a.meta.type_off[t] + jl) * a.S + lane / lph];
    const float4 v = make_float4(st.x, st.y > 0.f ? 1.f / st.y : 0.f, s, 0.f);
#pragma unroll
    for (int k = 0; k < kMaxRels; ++k) {
      const int64_t rk = __shfl_sync(kAll, row, k);
      if (rk >= 0 && lane % lph == 0) a.rstat[rk * a.S + lane / lph] = v;
    }
  }
}

// sum over the runs [beg, end) of one row (relation r, target j) of de K(i), with
// de = alpha (<dS_r(j), V(i)> - D_j) and alpha from the saved softmax statistics.
template <typename T, int D>
__device__ __forceinline__ void dst_edges(const HgtArgs& a, int64_t beg, int64_t end, RunWindow win,
                                          const float (&q)[D / 32], const float (&g)[D / 32], float m, float inv_l,
                                          float Dh, int lph, float (&acc)[D / 32]) {
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31;
  const T* KV = (const T*)a.KV + lane * E;
  for (int64_t w0 = beg; w0 < end; w0 += 32) {
    if (w0 > beg) win.load(a.dcol, a.dcnt, w0, end);
    const int n = (int)min((int64_t)32, end - w0);
    for (int b = 0; b < n; b += kBatch) {
      const int nb = min(kBatch, n - b);
      RawSlice<T, E> k[kBatch], v[kBatch];
      float w[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int64_t src = __shfl_sync(kAll, win.col, b + u);
        w[u] = (float)__shfl_sync(kAll, win.cnt, b + u);
        if (u < nb) {
          k[u].load(KV + src * 2 * D);
          v[u].load(KV + src * 2 * D + D);
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (u >= nb) break;
        float kf[E], vf[E], s = 0.f, da = 0.f;
        k[u].get(kf);
        v[u].get(vf);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          s = fmaf(kf[e], q[e], s);
          da = fmaf(g[e], vf[e], da);
        }
        s = head_sum(s, lph);
        da = head_sum(da, lph);
        const float alpha = expf(s - m) * inv_l;
        const float de = w[u] * alpha * (da - Dh);  // the run's w edges
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = fmaf(de, kf[e], acc[e]);
      }
    }
  }
}

// Adds the warps' sums of N floats per lane in warp order into warp 0's.
template <int N>
__device__ __forceinline__ void add_warps(float (&v)[N], float (*part)[32][N], int nwarps) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int e = 0; e < N; ++e) part[warp][lane][e] = v[e];
  __syncthreads();
  if (warp == 0)
    for (int w = 1; w < nwarps; ++w)
#pragma unroll
      for (int e = 0; e < N; ++e) v[e] += part[w][lane][e];
}

template <typename T, int D>
__global__ void __launch_bounds__(32 * kChunkWarps) hgt_bwd_dst_chunks(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  __shared__ float part[kChunkWarps][32][E];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lph = 32 / a.S, h = lane / lph;
  const int nchunks = a.dchunk_ofs[a.csr_rows];
  for_chunks(a.dptr, a.dchunk_ofs, a.dchunk_row, nchunks, [&](int c, int row, int64_t cb, int64_t ce) {
    const int64_t share = chunk_share(ce - cb), beg = cb + warp * share, end = min(ce, beg + share);
    const int64_t mr = a.mrow[row];
    const float4 st = a.rstat[mr * a.S + h];
    float q[E], g[E], acc[E];
    load_slice<T, E>((const T*)a.Qp + mr * D + lane * E, q);
    load_slice<T, E>((const T*)a.dS + mr * D + lane * E, g);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    RunWindow win;
    win.load(a.dcol, a.dcnt, beg, end);
    dst_edges<T, D>(a, beg, end, win, q, g, st.x, st.y, st.z, lph, acc);
    add_warps<E>(acc, part, kChunkWarps);
    if (warp == 0)
#pragma unroll
      for (int e = 0; e < E; ++e) a.part[(int64_t)c * D + lane * E + e] = acc[e];
    __syncthreads();
  });
}

// acc += the partials [c0, c1) of one row in order, N floats per lane at p + c * stride; kBatch
// partials are loaded before the first is added.
template <int N>
__device__ __forceinline__ void add_parts(const float* __restrict__ p, int64_t stride, int c0, int c1,
                                          float (&acc)[N]) {
  for (int c = c0; c < c1; c += kBatch) {
    float v[kBatch][N];
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (c + u < c1)
#pragma unroll
        for (int e = 0; e < N; ++e) v[u][e] = p[(int64_t)(c + u) * stride + e];
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      if (c + u < c1)
#pragma unroll
        for (int e = 0; e < N; ++e) acc[e] += v[u][e];
  }
}

// dQ'_r(j) for every stored row (hub rows: their chunk partials in order).  A warp claims kRowClaim
// compact rows; the next row's slices, statistics and first window load while a row is summed.
constexpr int kRowClaim = 8;
template <typename T, int D>
__global__ void __launch_bounds__(32 * kEdgeWarps, D <= 128 ? 6 : 1) hgt_bwd_dst_rows(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31, lph = 32 / a.S, h = lane / lph;
  const int64_t total = *a.mcount;
  const int nc = claim_size(total, kRowClaim), hub = hub_runs(a.dchunk_ofs[a.csr_rows]);
  for (int64_t x0 = claim(a.work + 1, nc); x0 < total; x0 = claim(a.work + 1, nc)) {
    const int nn = (int)min((int64_t)nc, total - x0);
    int eb = 0, ee = 0, cb = 0, ce = 0;
    if (lane < nn) {
      const int64_t cr = a.mlist[x0 + lane];
      eb = a.dptr[cr];
      ee = a.dptr[cr + 1];
      cb = a.dchunk_ofs[cr];
      ce = a.dchunk_ofs[cr + 1];
    }
    RawSlice<T, E> q, g, qn, gn;
    float4 st, stn;
    RunWindow win, wn;
    auto fetch = [&](int i) {
      const int64_t mr = x0 + i;
      qn.load((const T*)a.Qp + mr * D + lane * E);
      gn.load((const T*)a.dS + mr * D + lane * E);
      stn = __ldg(a.rstat + mr * a.S + h);
      wn.load(a.dcol, a.dcnt, __shfl_sync(kAll, eb, i), __shfl_sync(kAll, ee, i));
    };
    fetch(0);
    for (int i = 0; i < nn; ++i) {
      q = qn;
      g = gn;
      st = stn;
      win = wn;
      if (i + 1 < nn) fetch(i + 1);
      const int c0 = __shfl_sync(kAll, cb, i), c1 = __shfl_sync(kAll, ce, i);
      const int b = __shfl_sync(kAll, eb, i), e1 = __shfl_sync(kAll, ee, i);
      float acc[E];
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] = 0.f;
      if (e1 - b > hub) {
        add_parts<E>(a.part + lane * E, D, c0, c1, acc);
      } else {
        float qf[E], gf[E];
        q.get(qf);
        g.get(gf);
        dst_edges<T, D>(a, b, e1, win, qf, gf, st.x, st.y, st.z, lph, acc);
      }
      store_slice<T, E>((T*)a.dQp + (x0 + i) * D + lane * E, acc);
    }
  }
}

// Out-runs [beg, end) of source i (node-major list; each entry is the compact row of the edge's
// target): dK(i) += de Q'_r(j) in acc[0 .. E), dV(i) += alpha dS_r(j) in acc[E .. 2 E).
template <typename T, int D>
__device__ __forceinline__ void src_edges(const HgtArgs& a, int64_t beg, int64_t end, RunWindow win,
                                          const float (&k)[D / 32], const float (&v)[D / 32], int lph,
                                          float (&acc)[D / 16]) {
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31, h = lane / lph;
  const T* Qp = (const T*)a.Qp + lane * E;
  const T* dS = (const T*)a.dS + lane * E;
  for (int64_t w0 = beg; w0 < end; w0 += 32) {
    if (w0 > beg) win.load(a.scol, a.scnt, w0, end);
    const int n = (int)min((int64_t)32, end - w0);
    for (int b = 0; b < n; b += kBatch) {
      const int nb = min(kBatch, n - b);
      RawSlice<T, E> q[kBatch], g[kBatch];
      float4 st[kBatch];
      float w[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int64_t row = __shfl_sync(kAll, win.col, b + u);
        w[u] = (float)__shfl_sync(kAll, win.cnt, b + u);
        if (u < nb) {
          q[u].load(Qp + row * D);
          g[u].load(dS + row * D);
          st[u] = __ldg(a.rstat + row * a.S + h);
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (u >= nb) break;
        float qf[E], gf[E], s = 0.f, da = 0.f;
        q[u].get(qf);
        g[u].get(gf);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          s = fmaf(k[e], qf[e], s);
          da = fmaf(gf[e], v[e], da);
        }
        s = head_sum(s, lph);
        da = head_sum(da, lph);
        const float alpha = w[u] * expf(s - st[u].x) * st[u].y;  // the run's w edges
        const float de = alpha * (da - st[u].z);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          acc[e] = fmaf(de, qf[e], acc[e]);
          acc[E + e] = fmaf(alpha, gf[e], acc[E + e]);
        }
      }
    }
  }
}

// Partials of the source pass: lane-major, 2 E floats per lane (dK then dV).
template <typename T, int D>
__global__ void __launch_bounds__(32 * kChunkWarps) hgt_bwd_src_chunks(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  __shared__ float part[kChunkWarps][32][2 * E];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lph = 32 / a.S;
  const int nchunks = a.schunk_ofs[a.N];
  const T* KV = (const T*)a.KV;
  for_chunks(a.sptr, a.schunk_ofs, a.schunk_row, nchunks, [&](int c, int i, int64_t cb, int64_t ce) {
    const int64_t share = chunk_share(ce - cb), beg = cb + warp * share, end = min(ce, beg + share);
    float k[E], v[E], acc[2 * E];
    load_slice<T, E>(KV + (int64_t)i * 2 * D + lane * E, k);
    load_slice<T, E>(KV + (int64_t)i * 2 * D + D + lane * E, v);
#pragma unroll
    for (int e = 0; e < 2 * E; ++e) acc[e] = 0.f;
    RunWindow win;
    win.load(a.scol, a.scnt, beg, end);
    src_edges<T, D>(a, beg, end, win, k, v, lph, acc);
    add_warps<2 * E>(acc, part, kChunkWarps);
    if (warp == 0)
#pragma unroll
      for (int e = 0; e < 2 * E; ++e) a.part[((int64_t)c * 32 + lane) * 2 * E + e] = acc[e];
    __syncthreads();
  });
}

// dK(i), dV(i) of every node (zeros without out-edges); claims and prefetch as in hgt_bwd_dst_rows.
template <typename T, int D>
__global__ void __launch_bounds__(32 * kEdgeWarps, D <= 128 ? 6 : 1) hgt_bwd_src_nodes(HgtArgs a) {
  pdl_begin();
  constexpr int E = D / 32;
  const int lane = threadIdx.x & 31, lph = 32 / a.S;
  const T* KV = (const T*)a.KV;
  const int nc = claim_size(a.N, kRowClaim), hub = hub_runs(a.schunk_ofs[a.N]);
  for (int64_t x0 = claim(a.work + 2, nc); x0 < a.N; x0 = claim(a.work + 2, nc)) {
    const int nn = (int)min((int64_t)nc, a.N - x0);
    int eb = 0, ee = 0, cb = 0, ce = 0;
    if (lane < nn) {
      eb = a.sptr[x0 + lane];
      ee = a.sptr[x0 + lane + 1];
      cb = a.schunk_ofs[x0 + lane];
      ce = a.schunk_ofs[x0 + lane + 1];
    }
    RawSlice<T, E> k, v, kn, vn;
    RunWindow win, wn;
    auto fetch = [&](int i) {
      const int b = __shfl_sync(kAll, eb, i), e = __shfl_sync(kAll, ee, i);
      if (b == e) return;
      kn.load(KV + (x0 + i) * 2 * D + lane * E);
      vn.load(KV + (x0 + i) * 2 * D + D + lane * E);
      wn.load(a.scol, a.scnt, b, e);
    };
    fetch(0);
    for (int i = 0; i < nn; ++i) {
      k = kn;
      v = vn;
      win = wn;
      if (i + 1 < nn) fetch(i + 1);
      const int c0 = __shfl_sync(kAll, cb, i), c1 = __shfl_sync(kAll, ce, i);
      const int b = __shfl_sync(kAll, eb, i), e1 = __shfl_sync(kAll, ee, i);
      float acc[2 * E];
#pragma unroll
      for (int e = 0; e < 2 * E; ++e) acc[e] = 0.f;
      if (e1 - b > hub) {
        add_parts<2 * E>(a.part + lane * 2 * E, 2 * D, c0, c1, acc);
      } else if (e1 > b) {
        float kf[E], vf[E];
        k.get(kf);
        v.get(vf);
        src_edges<T, D>(a, b, e1, win, kf, vf, lph, acc);
      }
      float o[E];
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = acc[e];
      store_slice<T, E>((T*)a.dK + (x0 + i) * D + lane * E, o);
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = acc[E + e];
      store_slice<T, E>((T*)a.dV + (x0 + i) * D + lane * E, o);
    }
  }
}

// dW_msg[r][s] = the diagonal blocks of the dense gradient G[r] (d x d); dW_att[r][s] = c_r times the
// blocks of Gq[r] = dQ'_r^T Q; dmu[r] = <blockdiag(W_att[r]), Gq[r]> / sqrt(d_h) (one block per relation,
// fixed-order reduction).
template <typename T>
__global__ void __launch_bounds__(256) hgt_finish(const float* __restrict__ G, const float* __restrict__ Gq,
                                                  const T* __restrict__ W_att, const float* __restrict__ mu, int d,
                                                  int S, float* __restrict__ dW_msg, float* __restrict__ dW_att,
                                                  float* __restrict__ dmu) {
  pdl_begin();
  __shared__ double red[256];  // the sum's terms cancel: in fp32 its rounding was most of dmu's error
  const int r = blockIdx.x, dh = d / S;
  const float rs = rsqrtf((float)dh);
  const float c = mu[r] * rs;
  double acc = 0.0;
  for (int q = threadIdx.x; q < S * dh * dh; q += blockDim.x) {
    const int s = q / (dh * dh), a = (q / dh) % dh, b = q % dh;
    const int64_t gi = (int64_t)r * d * d + (int64_t)(s * dh + a) * d + s * dh + b;
    dW_msg[(int64_t)r * S * dh * dh + q] = G[gi];
    dW_att[(int64_t)r * S * dh * dh + q] = c * Gq[gi];
    acc = fma((double)to_f32(W_att[(int64_t)r * S * dh * dh + q]), (double)Gq[gi], acc);
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)blockDim.x; ++k) t += red[k];
    dmu[r] = (float)(t * (double)rs);
  }
}

}  // namespace
}  // namespace hg

namespace hg {
namespace {

struct HgtLayout {
  LayerLayout L;
  // saved
  void* KV;       // N x 2d
  void* Qp;       // csr_rows x d
  float2* stats;  // N x S
  void* BDmsg;    // R x d x d  blockdiag(W_msg[r])
  // scratch
  void* BDattT;   // R x d x d  blockdiag(W_att[r])^T
  void* BDatt;    // R x d x d  blockdiag(W_att[r])
  void* WKt;      // T x d x d
  void* WVt;      // T x d x d
  void* WQt;      // T x d x d
  float4* rstat;  // csr_rows x S
  void* dQp;      // csr_rows x d
  void* dK;       // N x d
  void* dV;       // N x d
  void* Qbuf;     // N x d: Q (forward), recomputed in the backward
  void* dQ;       // N x d
  float* part;    // chunk partials (L.agg_part)
  float* cs;      // column-sum partials
  float* Gw;      // R x d x d
  float* Gq;      // R x d x d
};

// rows per block of the bias sums: 128, or more so that there are at most eight blocks per SM
constexpr int64_t kColRows = 128;
int64_t col_rows(int64_t n) { return std::max(kColRows, ceil_div(n, 152 * 8)); }

int64_t max_type_rows(const GraphMeta& m) {
  int64_t r = 1;
  for (int t = 0; t < m.num_types; ++t) r = std::max(r, m.type_off[t + 1] - m.type_off[t]);
  return r;
}

void carve_hgt(const hg_graph* g, const hg_hgt_params* p, void* saved, void* scratch, HgtLayout* H,
               size_t* saved_bytes, size_t* scratch_bytes) {
  const GraphMeta& m = g->meta;
  const int d = p->d, S = p->heads;
  const size_t b = p->dtype == HG_F32 ? 4 : 2;
  const int64_t N = m.type_off[m.num_types];
  const size_t dd = (size_t)d * d;
  size_t ls = 0, lk = 0;
  // the chunk partials are the layer's: the projection has none of its own
  const int64_t pc = std::max<int64_t>(g->chunk_cap_csr * (2 * S + d), g->chunk_cap_node * 2 * d);
  carve_layer(g, d, p->dtype, saved, scratch, &H->L, &ls, &lk, false, pc);
  H->part = H->L.agg_part;
  Carve s(saved), k(scratch);
  s.used = align_up(ls);
  k.used = align_up(lk);
  H->KV = s.take<char>((size_t)std::max<int64_t>(N, 1) * 2 * d * b);
  H->Qp = s.take<char>((size_t)std::max<int64_t>(g->csr_rows, 1) * d * b);
  H->stats = s.take<float2>((size_t)std::max<int64_t>(N, 1) * S);
  H->BDmsg = s.take<char>(m.num_rels * dd * b);
  H->BDattT = k.take<char>(m.num_rels * dd * b);
  H->BDatt = k.take<char>(m.num_rels * dd * b);
  H->WKt = k.take<char>(m.num_types * dd * b);
  H->WVt = k.take<char>(m.num_types * dd * b);
  H->WQt = k.take<char>(m.num_types * dd * b);
  H->rstat = k.take<float4>((size_t)std::max<int64_t>(g->csr_rows, 1) * S);
  H->dQp = k.take<char>((size_t)std::max<int64_t>(g->csr_rows, 1) * d * b);
  H->dK = k.take<char>((size_t)std::max<int64_t>(N, 1) * d * b);
  H->dV = k.take<char>((size_t)std::max<int64_t>(N, 1) * d * b);
  H->Qbuf = k.take<char>((size_t)std::max<int64_t>(N, 1) * d * b);
  H->dQ = k.take<char>((size_t)std::max<int64_t>(N, 1) * d * b);
  H->cs = k.take<float>((size_t)152 * 8 * d);
  H->Gw = k.take<float>(m.num_rels * dd);
  H->Gq = k.take<float>(m.num_rels * dd);
  if (saved_bytes) *saved_bytes = s.used;
  if (scratch_bytes) *scratch_bytes = k.used;
}

hg_layer_params projection_params(const hg_hgt_params* p, const HgtLayout& H) {
  hg_layer_params lp{};
  lp.d = p->d;
  lp.dtype = p->dtype;
  lp.act = p->act;
  lp.layernorm = p->layernorm;
  lp.ln_eps = p->ln_eps;
  lp.W_rel = H.BDmsg;
  lp.W_agg = p->W_agg;
  lp.b_agg = p->b_agg;
  lp.ln_gamma = p->ln_gamma;
  lp.ln_beta = p->ln_beta;
  return lp;
}

HgtArgs edge_args(const hg_graph* g, const hg_hgt_params* p, const HgtLayout& H) {
  HgtArgs a{};
  a.meta = g->meta;
  for (int t = 0; t < kMaxTypes; ++t) {
    int k = 0;
    for (int r = 0; r < kMaxRels; ++r) a.rslot[t][r] = -1;
    for (int r = 0; r < g->meta.num_rels; ++r)
      if (t < g->meta.num_types && g->meta.rel_dst[r] == t) a.rslot[t][k++] = (int8_t)r;
  }
  a.N = g->meta.type_off[g->meta.num_types];
  a.csr_rows = g->csr_rows;
  a.S = p->heads;
  a.dptr = g->agg_ptr;
  a.dcol = g->agg_col;
  a.dcnt = g->agg_cnt;
  a.dchunk_ofs = g->agg_chunk_ofs;
  a.dchunk_row = g->agg_chunk_row;
  a.sptr = g->bagg_ptr;
  a.scol = g->bagg_col;
  a.scnt = g->bagg_cnt;
  a.schunk_ofs = g->bagg_chunk_ofs;
  a.schunk_row = g->bagg_chunk_row;
  a.mrow = g->mrow;
  a.mlist = g->mlist;
  a.mcount = g->mbase + g->meta.num_rels;
  a.nperm = g->nperm;
  a.nzero = g->nzero;
  a.work = H.L.work;
  a.KV = H.KV;
  a.Qp = H.Qp;
  a.Srows = H.L.M;
  a.dS = H.L.dMs;
  a.stats = H.stats;
  a.rstat = H.rstat;
  a.dQp = H.dQp;
  a.dK = H.dK;
  a.dV = H.dV;
  a.part = H.part;
  return a;
}

// Relations into the busiest type (the node kernels keep one slot per relation of a type).
int max_rels_per_type(const GraphMeta& m) {
  int best = 0;
  for (int t = 0; t < m.num_types; ++t) {
    int k = 0;
    for (int r = 0; r < m.num_rels; ++r) k += m.rel_dst[r] == t;
    best = std::max(best, k);
  }
  return best;
}

unsigned grid_of(int64_t threads) { return (unsigned)std::max<int64_t>(1, ceil_div(threads, 256)); }
unsigned chunk_blocks(int64_t cap) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>(cap, 152 * 8)); }
// CTAs of a claiming kernel over at most n items: what the SMs hold, or fewer for few items
unsigned claim_blocks(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, kEdgeWarps), 152 * 6));
}

template <typename T, int D>
hg_status gemm(const void* A, int64_t lda, const void* B, const void* bias, int K, int64_t n, void* out, int64_t ldo,
               int ocol0, int accumulate, cudaStream_t s, const float* scale_ptr = nullptr, float scale_mul = 1.f,
               const RowMap& map = RowMap{}) {
  if (n <= 0) return HG_OK;
  if constexpr (sizeof(T) == 2) {  // bf16: tensor cores (every product here has K = lda = D)
    if (lda == D && K == D)
      return rows_gemm_tc(D, A, n, B, bias, out, ldo, ocol0, accumulate, scale_ptr, scale_mul, s, map);
  }
  return launch("hgt_gemm_simt", hgt_gemm_simt<T, D>, dim3((unsigned)ceil_div(n, kBM)), dim3(256),
                sizeof(float) * kKC * D, s, (const T*)A, lda, (const T*)B, (const T*)bias, K, n, (T*)out, ldo, ocol0,
                accumulate, scale_ptr, scale_mul, map);
}

// relation r's stored rows
RowMap rel_rows(const hg_graph* g, int r, bool scatter) {
  return RowMap{g->mlist, g->mbase, r, g->meta.row_base[r], scatter ? 1 : 0};
}

template <typename T, int D>
hg_status colsum(const void* X, int64_t n, float* cs, float* out, float* tmp, cudaStream_t s) {
  if (n <= 0) {
    HG_CUDA(cudaMemsetAsync(out, 0, sizeof(float) * D, s));
    return HG_OK;
  }
  const int blocks = (int)ceil_div(n, col_rows(n));
  HG_TRY(launch("hgt_colsum", (hgt_colsum<T, D>), dim3(blocks), dim3(256), 0, s, (const T*)X, (int64_t)D, n,
                col_rows(n), cs));
  return reduce_partials(cs, D, blocks, D, out, tmp, s);
}

hg_status wgrad(hg_dtype dt, int d, const void* X, int64_t x0, const void* Y, int64_t y0, int64_t n, float* out,
                const LayerLayout& L, cudaStream_t s) {
  if (n <= 0) {
    HG_CUDA(cudaMemsetAsync(out, 0, sizeof(float) * d * d, s));
    return HG_OK;
  }
  if (dt == HG_BF16) {
    float* outs[1] = {out};
    return tc_weight_grad(d, X, &x0, 1, Y, y0, n, L.wpart, outs, L.rtmp, s);
  }
  return weight_grad(dt, d, X, x0, Y, y0, n, L.wpart, out, L.rtmp, s);
}

template <typename T, int D>
hg_status hgt_fwd_t(const hg_graph* g, const hg_hgt_params* p, const void* H_in, void* H_out, const HgtLayout& H,
                    cudaStream_t s) {
  const GraphMeta& m = g->meta;
  const int S = p->heads;
  const int64_t N = m.type_off[m.num_types];
  const size_t dd = (size_t)D * D;
  const T* Hin = (const T*)H_in;
  const float rs = (float)(1.0 / std::sqrt((double)(D / S)));
  // block-diagonal attention (transposed) and message matrices
  HG_TRY(launch("hgt_blockdiag", hgt_blockdiag<T>, dim3(grid_of((int64_t)m.num_rels * dd)), dim3(256), 0, s,
                (const T*)p->W_att, m.num_rels, D, S, 1, (T*)H.BDattT));
  HG_TRY(launch("hgt_blockdiag", hgt_blockdiag<T>, dim3(grid_of((int64_t)m.num_rels * dd)), dim3(256), 0, s,
                (const T*)p->W_msg, m.num_rels, D, S, 0, (T*)H.BDmsg));
  // K, V and Q of every node, Q' of every stored (relation, target) row
  for (int t = 0; t < m.num_types; ++t) {
    const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
    HG_TRY((gemm<T, D>(Hin + off * D, D, (const T*)p->W_K + t * dd, (const T*)p->b_K + (size_t)t * D, D, n,
                       (T*)H.KV + off * 2 * D, 2 * D, 0, 0, s)));
    HG_TRY((gemm<T, D>(Hin + off * D, D, (const T*)p->W_V + t * dd, (const T*)p->b_V + (size_t)t * D, D, n,
                       (T*)H.KV + off * 2 * D, 2 * D, D, 0, s)));
    HG_TRY((gemm<T, D>(Hin + off * D, D, (const T*)p->W_Q + t * dd, (const T*)p->b_Q + (size_t)t * D, D, n,
                       (T*)H.Qbuf + off * D, D, 0, 0, s)));
  }
  for (int r = 0; r < m.num_rels; ++r) {  // Q'_r = c_r Q blockdiag(W_att[r])^T, c_r = mu[r] / sqrt(d_h)
    const int t = m.rel_dst[r];
    const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
    HG_TRY((gemm<T, D>((const T*)H.Qbuf + off * D, D, (const T*)H.BDattT + r * dd, nullptr, D, n,
                       H.Qp, D, 0, 0, s, p->mu + r, rs, rel_rows(g, r, false))));
  }
  // Eq. 6-10: softmax over the in-edges, weighted value sums per relation row
  const HgtArgs a = edge_args(g, p, H);
  HG_TRY(launch("hgt_fwd_chunks", hgt_fwd_chunks<T, D>, dim3(chunk_blocks(g->chunk_cap_csr)), dim3(32 * kChunkWarps), 0,
                s, a));
  HG_CUDA(cudaMemsetAsync(a.work, 0, 3 * sizeof(int32_t), s));
  const dim3 cb(32 * kEdgeWarps);
  if (max_rels_per_type(m) <= 4)
    HG_TRY(launch("hgt_fwd_nodes", hgt_fwd_nodes<T, D, 4>, dim3(claim_blocks(N)), cb, 0, s, a));
  else
    HG_TRY(launch("hgt_fwd_nodes", hgt_fwd_nodes<T, D, kMaxRels>, dim3(claim_blocks(N)), cb, 0, s, a));
  // Eq. 11 on S_r with W_rel = blockdiag(W_msg[r])
  const hg_layer_params lp = projection_params(p, H);
  return project_forward(g, &lp, H_in, H_out, H.L, s);
}

template <typename T, int D>
hg_status hgt_bwd_t(const hg_graph* g, const hg_hgt_params* p, const void* H_in, const void* dH_out, void* dH_in,
                    const hg_hgt_grads* gr, const HgtLayout& H, cudaStream_t s) {
  constexpr hg_dtype kDt = sizeof(T) == 2 ? HG_BF16 : HG_F32;
  const GraphMeta& m = g->meta;
  const int S = p->heads;
  const int64_t N = m.type_off[m.num_types];
  const size_t dd = (size_t)D * D;
  const T* Hin = (const T*)H_in;
  const float rs = (float)(1.0 / std::sqrt((double)(D / S)));
  // Eq. 11 backward: dY (residual), dS_r (no degree scaling), dW of blockdiag(W_msg), dW_agg, db, LN
  const hg_layer_params lp = projection_params(p, H);
  hg_layer_grads lg{};
  lg.dW_rel = H.Gw;
  lg.dW_agg = gr->dW_agg;
  lg.db_agg = gr->db_agg;
  lg.dln_gamma = gr->dln_gamma;
  lg.dln_beta = gr->dln_beta;
  HG_TRY(project_backward(g, &lp, H_in, dH_out, &lg, H.L, false, s));
  // attention backward: target pass (dQ'), source pass (dK, dV)
  const HgtArgs a = edge_args(g, p, H);
  const dim3 cb(32 * kEdgeWarps), hb(32 * kChunkWarps);
  HG_CUDA(cudaMemsetAsync(a.work, 0, 3 * sizeof(int32_t), s));
  HG_TRY(launch("hgt_bwd_dstats", hgt_bwd_dstats<T, D>, dim3(std::min(grid_of(N * 32), 152u * 16)), dim3(256), 0, s, a));
  HG_TRY(launch("hgt_bwd_dst_chunks", hgt_bwd_dst_chunks<T, D>, dim3(chunk_blocks(g->chunk_cap_csr)), hb, 0, s, a));
  HG_TRY(launch("hgt_bwd_dst_rows", hgt_bwd_dst_rows<T, D>, dim3(claim_blocks(g->csr_rows)), cb, 0, s, a));
  HG_TRY(launch("hgt_bwd_src_chunks", hgt_bwd_src_chunks<T, D>, dim3(chunk_blocks(g->chunk_cap_node)), hb, 0, s, a));
  HG_TRY(launch("hgt_bwd_src_nodes", hgt_bwd_src_nodes<T, D>, dim3(claim_blocks(N)), cb, 0, s, a));
  // weights of the backward products (exact copies and transposes)
  HG_TRY(launch("hgt_blockdiag", hgt_blockdiag<T>, dim3(grid_of((int64_t)m.num_rels * dd)), dim3(256), 0, s,
                (const T*)p->W_att, m.num_rels, D, S, 0, (T*)H.BDatt));
  HG_TRY(launch("hgt_transpose", hgt_transpose<T>, dim3(grid_of((int64_t)m.num_types * dd)), dim3(256), 0, s,
                (const T*)p->W_K, m.num_types, D, (T*)H.WKt));
  HG_TRY(launch("hgt_transpose", hgt_transpose<T>, dim3(grid_of((int64_t)m.num_types * dd)), dim3(256), 0, s,
                (const T*)p->W_V, m.num_types, D, (T*)H.WVt));
  HG_TRY(launch("hgt_transpose", hgt_transpose<T>, dim3(grid_of((int64_t)m.num_types * dd)), dim3(256), 0, s,
                (const T*)p->W_Q, m.num_types, D, (T*)H.WQt));
  // dQ = sum_r c_r dQ'_r blockdiag(W_att[r]) per target type, added at each stored row's node
  if (N > 0) HG_CUDA(cudaMemsetAsync(H.dQ, 0, (size_t)N * D * sizeof(T), s));
  for (int r = 0; r < m.num_rels; ++r) {
    const int t = m.rel_dst[r];
    const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
    HG_TRY((gemm<T, D>(H.dQp, D, (const T*)H.BDatt + r * dd, nullptr, D, n, (T*)H.dQ + off * D, D, 0, 1, s,
                       p->mu + r, rs, rel_rows(g, r, true))));
  }
  // dH_in = dY + dK W_K^T + dV W_V^T + dQ W_Q^T
  if (dH_in) {
    HG_CUDA(cudaMemcpyAsync(dH_in, H.L.dY, (size_t)N * D * sizeof(T), cudaMemcpyDeviceToDevice, s));
    T* dH = (T*)dH_in;
    for (int t = 0; t < m.num_types; ++t) {
      const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
      HG_TRY((gemm<T, D>((const T*)H.dK + off * D, D, (const T*)H.WKt + t * dd, nullptr, D, n, dH + off * D, D, 0, 1,
                         s)));
      HG_TRY((gemm<T, D>((const T*)H.dV + off * D, D, (const T*)H.WVt + t * dd, nullptr, D, n, dH + off * D, D, 0, 1,
                         s)));
      HG_TRY((gemm<T, D>((const T*)H.dQ + off * D, D, (const T*)H.WQt + t * dd, nullptr, D, n, dH + off * D, D, 0, 1,
                         s)));
    }
  }
  // weight gradients of the three typed maps: dW = H^T dZ, db = column sums of dZ; Q recomputed for
  // the attention matrices' gradients
  for (int t = 0; t < m.num_types; ++t) {
    const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
    HG_TRY(wgrad(kDt, D, H_in, off, H.dK, off, n, gr->dW_K + t * dd, H.L, s));
    HG_TRY(wgrad(kDt, D, H_in, off, H.dV, off, n, gr->dW_V + t * dd, H.L, s));
    HG_TRY((colsum<T, D>((const T*)H.dK + off * D, n, H.cs, gr->db_K + (size_t)t * D, H.L.rtmp, s)));
    HG_TRY((colsum<T, D>((const T*)H.dV + off * D, n, H.cs, gr->db_V + (size_t)t * D, H.L.rtmp, s)));
    HG_TRY(wgrad(kDt, D, H_in, off, H.dQ, off, n, gr->dW_Q + t * dd, H.L, s));
    HG_TRY((colsum<T, D>((const T*)H.dQ + off * D, n, H.cs, gr->db_Q + (size_t)t * D, H.L.rtmp, s)));
    HG_TRY((gemm<T, D>(Hin + off * D, D, (const T*)p->W_Q + t * dd, (const T*)p->b_Q + (size_t)t * D, D, n,
                       (T*)H.Qbuf + off * D, D, 0, 0, s)));
  }
  for (int r = 0; r < m.num_rels; ++r) {  // Gq[r] = dQ'_r^T Q over the stored rows
    const int t = m.rel_dst[r];
    const int64_t off = m.type_off[t], n = m.type_off[t + 1] - off;
    float* out = H.Gq + r * dd;
    if (kDt == HG_BF16) {
      HG_TRY(tc_weight_grad_rows(D, H.dQp, g->csr_rows, g->mlist, g->mbase, r, m.row_base[r], H.Qbuf, off, n,
                                 H.L.wpart, out, H.L.rtmp, s));
    } else if (n > 0) {
      HG_TRY(weight_grad(kDt, D, H.dQp, 0, H.Qbuf, off, n, H.L.wpart, out, H.L.rtmp, s, rel_rows(g, r, false)));
    } else {
      HG_CUDA(cudaMemsetAsync(out, 0, sizeof(float) * dd, s));
    }
  }
  return launch("hgt_finish", hgt_finish<T>, dim3(m.num_rels), dim3(256), 0, s, (const float*)H.Gw,
                (const float*)H.Gq, (const T*)p->W_att, p->mu, D, S, gr->dW_msg, gr->dW_att, gr->dmu);
}

#define HG_HGT_DISPATCH(dtype, d, FN, ...)                                                  \
  do {                                                                                      \
    if (dtype == HG_F32) {                                                                  \
      if (d == 64) return FN<float, 64>(__VA_ARGS__);                                       \
      if (d == 128) return FN<float, 128>(__VA_ARGS__);                                     \
      if (d == 256) return FN<float, 256>(__VA_ARGS__);                                     \
    } else {                                                                                \
      if (d == 64) return FN<__nv_bfloat16, 64>(__VA_ARGS__);                               \
      if (d == 128) return FN<__nv_bfloat16, 128>(__VA_ARGS__);                             \
      if (d == 256) return FN<__nv_bfloat16, 256>(__VA_ARGS__);                             \
    }                                                                                       \
    set_error("unsupported feature width %d", d);                                           \
    return HG_ERR_UNSUPPORTED;                                                              \
  } while (0)

hg_status check_hgt(const hg_graph* g, const hg_hgt_params* p) {
  HG_REQUIRE(g && p, "graph and params must be non-null");
  if (!(p->d == 64 || p->d == 128 || p->d == 256) || !(p->dtype == HG_F32 || p->dtype == HG_BF16)) {
    set_error("unsupported d=%d / dtype=%d", p->d, (int)p->dtype);
    return HG_ERR_UNSUPPORTED;
  }
  HG_REQUIRE(p->heads >= 1 && p->heads <= 32 && (p->heads & (p->heads - 1)) == 0,
             "heads must be a power of two in [1, 32]");
  HG_REQUIRE(p->act == HG_ACT_RELU || p->act == HG_ACT_GELU_TANH || p->act == HG_ACT_NONE, "unknown activation");
  HG_REQUIRE(p->W_K && p->W_Q && p->W_V && p->b_K && p->b_Q && p->b_V && p->W_att && p->W_msg && p->mu && p->W_agg &&
                 p->b_agg,
             "every parameter pointer must be non-null");
  HG_REQUIRE(!p->layernorm || (p->ln_gamma && p->ln_beta && p->ln_eps > 0.f), "layernorm needs gamma, beta, eps > 0");
  return HG_OK;
}

hg_status check_buf256(const void* q, const char* name) {
  HG_REQUIRE(q != nullptr, "%s must be non-null", name);
  HG_REQUIRE(((uintptr_t)q & 255) == 0, "%s must be 256-byte aligned", name);
  return HG_OK;
}

}  // namespace
}  // namespace hg

using namespace hg;

extern "C" hg_status hg_hgt_workspace_size(const hg_graph* graph, const hg_hgt_params* params, size_t* saved_bytes,
                                          size_t* scratch_bytes) {
  clear_error();
  HG_TRY(check_hgt(graph, params));
  HG_REQUIRE(saved_bytes && scratch_bytes, "saved_bytes and scratch_bytes must be non-null");
  HgtLayout H;
  carve_hgt(graph, params, nullptr, nullptr, &H, saved_bytes, scratch_bytes);
  return HG_OK;
}

extern "C" hg_status hg_hgt_fwd(const hg_graph* graph, const hg_hgt_params* params, const void* H_in, void* H_out,
                               void* saved, void* scratch, hg_stream stream) {
  clear_error();
  HG_TRY(device_guard());
  HG_TRY(check_hgt(graph, params));
  HG_TRY(check_buf256(H_in, "H_in"));
  HG_TRY(check_buf256(H_out, "H_out"));
  HG_TRY(check_buf256(saved, "saved"));
  HG_TRY(check_buf256(scratch, "scratch"));
  HG_REQUIRE(H_in != H_out, "H_in and H_out must not alias");
  HgtLayout H;
  carve_hgt(graph, params, saved, scratch, &H, nullptr, nullptr);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  HG_HGT_DISPATCH(params->dtype, params->d, hgt_fwd_t, graph, params, H_in, H_out, H, s);
}

extern "C" hg_status hg_hgt_bwd(const hg_graph* graph, const hg_hgt_params* params, const void* H_in,
                               const void* saved, const void* dH_out, void* dH_in, const hg_hgt_grads* grads,
                               void* scratch, hg_stream stream) {
  clear_error();
  HG_TRY(device_guard());
  HG_TRY(check_hgt(graph, params));
  HG_TRY(check_buf256(H_in, "H_in"));
  HG_TRY(check_buf256(saved, "saved"));
  HG_TRY(check_buf256(dH_out, "dH_out"));
  HG_TRY(check_buf256(scratch, "scratch"));
  HG_REQUIRE(dH_in == nullptr || ((uintptr_t)dH_in & 255) == 0, "dH_in must be 256-byte aligned");
  HG_REQUIRE(dH_in != dH_out, "dH_in and dH_out must not alias");
  HG_REQUIRE(grads && grads->dW_K && grads->dW_Q && grads->dW_V && grads->db_K && grads->db_Q && grads->db_V &&
                 grads->dW_att && grads->dW_msg && grads->dmu && grads->dW_agg && grads->db_agg,
             "every gradient pointer must be non-null");
  HG_REQUIRE(!params->layernorm || (grads->dln_gamma && grads->dln_beta), "layernorm needs dln_gamma and dln_beta");
  HgtLayout H;
  carve_hgt(graph, params, const_cast<void*>(saved), scratch, &H, nullptr, nullptr);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  HG_HGT_DISPATCH(params->dtype, params->d, hgt_bwd_t, graph, params, H_in, dH_out, dH_in, grads, H, s);
}
