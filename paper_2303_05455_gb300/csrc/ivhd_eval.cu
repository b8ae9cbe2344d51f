// ivhd_eval.cu -- embedding quality on sampled rows (Sec. 4.1).
//
// Both criteria need the nearest embedded neighbours of a query point y_q,
// ascending by (FP32 squared distance dx*dx rounded, then fma(dy, dy, .);
// index).
//   Q_NX(k):  hits = |embedded kNN(q) ∩ input kNN row q|       (rank criteria)
//   cf_nn:    hits = #embedded neighbours with q's class label  (Eq. 4.4)
// Hits are integer-summed, so the result is exact and order independent.
// A sampled row id outside [0, M) is never dereferenced: it is counted in a
// second counter, and the call returns IVHD_ERR_INDEX.
//
// The points are 2-D, so a spatial index prunes almost all of the M distance
// evaluations of a query: the points are grouped by the cells of a grid in
// Z-order (count, scan, scatter), 32 consecutive points form a leaf and 32
// leaves a node, each with its bounding box.  A warp searches one query: its
// own leaf and its neighbours first, then every node and leaf whose box is
// not farther than the current kk-th neighbour.  The box distance goes
// through the same rounded operations as the point distances, each of which
// is monotone in |dx| and |dy|, so a box's value never exceeds that of a
// point inside it: pruning by ">" loses no neighbour and no tie, and the
// lists are those of the full scan, bit for bit.  70,000 points, all rows,
// k = 5 and cf_10: 9.86 ms for the two calls with the full scan (every thread
// evaluating all 4.9e9 pairs), 0.49 ms with the index.
//
// The full scan stays for what the index does not take: positions that are not
// finite (their distances have no order a box could bound) and sets for which
// its memory cannot be had.
#include "ivhd_internal.cuh"

namespace ivhd {
namespace {

constexpr int kEvalThreads = 128;
constexpr int kEvalTile = 2048;

template <bool kQnx>
__global__ void __launch_bounds__(kEvalThreads) k_lowd(const float2* __restrict__ Y, int64_t M,
                                                       const int64_t* __restrict__ rows,
                                                       int64_t nrows, int kk,
                                                       const int32_t* __restrict__ knn,
                                                       const int32_t* __restrict__ labels,
                                                       int32_t* __restrict__ out_lowd,
                                                       unsigned long long* __restrict__ hits,
                                                       unsigned long long* __restrict__ bad,
                                                       const uint32_t* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;  // the index answers this call
  extern __shared__ __align__(16) unsigned char smem[];
  float2* tile = reinterpret_cast<float2*>(smem);
  float* ld = reinterpret_cast<float*>(tile + kEvalTile) + threadIdx.x * kk;
  int* lj = reinterpret_cast<int*>(reinterpret_cast<float*>(tile + kEvalTile) + kEvalThreads * kk) +
            threadIdx.x * kk;
  const int64_t qi = (int64_t)blockIdx.x * kEvalThreads + threadIdx.x;
  const int64_t q = qi < nrows ? rows[qi] : 0;
  const bool in_range = q >= 0 && q < M;
  if (qi < nrows && !in_range) atomicAdd(bad, 1ull);
  const bool act = qi < nrows && in_range;
  const float2 yq = act ? Y[q] : make_float2(0.f, 0.f);
  int n = 0;
  float worst = INFINITY;
  for (int64_t t0 = 0; t0 < M; t0 += kEvalTile) {
    const int tn = (int)min((int64_t)kEvalTile, M - t0);
    __syncthreads();
    for (int e = threadIdx.x; e < tn; e += kEvalThreads) tile[e] = Y[t0 + e];
    __syncthreads();
    if (!act) continue;
    for (int e = 0; e < tn; ++e) {
      const float2 yj = tile[e];
      const float dx = __fsub_rn(yj.x, yq.x);
      const float dy = __fsub_rn(yj.y, yq.y);
      const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
      if (n == kk && !(d2 < worst)) continue;  // later candidates have larger ids
      const int j = (int)(t0 + e);
      if (j == q) continue;
      int pos = (n < kk) ? n : kk - 1;
      while (pos > 0 && (ld[pos - 1] > d2)) {
        ld[pos] = ld[pos - 1];
        lj[pos] = lj[pos - 1];
        --pos;
      }
      ld[pos] = d2;
      lj[pos] = j;
      if (n < kk) ++n;
      if (n == kk) worst = ld[kk - 1];
    }
  }
  if (!act) return;
  int h = 0;
  for (int s = 0; s < n; ++s) {
    const int j = lj[s];
    if (out_lowd) out_lowd[qi * kk + s] = j;
    if (kQnx) {
      for (int u = 0; u < kk; ++u)
        if (knn[q * kk + u] == j) {
          ++h;
          break;
        }
    } else {
      h += (labels[j] == labels[q]);
    }
  }
  atomicAdd(hits, (unsigned long long)h);
}

// ---- spatial index ----------------------------------------------------------

constexpr int kLeaf = 32;              // points per leaf (one warp load)
constexpr int kNode = 1024;            // points per node (32 leaves)
constexpr int kMaxCellBits = 10;       // at most 1,024 x 1,024 cells
constexpr int kCellTile = 4096;        // cells scanned per block
constexpr int kTreeWarps = 8;          // queries per block
constexpr int64_t kMaxIndexed = (int64_t)1 << 30;

// Scratch of one call.  head: [0..1] complements of the ordered minimum of x
// and y, [2..3] their ordered maximum, [4] non-zero when a position is not finite.
struct Index {
  uint32_t* head;
  int32_t* cells;   // counts, then exclusive offsets within each tile of cells
  int32_t* base;    // first position of every tile of cells
  int32_t* rank;    // arrival of each point in its cell, then its sorted position
  float4* pts;      // (x, y, id as bits, unused) in cell order; id -1 past the end
  float4* leaf;     // boxes (lo x, lo y, hi x, hi y)
  float4* node;
  int64_t M, nodes;
  int bits;
};

// Floats as unsigned integers of the same order.
__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__global__ void __launch_bounds__(256) k_eval_bounds(const float2* __restrict__ Y, Index I) {
  uint32_t v[4] = {0u, 0u, 0u, 0u};
  bool bad = false;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < I.M; i += (int64_t)gridDim.x * 256) {
    const float2 y = Y[i];
    bad |= !(isfinite(y.x) && isfinite(y.y));
    const uint32_t ox = ordered(y.x), oy = ordered(y.y);
    v[0] = max(v[0], ~ox);
    v[1] = max(v[1], ~oy);
    v[2] = max(v[2], ox);
    v[3] = max(v[3], oy);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = __reduce_max_sync(0xffffffffu, v[q]);
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicMax(I.head + q, v[q]);
    if (bad) atomicOr(I.head + 4, 1u);
  }
}

// Z-order cell of a point; any cell is a correct one (boxes are taken from the
// points), so the rounding here decides nothing.
__device__ __forceinline__ uint32_t cell_of(float2 y, const Index& I) {
  const float n = (float)(1 << I.bits);
  const float lx = unordered(~I.head[0]), ly = unordered(~I.head[1]);
  const float sx = n / (unordered(I.head[2]) - lx), sy = n / (unordered(I.head[3]) - ly);
  const int m = (1 << I.bits) - 1;
  uint32_t cx = (uint32_t)min(max((int)((y.x - lx) * sx), 0), m);
  uint32_t cy = (uint32_t)min(max((int)((y.y - ly) * sy), 0), m);
  uint32_t z = 0;
#pragma unroll
  for (int b = 0; b < kMaxCellBits; ++b)
    z |= ((cx >> b) & 1u) << (2 * b) | ((cy >> b) & 1u) << (2 * b + 1);
  return z;
}

__global__ void __launch_bounds__(256) k_eval_count(const float2* __restrict__ Y, Index I) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i < I.M) I.rank[i] = atomicAdd(I.cells + cell_of(Y[i], I), 1);
}

// Exclusive scan of n counts within tiles of kCellTile; the tiles' sums to `sums`.
__global__ void __launch_bounds__(1024) k_eval_scan(int32_t* __restrict__ a, int n,
                                                    int32_t* __restrict__ sums) {
  __shared__ int32_t wsum[32];
  const int at = blockIdx.x * kCellTile + (int)threadIdx.x * 4;
  int32_t v[4], tot = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[q] = at + q < n ? a[at + q] : 0;
    tot += v[q];
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  if (w == 0) {
    int32_t s = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    wsum[lane] = s;
  }
  __syncthreads();
  int32_t run = incl - tot + (w > 0 ? wsum[w - 1] : 0);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (at + q < n) a[at + q] = run;
    run += v[q];
  }
  if (threadIdx.x == 1023 && sums) sums[blockIdx.x] = wsum[31];
}

__global__ void __launch_bounds__(256) k_eval_scatter(const float2* __restrict__ Y, Index I) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= I.nodes * kNode) return;
  if (i >= I.M) {
    I.pts[i] = make_float4(0.f, 0.f, __int_as_float(-1), 0.f);
    return;
  }
  const float2 y = Y[i];
  const uint32_t c = cell_of(y, I);
  const int32_t p = I.base[c / kCellTile] + I.cells[c] + I.rank[i];
  I.rank[i] = p;
  I.pts[p] = make_float4(y.x, y.y, __int_as_float((int)i), 0.f);
}

__global__ void __launch_bounds__(kNode) k_eval_boxes(Index I) {
  __shared__ float4 sh[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float4 p = I.pts[(int64_t)blockIdx.x * kNode + threadIdx.x];
  const bool on = __float_as_int(p.z) >= 0;
  const float inf = __int_as_float(0x7f800000);
  float4 b = on ? make_float4(p.x, p.y, p.x, p.y) : make_float4(inf, inf, -inf, -inf);
  for (int level = 0; level < 2; ++level) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      b.x = fminf(b.x, __shfl_xor_sync(0xffffffffu, b.x, o));
      b.y = fminf(b.y, __shfl_xor_sync(0xffffffffu, b.y, o));
      b.z = fmaxf(b.z, __shfl_xor_sync(0xffffffffu, b.z, o));
      b.w = fmaxf(b.w, __shfl_xor_sync(0xffffffffu, b.w, o));
    }
    if (level == 1) break;
    if (lane == 0) {
      sh[w] = b;
      I.leaf[(int64_t)blockIdx.x * 32 + w] = b;
    }
    __syncthreads();
    if (w != 0) return;
    b = sh[lane];
  }
  if (lane == 0) I.node[blockIdx.x] = b;
}

__device__ __forceinline__ float box_d2(float4 b, float2 y) {
  const float dx = b.x > y.x ? __fsub_rn(b.x, y.x) : (y.x > b.z ? __fsub_rn(b.z, y.x) : 0.f);
  const float dy = b.y > y.y ? __fsub_rn(b.y, y.y) : (y.y > b.w ? __fsub_rn(b.w, y.y) : 0.f);
  return __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
}

// One warp per sampled row; the kk best (distance bits, id) keys ascend over
// the lanes and the R registers of each (kk <= 32 R).
template <bool kQnx, int R>
__global__ void __launch_bounds__(32 * kTreeWarps)
    k_eval_tree(Index I, const float2* __restrict__ Y, const int64_t* __restrict__ rows,
                int64_t nrows, int kk, const int32_t* __restrict__ knn,
                const int32_t* __restrict__ labels, int32_t* __restrict__ out_lowd,
                unsigned long long* __restrict__ hits, unsigned long long* __restrict__ bad) {
  if (I.head[4] != 0) return;  // positions that are not finite: the full scan answers
  __shared__ int block_hits;
  if (threadIdx.x == 0) block_hits = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t qi = (int64_t)blockIdx.x * kTreeWarps + (threadIdx.x >> 5);
  const int64_t q = qi < nrows ? rows[qi] : -1;
  if (qi < nrows && q >= 0 && q < I.M) {
    const float2 yq = Y[q];
    constexpr unsigned long long kNone = ~0ull;
    unsigned long long list[R];
#pragma unroll
    for (int r = 0; r < R; ++r) list[r] = kNone;
    unsigned long long worst = kNone;  // key of the kk-th best; its distance reads as NaN while open
    float wd = __uint_as_float(0xffffffffu);
    auto visit = [&](int64_t l) {
      const float4 p = I.pts[l * kLeaf + lane];
      const int j = __float_as_int(p.z);
      const float dx = __fsub_rn(p.x, yq.x), dy = __fsub_rn(p.y, yq.y);
      const float d2 = __fmaf_rn(dy, dy, __fmul_rn(dx, dx));
      const unsigned long long key =
          (j < 0 || j == (int)q) ? kNone
                                 : ((unsigned long long)__float_as_uint(d2) << 32) | (uint32_t)j;
      unsigned m = __ballot_sync(0xffffffffu, key < worst);
      while (m) {
        const unsigned long long x = __shfl_sync(0xffffffffu, key, __ffs((int)m) - 1);
        m &= m - 1;
        if (x >= worst) continue;
        // every element above x moves one place up, x takes the first such place
#pragma unroll
        for (int r = R - 1; r >= 0; --r) {
          unsigned long long prev = __shfl_up_sync(0xffffffffu, list[r], 1);
          const unsigned long long last = r > 0 ? __shfl_sync(0xffffffffu, list[r > 0 ? r - 1 : 0], 31) : 0ull;
          if (lane == 0) prev = last;
          if (list[r] > x) list[r] = prev > x ? prev : x;
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (r == (kk - 1) >> 5) worst = __shfl_sync(0xffffffffu, list[r], (kk - 1) & 31);
        wd = __uint_as_float((uint32_t)(worst >> 32));
      }
    };
    const int64_t leaves = I.nodes * 32;
    const int64_t own = I.rank[q] / kLeaf;
    const int64_t l0 = max(own - R, (int64_t)0), l1 = min(own + R, leaves - 1);
    for (int64_t l = l0; l <= l1; ++l) visit(l);
    for (int64_t s0 = 0; s0 < I.nodes; s0 += 32) {
      const bool in = s0 + lane < I.nodes;
      const float nb = in ? box_d2(I.node[s0 + lane], yq) : 0.f;
      unsigned mn = __ballot_sync(0xffffffffu, in && !(nb > wd));
      while (mn) {
        const int s = __ffs((int)mn) - 1;
        mn &= mn - 1;
        if (__shfl_sync(0xffffffffu, nb, s) > wd) continue;
        const int64_t l = (s0 + s) * 32 + lane;
        const float lb = box_d2(I.leaf[l], yq);
        unsigned ml = __ballot_sync(0xffffffffu, (l < l0 || l > l1) && !(lb > wd));
        while (ml) {
          const int t = __ffs((int)ml) - 1;
          ml &= ml - 1;
          if (!(__shfl_sync(0xffffffffu, lb, t) > wd)) visit((s0 + s) * 32 + t);
        }
      }
    }
    int h = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int s = r * 32 + lane;
      bool hit = false;
      if (s < kk) {
        const int j = (int)(uint32_t)list[r];
        if (out_lowd) out_lowd[qi * kk + s] = j;
        if (kQnx) {
          for (int u = 0; u < kk; ++u) hit |= knn[q * kk + u] == j;
        } else {
          hit = labels[j] == labels[q];
        }
      }
      h += __popc(__ballot_sync(0xffffffffu, hit));
    }
    if (lane == 0) atomicAdd(&block_hits, h);
  } else if (qi < nrows && lane == 0) {
    atomicAdd(bad, 1ull);
  }
  __syncthreads();
  if (threadIdx.x == 0 && block_hits) atomicAdd(hits, (unsigned long long)block_hits);
}

// Builds the index over Y in `mem` (index_bytes) and answers the rows with it.
// Cells: about four points each where the points are spread evenly.
int cell_bits(int64_t M) {
  int b = 1;
  while (b < kMaxCellBits && ((int64_t)4 << (2 * b)) < M) ++b;
  return b;
}
size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }
Index index_of(unsigned char* mem, int64_t M, size_t* bytes) {
  Index I{};
  I.M = M;
  I.nodes = (M + kNode - 1) / kNode;
  I.bits = cell_bits(M);
  const size_t cells = (size_t)1 << (2 * I.bits);
  size_t at = 0;
  auto take = [&](size_t n) {
    unsigned char* p = mem + at;
    at += align256(n);
    return p;
  };
  I.head = (uint32_t*)take(32);
  I.cells = (int32_t*)take(cells * 4);
  I.base = (int32_t*)take((cells / kCellTile + 1) * 4);
  I.rank = (int32_t*)take((size_t)M * 4);
  I.pts = (float4*)take((size_t)I.nodes * kNode * 16);
  I.leaf = (float4*)take((size_t)I.nodes * 32 * 16);
  I.node = (float4*)take((size_t)I.nodes * 16);
  *bytes = at;
  return I;
}

template <bool kQnx>
cudaError_t launch_tree(const Index& I, const float2* Y, const int64_t* rows, int64_t nrows, int kk,
                        const int32_t* knn, const int32_t* labels, int32_t* out_lowd,
                        unsigned long long* hits, cudaStream_t s) {
  const int cells = 1 << (2 * I.bits);
  const int tiles = (cells + kCellTile - 1) / kCellTile;
  cudaError_t e = cudaMemsetAsync(I.head, 0, 256 + (size_t)cells * 4, s);  // head, then the counts
  if (e != cudaSuccess) return e;
  const unsigned nb = (unsigned)((I.M + 255) / 256);
  k_eval_bounds<<<nb < 608 ? nb : 608, 256, 0, s>>>(Y, I);
  k_eval_count<<<nb, 256, 0, s>>>(Y, I);
  k_eval_scan<<<tiles, 1024, 0, s>>>(I.cells, cells, I.base);
  k_eval_scan<<<1, 1024, 0, s>>>(I.base, tiles, nullptr);
  k_eval_scatter<<<(unsigned)(I.nodes * (kNode / 256)), 256, 0, s>>>(Y, I);
  k_eval_boxes<<<(unsigned)I.nodes, kNode, 0, s>>>(I);
  const unsigned grid = (unsigned)((nrows + kTreeWarps - 1) / kTreeWarps);
  if (kk <= 32)
    k_eval_tree<kQnx, 1><<<grid, 32 * kTreeWarps, 0, s>>>(I, Y, rows, nrows, kk, knn, labels,
                                                          out_lowd, hits, hits + 1);
  else if (kk <= 64)
    k_eval_tree<kQnx, 2><<<grid, 32 * kTreeWarps, 0, s>>>(I, Y, rows, nrows, kk, knn, labels,
                                                          out_lowd, hits, hits + 1);
  else
    k_eval_tree<kQnx, 4><<<grid, 32 * kTreeWarps, 0, s>>>(I, Y, rows, nrows, kk, knn, labels,
                                                          out_lowd, hits, hits + 1);
  return cudaGetLastError();
}

template <bool kQnx>
ivhd_status run_lowd(const float* Y, int64_t M, const int32_t* knn, const int32_t* labels, int kk,
                     const int64_t* rows, int64_t nrows, int32_t* out_lowd, double* out,
                     void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const size_t sm = (size_t)kEvalTile * sizeof(float2) + (size_t)kEvalThreads * kk * 8;
  unsigned long long* hits_d = nullptr;  // [0] hits, [1] rows outside [0, M)
  cudaError_t e = dev_alloc((void**)&hits_d, 2 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return IVHD_ERR_OOM;
  e = cudaMemsetAsync(hits_d, 0, 2 * sizeof(unsigned long long), s);
  // the spatial index; without memory for it the full scan answers alone
  unsigned char* mem = nullptr;
  size_t bytes = 0;
  Index I{};
  if (e == cudaSuccess && M <= kMaxIndexed) {
    index_of(nullptr, M, &bytes);
    if (dev_alloc((void**)&mem, bytes, s) != cudaSuccess) {
      mem = nullptr;
      cudaGetLastError();
    }
  }
  if (e == cudaSuccess && mem) {
    I = index_of(mem, M, &bytes);
    e = launch_tree<kQnx>(I, (const float2*)Y, rows, nrows, kk, knn, labels, out_lowd, hits_d, s);
  }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_lowd<kQnx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess) {
    const unsigned grid = (unsigned)((nrows + kEvalThreads - 1) / kEvalThreads);
    k_lowd<kQnx><<<grid, kEvalThreads, sm, s>>>((const float2*)Y, M, rows, nrows, kk, knn, labels,
                                               out_lowd, hits_d, hits_d + 1,
                                               mem ? I.head + 4 : nullptr);
    e = cudaGetLastError();
  }
  dev_free(mem, s);
  unsigned long long hits[2] = {0, 0};
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hits, hits_d, sizeof(hits), cudaMemcpyDeviceToHost, s);
  dev_free(hits_d, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return IVHD_ERR_CUDA;
  if (hits[1] != 0) return IVHD_ERR_INDEX;
  *out = (double)hits[0] / ((double)kk * (double)nrows);
  return IVHD_OK;
}

}  // namespace
}  // namespace ivhd

using namespace ivhd;

extern "C" ivhd_status ivhd_eval_qnx(const float* Y, int64_t M, const int32_t* knn, int32_t k,
                                     const int64_t* rows, int64_t nrows, int32_t* out_lowd,
                                     double* out_q, void* stream) {
  if (!Y || !knn || !rows || !out_q || M < 2 || nrows < 1) return IVHD_ERR_ARG;
  if (k < 1 || (int64_t)k > M - 1 || k > 128) return IVHD_ERR_ARG;
  return run_lowd<true>(Y, M, knn, nullptr, k, rows, nrows, out_lowd, out_q, stream);
}

extern "C" ivhd_status ivhd_eval_cf(const float* Y, int64_t M, const int32_t* labels, int32_t nn,
                                    const int64_t* rows, int64_t nrows, double* out_cf,
                                    void* stream) {
  if (!Y || !labels || !rows || !out_cf || M < 2 || nrows < 1) return IVHD_ERR_ARG;
  if (nn < 1 || (int64_t)nn > M - 1 || nn > 128) return IVHD_ERR_ARG;
  return run_lowd<false>(Y, M, nullptr, labels, nn, rows, nrows, nullptr, out_cf, stream);
}
