// ivhd_knn_tc.cu -- kNN graph build (the set-up step of Sec. 5.1) on the
// 5th-generation tensor cores: a distance GEMM with the top-k selection fused
// into its epilogue.
//
// Squared distances come from the Gram matrix, |x_i - x_j|^2 = n_i + n_j - 2 <x_i, x_j>.
//
// uint8 data: the GEMM runs on x - 128 in BF16.  Every value in [-128, 127]
//   is exact in BF16, every product (at most 2^14) is exact in FP32, and with
//   N <= 1024 every partial sum stays below 2^24, so the tensor cores return
//   <x_i, x_j> exactly whatever their summation order; with the norms of the
//   shifted rows (exact int32) the distances are the exact integers and the
//   fused top-k (ties to the lower index) is final.
// FP32 data: x = hi + lo + r with hi = bf16(x), lo = bf16(x - hi) and
//   |r| <= 2^-16 |x|; the GEMM over K = 3N of [hi, hi, lo] . [hi, lo, hi] gives
//   <x_i, x_j> to about 2^-14 of sum_d |x_id x_jd|, so the approximate
//   distance dt_ij is within eps (n_i + n_j) of the exact FP32-chain distance,
//   eps = 2^-13 + N 2^-19 (the split, the FP32 accumulation of 3N products and
//   the chain's own rounding, with a margin of several times).  The epilogue
//   keeps, per row, the kList smallest keys kappa_j = dt_ij - eps n_j, each a
//   lower bound of d_ij + eps n_i.  A re-rank pass recomputes the listed
//   distances with the FP32 chain of the exact kernel, keeps the k best (ties to
//   the lower index) and certifies the row: every vertex outside the list has
//   kappa_j >= tau (the list's largest key), hence d_ij >= tau - eps n_i, so
//   the row is final when its exact k-th distance is below tau - eps n_i.
//   Other rows are recomputed by the exact CUDA-core kernel.
//
// Query rows are the rows of X itself for the kNN graph (a row never lists
// itself), or a separate set of new points searched against X as the base set
// (the nearest-neighbour placement of Progressive UMAP, Sec. 2.4.3); the
// arithmetic and the certificate are the same, with n_i the query's norm.
//
// A pair of CTAs (a cluster of two, cta_group::2) owns 256 query rows, 128
// tensor-memory lanes each, and sweeps all candidates in tiles of 256 columns:
//   warps 0, 10        TMA producers: this CTA's 128 x 64 query slice, and its
//                      half (128 x 64) of the candidate slice, into a 6-stage
//                      ring (128-byte swizzle); 32 KB from L2 per 512 clocks of
//                      MMAs instead of 48 KB with a tile per CTA (one warp's
//                      copies reach about 50 bytes per clock, two warps' 93)
//   warp 1             (rank 0) MMA issuer: tcgen05.mma M=256 N=256 K=16 into one
//                      of two 256-column accumulators in tensor memory, so the
//                      epilogue of tile t overlaps the MMAs of tile t+1
//   warps 2-9          epilogue: thread = query row; tcgen05.ld of 16 columns at
//                      a time, distance, test against the row's threshold, a
//                      queue in shared memory and a list in registers
// Every wait is bounded; a timeout sets an error flag and all roles stop.
// What bounds it: float, handling the candidates that pass (with one producer,
// M = 100,000 x 100, K = 320: 3.6 ms with the epilogue doing nothing, 3.7 ms
// with its tests but no candidate passing, 5 ms in all); uint8, the MMAs.
#include <climits>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "ivhd_internal.cuh"
#include "ivhd_knn_tc.cuh"
#include "ivhd_tc.cuh"

namespace ivhd {
namespace {

using namespace tc;

constexpr int kTM = 128;  // query rows per CTA (two CTAs share a 256-row tile)
constexpr int kTN = 256;  // candidate columns per accumulator tile, half of them loaded by each CTA
constexpr int kTStages = 6;
constexpr int kEpiWarps = 8;  // two warpgroups: each reads one 128-column half of a tile
constexpr int kTcThreads = 32 * (3 + kEpiWarps);
constexpr int kMaxKnnSegments = 32;  // column segments of one kNN launch (short query sets)
constexpr int kGroup = 8;            // columns tested and queued together in the epilogue
constexpr int kChunk = 16;           // columns read from tensor memory at once
constexpr int kQueue = 14;           // candidates a row holds back before its list takes them

struct KnnSmem {
  static constexpr int a_bytes = kTM * kBK * 2;
  static constexpr int b_bytes = kTN / 2 * kBK * 2;
  static constexpr int stage_bytes = a_bytes + b_bytes;
  static constexpr int bar_offset = kTStages * stage_bytes;
  static constexpr int nrm_offset = bar_offset + 256;  // 8 warps x 128 column terms
  static constexpr int queue_offset = nrm_offset + kEpiWarps * (kTN / 2) * 4;
  static constexpr int total = queue_offset + kQueue * 32 * kEpiWarps * 8 + 1024;  // + slack
};

template <class D>
__device__ __forceinline__ bool better(D d, int j, D bd, int bj) {
  return d < bd || (d == bd && j < bj);
}

// Inserts (d, j) into the ascending list (dl, jl) of L entries, dropping the
// last.  Candidates arrive in increasing j, so an equal key goes behind the
// ones already listed (the lower index wins the tie) and "<" is the order.
// Every entry looks at its left neighbour only: no chain of dependent selects.
template <class D, int L>
__device__ __forceinline__ void list_insert(D d, int j, D (&dl)[L], int (&jl)[L]) {
#pragma unroll
  for (int q = L - 1; q > 0; --q) {
    const bool here = d < dl[q], left = d < dl[q - 1];
    dl[q] = left ? dl[q - 1] : (here ? d : dl[q]);
    jl[q] = left ? jl[q - 1] : (here ? j : jl[q]);
  }
  if (d < dl[0]) {
    dl[0] = d;
    jl[0] = j;
  }
}

// Floats as integers of the same order, and back.
__device__ __forceinline__ int ordered_int(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float ordered_float(int i) {
  return __int_as_float(i ^ ((i >> 31) & 0x7fffffff));
}

// Twice the certificate's bound over a row's distances: a vertex whose key is
// above the k-th smallest key by this much or more is not among the k nearest
// (d_k <= kappa_k + 2 eps max n_j + eps n_i, and d_j >= kappa_j - eps n_i).
__device__ __forceinline__ float key_slack(float eps_coef, float ni, float n_max) {
  return 2.f * eps_coef * (ni + n_max);
}

// U8: exact integer keys; L: list length (kKnnList for float, 8 or kKnnList for uint8).
template <bool U8, int L>
__global__ void __launch_bounds__(kTcThreads, 1)
    k_knn_tc(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
             const float* __restrict__ nrm_f, const int32_t* __restrict__ nrm_i,
             const float* __restrict__ qnrm_f, const int32_t* __restrict__ qnrm_i, int Mq, int M,
             int Kp, bool self, int k, int seg_tiles, float eps_coef,
             int32_t* __restrict__ bounds, int32_t* __restrict__ out_ids,
             float* __restrict__ out_d, int32_t* __restrict__ err) {
  using D = typename std::conditional<U8, int32_t, float>::type;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + KnnSmem::bar_offset);
  uint64_t* empty = full + kTStages;
  uint64_t* acc_full = empty + kTStages;  // [2]
  uint64_t* acc_empty = acc_full + 2;     // [2]
  uint64_t* done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kCols = 2 * kTN;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();  // 0: the CTA that issues the MMAs of the pair
  const int m0 = blockIdx.x * kTM;
  const int nk = Kp / kBK;
  // this CTA's column segment: tiles t0 .. t0 + n_tiles - 1 (blockIdx.y of gridDim.y)
  const int all_tiles = (M + kTN - 1) / kTN;
  const int t0 = (int)blockIdx.y * seg_tiles;
  const int n_tiles = max(0, min(all_tiles - t0, seg_tiles));

  if (threadIdx.x == 0) {
    for (int s = 0; s < kTStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kEpiWarps);  // every epilogue warp of both CTAs arrives
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  pair_sync();  // both CTAs' barriers are set up before either signals the other's
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 || warp == 2 + kEpiWarps) {
    // producers: this CTA's query slice (re-read from L2 for every tile), and its
    // half of the candidate slice; the bytes of both CTAs are counted by the
    // barrier of rank 0
    const bool second = warp != 0;
    const uint32_t full0 = pair_addr(full, 0);
    int s = 0;
    uint32_t lap = 0;
    bool ok = true;
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int y = second ? (t0 + t) * kTN + (int)rank * (kTN / 2) : m0;
      for (int kt = 0; kt < nk; ++kt) {
        if (lap > 0) ok = __all_sync(0xffffffffu, pair_wait(&empty[s], (lap - 1) & 1, abort_flag));
        if (!ok) break;
        if (elect_one()) {
          if (rank == 0 && !second) mbar_expect_tx(&full[s], 2 * KnnSmem::stage_bytes);
          tma_load_2d_pair(smem + s * KnnSmem::stage_bytes + (second ? KnnSmem::a_bytes : 0),
                           second ? &map_b : &map_a, kt * kBK, y, full0 + (uint32_t)s * 8u);
        }
        if (++s == kTStages) {
          s = 0;
          ++lap;
        }
      }
    }
    if (!ok) {
      if (lane == 0) atomicOr(err, 1);
      // a copy in flight lands within microseconds: after an abort, time for
      // it before the shared memory goes away
      for (int it = 0; it < 2000; ++it) __nanosleep(1000);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(2 * kTM, kTN);
      const uint64_t desc = smem_desc_sw128(smem_u32(smem));
      int s = 0;
      uint32_t lap = 0;
      bool ok = true;
      auto wait = [&](uint64_t* bar, uint32_t parity, int code) {
        ok = __all_sync(0xffffffffu, pair_wait(bar, parity, abort_flag));
        if (!ok && lane == 0) atomicOr(err, code);
        asm volatile("tcgen05.fence::after_thread_sync;");
        return ok;
      };
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int b = t & 1;
        if (t >= 2 && !wait(&acc_empty[b], ((t >> 1) - 1) & 1, 2)) break;
        const uint32_t dst = tmem + (uint32_t)(b * kTN);
        for (int kt = 0; kt < nk; ++kt) {
          if (!wait(&full[s], lap & 1, 4)) break;
          if (elect_one()) {
            const uint64_t a = desc + (uint64_t)(s * (KnnSmem::stage_bytes >> 4));
            umma_slab_pair(dst, a, a + (KnnSmem::a_bytes >> 4), idesc, kt == 0, kBK / 16);
            umma_commit_pair(&empty[s]);
            if (kt + 1 == nk) umma_commit_pair(&acc_full[b]);
          }
          __syncwarp();
          if (++s == kTStages) {
            s = 0;
            ++lap;
          }
        }
      }
      // every MMA issued above has finished before tensor memory is released
      // and either CTA's shared memory goes away
      if (elect_one()) umma_commit_pair(done);
      if (!mbar_wait(done, 0) && lane == 0) atomicOr(err, 8);
    }
  } else {
    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. 32 (w % 4) + 31
    // (its row quarter) of one 128-column half of each tile: warps 2-5 the
    // first half, warps 6-9 the second, so every row has one list per half.
    // Keys: uint8, the exact distance; float, the lower-bound key
    // kappa_j = dt_j - eps n_j = n_i + (1 - eps) n_j - 2 <x_i, x_j>~ (see the
    // top); both without n_i, which every key of a row shares, until the end.
    //
    // A column is one FMA and one minimum; eight columns share one test against
    // the row's threshold.  What passes is queued in shared memory (a store per
    // candidate, whatever the other rows do) and goes to the lists when some row
    // of the warp has a full queue, all rows together: inserting each candidate
    // at once made the whole warp walk one row's list, and that, not the tensor
    // cores, set the time (whole build, 300,000 x 100 floats, k = 5: 70.4 -> 44.2 ms
    // with queues, 42.7 with appends that do not branch, loads that run ahead and
    // shared bounds, 38.8 with the second producer; 70,000 x 784 bytes 6.00 ->
    // 5.59 -> 5.01 -> 4.44 ms; 38.4 and 4.24 since the operands are prepared in
    // one pass).
    // uint8: the float key and the float threshold are within 2 of the exact
    // integers (magnitudes below 2^26), so the test allows 16 and the queue takes
    // the exact keys.
    constexpr int kHalf = kTN / 2;
    const int quarter = warp & 3;
    const int half = (warp - 2) >> 2;
    const int r = quarter * 32 + lane;
    const int i = m0 + r;
    // the half-tile's 128 column terms, staged per warp; each lane prefetches
    // its 4 terms of the next tile into registers while the current one is processed
    const uint32_t nbuf = smem_u32(smem + KnnSmem::nrm_offset) + (uint32_t)(warp - 2) * kHalf * 4;
    constexpr int kPer = kHalf / 32;
    constexpr int kQueueStride = 32 * kEpiWarps * 8;  // bytes from one entry of a row to the next
    const uint32_t queue = smem_u32(smem + KnnSmem::queue_offset) + ((warp - 2) * 32 + lane) * 8;
    const D kMaxKey = U8 ? (D)INT_MAX : (D)__int_as_float(0x7f800000);
    const float kInf = __int_as_float(0x7f800000);
    const float col_scale = 1.f - eps_coef;
    const bool has_row = i < Mq;
    int shared_bound = INT_MAX;  // bounds[i] as of the last fetch
    float pn[kPer];
    auto fetch = [&](int t) {
#pragma unroll
      for (int e = 0; e < kPer; ++e) {
        const int jc = (t0 + t) * kTN + half * kHalf + e * 32 + lane;
        if constexpr (U8)
          pn[e] = (jc < M) ? (float)nrm_i[jc] : 0.f;  // at most 2^24: exact
        else
          pn[e] = (jc < M) ? col_scale * nrm_f[jc] : 0.f;
      }
      if (has_row) shared_bound = *reinterpret_cast<volatile int32_t*>(bounds + i);
    };
    D dl[L];
    int jl[L];
#pragma unroll
    for (int q = 0; q < L; ++q) {
      dl[q] = kMaxKey;
      jl[q] = INT_MAX;
    }
    const D ni = (i < Mq) ? (U8 ? (D)qnrm_i[i] : (D)qnrm_f[i]) : (D)0;
    const int iself = self ? i : -1;  // the column a row never lists (self-kNN only)
    // A candidate is of use only below the list's last key, and below the k-th
    // key (uint8) or, float, the k-th key plus what separates its distance's
    // upper bound from a lower bound: slack = 2 eps (n_i + max n_j).
    const float slack = U8 ? 0.f : key_slack(eps_coef, (float)ni, nrm_f[M]);
    // The row's lists (the other half's, and those of the other column segments)
    // share the smallest of their bounds: together they let pass about as much
    // as one list would, and a segment that starts late starts with a bound.
    // (uint8: a key equal to another list's k-th may have the lower index, so
    // only larger ones are dropped.)
    D thr = kMaxKey;
    float thr_f = kInf;
    auto tighten = [&](D t) {
      thr = min(thr, t);
      thr_f = U8 ? (thr == (D)INT_MAX ? kInf : (float)thr + 16.f) : (float)thr;
    };
    uint32_t qa = queue;         // end of the row's queue
    auto flush = [&]() {
      const int held = (int)(qa - queue) / kQueueStride;
      const int most = __reduce_max_sync(0xffffffffu, held);
      for (int q = 0; q < most; ++q) {
        D d = kMaxKey;
        int j = INT_MAX;
        if (q < held) {
          const int2 e = ld_shared_i2(queue + q * kQueueStride);
          d = U8 ? (D)e.x : (D)__int_as_float(e.x);
          j = e.y;
        }
        list_insert<D, L>(d, j, dl, jl);
      }
      qa = queue;
      D dk = dl[L - 1];  // the k-th key: the smallest from there on
#pragma unroll
      for (int q = 0; q < L; ++q)
        if (q >= k - 1) dk = min(dk, dl[q]);
      if constexpr (U8) {
        if (has_row && dk != INT_MAX) atomicMin(bounds + i, dk + 1);
        tighten(dk);
      } else {
        if (has_row && dk < kInf) atomicMin(bounds + i, ordered_int(dk + slack));
        tighten(fminf(dl[L - 1], dk + slack));
      }
    };
    // kChunk columns from c0 of this half tile, which starts at column n0
    auto process = [&](const uint32_t(&v)[kChunk], int n0, int c0) {
      const int jb = n0 + c0;
      if (jb >= M) return;
      float d[kChunk];
#pragma unroll
      for (int q = 0; q < kChunk; q += 4) {
        const float4 w = ld_shared_f4(nbuf + (c0 + q) * 4);
        d[q + 0] = fmaf(-2.f, __uint_as_float(v[q + 0]), w.x);
        d[q + 1] = fmaf(-2.f, __uint_as_float(v[q + 1]), w.y);
        d[q + 2] = fmaf(-2.f, __uint_as_float(v[q + 2]), w.z);
        d[q + 3] = fmaf(-2.f, __uint_as_float(v[q + 3]), w.w);
      }
      if (jb + kChunk - 1 >= M || (jb <= iself && iself <= jb + kChunk - 1)) {
#pragma unroll
        for (int q = 0; q < kChunk; ++q)
          if (jb + q >= M || jb + q == iself) d[q] = kInf;
      }
      unsigned any[kChunk / kGroup];
#pragma unroll
      for (int g = 0; g < kChunk; g += kGroup) {
        const float a = fminf(fminf(d[g], d[g + 1]), fminf(d[g + 2], d[g + 3]));
        const float b = fminf(fminf(d[g + 4], d[g + 5]), fminf(d[g + 6], d[g + 7]));
        any[g / kGroup] = __ballot_sync(0xffffffffu, fminf(a, b) < thr_f);
      }
#pragma unroll
      for (int g = 0; g < kChunk; g += kGroup) {
        if (any[g / kGroup] == 0) continue;
        if constexpr (U8) {
#pragma unroll
          for (int q = 0; q < kGroup; q += 4) {
            const float4 w = ld_shared_f4(nbuf + (c0 + g + q) * 4);
            const float nj[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int key = (int)nj[u] - 2 * __float2int_rn(__uint_as_float(v[g + q + u]));
              append_shared<kQueueStride>(qa, d[g + q + u] < thr_f && key < thr, key, jb + g + q + u);
            }
          }
        } else {
#pragma unroll
          for (int q = 0; q < kGroup; ++q)
            append_shared<kQueueStride>(qa, d[g + q] < thr_f, __float_as_int(d[g + q]), jb + g + q);
        }
        if (__any_sync(0xffffffffu, qa > queue + (kQueue - kGroup) * kQueueStride)) flush();
      }
    };
    bool ok = true;
    fetch(0);
    for (int t = 0; t < n_tiles; ++t) {
      const int b = t & 1;
      if (!pair_wait(&acc_full[b], (t >> 1) & 1, abort_flag)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) {  // the warp stays together below
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      __syncwarp();
#pragma unroll
      for (int e = 0; e < kPer; ++e) st_shared_f32(nbuf + (e * 32 + lane) * 4, pn[e]);
      __syncwarp();
      tighten(U8 ? (D)shared_bound : (D)ordered_float(shared_bound));
      if (t + 1 < n_tiles) fetch(t + 1);
      const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * kTN + half * kHalf);
      const int n0 = (t0 + t) * kTN + half * kHalf;
      // the load of the next columns runs while the current ones are tested
      uint32_t va[kChunk], vb[kChunk];
      tmem_ld16_nowait(tbase, va);
#pragma unroll 1
      for (int c0 = 0; c0 < kHalf; c0 += 2 * kChunk) {
        tmem_wait_ld16(va);
        tmem_ld16_nowait(tbase + c0 + kChunk, vb);
        process(va, n0, c0);
        tmem_wait_ld16(vb);
        if (c0 + 2 * kChunk < kHalf) tmem_ld16_nowait(tbase + c0 + 2 * kChunk, va);
        process(vb, n0, c0 + kChunk);
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(pair_addr(&acc_empty[b], 0));
    }
    if (ok) flush();
    if (ok && i < Mq) {
      // the row's list for this segment and half:
      // out_ids / out_key [((i * segments + segment) * 2 + half) * L + q]
      const int64_t o = (((int64_t)i * gridDim.y + blockIdx.y) * 2 + half) * L;
#pragma unroll
      for (int q = 0; q < L; ++q) {
        out_ids[o + q] = jl[q];
        const D key = jl[q] == INT_MAX ? kMaxKey : dl[q] + ni;
        if constexpr (U8)
          reinterpret_cast<int32_t*>(out_d)[o + q] = key;
        else
          out_d[o + q] = key;
      }
    }
    if (!ok && lane == 0) atomicOr(err, 16);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  pair_sync();  // no MMA, copy or arrival of the pair is outstanding
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}

// ---- operand preparation ---------------------------------------------------

// Both kernels write a row's operands and its norm from one read of it, a warp
// per row over a resident grid.  uint8 is bound by the operands' stores, float by
// the FP64 sums (504 MB would take 74 us): 300,000 x 100 floats 476 -> 259 us (a thread per element, and a thread per row for the
// norms), 70,000 x 784 bytes 248 -> 33 us.
constexpr int kPrepWarps = 8;
inline unsigned prep_blocks(int64_t M, int sms) {
  const int64_t all = (M + kPrepWarps - 1) / kPrepWarps, resident = (int64_t)sms * 8;
  return (unsigned)(all < resident ? all : resident);
}

// FP32: A = [hi | hi | lo], B = [hi | lo | hi] along K (3N, zero-padded to Kp);
// either output may be null (queries fill A, the base set B).  Norms: an FP64 sum,
// rounded once; the largest goes to nrm[M], which starts at zero (norms are not
// negative, so their bits order as integers).
// V: features per access; 4 needs N % 4 == 0 and X on 16 bytes, then every part of
// an operand row starts on 8 (Kp is a multiple of 64).
template <int V>
__global__ void k_prep_f32(const float* __restrict__ X, int64_t M, int N, int Kp,
                           __nv_bfloat16* __restrict__ A, __nv_bfloat16* __restrict__ B,
                           float* __restrict__ nrm) {
  struct __align__(2 * V) Part {
    __nv_bfloat16 v[V];
  };
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * kPrepWarps;
  unsigned top = 0;
  for (int64_t i = (int64_t)blockIdx.x * kPrepWarps + (threadIdx.x >> 5); i < M; i += warps) {
    __nv_bfloat16* a = A ? A + i * Kp : nullptr;
    __nv_bfloat16* b = B ? B + i * Kp : nullptr;
    double sum = 0.0;
    for (int d = lane * V; d < N; d += 32 * V) {
      float x[V];
      if constexpr (V == 4) {
        const float4 w = *reinterpret_cast<const float4*>(X + i * N + d);
        x[0] = w.x, x[1] = w.y, x[2] = w.z, x[3] = w.w;
      } else {
        x[0] = X[i * N + d];
      }
      Part hi, lo;
#pragma unroll
      for (int u = 0; u < V; ++u) {
        hi.v[u] = __float2bfloat16_rn(x[u]);
        lo.v[u] = __float2bfloat16_rn(x[u] - __bfloat162float(hi.v[u]));
        sum += (double)x[u] * (double)x[u];
      }
      if (a) {
        *reinterpret_cast<Part*>(a + d) = hi;
        *reinterpret_cast<Part*>(a + N + d) = hi;
        *reinterpret_cast<Part*>(a + 2 * N + d) = lo;
      }
      if (b) {
        *reinterpret_cast<Part*>(b + d) = hi;
        *reinterpret_cast<Part*>(b + N + d) = lo;
        *reinterpret_cast<Part*>(b + 2 * N + d) = hi;
      }
    }
    for (int c = 3 * N + lane; c < Kp; c += 32) {
      if (a) a[c] = __float2bfloat16_rn(0.f);
      if (b) b[c] = __float2bfloat16_rn(0.f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float n = (float)sum;
    if (lane == 0) nrm[i] = n;
    top = max(top, __float_as_uint(n));
  }
  if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(nrm + M), top);
}

// uint8: A = B = x - 128 (zero-padded to Kp); norms of the shifted rows.
// Eight columns per lane and store; V: bytes per load (8 needs N % 8 == 0 and X on 8).
template <int V>
__global__ void k_prep_u8(const uint8_t* __restrict__ X, int64_t M, int N, int Kp,
                          __nv_bfloat16* __restrict__ A, int32_t* __restrict__ nrm) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * kPrepWarps;
  for (int64_t i = (int64_t)blockIdx.x * kPrepWarps + (threadIdx.x >> 5); i < M; i += warps) {
    const uint8_t* x = X + i * N;
    int32_t sum = 0;
    for (int c = lane * 8; c < Kp; c += 256) {
      uint8_t t[8];
      if constexpr (V == 8) {
        uint2 w = make_uint2(0x80808080u, 0x80808080u);  // 128: the shifted value is 0
        if (c < N) w = *reinterpret_cast<const uint2*>(x + c);
        memcpy(t, &w, 8);
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) t[u] = c + u < N ? x[c + u] : 128;
      }
      __nv_bfloat16 o[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int v = (int)t[u] - 128;
        o[u] = __float2bfloat16_rn((float)v);
        sum += v * v;
      }
      uint4 w;
      memcpy(&w, o, 16);
      *reinterpret_cast<uint4*>(A + i * Kp + c) = w;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) nrm[i] = sum;
  }
}

// ---- FP32 re-rank and certificate (warp per row, lane = candidate) --------

template <class D>
__device__ __forceinline__ void cas(D& d, int& j, int lane, int mask, bool up) {
  const D od = __shfl_xor_sync(0xffffffffu, d, mask);
  const int oj = __shfl_xor_sync(0xffffffffu, j, mask);
  const bool lower = (lane & mask) == 0;
  // the lower lane keeps the smaller pair when sorting up
  const bool mine_better = better(d, j, od, oj);
  const bool keep = (lower == up) ? mine_better : !mine_better;
  if (!keep) {
    d = od;
    j = oj;
  }
}

// Exact FP32-chain distance of rows i and j (the order of the exact kernel);
// vec: both rows start on 16 bytes (N % 4 == 0), four features per load.
__device__ __forceinline__ float chain_dist(const float* __restrict__ xi,
                                            const float* __restrict__ xj, int N, bool vec) {
  float acc = 0.f;
  if (vec) {
    const float4* a = reinterpret_cast<const float4*>(xi);
    const float4* b = reinterpret_cast<const float4*>(xj);
#pragma unroll 4
    for (int q = 0; q < N / 4; ++q) {
      const float4 u = a[q], w = b[q];
      float t = __fsub_rn(u.x, w.x);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(u.y, w.y);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(u.z, w.z);
      acc = __fmaf_rn(t, t, acc);
      t = __fsub_rn(u.w, w.w);
      acc = __fmaf_rn(t, t, acc);
    }
    return acc;
  }
#pragma unroll 4
  for (int q = 0; q < N; ++q) {
    const float diff = __fsub_rn(xi[q], xj[q]);
    acc = __fmaf_rn(diff, diff, acc);
  }
  return acc;
}

// Bitonic sort of one (d, j) pair per lane across the warp, ascending.  SORTED:
// lanes already in sorted runs of this length, every other one descending.
template <int SORTED = 1, class D>
__device__ __forceinline__ void warp_sort(D& d, int& j, int lane) {
#pragma unroll
  for (int kk = 2 * SORTED; kk <= 32; kk <<= 1)
#pragma unroll
    for (int m = kk >> 1; m > 0; m >>= 1) cas(d, j, lane, m, (lane & kk) == 0);
}

// The 32 smallest of a warp's sorted (d, j) and the sorted (dn, jn): the first
// against the second reversed is bitonic, and a bitonic merge sorts it.
template <class D>
__device__ __forceinline__ void warp_merge(D& d, int& j, D dn, int jn, int lane) {
  const D rd = __shfl_sync(0xffffffffu, dn, 31 - lane);
  const int rj = __shfl_sync(0xffffffffu, jn, 31 - lane);
  if (better(rd, rj, d, j)) {
    d = rd;
    j = rj;
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) cas(d, j, lane, m, true);
}

// Warp per row: the row's n_lists candidate lists (two half-tile lists per
// column segment, L candidates each) are merged into the 32 smallest keys, and
// those within the slack of the k-th key are re-ranked by the exact FP32 chain
// (about eight of 64 at k = 5; re-ranking all of them took 3.25 ms of the
// 300,000 x 100 build).  When more than 32 are within the slack, all
// candidates are re-ranked, 32 per pass.
// Certificate: what a list left out has kappa_j >= min(its largest key if it is
// full, its k-th key + slack), what was not re-ranked has kappa_j > the
// merged k-th key + slack; with tau the smallest of these, d_ij >= tau - eps n_i,
// so the row is final when its exact k-th distance is below that.
template <int L>
__global__ void k_rerank(const float* __restrict__ Q, int Mq, const float* __restrict__ X, int M,
                         int N, int k, int n_lists, const int32_t* __restrict__ cand,
                         const float* __restrict__ key, const float* __restrict__ qnrm,
                         const float* __restrict__ nrm, float eps_coef, int32_t* __restrict__ out,
                         int32_t* __restrict__ fb_rows, int32_t* __restrict__ n_fb,
                         int32_t* __restrict__ max_err_bits) {
  static_assert(L == 16 || L == 32, "lists of 16 or 32 entries");
  constexpr int kPer = 32 / L;  // lists per pass (lane = entry)
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= Mq) return;
  const float* xi = Q + i * N;
  const bool vec = N % 4 == 0 && ((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(X)) & 15) == 0;
  const float inf = __int_as_float(0x7f800000);
  const float slack = key_slack(eps_coef, qnrm[i], nrm[M]);
  // L = 32: pass p reads list p; L = 16: lanes 0-15 list 2p, lanes 16-31 list 2p + 1
  auto entry = [&](int pass) {
    return (i * n_lists + pass * kPer + ((L == 32) ? 0 : (lane >> 4))) * L + (lane & (L - 1));
  };
  auto listed = [&](int j) { return j >= 0 && j < M; };
  float rel = 0.f;
  auto exact = [&](int j, float kj) {
    const float dc = chain_dist(xi, X + (int64_t)j * N, N, vec);
    // the approximate distance is the key plus eps n_j
    rel = fmaxf(rel, fabsf(fmaf(eps_coef, nrm[j], kj) - dc) / fmaxf(qnrm[i] + nrm[j], 1e-30f));
    return dc;
  };
  float tau = inf;
  float kd = inf;  // the running 32 smallest keys, sorted across the lanes
  int kj = INT_MAX;
  for (int pass = 0; pass < n_lists / kPer; ++pass) {
    const int64_t o = entry(pass);
    int j0 = cand[o];
    float k0 = key[o];
#pragma unroll
    for (int hh = 0; hh < kPer; ++hh) {
      const int last = hh * L + L - 1, kth = hh * L + k - 1;
      const float klast = __shfl_sync(0xffffffffu, k0, last), kk = __shfl_sync(0xffffffffu, k0, kth);
      if (listed(__shfl_sync(0xffffffffu, j0, last))) tau = fminf(tau, klast);
      if (listed(__shfl_sync(0xffffffffu, j0, kth))) tau = fminf(tau, kk + slack);
    }
    if (!listed(j0)) {
      k0 = inf;
      j0 = INT_MAX;
    }
    warp_sort(k0, j0, lane);
    if (pass == 0) {
      kd = k0;
      kj = j0;
    } else {
      warp_merge(kd, kj, k0, j0, lane);
    }
  }
  const float bound = __shfl_sync(0xffffffffu, kd, k - 1) + slack;
  float d = inf;
  int j = INT_MAX;
  if (__shfl_sync(0xffffffffu, kd, 31) > bound || !listed(__shfl_sync(0xffffffffu, kj, 31))) {
    if (listed(kj) && !(kd > bound)) {
      d = exact(kj, kd);
      j = kj;
    }
    if (listed(__shfl_sync(0xffffffffu, kj, k - 1))) tau = fminf(tau, bound);
    warp_sort(d, j, lane);
  } else {
    for (int pass = 0; pass < n_lists / kPer; ++pass) {
      const int64_t o = entry(pass);
      const int j0 = cand[o];
      float dc = inf;
      int jc = INT_MAX;
      if (listed(j0)) {
        dc = exact(j0, key[o]);
        jc = j0;
      }
      warp_sort(dc, jc, lane);
      if (pass == 0) {
        d = dc;
        j = jc;
      } else {
        warp_merge(d, j, dc, jc, lane);
      }
    }
  }
  float mrel = rel;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mrel = fmaxf(mrel, __shfl_xor_sync(0xffffffffu, mrel, o));
  const float dk = __shfl_sync(0xffffffffu, d, k - 1);
  const bool certified = dk < tau - eps_coef * qnrm[i];
  if (certified) {
    if (lane < k) out[i * k + lane] = j;
  } else if (lane == 0) {
    fb_rows[atomicAdd(n_fb, 1)] = (int32_t)i;
  }
  if (lane == 0) atomicMax(max_err_bits, __float_as_int(mrel));
}

// uint8: the n_lists exact lists of each row (ascending by (distance, index))
// merged into the k <= 32 nearest: a warp per row, 32 / L lists per pass, every
// other one read backwards as the sort wants it; a pass without a candidate
// before the k-th so far is skipped (10,000 queries, 34 lists of 8: 41 -> 16 us;
// 70,000 rows, 6 lists: 26 -> 27; a thread per row left most of the chip idle).
template <int L>
__global__ void k_merge_u8(const int32_t* __restrict__ ids, const int32_t* __restrict__ keys,
                           int64_t M, int k, int n_lists, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31, n = n_lists * L;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= M) return;
  // (one list per pass, L = 32: ascending, nothing to sort)
  const int from = (L < 32 && (lane & L)) ? (lane ^ (L - 1)) : lane;
  int32_t d = INT_MAX, j = INT_MAX;
  for (int at0 = 0; at0 < n; at0 += 32) {
    int32_t dc = INT_MAX, jc = INT_MAX;
    if (at0 + from < n) {
      dc = keys[i * n + at0 + from];
      jc = ids[i * n + at0 + from];
    }
    if (at0 > 0) {
      const int32_t dk = __shfl_sync(0xffffffffu, d, k - 1);
      const int32_t jk = __shfl_sync(0xffffffffu, j, k - 1);
      if (!__any_sync(0xffffffffu, better(dc, jc, dk, jk))) continue;
    }
    warp_sort<L>(dc, jc, lane);
    if (at0 == 0) {
      d = dc;
      j = jc;
    } else {
      warp_merge(d, j, dc, jc, lane);
    }
  }
  if (lane < k) out[i * k + lane] = j;
}

template <bool U8, int L>
cudaError_t launch_tc(const CUtensorMap& ma, const CUtensorMap& mb, const float* nrm_f,
                      const int32_t* nrm_i, const float* qnrm_f, const int32_t* qnrm_i, int Mq,
                      int M, int Kp, bool self, int k, int segments, int seg_tiles, float eps_coef,
                      int32_t* bounds, int32_t* out_ids, float* out_d, int32_t* err,
                      cudaStream_t s) {
  // no bound yet: larger than any key, and as a float 3.4e38
  const cudaError_t e0 = cudaMemsetAsync(bounds, 0x7f, (size_t)Mq * sizeof(int32_t), s);
  if (e0 != cudaSuccess) return e0;
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_knn_tc<U8, L>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         KnnSmem::total);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (unsigned)((Mq + 2 * kTM - 1) / (2 * kTM)), (unsigned)segments);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = KnnSmem::total;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_knn_tc<U8, L>, ma, mb, nrm_f, nrm_i, qnrm_f, qnrm_i, Mq, M, Kp,
                            self, k, seg_tiles, eps_coef, bounds, out_ids, out_d, err);
}

}  // namespace

bool knn_tc_supported(const KnnProblem& P) {
  if (P.k < 1 || P.k > kKnnList || P.M < 2 || P.M > (1 << 30) || P.Mq < 1 || P.Mq > (1 << 30))
    return false;
  if (P.dtype == IVHD_KNN_U8) return P.N <= 1024;
  return (int64_t)3 * P.N <= 65536;
}

// Device scratch freed on scope exit (stream-ordered).
namespace {
struct Bufs {
  cudaStream_t s;
  void* p[12] = {};
  int n = 0;
  bool ok = true;
  explicit Bufs(cudaStream_t st) : s(st) {}
  template <class T>
  T* get(int64_t count) {
    void* q = nullptr;
    if (n == (int)(sizeof(p) / sizeof(p[0])) ||
        dev_alloc(&q, (size_t)(count > 0 ? count : 1) * sizeof(T), s) != cudaSuccess) {
      ok = false;
      return nullptr;
    }
    p[n++] = q;
    return (T*)q;
  }
  ~Bufs() {
    for (int q = 0; q < n; ++q) dev_free(p[q], s);
  }
};
}  // namespace

int knn_tc_kp(int32_t dtype, int32_t N) {
  const int64_t K = dtype == IVHD_KNN_U8 ? (int64_t)N : 3 * (int64_t)N;
  return (int)(((K + kBK - 1) / kBK) * kBK);
}

static int sm_count() {
  int sms = 0, dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess &&
                 cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess
             ? sms
             : 0;
}

// The M x Kp operands (either may be null), the M norms and, at nrm[M], the
// largest of them.
static cudaError_t prep_f32(const float* X, int64_t M, int N, __nv_bfloat16* A, __nv_bfloat16* B,
                            float* nrm, int sms, cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(nrm + M, 0, sizeof(float), s);
  if (e != cudaSuccess) return e;
  const int Kp = knn_tc_kp(IVHD_KNN_F32, N);
  const unsigned g = prep_blocks(M, sms);
  if (N % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0)
    k_prep_f32<4><<<g, 32 * kPrepWarps, 0, s>>>(X, M, N, Kp, A, B, nrm);
  else
    k_prep_f32<1><<<g, 32 * kPrepWarps, 0, s>>>(X, M, N, Kp, A, B, nrm);
  return cudaGetLastError();
}

static cudaError_t prep_u8(const uint8_t* X, int64_t M, int N, __nv_bfloat16* A, int32_t* nrm,
                           int sms, cudaStream_t s) {
  const int Kp = knn_tc_kp(IVHD_KNN_U8, N);
  const unsigned g = prep_blocks(M, sms);
  if (N % 8 == 0 && (reinterpret_cast<uintptr_t>(X) & 7) == 0)
    k_prep_u8<8><<<g, 32 * kPrepWarps, 0, s>>>(X, M, N, Kp, A, nrm);
  else
    k_prep_u8<1><<<g, 32 * kPrepWarps, 0, s>>>(X, M, N, Kp, A, nrm);
  return cudaGetLastError();
}

cudaError_t knn_tc_prepare_base(const void* X, int32_t dtype, int64_t M, int32_t N,
                                __nv_bfloat16* B, void* nrm, cudaStream_t s) {
  const int sms = sm_count();
  if (sms == 0) return cudaErrorInvalidDevice;
  if (dtype == IVHD_KNN_U8) return prep_u8((const uint8_t*)X, M, N, B, (int32_t*)nrm, sms, s);
  return prep_f32((const float*)X, M, N, nullptr, B, (float*)nrm, sms, s);
}

ivhd_status knn_tc_build(const KnnProblem& P, int32_t* out_knn, cudaStream_t s,
                         KnnTcStats* stats, const KnnBase* base) {
  const bool u8 = P.dtype == IVHD_KNN_U8;
  const int64_t M = P.M, Mq = P.Mq;
  const int N = P.N, k = P.k;
  const int Kp = knn_tc_kp(P.dtype, N);
  if (base && P.self) return IVHD_ERR_ARG;
  Bufs b(s);
  // A: the query rows' operand, B: the base rows' (prepared once in an index,
  // or here); one array when they coincide (uint8 self)
  __nv_bfloat16* B = base ? const_cast<__nv_bfloat16*>(base->B) : b.get<__nv_bfloat16>(M * Kp);
  __nv_bfloat16* A = (u8 && P.self) ? B : b.get<__nv_bfloat16>(Mq * Kp);
  int32_t* err = b.get<int32_t>(8);  // err, n_fb, max-err bits
  int32_t* bounds = b.get<int32_t>(Mq);
  if (!b.ok) return IVHD_ERR_OOM;
  cudaError_t e = cudaMemsetAsync(err, 0, 8 * sizeof(int32_t), s);
  int32_t* n_fb = err + 1;
  int32_t* maxerr_bits = err + 2;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, Mq, Kp, Kp, kTM) || !make_map(&mb, B, M, Kp, Kp, kTN / 2))
    return IVHD_ERR_CUDA;
  const float eps_coef = (float)(1.0 / 8192.0 + (double)N / 524288.0);
  // Short query sets: the columns are split into segments (one CTA per row
  // block and segment, one CTA per SM at a time), choosing the count that
  // minimises waves x (tiles per segment + a fixed cost of about two tiles per
  // CTA); a segment keeps at least 4 tiles of 256 columns.  Each segment
  // yields its own lists, merged per row afterwards.
  const int sms = sm_count();
  if (sms == 0) return IVHD_ERR_CUDA;
  const int64_t row_blocks = 2 * ((Mq + 2 * kTM - 1) / (2 * kTM));
  const int all_tiles = (int)((M + kTN - 1) / kTN);
  int want = 1;
  int64_t best_cost = INT64_MAX;
  for (int S = 1; S <= kMaxKnnSegments && (S == 1 || all_tiles / S >= 4); ++S) {
    const int64_t waves = (row_blocks * S + sms - 1) / sms;
    const int64_t cost = waves * ((all_tiles + S - 1) / S + 2);
    if (cost < best_cost) {
      best_cost = cost;
      want = S;
    }
  }
  const int seg_tiles = (all_tiles + want - 1) / want;
  const int segs = (all_tiles + seg_tiles - 1) / seg_tiles;  // every segment has tiles
  const int n_lists = 2 * segs;
  if (u8) {
    const int L = (k <= 8) ? 8 : kKnnList;
    int32_t* nrm = base ? (int32_t*)const_cast<void*>(base->nrm) : b.get<int32_t>(M);
    int32_t* qnrm = P.self ? nrm : b.get<int32_t>(Mq);
    int32_t* lids = b.get<int32_t>(Mq * n_lists * L);
    int32_t* lkeys = b.get<int32_t>(Mq * n_lists * L);
    if (!b.ok) return IVHD_ERR_OOM;
    if (e == cudaSuccess) {
      if (!base) e = prep_u8((const uint8_t*)P.X, M, N, B, nrm, sms, s);
      if (!P.self && e == cudaSuccess) e = prep_u8((const uint8_t*)P.Q, Mq, N, A, qnrm, sms, s);
    }
    if (e == cudaSuccess) {
      e = (L == 8) ? launch_tc<true, 8>(ma, mb, nullptr, nrm, nullptr, qnrm, (int)Mq, (int)M, Kp,
                                        P.self, k, segs, seg_tiles, 0.f, bounds, lids, (float*)lkeys, err,
                                        s)
                   : launch_tc<true, kKnnList>(ma, mb, nullptr, nrm, nullptr, qnrm, (int)Mq,
                                               (int)M, Kp, P.self, k, segs, seg_tiles, 0.f, bounds, lids,
                                               (float*)lkeys, err, s);
    }
    if (e == cudaSuccess) {
      const unsigned g8 = (unsigned)((Mq + 7) / 8);
      if (L == 8)
        k_merge_u8<8><<<g8, 256, 0, s>>>(lids, lkeys, Mq, k, n_lists, out_knn);
      else
        k_merge_u8<kKnnList><<<g8, 256, 0, s>>>(lids, lkeys, Mq, k, n_lists, out_knn);
      e = cudaGetLastError();
    }
  } else {
    float* nrm = base ? (float*)const_cast<void*>(base->nrm) : b.get<float>(M + 1);
    float* qnrm = P.self ? nrm : b.get<float>(Mq + 1);
    const int L = (k <= 8) ? 16 : kKnnList;  // candidates per row and half
    int32_t* cand = b.get<int32_t>(Mq * n_lists * L);
    float* cd = b.get<float>(Mq * n_lists * L);
    int32_t* fb = b.get<int32_t>(Mq);
    if (!b.ok) return IVHD_ERR_OOM;
    const float* X = (const float*)P.X;
    const float* Q = (const float*)P.Q;
    if (e == cudaSuccess) {
      if (P.self) {
        e = prep_f32(X, M, N, A, B, nrm, sms, s);
      } else {
        if (!base) e = prep_f32(X, M, N, nullptr, B, nrm, sms, s);
        if (e == cudaSuccess) e = prep_f32(Q, Mq, N, A, nullptr, qnrm, sms, s);
      }
    }
    if (e == cudaSuccess) {
      e = (L == 16) ? launch_tc<false, 16>(ma, mb, nrm, nullptr, qnrm, nullptr, (int)Mq, (int)M,
                                           Kp, P.self, k, segs, seg_tiles, eps_coef, bounds, cand, cd, err, s)
                    : launch_tc<false, kKnnList>(ma, mb, nrm, nullptr, qnrm, nullptr, (int)Mq,
                                                 (int)M, Kp, P.self, k, segs, seg_tiles, eps_coef,
                                                 bounds, cand, cd, err, s);
    }
    if (e == cudaSuccess) {
      const unsigned g8 = (unsigned)((Mq + 7) / 8);
      if (L == 16)
        k_rerank<16><<<g8, 256, 0, s>>>(Q, (int)Mq, X, (int)M, N, k, n_lists, cand, cd, qnrm,
                                        nrm, eps_coef, out_knn, fb, n_fb, maxerr_bits);
      else
        k_rerank<kKnnList><<<g8, 256, 0, s>>>(Q, (int)Mq, X, (int)M, N, k, n_lists, cand, cd,
                                              qnrm, nrm, eps_coef, out_knn, fb, n_fb,
                                              maxerr_bits);
      e = cudaGetLastError();
    }
    // rows without a certificate: the exact CUDA-core kernel on just those rows
    if (e == cudaSuccess) e = knn_exact_rows_f32(P, fb, n_fb, out_knn, s);
  }
  int32_t h[8] = {};
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, err, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return IVHD_ERR_CUDA;
  if (stats) {
    stats->fallback_rows = u8 ? 0 : h[1];
    float mre = 0.f;
    std::memcpy(&mre, &h[2], sizeof(mre));
    stats->max_rel_err = u8 ? 0.f : mre;
    stats->eps_coef = u8 ? 0.f : eps_coef;
  }
  return h[0] ? IVHD_ERR_TIMEOUT : IVHD_OK;
}

}  // namespace ivhd
