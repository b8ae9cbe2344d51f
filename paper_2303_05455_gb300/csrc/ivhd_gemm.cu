// ivhd_gemm.cu -- BF16 x BF16 -> FP32 GEMM on the 5th-generation tensor cores.
//
//   C[m, n] = sum_k A[m, k] B[n, k]        (A: M x K, B: N x K, both row-major = K-major)
//
// with a fused epilogue (bias, GELU, GELU derivative, BF16 or FP32 output).  It
// carries the dense layers of the learned warm start (an MLP that maps features
// to 2-D positions, trained on IVHD embeddings).
//
// Persistent kernel, looping over 128 x BN output tiles, one CTA per SM (BN = 256,
// or 128 when that keeps more SMs busy or pads N less) or two (BN = 64, for
// products of few tiles: their time is the epilogue's, and twice the warps work
// on it; batch 4,096, hidden 512, under ncu: W1 forward 20.5 -> 17.0 us, W2
// forward 17.0 -> 14.0, dH 18.2 -> 15.5, dW1 16.3 -> 12.9):
//   warps 0, 10        TMA producers: 128 x 64 A and BN x 64 B tiles into a
//                      4- or 6-stage shared-memory ring (128-byte swizzle), one
//                      mbarrier with a transaction count per stage
//   warp 1             MMA issuer: four tcgen05.mma (K = 16 each) per stage into
//                      one of two tensor-memory accumulators; tcgen05.commit
//                      frees the stage, a commit per tile hands the
//                      accumulator to the epilogue
//   warps 2-9          epilogue: tcgen05.ld of their 32 accumulator lanes (two
//                      warps per lane quadrant, each half of the tile's
//                      columns), fused element-wise op, vector global stores;
//                      while they drain one accumulator the MMA warp fills the
//                      other.  Eight epilogue warps rather than four: the
//                      epilogue (the GELU chains above all) is bound by its own
//                      instruction latency with one warp per SM sub-partition
//                      (training step 0.130 -> 0.118 ms)
// Every mbarrier wait is bounded; on timeout the kernel raises an error flag,
// leaves its copies in flight the time to land, frees tensor memory and returns.
#include <atomic>
#include <mutex>
#include <unordered_map>

#include "ivhd_gelu.cuh"
#include "ivhd_gemm.cuh"
#include "ivhd_internal.cuh"
#include "ivhd_tc.cuh"

namespace ivhd {

namespace tc {

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

bool make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld,
              int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// Encoded maps of the operands seen so far, keyed by address and geometry: an
// encoding depends on nothing else, so a cached map equals a fresh one.  The
// GEMMs of the warm-start network reuse a few fixed buffers, so this removes
// the host-side encoding from every call after the first.
namespace {
struct MapKey {
  const void* base;
  int64_t rows, cols, ld;
  int box_rows;
  bool operator==(const MapKey& o) const {
    return base == o.base && rows == o.rows && cols == o.cols && ld == o.ld &&
           box_rows == o.box_rows;
  }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    uint64_t h = (uint64_t)(uintptr_t)k.base;
    for (uint64_t v : {(uint64_t)k.rows, (uint64_t)k.cols, (uint64_t)k.ld, (uint64_t)k.box_rows})
      h = (h ^ v) * 0x100000001b3ull;
    return (size_t)h;
  }
};
constexpr size_t kMapCacheMax = 1024;
}  // namespace

bool make_map_cached(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld,
                     int box_rows) {
  static std::mutex mu;
  static auto* cache = new std::unordered_map<MapKey, CUtensorMap, MapKeyHash>;
  const MapKey key{base, rows, cols, ld, box_rows};
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache->find(key);
    if (it != cache->end()) {
      *map = it->second;
      return true;
    }
  }
  if (!make_map(map, base, rows, cols, ld, box_rows)) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (cache->size() >= kMapCacheMax) cache->clear();
  (*cache)[key] = *map;
  return true;
}

}  // namespace tc

namespace {

using namespace tc;

constexpr int kBM = 128;
constexpr int kEpiWarps = 8;       // two per tensor-memory lane quadrant, each half the columns
constexpr int kGemmThreads = 32 * (3 + kEpiWarps);  // warps 0, 10 TMA, warp 1 MMA, warps 2-9 epilogue

__device__ __forceinline__ bool aligned16(const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0;
}

constexpr int kCols = 16;  // accumulator columns handled at once: 8 pairs for the packed FP32 pipe

// kCols BF16 values (round to nearest even) stored as 16-byte words.
__device__ __forceinline__ void store_bf16(__nv_bfloat16* o, const float* t) {
  uint32_t w[kCols / 2];
#pragma unroll
  for (int q = 0; q < kCols / 2; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(t[2 * q], t[2 * q + 1]);
    memcpy(&w[q], &h, 4);
  }
#pragma unroll
  for (int q = 0; q < kCols / 8; ++q)
    reinterpret_cast<uint4*>(o)[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// The transposed copy of kCols BF16 values of one row: column col0 + q of this
// row goes to out_t[(col0 + q) * ld_t + row].  The lanes of a warp hold
// consecutive rows, so each store is one contiguous 64-byte run.
__device__ __forceinline__ void store_bf16_t(__nv_bfloat16* out_t, int64_t ld_t, int row,
                                             int col0, int N, const float* t) {
#pragma unroll
  for (int q = 0; q < kCols; ++q)
    if (col0 + q < N) out_t[(int64_t)(col0 + q) * ld_t + row] = __float2bfloat16_rn(t[q]);
}

// Epilogue of kCols consecutive accumulator columns of one row: v[q] = C[row, col0 + q].
// Vector accesses where the columns are in range and 16-byte aligned, else
// element by element; the value written per element is the same either way.
__device__ __forceinline__ void ep_apply(const GemmEpilogue& ep, int row, int col0, int N,
                                         const float* v) {
  const int64_t off = (int64_t)row * ep.ld_out + col0;
  const bool full = col0 + kCols <= N;
  if (ep.kind == kEpStoreF32) {
    float* o = ep.out_f32 + off;
    if (full && aligned16(o)) {
#pragma unroll
      for (int q = 0; q < kCols / 4; ++q)
        reinterpret_cast<float4*>(o)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    } else {
#pragma unroll
      for (int q = 0; q < kCols; ++q)
        if (col0 + q < N) o[q] = v[q];
    }
  } else if (ep.kind == kEpBiasGelu) {
    // z = acc + bias is kept (FP32) for the backward pass (when out_f32 is
    // given: training); h = GELU(z) in BF16
    float* z = ep.out_f32 ? ep.out_f32 + off : nullptr;
    __nv_bfloat16* h = ep.out_bf16 + off;
    float t[kCols], g[kCols];
    const bool vec_bias = full && aligned16(ep.bias + col0);
#pragma unroll
    for (int q = 0; q < kCols; q += 4) {
      float4 b;
      if (vec_bias) {
        b = __ldg(reinterpret_cast<const float4*>(ep.bias + col0 + q));
      } else {
        b.x = col0 + q < N ? ep.bias[col0 + q] : 0.f;
        b.y = col0 + q + 1 < N ? ep.bias[col0 + q + 1] : 0.f;
        b.z = col0 + q + 2 < N ? ep.bias[col0 + q + 2] : 0.f;
        b.w = col0 + q + 3 < N ? ep.bias[col0 + q + 3] : 0.f;
      }
      const F2 z0 = f2_add(f2(v[q], v[q + 1]), f2(b.x, b.y)), z1 = f2_add(f2(v[q + 2], v[q + 3]), f2(b.z, b.w));
      const float2 t0 = f2_get(z0), t1 = f2_get(z1), g0 = gelu2(z0), g1 = gelu2(z1);
      t[q] = t0.x, t[q + 1] = t0.y, t[q + 2] = t1.x, t[q + 3] = t1.y;
      g[q] = g0.x, g[q + 1] = g0.y, g[q + 2] = g1.x, g[q + 3] = g1.y;
    }
    if (full && (!z || aligned16(z)) && aligned16(h)) {
      if (z) {
#pragma unroll
        for (int q = 0; q < kCols / 4; ++q)
          reinterpret_cast<float4*>(z)[q] =
              make_float4(t[4 * q], t[4 * q + 1], t[4 * q + 2], t[4 * q + 3]);
      }
      store_bf16(h, g);
    } else {
#pragma unroll
      for (int q = 0; q < kCols; ++q)
        if (col0 + q < N) {
          if (z) z[q] = t[q];
          h[q] = __float2bfloat16_rn(g[q]);
        }
    }
    if (ep.out_bf16_t) store_bf16_t(ep.out_bf16_t, ep.ld_t, row, col0, N, g);
  } else if (ep.kind == kEpGeluGrad) {
    // dZ = acc * GELU'(z) in BF16 (acc is dH)
    const float* z = ep.aux_f32 + off;
    __nv_bfloat16* o = ep.out_bf16 + off;
    float zz[kCols], t[kCols];
    if (full && aligned16(z)) {
#pragma unroll
      for (int q = 0; q < kCols / 4; ++q) {
        const float4 f = reinterpret_cast<const float4*>(z)[q];
        zz[4 * q] = f.x;
        zz[4 * q + 1] = f.y;
        zz[4 * q + 2] = f.z;
        zz[4 * q + 3] = f.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < kCols; ++q) zz[q] = (col0 + q < N) ? z[q] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < kCols; q += 2) {
      const float2 g = gelu_grad2(f2(zz[q], zz[q + 1]));
      t[q] = v[q] * g.x;
      t[q + 1] = v[q + 1] * g.y;
    }
    if (full && aligned16(o)) {
      store_bf16(o, t);
    } else {
#pragma unroll
      for (int q = 0; q < kCols; ++q)
        if (col0 + q < N) o[q] = __float2bfloat16_rn(t[q]);
    }
    if (ep.out_bf16_t) store_bf16_t(ep.out_bf16_t, ep.ld_t, row, col0, N, t);
  }
}

// Bounded wait that also stops when another role has given up.
__device__ __forceinline__ bool wait_or_stop(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  for (uint32_t it = 0; it < kSpinLimit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

template <int BN, int STAGES>
struct GemmSmem {
  static constexpr int a_bytes = kBM * kBK * 2;
  static constexpr int b_bytes = BN * kBK * 2;
  static constexpr int stage_bytes = a_bytes + b_bytes;
  static constexpr int bar_offset = STAGES * stage_bytes;
  static constexpr int total = bar_offset + 256 + 1024;  // + alignment slack
  // CTAs per SM: two where shared memory and tensor memory hold both
  static constexpr int per_sm = 2 * total <= 227 * 1024 && 4 * BN <= 512 ? 2 : 1;
};

// A work unit: output tile (tm, tn) and split-K slice z with its k-tiles
// [kt0, kt0 + nk).  Units are numbered so that the ones running at the same
// time on different SMs share operand tiles in L2: tiles go in groups of 8
// tile rows, column by column within a group.
struct Unit {
  int tm, tn, z, kt0, nk;
};
__device__ __forceinline__ Unit unit_of(int u, int tiles_m, int tiles_n, int splits, int nk_all) {
  constexpr int G = 8;
  const int per_z = tiles_m * tiles_n;
  const int z = u / per_z;
  const int t = u - z * per_z;
  const int first_m = (t / (G * tiles_n)) * G;
  const int gm = min(G, tiles_m - first_m);
  const int local = t - first_m * tiles_n;
  Unit r;
  r.tm = first_m + local % gm;
  r.tn = local / gm;
  r.z = z;
  const int per = (nk_all + splits - 1) / splits;
  r.kt0 = z * per;
  r.nk = max(0, min(nk_all, r.kt0 + per) - r.kt0);
  return r;
}

// Persistent: each CTA (one per SM, two with BN = 64) takes units blockIdx.x, blockIdx.x +
// gridDim.x, ...  Two accumulators in tensor memory (2 x BN columns): the MMA
// warp fills one while the epilogue warps drain the other.
//   full[s] / empty[s]      shared-memory stage s loaded (TMA) / consumed (MMA commit)
//   acc_full[b]             accumulator b complete (MMA commit)
//   acc_empty[b]            accumulator b read out (one arrival per epilogue warp)
template <int BN, int STAGES>
__global__ void __launch_bounds__(kGemmThreads, GemmSmem<BN, STAGES>::per_sm)
    k_gemm_bf16_tn(const __grid_constant__ CUtensorMap map_a,
                   const __grid_constant__ CUtensorMap map_b, GemmEpilogue ep, int M, int N,
                   int K, int splits, int32_t* __restrict__ err) {
  using S = GemmSmem<BN, STAGES>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::bar_offset);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kTmemCols = 2 * BN;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int tiles_m = (M + kBM - 1) / kBM, tiles_n = (N + BN - 1) / BN;
  const int nk_all = (K + kBK - 1) / kBK;
  const int units = tiles_m * tiles_n * splits;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;
  // What precedes in the stream is complete from here on.  The next kernel may be
  // launched once every CTA is here: each holds its tensor memory by then, so a
  // waiting CTA of the next kernel cannot keep it from one of this kernel.
  depend();

  if (warp == 0 || warp == 2 + kEpiWarps) {
    // TMA producers, one for each operand (one warp's copies reach about 50
    // bytes per clock, two warps' 93); the first announces the bytes of both
    const bool second = warp != 0;
    int s = 0;
    uint32_t lap = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
      const Unit w = unit_of(u, tiles_m, tiles_n, splits, nk_all);
      const int y = second ? w.tn * BN : w.tm * kBM;
      for (int kt = 0; kt < w.nk; ++kt) {
        if (lap > 0) ok = __all_sync(0xffffffffu, wait_or_stop(&empty[s], (lap - 1) & 1, abort_flag));
        if (!ok) break;
        if (elect_one()) {
          if (!second) mbar_expect_tx(&full[s], S::stage_bytes);
          tma_load_2d(smem + s * S::stage_bytes + (second ? S::a_bytes : 0), second ? &map_b : &map_a,
                      (w.kt0 + kt) * kBK, y, &full[s]);
        }
        if (++s == STAGES) {
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
    // MMA issuer
    constexpr uint32_t idesc = instr_desc_bf16(kBM, BN);
    const uint64_t desc = smem_desc_sw128(smem_u32(smem));
    int s = 0, j = 0;
    uint32_t lap = 0;
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity, int code) {
      ok = __all_sync(0xffffffffu, wait_or_stop(bar, parity, abort_flag));
      if (!ok && lane == 0) atomicOr(err, code);
      asm volatile("tcgen05.fence::after_thread_sync;");
      return ok;
    };
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++j) {
      const Unit w = unit_of(u, tiles_m, tiles_n, splits, nk_all);
      const int b = j & 1;
      if (j >= 2 && !wait(&acc_empty[b], ((j >> 1) - 1) & 1, 8)) break;
      const uint32_t d = tmem + (uint32_t)(b * BN);
      for (int kt = 0; kt < w.nk; ++kt) {
        if (!wait(&full[s], lap & 1, 2)) break;
        if (elect_one()) {
          const uint64_t da = desc + (uint64_t)(s * (S::stage_bytes >> 4)), db = da + (S::a_bytes >> 4);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            umma_bf16(d, da + 2 * kk, db + 2 * kk, idesc, (kt > 0 || kk > 0) ? 1u : 0u);
          umma_commit(&empty[s]);
        }
        __syncwarp();
        if (++s == STAGES) {
          s = 0;
          ++lap;
        }
      }
      // this unit's MMAs (an empty slice arrives at once)
      if (ok && elect_one()) umma_commit(&acc_full[b]);
      __syncwarp();
    }
    // every MMA issued above has finished before tensor memory is released
    if (elect_one()) umma_commit(done);
    if (!mbar_wait(done, 0) && lane == 0) atomicOr(err, 16);
  } else {
    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31
    const int q = warp & 3;
    const int half = (warp - 2) / 4;  // warps 2-5: first BN / 2 columns; 6-9: the rest
    int j = 0;
    for (int u = blockIdx.x; u < units; u += gridDim.x, ++j) {
      const Unit w = unit_of(u, tiles_m, tiles_n, splits, nk_all);
      const int b = j & 1;
      // warp-uniform decisions: tcgen05.ld below is executed by all 32 lanes together
      if (!__all_sync(0xffffffffu, wait_or_stop(&acc_full[b], (j >> 1) & 1, abort_flag))) {
        if (lane == 0) atomicOr(err, 4);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      const int row = w.tm * kBM + q * 32 + lane;
      GemmEpilogue epz = ep;
      if (splits > 1) epz.out_f32 += (int64_t)w.z * ep.split_stride;
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN);
#pragma unroll 1
      for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += kCols) {
        float v[kCols];
        if (w.nk > 0) {
          tmem_ld16(taddr + (uint32_t)c, v);
        } else {
#pragma unroll
          for (int t = 0; t < kCols; ++t) v[t] = 0.f;  // an empty K slice contributes zero
        }
        const int col0 = w.tn * BN + c;
        if (row < M && col0 < N) ep_apply(epz, row, col0, N, v);
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[b]);
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols));
}

// ---- host side --------------------------------------------------------------

int sm_count() {
  static int count[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 148;
  if (!count[dev]) {
    int c = 0;
    if (cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || c < 1)
      c = 148;
    count[dev] = c;
  }
  return count[dev];
}

template <int BN, int STAGES>
cudaError_t launch_bn(const CUtensorMap& ma, const CUtensorMap& mb, const GemmEpilogue& ep, int M,
                      int N, int K, int splits, int32_t* err, cudaStream_t s, bool dependent) {
  const int smem = GemmSmem<BN, STAGES>::total;
  static bool attr_set[64] = {};  // one attribute call per instantiation and device
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_bf16_tn<BN, STAGES>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  const int64_t units = (int64_t)((M + kBM - 1) / kBM) * ((N + BN - 1) / BN) * splits;
  const int slots = sm_count() * GemmSmem<BN, STAGES>::per_sm;
  const int grid = (int)(units < slots ? units : slots);
  return launch_dependent(dependent, k_gemm_bf16_tn<BN, STAGES>, dim3(grid), dim3(kGemmThreads),
                          smem, s, ma, mb, ep, M, N, K, splits, err);
}

}  // namespace

cudaError_t gemm_bf16_tn(const __nv_bfloat16* A, int64_t lda, const __nv_bfloat16* B, int64_t ldb,
                         int M, int N, int K, const GemmEpilogue& ep, int32_t* err,
                         cudaStream_t s, int splits, bool dependent) {
  if (splits < 1 || (splits > 1 && ep.kind != kEpStoreF32)) return cudaErrorInvalidValue;
  // 256-column tiles when they keep every SM busy and pad N no more than
  // 128-column ones; 64-column tiles, two CTAs per SM, when 128-column ones
  // would not give every SM two: the epilogue is then most of the time, and
  // twice the warps work on it (the network's products at batch 4,096, below)
  const int64_t tiles_m = (M + kBM - 1) / kBM;
  const int64_t n256 = (N + 255) / 256, n128 = (N + 127) / 128;
  const bool wide = tiles_m * n256 * splits >= sm_count() && n256 * 256 <= n128 * 128;
  const bool narrow = !wide && tiles_m * n128 * splits < 2 * sm_count();
  const int BN = wide ? 256 : narrow ? 64 : 128;
  CUtensorMap ma, mb;
  if (!make_map_cached(&ma, A, M, K, lda, kBM)) return cudaErrorInvalidValue;
  if (!make_map_cached(&mb, B, N, K, ldb, BN)) return cudaErrorInvalidValue;
  if (wide) return launch_bn<256, 4>(ma, mb, ep, M, N, K, splits, err, s, dependent);
  if (narrow) return launch_bn<64, 4>(ma, mb, ep, M, N, K, splits, err, s, dependent);
  return launch_bn<128, 6>(ma, mb, ep, M, N, K, splits, err, s, dependent);
}

// out[i] = sum_z part[z * stride + i] over `splits` slices in order (deterministic).
__global__ void k_sum_slices(const float* __restrict__ part, int64_t n, int64_t stride, int splits,
                             float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float t = 0.f;
  for (int z = 0; z < splits; ++z) t += part[z * stride + i];
  out[i] = t;
}

cudaError_t sum_slices(const float* part, int64_t n, int64_t stride, int splits, float* out,
                       cudaStream_t s) {
  k_sum_slices<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, n, stride, splits, out);
  return cudaGetLastError();
}

}  // namespace ivhd

using namespace ivhd;

// Error flags of ivhd_gemm_bf16_tn calls: a fixed set of slots in the
// library's device memory, taken in turn, so a call allocates nothing.  A slot
// is reused only after kErrSlots later calls; each call clears its slot first.
constexpr int kErrSlots = 256;
static __device__ int32_t g_gemm_err[kErrSlots];

extern "C" ivhd_status ivhd_gemm_bf16_tn(const void* A, const void* B, float* C, int64_t M,
                                         int64_t N, int64_t K, void* stream) {
  if (!A || !B || !C || M < 1 || N < 1 || K < 1) return IVHD_ERR_ARG;
  if (M > (1 << 30) || N > (1 << 30) || K > (1 << 30) || (K % 8) != 0) return IVHD_ERR_ARG;
  if (((uintptr_t)A & 15) || ((uintptr_t)B & 15) || ((uintptr_t)C & 15)) return IVHD_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  static std::atomic<uint32_t> next{0};
  int32_t* slots = nullptr;
  cudaError_t e = cudaGetSymbolAddress((void**)&slots, g_gemm_err);
  if (e != cudaSuccess) return IVHD_ERR_CUDA;
  int32_t* err = slots + (next.fetch_add(1) % kErrSlots);
  int32_t herr = 0;
  e = cudaMemsetAsync(err, 0, sizeof(int32_t), s);
  GemmEpilogue ep{};
  ep.kind = kEpStoreF32;
  ep.split_stride = 0;
  ep.out_f32 = C;
  ep.ld_out = N;
  if (e == cudaSuccess)
    e = gemm_bf16_tn((const __nv_bfloat16*)A, K, (const __nv_bfloat16*)B, K, (int)M, (int)N,
                     (int)K, ep, err, s, 1);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e == cudaErrorInvalidValue ? IVHD_ERR_ARG : IVHD_ERR_CUDA;
  return herr ? IVHD_ERR_TIMEOUT : IVHD_OK;
}
