// ivhd_mlp_place.cu -- the warm-start network applied to new rows in one kernel:
//
//   y = W3 bf16(GELU(W2 bf16(GELU(W1 x + b1)) + b2)) + b3
//
// with the values of the layer-by-layer path (BF16 operands, FP32 accumulation,
// bias and GELU in FP32, activations rounded to BF16, FP32 output layer; the
// output layer's sum runs in another fixed order).  The activations never
// leave the SM: a layer at a time wrote and re-read 2 KB per row, and its GEMMs
// were bound by that epilogue.  1.4e6 rows of 784 bytes, hidden 512: 5.63 ms
// layer by layer, 2.36 ms here (the MMAs need 1.0 ms at the tensor cores' rate).
//
// A pair of CTAs (cta_group::2) takes 256 rows at a time, 128 each, and loops
// over such tiles (persistent).  The hidden layers are computed in chunks of
// at most 256 columns, one tensor-memory buffer (128 lanes x 256 columns) each,
// so that the epilogue of one chunk runs beside the MMAs of the next:
//
//   MMA       L1c0      L1c1      L2c0 (K of c0) (K of c1)   L2c1     L1c0' ...
//   epilogue            E1c0      E1c1                       E2c0     E2c1 ...
//
// E1 writes BF16 activations to shared memory as the K-major, 128-byte-swizzled
// A operand of layer 2; E2 adds the row's two outputs from its columns.
//   warp 0      TMA: stages of two 16 KB slabs (128 x 64; x and W1, or two of W2)
//               into a ring; every CTA loads its own rows of x and half of the
//               weights' rows
//   warp 1      MMA issuer (rank 0)
//   warps 2-17  epilogue: four warps per tensor-memory lane quadrant, a quarter
//               of the chunk's columns each
//   warp 18     TMA: the second slab of every stage (copies issued by one warp
//               reach about 50 bytes per clock, by two about 93)
// Waits are bounded; on timeout an error flag is raised and all roles stop.
#include "ivhd_gelu.cuh"
#include "ivhd_gemm.cuh"
#include "ivhd_internal.cuh"
#include "ivhd_mlp_place.cuh"
#include "ivhd_tc.cuh"

namespace ivhd {
namespace {

using namespace tc;

constexpr int kRows = 128;             // rows per CTA
constexpr int kChunkN = 256;           // hidden columns per chunk
constexpr int kMaxHidden = 2 * kChunkN;
constexpr int kSlab = kRows * kBK * 2; // 16 KB: 128 rows x 64 columns
constexpr int kStage = 2 * kSlab;      // layer 1: x and W1; layer 2: two slabs of W2
constexpr int kStages = 3;
constexpr int kParts = 4;              // column quarters of a chunk
constexpr int kEpi = 4 * kParts;       // epilogue warps
constexpr int kThreads = 32 * (3 + kEpi);

// Shared memory: the layer-1 activations (up to 128 KB), the ring, the barriers.
__host__ __device__ constexpr int h1_slabs(int H) { return (H + kBK - 1) / kBK; }
constexpr int kBars = 512;
__host__ __device__ constexpr int smem_bytes(int H) {
  return (h1_slabs(H) > kParts ? h1_slabs(H) : kParts) * kSlab + kStages * kStage + kBars + 1024;
}

// Barrier `id` over n threads; whether ok was set in all of them.
__device__ __forceinline__ bool bar_and(int id, int n, bool ok) {
  int all;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.s32 q, %1, 0;\n"
      "barrier.cta.red.and.pred p, %2, %3, q;\n"
      "selp.s32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(all)
      : "r"((int)ok), "r"(id), "r"(n)
      : "memory");
  return all != 0;
}

__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_place(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w1,
                const __grid_constant__ CUtensorMap map_w2, const float* __restrict__ b1,
                const float* __restrict__ b2, const float* __restrict__ W3,
                const float* __restrict__ b3, int rows, int n_in, int H, float2* __restrict__ y,
                float2* __restrict__ y_copy, int32_t* __restrict__ err) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int nk2 = h1_slabs(H);
  unsigned char* ring = smem + (nk2 > kParts ? nk2 : kParts) * kSlab;
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kStages * kStage);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;  // [2] a chunk's accumulator is complete
  uint64_t* acc_done = acc_full + 2;     // [2] a chunk is read out (layer 1: and its activations written)
  uint64_t* done = acc_done + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
  const int n_tiles = (rows + 2 * kRows - 1) / (2 * kRows);
  const int nc = (H + kChunkN - 1) / kChunkN;  // 1 or 2
  const int nk1 = (n_in + kBK - 1) / kBK;
  auto width = [&](int c) { return min(kChunkN, H - c * kChunkN); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int c = 0; c < 2; ++c) {
      mbar_init(&acc_full[c], 1);
      mbar_init(&acc_done[c], 2 * kEpi);  // the epilogue warps of both CTAs
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(2 * kChunkN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  pair_sync();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;

  // The ring's stages in order: a thread's position in it, without divisions (one
  // thread loads and one issues; what they do per stage is what they can give).
  struct Cursor {
    int s = 0;
    uint32_t lap = 0;
    __device__ __forceinline__ void next() {
      if (++s == kStages) {
        s = 0;
        ++lap;
      }
    }
  };

  if (warp == 0 || warp == 2 + kEpi) {
    // the first and the second slab of every stage; the first producer of rank 0
    // announces the bytes of all
    const int second = warp != 0;
    Cursor c;
    bool ok = true;
    const uint32_t full0 = pair_addr(full, 0);
    auto load = [&](const CUtensorMap* map, int x, int y, int slabs) {
      if (c.lap > 0) ok = __all_sync(0xffffffffu, pair_wait(&empty[c.s], (c.lap - 1) & 1, abort_flag));
      if (!ok) return;
      if (elect_one()) {
        if (rank == 0 && !second) mbar_expect_tx(&full[c.s], 2 * slabs * kSlab);
        if (second < slabs)
          tma_load_2d_pair(ring + c.s * kStage + second * kSlab, map, x, y, full0 + (uint32_t)c.s * 8u);
      }
      c.next();
    };
    for (int t = pair; t < n_tiles && ok; t += n_pairs) {
      for (int n = 0; n < nc && ok; ++n) {
        const int y = second ? n * kChunkN + (int)rank * (width(n) / 2) : (2 * t + (int)rank) * kRows;
        for (int k = 0; k < nk1 && ok; ++k) load(second ? &map_w1 : &map_x, k * kBK, y, 2);
      }
      for (int n = 0; n < nc && ok; ++n) {
        const int y = n * kChunkN + (int)rank * (width(n) / 2);
        for (int k = 0; k < nk2 && ok; k += 2)
          load(&map_w2, (k + second) * kBK, y, min(2, nk2 - k));
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
      Cursor c;
      bool ok = true;
      auto wait = [&](uint64_t* bar, uint32_t parity, int code) {
        ok = __all_sync(0xffffffffu, pair_wait(bar, parity, abort_flag));
        if (!ok && lane == 0) atomicOr(err, code);
        asm volatile("tcgen05.fence::after_thread_sync;");
        return ok;
      };
      const uint64_t ring_desc = smem_desc_sw128(smem_u32(ring)), h1_desc = smem_desc_sw128(smem_u32(smem));
      int i = 0;  // tiles of this pair so far
      for (int t = pair; t < n_tiles && ok; t += n_pairs, ++i) {
        for (int n = 0; n < nc && ok; ++n) {
          if (i > 0 && !wait(&acc_done[n], 1, 4)) break;  // the previous tile's layer 2
          const uint32_t dst = tmem + (uint32_t)(n * kChunkN), idesc = instr_desc_bf16(2 * kRows, width(n));
          for (int k = 0; k < nk1; ++k) {
            if (!wait(&full[c.s], c.lap & 1, 2)) break;
            if (elect_one()) {
              const uint64_t a = ring_desc + (uint64_t)(c.s * (kStage >> 4));
              umma_slab_pair(dst, a, a + (kSlab >> 4), idesc, k == 0, min(kBK / 16, (n_in - k * kBK + 15) / 16));
              umma_commit_pair(&empty[c.s]);
              if (k + 1 == nk1) umma_commit_pair(&acc_full[n]);
            }
            __syncwarp();
            c.next();
          }
        }
        for (int n = 0; n < nc && ok; ++n) {
          const uint32_t dst = tmem + (uint32_t)(n * kChunkN), idesc = instr_desc_bf16(2 * kRows, width(n));
          for (int k = 0; k < nk2; k += 2) {
            // layer 1's chunk k / 4 holds these activations (the first wait for a
            // chunk also frees its accumulator)
            if (n == 0 && k % (kChunkN / kBK) == 0 && !wait(&acc_done[k / (kChunkN / kBK)], 0, 8)) break;
            if (!wait(&full[c.s], c.lap & 1, 2)) break;
            if (elect_one()) {
              const uint64_t b = ring_desc + (uint64_t)(c.s * (kStage >> 4));
              const uint64_t a = h1_desc + (uint64_t)(k * (kSlab >> 4));
              umma_slab_pair(dst, a, b, idesc, k == 0, min(kBK / 16, (H - k * kBK) / 16));
              if (k + 1 < nk2)
                umma_slab_pair(dst, a + (kSlab >> 4), b + (kSlab >> 4), idesc, false,
                               min(kBK / 16, (H - (k + 1) * kBK) / 16));
              umma_commit_pair(&empty[c.s]);
              if (k + 2 >= nk2) umma_commit_pair(&acc_full[n]);
            }
            __syncwarp();
            c.next();
          }
        }
      }
      if (elect_one()) umma_commit_pair(done);
      if (!mbar_wait(done, 0) && lane == 0) atomicOr(err, 16);
    }
  } else {
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int r = quarter * 32 + lane;
    const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t h1_s = smem_u32(smem) + (uint32_t)r * 128u;
    // the row's partial sums: in the units of its layer-1 activations (free
    // once layer 2 is complete) that only the part-0 warps write, who add them
    const uint32_t sum_s = h1_s + (uint32_t)((r & 7) * 16);
    auto param = [&](const float* p, int col) { return __ldg(reinterpret_cast<const float4*>(p + col)); };
    bool ok = true;
    auto wait = [&](int c, uint32_t parity) {
      if (!pair_wait(&acc_full[c], parity, abort_flag)) ok = false;
      ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is executed by the warp together
      if (!ok && lane == 0) atomicOr(err, 32);
      asm volatile("tcgen05.fence::after_thread_sync;");
      return ok;
    };
    int i = 0;
    for (int t = pair; t < n_tiles && ok; t += n_pairs, ++i) {
      for (int c = 0; c < nc; ++c) {
        if (!ok || !wait(c, 0)) break;
        const int w = width(c);
        // this warp's columns of the chunk: groups of 16, part, part + 4, ...
        for (int q0 = part * 16; q0 < w; q0 += 16 * kParts) {
          uint32_t v[16];
          tmem_ld16_nowait(lanes + (uint32_t)(c * kChunkN + q0), v);
          tmem_wait_ld16(v);
          const int col = c * kChunkN + q0;
          uint32_t h[8];
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            const float4 b = param(b1, col + q);
            const float2 g0 = gelu2(f2_add(f2(__uint_as_float(v[q]), __uint_as_float(v[q + 1])), f2(b.x, b.y)));
            const float2 g1 = gelu2(f2_add(f2(__uint_as_float(v[q + 2]), __uint_as_float(v[q + 3])), f2(b.z, b.w)));
            const __nv_bfloat162 lo = __floats2bfloat162_rn(g0.x, g0.y);
            const __nv_bfloat162 hi = __floats2bfloat162_rn(g1.x, g1.y);
            memcpy(&h[q / 2], &lo, 4);
            memcpy(&h[q / 2 + 1], &hi, 4);
          }
          // 16-byte units of the row, swizzled as the TMA writes an operand
          const uint32_t slab = h1_s + (uint32_t)(col / kBK) * kSlab;
          const uint32_t u = (uint32_t)(col % kBK) / 8u;
          st_shared_u4(slab + ((u ^ (r & 7)) * 16u), h[0], h[1], h[2], h[3]);
          st_shared_u4(slab + (((u + 1u) ^ (r & 7)) * 16u), h[4], h[5], h[6], h[7]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_release(pair_addr(&acc_done[c], 0));
      }
      F2 s0 = f2_same(0.f), s1 = s0;
      for (int c = 0; c < nc && ok; ++c) {
        if (!wait(c, 1)) break;
        const int w = width(c);
        for (int q0 = part * 16; q0 < w; q0 += 16 * kParts) {
          uint32_t v[16];
          tmem_ld16_nowait(lanes + (uint32_t)(c * kChunkN + q0), v);
          tmem_wait_ld16(v);
          const int col = c * kChunkN + q0;
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            const float4 b = param(b2, col + q);
            const float4 u = param(W3, col + q);
            const float4 x = param(W3 + H, col + q);
            const float2 g0 = gelu2(f2_add(f2(__uint_as_float(v[q]), __uint_as_float(v[q + 1])), f2(b.x, b.y)));
            const float2 g1 = gelu2(f2_add(f2(__uint_as_float(v[q + 2]), __uint_as_float(v[q + 3])), f2(b.z, b.w)));
            const float2 h0 = __bfloat1622float2(__floats2bfloat162_rn(g0.x, g0.y));
            const float2 h1 = __bfloat1622float2(__floats2bfloat162_rn(g1.x, g1.y));
            // even and odd columns apart, two sums per output
            s0 = f2_fma(f2(u.x, u.y), f2(h0.x, h0.y), s0);
            s1 = f2_fma(f2(x.x, x.y), f2(h0.x, h0.y), s1);
            s0 = f2_fma(f2(u.z, u.w), f2(h1.x, h1.y), s0);
            s1 = f2_fma(f2(x.z, x.w), f2(h1.x, h1.y), s1);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(pair_addr(&acc_done[c], 0));
      }
      // the quarter's four column parts, added in order.  The four warps leave
      // together when one of them has given up.
      const float2 t0 = f2_get(s0), t1 = f2_get(s1);
      st_shared_f2(sum_s + (uint32_t)part * kSlab, t0.x + t0.y, t1.x + t1.y);
      ok = bar_and(1 + quarter, 32 * kParts, ok);
      if (!ok) break;
      const int row = (2 * t + (int)rank) * kRows + r;
      if (part == 0 && row < rows) {
        float2 o = ld_shared_f2(sum_s);
        for (int q = 1; q < kParts; ++q) {
          const float2 v = ld_shared_f2(sum_s + (uint32_t)q * kSlab);
          o.x += v.x;
          o.y += v.y;
        }
        o.x += b3[0];
        o.y += b3[1];
        y[row] = o;
        if (y_copy) y_copy[row] = o;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  pair_sync();  // no MMA, copy or arrival of the pair is outstanding
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(2 * kChunkN));
}

}  // namespace

bool mlp_place_supported(int hidden) { return hidden <= kMaxHidden; }

int mlp_place_rows(int max_rows) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 2)
    return max_rows;
  const int round = sms / 2 * 2 * kRows;  // one tile for every pair of SMs
  return max_rows < round ? max_rows : max_rows / round * round;
}

cudaError_t mlp_place(const MlpPlace& P, int rows, const __nv_bfloat16* x, float* y, float* y_copy,
                      cudaStream_t s) {
  CUtensorMap mx, m1, m2;
  if (!make_map_cached(&mx, x, rows, P.n_in, P.n_in, kRows) ||
      !make_map_cached(&m1, P.w1, P.hidden, P.n_in, P.n_in, kRows) ||
      !make_map_cached(&m2, P.w2, P.hidden, P.hidden, P.hidden, kRows))
    return cudaErrorInvalidValue;
  static bool attr_set[64] = {};
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    e = cudaFuncSetAttribute(k_mlp_place, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem_bytes(kMaxHidden));
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  const int tiles = (rows + 2 * kRows - 1) / (2 * kRows), pairs = sms / 2 > 0 ? sms / 2 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (unsigned)(tiles < pairs ? tiles : pairs));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes(P.hidden);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mlp_place, mx, m1, m2, P.b1, P.b2, P.W3, P.b3, rows, P.n_in,
                            P.hidden, (float2*)y, (float2*)y_copy, P.err);
}

}  // namespace ivhd
