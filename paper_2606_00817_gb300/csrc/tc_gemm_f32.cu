// tc_gemm_f32.cu -- one FP32 layer Y = ReLU(A W^T + b) on the tensor cores,
// by splitting every FP32 operand into three bf16 values
//   x = x0 + x1 + x2   (x0 = bf16(x), x1 = bf16(x - x0), x2 = x - x0 - x1)
// which is exact for normal numbers (3 x 8 significand bits; every remainder
// is a float32 subtraction without rounding), and summing the six products
//   a2 w0 + a0 w2 + a1 w1 + a1 w0 + a0 w1 + a0 w0
// of bf16 operands, each exact in FP32. Of the three products left out a1 w2 and
// a2 w1 reach 2^-25 of |a w| (|x1| <= 2^-8 |x|, |x2| <= 2^-17 |x|), a2 w2 2^-34, all
// of random sign (the pieces are rounded to nearest). An infinite activation
// meets each weight once, in a2 w0, and gives what an FP32 FMA gives (unless the
// weight is so small, under 2^-133, that its first piece is 0).
//
// What bounds it: the tensor pipe, at six bf16 MMAs per FP32 one, and between
// two tiles the outputs (the epilogue warps hold a tile's sums in registers, so
// the MMAs run at most two accumulators ahead of them). Measured through the
// 126 -> 1280 x 8 field: 16,387 rays 1.50 ms against 9.53 ms on FFMA
// (sgemm_relu_kernel), without any output stores 1.18, without operand loads or
// without reading the accumulators no less; 140,000 rays 11.8 ms, 1 ray 0.24
// against 1.40 ms; at 256 x 3, 5,000 rays 0.06 against 0.128 ms. It wins at every
// batch size, so a width that is a multiple of 256 always takes it; other widths
// keep the FFMA layers.
//
// Precision. The MMA adds into its FP32 accumulator without rounding to
// nearest, so a long sum in TMEM would drift. An accumulator therefore only
// ever holds 32 of K (the small products first, a0 w0 last); the epilogue
// warps add these in registers in ordinary FP32, and while they drain one
// accumulator the MMAs of the next fill the other. Against 64 bits the
// outputs are as near as on FFMA or nearer: t at 1280 x 8 4.1e-8 (FFMA 4.7e-8),
// with 1.7 times the weights 6.6e-7 (2.2e-6), at 256 x 3 6.3e-8 (6.9e-8).
// Draining every 64 of K cost 3 % less time on 140,000 rays but left a bias
// that 32 halves.
//
// Shape: as the pair kernel (tc_gemm_pair.cu), a cluster of two CTAs owns a
// 256 x 256 tile (cta_group::2, M = N = 256). A stage is one K block of 64 of
// all planes: 3 x 16 KB of A and 3 x 16 KB of W per CTA; two stages fill
// shared memory, and each is 24 MMAs long (about 3,000 cycles), which hides
// the 96 KB load of the other. 8 epilogue warps hold 128 columns each of
// their row in 128 registers per thread.
//
// Waits are bounded and an abort drains as in the pair kernel.
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "f32_split.cuh"
#include "kernels.h"
#include "ptx_sm103.cuh"

namespace ddf {

namespace {

constexpr uint64_t kF32DrainNs = 1000000000ull;
constexpr int kF32Epi = 8;                       // epilogue warps
constexpr int kF32Threads = 32 * (2 + kF32Epi);
constexpr int kF32Stages = 2;
constexpr int kF32Plane = 128 * 128;             // 128 rows x 64 bf16: 16 KB
constexpr int kF32Operand = 3 * kF32Plane;       // the three planes of A (or W)
constexpr int kF32Stage = 2 * kF32Operand;
constexpr int kF32Ctrl = 128;
constexpr int kF32Smem = kF32Stages * kF32Stage + kF32Ctrl + 1024;
static_assert(kF32Smem <= 227 * 1024, "shared memory of one CTA");

// The six products, smallest first: plane of A, plane of W.
__device__ constexpr int kProdA[6] = {2, 0, 1, 1, 0, 0};
__device__ constexpr int kProdW[6] = {0, 2, 1, 0, 1, 0};

// The tiles of a layer on `slots` clusters: whole waves of 256 x 256 tiles, and
// each tile left over in 1 << lg parts of 256 >> lg columns, as many as one wave
// holds (a part of 64 columns takes a third of a tile's time, by its operands).
// 1280 x 8, undivided and so: 1 ray (5 tiles of 76) 337 and 243 us, 1,000 rays (20)
// 406 and 314, 4,099 rays (a wave and 9) 739 and 609.
// The parts come first: the clusters that begin with one are out of step with the
// others from then on, and their outputs' stores do not all fall together (1,506 and
// 1,484 us).
struct F32Plan {
  int parts, lg, tiles;
};
__host__ __device__ inline F32Plan f32_plan(int M, int N, int slots) {
  const int all = (M + 255) / 256 * (N / 256), big = all / slots * slots, rest = all - big;
  const int lg = 4 * rest <= slots ? 2 : 2 * rest <= slots ? 1 : 0;
  return F32Plan{rest << lg, lg, big + (rest << lg)};
}
struct F32Tile {
  int m0, n0, n;  // first row and column, columns
};
__device__ __forceinline__ int f32_columns(const F32Plan& f, int t) {
  return t < f.parts ? 256 >> f.lg : 256;
}
__device__ __forceinline__ F32Tile f32_tile(const F32Plan& f, int t, int num_n) {
  const int n = f32_columns(f, t);
  const int sub = t < f.parts ? t & ((1 << f.lg) - 1) : 0;
  t = t < f.parts ? t >> f.lg : t - f.parts + (f.parts >> f.lg);
  const int m = t / num_n;
  return F32Tile{m * 256, (t - m * num_n) * 256 + sub * n, n};
}

// The pieces of COLS outputs (>= 0, no NaN), as f32_split gives them, 16 at a time,
// plane by plane and packed in pairs. An infinity's pieces come out as bf16's
// largest value, infinity and NaN, which the sum of all third pieces shows; they
// are then looked for and stored again. With the selects of f32_split for each
// output the drain has too few registers (16,387 rays 1,471 us without a rule for
// infinities, 1,503 with the selects, 1,474 so).
template <int COLS>
__device__ __forceinline__ void f32_store_planes(float* x, __nv_bfloat16* dst, size_t plane) {
  const __nv_bfloat162 most = __halves2bfloat162(__ushort_as_bfloat16(0x7f7f),
                                                 __ushort_as_bfloat16(0x7f7f));
  __nv_bfloat162 sum = __halves2bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0));
#pragma unroll
  for (int c = 0; c < COLS; c += 16) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float &a = x[c + 2 * i], &b = x[c + 2 * i + 1];
        __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        if (j == 0) v = __hmin2(v, most);
        if (j == 2) sum = __hadd2(sum, v);
        w[i] = *reinterpret_cast<const uint32_t*>(&v);
        a -= __uint_as_float(w[i] << 16);
        b -= __uint_as_float(w[i] & 0xffff0000u);
      }
      st_global_256(dst + j * plane + c, w);
    }
  }
  if (__builtin_expect(__hbeq2(sum, sum), 1)) return;
  for (int i = 0; i < COLS; ++i) {
    if (!__hisnan(dst[2 * plane + i])) continue;
    dst[i] = dst[plane + i] = __ushort_as_bfloat16(0);
    dst[2 * plane + i] = __ushort_as_bfloat16(0x7f80);
  }
}

// One warp's part of a tile: COLS columns of its 32 rows, the accumulators of
// every 32 of K added up (`it` counts them), then bias, ReLU and the output at the
// row and column `where` gives (asked late: its registers are not there before).
// False when a wait gave up.
template <int COLS, class Wait, class Done, class Where>
__device__ __forceinline__ bool f32_drain(const TcF32Params& p, uint32_t trow, int blocks,
                                          uint32_t& it, Wait wait, Done done, Where where) {
  float acc[COLS];
#pragma unroll
  for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
  for (int kb = 0; kb < blocks; ++kb, ++it) {
    const int b = it & 1;
    if (!wait(b, (it >> 1) & 1)) return false;
    tc_fence_after();
#pragma unroll
    for (int c = 0; c < COLS / 16; ++c) {  // 16 columns at a time: 32 would spill
      uint32_t v[16];
      tmem_ld16_wait(trow + 256u * b + 16u * c, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[16 * c + i] += __uint_as_float(v[i]);
    }
    tc_fence_before();
    __syncwarp();
    done(b);
  }
  int row, n0;
  where(row, n0);
  if (row >= p.M) return true;
  const float4* bias = reinterpret_cast<const float4*>(p.bias + n0);
#pragma unroll
  for (int c = 0; c < COLS / 4; ++c) {
    const float4 bb = __ldg(bias + c);
    acc[4 * c + 0] = fmaxf(acc[4 * c + 0] + bb.x, 0.f);
    acc[4 * c + 1] = fmaxf(acc[4 * c + 1] + bb.y, 0.f);
    acc[4 * c + 2] = fmaxf(acc[4 * c + 2] + bb.z, 0.f);
    acc[4 * c + 3] = fmaxf(acc[4 * c + 3] + bb.w, 0.f);
  }
  // 32-byte stores: the lanes' rows lie apart, and with half-written sectors this
  // part took a third of a layer's time (16,387 rays 1.80 ms, now 1.53; TMA stores
  // from shared-memory boxes, for which only 32 KB are left, 1.69)
  if (p.out_f32 != nullptr) {  // the last layer: FP32 rows for the head
    float* dst = p.out_f32 + static_cast<size_t>(row) * p.N + n0;
#pragma unroll
    for (int c = 0; c < COLS / 8; ++c) {
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = __float_as_uint(acc[8 * c + i]);
      st_global_256(dst + 8 * c, w);
    }
  } else {  // the next layer's operand: three bf16 planes
    f32_store_planes<COLS>(acc, p.out_planes + static_cast<size_t>(row) * p.N + n0,
                           static_cast<size_t>(p.M) * p.N);
  }
  return true;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kF32Threads, 1)
    tc_gemm_f32_kernel(const __grid_constant__ CUtensorMap tmA,
                       const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmB32, const TcF32Params p,
                       const int slots) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kF32Stages * kF32Stage);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (2 + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (4 + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (6 + b); };
  const uint32_t mdone_bar = bar0 + 8u * 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 9);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile uint32_t* issued = reinterpret_cast<volatile uint32_t*>(tmem_slot + 2);  // [2]

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0: leader, issues the MMAs
  const int pair = blockIdx.x >> 1;
  const int npairs = gridDim.x >> 1;

  cluster_arrive_relaxed();  // this CTA has started
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
      mbar_init(tfull_bar(s), 1);
      mbar_init(tempty_bar(s), 2 * kF32Epi);  // every epilogue warp of both CTAs
    }
    mbar_init(mdone_bar, 1);
    *abort_flag = 0;
    issued[0] = 0;
    issued[1] = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  cluster_wait();  // and so has the peer, with which warp 1 allocates TMEM
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t full_leader0 = map_to_cta(full_bar(0), 0);
  const uint32_t abort_peer = map_to_cta(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u);
  auto raise_abort = [&]() {
    *abort_flag = 1;
    st_cluster_u32(abort_peer, 1u);
    atomicOr(p.status, kStatusPipelineTimeout);
  };

  const int num_n = p.N / 256;
  const F32Plan plan = f32_plan(p.M, p.N, slots);
  const int num_tiles = plan.tiles;
  const int num_kb = (p.K + 63) / 64;
  // plane j of A starts at row j M of the map, plane j of W at row j N; this CTA
  // brings 128 rows of A and half of the tile's rows of W
  auto load_stage = [&](int s, const F32Tile& t, int kb, uint32_t bar) {
    const uint32_t a = smem_u32(smem + s * kF32Stage);
    const int m0 = t.m0 + static_cast<int>(rank) * 128;
    const int n0 = t.n0 + static_cast<int>(rank) * (t.n / 2);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      tma_load_2d_pair(a + j * kF32Plane, &tmA, kb * 64, j * p.M + m0, bar);
      const uint32_t b = a + kF32Operand + j * kF32Plane;
      if (t.n == 256) {
        tma_load_2d_pair(b, &tmB, kb * 64, j * p.N + n0, bar);
      } else {
        for (int r = 0; r < t.n / 2; r += 32)
          tma_load_2d_pair(b + r * 128, &tmB32, kb * 64, j * p.N + n0 + r, bar);
      }
    }
  };
  auto stage_bytes = [](const F32Tile& t) {  // of both CTAs
    return static_cast<uint32_t>(2 * (kF32Operand + 3 * (t.n / 2) * 128));
  };

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------- producer
      uint32_t it = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        const F32Tile t = f32_tile(plan, tile, num_n);
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it & 1;
          if (!mbar_wait_bounded(empty_bar(s), ((it >> 1) & 1) ^ 1u, abort_flag, p.timeout_ns)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_arrive_expect_tx(full_bar(s), stage_bytes(t));
          load_stage(s, t, kb, full_leader0 + 8u * s);
        }
      }
      if (!ok) raise_abort();
      const uint32_t slot = smem_u32(const_cast<uint32_t*>(issued)) + 4u * rank;
      st_cluster_u32(map_to_cta(slot, 0), it);
      st_cluster_u32(map_to_cta(slot, 1), it);
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      // -------------------------------------------------------- MMA issuer
      uint32_t it = 0;  // one K block: one stage and one accumulator
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        const uint32_t idesc = mma_idesc(1u, f32_columns(plan, tile), 256);
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it & 1;
          const uint32_t ph = (it >> 1) & 1;
          const uint32_t a0 = smem_u32(smem + s * kF32Stage);
#pragma unroll
          for (int g = 0; g < 2 && ok; ++g) {  // accumulator g: the block's K half g
            if (!mbar_wait_bounded(tempty_bar(g), (it & 1) ^ 1u, abort_flag, p.timeout_ns) ||
                (g == 0 && !mbar_wait_bounded(full_bar(s), ph, abort_flag, p.timeout_ns))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(g * 256);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
#pragma unroll
              for (int j = 2 * g; j < 2 * g + 2; ++j)
                tc_mma_pair_f16(d_tmem, sw128_kmajor_desc(a0 + kProdA[q] * kF32Plane + 32u * j),
                                sw128_kmajor_desc(a0 + kF32Operand + kProdW[q] * kF32Plane + 32u * j),
                                idesc, (q != 0 || j != 2 * g) ? 1u : 0u);
            }
            if (g == 1) tc_commit_pair_multicast(empty_bar(s), 0x3);
            tc_commit_pair_multicast(tfull_bar(g), 0x3);
          }
          if (!ok) break;
        }
      }
      if (!ok) raise_abort();
      tc_commit_pair(mdone_bar);
      mbar_wait_bounded(mdone_bar, 0, nullptr, kF32DrainNs);
    }
  } else {
    // ---------------------------------------------------------- epilogue (both CTAs)
    const int q = warp & 3;            // TMEM lane quarter
    const int half = (warp - 2) / 4;   // half of the tile's columns
    const uint32_t tempty_leader0 = map_to_cta(tempty_bar(0), 0);
    const uint32_t trow = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    auto wait = [&](int b, uint32_t ph) {
      const bool ok = mbar_wait_bounded(tfull_bar(b), ph, abort_flag, p.timeout_ns);
      return __all_sync(0xffffffffu, ok) != 0;
    };
    auto done = [&](int b) {
      if (lane == 0) mbar_arrive_cluster(tempty_leader0 + 8u * b);
    };
    uint32_t it = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
      const int n = f32_columns(plan, tile);
      auto where = [&](int& row, int& n0) {
        const F32Tile t = f32_tile(f32_plan(p.M, p.N, slots), tile, p.N / 256);
        row = t.m0 + static_cast<int>(rank) * 128 + q * 32 + lane;
        n0 = t.n0 + t.n / 2 * half;
      };
      if (n == 256)
        ok = f32_drain<128>(p, trow + 128u * half, 2 * num_kb, it, wait, done, where);
      else if (n == 128)
        ok = f32_drain<64>(p, trow + 64u * half, 2 * num_kb, it, wait, done, where);
      else
        ok = f32_drain<32>(p, trow + 32u * half, 2 * num_kb, it, wait, done, where);
    }
    if (!ok && lane == 0) raise_abort();
  }

  // ---------------------------------------------------------- teardown
  tc_fence_before();
  cluster_sync_all();  // #1: no role issues anything new; issue counts published
  if (warp == 0 && lane == 0) {
    const uint32_t mine = issued[rank], other = issued[rank ^ 1u];
    // after an abort: copy this CTA's half of any stage the other producer
    // issued and this one did not, so that every armed phase completes
    for (uint32_t j = mine; j < other; ++j) {  // K block j of this pair's tiles
      const F32Tile t =
          f32_tile(plan, pair + static_cast<int>(j / num_kb) * npairs, num_n);
      if (rank == 0) mbar_arrive_expect_tx(full_bar(j & 1), stage_bytes(t));
      load_stage(j & 1, t, static_cast<int>(j % num_kb), full_leader0 + 8u * (j & 1));
    }
    if (rank == 0) {
      const uint32_t jmax = mine > other ? mine : other;
      for (uint32_t j = jmax > 2u ? jmax - 2u : 0u; j < jmax; ++j)
        mbar_wait_bounded(full_bar(j & 1), (j >> 1) & 1, nullptr, kF32DrainNs);
    }
  }
  tc_fence_before();
  cluster_sync_all();  // #2: every copy landed, every MMA finished
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// dst = three bf16 planes [3][N x ldd] of src [N x K], zero beyond K
// (ldd a multiple of 8).
__global__ void pack_planes_kernel(const float* __restrict__ src, int N, int K, int ldd,
                                   __nv_bfloat16* __restrict__ dst) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int per_row = ldd / 8;
  if (i >= static_cast<int64_t>(N) * per_row) return;
  const int n = static_cast<int>(i / per_row), k = static_cast<int>(i % per_row) * 8;
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = k + j < K ? src[static_cast<int64_t>(n) * K + k + j] : 0.f;
  uint4 w[3];
  f32_split8(v, w);
#pragma unroll
  for (int j = 0; j < 3; ++j)
    *reinterpret_cast<uint4*>(dst + (static_cast<size_t>(j) * N + n) * ldd + k) = w[j];
}

}  // namespace

int tc_gemm_f32_max_clusters() {
  if (cudaFuncSetAttribute(tc_gemm_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kF32Smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2, 1, 1);
  cfg.blockDim = dim3(kF32Threads, 1, 1);
  cfg.dynamicSmemBytes = kF32Smem;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tc_gemm_f32_kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_tc_gemm_f32(const CUtensorMap& tmA, const CUtensorMap& tmB,
                               const CUtensorMap& tmB32, const TcF32Params& p, int clusters,
                               cudaStream_t s) {
  if (p.M <= 0) return cudaSuccess;
  if (p.N % 256 != 0 || p.K <= 0 || clusters <= 0 ||
      3 * static_cast<int64_t>(p.M) > 0x7fffffff ||
      (p.out_f32 == nullptr) == (p.out_planes == nullptr) ||
      reinterpret_cast<uintptr_t>(p.out_f32) % 32 != 0 ||
      reinterpret_cast<uintptr_t>(p.out_planes) % 32 != 0 ||
      reinterpret_cast<uintptr_t>(p.bias) % 16 != 0)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(tc_gemm_f32_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kF32Smem);
  if (e != cudaSuccess) return e;
  const int tiles = f32_plan(p.M, p.N, clusters).tiles;
  tc_gemm_f32_kernel<<<2 * (tiles < clusters ? tiles : clusters), kF32Threads, kF32Smem, s>>>(
      tmA, tmB, tmB32, p, clusters);
  return cudaGetLastError();
}

cudaError_t launch_pack_planes(const float* src, int N, int K, int ldd, __nv_bfloat16* dst,
                               cudaStream_t s) {
  if (ldd % 8 != 0) return cudaErrorInvalidValue;
  const int64_t total = static_cast<int64_t>(N) * (ldd / 8);
  pack_planes_kernel<<<static_cast<unsigned>((total + 255) / 256), 256, 0, s>>>(src, N, K, ldd,
                                                                                dst);
  return cudaGetLastError();
}

}  // namespace ddf
