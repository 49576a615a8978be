// tc_small.cu -- the layers of a wide field for a few hundred rays (bf16 and
// e4m3), the encoding and the heads that go with them.
//
// With one or two row blocks the 128 x 256 tile of tc_gemm.cu gives ten CTAs
// at width 1280, and each takes in 960 KB of operands through one SM's port:
// 16 us a layer whatever the batch, 8 layers one after another. Here a CTA
// computes 128 x 64 (480 KB, four times the CTAs), and the layers are launched
// with programmatic dependence: a CTA sets itself up and requests the first
// nine stages' weights while the layer before is still running, and waits for
// that layer (griddepcontrol.wait) only before its first activations.
// Measured at 1280 x 8, a whole call: 193 rays 127 -> 70 us (e4m3 112 -> 50), 1,500
// rays (two waves of tiles) 130 -> 129 (113 -> 90); at 512 x 6, 1,000 rays 75 -> 40.
//
// The arithmetic is that of the default tiles, in their order: K ascending in
// the same steps, the same epilogue expressions. The head's chains run over
// blocks of 256 (or 128) columns and so cannot be folded into 64-column tiles;
// the last layer writes its FP32 activations and small_heads_kernel runs the
// chains. The results are the same bits.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "epilogue.cuh"
#include "heads.cuh"
#include "kernels.h"
#include "ptx_sm103.cuh"

namespace ddf {

namespace {

constexpr uint64_t kSmDrainNs = 1000000000ull;
constexpr int kSmStages = 9;
constexpr int kSmA = 128 * 128;   // 128 rows x 128 bytes of K
constexpr int kSmB = 64 * 128;
constexpr int kSmStage = kSmA + kSmB;
constexpr int kSmEpi = 8;         // epilogue warps: a lane quarter and 32 columns each
constexpr int kSmThreads = 32 * (2 + kSmEpi);
constexpr int kSmCtrl = 256;
constexpr int kSmSmem = kSmStages * kSmStage + kSmCtrl + 2 * 64 * 4 + 1024;
static_assert(kSmSmem <= 227 * 1024, "shared memory of one CTA");

// This grid's memory may be used by the next one's prologue only; it has what
// the previous grid wrote once the wait returns.
__device__ __forceinline__ void grid_dependents_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

enum SmallOut { kOutBf16 = 0, kOutFp8 = 1, kOutF32 = 2 };

template <bool IN_FP8, int OUT>
__global__ void __launch_bounds__(kSmThreads, 1)
    tc_small_kernel(const __grid_constant__ CUtensorMap tmA,
                    const __grid_constant__ CUtensorMap tmB, const TcGemmParams p) {
  constexpr int BK = IN_FP8 ? 128 : 64;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kSmStages * kSmStage);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kSmStages + s); };
  const uint32_t done_bar = bar0 + 8u * (2 * kSmStages);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kSmStages + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* svec = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kSmCtrl);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_n = p.N / 64;
  const int m0 = static_cast<int>(blockIdx.x) / num_n * 128;
  const int n0 = static_cast<int>(blockIdx.x) % num_n * 64;
  const int num_kb = (p.K + BK - 1) / BK;
  const int first = num_kb < kSmStages ? num_kb : kSmStages;
  auto a_dst = [&](int s) { return smem_u32(smem + s * kSmStage); };
  auto raise_abort = [&]() {
    *abort_flag = 1;
    atomicOr(p.status, kStatusPipelineTimeout);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kSmStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    for (int s = 0; s < first; ++s) {  // weights do not depend on the layer before
      mbar_arrive_expect_tx(full_bar(s), kSmStage);
      tma_load_2d(a_dst(s) + kSmA, &tmB, s * BK, n0, full_bar(s));
    }
    grid_dependents_launch();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 64);
    tmem_relinquish();
  }
  // the tile's bias and column scales, an output's power-of-two scale folded in
  if (threadIdx.x >= 64 && threadIdx.x < 128) {
    const int i = threadIdx.x - 64;
    svec[i] = __ldg(p.bias + n0 + i) * p.out_scale;
    if (p.col_scale != nullptr) svec[64 + i] = __ldg(p.col_scale + n0 + i) * p.out_scale;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------- producer
      grid_dependency_wait();
      for (int s = 0; s < first; ++s) tma_load_2d(a_dst(s), &tmA, s * BK, m0, full_bar(s));
      bool ok = true;
      int it = first;
      for (; it < num_kb; ++it) {
        const int s = it % kSmStages;
        if (!mbar_wait_bounded(empty_bar(s), ((it / kSmStages) & 1) ^ 1u, abort_flag,
                               p.timeout_ns)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(full_bar(s), kSmStage);
        tma_load_2d(a_dst(s) + kSmA, &tmB, it * BK, n0, full_bar(s));
        tma_load_2d(a_dst(s), &tmA, it * BK, m0, full_bar(s));
      }
      if (!ok) raise_abort();
      // no exit with a copy in flight
      for (int j = it > kSmStages ? it - kSmStages : 0; j < it; ++j)
        mbar_wait_bounded(full_bar(j % kSmStages), (j / kSmStages) & 1, nullptr, kSmDrainNs);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // -------------------------------------------------------- MMA issuer
      constexpr uint32_t idesc = mma_idesc(IN_FP8 ? 0u : 1u, 64, 128);
      bool ok = true;
      for (int it = 0; it < num_kb; ++it) {
        const int s = it % kSmStages;
        if (!mbar_wait_bounded(full_bar(s), (it / kSmStages) & 1, abort_flag, p.timeout_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t ad = sw128_kmajor_desc(a_dst(s) + 32u * j);
          const uint64_t bd = sw128_kmajor_desc(a_dst(s) + kSmA + 32u * j);
          const uint32_t acc = (it != 0 || j != 0) ? 1u : 0u;
          if constexpr (IN_FP8)
            tc_mma_f8(tmem, ad, bd, idesc, acc);
          else
            tc_mma_f16(tmem, ad, bd, idesc, acc);
        }
        tc_commit(empty_bar(s));
      }
      if (!ok) raise_abort();
      tc_commit(done_bar);  // arrives once every MMA above has finished
      mbar_wait_bounded(done_bar, 0, nullptr, kSmDrainNs);
    }
  } else {
    // ---------------------------------------------------------- epilogue
    const int q = warp & 3, half = (warp - 2) / 4;
    // as long as the MMA issuer may take over all its stages, and then some
    bool ok = mbar_wait_bounded(done_bar, 0, abort_flag, p.timeout_ns) && *abort_flag == 0;
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) {
      if (lane == 0) raise_abort();
    } else {
      tc_fence_after();
      grid_dependency_wait();  // the output buffer is the layer before's input
      uint32_t v[32];
      tmem_ld32(tmem + (static_cast<uint32_t>(q * 32) << 16) + 32u * half, v);
      tmem_wait_ld_regs(v);
      const EpiVectors ev{svec, p.col_scale != nullptr ? svec + 64 : nullptr, nullptr, nullptr,
                          p.out_scale};
      float x[32];
      epi_affine32(ev, v, 32 * half, x);
      const int row = m0 + q * 32 + lane;
      if (row < p.M) {
        const size_t at = static_cast<size_t>(row) * p.ldo + n0 + 32 * half;
        if constexpr (OUT == kOutF32) {
          uint32_t w[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(fmaxf(x[j], 0.f));
#pragma unroll
          for (int j = 0; j < 4; ++j) st_global_256(p.out_f32 + at + 8 * j, w + 8 * j);
        } else if constexpr (OUT == kOutFp8) {
          uint32_t w[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            w[k] = epi_pack_e4m3x4_relu(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
          st_global_256(static_cast<uint8_t*>(p.out) + at, w);
        } else {
          uint32_t w[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) w[k] = epi_pack_bf16x2_relu(x[2 * k], x[2 * k + 1]);
          st_global_256(static_cast<__nv_bfloat16*>(p.out) + at, w);
          st_global_256(static_cast<__nv_bfloat16*>(p.out) + at + 16, w + 8);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 64);
  }
}

// The sinusoidal encoding of encode_kernel (simt.cu) with six threads a ray,
// one coordinate each: with one, its 60 sin / cos pairs in a row take 7 us.
constexpr int kSmEncRays = 32;

__global__ void __launch_bounds__(6 * kSmEncRays)
small_encode_kernel(const __grid_constant__ RaySoA rays, int64_t M, int L, int ld,
                    __nv_bfloat16* __restrict__ out) {
  grid_dependents_launch();
  const int c = threadIdx.x / kSmEncRays;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * kSmEncRays + threadIdx.x % kSmEncRays;
  if (r >= M) return;
  __nv_bfloat16* row = out + r * ld;
  const float e = ray_ld(rays, c, r);
  row[c] = __float2bfloat16_rn(e);
  uint32_t* pair = reinterpret_cast<uint32_t*>(row + 6) + c * L;  // ld is a multiple of 8
  for (int k = 0; k < L; ++k) {
    float sn, cs;
    sincospif(e * __int_as_float((127 + k) << 23), &sn, &cs);  // 2^k exactly
    pair[k] = epi_pack_bf16x2(sn, cs);
  }
  if (c == 0)
    for (int col = 6 + 12 * L; col < ld; col += 2) *reinterpret_cast<uint32_t*>(row + col) = 0u;
}

// Heads from FP32 activations X [M x W]: per ray, output and block of `blk`
// columns one chain of FMAs in column order, then the blocks in order, as the
// default tiles and finish_heads_kernel add them.
constexpr int kSmHeadRays = 8;
__host__ __device__ constexpr int sm_heads_bytes(int nb, int blk) {
  return ((2 + kSmHeadRays) * nb * (blk + 1) + kSmHeadRays * nb * 2) * 4;
}
// of the widest field, in blocks of 128
constexpr int kSmHeadsLimit = sm_heads_bytes(kMaxStagedColumns / 128, 128);

__global__ void __launch_bounds__(256)
small_heads_kernel(const float* __restrict__ X, int M, int W, int blk,
                   const float* __restrict__ wo, const float* __restrict__ bo,
                   const __grid_constant__ HeadOut o) {
  extern __shared__ float hsm[];
  const int nb = W / blk, ldb = blk + 1;  // chains of one warp on different banks
  float* sw = hsm;                        // [2][nb][ldb]
  float* sx = sw + 2 * nb * ldb;          // [kSmHeadRays][nb][ldb]
  float* sp = sx + kSmHeadRays * nb * ldb;  // [kSmHeadRays][nb][2]
  for (int i = threadIdx.x; i < 2 * W; i += blockDim.x)
    sw[(i / blk) * ldb + i % blk] = __ldg(wo + i);
  grid_dependency_wait();
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * kSmHeadRays;
  const int rows = static_cast<int>(M - r0 < kSmHeadRays ? M - r0 : kSmHeadRays);
  for (int i = threadIdx.x; i < rows * W / 4; i += blockDim.x) {
    const float4 x = __ldcg(reinterpret_cast<const float4*>(X + r0 * W) + i);
    float* d = sx + (4 * i / blk) * ldb + 4 * i % blk;
    d[0] = x.x;
    d[1] = x.y;
    d[2] = x.z;
    d[3] = x.w;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < rows * nb * 2; i += blockDim.x) {
    const int k = i >> 1, out = i & 1, b = k % nb;
    const float* x = sx + k * ldb;
    const float* w = sw + (out * nb + b) * ldb;
    float h = 0.f;
#pragma unroll 16
    for (int j = 0; j < blk; ++j) h = fmaf(x[j], w[j], h);
    sp[i] = h;
  }
  __syncthreads();
  if (static_cast<int>(threadIdx.x) < rows) {
    float z0 = 0.f, z1 = 0.f;
    for (int b = 0; b < nb; ++b) {
      z0 += sp[(threadIdx.x * nb + b) * 2];
      z1 += sp[(threadIdx.x * nb + b) * 2 + 1];
    }
    write_heads(o, r0 + threadIdx.x, z0 + bo[0], z1 + bo[1]);
  }
}

template <typename... A>
cudaError_t launch_dependent(void (*kern)(A...), int grid, int block, int smem, cudaStream_t s,
                             A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <bool IN_FP8, int OUT>
cudaError_t launch_layer(const CUtensorMap& tmA, const CUtensorMap& tmB, const TcGemmParams& p,
                         cudaStream_t s) {
  auto kern = tc_small_kernel<IN_FP8, OUT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmSmem);
  if (e != cudaSuccess) return e;
  return launch_dependent<CUtensorMap, CUtensorMap, TcGemmParams>(
      kern, (p.M + 127) / 128 * (p.N / 64), kSmThreads, kSmSmem, s, tmA, tmB, p);
}

}  // namespace

cudaError_t load_small_kernels(bool fp8) {
  // e4m3: the first layer, the others, the last one, a single one
  const void* bf16[] = {(const void*)tc_small_kernel<false, kOutBf16>,
                        (const void*)tc_small_kernel<false, kOutF32>};
  const void* e4m3[] = {(const void*)tc_small_kernel<false, kOutFp8>,
                        (const void*)tc_small_kernel<true, kOutFp8>,
                        (const void*)tc_small_kernel<true, kOutF32>,
                        (const void*)tc_small_kernel<false, kOutF32>};
  const void* both[] = {(const void*)small_encode_kernel, (const void*)small_heads_kernel};
  cudaError_t e = load_kernels(both, 2);
  if (e == cudaSuccess) e = fp8 ? load_kernels(e4m3, 4) : load_kernels(bf16, 2);
  return e;
}

cudaError_t launch_small_layer(bool in_fp8, bool out_fp8, const CUtensorMap& tmA,
                               const CUtensorMap& tmB, const TcGemmParams& p, cudaStream_t s) {
  if (p.M <= 0) return cudaSuccess;
  if (p.N % 64 != 0 || p.bias == nullptr || (p.out_f32 == nullptr) == (p.out == nullptr) ||
      reinterpret_cast<uintptr_t>(p.out_f32) % 32 != 0 || !epi_out_aligned(p, out_fp8))
    return cudaErrorInvalidValue;
  if (p.out_f32 != nullptr)
    return in_fp8 ? launch_layer<true, kOutF32>(tmA, tmB, p, s)
                  : launch_layer<false, kOutF32>(tmA, tmB, p, s);
  if (out_fp8)
    return in_fp8 ? launch_layer<true, kOutFp8>(tmA, tmB, p, s)
                  : launch_layer<false, kOutFp8>(tmA, tmB, p, s);
  if (in_fp8) return cudaErrorInvalidValue;
  return launch_layer<false, kOutBf16>(tmA, tmB, p, s);
}

cudaError_t launch_small_encode(const RaySoA& rays, int64_t M, int L, int ld, __nv_bfloat16* out,
                                cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  small_encode_kernel<<<static_cast<unsigned>((M + kSmEncRays - 1) / kSmEncRays), 6 * kSmEncRays,
                        0, s>>>(rays, M, L, ld, out);
  return cudaGetLastError();
}

cudaError_t launch_small_heads(const float* X, int M, int W, int blk, const float* wo,
                               const float* bo, const HeadOut& o, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (W % blk != 0 || blk % 4 != 0) return cudaErrorInvalidValue;
  const int nb = W / blk;
  const int smem = sm_heads_bytes(nb, blk);
  if (smem > kSmHeadsLimit) return cudaErrorInvalidValue;
  // a constant: the limit is the function's, and host threads with other fields set it too
  cudaError_t e = cudaFuncSetAttribute(
      small_heads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmHeadsLimit);
  if (e != cudaSuccess) return e;
  return launch_dependent<const float*, int, int, int, const float*, const float*, HeadOut>(
      small_heads_kernel, (M + kSmHeadRays - 1) / kSmHeadRays, 256, smem, s, X, M, W, blk, wo, bo,
      o);
}

}  // namespace ddf
