// tc_steps.cu -- the kernels of a sphere-tracing step (Sec. 4.4) whose number
// of rays only the device knows: encoding of the current points, the layers,
// the update with compaction.
//
// A trace is launched for its step limit, and after a dozen steps a few
// thousand rays are left, then a few, then none. What such steps cost is
// latency: with the general kernels some 65 us each at 512 x 6, rays or no
// rays. Here
//   * every kernel is launched with programmatic dependence on the one before
//     and passes the permission on as soon as its own predecessor is complete,
//     so starting up overlaps the predecessor's work; a step without rays is a
//     chain of kernels that read one number;
//   * a layer looks at the count and takes 128 x 256 tiles where those fill the
//     GPU, else 128 x 64 tiles, four times the CTAs with half the operand bytes
//     each, and asks for its first stages' weights before the layer before has
//     finished;
//   * encoding and update run on a fixed grid, several threads a ray.
// 65,536 rays through 51 -> 512 x 6, 128 steps allowed, 77 used: 8.40 -> 4.79 ms;
// a step with few rays 65 -> 30 us.
//
// The arithmetic and its order are those of encode_points_kernel and
// tc_gemm_kernel (128 x bn tiles, 4 epilogue warps): the same bits. In the small
// tiles the last layer writes FP32 activations and the update runs the head's
// chains over blocks of bn columns.
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "kernels.h"
#include "ptx_sm103.cuh"

namespace ddf {

namespace {

constexpr uint64_t kStDrainNs = 1000000000ull;
constexpr int kStSlots = 8;
constexpr int kStRing = 192 * 1024;
constexpr int kStA = 128 * 128;
constexpr int kStEpi = 8;
constexpr int kStThreads = 32 * (2 + kStEpi);
constexpr int kStCtrl = 256;
constexpr int kStMaxSmem = 226 * 1024;  // allowed to every kernel here, whatever the field

__device__ __forceinline__ void st_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void st_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Whether `rows` rows leave SMs without a 128 x bn tile, so that 128 x 64 tiles
// are taken. Every kernel of a step decides this alike.
__device__ __forceinline__ bool small_tiles(int rows, int N, int bn, int sms) {
  return (rows + 127) / 128 * (N / bn) < sms;
}

template <bool LAST>
__global__ void __launch_bounds__(kStThreads, 1)
    tc_step_kernel(const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmB64, const TcGemmParams p, int bn_big) {
  // the count is older than the layer before, whose start (the permission to
  // launch this kernel) came after the count's writer was complete
  __shared__ int s_rows;  // one reading for the block
  if (threadIdx.x == 0) s_rows = min(__ldcg(p.m_dev), p.M);
  __syncthreads();
  const int rows = s_rows;
  const bool small = small_tiles(rows, p.N, bn_big, static_cast<int>(gridDim.x));
  const int bn = small ? 64 : bn_big;
  const int num_n = p.N / bn;
  const int tiles = (rows + 127) / 128 * num_n;
  if (static_cast<int>(blockIdx.x) >= tiles) {  // still a link of the chain
    if (threadIdx.x == 0) {
      st_wait();
      st_launch_dependents();
    }
    return;
  }
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStRing);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStSlots + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * kStSlots + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * kStSlots + 2 + b); };
  const uint32_t mdone_bar = bar0 + 8u * (2 * kStSlots + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStSlots + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stage_bytes = kStA + bn * 128;
  const int slots = kStRing / stage_bytes;  // 4 (256), 6 (128) or 8 (64)
  const int num_kb = (p.K + 63) / 64;
  const CUtensorMap* const mapB = small ? &tmB64 : &tmB;
  auto stage = [&](int s) { return smem_u32(smem + s * stage_bytes); };
  auto raise_abort = [&]() {
    *abort_flag = 1;
    atomicOr(p.status, kStatusPipelineTimeout);
  };
  const int ahead = num_kb < slots ? num_kb : slots;  // weight stages requested early

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStSlots; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull_bar(b), 1);
      mbar_init(tempty_bar(b), kStEpi);
    }
    mbar_init(mdone_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    const int n0 = static_cast<int>(blockIdx.x) % num_n * bn;
    for (int s = 0; s < ahead; ++s) {
      mbar_arrive_expect_tx(full_bar(s), stage_bytes);
      tma_load_2d(stage(s) + kStA, mapB, s * 64, n0, full_bar(s));
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  const EpiVectors ev = stage_epi_vectors(p, reinterpret_cast<float*>(smem + kStRing + kStCtrl));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------- producer
      st_wait();
      st_launch_dependents();
      int slot = 0, issued = 0;
      uint32_t ph = 0;
      bool ok = true, first = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int m0 = tile / num_n * 128, n0 = tile % num_n * bn;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!(first && kb < ahead)) {
            if (!mbar_wait_bounded(empty_bar(slot), ph ^ 1u, abort_flag, p.timeout_ns)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(full_bar(slot), stage_bytes);
            tma_load_2d(stage(slot) + kStA, mapB, kb * 64, n0, full_bar(slot));
          }
          tma_load_2d(stage(slot), &tmA, kb * 64, m0, full_bar(slot));
          if (++slot == slots) {
            slot = 0;
            ph ^= 1u;
          }
          if (issued < slots) ++issued;
        }
        first = false;
      }
      if (!ok) raise_abort();
      for (; issued > 0; --issued) {  // no exit with a copy in flight
        if (--slot < 0) {
          slot = slots - 1;
          ph ^= 1u;
        }
        mbar_wait_bounded(full_bar(slot), ph, nullptr, kStDrainNs);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // -------------------------------------------------------- MMA issuer
      const uint32_t idesc = mma_idesc(1u, bn, 128);
      int slot = 0, local = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++local) {
        const int b = local & 1;
        if (!mbar_wait_bounded(tempty_bar(b), ((local >> 1) & 1) ^ 1u, abort_flag, p.timeout_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(b * 256);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait_bounded(full_bar(slot), ph, abort_flag, p.timeout_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = sw128_kmajor_desc(stage(slot));
          const uint64_t bd = sw128_kmajor_desc(stage(slot) + kStA);
#pragma unroll
          for (int j = 0; j < 4; ++j)  // 32 bytes of K: 2 in units of 16 bytes
            tc_mma_f16(d_tmem, ad + 2 * j, bd + 2 * j, idesc, (kb != 0 || j != 0) ? 1u : 0u);
          tc_commit(empty_bar(slot));
          if (++slot == slots) {
            slot = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        tc_commit(tfull_bar(b));
      }
      if (!ok) raise_abort();
      tc_commit(mdone_bar);
      mbar_wait_bounded(mdone_bar, 0, nullptr, kStDrainNs);
    }
  } else {
    // ---------------------------------------------------------- epilogue
    const int q = warp & 3, half = (warp - 2) / 4;
    int local = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++local) {
      const int b = local & 1;
      bool ok = mbar_wait_bounded(tfull_bar(b), (local >> 1) & 1, abort_flag, p.timeout_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) raise_abort();
        break;
      }
      tc_fence_after();
      if (local == 0) st_wait();  // the outputs replace what the layer before read
      const int n_blk = tile % num_n, n0 = n_blk * bn;
      const int row = tile / num_n * 128 + q * 32 + lane;
      const bool row_ok = row < rows;
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                             static_cast<uint32_t>(b * 256);
      const int chunks = bn / 64;  // 32-column chunks of this warp's half
      float h0 = 0.f, h1 = 0.f;
      if (!LAST) {
        epi_row<false>(p, ev, tbase, row, row_ok, n0, half * chunks, (half + 1) * chunks, h0, h1);
      } else if (small) {
        uint32_t v[32];
        tmem_ld32(tbase + 32u * half, v);
        tmem_wait_ld_regs(v);
        float x[32];
        epi_affine32(ev, v, n0 + 32 * half, x);
        if (row_ok) {
          uint32_t w[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(fmaxf(x[j], 0.f));
          float* dst = p.out_f32 + static_cast<size_t>(row) * p.N + n0 + 32 * half;
#pragma unroll
          for (int j = 0; j < 4; ++j) st_global_256(dst + 8 * j, w + 8 * j);
        }
      } else if (half == 0) {  // the block's chain is one thread's
        epi_row<false, true>(p, ev, tbase, row, row_ok, n0, 0, bn / 32, h0, h1);
        if (row_ok) p.head_part[static_cast<size_t>(n_blk) * p.M + row] = make_float2(h0, h1);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar(b));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// The current points' encoding (as encode_points_kernel), three threads a ray,
// on a fixed grid. Also clears the count this step's update will write.
constexpr int kStEncRays = 64;

__global__ void __launch_bounds__(3 * kStEncRays)
step_encode_kernel(const __grid_constant__ RaySoA rays, const float* __restrict__ t,
                   const int* __restrict__ idx, const int* __restrict__ count,
                   int* __restrict__ next_count, int cap, int L, int ld,
                   __nv_bfloat16* __restrict__ out) {
  extern __shared__ __align__(16) __nv_bfloat16 esm[];  // [kStEncRays][ld + 8]
  st_wait();
  st_launch_dependents();
  const int rows = min(__ldcg(count), cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) *next_count = 0;
  const int sld = ld + 8;
  const int c = threadIdx.x / kStEncRays, j = threadIdx.x % kStEncRays;
  for (int r0 = blockIdx.x * kStEncRays; r0 < rows; r0 += gridDim.x * kStEncRays) {
    const int m = min(rows - r0, kStEncRays);
    if (j < m) {
      const int i = __ldcg(idx + r0 + j);
      const float e = fmaf(__ldcg(t + i), rays.p[3 + c][i], rays.p[c][i]);
      __nv_bfloat16* row = esm + j * sld;
      row[c] = __float2bfloat16_rn(e);
      for (int k = 0; k < L; ++k) {
        float sn, cs;
        sincospif(e * __int_as_float((127 + k) << 23), &sn, &cs);  // 2^k exactly
        row[3 + 2 * (c * L + k)] = __float2bfloat16_rn(sn);
        row[4 + 2 * (c * L + k)] = __float2bfloat16_rn(cs);
      }
      if (c == 0)
        for (int col = 3 + 6 * L; col < ld; ++col) row[col] = __float2bfloat16_rn(0.f);
    }
    __syncthreads();
    const int per_row = ld / 8;
    for (int q = threadIdx.x; q < m * per_row; q += blockDim.x) {
      const int r = q / per_row, col = (q - r * per_row) * 8;
      *reinterpret_cast<uint4*>(out + static_cast<int64_t>(r0 + r) * ld + col) =
          *reinterpret_cast<const uint4*>(esm + r * sld + col);
    }
    __syncthreads();
  }
}

// The step's outcome per active ray: s = the head's sum, steps += 1; s < eps is a
// hit; else t += s, and the ray stays active unless t > t_max or it has used
// max_steps evaluations. On a fixed grid of 256-thread blocks; `small_tiles` decides where s comes from: the head partials
// of the 128 x bn tiles, or chains over X here, a block of bn columns a thread.
constexpr int kStUpdThreads = 256;
constexpr int kStUpdRays = 16;  // rays of a block at a time in the small case

__global__ void __launch_bounds__(kStUpdThreads)
step_update_kernel(const __grid_constant__ StepUpdate u) {
  extern __shared__ float usm[];
  st_wait();
  st_launch_dependents();
  const int cnt = min(__ldcg(u.count_in), u.cap);
  const int lane = threadIdx.x & 31;
  const float hb = __ldg(u.head_b);
  // one ray's step; the whole warp takes part in the compaction
  auto finish = [&](bool mine, int j, float s) {
    bool keep = false;
    int i = 0;
    if (mine) {
      i = __ldcg(u.idx_in + j);
      const int st = u.steps[i] + 1;
      u.steps[i] = st;
      if (s < u.eps) {
        u.hit[i] = 1;
      } else {
        const float tn = u.t[i] + s;
        u.t[i] = tn;
        keep = !(tn > u.t_max) && st < u.max_steps;
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    int base = 0;
    if (lane == 0 && m != 0u) base = atomicAdd(u.count_out, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (keep) u.idx_out[base + __popc(m & ((1u << lane) - 1u))] = i;
  };
  const int nb = u.N / u.bn;
  if (!small_tiles(cnt, u.N, u.bn, u.sms)) {
    for (int j0 = blockIdx.x * kStUpdThreads; j0 < cnt; j0 += gridDim.x * kStUpdThreads) {
      const int j = j0 + static_cast<int>(threadIdx.x);
      float s = hb;
      if (j < cnt)
        for (int b = 0; b < nb; ++b) s += __ldcg(&u.part[static_cast<size_t>(b) * u.cap + j].x);
      finish(j < cnt, j, s);
    }
    return;
  }
  const int ldb = u.bn + 1;         // chains of one warp on different banks
  float* sw = usm;                  // [nb][ldb]
  float* sx = sw + nb * ldb;        // [kStUpdRays][nb][ldb]
  float* sp = sx + kStUpdRays * nb * ldb;  // [kStUpdRays][nb]
  for (int j0 = blockIdx.x * kStUpdRays; j0 < cnt; j0 += gridDim.x * kStUpdRays) {
    const int m = min(cnt - j0, kStUpdRays);
    for (int i = threadIdx.x; i < u.N; i += kStUpdThreads)
      sw[(i / u.bn) * ldb + i % u.bn] = __ldg(u.head_w + i);
    for (int i = threadIdx.x; i < m * u.N / 4; i += kStUpdThreads) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(u.x + static_cast<size_t>(j0) * u.N) + i);
      float* d = sx + (4 * i / u.bn) * ldb + 4 * i % u.bn;
      d[0] = x.x;
      d[1] = x.y;
      d[2] = x.z;
      d[3] = x.w;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < m * nb; k += kStUpdThreads) {
      const float* x = sx + k * ldb;
      const float* w = sw + (k % nb) * ldb;
      float h = 0.f;
#pragma unroll 16
      for (int c = 0; c < u.bn; ++c) h = fmaf(x[c], w[c], h);
      sp[k] = h;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      float s = hb;
      if (static_cast<int>(threadIdx.x) < m)
        for (int b = 0; b < nb; ++b) s += sp[threadIdx.x * nb + b];
      finish(static_cast<int>(threadIdx.x) < m, j0 + threadIdx.x, s);
    }
    __syncthreads();
  }
}

template <typename... A>
cudaError_t launch_chained(void (*kern)(A...), bool first, int grid, int block, int smem,
                           cudaStream_t s, A... args) {
  if (smem > kStMaxSmem) return cudaErrorInvalidValue;
  if (first) {  // a thousand launches follow: not on each of them
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kStMaxSmem);
    if (e != cudaSuccess) return e;
  }
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

}  // namespace

int64_t step_small_rows(int N, int bn, int sms) { return 128 * (static_cast<int64_t>(sms) / (N / bn) + 1); }

cudaError_t launch_step_encode(const RaySoA& rays, const float* t, const int* idx, const int* count,
                               int* next_count, int cap, int L, int ld, __nv_bfloat16* out, int sms,
                               bool first, cudaStream_t s) {
  if (cap <= 0 || ld % 8 != 0) return cudaErrorInvalidValue;
  const int blocks = (cap + kStEncRays - 1) / kStEncRays;
  return launch_chained<RaySoA, const float*, const int*, const int*, int*, int, int, int,
                        __nv_bfloat16*>(step_encode_kernel, first, blocks < 4 * sms ? blocks : 4 * sms,
                                        3 * kStEncRays, kStEncRays * (ld + 8) * 2, s, rays, t, idx,
                                        count, next_count, cap, L, ld, out);
}

cudaError_t launch_step_layer(const CUtensorMap& tmA, const CUtensorMap& tmB,
                              const CUtensorMap& tmB64, const TcGemmParams& p, int bn, int sms,
                              bool first, cudaStream_t s) {
  const bool last = p.mode == 1;
  if (p.m_dev == nullptr || (bn != 128 && bn != 256) || p.N % bn != 0 || p.bias == nullptr ||
      (last && (p.head_w == nullptr || p.head_part == nullptr || p.out_f32 == nullptr ||
                reinterpret_cast<uintptr_t>(p.out_f32) % 32 != 0)) ||
      !epi_out_aligned(p, false))
    return cudaErrorInvalidValue;
  const int smem = kStRing + kStCtrl + epi_vector_bytes(p.N) + 1024;
  return last ? launch_chained<CUtensorMap, CUtensorMap, CUtensorMap, TcGemmParams, int>(
                    tc_step_kernel<true>, first, sms, kStThreads, smem, s, tmA, tmB, tmB64, p, bn)
              : launch_chained<CUtensorMap, CUtensorMap, CUtensorMap, TcGemmParams, int>(
                    tc_step_kernel<false>, first, sms, kStThreads, smem, s, tmA, tmB, tmB64, p, bn);
}

cudaError_t launch_step_update(const StepUpdate& u, bool first, cudaStream_t s) {
  if (u.cap <= 0 || u.N % u.bn != 0 || u.bn % 4 != 0) return cudaErrorInvalidValue;
  const int nb = u.N / u.bn;
  const int smem = ((1 + kStUpdRays) * nb * (u.bn + 1) + kStUpdRays * nb) * 4;
  const int blocks = (u.cap + kStUpdRays - 1) / kStUpdRays;
  return launch_chained<StepUpdate>(step_update_kernel, first, blocks < 2 * u.sms ? blocks : 2 * u.sms,
                                    kStUpdThreads, smem, s, u);
}

}  // namespace ddf
