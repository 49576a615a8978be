// tc_steps.cu -- layers whose cost is latency and the last wave of tiles: the
// steps of a sphere trace (Sec. 4.4), whose number of rays only the device
// knows, and queries of a few thousand rays (bf16 and e4m3).
//
// A trace is launched for its step limit, and after a dozen steps a few
// thousand rays are left, then a few, then none; with the general kernels a step
// costs some 65 us at 512 x 6, rays or no rays. A query of 4,099 rays through
// 1280 x 8 has 165 tiles a layer for 152 SMs: two waves, the second nearly empty,
// and between two layers the SMs drain and fill. Here
//   * every kernel is launched with programmatic dependence on the one before
//     and passes the permission on as soon as its own predecessor is complete,
//     so starting up overlaps the predecessor's work; a step without rays is a
//     chain of kernels that read one number;
//   * a layer works out its tiles from the rows (tile_plan): whole waves of
//     128 x 256 tiles, and the rest, if it is little, in tiles of 64 columns; it
//     asks for its first stages' weights before the layer before has finished;
//   * a trace's encoding and update run on a fixed grid, several threads a ray.
// 65,536 rays through 51 -> 512 x 6, 128 steps allowed, 77 used: 8.44 -> 4.73 ms; a
// step with few rays 65 -> 30 us. 4,099 rays through 126 -> 1280 x 8 in caller's
// scratch 200 -> 128 us; e4m3 147 -> 93; 8,192 rays 254 -> 184. What bounds a wave
// is the operands' way into the SM, 48 KB for 524 cycles of MMAs.
//
// The arithmetic and its order are those of the encoders and tc_gemm_kernel (128
// x bn tiles, 4 epilogue warps): the same bits. A head's chain runs over a block
// of bn columns, so the last layer writes a split tile's FP32 activations, and
// the update or the heads run the chains.
#include <cuda_bf16.h>

#include <algorithm>

#include "epilogue.cuh"
#include "heads.cuh"
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

template <bool IN_FP8, bool OUT_FP8, bool LAST>
__global__ void __launch_bounds__(kStThreads, 1)
    tc_step_kernel(const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmB64, const TcGemmParams p,
                   const StepTiles st) {
  constexpr int BK = IN_FP8 ? 128 : 64;
  int rows = p.M;
  if (p.m_dev != nullptr) {
    // the count is older than the layer before, whose start (the permission to
    // launch this kernel) came after the count's writer was complete
    __shared__ int s_rows;  // one reading for the block
    if (threadIdx.x == 0) s_rows = min(__ldcg(p.m_dev), p.M);
    __syncthreads();
    rows = s_rows;
  }
  const TilePlan plan = tile_plan(rows, st);
  if (static_cast<int>(blockIdx.x) >= plan.tiles) {  // still a link of the chain
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
  const int num_n = st.num_n, bn = 1 << st.lg_bn;
  const int slot_bytes = kStA + (plan.big > 0 ? bn : 64) * 128;
  const int slots = kStRing / slot_bytes;  // 4 (256 columns), 6 (128) or 8 (64)
  const int num_kb = (p.K + BK - 1) / BK;
  // tile t: row block, first column, columns
  struct Tile {
    int m0, n0, bn;
  };
  auto tile_at = [&](int t) {
    int sub = 0, w = bn;
    if (t >= plan.big) {
      sub = (t - plan.big) & ((1 << plan.lg_split) - 1);
      t = plan.big + ((t - plan.big) >> plan.lg_split);
      w = 64;
    }
    const int m = t / num_n;
    return Tile{m * 128, (t - m * num_n) * bn + sub * w, w};
  };
  auto load_b = [&](uint32_t dst, int kb, const Tile& t, uint32_t bar) {
    mbar_arrive_expect_tx(bar, kStA + t.bn * 128);
    tma_load_2d(dst, t.bn == bn ? &tmB : &tmB64, kb * BK, t.n0, bar);
  };
  auto stage = [&](int s) { return smem_u32(smem + s * slot_bytes); };
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
    const Tile t = tile_at(blockIdx.x);
    for (int s = 0; s < ahead; ++s) load_b(stage(s) + kStA, s, t, full_bar(s));
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
      for (int tile = blockIdx.x; tile < plan.tiles && ok; tile += gridDim.x) {
        const Tile t = tile_at(tile);
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!(first && kb < ahead)) {
            if (!mbar_wait_bounded(empty_bar(slot), ph ^ 1u, abort_flag, p.timeout_ns)) {
              ok = false;
              break;
            }
            load_b(stage(slot) + kStA, kb, t, full_bar(slot));
          }
          tma_load_2d(stage(slot), &tmA, kb * BK, t.m0, full_bar(slot));
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
      int slot = 0, local = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < plan.tiles && ok; tile += gridDim.x, ++local) {
        const int b = local & 1;
        const uint32_t idesc =
            mma_idesc(IN_FP8 ? 0u : 1u, tile < plan.big ? bn : 64, 128);
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
          for (int j = 0; j < 4; ++j) {  // 32 bytes of K: 2 in units of 16 bytes
            const uint32_t acc = (kb != 0 || j != 0) ? 1u : 0u;
            if constexpr (IN_FP8)
              tc_mma_f8(d_tmem, ad + 2 * j, bd + 2 * j, idesc, acc);
            else
              tc_mma_f16(d_tmem, ad + 2 * j, bd + 2 * j, idesc, acc);
          }
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
    for (int tile = blockIdx.x; tile < plan.tiles; tile += gridDim.x, ++local) {
      const int b = local & 1;
      bool ok = mbar_wait_bounded(tfull_bar(b), (local >> 1) & 1, abort_flag, p.timeout_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) raise_abort();
        break;
      }
      tc_fence_after();
      if (local == 0) st_wait();  // the outputs replace what the layer before read
      const Tile t = tile_at(tile);
      const int row = t.m0 + q * 32 + lane;
      const bool row_ok = row < rows;
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                             static_cast<uint32_t>(b * 256);
      const int chunks = t.bn / 64;  // 32-column chunks of this warp's half
      float h0 = 0.f, h1 = 0.f;
      if (!LAST) {
        epi_row<OUT_FP8>(p, ev, tbase, row, row_ok, t.n0, half * chunks, (half + 1) * chunks, h0,
                         h1);
      } else if (t.bn < bn) {  // a part of a block: its FP32 activations
        const int blk = (tile - plan.big) >> plan.lg_split;
        float* dst = p.out_f32 + (static_cast<size_t>(blk) * 128 + q * 32 + lane) * bn +
                     (t.n0 & (bn - 1));
        uint32_t v[32];
        tmem_ld32(tbase + 32u * half, v);
        tmem_wait_ld_regs(v);
        float x[32];
        epi_affine32(ev, v, t.n0 + 32 * half, x);
        if (row_ok) {
          uint32_t w[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(fmaxf(x[j], 0.f));
#pragma unroll
          for (int j = 0; j < 4; ++j) st_global_256(dst + 32 * half + 8 * j, w + 8 * j);
        }
      } else if (half == 0) {  // the block's chain is one thread's
        epi_row<false, true>(p, ev, tbase, row, row_ok, t.n0, 0, bn / 32, h0, h1);
        if (row_ok)
          p.head_part[static_cast<size_t>(t.n0 >> st.lg_bn) * p.M + row] = make_float2(h0, h1);
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
// max_steps evaluations. On a fixed grid of 256-thread blocks. The tile plan of the
// count decides where s comes from: rows whose tiles were all whole add up the
// head partials these left, the others run the chains of their split tiles here
// over X, a block of bn columns a thread.
constexpr int kStUpdThreads = 256;
constexpr int kStUpdRays = 16;  // rays of a block at a time where tiles were split

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
  const int nb = u.tiles.num_n, lg = u.tiles.lg_bn, bn = 1 << lg;
  const TilePlan plan = tile_plan(cnt, u.tiles);
  // rows of partials only
  const int whole = plan.lg_split == 0 ? cnt : min(cnt, plan.big / nb * 128);
  for (int j0 = blockIdx.x * kStUpdThreads; j0 < whole; j0 += gridDim.x * kStUpdThreads) {
    const int j = j0 + static_cast<int>(threadIdx.x);
    float s = hb;
    if (j < whole)
      for (int b = 0; b < nb; ++b) s += __ldcg(&u.part[static_cast<size_t>(b) * u.cap + j].x);
    finish(j < whole, j, s);
  }
  const int ldb = bn + 1;           // chains of one warp on different banks
  float* sw = usm;                  // [nb][ldb]
  float* sx = sw + nb * ldb;        // [kStUpdRays][nb][ldb]
  float* sp = sx + kStUpdRays * nb * ldb;  // [kStUpdRays][nb]
  for (int j0 = whole + blockIdx.x * kStUpdRays; j0 < cnt; j0 += gridDim.x * kStUpdRays) {
    const int m = min(cnt - j0, kStUpdRays);
    const int t0 = j0 / 128 * nb;          // the row block's first tile
    const int b0 = max(0, plan.big - t0);  // blocks before it: partials
    const int nx = (nb - b0) << lg;
    const float* X = u.x + ((static_cast<size_t>(t0 + b0 - plan.big) * 128 + j0 % 128) << lg);
    for (int i = threadIdx.x; i < nx; i += kStUpdThreads)
      sw[(b0 + (i >> lg)) * ldb + (i & (bn - 1))] = __ldg(u.head_w + (b0 << lg) + i);
    for (int i = threadIdx.x; i < m * nx / 4; i += kStUpdThreads) {
      const int r = 4 * i / nx, k = 4 * i - r * nx, b = k >> lg, c = k & (bn - 1);
      const float4 x = __ldcg(
          reinterpret_cast<const float4*>(X + ((static_cast<size_t>(b) * 128 + r) << lg) + c));
      float* d = sx + (r * nb + b0 + b) * ldb + c;
      d[0] = x.x;
      d[1] = x.y;
      d[2] = x.z;
      d[3] = x.w;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < m * nb; k += kStUpdThreads) {
      const int b = k % nb;
      float h = 0.f;
      if (b < b0) {
        h = __ldcg(&u.part[static_cast<size_t>(b) * u.cap + j0 + k / nb].x);
      } else {
        const float* x = sx + k * ldb;
        const float* w = sw + b * ldb;
#pragma unroll 16
        for (int c = 0; c < bn; ++c) h = fmaf(x[c], w[c], h);
      }
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

// The heads of a query: per ray, output and block of bn columns the partial a
// whole tile left or, where the tile was split, the chain over its FP32
// activations; then the blocks in order, as finish_heads_kernel.
constexpr int kStHeadRays = 8;

__global__ void __launch_bounds__(256)
step_heads_kernel(const float2* __restrict__ part, const float* __restrict__ X, int M,
                  const StepTiles st, const float* __restrict__ wo, const float* __restrict__ bo,
                  const __grid_constant__ HeadOut o) {
  extern __shared__ float hsm[];
  const int nb = st.num_n, lg = st.lg_bn, bn = 1 << lg, ldb = bn + 1;
  const TilePlan plan = tile_plan(M, st);
  float* sw = hsm;                          // [2][nb][ldb]
  float* sx = sw + 2 * nb * ldb;            // [kStHeadRays][nb][ldb]
  float* sp = plan.lg_split == 0 ? hsm : sx + kStHeadRays * nb * ldb;  // [kStHeadRays][nb][2]
  const int j0 = blockIdx.x * kStHeadRays;
  const int m = min(M - j0, kStHeadRays);
  const int t0 = j0 / 128 * nb;
  const int b0 = plan.lg_split == 0 ? nb : min(nb, max(0, plan.big - t0));
  const int nx = (nb - b0) << lg;
  for (int i = threadIdx.x; i < 2 * nx; i += blockDim.x) {
    const int r = i >= nx ? 1 : 0, k = i - r * nx;
    sw[(r * nb + b0 + (k >> lg)) * ldb + (k & (bn - 1))] =
        __ldg(wo + ((r * nb + b0) << lg) + k);
  }
  st_wait();
  const float* x0 = X + (static_cast<ptrdiff_t>(t0 + b0 - plan.big) * 128 + j0 % 128) * bn;
  for (int i = threadIdx.x; i < m * nx / 4; i += blockDim.x) {
    const int r = 4 * i / nx, k = 4 * i - r * nx, b = k >> lg, c = k & (bn - 1);
    const float4 x = __ldcg(
        reinterpret_cast<const float4*>(x0 + ((static_cast<size_t>(b) * 128 + r) << lg) + c));
    float* d = sx + (r * nb + b0 + b) * ldb + c;
    d[0] = x.x;
    d[1] = x.y;
    d[2] = x.z;
    d[3] = x.w;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m * nb * 2; i += blockDim.x) {
    const int k = i >> 1, out = i & 1, b = k % nb;
    float h = 0.f;
    if (b < b0) {
      const float2 v = __ldcg(&part[static_cast<size_t>(b) * M + j0 + k / nb]);
      h = out == 0 ? v.x : v.y;
    } else {
      const float* x = sx + k * ldb;
      const float* w = sw + (out * nb + b) * ldb;
#pragma unroll 16
      for (int c = 0; c < bn; ++c) h = fmaf(x[c], w[c], h);
    }
    sp[i] = h;
  }
  __syncthreads();
  if (static_cast<int>(threadIdx.x) < m) {
    float z0 = 0.f, z1 = 0.f;
    for (int b = 0; b < nb; ++b) {
      z0 += sp[(threadIdx.x * nb + b) * 2];
      z1 += sp[(threadIdx.x * nb + b) * 2 + 1];
    }
    write_heads(o, j0 + threadIdx.x, z0 + bo[0], z1 + bo[1]);
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

cudaError_t launch_step_encode(const RaySoA& rays, const float* t, const int* idx, const int* count,
                               int* next_count, int cap, int L, int ld, __nv_bfloat16* out, int sms,
                               bool first, cudaStream_t s) {
  if (cap <= 0 || ld % 8 != 0) return cudaErrorInvalidValue;
  const int blocks = (cap + kStEncRays - 1) / kStEncRays;
  return launch_chained<RaySoA, const float*, const int*, const int*, int*, int, int, int,
                        __nv_bfloat16*>(step_encode_kernel, first, std::min(blocks, 4 * sms),
                                        3 * kStEncRays, kStEncRays * (ld + 8) * 2, s, rays, t, idx,
                                        count, next_count, cap, L, ld, out);
}

namespace {

template <bool IN_FP8, bool OUT_FP8, bool LAST>
cudaError_t launch_layer(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB64,
                         const TcGemmParams& p, const StepTiles& st, bool first, cudaStream_t s) {
  const int grid =
      p.m_dev != nullptr ? st.sms : std::min(st.sms, tile_plan(p.M, st).tiles);
  return launch_chained<CUtensorMap, CUtensorMap, CUtensorMap, TcGemmParams, StepTiles>(
      tc_step_kernel<IN_FP8, OUT_FP8, LAST>, first, grid, kStThreads,
      kStRing + kStCtrl + epi_vector_bytes(p.N) + 1024, s, tmA, tmB, tmB64, p, st);
}

}  // namespace

cudaError_t load_step_query_kernels(bool fp8) {
  const void* bf16[] = {(const void*)tc_step_kernel<false, false, false>,
                        (const void*)tc_step_kernel<false, false, true>};
  const void* e4m3[] = {(const void*)tc_step_kernel<false, true, false>,
                        (const void*)tc_step_kernel<true, true, false>,
                        (const void*)tc_step_kernel<true, false, true>,
                        (const void*)tc_step_kernel<false, false, true>};
  const void* heads = (const void*)step_heads_kernel;
  cudaError_t e = load_kernels(&heads, 1);
  if (e == cudaSuccess) e = fp8 ? load_kernels(e4m3, 4) : load_kernels(bf16, 2);
  return e;
}

cudaError_t launch_step_layer(bool in_fp8, bool out_fp8, const CUtensorMap& tmA,
                              const CUtensorMap& tmB, const CUtensorMap& tmB64,
                              const TcGemmParams& p, const StepTiles& st, bool first,
                              cudaStream_t s) {
  const bool last = p.mode == 1;
  if (p.M <= 0) return cudaSuccess;
  if ((st.lg_bn != 7 && st.lg_bn != 8) || p.N != st.num_n << st.lg_bn || p.bias == nullptr ||
      st.sms < 1 ||
      (last && (p.head_w == nullptr || p.head_part == nullptr ||
                (p.out_f32 == nullptr && st.x_tiles > 0) || out_fp8 ||
                reinterpret_cast<uintptr_t>(p.out_f32) % 32 != 0)) ||
      !epi_out_aligned(p, out_fp8))
    return cudaErrorInvalidValue;
  if (last)
    return in_fp8 ? launch_layer<true, false, true>(tmA, tmB, tmB64, p, st, first, s)
                  : launch_layer<false, false, true>(tmA, tmB, tmB64, p, st, first, s);
  if (out_fp8)
    return in_fp8 ? launch_layer<true, true, false>(tmA, tmB, tmB64, p, st, first, s)
                  : launch_layer<false, true, false>(tmA, tmB, tmB64, p, st, first, s);
  if (in_fp8) return cudaErrorInvalidValue;
  return launch_layer<false, false, false>(tmA, tmB, tmB64, p, st, first, s);
}

cudaError_t launch_step_update(const StepUpdate& u, bool first, cudaStream_t s) {
  if (u.cap <= 0) return cudaErrorInvalidValue;
  const int nb = u.tiles.num_n;
  const int smem = ((1 + kStUpdRays) * nb * ((1 << u.tiles.lg_bn) + 1) + kStUpdRays * nb) * 4;
  const int blocks = (u.cap + kStUpdRays - 1) / kStUpdRays, most = 2 * u.tiles.sms;
  return launch_chained<StepUpdate>(step_update_kernel, first, blocks < most ? blocks : most,
                                    kStUpdThreads, smem, s, u);
}

cudaError_t launch_step_heads(const float2* part, const float* X, int M, const StepTiles& st,
                              const float* wo, const float* bo, const HeadOut& o,
                              cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  const int nb = st.num_n;
  const bool split = tile_plan(M, st).lg_split > 0;  // else no chains are run here
  const int smem = (split ? (2 + kStHeadRays) * nb * ((1 << st.lg_bn) + 1) : 0) * 4 +
                   kStHeadRays * nb * 8;
  return launch_chained<const float2*, const float*, int, StepTiles, const float*, const float*,
                        HeadOut>(step_heads_kernel, true, (M + kStHeadRays - 1) / kStHeadRays, 256,
                                 smem, s, part, X, M, st, wo, bo, o);
}

}  // namespace ddf
