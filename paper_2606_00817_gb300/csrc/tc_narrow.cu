// tc_narrow.cu -- a whole bf16 ray query of a narrow field (width 128 or 256)
// in one kernel: encoding (Sec. 4.3), every ReLU layer and the heads.
//
// Layer by layer, a narrow field is bound by its launches: each of the
// H + 2 kernels runs for 3-8 us, mostly start-up, one TMA round trip and the
// way of the activations through L2. Here a group of 256 threads takes 128
// rays through all layers: the encoded rays and then each layer's activations
// live in one shared-memory tile (128-byte-swizzled K-major operand of
// tcgen05.mma, overwritten in place once the layer's MMAs are done), the
// accumulator (128 x W) in TMEM, and only the weights are loaded, as chunks of
// W rows x 64 K through TMA:
//   * resident: all chunks of the field fit in shared memory (width 128, up to
//     5 layers); they are loaded once per CTA, and two groups (two tiles) run
//     side by side where there is room, one in its MMAs while the other drains;
//   * streamed: a ring of chunks, refilled as the MMAs release them, so the
//     next layer's weights arrive while a layer drains. One group.
// Measured, a whole call: 78 -> 128 x 4, 16,384 rays 42 us by layers, 22 us so (near
// the host cost of a call), 300,000 rays 166 and 101 us; 102 -> 256 x 3, 100,000
// rays 102 and 73 us, 300,000 rays 241 and 185, 1,000,000 rays 708 and 585 us. It wins
// at every size measured.
//
// The arithmetic is that of the layer kernels, in their order (encode_kernel,
// K ascending in steps of 16, ReLU(acc + b) rounded to bf16, the head's FP32
// dot products column by column in blocks of min(W, 256)), so the results are
// the same bits as those of the default tiles.
//
// Waits are bounded; a timeout raises the abort flag and a status bit, and the
// CTA waits for its copies and MMAs in flight before it releases TMEM.
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "heads.cuh"
#include "kernels.h"
#include "ptx_sm103.cuh"

namespace ddf {

namespace {

constexpr uint64_t kNwDrainNs = 1000000000ull;
constexpr int kNwGroup = 256;     // threads of a group
constexpr int kNwSlots = 16;      // most chunks a ring holds
constexpr int kNwBlock = 16384;   // 128 rows x 64 K of a tile
constexpr int kNwCtrl = 512;
constexpr int kNwSmemMax = 227 * 1024 - 1024;  // less the base alignment
constexpr int kNwSmemLimit = 227 * 1024;

// Byte offset of element pair (even column c) of row r in the operand tile.
__device__ __forceinline__ uint32_t nw_off(int r, int c) {
  return static_cast<uint32_t>((c >> 6) * kNwBlock + r * 128 + ((((c >> 3) & 7) ^ (r & 7)) << 4) +
                               ((c & 7) << 1));
}

struct NwShape {
  int kb1;      // 64-wide K blocks of the encoding
  int a_bytes;  // operand tile of one group
  int slots;    // ring chunks
  int groups;
  bool resident;
  int smem;
};

// How a field of this shape is laid out; slots 0: it does not fit.
NwShape nw_shape(int L, int W, int H) {
  NwShape s{};
  s.kb1 = (6 + 12 * L + 63) / 64;
  s.a_bytes = kNwBlock * (s.kb1 > W / 64 ? s.kb1 : W / 64);
  const int chunk = W * 128;
  const int chunks = s.kb1 + (H - 1) * (W / 64);
  const int vec = (H * W + 2 * W + 4 + 2 * 128) * 4;
  for (int g = W == 128 ? 2 : 1; g >= 1; --g) {
    const int room = (kNwSmemMax - kNwCtrl - vec - g * s.a_bytes) / chunk;
    s.groups = g;
    s.resident = chunks <= room && chunks <= kNwSlots;
    s.slots = s.resident ? chunks : (room < kNwSlots ? room : kNwSlots);
    s.smem = g * s.a_bytes + s.slots * chunk + vec + kNwCtrl + 1024;
    if (s.resident) return s;
  }
  if (s.slots < 3) s.slots = 0;  // a shorter ring cannot hide a load
  return s;
}

template <int W>
__global__ void __launch_bounds__(2 * kNwGroup + 32, 1)
    tc_narrow_kernel(const __grid_constant__ NarrowMaps maps,
                     const __grid_constant__ NarrowParams p, const NwShape sh,
                     const __grid_constant__ RaySoA rays, const __grid_constant__ HeadOut out) {
  constexpr int kChunk = W * 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* ring = smem + sh.groups * sh.a_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + sh.slots * kChunk);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kNwSlots + s); };
  auto done_bar = [&](int g) { return bar0 + 8u * (2 * kNwSlots + g); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kNwSlots + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* sbias = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kNwCtrl);
  float* shw = sbias + p.H * W;  // two head rows, then the head bias (4 floats)
  float* sz = shw + 2 * W + 4;   // z1 of each group's rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int groups = sh.groups;
  const bool producer = warp == groups * (kNwGroup / 32);

  const int64_t tiles = (p.M + 127) / 128;
  const int kbh = W / 64;                       // K blocks of a hidden layer
  const int chunks = sh.kb1 + (p.H - 1) * kbh;  // of one tile

  // The producer thread: barriers, then weight chunks for as long as the ring
  // has room, before the rest of the CTA is even set up.
  int64_t loaded = 0;  // chunks issued
  int load_slot = 0, load_layer = 0, load_kb = 0;  // of the next one
  uint32_t load_ph = 0;
  auto load_chunk = [&]() {
    mbar_arrive_expect_tx(full_bar(load_slot), kChunk);
    tma_load_2d(smem_u32(ring + load_slot * kChunk), &maps.m[load_layer], load_kb * 64, 0,
                full_bar(load_slot));
    ++loaded;
    if (++load_slot == sh.slots) {
      load_slot = 0;
      load_ph ^= 1u;
    }
    if (++load_kb == (load_layer == 0 ? sh.kb1 : kbh)) {
      load_kb = 0;
      load_layer = load_layer + 1 == p.H ? 0 : load_layer + 1;
    }
  };
  int64_t total = 0;  // chunks this CTA needs
  if (producer && lane == 0) {
    for (int l = 0; l < p.H; ++l) tma_prefetch_desc(&maps.m[l]);
    for (int s = 0; s < sh.slots; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int g = 0; g < groups; ++g) mbar_init(done_bar(g), 1);
    *abort_flag = 0;
    fence_mbar_init();
    // tiles of this CTA pass through its groups in turn; a streamed field has one group
    const int64_t mine = tiles > blockIdx.x ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    total = sh.resident ? (mine > 0 ? chunks : 0) : mine * chunks;
    while (loaded < total && loaded < sh.slots) load_chunk();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), groups * W);
    tmem_relinquish();
  }
  {  // biases, head rows and head bias, all loads of a round in flight at once
    const int nb = p.H * W, nv = nb + 2 * W + 2;
    for (int i0 = tid; i0 < nv; i0 += 4 * blockDim.x) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * blockDim.x;
        if (i < nv)
          v[j] = __ldg(i < nb ? p.bias[i / W] + i % W
                              : i < nb + 2 * W ? p.head_w + (i - nb) : p.head_b + (i - nb - 2 * W));
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int i = i0 + j * blockDim.x;
        if (i < nv) sbias[i] = v[j];
      }
    }
  }

  // Encodes the rays of `tile` into group g's operand tile: 2 threads a ray, 3
  // coordinates each.
  const int g = warp >> 3;
  const int gt = tid - g * kNwGroup;  // thread of the group
  uint8_t* const sA = smem + g * sh.a_bytes;
  auto encode = [&](int64_t tile) {
    const int er = gt & 127, part = gt >> 7;
    const int64_t row = tile * 128 + er;
    float e[3] = {0.f, 0.f, 0.f};
    if (row < p.M) {
#pragma unroll
      for (int c = 0; c < 3; ++c) e[c] = ray_ld(rays, 3 * part + c, row);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int col = 3 * part + c;
      *reinterpret_cast<__nv_bfloat16*>(sA + nw_off(er, col & ~1) + ((col & 1) << 1)) =
          __float2bfloat16_rn(e[c]);
    }
    for (int k = 0; k < p.L; ++k) {  // three independent chains at a time
      const float f = __int_as_float((127 + k) << 23);  // 2^k exactly
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float sn, cs;
        sincospif(e[c] * f, &sn, &cs);
        *reinterpret_cast<uint32_t*>(sA + nw_off(er, 6 + 2 * ((3 * part + c) * p.L + k))) =
            epi_pack_bf16x2(sn, cs);
      }
    }
    if (part == 0)
      for (int col = 6 + 12 * p.L; col < sh.kb1 * 64; col += 2)
        *reinterpret_cast<uint32_t*>(sA + nw_off(er, col)) = 0u;
  };
  const int64_t tile0 = blockIdx.x + static_cast<int64_t>(gridDim.x) * g;
  if (!producer && tile0 < tiles) encode(tile0);  // beside the first loads
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  auto raise_abort = [&]() {
    *abort_flag = 1;
    atomicOr(p.status, kStatusPipelineTimeout);
  };

  if (producer) {
    if (lane == 0) {
      bool ok = true;
      while (loaded < total) {
        if (!mbar_wait_bounded(empty_bar(load_slot), load_ph ^ 1u, abort_flag, p.timeout_ns)) {
          ok = false;
          break;
        }
        load_chunk();
      }
      if (!ok) raise_abort();
      // no exit with a copy in flight: back over the last chunks
      for (int64_t j = loaded < sh.slots ? loaded : sh.slots; j > 0; --j) {
        if (--load_slot < 0) {
          load_slot = sh.slots - 1;
          load_ph ^= 1u;
        }
        mbar_wait_bounded(full_bar(load_slot), load_ph, nullptr, kNwDrainNs);
      }
    }
  } else {
    const uint32_t a0 = smem_u32(sA);
    const int q = warp & 3, half = (gt >> 7);        // TMEM lane quarter, column half
    const int r = q * 32 + lane;                     // this thread's row of the accumulator
    const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(g * W);
    const uint32_t trow = d_tmem + (static_cast<uint32_t>(q * 32) << 16);
    constexpr uint32_t idesc = mma_idesc(1u, W, 128);
    auto group_sync = [&]() {
      asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kNwGroup) : "memory");
    };
    auto group_and = [&](bool v) {  // a barrier of the group; true if v is for all its threads
      uint32_t all;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.u32 p, %3, 0;\n\t"
          "bar.red.and.pred q, %1, %2, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(all)
          : "r"(g + 1), "n"(kNwGroup), "r"(v ? 1u : 0u)
          : "memory");
      return all != 0;
    };
    int slot = 0;         // streamed: the next chunk's, and its phase (64-bit counters
    uint32_t sph = 0;     // and their divisions cost 400 cycles a chunk)
    uint32_t dphase = 0;  // layers finished, mod 2
    bool ok = true;
    for (int64_t tile = tile0; tile < tiles && ok;
         tile += static_cast<int64_t>(gridDim.x) * groups) {
      if (tile != tile0) encode(tile);
      for (int l = 0; l < p.H; ++l) {
        fence_proxy_async_smem();  // this thread's part of the tile, for the MMAs
        tc_fence_before();
        group_sync();
        if (gt == 0) {
          tc_fence_after();
          const int kbs = l == 0 ? sh.kb1 : kbh;
          const int first = l == 0 ? 0 : sh.kb1 + (l - 1) * kbh;
          for (int kb = 0; kb < kbs && ok; ++kb) {
            const int s = sh.resident ? first + kb : slot;
            const uint32_t ph = sh.resident ? 0u : sph;
            if (!mbar_wait_bounded(full_bar(s), ph, abort_flag, p.timeout_ns)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t ab = a0 + kb * kNwBlock, bb = smem_u32(ring + s * kChunk);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              tc_mma_f16(d_tmem, sw128_kmajor_desc(ab + 32u * j), sw128_kmajor_desc(bb + 32u * j),
                         idesc, (kb != 0 || j != 0) ? 1u : 0u);
            if (!sh.resident) {
              tc_commit(empty_bar(s));
              if (++slot == sh.slots) {
                slot = 0;
                sph ^= 1u;
              }
            }
          }
          tc_commit(done_bar(g));  // arrives once every MMA above has finished
          ok = mbar_wait_bounded(done_bar(g), dphase, nullptr, p.timeout_ns) && ok;
        }
        dphase ^= 1u;
        ok = group_and(ok);  // the group goes on, or gives up, together
        if (!ok) break;
        tc_fence_after();
        if (l + 1 < p.H) {  // ReLU(acc + b) in bf16 over the tile: the next operand
          const EpiVectors ev{sbias + l * W, nullptr, nullptr, nullptr, 1.f};
#pragma unroll
          for (int c = 0; c < W / 64; ++c) {
            const int col = half * (W / 2) + 32 * c;
            uint32_t v[32];
            tmem_ld32(trow + col, v);
            tmem_wait_ld_regs(v);
            float x[32];
            epi_affine32(ev, v, col, x);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              uint4 w;
              w.x = epi_pack_bf16x2_relu(x[8 * k + 0], x[8 * k + 1]);
              w.y = epi_pack_bf16x2_relu(x[8 * k + 2], x[8 * k + 3]);
              w.z = epi_pack_bf16x2_relu(x[8 * k + 4], x[8 * k + 5]);
              w.w = epi_pack_bf16x2_relu(x[8 * k + 6], x[8 * k + 7]);
              *reinterpret_cast<uint4*>(sA + nw_off(r, col + 8 * k)) = w;
            }
          }
        } else {
          // the FP32 head, column by column: z0 by the threads of half 0, z1 by
          // those of half 1, which pass it on through shared memory
          const float* hw = shw + half * W;
          const float* bias = sbias + l * W;
          float z = 0.f;
#pragma unroll 1
          for (int c = 0; c < W / 32; ++c) {
            uint32_t v[32];
            tmem_ld32(trow + 32 * c, v);
            tmem_wait_ld_regs(v);
            const float4* b4 = reinterpret_cast<const float4*>(bias + 32 * c);
            const float4* w4 = reinterpret_cast<const float4*>(hw + 32 * c);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float4 b = b4[k], w = w4[k];
              z = fmaf(fmaxf(__uint_as_float(v[4 * k + 0]) + b.x, 0.f), w.x, z);
              z = fmaf(fmaxf(__uint_as_float(v[4 * k + 1]) + b.y, 0.f), w.y, z);
              z = fmaf(fmaxf(__uint_as_float(v[4 * k + 2]) + b.z, 0.f), w.z, z);
              z = fmaf(fmaxf(__uint_as_float(v[4 * k + 3]) + b.w, 0.f), w.w, z);
            }
          }
          z = (0.f + z) + shw[2 * W + half];
          if (half == 1) sz[g * 128 + r] = z;
          group_sync();
          const int64_t row = tile * 128 + r;
          if (half == 0 && row < p.M) write_heads(out, row, z, sz[g * 128 + r]);
        }
      }
      // the accumulator is read before the next tile's MMAs
      tc_fence_before();
      group_sync();
    }
    if (!ok && gt == 0) {
      raise_abort();
      mbar_wait_bounded(done_bar(g), dphase ^ 1u, nullptr, kNwDrainNs);  // MMAs in flight
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, groups * W);
  }
}

template <int W>
cudaError_t launch_w(const NarrowMaps& maps, const NarrowParams& p, const NwShape& s,
                     const RaySoA& rays, const HeadOut& out, int num_sms, cudaStream_t st) {
  // a constant: the limit is the function's, and host threads with other fields set it too
  cudaError_t e = cudaFuncSetAttribute(
      tc_narrow_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNwSmemLimit);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (p.M + 127) / 128;
  const int grid = static_cast<int>(tiles < num_sms ? tiles : num_sms);
  tc_narrow_kernel<W><<<grid, s.groups * kNwGroup + 32, s.smem, st>>>(maps, p, s, rays, out);
  return cudaGetLastError();
}

}  // namespace

bool tc_narrow_supported(int L, int W, int H) {
  return (W == 128 || W == 256) && H >= 1 && H <= kNarrowLayers && nw_shape(L, W, H).slots > 0;
}

cudaError_t launch_tc_narrow(const NarrowMaps& maps, const NarrowParams& p, const RaySoA& rays,
                             const HeadOut& out, int W, int num_sms, cudaStream_t st) {
  if (p.M <= 0) return cudaSuccess;
  if (!tc_narrow_supported(p.L, W, p.H)) return cudaErrorInvalidValue;
  const NwShape s = nw_shape(p.L, W, p.H);
  return W == 128 ? launch_w<128>(maps, p, s, rays, out, num_sms, st)
                  : launch_w<256>(maps, p, s, rays, out, num_sms, st);
}

}  // namespace ddf
