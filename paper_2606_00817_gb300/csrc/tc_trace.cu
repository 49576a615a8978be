// tc_trace.cu -- sphere tracing of an SDF field (Sec. 4.4) of width 128 to 512
// in one persistent kernel.
//
// Layer by layer a trace is bound by latency: each of up to 128 steps is an
// encoding, H layer launches and an update, some 65 us whether 65,536 rays are
// still marching or three, and the host, which does not know, launches all of
// them. Here a thread-block cluster of W / 128 CTAs owns 128 lanes. A lane
// holds one ray until it hits, leaves or runs out of steps, and then takes the
// next ray from a global counter, so there are no lists, no compaction and no
// launches in between; the kernel ends when the last ray does.
//
// A step of a cluster: every CTA encodes the 128 current points into its
// operand tile (128 x W bf16 in shared memory, 128-byte-swizzled K-major);
// per layer CTA r computes output columns [128 r, 128 r + 128) (its weights
// streamed by TMA through a ring that runs ahead across layers and steps),
// writes them, as its part of the next layer's operand, into its own tile, and
// copies that part (32 KB, contiguous) into the peers' tiles. What bounds it is
// the chain of a step: per layer the MMAs (2,048 cycles at W = 512), a cluster
// handshake, the epilogue and the copies. (Storing the outputs to the peers from
// the registers, 16 bytes a thread, took 9,500 cycles a layer.)
// Up to 128 steps, 8.4 a ray: 300 rays through 39 -> 256 x 4 3.97 -> 0.59 ms,
// 3,000 rays 4.59 -> 1.07; through 51 -> 512 x 6 6.46 -> 2.34 and 6.58 -> 2.34. Larger
// batches take the step kernels (tc_steps.cu).
//
// The arithmetic is that of the layer kernels in their order, so t, hit and
// steps are the same bits: K ascending, ReLU(acc + b) rounded to bf16, the head's
// FP32 chain over blocks of 256 (or 128) columns, handed from CTA to CTA inside a
// block, then the blocks in order.
//
// Handshakes are mbarriers in every CTA that the peers arrive on (release /
// acquire at cluster scope): "all CTAs have read their tiles", the bytes of the
// peers' parts, "chain", "blocks", "next rays". Every wait is
// bounded; a CTA that gives up raises a status bit and goes to the final cluster
// barrier, its peers follow when their own waits run out.
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "kernels.h"
#include "ptx_sm103.cuh"

namespace ddf {

namespace {

constexpr uint64_t kTrDrainNs = 1000000000ull;
constexpr int kTrThreads = 256 + 32;  // 8 compute warps, the producer
constexpr int kTrBlock = 16384;       // 128 rows x 64 K: a K block of the tile, and a weight chunk
constexpr int kTrSlots = 8;           // most ring slots
constexpr int kTrCtrl = 512;
constexpr int kTrSmemMax = 227 * 1024 - 1024;  // less the base alignment
constexpr int kTrSmemLimit = 227 * 1024;

struct TrShape {
  int kb1;    // K blocks of the encoding
  int slots;  // ring chunks
  int smem;
};

// Floats behind the control block: biases [H x 128], head slice [128], incoming
// chain [128], blocks [4 x 128].
__host__ __device__ constexpr int tr_floats(int H) { return H * 128 + 128 + 128 + 4 * 128; }

TrShape tr_shape(int L, int C, int H) {
  TrShape s{};
  s.kb1 = (3 + 6 * L + 63) / 64;
  const int tile = kTrBlock * (2 * C > s.kb1 ? 2 * C : s.kb1);
  const int rest = kTrCtrl + tr_floats(H) * 4;
  const int room = (kTrSmemMax - tile - rest) / kTrBlock;
  s.slots = room < kTrSlots ? room : kTrSlots;
  s.smem = tile + s.slots * kTrBlock + rest + 1024;
  return s;
}

__device__ __forceinline__ uint32_t tr_off(int r, int c) {  // byte offset of element c of row r
  return static_cast<uint32_t>((c >> 6) * kTrBlock + r * 128 + ((((c >> 3) & 7) ^ (r & 7)) << 4) +
                               ((c & 7) << 1));
}

__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint32_t bar, uint32_t parity,
                                                          uint64_t timeout_ns) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((i & 15u) == 0u && globaltimer_ns() - t0 > timeout_ns) return false;
  }
}

// `bytes` of this CTA's shared memory to the peer address dst; counted as
// transaction bytes on the peer's barrier.
__device__ __forceinline__ void bulk_copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes,
                                                  uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(dst), "r"(src), "r"(bytes), "r"(bar_cluster)
      : "memory");
}

template <int C>
__global__ void __launch_bounds__(kTrThreads, 1)
    tc_trace_kernel(const __grid_constant__ TraceMaps maps, const __grid_constant__ TraceParams p,
                    const TrShape sh) {
  constexpr int kBlk = C % 2 == 0 ? 2 : 1;  // CTAs of one head chain: blocks of 256 or 128 columns
  constexpr int kBlocks = C / kBlk;
  extern __shared__ uint8_t smem_raw[];
  // the same offset in every CTA of the cluster (peers' addresses are mapped from it)
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* const sA = smem;
  uint8_t* const ring = smem + kTrBlock * (2 * C > sh.kb1 ? 2 * C : sh.kb1);
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + sh.slots * kTrBlock);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kTrSlots + s); };
  const uint32_t done_bar = bar0 + 8u * (2 * kTrSlots);
  const uint32_t read_bar = done_bar + 8u;    // C arrivals: every CTA's MMAs have read their tile
  const uint32_t write_bar = done_bar + 16u;  // own arrival and the bytes of the peers' parts
  const uint32_t chain_bar = done_bar + 24u;  // 1 arrival: the chain so far
  const uint32_t block_bar = done_bar + 32u;  // kBlocks arrivals: the head's blocks
  const uint32_t next_bar = done_bar + 40u;   // 1 arrival: the next rays' first index
  int* ctrl = reinterpret_cast<int*>(bars + 2 * kTrSlots + 6);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ctrl);
  volatile int* stop_flag = reinterpret_cast<volatile int*>(ctrl + 1);
  volatile int* s_base = ctrl + 2;  // written by rank 0
  unsigned* s_mask = reinterpret_cast<unsigned*>(ctrl + 4);  // [4] finished, [4] active
  float* sbias = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kTrCtrl);
  float* shw = sbias + p.H * 128;
  float* s_chain = shw + 128;
  float* s_block = s_chain + 128;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int cluster = blockIdx.x / C, clusters = gridDim.x / C;

  if (tid == 0) {
    for (int s = 0; s < sh.slots; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(done_bar, 1);
    mbar_init(read_bar, C);
    mbar_init(write_bar, 1);
    mbar_init(chain_bar, 1);
    mbar_init(block_bar, kBlocks);
    mbar_init(next_bar, 1);
    *stop_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), 128);
    tmem_relinquish();
  }
  for (int i = tid; i < p.H * 128; i += kTrThreads)
    sbias[i] = __ldg(p.bias[i >> 7] + 128 * rank + (i & 127));
  for (int i = tid; i < 128; i += kTrThreads) shw[i] = __ldg(p.head_w + 128 * rank + i);
  tc_fence_before();
  cluster_sync_all();  // barriers of every CTA initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 8) {
    if (lane == 0) {
      // -------------------------------------------------------- producer
      int slot = 0, layer = 0, kb = 0, issued = 0;
      uint32_t ph = 0;
      for (;;) {
        if (!mbar_wait_bounded(empty_bar(slot), ph ^ 1u, stop_flag, p.timeout_ns)) break;
        if (*stop_flag) break;
        mbar_arrive_expect_tx(full_bar(slot), kTrBlock);
        tma_load_2d(smem_u32(ring + slot * kTrBlock), &maps.m[layer], kb * 64, 128 * rank,
                    full_bar(slot));
        if (++kb == (layer == 0 ? sh.kb1 : 2 * C)) {
          kb = 0;
          layer = layer + 1 == p.H ? 0 : layer + 1;
        }
        if (++slot == sh.slots) {
          slot = 0;
          ph ^= 1u;
        }
        if (issued < sh.slots) ++issued;
      }
      // no exit with a copy in flight: the last `issued` chunks, newest last
      for (int j = 0; j < issued; ++j) {
        if (--slot < 0) {
          slot = sh.slots - 1;
          ph ^= 1u;
        }
        mbar_wait_bounded(full_bar(slot), ph, nullptr, kTrDrainNs);
      }
    }
  } else {
    const int q = warp & 3, half = warp >> 2;
    const int r = q * 32 + lane;  // this thread's lane of the cluster (two threads each)
    const uint32_t trow = tmem + (static_cast<uint32_t>(q * 32) << 16);
    const uint32_t a0 = smem_u32(sA);
    constexpr uint32_t idesc = mma_idesc(1u, 128, 128);
    auto group_sync = [&]() { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    auto group_and = [&](bool v) {
      uint32_t all;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\t"
          "setp.ne.u32 p, %1, 0;\n\t"
          "bar.red.and.pred q, 1, 256, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(all)
          : "r"(v ? 1u : 0u)
          : "memory");
      return all != 0;
    };
    auto arrive_all = [&](uint32_t bar) {  // one thread
#pragma unroll
      for (int c = 0; c < C; ++c) mbar_arrive_release_cluster(map_to_cta(bar, c));
    };

    // the lane's ray
    int idx = cluster * 128 + r;
    if (idx >= p.n) idx = -1;
    float o[3] = {0.f, 0.f, 0.f}, d[3] = {0.f, 0.f, 0.f}, t = 0.f;
    int steps = 0;
    auto load_ray = [&]() {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        o[c] = __ldg(p.rays.p[c] + idx);
        d[c] = __ldg(p.rays.p[3 + c] + idx);
      }
      t = 0.f;
      steps = 0;
    };
    if (idx >= 0) load_ray();

    int slot = 0;               // of the next weight chunk, and its phase (64-bit
    uint32_t sph = 0;           // counters and their divisions took 400 cycles a chunk)
    uint32_t dph = 0, rph = 0, wph = 0, cph = 0, bph = 0, nph = 0;
    bool ok = true, more = true;  // more: the counter may still have rays
    bool awaited = false;         // (thread 0) peers' copies may be on their way here
    uint32_t awaited_phase = 0;
    bool any = cluster * 128 < p.n;
    while (any && ok) {
      {  // encode the current point: the pairs of bands in turn by the lane's two threads
        float e[3] = {0.f, 0.f, 0.f};
        if (idx >= 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) e[c] = fmaf(t, d[c], o[c]);
        }
        auto put = [&](int col, float v) {
          *reinterpret_cast<__nv_bfloat16*>(sA + tr_off(r, col)) = __float2bfloat16_rn(v);
        };
        if (half == 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) put(c, e[c]);
        }
        for (int k = half; k < p.L; k += 2) {
          const float f = __int_as_float((127 + k) << 23);  // 2^k exactly
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            float sn, cs;
            sincospif(e[c] * f, &sn, &cs);
            const int col = 3 + 2 * (c * p.L + k);
            put(col, sn);
            put(col + 1, cs);
          }
        }
        if (half == 1)
          for (int col = 3 + 6 * p.L; col < sh.kb1 * 64; ++col) put(col, 0.f);
      }
      fence_proxy_async_smem();
      tc_fence_before();
      group_sync();
      float s = 0.f;  // the SDF value
      for (int l = 0; l < p.H; ++l) {
        if (tid == 0) {
          if (l > 0)  // the peers' parts of this layer's operand are here
            awaited = !(ok = mbar_wait_cluster_bounded(write_bar, wph, p.timeout_ns));
          tc_fence_after();
          const int kbs = l == 0 ? sh.kb1 : 2 * C;
          for (int kb = 0; kb < kbs && ok; ++kb) {
            if (!mbar_wait_bounded(full_bar(slot), sph, stop_flag, p.timeout_ns)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t ab = a0 + kb * kTrBlock, bb = smem_u32(ring + slot * kTrBlock);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              tc_mma_f16(tmem, sw128_kmajor_desc(ab + 32u * j), sw128_kmajor_desc(bb + 32u * j),
                         idesc, (kb != 0 || j != 0) ? 1u : 0u);
            tc_commit(empty_bar(slot));
            if (++slot == sh.slots) {
              slot = 0;
              sph ^= 1u;
            }
          }
          tc_commit(done_bar);
          ok = mbar_wait_bounded(done_bar, dph, nullptr, p.timeout_ns) && ok;
        }
        if (l > 0) wph ^= 1u;
        dph ^= 1u;
        const bool last = l == p.H - 1;
        // once every CTA has read its tile, the peers' parts in it may be replaced,
        // and this CTA's own: the copies of it that the peers read have landed
        if (!last && tid == 0 && ok) {
          mbar_arrive_expect_tx(write_bar, (C - 1) * 2 * kTrBlock);
          awaited = true;
          awaited_phase = wph;
          arrive_all(read_bar);
          ok = mbar_wait_cluster_bounded(read_bar, rph, p.timeout_ns);
        }
        if (!last) rph ^= 1u;
        ok = group_and(ok);
        if (!ok) break;
        tc_fence_after();
        const float* bias = sbias + l * 128;
        if (!last) {
          const EpiVectors ev{bias, nullptr, nullptr, nullptr, 1.f};
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int col = 64 * half + 32 * c;
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
              *reinterpret_cast<uint4*>(sA + tr_off(r, 128 * rank + col + 8 * k)) = w;
            }
          }
          fence_proxy_async_smem();  // for the copies and the MMAs
          tc_fence_before();
          group_sync();
          if (tid == 0) {
            const uint32_t part = a0 + static_cast<uint32_t>(2 * rank) * kTrBlock;
#pragma unroll
            for (int c = 1; c < C; ++c) {
              const int peer = (rank + c) % C;
              bulk_copy_to_peer(map_to_cta(part, peer), part, 2 * kTrBlock,
                                map_to_cta(write_bar, peer));
            }
          }
        } else {
          // the head: this CTA's 128 columns of its block's chain
          float h = 0.f;
          if (kBlk > 1 && rank % kBlk != 0) {
            if (tid == 0) ok = mbar_wait_cluster_bounded(chain_bar, cph, p.timeout_ns);
            cph ^= 1u;
            ok = group_and(ok);
            if (!ok) break;
            h = s_chain[r];
          }
          if (half == 0) {
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t v[32];
              tmem_ld32(trow + 32 * c, v);
              tmem_wait_ld_regs(v);
              const float4* b4 = reinterpret_cast<const float4*>(bias + 32 * c);
              const float4* w4 = reinterpret_cast<const float4*>(shw + 32 * c);
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float4 b = b4[k], w = w4[k];
                h = fmaf(fmaxf(__uint_as_float(v[4 * k + 0]) + b.x, 0.f), w.x, h);
                h = fmaf(fmaxf(__uint_as_float(v[4 * k + 1]) + b.y, 0.f), w.y, h);
                h = fmaf(fmaxf(__uint_as_float(v[4 * k + 2]) + b.z, 0.f), w.z, h);
                h = fmaf(fmaxf(__uint_as_float(v[4 * k + 3]) + b.w, 0.f), w.w, h);
              }
            }
            if (kBlk > 1 && rank % kBlk != kBlk - 1) {
              st_cluster_u32(map_to_cta(smem_u32(s_chain + r), rank + 1), __float_as_uint(h));
            } else {
#pragma unroll
              for (int c = 0; c < C; ++c)
                st_cluster_u32(map_to_cta(smem_u32(s_block + (rank / kBlk) * 128 + r), c),
                               __float_as_uint(h));
            }
          }
          tc_fence_before();
          group_sync();
          if (tid == 0) {
            if (kBlk > 1 && rank % kBlk != kBlk - 1)
              mbar_arrive_release_cluster(map_to_cta(chain_bar, rank + 1));
            else
              arrive_all(block_bar);
            ok = mbar_wait_cluster_bounded(block_bar, bph, p.timeout_ns);
          }
          bph ^= 1u;
          ok = group_and(ok);
          if (!ok) break;
          s = __ldg(p.head_b);
#pragma unroll
          for (int b = 0; b < kBlocks; ++b) s += s_block[b * 128 + r];
        }
      }
      if (!ok) break;

      // the step's outcome, the same in every CTA
      bool finished = false;
      if (idx >= 0) {
        ++steps;
        bool hit = false;
        if (s < p.eps) {
          hit = finished = true;
        } else {
          t = t + s;
          finished = t > p.t_max || steps >= p.max_steps;
        }
        if (finished && rank == 0 && half == 0) {
          p.out_t[idx] = t;
          p.out_hit[idx] = hit ? 1 : 0;
          if (p.out_steps != nullptr) p.out_steps[idx] = steps;
        }
      }
      const unsigned fm = __ballot_sync(0xffffffffu, finished || idx < 0);
      const unsigned am = __ballot_sync(0xffffffffu, idx >= 0 && !finished);
      if (half == 0 && lane == 0) {
        s_mask[q] = fm;
        s_mask[4 + q] = am;
      }
      group_sync();
      int free_lanes = 0, before = 0;
      any = false;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const unsigned m = s_mask[w];
        free_lanes += __popc(m);
        before += w < q ? __popc(m) : w == q ? __popc(m & ((1u << lane) - 1u)) : 0;
        any = any || s_mask[4 + w] != 0;
      }
      if (finished) idx = -1;
      if (more && free_lanes > 0) {
        if (tid == 0) {
          if (rank == 0) {
            const int base = clusters * 128 + atomicAdd(p.queue, free_lanes);
#pragma unroll
            for (int c = 0; c < C; ++c)
              st_cluster_u32(map_to_cta(smem_u32(const_cast<int*>(s_base)), c),
                             static_cast<uint32_t>(base));
            arrive_all(next_bar);
          }
          ok = mbar_wait_cluster_bounded(next_bar, nph, p.timeout_ns);
        }
        nph ^= 1u;
        ok = group_and(ok);
        if (!ok) break;
        const int base = *s_base;
        more = base + free_lanes < p.n;
        any = any || base < p.n;
        if (idx < 0 && base + before < p.n) {
          idx = base + before;
          load_ray();
        }
      }
      group_sync();  // s_mask and s_base are read before the next step writes them
    }
    if (tid == 0) {
      if (!ok) {
        atomicOr(p.status, kStatusPipelineTimeout);
        mbar_wait_bounded(done_bar, dph ^ 1u, nullptr, kTrDrainNs);  // MMAs in flight
        if (awaited) mbar_wait_bounded(write_bar, awaited_phase, nullptr, kTrDrainNs);
      }
      *stop_flag = 1;  // the producer has run ahead
    }
  }
  tc_fence_before();
  cluster_sync_all();  // no CTA leaves while a peer may write to it
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

template <int C>
cudaError_t configure(const TrShape& s, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  // a constant: the limit is the function's, and host threads with other fields set it too
  cudaError_t e = cudaFuncSetAttribute(
      tc_trace_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrSmemLimit);
  if (e != cudaSuccess) return e;
  *cfg = cudaLaunchConfig_t{};
  cfg->blockDim = dim3(kTrThreads);
  cfg->dynamicSmemBytes = s.smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  return cudaSuccess;
}

template <int C>
int max_clusters(const TrShape& s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  int n = 0;
  if (configure<C>(s, &cfg, at) != cudaSuccess) return cudaGetLastError(), 0;
  cfg.gridDim = dim3(C);
  if (cudaOccupancyMaxActiveClusters(&n, tc_trace_kernel<C>, &cfg) != cudaSuccess)
    return cudaGetLastError(), 0;
  return n;
}

template <int C>
cudaError_t launch_c(const TrShape& s, const TraceMaps& maps, const TraceParams& p, int clusters,
                     cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  cudaError_t e = configure<C>(s, &cfg, at);
  if (e != cudaSuccess) return e;
  const int64_t need = (static_cast<int64_t>(p.n) + 127) / 128;
  cfg.gridDim = dim3(static_cast<unsigned>(C * (need < clusters ? need : clusters)));
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, tc_trace_kernel<C>, maps, p, s);
}

}  // namespace

// Clusters of the trace kernel that fit the current device at once; 0: the
// field's shape is not one it takes.
int tc_trace_clusters(int L, int W, int H) {
  // with one layer a CTA could be two steps ahead of a peer that still reads its blocks
  if (W % 128 != 0 || W > 512 || H < 2 || H > kTraceLayers) return 0;
  const TrShape s = tr_shape(L, W / 128, H);
  if (s.slots < 3 || s.kb1 > 2 * (W / 128)) return 0;
  switch (W / 128) {
    case 1: return max_clusters<1>(s);
    case 2: return max_clusters<2>(s);
    case 3: return max_clusters<3>(s);
    default: return max_clusters<4>(s);
  }
}

cudaError_t launch_tc_trace(int L, int W, const TraceMaps& maps, const TraceParams& p, int clusters,
                            cudaStream_t st) {
  if (p.n <= 0) return cudaSuccess;
  if (clusters <= 0 || W % 128 != 0 || W > 512 || p.H < 2 || p.H > kTraceLayers || p.L != L)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(p.queue, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  const TrShape s = tr_shape(L, W / 128, p.H);
  switch (W / 128) {
    case 1: return launch_c<1>(s, maps, p, clusters, st);
    case 2: return launch_c<2>(s, maps, p, clusters, st);
    case 3: return launch_c<3>(s, maps, p, clusters, st);
    default: return launch_c<4>(s, maps, p, clusters, st);
  }
}

}  // namespace ddf
