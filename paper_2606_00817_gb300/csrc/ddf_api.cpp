// ddf_api.cpp -- the C ABI of libddf.so (declared in include/ddf.h).
//
// Host-side runtime of the DDF query path: argument checking, weight upload
// and derivation of the per-precision device copies, workspace management,
// TMA tensor-map construction, the per-chunk launch sequence
//   encode -> H dense layers -> heads
// (one network evaluation per ray, Sec. 3.3), the pipelined host-buffer
// query, device status words and per-kernel-class event timing.
#include "ddf.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "handle.h"
#include "kernels.h"

namespace ddfi {

thread_local std::string g_last_error;

ddf_status fail(ddf_status s, const std::string& msg) {
  g_last_error = msg;
  return s;
}

ddf_status cuda_fail(cudaError_t e, const char* what) {
  const ddf_status s = (e == cudaErrorMemoryAllocation) ? DDF_ERR_OOM : DDF_ERR_CUDA;
  return fail(s, std::string(what) + ": " + cudaGetErrorString(e));
}


int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }


PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// Row-major [rows x inner] matrix of 1- or 2-byte elements, 128-byte-swizzled
// boxes of [box_rows x (128 bytes)].
bool make_tmap(CUtensorMap* m, const void* base, bool one_byte, uint64_t inner, uint64_t rows,
               uint64_t row_bytes, uint32_t box_rows) {
  auto fn = get_encode_fn();
  if (fn == nullptr) return false;
  const cuuint64_t dims[2] = {inner, rows};
  const cuuint64_t strides[1] = {row_bytes};
  const cuuint32_t box[2] = {one_byte ? 128u : 64u, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(m, one_byte ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                        2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}


}  // namespace ddfi


namespace ddfi {

// Injected allocation failure (ddf_debug_fail_allocation): the allocation
// that finds the counter at 0 fails and disables it; -1 = off.
std::atomic<int64_t> g_fail_alloc_after{-1};

ddf_status dev_alloc(ddf_s* h, void** p, size_t bytes) {
  *p = nullptr;
  if (bytes == 0) bytes = 16;
  int64_t k = g_fail_alloc_after.load();
  while (k >= 0 && !g_fail_alloc_after.compare_exchange_weak(k, k - 1)) {
  }
  if (k == 0)
    return fail(DDF_ERR_OOM, "device allocation of " + std::to_string(bytes) +
                                 " bytes refused (injected failure)");
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(DDF_ERR_OOM, "cudaMalloc of " + std::to_string(bytes) + " bytes failed: " +
                                 cudaGetErrorString(e));
  }
  h->owned.push_back(*p);
  return DDF_OK;
}

void dev_free(ddf_s* h, void* p) {
  if (p == nullptr) return;
  auto it = std::find(h->owned.begin(), h->owned.end(), p);
  if (it != h->owned.end()) h->owned.erase(it);
  cudaFree(p);
}

// Frees every per-layer weight buffer and the master blob, so that a weight
// load that failed half way starts from nothing on its next attempt.
void release_weight_buffers(ddf_s* h) {
  for (auto* v : {&h->wf, &h->bias, &h->wscale, &h->colscale}) {
    for (float* q : *v) dev_free(h, q);
    v->clear();
  }
  for (__nv_bfloat16* q : h->wb) dev_free(h, q);
  for (__nv_bfloat16* q : h->wcal) dev_free(h, q);
  for (__nv_bfloat16* q : h->wp) dev_free(h, q);
  for (uint8_t* q : h->wq) dev_free(h, q);
  h->wb.clear();
  h->tmBig.clear();
  h->tmSmall.clear();
  h->tmTrace.clear();
  h->tmStep.clear();
  h->tmF32.clear();
  h->wcal.clear();
  h->wp.clear();
  h->wq.clear();
  dev_free(h, h->head_w);
  dev_free(h, h->head_b);
  dev_free(h, h->d_blob);
  h->head_w = h->head_b = h->d_blob = nullptr;
  h->loaded = false;
}

bool valid_config(const ddf_config* c, std::string* why) {
  if (c == nullptr) return *why = "config is NULL", false;
  if (c->octaves < 0 || c->octaves > 16) return *why = "octaves must be in [0, 16]", false;
  if (c->width < 8 || c->width > 8192 || c->width % 8 != 0)
    return *why = "width must be a multiple of 8 in [8, 8192]", false;
  if (c->hidden_layers < 1 || c->hidden_layers > 64)
    return *why = "hidden_layers must be in [1, 64]", false;
  if (c->precision < DDF_FP32 || c->precision > DDF_FP8_E4M3)
    return *why = "unknown precision", false;
  if (c->device < 0) return *why = "device must be >= 0", false;
  if (c->kind != DDF_KIND_RAY && c->kind != DDF_KIND_SDF && c->kind != DDF_KIND_HASHGRID)
    return *why = "unknown kind", false;
  if (c->kind == DDF_KIND_SDF && c->precision != DDF_BF16)
    return *why = "SDF fields run in bf16 only", false;
  if (c->kind == DDF_KIND_HASHGRID) {
    if (c->octaves != 4 || c->width != 64 || c->hidden_layers > 4)
      return *why = "hash-grid fields: 4 direction bands, width 64, 1..4 hidden layers", false;
    if (c->precision == DDF_FP8_E4M3) return *why = "hash-grid fields run in bf16 or FP32", false;
  }
  return true;
}

size_t input_width(const ddf_config& c) {
  if (c.kind == DDF_KIND_HASHGRID) return 59;  // 16 levels x 2 features + 27 direction values
  return c.kind == DDF_KIND_SDF ? 3 + 6 * static_cast<size_t>(c.octaves)
                                : 6 + 12 * static_cast<size_t>(c.octaves);
}

size_t head_rows(const ddf_config& c) { return c.kind == DDF_KIND_SDF ? 1 : 2; }

size_t param_count(const ddf_config& c) {
  if (c.kind == DDF_KIND_HASHGRID) return hg_param_count(c);
  const size_t d_in = input_width(c);
  const size_t W = c.width;
  const size_t hr = head_rows(c);
  return d_in * W + W + (c.hidden_layers - 1) * (W * W + W) + hr * W + hr;
}

cudaEvent_t prof_event(ddf_s* h) {
  if (h->ev_used == h->ev_pool.size()) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    h->ev_pool.push_back(e);
  }
  return h->ev_pool[h->ev_used++];
}


// Most head partials any tile writes per row: N/128 blocks x 2 epilogue halves.
int max_partials(int W) { return (W / 128) * 2; }

void clear_graphs(ddf_s* h);

// Fields whose small batches run on the tiles of tc_small.cu (narrow ones have
// their own kernel).
bool small_batches(const ddf_s* h) {
  return h->cfg.kind == DDF_KIND_RAY && h->cfg.precision != DDF_FP32 && !h->narrow;
}

ddf_status ensure_workspace(ddf_s* h, int64_t rows) {
  if (rows <= h->ws_rows || h->cfg.kind == DDF_KIND_HASHGRID) return DDF_OK;  // no workspace
  clear_graphs(h);  // cached graphs point at the old buffers
  dev_free(h, h->ws_enc);
  dev_free(h, h->ws_act[0]);
  dev_free(h, h->ws_act[1]);
  dev_free(h, h->ws_part);
  h->ws_enc = h->ws_act[0] = h->ws_act[1] = nullptr;
  h->ws_part = nullptr;
  h->ws_x = nullptr;
  h->ws_x_rows = 0;
  h->ws_rows = 0;
  const int W = h->cfg.width;
  const bool f32 = h->cfg.precision == DDF_FP32;
  // e4m3 activations need 1 byte, but the calibration pass of an FP8 handle
  // runs the layers in bf16 through the same buffers
  const bool planes = f32 && h->f32_clusters > 0;  // three bf16 planes of one pass's rows
  const size_t elem = planes ? 6 : f32 ? 4 : 2;
  const size_t r = static_cast<size_t>(planes ? std::min(rows, h->f32_pass) : rows);
  ddf_status st;
  if ((st = dev_alloc(h, &h->ws_enc, r * (f32 ? h->kp32 : h->kp16) * elem)) != DDF_OK) return st;
  // the buffer the last layer would write holds a small batch's FP32 activations
  const int xi = (h->cfg.hidden_layers - 1) & 1;
  const int64_t xr = small_batches(h) ? std::min(rows, small_rows(W, h->num_sms)) : 0;
  for (int i = 0; i < 2; ++i) {
    const size_t bytes = std::max(r * W * elem, i == xi ? static_cast<size_t>(xr) * W * 4 : 0);
    if ((st = dev_alloc(h, &h->ws_act[i], bytes)) != DDF_OK) return st;
  }
  h->ws_x = xr > 0 ? static_cast<float*>(h->ws_act[xi]) : nullptr;
  h->ws_x_rows = xr;
  if (!f32) {
    void* p;
    if ((st = dev_alloc(h, &p, static_cast<size_t>(rows) * max_partials(W) * sizeof(float2))) != DDF_OK)
      return st;
    h->ws_part = static_cast<float2*>(p);
  }
  h->ws_rows = rows;
  return DDF_OK;
}

constexpr int64_t kNoSplit = INT64_MAX;

// The rays from row `off` on. A batch that joins two sets of arrays keeps
// its split relative to the new first row; once `off` is past the split the
// second set becomes the only one.
ddf::RaySoA shift_rays(ddf::RaySoA r, int64_t off) {
  if (r.split != kNoSplit && off >= r.split) {
    for (int c = 0; c < 6; ++c) {
      r.p[c] = r.q[c] + (off - r.split);
      r.q[c] = nullptr;
    }
    r.split = kNoSplit;
    return r;
  }
  for (int c = 0; c < 6; ++c) r.p[c] += off;
  if (r.split != kNoSplit) r.split -= off;
  return r;
}

// Advances every output that is present (null outputs stay null); past the
// split of a mixed batch only the second part's visibility and hit flags
// remain.
ddf::HeadOut shift_out(ddf::HeadOut o, int64_t off) {
  if (o.split != kNoSplit && off >= o.split) {
    const int64_t k = off - o.split;
    o.t = nullptr;
    o.z0 = nullptr;
    o.occluded = nullptr;
    o.vis = o.vis2 != nullptr ? o.vis2 + k : nullptr;
    o.hit = o.hit2 != nullptr ? o.hit2 + k : nullptr;
    o.vis2 = nullptr;
    o.hit2 = nullptr;
    o.split = kNoSplit;
    o.rays = shift_rays(o.rays, off);
    return o;
  }
  if (o.t != nullptr) o.t += off;
  if (o.vis != nullptr) o.vis += off;
  if (o.hit != nullptr) o.hit += off;
  if (o.z0 != nullptr) o.z0 += off;
  if (o.occluded != nullptr) o.occluded += off;
  if (o.split != kNoSplit) o.split -= off;
  o.rays = shift_rays(o.rays, off);
  return o;
}

// One pass of an FP32 query on the tensor cores: the encoding and every
// activation as three bf16 planes (tc_gemm_f32.cu), FP32 rows for the head.
ddf_status forward_f32_tc(ddf_s* h, ddf::RaySoA rays, int m, ddf::HeadOut out, cudaStream_t st) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  {
    ProfScope ps(h, kProfEncode, st);
    DDF_CK(ddf::launch_encode_planes(rays, m, h->cfg.octaves, h->kp32,
                                     static_cast<__nv_bfloat16*>(h->ws_enc), st));
  }
  for (int l = 0; l < H; ++l) {
    const void* a_base = l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1];
    ddf::TcF32Params p{};
    p.M = m;
    p.N = W;
    p.K = l == 0 ? h->kp32 : W;
    p.bias = h->bias[l];
    if (l == H - 1)
      p.out_f32 = static_cast<float*>(h->ws_act[l & 1]);
    else
      p.out_planes = static_cast<__nv_bfloat16*>(h->ws_act[l & 1]);
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    CUtensorMap tmA;
    if (!make_tmap(&tmA, a_base, false, p.K, 3 * static_cast<uint64_t>(m),
                   static_cast<uint64_t>(p.K) * 2, 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
    ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
    DDF_CK(ddf::launch_tc_gemm_f32(tmA, h->tmB[l], h->tmF32[l], p, h->f32_clusters, st));
  }
  ProfScope ps(h, kProfHead, st);
  DDF_CK(ddf::launch_head_f32(static_cast<const float*>(h->ws_act[(H - 1) & 1]), m, W, h->head_w,
                              h->head_b, out, st));
  return DDF_OK;
}

ddf_status forward_f32(ddf_s* h, ddf::RaySoA rays, int m, ddf::HeadOut out, cudaStream_t st) {
  const int W = h->cfg.width;
  if (h->f32_clusters > 0) {
    for (int64_t off = 0; off < m; off += h->f32_pass) {
      const ddf_status s =
          forward_f32_tc(h, shift_rays(rays, off),
                         static_cast<int>(std::min<int64_t>(h->f32_pass, m - off)),
                         shift_out(out, off), st);
      if (s != DDF_OK) return s;
    }
    return DDF_OK;
  }
  {
    ProfScope ps(h, kProfEncode, st);
    DDF_CK(ddf::launch_encode_f32(rays, m, h->cfg.octaves, h->kp32, static_cast<float*>(h->ws_enc), st));
  }
  const float* A = static_cast<const float*>(h->ws_enc);
  int K = h->kp32;
  for (int l = 0; l < h->cfg.hidden_layers; ++l) {
    float* C = static_cast<float*>(h->ws_act[l & 1]);
    ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
    DDF_CK(ddf::launch_sgemm_relu(A, h->wf[l], h->bias[l], C, m, W, K, st));
    A = C;
    K = W;
  }
  ProfScope ps(h, kProfHead, st);
  DDF_CK(ddf::launch_head_f32(A, m, W, h->head_w, h->head_b, out, st));
  return DDF_OK;
}

// A few hundred rays through a wide bf16 or e4m3 field (tc_small.cu).
ddf_status forward_small(ddf_s* h, ddf::RaySoA rays, int m, ddf::HeadOut out, cudaStream_t st) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  const bool fp8 = h->cfg.precision == DDF_FP8_E4M3;
  {
    ProfScope ps(h, kProfEncode, st);
    DDF_CK(ddf::launch_small_encode(rays, m, h->cfg.octaves, h->kp16,
                                    static_cast<__nv_bfloat16*>(h->ws_enc), st));
  }
  for (int l = 0; l < H; ++l) {
    const bool in_fp8 = fp8 && l > 0, last = l == H - 1, out_fp8 = fp8 && !last;
    ddf::TcGemmParams p{};
    p.M = m;
    p.N = W;
    p.K = l == 0 ? h->kp16 : W;
    p.bias = h->bias[l];
    p.col_scale = in_fp8 ? h->colscale[l] : nullptr;
    p.out_scale = out_fp8 ? 1.0f / h->act_scales[l] : 1.0f;
    p.ldo = W;
    if (last)
      p.out_f32 = h->ws_x;
    else
      p.out = h->ws_act[l & 1];
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    CUtensorMap tmA;
    if (!make_tmap(&tmA, l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1], in_fp8, p.K, m,
                   static_cast<uint64_t>(p.K) * (in_fp8 ? 1 : 2), 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
    ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
    DDF_CK(ddf::launch_small_layer(in_fp8, out_fp8, tmA, h->tmSmall[l], p, st));
  }
  ProfScope ps(h, kProfHead, st);
  DDF_CK(ddf::launch_small_heads(h->ws_x, m, W, W % 256 == 0 ? 256 : 128, h->head_w, h->head_b,
                                 out, st));
  return DDF_OK;
}

// A few thousand rays through a wide bf16 or e4m3 field (tc_steps.cu).
ddf_status forward_mid(ddf_s* h, ddf::RaySoA rays, int m, ddf::HeadOut out, cudaStream_t st) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  const bool fp8 = h->cfg.precision == DDF_FP8_E4M3;
  // the buffer the last layer would write holds its split tiles
  float* const x = static_cast<float*>(h->ws_act[(H - 1) & 1]);
  const int64_t x_bytes = static_cast<int64_t>(m) * W * (fp8 ? 1 : 2);
  const ddf::StepTiles mid{W / h->bn, h->bn == 256 ? 8 : 7, h->num_sms, h->num_sms};
  ddf::StepTiles end = mid;
  end.x_tiles = static_cast<int>(x_bytes / (128 * 4 * h->bn));
  {
    ProfScope ps(h, kProfEncode, st);
    DDF_CK(ddf::launch_small_encode(rays, m, h->cfg.octaves, h->kp16,
                                    static_cast<__nv_bfloat16*>(h->ws_enc), st));
  }
  for (int l = 0; l < H; ++l) {
    const bool in_fp8 = fp8 && l > 0, last = l == H - 1, out_fp8 = fp8 && !last;
    ddf::TcGemmParams p{};
    p.M = m;
    p.N = W;
    p.K = l == 0 ? h->kp16 : W;
    p.bias = h->bias[l];
    p.col_scale = in_fp8 ? h->colscale[l] : nullptr;
    p.out_scale = out_fp8 ? 1.0f / h->act_scales[l] : 1.0f;
    p.out = h->ws_act[l & 1];
    p.ldo = W;
    p.head_w = h->head_w;
    p.head_part = h->ws_part;
    p.out_f32 = last ? x : nullptr;
    p.mode = last ? 1 : 0;
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    CUtensorMap tmA;
    if (!make_tmap(&tmA, l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1], in_fp8, p.K, m,
                   static_cast<uint64_t>(p.K) * (in_fp8 ? 1 : 2), 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
    ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
    DDF_CK(ddf::launch_step_layer(in_fp8, out_fp8, tmA, h->tmB[l], h->tmSmall[l], p,
                                  last ? end : mid, true, st));
  }
  ProfScope ps(h, kProfHead, st);
  DDF_CK(ddf::launch_step_heads(h->ws_part, x, m, end, h->head_w, h->head_b, out, st));
  return DDF_OK;
}

ddf_status forward_tc(ddf_s* h, ddf::RaySoA rays, int m, ddf::HeadOut out, cudaStream_t st) {
  const int W = h->cfg.width;
  const int H = h->cfg.hidden_layers;
  const bool fp8 = h->cfg.precision == DDF_FP8_E4M3;
  if (h->narrow && h->tile_auto) {
    ddf::NarrowParams p{};
    p.M = m;
    p.L = h->cfg.octaves;
    p.H = H;
    for (int l = 0; l < H; ++l) p.bias[l] = h->bias[l];
    p.head_w = h->head_w;
    p.head_b = h->head_b;
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    ProfScope ps(h, kProfGemm, st);
    DDF_CK(ddf::launch_tc_narrow(h->narrow_maps, p, rays, out, W, h->num_sms, st));
    return DDF_OK;
  }
  if (h->tile_auto && !h->tmSmall.empty() && m <= small_rows(W, h->num_sms) && m <= h->ws_x_rows)
    return forward_small(h, rays, m, out, st);
  if (h->tile_auto && !h->tmSmall.empty() && (h->tmBig.empty() || m < mid_rows(W, h->num_sms, fp8)))
    return forward_mid(h, rays, m, out, st);
  // the tiles in force: those set, or by the batch where none were (kPairRows)
  const bool big = h->tile_auto && !h->tmBig.empty() && m >= kPairRows;
  ddf::TcTile tile_h = h->tile, tile_1 = h->tile_first;
  if (big) {
    tile_h = ddf::TcTile{256, 4, true, true, false};
    if (h->cfg.kind == DDF_KIND_RAY && H > 1 && ddf::tc_layer1_supported(h->cfg.octaves, W))
      tile_1 = ddf::TcTile{256, 8, false, true, true};
    else if (H > 1)
      tile_1 = tile_h;
  }
  const std::vector<CUtensorMap>& tmB = big ? h->tmBig : h->tmB;
  // layer 1 may build the encoding itself (ddf_set_tile checked the shape)
  const bool fused1 = tile_1.fused && h->cfg.kind == DDF_KIND_RAY;
  if (!fused1) {
    ProfScope ps(h, kProfEncode, st);
    if (h->cfg.kind == DDF_KIND_SDF)  // points in rays.p[0..2]
      DDF_CK(ddf::launch_encode_points_bf16(rays.p[0], rays.p[1], rays.p[2], m, h->cfg.octaves,
                                            h->kp16, static_cast<__nv_bfloat16*>(h->ws_enc), st));
    else
      DDF_CK(ddf::launch_encode_bf16(rays, m, h->cfg.octaves, h->kp16,
                                     static_cast<__nv_bfloat16*>(h->ws_enc), st));
  }
  for (int l = 0; l < H; ++l) {
    const bool in_fp8 = fp8 && l > 0;
    const bool last = l == H - 1;
    const bool out_fp8 = fp8 && !last;
    const void* a_base = l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1];
    const int K = l == 0 ? h->kp16 : W;
    ddf::TcGemmParams p{};
    p.M = m;
    p.N = W;
    p.K = K;
    p.bias = h->bias[l];
    p.col_scale = in_fp8 ? h->colscale[l] : nullptr;
    p.out_scale = out_fp8 ? 1.0f / h->act_scales[l] : 1.0f;
    p.out = last ? nullptr : h->ws_act[l & 1];
    p.ldo = W;
    p.head_w = h->head_w;
    p.head_part = h->ws_part;
    p.mode = last ? 1 : 0;
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
    const ddf::TcTile& t = l == 0 ? tile_1 : tile_h;
    if (l == 0 && fused1) {
      CUtensorMap tmO;  // the layer's output, written by TMA stores of 32-row boxes
      if (!make_tmap(&tmO, p.out, out_fp8, W, m, static_cast<uint64_t>(W) * (out_fp8 ? 1 : 2), 32))
        return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an output map");
      const int grid = static_cast<int>(std::min<int64_t>((m + 127) / 128, h->num_sms));
      DDF_CK(ddf::launch_tc_layer1(t.epi_warps, out_fp8, tmB[0], tmO, rays, h->cfg.octaves, p,
                                   grid, st));
      continue;
    }
    const uint64_t row_bytes = static_cast<uint64_t>(K) * (in_fp8 ? 1 : 2);
    CUtensorMap tmA;
    if (!make_tmap(&tmA, a_base, in_fp8, K, m, row_bytes, 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
    if (t.pair) {
      const int64_t tiles = ((m + 255) / 256) * static_cast<int64_t>(W / 256);
      const int clusters = static_cast<int>(std::min<int64_t>(tiles, h->pair_clusters));
      CUtensorMap tmO;  // staged outputs leave shared memory by TMA stores of 32-row boxes
      const bool tma_out = t.staged && !last;
      if (tma_out) {
        if (!make_tmap(&tmO, p.out, out_fp8, W, m, static_cast<uint64_t>(W) * (out_fp8 ? 1 : 2), 32))
          return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an output map");
        p.tma_out = 1;
      }
      DDF_CK(ddf::launch_tc_gemm_pair(in_fp8, out_fp8, t.staged, t.epi_warps, tmA, tmB[l], p,
                                      clusters, st, tma_out ? &tmO : nullptr));
    } else {
      const int64_t tiles = ((m + 127) / 128) * static_cast<int64_t>(W / t.bn);
      const int grid = static_cast<int>(std::min<int64_t>(tiles, h->num_sms));
      DDF_CK(ddf::launch_tc_gemm(t, in_fp8, out_fp8, tmA, tmB[l], p, grid, st));
    }
  }
  ProfScope ps(h, kProfHead, st);
  const ddf::TcTile& tl = H == 1 ? tile_1 : tile_h;  // the last layer writes the partials
  const int nparts = (tl.pair ? W / 256 : W / tl.bn) * (tl.epi_warps / 4);
  DDF_CK(ddf::launch_finish_heads(h->ws_part, nparts, m, h->head_b, out, st));
  return DDF_OK;
}

// The weight maps of the tiles that batches take by their size (kPairRows,
// small_rows), once the weights are loaded; none where those tiles do not exist.
ddf_status build_size_maps(ddf_s* h) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  h->tmBig.clear();
  h->tmSmall.clear();
  if (small_batches(h)) {
    std::vector<CUtensorMap> maps(H);
    for (int l = 0; l < H; ++l) {
      const int kp = l == 0 ? h->kp16 : W;
      const bool ok = h->wb[l] != nullptr
                          ? make_tmap(&maps[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, 64)
                          : make_tmap(&maps[l], h->wq[l], true, W, W, W, 64);
      if (!ok) return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
    }
    h->tmSmall = maps;
  }
  if (h->cfg.precision == DDF_FP32 || W % 256 != 0 || h->pair_clusters <= 0) return DDF_OK;
  std::vector<CUtensorMap> maps(H);
  for (int l = 0; l < H; ++l) {
    const bool whole = l == 0 && (H == 1 || (h->cfg.kind == DDF_KIND_RAY &&
                                             ddf::tc_layer1_supported(h->cfg.octaves, W)));
    const uint32_t box = whole ? 256u : 128u;  // layer 1 fused (or alone): 256 rows
    const int kp = l == 0 ? h->kp16 : W;
    const bool ok = h->wb[l] != nullptr
                        ? make_tmap(&maps[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, box)
                        : make_tmap(&maps[l], h->wq[l], true, W, W, W, box);
    if (!ok) return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
  }
  h->tmBig = maps;
  return DDF_OK;
}

// (Re)builds the TMA maps of the weight matrices for the current N tile.
ddf_status build_weight_maps(ddf_s* h) {
  const int W = h->cfg.width;
  for (int l = 0; l < h->cfg.hidden_layers; ++l) {
    const ddf::TcTile& t = l == 0 ? h->tile_first : h->tile;
    const uint32_t box_rows = t.pair ? 128u : static_cast<uint32_t>(t.bn);
    bool ok = true;
    if (h->wb[l] != nullptr) {
      const int kp = l == 0 ? h->kp16 : W;
      ok = make_tmap(&h->tmB[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, box_rows);
    } else if (h->wq[l] != nullptr) {
      ok = make_tmap(&h->tmB[l], h->wq[l], true, W, W, W, box_rows);
    }
    if (!ok) return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
  }
  return DDF_OK;
}

ddf_status check_rays(const float* const rays[6], int64_t n) {
  if (n < 0) return fail(DDF_ERR_INVALID_ARG, "n must be >= 0");
  if (n > 0 && rays == nullptr) return fail(DDF_ERR_INVALID_ARG, "rays is NULL");
  for (int c = 0; n > 0 && c < 6; ++c) {
    if (rays[c] == nullptr) return fail(DDF_ERR_INVALID_ARG, "a ray array pointer is NULL");
    if (reinterpret_cast<uintptr_t>(rays[c]) % 4 != 0)
      return fail(DDF_ERR_INVALID_ARG, "ray arrays must be 4-byte aligned");
  }
  return DDF_OK;
}

// Ready for a query of the given field kind (ray queries by default).
ddf_status check_ready(ddf_s* h, int kind = DDF_KIND_RAY) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  if (!h->loaded) return fail(DDF_ERR_BAD_WEIGHTS, "no weights loaded");
  const bool match = h->cfg.kind == kind ||
                     (kind == DDF_KIND_RAY && h->cfg.kind == DDF_KIND_HASHGRID);  // ray queries
  if (!match)
    return fail(DDF_ERR_INVALID_ARG, kind == DDF_KIND_RAY ? "not a ray (DDF) field"
                                                          : "not an SDF field");
  if (h->cfg.precision == DDF_FP8_E4M3 && h->cfg.hidden_layers > 1 && !h->scales_set)
    return fail(DDF_ERR_INVALID_ARG, "FP8 needs activation scales (ddf_set_act_scales)");
  return DDF_OK;
}

ddf_status run_query_soa(ddf_s* h, ddf::RaySoA r, int64_t n, ddf::HeadOut out, cudaStream_t st) {
  DDF_REQUIRE_ALIGNED(out.t, 4);
  DDF_REQUIRE_ALIGNED(out.vis, 4);
  DDF_REQUIRE_ALIGNED(out.z0, 4);
  DDF_REQUIRE_ALIGNED(out.vis2, 4);
  const int64_t rows = std::min<int64_t>(n, h->chunk);
  ddf_status s = ensure_workspace(h, rows);
  if (s != DDF_OK) return s;
  out.rays = r;
  if (h->cfg.kind == DDF_KIND_HASHGRID) {  // one fused kernel per part, no chunks needed
    if (r.split == kNoSplit || r.split >= n) return hg_query(h, r, n, out, st);
    const int64_t n1 = r.split;
    ddf::RaySoA r1 = r;
    r1.split = kNoSplit;
    ddf::HeadOut o1 = out;
    o1.split = kNoSplit;
    o1.vis2 = nullptr;
    o1.hit2 = nullptr;
    o1.rays = r1;
    if (n1 > 0 && (s = hg_query(h, r1, n1, o1, st)) != DDF_OK) return s;
    return hg_query(h, shift_rays(r, n1), n - n1, shift_out(out, n1), st);
  }
  for (int64_t off = 0; off < n; off += h->chunk) {
    const int m = static_cast<int>(std::min<int64_t>(h->chunk, n - off));
    const ddf::RaySoA rc = shift_rays(r, off);
    const ddf::HeadOut oc = shift_out(out, off);
    s = h->cfg.precision == DDF_FP32 ? forward_f32(h, rc, m, oc, st) : forward_tc(h, rc, m, oc, st);
    if (s != DDF_OK) return s;
  }
  return DDF_OK;
}

ddf_status run_query(ddf_s* h, const float* const rays[6], int64_t n, ddf::HeadOut out,
                     cudaStream_t st) {
  ddf::RaySoA r;
  for (int c = 0; c < 6; ++c) r.p[c] = rays[c];
  return run_query_soa(h, r, n, out, st);
}

void clear_graphs(ddf_s* h) {
  for (auto& g : h->graphs) cudaGraphExecDestroy(g.exec);
  h->graphs.clear();
}

// Identity of a query for the graph cache: everything its launches bake in.
std::vector<uint64_t> query_key(int kind, const float* const rays[6], int64_t n,
                                std::initializer_list<const void*> ptrs, const float* light,
                                int64_t extra) {
  std::vector<uint64_t> k{static_cast<uint64_t>(kind), static_cast<uint64_t>(n),
                          static_cast<uint64_t>(extra)};
  for (int c = 0; c < 6; ++c) k.push_back(reinterpret_cast<uintptr_t>(rays[c]));
  for (const void* p : ptrs) k.push_back(reinterpret_cast<uintptr_t>(p));
  for (int c = 0; light != nullptr && c < 3; ++c) {
    uint32_t bits;
    std::memcpy(&bits, &light[c], 4);
    k.push_back(bits);
  }
  return k;
}

// Enqueues a query on st: directly, or in graph mode by replaying the CUDA
// graph captured (on a private stream) the first time this key was seen.
// Workspaces must already be large enough: nothing is allocated while capturing.
template <class K, class F>
ddf_status enqueue(ddf_s* h, K make_key, cudaStream_t st, F body) {
  if (!h->graph_mode) return body(st);
  const std::vector<uint64_t> key = make_key();
  for (auto& g : h->graphs) {
    if (g.key == key) {
      DDF_CK(cudaGraphLaunch(g.exec, st));
      return DDF_OK;
    }
  }
  if (h->s_graph == nullptr) DDF_CK(cudaStreamCreateWithFlags(&h->s_graph, cudaStreamNonBlocking));
  const bool keep_prof = h->prof;
  h->prof = false;
  DDF_CK(cudaStreamBeginCapture(h->s_graph, cudaStreamCaptureModeRelaxed));
  const ddf_status s = body(h->s_graph);
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamEndCapture(h->s_graph, &graph);
  h->prof = keep_prof;
  if (s != DDF_OK) {
    if (graph != nullptr) cudaGraphDestroy(graph);
    return s;
  }
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
  if (h->graphs.size() >= 8) {
    cudaGraphExecDestroy(h->graphs.front().exec);
    h->graphs.erase(h->graphs.begin());
  }
  h->graphs.push_back({key, exec});
  DDF_CK(cudaGraphLaunch(exec, st));
  return DDF_OK;
}

ddf_status ensure_ao_buffers(ddf_s* h, int64_t rows) {
  if (rows <= h->ao_rows) return DDF_OK;
  clear_graphs(h);  // cached graphs may point at the old buffers
  dev_free(h, h->ao_vis);
  dev_free(h, h->ao_hit);
  h->ao_vis = nullptr;
  h->ao_hit = nullptr;
  h->ao_rows = 0;
  void* p;
  ddf_status s;
  if ((s = dev_alloc(h, &p, rows * sizeof(float))) != DDF_OK) return s;
  h->ao_vis = static_cast<float*>(p);
  if ((s = dev_alloc(h, &p, rows)) != DDF_OK) return s;
  h->ao_hit = static_cast<uint8_t*>(p);
  h->ao_rows = rows;
  return DDF_OK;
}

// Layers 1..H-1 in bf16 on the calibration weights, recording max |h_l| of
// every hidden activation that feeds an e4m3 layer into amax[l].
ddf_status calibrate_chunk(ddf_s* h, ddf::RaySoA rays, int m, float* amax, cudaStream_t st) {
  const int W = h->cfg.width;
  DDF_CK(ddf::launch_encode_bf16(rays, m, h->cfg.octaves, h->kp16,
                                 static_cast<__nv_bfloat16*>(h->ws_enc), st));
  const ddf::TcTile tile{h->bn, 4};
  for (int l = 0; l + 1 < h->cfg.hidden_layers; ++l) {
    const void* a_base = l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1];
    const int K = l == 0 ? h->kp16 : W;
    CUtensorMap tmA;
    if (!make_tmap(&tmA, a_base, false, K, m, static_cast<uint64_t>(K) * 2, 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
    ddf::TcGemmParams p{};
    p.M = m;
    p.N = W;
    p.K = K;
    p.bias = h->bias[l];
    p.out_scale = 1.0f;
    p.out = h->ws_act[l & 1];
    p.ldo = W;
    p.mode = 0;
    p.status = h->status_dev;
    p.timeout_ns = h->timeout_ns;
    p.amax = amax + l;
    const int64_t tiles = ((m + 127) / 128) * static_cast<int64_t>(W / tile.bn);
    const int grid = static_cast<int>(std::min<int64_t>(tiles, h->num_sms));
    DDF_CK(ddf::launch_tc_gemm(tile, false, false, tmA, h->tmBcal[l], p, grid, st));
  }
  return DDF_OK;
}

ddf_status ensure_plain_maps(ddf_s* h) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  if (static_cast<int>(h->tmBtr.size()) == H) return DDF_OK;
  std::vector<CUtensorMap> maps(H);
  for (int l = 0; l < H; ++l) {
    const int kp = l == 0 ? h->kp16 : W;
    if (h->wb[l] == nullptr) return fail(DDF_ERR_UNSUPPORTED, "no bf16 weights for this layer");
    if (!make_tmap(&maps[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, h->bn))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
  }
  h->tmBtr = maps;
  return DDF_OK;
}

// Weight maps of the narrow tiles of a tracing step.
ddf_status ensure_step_maps(ddf_s* h) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  if (static_cast<int>(h->tmStep.size()) == H) return DDF_OK;
  std::vector<CUtensorMap> maps(H);
  for (int l = 0; l < H; ++l) {
    const int kp = l == 0 ? h->kp16 : W;
    if (!make_tmap(&maps[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, 64))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
  }
  h->tmStep = maps;
  return DDF_OK;
}

ddf_status ensure_trace_buffers(ddf_s* h, int64_t rows) {
  if (rows <= h->trc_rows) return DDF_OK;
  dev_free(h, h->trc_idx[0]);
  dev_free(h, h->trc_idx[1]);
  dev_free(h, h->trc_steps);
  h->trc_idx[0] = h->trc_idx[1] = h->trc_steps = nullptr;
  h->trc_rows = 0;
  void* p;
  ddf_status s;
  for (int i = 0; i < 2; ++i) {
    if ((s = dev_alloc(h, &p, rows * sizeof(int))) != DDF_OK) return s;
    h->trc_idx[i] = static_cast<int*>(p);
  }
  if ((s = dev_alloc(h, &p, rows * sizeof(int))) != DDF_OK) return s;
  h->trc_steps = static_cast<int*>(p);
  // FP32 activations of the last layer's split tiles: fewer tiles than SMs
  dev_free(h, h->trc_x);
  h->trc_x = nullptr;
  const int64_t xe = std::min<int64_t>(round_up(rows, 128) * h->cfg.width,
                                       int64_t{128} * 256 * h->num_sms);
  if ((s = dev_alloc(h, &p, xe * sizeof(float))) != DDF_OK) return s;
  h->trc_x = static_cast<float*>(p);
  if (h->trc_count == nullptr) {
    if ((s = dev_alloc(h, &p, 2 * sizeof(int))) != DDF_OK) return s;
    h->trc_count = static_cast<int*>(p);
  }
  h->trc_rows = rows;
  return DDF_OK;
}

// A trace by one persistent kernel (tc_trace.cu), for the fields and batches it
// serves.
ddf_status trace_in_one(ddf_s* h, const float* const rays[6], int n, int max_steps, float eps,
                        float t_max, float* out_t, uint8_t* out_hit, int32_t* out_steps,
                        cudaStream_t st) {
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  ddf_status s;
  if (h->trc_queue == nullptr) {
    void* q;
    if ((s = dev_alloc(h, &q, sizeof(int))) != DDF_OK) return s;
    h->trc_queue = static_cast<int*>(q);
  }
  if (static_cast<int>(h->tmTrace.size()) != H) {
    std::vector<CUtensorMap> maps(H);
    for (int l = 0; l < H; ++l) {
      const int kp = l == 0 ? h->kp16 : W;
      if (!make_tmap(&maps[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2, 128))
        return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
    }
    h->tmTrace = maps;
  }
  ddf::TraceMaps maps{};
  ddf::TraceParams p{};
  for (int c = 0; c < 6; ++c) p.rays.p[c] = rays[c];
  p.n = n;
  p.L = h->cfg.octaves;
  p.H = H;
  p.max_steps = max_steps;
  p.eps = eps;
  p.t_max = t_max;
  for (int l = 0; l < H; ++l) {
    maps.m[l] = h->tmTrace[l];
    p.bias[l] = h->bias[l];
  }
  p.head_w = h->head_w;
  p.head_b = h->head_b;
  p.out_t = out_t;
  p.out_hit = out_hit;
  p.out_steps = out_steps;
  p.queue = h->trc_queue;
  p.status = h->status_dev;
  p.timeout_ns = h->timeout_ns;
  ProfScope ps(h, kProfGemm, st);
  DDF_CK(ddf::launch_tc_trace(h->cfg.octaves, W, maps, p, h->trc_clusters, st));
  return DDF_OK;
}

}  // namespace ddfi

using namespace ddfi;

extern "C" {

ddf_status ddf_sdf_eval(ddf_handle h, const float* const points[3], int64_t n, float* out_s,
                        void* stream) {
  ddf_status s = check_ready(h, DDF_KIND_SDF);
  if (s != DDF_OK) return s;
  if (n < 0) return fail(DDF_ERR_INVALID_ARG, "n must be >= 0");
  if (n == 0) return DDF_OK;
  if (points == nullptr || points[0] == nullptr || points[1] == nullptr || points[2] == nullptr ||
      out_s == nullptr)
    return fail(DDF_ERR_INVALID_ARG, "a pointer is NULL");
  for (int c = 0; c < 3; ++c) DDF_REQUIRE_ALIGNED(points[c], 4);
  DDF_REQUIRE_ALIGNED(out_s, 4);
  DeviceGuard g(h->cfg.device);
  const float* as_rays[6] = {points[0], points[1], points[2], points[0], points[1], points[2]};
  ddf::HeadOut o{};
  o.z0 = out_s;
  return run_query(h, as_rays, n, o, static_cast<cudaStream_t>(stream));
}

ddf_status ddf_sphere_trace(ddf_handle h, const float* const rays[6], int64_t n, int32_t max_steps,
                            float eps, float t_max, float* out_t, uint8_t* out_hit,
                            int32_t* out_steps, void* stream) {
  ddf_status s = check_ready(h, DDF_KIND_SDF);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (n == 0) return DDF_OK;
  if (n > h->chunk) return fail(DDF_ERR_INVALID_ARG, "trace at most chunk_rays rays per call");
  if (max_steps < 1 || !(eps > 0.f) || !std::isfinite(eps) || !(t_max >= 0.f) ||
      !std::isfinite(t_max))
    return fail(DDF_ERR_INVALID_ARG, "max_steps >= 1, finite eps > 0 and finite t_max >= 0 required");
  if (out_t == nullptr || out_hit == nullptr) return fail(DDF_ERR_INVALID_ARG, "output is NULL");
  DDF_REQUIRE_ALIGNED(out_t, 4);
  DDF_REQUIRE_ALIGNED(out_steps, 4);
  DeviceGuard g(h->cfg.device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int W = h->cfg.width, H = h->cfg.hidden_layers, cap = static_cast<int>(n);
  if (h->trc_clusters < 0) h->trc_clusters = ddf::tc_trace_clusters(h->cfg.octaves, W, H);
  if (h->trc_clusters > 0 && h->tile_auto && n <= trace_rays(W, h->trc_clusters))
    return trace_in_one(h, rays, cap, max_steps, eps, t_max, out_t, out_hit, out_steps, st);
  if ((s = ensure_workspace(h, cap)) != DDF_OK) return s;
  if ((s = ensure_trace_buffers(h, cap)) != DDF_OK) return s;
  if ((s = ensure_plain_maps(h)) != DDF_OK) return s;
  if ((s = ensure_step_maps(h)) != DDF_OK) return s;
  std::vector<CUtensorMap> tmA(H);
  for (int l = 0; l < H; ++l) {
    const int K = l == 0 ? h->kp16 : W;
    if (!make_tmap(&tmA[l], l == 0 ? h->ws_enc : h->ws_act[(l - 1) & 1], false, K, cap,
                   static_cast<uint64_t>(K) * 2, 128))
      return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for an activation map");
  }
  int* steps = out_steps != nullptr ? out_steps : h->trc_steps;
  ddf::RaySoA r;
  for (int c = 0; c < 6; ++c) r.p[c] = rays[c];
  const ddf::StepTiles tiles{W / h->bn, h->bn == 256 ? 8 : 7, h->num_sms, h->num_sms};
  DDF_CK(ddf::launch_trace_init(cap, h->trc_idx[0], h->trc_count, out_t, steps, out_hit, st));
  for (int it = 0; it < max_steps; ++it) {
    int* cin = h->trc_count + (it & 1);
    int* cout = h->trc_count + ((it + 1) & 1);
    const int* iin = h->trc_idx[it & 1];
    int* iout = h->trc_idx[(it + 1) & 1];
    {
      ProfScope ps(h, kProfEncode, st);
      DDF_CK(ddf::launch_step_encode(r, out_t, iin, cin, cout, cap, h->cfg.octaves, h->kp16,
                                     static_cast<__nv_bfloat16*>(h->ws_enc), h->num_sms, it == 0, st));
    }
    for (int l = 0; l < H; ++l) {
      const bool last = l == H - 1;
      const int K = l == 0 ? h->kp16 : W;
      ddf::TcGemmParams p{};
      p.M = cap;
      p.m_dev = cin;
      p.N = W;
      p.K = K;
      p.bias = h->bias[l];
      p.out_scale = 1.0f;
      p.out = last ? nullptr : h->ws_act[l & 1];
      p.ldo = W;
      p.head_w = h->head_w;
      p.head_part = h->ws_part;
      p.out_f32 = last ? h->trc_x : nullptr;
      p.mode = last ? 1 : 0;
      p.status = h->status_dev;
      p.timeout_ns = h->timeout_ns;
      ProfScope ps(h, l == 0 ? kProfFirst : kProfGemm, st);
      DDF_CK(ddf::launch_step_layer(false, false, tmA[l], h->tmBtr[l], h->tmStep[l], p, tiles,
                                    it == 0 && (l == 0 || last), st));
    }
    ProfScope ps(h, kProfHead, st);
    ddf::StepUpdate u{};
    u.part = h->ws_part;
    u.x = h->trc_x;
    u.head_w = h->head_w;
    u.head_b = h->head_b;
    u.tiles = tiles;
    u.cap = cap;
    u.max_steps = max_steps;
    u.eps = eps;
    u.t_max = t_max;
    u.count_in = cin;
    u.idx_in = iin;
    u.t = out_t;
    u.steps = steps;
    u.hit = out_hit;
    u.idx_out = iout;
    u.count_out = cout;
    DDF_CK(ddf::launch_step_update(u, it == 0, st));
  }
  return DDF_OK;
}

size_t ddf_param_count(const ddf_config* cfg) {
  std::string why;
  return valid_config(cfg, &why) ? param_count(*cfg) : 0;
}

const char* ddf_last_error(void) { return g_last_error.c_str(); }

ddf_status ddf_debug_fail_allocation(int64_t after) {
  g_fail_alloc_after.store(after < 0 ? -1 : after);
  return DDF_OK;
}

ddf_status ddf_create(const ddf_config* cfg, ddf_handle* out) {
  if (out == nullptr) return fail(DDF_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  std::string why;
  if (!valid_config(cfg, &why)) return fail(DDF_ERR_INVALID_ARG, why);
  const bool layered = cfg->kind != DDF_KIND_HASHGRID;
  if (layered && cfg->precision != DDF_FP32 && cfg->width % 128 != 0)
    return fail(DDF_ERR_UNSUPPORTED, "tensor-core precisions need width % 128 == 0");
  if (layered && cfg->precision != DDF_FP32 && cfg->width > 2048)
    return fail(DDF_ERR_UNSUPPORTED, "tensor-core precisions support width <= 2048");
  int ndev = 0;
  DDF_CK(cudaGetDeviceCount(&ndev));
  if (cfg->device >= ndev) return fail(DDF_ERR_INVALID_ARG, "device ordinal out of range");
  DeviceGuard g(cfg->device);
  if (!g.ok) return fail(DDF_ERR_CUDA, "cudaSetDevice failed");
  int major = 0, minor = 0;
  DDF_CK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, cfg->device));
  DDF_CK(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, cfg->device));
  if (cfg->precision != DDF_FP32) {
    if (major != 10 || minor != 3)
      return fail(DDF_ERR_UNSUPPORTED, "tensor-core precisions are built for sm_103a only");
    if (get_encode_fn() == nullptr)
      return fail(DDF_ERR_UNSUPPORTED, "cuTensorMapEncodeTiled is not available");
  }
  ddf_s* h = new ddf_s();
  h->cfg = *cfg;
  h->d_in = static_cast<int>(input_width(*cfg));
  h->kp32 = static_cast<int>(round_up(h->d_in, 8));
  h->kp16 = static_cast<int>(round_up(h->d_in, 8));
  h->bn = (cfg->width % 256 == 0) ? 256 : 128;
  h->tile = ddf::TcTile{h->bn, 4};
  h->tile_first = h->tile;
  if (layered && cfg->precision != DDF_FP32 && cfg->width % 256 == 0)
    h->pair_clusters = std::min(ddf::tc_gemm_pair_max_clusters(false),
                                ddf::tc_gemm_pair_max_clusters(true));
  if (layered && cfg->precision == DDF_FP32 && cfg->width % 256 == 0 && major == 10 &&
      minor == 3 && get_encode_fn() != nullptr)
    h->f32_clusters = ddf::tc_gemm_f32_max_clusters();
  h->narrow = cfg->kind == DDF_KIND_RAY && cfg->precision == DDF_BF16 &&
              ddf::tc_narrow_supported(cfg->octaves, cfg->width, cfg->hidden_layers);
  cudaError_t e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, cfg->device);
  void* p = nullptr;
  if (e != cudaSuccess || dev_alloc(h, &p, sizeof(uint32_t)) != DDF_OK) {
    delete h;
    return e != cudaSuccess ? cuda_fail(e, "cudaDeviceGetAttribute") : DDF_ERR_OOM;
  }
  h->status_dev = static_cast<uint32_t*>(p);
  if ((e = cudaMemset(h->status_dev, 0, sizeof(uint32_t))) != cudaSuccess) {
    ddf_destroy(h);
    return cuda_fail(e, "cudaMemset");
  }
  *out = h;
  return DDF_OK;
}

ddf_status ddf_destroy(ddf_handle h) {
  if (h == nullptr) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  cudaDeviceSynchronize();
  for (void* p : h->owned) cudaFree(p);
  for (auto& e : h->ev_pool) cudaEventDestroy(e);
  for (int b = 0; b < 2; ++b) {
    for (int c = 0; c < 6; ++c)
      if (h->hp_rays[b][c]) cudaFree(h->hp_rays[b][c]);
    if (h->hp_t[b]) cudaFree(h->hp_t[b]);
    if (h->hp_v[b]) cudaFree(h->hp_v[b]);
    if (h->hp_occ[b]) cudaFree(h->hp_occ[b]);
    if (h->ev_in[b]) cudaEventDestroy(h->ev_in[b]);
    if (h->ev_comp[b]) cudaEventDestroy(h->ev_comp[b]);
  }
  if (h->s_copy) cudaStreamDestroy(h->s_copy);
  if (h->s_comp) cudaStreamDestroy(h->s_comp);
  for (int b = 0; b < 2; ++b) {
    if (h->ev_gemm[b]) cudaEventDestroy(h->ev_gemm[b]);
    if (h->ev_red[b]) cudaEventDestroy(h->ev_red[b]);
  }
  if (h->ev_join) cudaEventDestroy(h->ev_join);
  if (h->s_red) cudaStreamDestroy(h->s_red);
  clear_graphs(h);
  if (h->s_graph) cudaStreamDestroy(h->s_graph);
  delete h;
  return DDF_OK;
}

ddf_status ddf_load_weights(ddf_handle h, const float* host_blob, size_t n_floats) {
  if (h == nullptr || host_blob == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  const size_t need = param_count(h->cfg);
  if (n_floats != need)
    return fail(DDF_ERR_BAD_WEIGHTS, "blob has " + std::to_string(n_floats) + " floats, config needs " +
                                         std::to_string(need));
  for (size_t i = 0; i < n_floats; ++i)
    if (!std::isfinite(host_blob[i]))
      return fail(DDF_ERR_BAD_WEIGHTS, "non-finite weight at index " + std::to_string(i));
  DeviceGuard g(h->cfg.device);
  if (h->cfg.kind == DDF_KIND_HASHGRID) {
    const ddf_status r = hg_load(h, host_blob);
    if (r == DDF_OK) h->loaded = true;
    return r;
  }
  const int W = h->cfg.width, H = h->cfg.hidden_layers;
  const int prec = h->cfg.precision;
  cudaStream_t st = nullptr;
  ddf_status s;
  auto alloc_buffers = [&]() -> ddf_status {
    void* p;
    if ((s = dev_alloc(h, &p, need * sizeof(float))) != DDF_OK) return s;
    h->d_blob = static_cast<float*>(p);
    h->wf.assign(H, nullptr);
    h->bias.assign(H, nullptr);
    h->wp.assign(H, nullptr);
    h->wb.assign(H, nullptr);
    h->wq.assign(H, nullptr);
    h->wscale.assign(H, nullptr);
    h->colscale.assign(H, nullptr);
    h->wcal.assign(H, nullptr);
    h->tmB.assign(H, CUtensorMap{});
    h->tmBcal.assign(H, CUtensorMap{});
    h->tmF32.assign(H, CUtensorMap{});
    for (int l = 0; l < H; ++l) {
      const int K = l == 0 ? h->d_in : W;
      if ((s = dev_alloc(h, &p, W * sizeof(float))) != DDF_OK) return s;
      h->bias[l] = static_cast<float*>(p);
      if (prec == DDF_FP32) {
        const int kp = l == 0 ? h->kp32 : W;
        if (h->f32_clusters == 0) {
          if ((s = dev_alloc(h, &p, static_cast<size_t>(W) * kp * sizeof(float))) != DDF_OK)
            return s;
          h->wf[l] = static_cast<float*>(p);
        } else {
          if ((s = dev_alloc(h, &p, static_cast<size_t>(W) * kp * 6)) != DDF_OK) return s;
          h->wp[l] = static_cast<__nv_bfloat16*>(p);
          const uint64_t rows = 3 * static_cast<uint64_t>(W), pitch = static_cast<uint64_t>(kp) * 2;
          if (!make_tmap(&h->tmB[l], h->wp[l], false, kp, rows, pitch, 128) ||
              !make_tmap(&h->tmF32[l], h->wp[l], false, kp, rows, pitch, 32))
            return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
        }
      } else if (prec == DDF_BF16 || l == 0) {
        const int kp = l == 0 ? h->kp16 : W;
        if ((s = dev_alloc(h, &p, static_cast<size_t>(W) * kp * 2)) != DDF_OK) return s;
        h->wb[l] = static_cast<__nv_bfloat16*>(p);
        if (!make_tmap(&h->tmB[l], h->wb[l], false, kp, W, static_cast<uint64_t>(kp) * 2,
                       (l == 0 ? h->tile_first : h->tile).pair ? 128u : (l == 0 ? h->tile_first : h->tile).bn))
          return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
        if (h->narrow && !make_tmap(&h->narrow_maps.m[l], h->wb[l], false, kp, W,
                                    static_cast<uint64_t>(kp) * 2, static_cast<uint32_t>(W)))
          return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
      } else {
        if ((s = dev_alloc(h, &p, static_cast<size_t>(W) * W)) != DDF_OK) return s;
        h->wq[l] = static_cast<uint8_t*>(p);
        if ((s = dev_alloc(h, &p, W * sizeof(float))) != DDF_OK) return s;
        h->wscale[l] = static_cast<float*>(p);
        if ((s = dev_alloc(h, &p, W * sizeof(float))) != DDF_OK) return s;
        h->colscale[l] = static_cast<float*>(p);
        if (!make_tmap(&h->tmB[l], h->wq[l], true, W, W, W, h->tile.pair ? 128u : h->tile.bn))
          return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
        // bf16 copy for the activation-scale calibration pass
        if ((s = dev_alloc(h, &p, static_cast<size_t>(W) * W * 2)) != DDF_OK) return s;
        h->wcal[l] = static_cast<__nv_bfloat16*>(p);
      }
      (void)K;
    }
    if (prec == DDF_FP8_E4M3) {
      for (int l = 0; l < H; ++l) {
        const int kp = l == 0 ? h->kp16 : W;
        const __nv_bfloat16* w = l == 0 ? h->wb[0] : h->wcal[l];
        if (!make_tmap(&h->tmBcal[l], w, false, kp, W, static_cast<uint64_t>(kp) * 2, h->bn))
          return fail(DDF_ERR_CUDA, "cuTensorMapEncodeTiled failed for a weight map");
      }
    }
    if ((s = dev_alloc(h, &p, 2 * W * sizeof(float))) != DDF_OK) return s;
    h->head_w = static_cast<float*>(p);
    if ((s = dev_alloc(h, &p, 4 * sizeof(float))) != DDF_OK) return s;
    h->head_b = static_cast<float*>(p);
    return DDF_OK;
  };
  if (h->d_blob == nullptr && (s = alloc_buffers()) != DDF_OK) {
    release_weight_buffers(h);  // the next load allocates again from nothing
    return s;
  }
  if (h->tmBig.empty() && h->tmSmall.empty() && (s = build_size_maps(h)) != DDF_OK) return s;
  DDF_CK(cudaMemcpy(h->d_blob, host_blob, need * sizeof(float), cudaMemcpyHostToDevice));
  size_t off = 0;
  for (int l = 0; l < H; ++l) {
    const int K = l == 0 ? h->d_in : W;
    const float* w = h->d_blob + off;
    off += static_cast<size_t>(W) * K;
    DDF_CK(cudaMemcpy(h->bias[l], h->d_blob + off, W * sizeof(float), cudaMemcpyDeviceToDevice));
    off += W;
    if (prec == DDF_FP32) {
      if (h->f32_clusters == 0)
        DDF_CK(ddf::launch_pack_f32(w, W, K, l == 0 ? h->kp32 : W, h->wf[l], st));
      else
        DDF_CK(ddf::launch_pack_planes(w, W, K, l == 0 ? h->kp32 : W, h->wp[l], st));
    } else if (prec == DDF_BF16 || l == 0) {
      DDF_CK(ddf::launch_pack_bf16(w, W, K, l == 0 ? h->kp16 : W, h->wb[l], st));
      // the transposed copies of a handle that has trained (input gradients)
      if (prec == DDF_BF16 && l > 0 && static_cast<int>(h->wt.size()) > l && h->wt[l] != nullptr)
        DDF_CK(ddf::launch_pack_bf16_t(w, W, W, h->wt[l], st));
    } else {
      DDF_CK(ddf::launch_quant_e4m3(w, W, K, W, h->wq[l], h->wscale[l], st));
      DDF_CK(ddf::launch_pack_bf16(w, W, K, W, h->wcal[l], st));
    }
  }
  // head rows: (t, vis) for a ray field; the SDF field has one row, and the
  // second row of the device head stays zero
  const int hr = static_cast<int>(head_rows(h->cfg));
  DDF_CK(cudaMemset(h->head_w, 0, 2 * W * sizeof(float)));
  DDF_CK(cudaMemset(h->head_b, 0, 2 * sizeof(float)));
  DDF_CK(cudaMemcpy(h->head_w, h->d_blob + off, hr * W * sizeof(float), cudaMemcpyDeviceToDevice));
  off += hr * W;
  DDF_CK(cudaMemcpy(h->head_b, h->d_blob + off, hr * sizeof(float), cudaMemcpyDeviceToDevice));
  if (prec == DDF_FP8_E4M3 && h->scales_set) {
    for (int l = 1; l < H; ++l)
      DDF_CK(ddf::launch_scale_vec(h->wscale[l], h->act_scales[l - 1], W, h->colscale[l], st));
  }
  DDF_CK(cudaDeviceSynchronize());
  h->loaded = true;
  h->fwd_rows = 0;  // kept training activations belong to the old weights
  return DDF_OK;
}

ddf_status ddf_get_weights(ddf_handle h, float* host_blob, size_t n_floats) {
  if (h == nullptr || host_blob == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  if (!h->loaded) return fail(DDF_ERR_BAD_WEIGHTS, "no weights loaded");
  if (n_floats != param_count(h->cfg)) return fail(DDF_ERR_INVALID_ARG, "wrong blob size");
  DeviceGuard g(h->cfg.device);
  DDF_CK(cudaDeviceSynchronize());
  DDF_CK(cudaMemcpy(host_blob, h->d_blob, n_floats * sizeof(float), cudaMemcpyDeviceToHost));
  return DDF_OK;
}

ddf_status ddf_set_act_scales(ddf_handle h, const float* host_scales, int32_t n) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  if (h->cfg.precision != DDF_FP8_E4M3)
    return fail(DDF_ERR_INVALID_ARG, "activation scales apply to FP8 handles only");
  if (n != h->cfg.hidden_layers - 1) return fail(DDF_ERR_INVALID_ARG, "need hidden_layers - 1 scales");
  if (n > 0 && host_scales == nullptr) return fail(DDF_ERR_INVALID_ARG, "scales is NULL");
  for (int i = 0; i < n; ++i) {
    int ex;
    const float m = std::frexp(host_scales[i], &ex);
    if (!(host_scales[i] > 0.f) || !std::isfinite(host_scales[i]) || m != 0.5f)
      return fail(DDF_ERR_INVALID_ARG, "activation scales must be positive powers of two");
  }
  clear_graphs(h);  // the output scales are launch parameters
  h->act_scales.assign(host_scales, host_scales + n);
  h->scales_set = true;
  if (h->loaded) {
    DeviceGuard g(h->cfg.device);
    for (int l = 1; l < h->cfg.hidden_layers; ++l)
      DDF_CK(ddf::launch_scale_vec(h->wscale[l], h->act_scales[l - 1], h->cfg.width, h->colscale[l],
                                   nullptr));
    DDF_CK(cudaDeviceSynchronize());
  }
  return DDF_OK;
}

ddf_status ddf_query_rays(ddf_handle h, const float* const rays[6], int64_t n, float* out_t,
                          float* out_vis, void* stream) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (n > 0 && (out_t == nullptr || out_vis == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "output pointer is NULL");
  DDF_REQUIRE_ALIGNED(out_t, 4);
  DDF_REQUIRE_ALIGNED(out_vis, 4);
  if (n == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  if ((s = ensure_workspace(h, std::min<int64_t>(n, h->chunk))) != DDF_OK) return s;
  ddf::HeadOut o{};
  o.t = out_t;
  o.vis = out_vis;
  return enqueue(h, [&] { return query_key(0, rays, n, {out_t, out_vis}, nullptr, 0); },
                 static_cast<cudaStream_t>(stream),
                 [&](cudaStream_t st) { return run_query(h, rays, n, o, st); });
}

ddf_status ddf_query_shadow(ddf_handle h, const float* const rays[6], int64_t n,
                            const float light[3], float* out_t, float* out_vis,
                            uint8_t* out_occluded, void* stream) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (light == nullptr) return fail(DDF_ERR_INVALID_ARG, "light is NULL");
  if (n > 0 && (out_t == nullptr || out_vis == nullptr || out_occluded == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "output pointer is NULL");
  DDF_REQUIRE_ALIGNED(out_t, 4);
  DDF_REQUIRE_ALIGNED(out_vis, 4);
  if (n == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  if ((s = ensure_workspace(h, std::min<int64_t>(n, h->chunk))) != DDF_OK) return s;
  ddf::HeadOut o{};
  o.t = out_t;
  o.vis = out_vis;
  o.occluded = out_occluded;
  for (int i = 0; i < 3; ++i) o.light[i] = light[i];
  return enqueue(h, [&] { return query_key(1, rays, n, {out_t, out_vis, out_occluded}, light, 0); },
                 static_cast<cudaStream_t>(stream),
                 [&](cudaStream_t st) { return run_query(h, rays, n, o, st); });
}

ddf_status ddf_query_ao(ddf_handle h, const float* const rays[6], int64_t n_rays,
                        const int32_t* offsets, int64_t n_points, float* out_hard,
                        float* out_soft, void* stream) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n_rays)) != DDF_OK) return s;
  if (n_points < 0) return fail(DDF_ERR_INVALID_ARG, "n_points must be >= 0");
  if (n_points > 0 && (offsets == nullptr || out_hard == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "offsets or out_hard is NULL");
  DDF_REQUIRE_ALIGNED(offsets, 4);
  DDF_REQUIRE_ALIGNED(out_hard, 4);
  DDF_REQUIRE_ALIGNED(out_soft, 4);
  if (n_rays >= (int64_t{1} << 31)) return fail(DDF_ERR_INVALID_ARG, "n_rays must fit int32 offsets");
  if (n_points == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  if ((s = ensure_workspace(h, std::max<int64_t>(1, std::min<int64_t>(n_rays, h->chunk)))) != DDF_OK)
    return s;
  if ((s = ensure_ao_buffers(h, std::max<int64_t>(1, n_rays))) != DDF_OK) return s;
  ddf::HeadOut o{};
  o.vis = h->ao_vis;
  o.hit = h->ao_hit;
  return enqueue(h, [&] { return query_key(2, rays, n_rays, {offsets, out_hard, out_soft}, nullptr, n_points); },
                 static_cast<cudaStream_t>(stream), [&](cudaStream_t st) {
                   ddf_status r = n_rays > 0 ? run_query(h, rays, n_rays, o, st) : DDF_OK;
                   if (r != DDF_OK) return r;
                   DDF_CK(ddf::launch_ao_reduce(h->ao_hit, h->ao_vis, offsets, n_points, out_hard,
                                                out_soft, st));
                   return DDF_OK;
                 });
}

ddf_status ddf_query_mixed(ddf_handle h, const float* const shadow_rays[6], int64_t n_shadow,
                           const float light[3], float* out_t, float* out_vis,
                           uint8_t* out_occluded, const float* const ao_rays[6], int64_t n_ao_rays,
                           const int32_t* offsets, int64_t n_points, float* out_hard,
                           float* out_soft, void* stream) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(shadow_rays, n_shadow)) != DDF_OK) return s;
  if ((s = check_rays(ao_rays, n_ao_rays)) != DDF_OK) return s;
  if (n_shadow > 0 && (light == nullptr || out_t == nullptr || out_vis == nullptr ||
                       out_occluded == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "light or a shadow output is NULL");
  if (n_points < 0) return fail(DDF_ERR_INVALID_ARG, "n_points must be >= 0");
  if (n_points > 0 && (offsets == nullptr || out_hard == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "offsets or out_hard is NULL");
  if (n_points == 0 && n_ao_rays > 0)
    return fail(DDF_ERR_INVALID_ARG, "ambient-occlusion rays without shading points");
  DDF_REQUIRE_ALIGNED(out_t, 4);
  DDF_REQUIRE_ALIGNED(out_vis, 4);
  DDF_REQUIRE_ALIGNED(offsets, 4);
  DDF_REQUIRE_ALIGNED(out_hard, 4);
  DDF_REQUIRE_ALIGNED(out_soft, 4);
  if (n_ao_rays >= (int64_t{1} << 31)) return fail(DDF_ERR_INVALID_ARG, "n_ao_rays must fit int32 offsets");
  const int64_t n = n_shadow + n_ao_rays;
  if (n == 0 && n_points == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  if ((s = ensure_workspace(h, std::max<int64_t>(1, std::min<int64_t>(n, h->chunk)))) != DDF_OK)
    return s;
  if ((s = ensure_ao_buffers(h, std::max<int64_t>(1, n_ao_rays))) != DDF_OK) return s;
  ddf::RaySoA r;
  for (int c = 0; c < 6; ++c) {
    r.p[c] = n_shadow > 0 ? shadow_rays[c] : nullptr;
    r.q[c] = n_ao_rays > 0 ? ao_rays[c] : nullptr;
  }
  r.split = n_shadow;
  ddf::HeadOut o{};
  o.t = out_t;
  o.vis = out_vis;
  o.occluded = out_occluded;
  for (int i = 0; n_shadow > 0 && i < 3; ++i) o.light[i] = light[i];
  o.vis2 = h->ao_vis;
  o.hit2 = h->ao_hit;
  o.split = n_shadow;
  std::vector<uint64_t> key = query_key(
      3, r.p, n,
      {out_t, out_vis, out_occluded, offsets, out_hard, out_soft, r.q[0], r.q[1], r.q[2], r.q[3],
       r.q[4], r.q[5]},
      n_shadow > 0 ? light : nullptr, n_points);
  key.push_back(static_cast<uint64_t>(n_shadow));
  return enqueue(h, [&] { return key; }, static_cast<cudaStream_t>(stream), [&](cudaStream_t st) {
    ddf_status q = n > 0 ? run_query_soa(h, r, n, o, st) : DDF_OK;
    if (q != DDF_OK) return q;
    DDF_CK(ddf::launch_ao_reduce(h->ao_hit, h->ao_vis, offsets, n_points, out_hard, out_soft, st));
    return DDF_OK;
  });
}

ddf_status ddf_set_graph_mode(ddf_handle h, int32_t on) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  DeviceGuard g(h->cfg.device);
  if (!on) clear_graphs(h);
  h->graph_mode = on != 0;
  return DDF_OK;
}

ddf_status ddf_calibrate_fp8(ddf_handle h, const float* const rays[6], int64_t n, float* amax_out,
                             float* scales_out, void* stream) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  if (h->cfg.precision != DDF_FP8_E4M3) return fail(DDF_ERR_INVALID_ARG, "not an FP8 handle");
  if (!h->loaded) return fail(DDF_ERR_BAD_WEIGHTS, "no weights loaded");
  ddf_status s = check_rays(rays, n);
  if (s != DDF_OK) return s;
  if (n <= 0) return fail(DDF_ERR_INVALID_ARG, "calibration needs at least one ray");
  const int nl = h->cfg.hidden_layers - 1;
  if (nl == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = ensure_workspace(h, std::min<int64_t>(n, h->chunk))) != DDF_OK) return s;
  float* amax = nullptr;
  DDF_CK(cudaMalloc(&amax, nl * sizeof(float)));
  cudaMemsetAsync(amax, 0, nl * sizeof(float), st);
  ddf::RaySoA r;
  for (int c = 0; c < 6; ++c) r.p[c] = rays[c];
  for (int64_t off = 0; off < n && s == DDF_OK; off += h->chunk) {
    const int m = static_cast<int>(std::min<int64_t>(h->chunk, n - off));
    s = calibrate_chunk(h, shift_rays(r, off), m, amax, st);
  }
  std::vector<float> a(nl);
  const cudaError_t e1 = cudaStreamSynchronize(st);
  const cudaError_t e2 = cudaMemcpy(a.data(), amax, nl * sizeof(float), cudaMemcpyDeviceToHost);
  cudaFree(amax);
  if (s != DDF_OK) return s;
  if (e1 != cudaSuccess || e2 != cudaSuccess) return cuda_fail(e1 != cudaSuccess ? e1 : e2, "calibration");
  std::vector<float> sc(nl);
  for (int l = 0; l < nl; ++l) {
    // smallest power of two s with amax / s <= 448
    double q = static_cast<double>(a[l]) / 448.0;
    int ex = 0;
    const double m = std::frexp(q, &ex);  // q = m 2^ex, m in [0.5, 1)
    sc[l] = a[l] > 0.f ? static_cast<float>(std::ldexp(1.0, m == 0.5 ? ex - 1 : ex)) : 1.0f;
    if (amax_out != nullptr) amax_out[l] = a[l];
    if (scales_out != nullptr) scales_out[l] = sc[l];
  }
  return ddf_set_act_scales(h, sc.data(), nl);
}

namespace ddfi {

// Host-buffer pipeline: chunk i's rays are copied in on a copy stream while
// chunk i-1 is evaluated on a compute stream; results go back on the copy
// stream once the compute stream has finished the chunk.
ddf_status host_pipeline(ddf_s* h, const float* const rays[6], int64_t n, const float* light,
                         float* out_t, float* out_vis, uint8_t* out_occ) {
  const int64_t C = std::min<int64_t>(h->chunk, n);
  if (h->s_copy == nullptr) {
    DDF_CK(cudaStreamCreateWithFlags(&h->s_copy, cudaStreamNonBlocking));
    DDF_CK(cudaStreamCreateWithFlags(&h->s_comp, cudaStreamNonBlocking));
    for (int b = 0; b < 2; ++b) {
      DDF_CK(cudaEventCreateWithFlags(&h->ev_in[b], cudaEventDisableTiming));
      DDF_CK(cudaEventCreateWithFlags(&h->ev_comp[b], cudaEventDisableTiming));
    }
  }
  if (h->hp_rows < C) {
    for (int b = 0; b < 2; ++b) {
      for (int c = 0; c < 6; ++c) {
        cudaFree(h->hp_rays[b][c]);
        h->hp_rays[b][c] = nullptr;
      }
      cudaFree(h->hp_t[b]);
      cudaFree(h->hp_v[b]);
      cudaFree(h->hp_occ[b]);
      h->hp_t[b] = h->hp_v[b] = nullptr;
      h->hp_occ[b] = nullptr;
    }
    h->hp_rows = 0;
    for (int b = 0; b < 2; ++b) {
      for (int c = 0; c < 6; ++c) DDF_CK(cudaMalloc(&h->hp_rays[b][c], C * sizeof(float)));
      DDF_CK(cudaMalloc(&h->hp_t[b], C * sizeof(float)));
      DDF_CK(cudaMalloc(&h->hp_v[b], C * sizeof(float)));
      DDF_CK(cudaMalloc(&h->hp_occ[b], C));
    }
    h->hp_rows = C;
  }
  ddf_status s = ensure_workspace(h, C);
  if (s != DDF_OK) return s;
  const int64_t nchunks = (n + C - 1) / C;
  auto copy_in = [&](int64_t i) -> ddf_status {
    const int b = static_cast<int>(i & 1);
    const int64_t off = i * C, m = std::min<int64_t>(C, n - off);
    for (int c = 0; c < 6; ++c)
      DDF_CK(cudaMemcpyAsync(h->hp_rays[b][c], rays[c] + off, m * sizeof(float),
                             cudaMemcpyHostToDevice, h->s_copy));
    DDF_CK(cudaEventRecord(h->ev_in[b], h->s_copy));
    return DDF_OK;
  };
  if ((s = copy_in(0)) != DDF_OK) return s;
  for (int64_t i = 0; i < nchunks; ++i) {
    const int b = static_cast<int>(i & 1);
    const int64_t off = i * C, m = std::min<int64_t>(C, n - off);
    if (i + 1 < nchunks && (s = copy_in(i + 1)) != DDF_OK) return s;
    DDF_CK(cudaStreamWaitEvent(h->s_comp, h->ev_in[b], 0));
    ddf::HeadOut o{};
    o.t = h->hp_t[b];
    o.vis = h->hp_v[b];
    if (light != nullptr) {
      o.occluded = h->hp_occ[b];
      for (int k = 0; k < 3; ++k) o.light[k] = light[k];
    }
    const float* rp[6];
    for (int c = 0; c < 6; ++c) rp[c] = h->hp_rays[b][c];
    if ((s = run_query(h, rp, m, o, h->s_comp)) != DDF_OK) return s;
    DDF_CK(cudaEventRecord(h->ev_comp[b], h->s_comp));
    DDF_CK(cudaStreamWaitEvent(h->s_copy, h->ev_comp[b], 0));
    DDF_CK(cudaMemcpyAsync(out_t + off, h->hp_t[b], m * sizeof(float), cudaMemcpyDeviceToHost,
                           h->s_copy));
    DDF_CK(cudaMemcpyAsync(out_vis + off, h->hp_v[b], m * sizeof(float), cudaMemcpyDeviceToHost,
                           h->s_copy));
    if (light != nullptr)
      DDF_CK(cudaMemcpyAsync(out_occ + off, h->hp_occ[b], m, cudaMemcpyDeviceToHost, h->s_copy));
  }
  DDF_CK(cudaStreamSynchronize(h->s_copy));
  DDF_CK(cudaStreamSynchronize(h->s_comp));
  return DDF_OK;
}

}  // namespace ddfi

ddf_status ddf_query_rays_host(ddf_handle h, const float* const rays[6], int64_t n, float* out_t,
                               float* out_vis) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (n > 0 && (out_t == nullptr || out_vis == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "output pointer is NULL");
  if (n == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  return host_pipeline(h, rays, n, nullptr, out_t, out_vis, nullptr);
}

ddf_status ddf_query_shadow_host(ddf_handle h, const float* const rays[6], int64_t n,
                                 const float light[3], float* out_t, float* out_vis,
                                 uint8_t* out_occluded) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (light == nullptr) return fail(DDF_ERR_INVALID_ARG, "light is NULL");
  if (n > 0 && (out_t == nullptr || out_vis == nullptr || out_occluded == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "output pointer is NULL");
  if (n == 0) return DDF_OK;
  DeviceGuard g(h->cfg.device);
  return host_pipeline(h, rays, n, light, out_t, out_vis, out_occluded);
}

ddf_status ddf_check_status(ddf_handle h, uint32_t* out) {
  if (h == nullptr || out == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard g(h->cfg.device);
  DDF_CK(cudaDeviceSynchronize());
  DDF_CK(cudaMemcpy(out, h->status_dev, sizeof(uint32_t), cudaMemcpyDeviceToHost));
  DDF_CK(cudaMemset(h->status_dev, 0, sizeof(uint32_t)));
  return DDF_OK;
}

ddf_status ddf_set_timeout_ns(ddf_handle h, uint64_t ns) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  clear_graphs(h);
  h->timeout_ns = ns;
  return DDF_OK;
}

ddf_status ddf_set_chunk_rays(ddf_handle h, int64_t chunk) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  if (chunk < 128 || chunk > (int64_t{1} << 30))
    return fail(DDF_ERR_INVALID_ARG, "chunk must be in [128, 2^30]");
  clear_graphs(h);
  h->chunk = chunk;
  return DDF_OK;
}

ddf_status ddf_profile_enable(ddf_handle h, int32_t on) {
  if (h == nullptr) return fail(DDF_ERR_INVALID_ARG, "handle is NULL");
  h->prof = on != 0;
  return DDF_OK;
}

ddf_status ddf_profile_read(ddf_handle h, double ms[4], int64_t launches[4]) {
  if (h == nullptr || ms == nullptr || launches == nullptr)
    return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard g(h->cfg.device);
  DDF_CK(cudaDeviceSynchronize());
  for (int c = 0; c < kProfClasses; ++c) {
    ms[c] = 0.0;
    launches[c] = 0;
  }
  for (const auto& r : h->recs) {
    float t = 0.f;
    DDF_CK(cudaEventElapsedTime(&t, r.a, r.b));
    ms[r.cls] += t;
    launches[r.cls] += 1;
  }
  h->recs.clear();
  h->ev_used = 0;
  return DDF_OK;
}


ddf_status ddf_set_tile(ddf_handle h, int32_t which, const ddf_tile* tile) {
  if (h == nullptr || tile == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  if (which != 0 && which != 1) return fail(DDF_ERR_INVALID_ARG, "which must be 0 or 1");
  if (h->cfg.kind == DDF_KIND_HASHGRID)
    return fail(DDF_ERR_UNSUPPORTED, "hash-grid fields have one kernel shape");
  const int bn = tile->bn, ew = tile->epi_warps;
  if ((bn != 128 && bn != 256) || (ew != 4 && ew != 8))
    return fail(DDF_ERR_INVALID_ARG, "bn must be 128 or 256 and epi_warps 4 or 8");
  if (h->cfg.width % bn != 0) return fail(DDF_ERR_UNSUPPORTED, "width is not a multiple of bn");
  if (tile->cta_pair != 0 && bn != 256)
    return fail(DDF_ERR_INVALID_ARG, "the CTA-pair tile is bn 256");
  if (tile->fused_encode != 0) {
    if (which != 1) return fail(DDF_ERR_INVALID_ARG, "fused_encode is a layer-1 tile (which = 1)");
    if (bn != 256 || tile->cta_pair != 0 || tile->staged == 0)
      return fail(DDF_ERR_INVALID_ARG, "the fused layer-1 tile is bn 256, no pair, staged");
    if (h->cfg.kind != DDF_KIND_RAY || h->cfg.hidden_layers < 2 ||
        !ddf::tc_layer1_supported(h->cfg.octaves, h->cfg.width))
      return fail(DDF_ERR_UNSUPPORTED,
                  "fused_encode needs a ray field, >= 2 hidden layers, 6 + 12 octaves <= 128 "
                  "and width % 256 == 0");
  } else if (tile->staged != 0 && tile->cta_pair == 0) {
    return fail(DDF_ERR_INVALID_ARG, "staged stores exist for the CTA-pair and fused tiles only");
  }
  if (tile->cta_pair != 0 && h->pair_clusters <= 0)
    return fail(DDF_ERR_UNSUPPORTED, "CTA-pair clusters do not fit on this device");
  clear_graphs(h);  // weight maps and launch shapes change
  (which == 1 ? h->tile_first : h->tile) =
      ddf::TcTile{bn, ew, tile->cta_pair != 0, tile->staged != 0, tile->fused_encode != 0};
  if (h->bn != h->tile.bn) h->tmBtr.clear();  // boxes of the old bn
  h->bn = h->tile.bn;
  h->tile_auto = false;
  if (h->loaded && h->cfg.precision != DDF_FP32) {
    DeviceGuard g(h->cfg.device);
    DDF_CK(cudaDeviceSynchronize());  // launches in flight keep their own copies of the maps
    return build_weight_maps(h);
  }
  return DDF_OK;
}

ddf_status ddf_get_tile(ddf_handle h, int32_t which, ddf_tile* tile) {
  if (h == nullptr || tile == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL argument");
  if (which != 0 && which != 1) return fail(DDF_ERR_INVALID_ARG, "which must be 0 or 1");
  const ddf::TcTile& t = which == 1 ? h->tile_first : h->tile;
  tile->bn = t.bn;
  tile->epi_warps = t.epi_warps;
  tile->cta_pair = t.pair ? 1 : 0;
  tile->staged = t.staged ? 1 : 0;
  tile->fused_encode = t.fused ? 1 : 0;
  return DDF_OK;
}

namespace ddfi {

// the last kFusedCands candidates are layer-1 only (phase 2)
constexpr int kTileCands = 9;
constexpr int kFusedCands = 2;
constexpr int kMsSlots = 2 * kTileCands;
const ddf_tile kCands[kTileCands] = {{256, 4, 0, 0, 0}, {256, 8, 0, 0, 0}, {128, 4, 0, 0, 0},
                                     {128, 8, 0, 0, 0}, {256, 4, 1, 0, 0}, {256, 4, 1, 1, 0},
                                     {256, 8, 1, 1, 0}, {256, 4, 0, 1, 1}, {256, 8, 0, 1, 1}};

bool cand_ok(ddf_s* h, const ddf_tile& c) {
  if (c.fused_encode != 0)
    return h->cfg.kind == DDF_KIND_RAY && h->cfg.hidden_layers >= 2 &&
           ddf::tc_layer1_supported(h->cfg.octaves, h->cfg.width);
  return h->cfg.width % c.bn == 0 && (c.cta_pair == 0 || h->pair_clusters > 0);
}

}  // namespace ddfi

ddf_status ddf_autotune(ddf_handle h, const float* const rays[6], int64_t n, void* stream,
                        double* ms_out, int32_t n_out) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (n <= 0 || n > (int64_t{1} << 24)) return fail(DDF_ERR_INVALID_ARG, "tune on 1 .. 2^24 rays");
  if (ms_out != nullptr && n_out < kMsSlots)
    return fail(DDF_ERR_INVALID_ARG, "ms_out needs 16 entries");
  if (ms_out != nullptr)
    for (int i = 0; i < kMsSlots; ++i) ms_out[i] = -1.0;
  if (h->cfg.precision == DDF_FP32 || h->cfg.kind == DDF_KIND_HASHGRID)
    return DDF_OK;  // one kernel shape, nothing to choose
  DeviceGuard g(h->cfg.device);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* buf = nullptr;
  DDF_CK(cudaMalloc(&buf, 4 * n * sizeof(float)));
  std::vector<float> ref_t(n), ref_v(n), got_t(n), got_v(n);
  ddf_tile keep_h, keep_f;
  ddf_get_tile(h, 0, &keep_h);
  ddf_get_tile(h, 1, &keep_f);
  const bool keep_prof = h->prof, keep_auto = h->tile_auto;
  h->prof = false;
  bool have_ref = false;
  ddf_status result = DDF_OK;
  // Runs the query once with the current tiles and checks it against the
  // reference (the first configuration run); false if rejected.
  auto check = [&](bool* ok) -> ddf_status {
    *ok = false;
    ddf::HeadOut o{};
    o.t = buf + (have_ref ? 2 * n : 0);
    o.vis = o.t + n;
    ddf_status r = run_query(h, rays, n, o, st);
    if (r != DDF_OK) return r;
    if (cudaStreamSynchronize(st) != cudaSuccess) return fail(DDF_ERR_CUDA, "autotune: launch failed");
    std::vector<float>& tt = have_ref ? got_t : ref_t;
    std::vector<float>& vv = have_ref ? got_v : ref_v;
    cudaMemcpy(tt.data(), o.t, n * sizeof(float), cudaMemcpyDeviceToHost);
    cudaMemcpy(vv.data(), o.vis, n * sizeof(float), cudaMemcpyDeviceToHost);
    if (have_ref) {
      double worst = 0.0;
      for (int64_t i = 0; i < n; ++i) {
        worst = std::max(worst, std::fabs(double(got_t[i]) - ref_t[i]) / std::max(1.0, std::fabs(double(ref_t[i]))));
        worst = std::max(worst, std::fabs(double(got_v[i]) - ref_v[i]) / std::max(1.0, std::fabs(double(ref_v[i]))));
      }
      if (!(worst <= 1e-3)) return DDF_OK;  // rejected
    }
    have_ref = true;
    *ok = true;
    return DDF_OK;
  };
  // Device time of one query with the current tiles, from the per-launch
  // events of the profiling classes: every class (phase 1) or only the
  // encoding and layer 1 (phase 2). The events used here are released again.
  auto timed = [&](bool first_only, double* ms) -> ddf_status {
    const size_t k0 = h->recs.size(), e0 = h->ev_used;
    ddf::HeadOut o{};
    o.t = buf + 2 * n;
    o.vis = o.t + n;
    h->prof = true;
    ddf_status r = run_query(h, rays, n, o, st);
    h->prof = false;
    if (r == DDF_OK && cudaStreamSynchronize(st) != cudaSuccess)
      r = fail(DDF_ERR_CUDA, "autotune: launch failed");
    double sum = 0.0;
    for (size_t i = k0; r == DDF_OK && i < h->recs.size(); ++i) {
      const auto& rec = h->recs[i];
      if (first_only && rec.cls != kProfEncode && rec.cls != kProfFirst) continue;
      float t = 0.f;
      cudaEventElapsedTime(&t, rec.a, rec.b);
      sum += t;
    }
    h->recs.resize(k0);
    h->ev_used = e0;
    *ms = sum;
    return r;
  };
  // Candidates are checked once, then timed round-robin; each keeps its best
  // round, so a clock that drifts while the GPU warms up (power cap) affects
  // every candidate alike instead of the ones tried last.
  constexpr int kRounds = 3;
  auto tune = [&](int which_set, int n_cands, bool first_only, double* best_ms) -> int {
    std::vector<double> ms(n_cands, 1e30);
    std::vector<char> ok(n_cands, 0);
    for (int c = 0; c < n_cands && result == DDF_OK; ++c) {
      if (!cand_ok(h, kCands[c])) continue;
      if (which_set != 0 && (result = ddf_set_tile(h, 0, &kCands[c])) != DDF_OK) break;
      if ((result = ddf_set_tile(h, 1, &kCands[c])) != DDF_OK) break;
      bool pass = false;
      if ((result = check(&pass)) != DDF_OK) break;
      ok[c] = pass;
    }
    for (int round = 0; round < kRounds && result == DDF_OK; ++round) {
      for (int c = 0; c < n_cands && result == DDF_OK; ++c) {
        if (!ok[c]) continue;
        if (which_set != 0 && (result = ddf_set_tile(h, 0, &kCands[c])) != DDF_OK) break;
        if ((result = ddf_set_tile(h, 1, &kCands[c])) != DDF_OK) break;
        double t = 0.0;
        if ((result = timed(first_only, &t)) != DDF_OK) break;
        ms[c] = std::min(ms[c], t);
      }
    }
    int best = -1;
    for (int c = 0; c < n_cands; ++c) {
      if (!ok[c]) continue;
      best_ms[c] = ms[c];
      if (best < 0 || ms[c] < ms[best]) best = c;
    }
    return best;
  };
  // phase 1: one tile for every layer; phase 2: the first layer's own tile
  double p1[kTileCands], p2[kTileCands];
  for (int c = 0; c < kTileCands; ++c) p1[c] = p2[c] = -1.0;
  const int best_h = tune(1, kTileCands - kFusedCands, false, p1);
  int best_f = -1;
  if (result == DDF_OK && best_h >= 0) {
    result = ddf_set_tile(h, 0, &kCands[best_h]);
    if (result == DDF_OK) best_f = tune(0, kTileCands, true, p2);
  }
  // the kernels this batch takes where no tile is set, against the tiles just
  // chosen, unless they are among the candidates (from mid_rows on)
  const ddf_tile plain{h->cfg.width % 256 == 0 ? 256 : 128, 4, 0, 0, 0};
  const bool own = h->narrow || (!h->tmSmall.empty() &&
                                 (h->tmBig.empty() ||
                                  std::min<int64_t>(n, h->chunk) <
                                      mid_rows(h->cfg.width, h->num_sms,
                                               h->cfg.precision == DDF_FP8_E4M3)));
  auto choose = [&](bool untuned) -> ddf_status {
    ddf_status r = ddf_set_tile(h, 0, untuned ? &plain : &kCands[best_h]);
    if (r == DDF_OK) r = ddf_set_tile(h, 1, untuned ? &plain : &kCands[best_f]);
    h->tile_auto = r == DDF_OK && untuned;
    return r;
  };
  // Device time of a whole query, launches of which may overlap: enqueued behind
  // another one, so that the host is ahead.
  auto whole = [&](double* ms) -> ddf_status {
    ddf::HeadOut o{};
    o.t = buf + 2 * n;
    o.vis = o.t + n;
    cudaEvent_t a = nullptr, b = nullptr;
    ddf_status r = run_query(h, rays, n, o, st);
    float t = 0.f;
    cudaError_t e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    if (e == cudaSuccess) e = cudaEventRecord(a, st);
    if (r == DDF_OK && e == cudaSuccess) r = run_query(h, rays, n, o, st);
    if (e == cudaSuccess) e = cudaEventRecord(b, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, a, b);
    if (a != nullptr) cudaEventDestroy(a);
    if (b != nullptr) cudaEventDestroy(b);
    *ms = t;
    return r != DDF_OK || e == cudaSuccess ? r : cuda_fail(e, "autotune: timing a query");
  };
  bool untuned_wins = false;
  if (result == DDF_OK && best_f >= 0 && own && (result = choose(true)) == DDF_OK) {
    double best[2] = {1e30, 1e30};
    bool pass = false;
    result = check(&pass);
    for (int k = 0; k < 2 * kRounds && result == DDF_OK && pass; ++k) {
      double t = 0.0;
      if ((result = choose(k % 2 == 0)) == DDF_OK && (result = whole(&t)) == DDF_OK)
        best[k % 2] = std::min(best[k % 2], t);
    }
    untuned_wins = pass && best[0] <= best[1];
  }
  for (int c = 0; ms_out != nullptr && c < kTileCands; ++c) {
    ms_out[c] = p1[c];
    ms_out[kTileCands + c] = p2[c];
  }
  h->prof = keep_prof;
  cudaFree(buf);
  if (result != DDF_OK || best_h < 0 || best_f < 0) {
    ddf_set_tile(h, 0, &keep_h);
    ddf_set_tile(h, 1, &keep_f);
    h->tile_auto = keep_auto;
    return result != DDF_OK ? result : fail(DDF_ERR_CUDA, "autotune: no candidate passed");
  }
  return choose(untuned_wins);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Internal helpers for queries whose workspace is supplied by the caller
// instead of the handle (used by the allocation-free entry point in
// noalloc.cu). Not part of the public header.

namespace {

// Loads the kernels of every batch size for the handle's precision, once a
// device (asking for them again would cost a new handle's first call 7 us).
ddf_status load_size_kernels(ddf_s* h) {
  constexpr int kDevices = 64;
  static std::atomic<unsigned> loaded[kDevices] = {};  // bit 0: bf16, bit 1: e4m3
  const bool fp8 = h->cfg.precision == DDF_FP8_E4M3;
  const unsigned bit = fp8 ? 2u : 1u;
  const int dev = h->cfg.device;
  if (dev < kDevices && (loaded[dev].load(std::memory_order_relaxed) & bit) != 0) return DDF_OK;
  DDF_CK(ddf::load_small_kernels(fp8));
  DDF_CK(ddf::load_step_query_kernels(fp8));
  if (dev < kDevices) loaded[dev].fetch_or(bit, std::memory_order_relaxed);
  return DDF_OK;
}

}  // namespace

size_t ddf_internal_workspace_bytes(ddf_handle h, int64_t rows) {
  if (h->cfg.kind == DDF_KIND_HASHGRID) return 0;  // one fused kernel, no scratch
  const int W = h->cfg.width;
  const bool f32 = h->cfg.precision == DDF_FP32;
  const size_t act_elem = f32 ? 4 : (h->cfg.precision == DDF_BF16 ? 2 : 1);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  size_t total = up(static_cast<size_t>(rows) * (f32 ? h->kp32 * 4 : h->kp16 * 2));
  total += 2 * up(static_cast<size_t>(rows) * W * act_elem);
  if (!f32) total += up(static_cast<size_t>(rows) * max_partials(W) * sizeof(float2));
  return total;
}

int ddf_internal_device(ddf_handle h) { return h->cfg.device; }

// Runs ddf_query_rays with its encode / activation / partial-sum buffers
// carved out of `ws` (256-byte aligned, ws_bytes long) instead of the
// handle's own workspace. The caller has checked that ws is large enough for
// n rays in one chunk. The handle's workspace pointers are swapped in for the
// launches and restored before returning (launch parameters are captured at
// launch time); event timing is suspended so no event objects are created.
ddf_status ddf_internal_query_in_workspace(ddf_handle h, const float* const rays[6], int64_t n,
                                           float* out_t, float* out_vis, void* stream, void* ws,
                                           size_t ws_bytes) {
  ddf_status s = check_ready(h);
  if (s != DDF_OK) return s;
  if ((s = check_rays(rays, n)) != DDF_OK) return s;
  if (n > 0 && (out_t == nullptr || out_vis == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "output pointer is NULL");
  if (n == 0) return DDF_OK;
  if (ws == nullptr || ddf_internal_workspace_bytes(h, n) > ws_bytes)
    return fail(DDF_ERR_INVALID_ARG, "workspace too small for this batch");
  DeviceGuard g(h->cfg.device);
  // a batch of another size may come in a frame, or while a stream is captured;
  // other fields have the same kernels for every size
  if (h->tile_auto && !h->tmSmall.empty() && (s = load_size_kernels(h)) != DDF_OK) return s;
  const int W = h->cfg.width;
  const bool f32 = h->cfg.precision == DDF_FP32;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  // FP32 on the tensor cores keeps 6 bytes a value, of as many rows at a time
  // as fit (the same results, every row being independent of the others)
  const bool planes = f32 && h->f32_clusters > 0;
  int64_t rows = n;
  if (planes) {
    const size_t per_row = 6 * (static_cast<size_t>(h->kp32) + 2 * W);
    rows = std::min<int64_t>(n, static_cast<int64_t>((ws_bytes - 3 * 256) / per_row));
    if (rows > 256) rows = std::min<int64_t>(n, rows / 256 * 256);
    if (rows < 1) return fail(DDF_ERR_INVALID_ARG, "workspace too small for this batch");
  }
  const size_t act_elem = planes ? 6 : f32 ? 4 : (h->cfg.precision == DDF_BF16 ? 2 : 1);
  uint8_t* p = static_cast<uint8_t*>(ws);
  void* enc = p;
  p += up(static_cast<size_t>(rows) * (f32 ? h->kp32 * (planes ? 6 : 4) : h->kp16 * 2));
  void* act0 = p;
  p += up(static_cast<size_t>(rows) * W * act_elem);
  void* act1 = p;
  p += up(static_cast<size_t>(rows) * W * act_elem);
  float2* part = f32 ? nullptr : reinterpret_cast<float2*>(p);
  if (!f32) p += up(static_cast<size_t>(n) * max_partials(W) * sizeof(float2));
  // the small-batch tiles' FP32 activations, where the scratch has room
  const bool room = !f32 && small_batches(h) && n <= small_rows(W, h->num_sms) &&
                    static_cast<size_t>(p - static_cast<uint8_t*>(ws)) +
                            static_cast<size_t>(n) * W * sizeof(float) <= ws_bytes;
  float* const save_x = h->ws_x;
  const int64_t save_x_rows = h->ws_x_rows;
  h->ws_x = room ? reinterpret_cast<float*>(p) : nullptr;
  h->ws_x_rows = room ? n : 0;

  void* save_enc = h->ws_enc;
  void* save_act0 = h->ws_act[0];
  void* save_act1 = h->ws_act[1];
  float2* save_part = h->ws_part;
  const int64_t save_rows = h->ws_rows, save_chunk = h->chunk;
  const bool save_prof = h->prof;
  h->ws_enc = enc;
  h->ws_act[0] = act0;
  h->ws_act[1] = act1;
  h->ws_part = part;
  h->ws_rows = n;
  h->chunk = n;
  h->prof = false;
  const int64_t save_pass = h->f32_pass;
  if (planes) h->f32_pass = rows;
  ddf::HeadOut o{};
  o.t = out_t;
  o.vis = out_vis;
  s = run_query(h, rays, n, o, static_cast<cudaStream_t>(stream));
  h->f32_pass = save_pass;
  h->ws_enc = save_enc;
  h->ws_act[0] = save_act0;
  h->ws_act[1] = save_act1;
  h->ws_part = save_part;
  h->ws_x = save_x;
  h->ws_x_rows = save_x_rows;
  h->ws_rows = save_rows;
  h->chunk = save_chunk;
  h->prof = save_prof;
  return s;
}

// Records msg as the calling thread's last error and returns s.
ddf_status ddf_internal_set_error(ddf_status s, const char* msg) { return fail(s, msg); }

// ---------------------------------------------------------------------------
// Shadow and AO images (the application of Sec. 3.3).

namespace ddfi {

ddf_status camera_basis(const float camera[10], int32_t width, int32_t height,
                        ddf::GiCamera* cam) {
  // basis in double, as the pinhole model defines it
  double e[3], f[3], up[3];
  for (int c = 0; c < 3; ++c) e[c] = camera[c], f[c] = camera[3 + c] - camera[c], up[c] = camera[6 + c];
  const double fl = std::sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
  if (!(fl > 0.0)) return fail(DDF_ERR_INVALID_ARG, "eye and target coincide");
  for (double& v : f) v /= fl;
  double r[3] = {f[1] * up[2] - f[2] * up[1], f[2] * up[0] - f[0] * up[2], f[0] * up[1] - f[1] * up[0]};
  const double rl = std::sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
  if (!(rl > 0.0)) return fail(DDF_ERR_INVALID_ARG, "up is parallel to the view direction");
  for (double& v : r) v /= rl;
  const double u[3] = {r[1] * f[2] - r[2] * f[1], r[2] * f[0] - r[0] * f[2], r[0] * f[1] - r[1] * f[0]};
  const double th = std::tan(0.5 * static_cast<double>(camera[9]));
  if (!(th > 0.0) || !std::isfinite(th) || !(camera[9] < 3.14159265358979323846))
    return fail(DDF_ERR_INVALID_ARG, "fov_y must be in (0, pi)");
  for (int c = 0; c < 3; ++c) {
    if (!std::isfinite(e[c])) return fail(DDF_ERR_INVALID_ARG, "camera eye is not finite");
    cam->eye[c] = static_cast<float>(e[c]);
    cam->f[c] = static_cast<float>(f[c]);
    cam->r[c] = static_cast<float>(r[c]);
    cam->u[c] = static_cast<float>(u[c]);
  }
  cam->tan_half = static_cast<float>(th);
  cam->width = width;
  cam->height = height;
  return DDF_OK;
}

}  // namespace ddfi

extern "C" ddf_status ddf_render_gi(ddf_handle h, const float* spheres, int32_t n_spheres,
                                    const float* boxes, int32_t n_boxes, const float camera[10],
                                    int32_t width, int32_t height, const float light[3],
                                    int32_t ao_samples, uint64_t seed, float* out_shadow,
                                    float* out_ao, void* stream) {
  if (camera == nullptr || light == nullptr) return fail(DDF_ERR_INVALID_ARG, "NULL camera or light");
  if (width < 1 || height < 1 || static_cast<int64_t>(width) * height > (int64_t{1} << 26))
    return fail(DDF_ERR_INVALID_ARG, "width, height >= 1 and at most 2^26 pixels");
  const int k = out_ao != nullptr ? ao_samples : 0;
  if (out_ao != nullptr && (ao_samples < 1 || ao_samples > 1024))
    return fail(DDF_ERR_INVALID_ARG, "ao_samples must be in [1, 1024]");
  if (n_spheres < 0 || n_boxes < 0 || n_spheres > 1024 || n_boxes > 1024)
    return fail(DDF_ERR_INVALID_ARG, "0..1024 spheres and 0..1024 boxes");
  if ((n_spheres > 0 && spheres == nullptr) || (n_boxes > 0 && boxes == nullptr))
    return fail(DDF_ERR_INVALID_ARG, "primitive array is NULL");
  DDF_REQUIRE_ALIGNED(spheres, 4);
  DDF_REQUIRE_ALIGNED(boxes, 4);
  DDF_REQUIRE_ALIGNED(out_shadow, 4);
  DDF_REQUIRE_ALIGNED(out_ao, 4);
  ddf_status s = DDF_OK;
  if (h != nullptr && (s = check_ready(h)) != DDF_OK) return s;
  ddf::GiCamera cam{};
  if ((s = camera_basis(camera, width, height, &cam)) != DDF_OK) return s;
  int dev = 0;
  if (h != nullptr) dev = h->cfg.device;
  else DDF_CK(cudaGetDevice(&dev));
  DeviceGuard g(dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t npx = static_cast<int64_t>(width) * height;
  const int64_t n2 = npx * (1 + k);
  // shading points, normals, 6 ray arrays, t, hit flags
  const size_t bytes = npx * sizeof(float4) + 3 * npx * sizeof(float) + 7 * n2 * sizeof(float) + n2;
  uint8_t* buf = nullptr;
  DDF_CK(cudaMalloc(&buf, bytes));
  float4* sp = reinterpret_cast<float4*>(buf);
  float* nrm = reinterpret_cast<float*>(sp + npx);
  float* rp = nrm + 3 * npx;
  float* t = rp + 6 * n2;
  uint8_t* hit = reinterpret_cast<uint8_t*>(t + n2);
  ddf::RayOut ro;
  const float* rc[6];
  for (int c = 0; c < 6; ++c) ro.p[c] = rp + c * n2, rc[c] = ro.p[c];
  cudaError_t ce = ddf::launch_gi_primary(cam, spheres, n_spheres, boxes, n_boxes, sp, nrm, st);
  if (ce == cudaSuccess) ce = ddf::launch_gi_rays(sp, nrm, npx, k, seed, light, ro, st);
  if (ce != cudaSuccess) s = cuda_fail(ce, "gi ray generation");
  if (s == DDF_OK) {
    if (h != nullptr) {
      ddf::HeadOut o{};
      o.t = t;
      o.hit = hit;
      s = run_query(h, rc, n2, o, st);
    } else {
      ddf::RaySoA rs;
      for (int c = 0; c < 6; ++c) rs.p[c] = rc[c];
      ce = ddf::launch_cast_scene(spheres, n_spheres, boxes, n_boxes, rs, n2, t, hit, st);
      if (ce != cudaSuccess) s = cuda_fail(ce, "cast");
    }
  }
  if (s == DDF_OK) {
    ce = ddf::launch_gi_compose(sp, npx, k, light, t, hit, out_shadow, out_ao, st);
    if (ce != cudaSuccess) s = cuda_fail(ce, "gi compose");
  }
  ce = cudaStreamSynchronize(st);
  cudaFree(buf);
  if (s == DDF_OK && ce != cudaSuccess) s = cuda_fail(ce, "cudaStreamSynchronize");
  return s;
}

