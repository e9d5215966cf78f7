// The two small steps either side of the denoising loop that belong to the model adapter (paper, Sec. "Architecture":
// the adapter owns preprocessing, cache layout and action conversion): packing a backbone's padded per-layer K / V
// into the library's ragged prefix-KV layout, and converting the raw action chunk (x at t = 0) into robot actions.
// Both are pure data movement / element-wise work: coalesced 16-byte copies, one thread per output element.
#include <cstdio>
#include <new>

#include "../../include/phyai.h"
#include "kernels.h"

namespace phyai {
namespace {

thread_local char g_ad_err[256] = "";

// cu[0] = 0, cu[b + 1] = cu[b] + lens[b]; a length outside 0..p_max or a total beyond kv_tokens raises the status word
// (INVALID_ARG) and the pack kernel then copies nothing; with `clear` the word is written either way.  One block: a thread sums a run of lengths, the runs are scanned.
__global__ void __launch_bounds__(1024) k_kv_scan(const int* lens, int batch, int p_max, unsigned long long kv_tokens, int* cu, int* status, int clear) {
  __shared__ long long wsum[32];
  pdl_launch_dependents();
  const int per = (batch + 1023) / 1024, b0 = min(batch, (int)threadIdx.x * per), b1 = min(batch, b0 + per);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool bad = false;
  long long sum = 0;
  for (int b = b0; b < b1; ++b) {
    const int n = lens[b];
    if (n < 0 || n > p_max) bad = true;
    sum += max(n, 0);
  }
  long long run = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long v = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += v;
  }
  if (lane == 31) wsum[warp] = run;
  __syncthreads();
  long long acc = run - sum;
  for (int w = 0; w < warp; ++w) acc += wsum[w];
  if (threadIdx.x == 0) cu[0] = 0;
  for (int b = b0; b < b1; ++b) {
    acc += max(lens[b], 0);
    cu[b + 1] = (int)min(acc, 0x7fffffffLL);
  }
  if (b1 == batch && b0 < b1 && (unsigned long long)acc > kv_tokens) bad = true;
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0 && (bad || clear)) atomicExch(status, bad ? ST_INVALID_ARG : 0);
}

// src [L][B][p_max][row_bytes], dst [L][2][kv_tokens][row_bytes]: plane (l, kv) of request b, rows p < lens[b], go to
// rows cu[b] + p.  The rows of a request are one contiguous run on both sides: a block moves 16 KB of it (grid.x) of one
// plane (grid.y) and request (grid.z), its loads issued before the dependency wait (only the destination needs cu).  With
// `zero_tail` the entry grid.z = batch clears the rows past the last request (after an error: all rows).  For more requests than the
// threads of a block; else k_kv_pack_small.
constexpr int PACK_T = 256, PACK_U = 4, PACK_CHUNK = PACK_T * PACK_U;
__global__ void __launch_bounds__(PACK_T) k_kv_pack(const uint4* k, const uint4* v, const int* lens, const int* cu, const int* status, uint4* dst,
                                                    int batch, int p_max, unsigned long long kv_tokens, int row_chunks, int zero_tail) {
  const int layer = blockIdx.y >> 1, is_v = blockIdx.y & 1;
  uint4* out = dst + (size_t)blockIdx.y * kv_tokens * row_chunks;
  bool waited = false;
  for (int b = blockIdx.z; b < batch + zero_tail; b += gridDim.z) {
    if (b == batch) {
      if (!waited) pdl_wait();
      waited = true;
      const size_t lo = status_set(status) ? 0 : (size_t)cu[batch] * row_chunks, hi = kv_tokens * row_chunks;
      for (size_t i = lo + (size_t)blockIdx.x * PACK_T + threadIdx.x; i < hi; i += (size_t)gridDim.x * PACK_T) out[i] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const int n = min(max(lens[b], 0), p_max) * row_chunks;
    const uint4* src = (is_v ? v : k) + ((size_t)layer * batch + b) * p_max * row_chunks;
    uint4 x[PACK_U];
    const int i0 = (int)blockIdx.x * PACK_CHUNK + (int)threadIdx.x;
#pragma unroll
    for (int u = 0; u < PACK_U; ++u)
      if (i0 + u * PACK_T < n) x[u] = __ldcs(src + i0 + u * PACK_T);
    if (!waited) pdl_wait();
    waited = true;
    if ((int)blockIdx.x * PACK_CHUNK >= n || status_set(status)) continue;
    uint4* o = out + (size_t)cu[b] * row_chunks + i0;
#pragma unroll
    for (int u = 0; u < PACK_U; ++u)
      if (i0 + u * PACK_T < n) o[u * PACK_T] = x[u];
  }
}

// The same in one launch, for up to PACK_T requests: every block adds the lengths up itself while its loads are on their way, block
// (0, 0, 0) also writes cu and the status word.  Bound by HBM: with the post-processing launch of the actions 8 requests of the pi0 shape
// (258 MB moved) 45.8 us, behind a scan kernel 51.7; 1 request 20.8 / 26.8, 32 requests 166 / 175.  (Eight loads per thread instead of
// four 46.6 / 167.8; streaming stores 45.1 for 8 requests but 171 for 32.)
__global__ void __launch_bounds__(PACK_T) k_kv_pack_small(const uint4* k, const uint4* v, const int* lens, int* cu, int* status, uint4* dst, int batch,
                                                          int p_max, unsigned long long kv_tokens, int row_chunks, int clear) {
  __shared__ long long wsum[2][PACK_T / 32];
  const int layer = blockIdx.y >> 1, is_v = blockIdx.y & 1, b = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint4* out = dst + (size_t)blockIdx.y * kv_tokens * row_chunks;
  const int raw = tid < batch ? lens[tid] : 0;
  const int n = b < batch ? min(max(lens[b], 0), p_max) * row_chunks : 0;
  const uint4* src = (is_v ? v : k) + ((size_t)layer * batch + b) * p_max * row_chunks;
  uint4 x[PACK_U];
  const int i0 = (int)blockIdx.x * PACK_CHUNK + tid;
  const bool first = blockIdx.x == 0 && blockIdx.y == 0 && b == 0;
  if (b < batch && (int)blockIdx.x * PACK_CHUNK >= n && !first) return;
#pragma unroll
  for (int u = 0; u < PACK_U; ++u)
    if (i0 + u * PACK_T < n) x[u] = __ldcs(src + i0 + u * PACK_T);
  // ---- rows ahead of this request, all rows
  long long run = max(raw, 0);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long up = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += up;
  }
  if (lane == 31) wsum[0][warp] = run;
  bool bad = __syncthreads_or(raw < 0 || raw > p_max);
  long long total = 0;
#pragma unroll
  for (int w = 0; w < PACK_T / 32; ++w) {
    if (w == warp) run += total;
    total += wsum[0][w];
  }
  if (tid == (b > 0 ? b - 1 : 0)) wsum[1][0] = b > 0 ? run : 0;            // (inclusive sum of the request before)
  bad |= (unsigned long long)total > kv_tokens;
  __syncthreads();
  const long long pre = wsum[1][0];
  if (first) {
    if (tid < batch) cu[tid + 1] = (int)min(run, 0x7fffffffLL);
    if (tid == 0) {
      cu[0] = 0;
      if (bad || clear) atomicExch(status, bad ? ST_INVALID_ARG : 0);
    }
  }
  if (b == batch) {
    const size_t lo = bad ? 0 : (size_t)total * row_chunks, hi = kv_tokens * row_chunks;
    for (size_t i = lo + (size_t)blockIdx.x * PACK_T + tid; i < hi; i += (size_t)gridDim.x * PACK_T) out[i] = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  if (bad || (!clear && status_set(status))) return;      // (a word raised before: nothing is copied, unless the call clears it)
  uint4* o = out + (size_t)pre * row_chunks + i0;
#pragma unroll
  for (int u = 0; u < PACK_U; ++u)
    if (i0 + u * PACK_T < n) o[u * PACK_T] = x[u];
}

// out[b][h][a] = (clip(x[b][h][a]) + 1) / 2 * (q99[a] - q01[a]) + q01[a] for h < H_out, a < A_out
__global__ void k_postprocess(const float* x, const float* q01, const float* q99, float* out, int batch, int H, int A,
                              int H_out, int A_out, float lo, float hi, int do_clip) {
  const size_t total = (size_t)batch * H_out * A_out;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int a = (int)(i % A_out), hh = (int)((i / A_out) % H_out), b = (int)(i / ((size_t)A_out * H_out));
    float v = x[((size_t)b * H + hh) * A + a];
    if (do_clip) v = fminf(fmaxf(v, lo), hi);
    const float lo_q = q01 ? q01[a] : -1.0f, hi_q = q99 ? q99[a] : 1.0f;
    out[i] = (v + 1.0f) * 0.5f * (hi_q - lo_q) + lo_q;
  }
}

}  // namespace
}  // namespace phyai

extern "C" {

const char* phyai_adapter_last_error(void) { return phyai::g_ad_err; }

static phyai_status_t pack_prefix_kv(const phyai_kv_pack_desc_t* desc, const void* k, const void* v, const int32_t* lens, void* prefix_kv,
                                     uint64_t kv_tokens, int32_t* cu_prefix_lens, int32_t* status_word, int cleared, void* stream) {
  using namespace phyai;
  auto bad = [](const char* m) {
    snprintf(g_ad_err, sizeof(g_ad_err), "%s", m);
    return PHYAI_ERR_INVALID_ARG;
  };
  if (!desc || desc->struct_size != sizeof(phyai_kv_pack_desc_t)) return bad("desc is NULL or has a wrong struct_size");
  if (!k || !v || !lens || !prefix_kv || !cu_prefix_lens || !status_word) return bad("a pointer argument is NULL");
  if (!desc->n_layers || !desc->n_kv_heads || !desc->head_dim || !desc->batch || !desc->p_max)
    return bad("a size in desc is zero");
  if (desc->elem_bytes != 2 && desc->elem_bytes != 4) return bad("elem_bytes must be 2 (bfloat16) or 4 (float32)");
  const size_t row_bytes = (size_t)desc->n_kv_heads * desc->head_dim * desc->elem_bytes;
  if (row_bytes % 16) return bad("n_kv_heads * head_dim * elem_bytes must be a multiple of 16");
  if ((reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(prefix_kv)) & 15u)
    return bad("k, v and prefix_kv must be 16-byte aligned");
  if (kv_tokens > 0x7fffffffull || desc->batch > 65535u || desc->n_layers > 32767u || desc->p_max * (row_bytes / 16) > 0x7fffffffull)
    return bad("kv_tokens, batch, p_max or n_layers too large");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int chunks = (int)(row_bytes / 16), B = (int)desc->batch;
  const unsigned gx = (unsigned)(((size_t)desc->p_max * chunks + PACK_CHUNK - 1) / PACK_CHUNK);
  if (B <= PACK_T) {
    k_kv_pack_small<<<dim3(gx, desc->n_layers * 2, B + cleared), PACK_T, 0, st>>>(reinterpret_cast<const uint4*>(k), reinterpret_cast<const uint4*>(v), lens,
                                                                                  cu_prefix_lens, status_word, reinterpret_cast<uint4*>(prefix_kv), B,
                                                                                  (int)desc->p_max, (unsigned long long)kv_tokens, chunks, cleared);
    const cudaError_t es = cudaGetLastError();
    if (es == cudaSuccess) return PHYAI_OK;
    snprintf(g_ad_err, sizeof(g_ad_err), "kernel launch failed: %s", cudaGetErrorString(es));
    return PHYAI_ERR_CUDA;
  }
  k_kv_scan<<<1, 1024, 0, st>>>(lens, B, (int)desc->p_max, kv_tokens, cu_prefix_lens, status_word, cleared);
  cudaError_t e = launch_pdl(k_kv_pack, dim3(gx, desc->n_layers * 2, B + cleared < 65535 ? B + cleared : 65535), dim3(PACK_T), 0, st,
                             reinterpret_cast<const uint4*>(k), reinterpret_cast<const uint4*>(v), (const int*)lens, (const int*)cu_prefix_lens,
                             (const int*)status_word, reinterpret_cast<uint4*>(prefix_kv), B, (int)desc->p_max,
                             (unsigned long long)kv_tokens, chunks, cleared);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    snprintf(g_ad_err, sizeof(g_ad_err), "kernel launch failed: %s", cudaGetErrorString(e));
    return PHYAI_ERR_CUDA;
  }
  return PHYAI_OK;
}

phyai_status_t phyai_pack_prefix_kv(const phyai_kv_pack_desc_t* desc, const void* k, const void* v, const int32_t* lens, void* prefix_kv,
                                    uint64_t kv_tokens, int32_t* cu_prefix_lens, int32_t* status_word, void* stream) {
  return pack_prefix_kv(desc, k, v, lens, prefix_kv, kv_tokens, cu_prefix_lens, status_word, 0, stream);
}
phyai_status_t phyai_pack_prefix_kv_cleared(const phyai_kv_pack_desc_t* desc, const void* k, const void* v, const int32_t* lens,
                                            void* prefix_kv, uint64_t kv_tokens, int32_t* cu_prefix_lens, int32_t* status_word, void* stream) {
  return pack_prefix_kv(desc, k, v, lens, prefix_kv, kv_tokens, cu_prefix_lens, status_word, 1, stream);
}

phyai_status_t phyai_postprocess_actions(const float* x, uint32_t batch, uint32_t horizon, uint32_t action_dim,
                                         const float* q01, const float* q99, float clip_lo, float clip_hi,
                                         uint32_t out_horizon, uint32_t out_dim, float* out, void* stream) {
  using namespace phyai;
  if (!x || !out || !batch || !horizon || !action_dim || !out_horizon || !out_dim || out_horizon > horizon ||
      out_dim > action_dim || ((q01 == nullptr) != (q99 == nullptr))) {
    snprintf(g_ad_err, sizeof(g_ad_err), "NULL pointer, zero size, out_horizon > horizon, out_dim > action_dim, or only one of q01 / q99 given");
    return PHYAI_ERR_INVALID_ARG;
  }
  const size_t total = (size_t)batch * out_horizon * out_dim;
  const int blocks = (int)((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024);
  k_postprocess<<<blocks, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(x, q01, q99, out, (int)batch, (int)horizon,
                                                                           (int)action_dim, (int)out_horizon, (int)out_dim,
                                                                           clip_lo, clip_hi, clip_lo < clip_hi ? 1 : 0);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    snprintf(g_ad_err, sizeof(g_ad_err), "kernel launch failed: %s", cudaGetErrorString(e));
    return PHYAI_ERR_CUDA;
  }
  return PHYAI_OK;
}

}  // extern "C"

// Request-local K / V projections of a feature-handoff head: one GEMM on CTA pairs of the (tiled) feature rows against
// [Wk | Wv] of all layers, whose epilogue writes the bf16 rows of every layer's two planes.  The projector handle owns the
// packed weight images and the workspace, so that a run only enqueues kernels.  640 rows of 2048 features, 16 layers of
// 2 x 256 channels: 27 us (a 128-row tile GEMM with fp32 output and a conversion kernel per layer, 32 launches: 260 us).
struct phyai_kv_projector {
  int L = 0, nkv = 0, Dv = 0, max_tokens = 0, rows_pad = 0, N = 0, n_sm = 0;   // N: rows of the image, a multiple of 256
  __nv_bfloat16* wp = nullptr;    // packed [Wk | Wv] of layer 0, of layer 1, ...: blocks [N/128][Dv/64][128 x 64]
  __nv_bfloat16* xt = nullptr;    // tiled features [Dv / 64][rows_pad][64]
  int* status = nullptr;
};

namespace {
phyai_status_t proj_fail(phyai_status_t st, const char* msg, cudaError_t e = cudaSuccess) {
  using namespace phyai;
  if (e != cudaSuccess) snprintf(g_ad_err, sizeof(g_ad_err), "%s: %s", msg, cudaGetErrorString(e));
  else snprintf(g_ad_err, sizeof(g_ad_err), "%s", msg);
  return st;
}
}  // namespace

extern "C" void phyai_kv_projector_destroy(phyai_kv_projector_t* p) {
  if (!p) return;
  cudaFree(p->wp), cudaFree(p->xt), cudaFree(p->status);
  delete p;
}

extern "C" phyai_status_t phyai_kv_projector_create(const phyai_kv_proj_desc_t* desc, const void* const* wk,
                                                    const void* const* wv, uint64_t max_tokens, void* stream,
                                                    phyai_kv_projector_t** out) {
  using namespace phyai;
  g_ad_err[0] = 0;
  if (out) *out = nullptr;
  if (!desc || desc->struct_size != sizeof(phyai_kv_proj_desc_t) || !wk || !wv || !out)
    return proj_fail(PHYAI_ERR_INVALID_ARG, "NULL argument or wrong struct_size");
  const int L = (int)desc->n_layers, nkv = (int)(desc->n_kv_heads * desc->head_dim), Dv = (int)desc->feat_dim;
  if (L <= 0 || nkv <= 0 || Dv <= 0 || Dv % 64 || (2 * nkv) % 128 || max_tokens == 0 || max_tokens > (1u << 22))
    return proj_fail(PHYAI_ERR_INVALID_ARG,
                     "need feat_dim a multiple of 64, 2 * n_kv_heads * head_dim a multiple of 128, 1 <= max_tokens <= 2^22");
  for (int l = 0; l < L; ++l)
    if (!wk[l] || !wv[l]) return proj_fail(PHYAI_ERR_INVALID_ARG, "a per-layer weight pointer is NULL");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  phyai_kv_projector* p = new (std::nothrow) phyai_kv_projector();
  if (!p) return proj_fail(PHYAI_ERR_OOM, "host allocation failed");
  p->L = L, p->nkv = nkv, p->Dv = Dv, p->max_tokens = (int)max_tokens, p->rows_pad = ((int)max_tokens + 255) / 256 * 256;
  const size_t per_layer = 2 * (size_t)nkv, n_rows = (size_t)L * per_layer;
  p->N = (int)((n_rows + 255) / 256 * 256);
  if ((e = cudaMalloc(&p->wp, (size_t)Dv * p->N * 2)) != cudaSuccess || (e = cudaMalloc(&p->xt, (size_t)p->rows_pad * Dv * 2)) != cudaSuccess ||
      (e = cudaMalloc(&p->status, 4)) != cudaSuccess) {
    phyai_kv_projector_destroy(p);
    return proj_fail(PHYAI_ERR_OOM, "cudaMalloc", e);
  }
  cudaMemsetAsync(p->xt, 0, (size_t)p->rows_pad * Dv * 2, st);
  cudaMemsetAsync(p->status, 0, 4, st);
  cudaMemsetAsync(p->wp + n_rows * Dv, 0, (p->N - n_rows) * Dv * 2, st);
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) {
    phyai_kv_projector_destroy(p);
    return proj_fail(PHYAI_ERR_CUDA, "device attributes", e);
  }
  for (int l = 0; l < L; ++l) {
    launch_pack_tiled(wk[l], 1, p->wp + (size_t)l * Dv * per_layer, Dv, nkv, 0, st);
    launch_pack_tiled(wv[l], 1, p->wp + (size_t)l * Dv * per_layer, Dv, nkv, nkv, st);
  }
  e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    phyai_kv_projector_destroy(p);
    return proj_fail(PHYAI_ERR_CUDA, "weight packing", e);
  }
  *out = p;
  return PHYAI_OK;
}

extern "C" phyai_status_t phyai_kv_projector_run(phyai_kv_projector_t* p, const void* features, uint64_t tokens,
                                                 uint64_t kv_tokens, void* prefix_kv, void* stream) {
  using namespace phyai;
  g_ad_err[0] = 0;
  if (!p || !features || !prefix_kv) return proj_fail(PHYAI_ERR_INVALID_ARG, "NULL argument");
  if (tokens == 0 || tokens > (uint64_t)p->max_tokens || tokens > kv_tokens)
    return proj_fail(PHYAI_ERR_INVALID_ARG, "need 1 <= tokens <= max_tokens and tokens <= kv_tokens");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int M = (int)tokens;
  launch_rows_to_tiled(reinterpret_cast<const __nv_bfloat16*>(features), p->xt, M, p->Dv, p->rows_pad, st);
  PairGemm g{};
  g.epi = PG_PLANES, g.W = p->wp, g.w_rows = (uint64_t)p->N * (p->Dv / 64), g.X = p->xt, g.rows_pad = p->rows_pad;
  g.M = M, g.N = p->N, g.K = p->Dv, g.out = reinterpret_cast<__nv_bfloat16*>(prefix_kv), g.nkv = p->nkv, g.n_planes = 2 * p->L;
  g.plane_rows = kv_tokens, g.wait_limit = 1u << 28;
  int busy = 0;
  cudaError_t e = launch_pair_gemm(p->status, g, p->n_sm, &busy, st);
  if (e != cudaSuccess) return proj_fail(PHYAI_ERR_CUDA, "projection GEMM launch", e);
  e = cudaGetLastError();
  if (e != cudaSuccess) return proj_fail(PHYAI_ERR_CUDA, "kernel launch failed", e);
  return PHYAI_OK;
}

// One-shot form: create, run, synchronise, destroy.
extern "C" phyai_status_t phyai_project_features_kv(const phyai_kv_proj_desc_t* desc, const void* features,
                                                    const void* const* wk, const void* const* wv, uint64_t tokens,
                                                    uint64_t kv_tokens, void* prefix_kv, void* stream) {
  phyai_kv_projector_t* p = nullptr;
  phyai_status_t st = phyai_kv_projector_create(desc, wk, wv, tokens ? tokens : 1, stream, &p);
  if (st != PHYAI_OK) return st;
  st = phyai_kv_projector_run(p, features, tokens, kv_tokens, prefix_kv, stream);
  cudaError_t e = cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream));
  int hs = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&hs, p->status, 4, cudaMemcpyDeviceToHost);
  phyai_kv_projector_destroy(p);
  if (st != PHYAI_OK) return st;
  if (e != cudaSuccess) return proj_fail(PHYAI_ERR_CUDA, "feature K/V projection", e);
  if (hs != 0) return proj_fail(PHYAI_ERR_TIMEOUT, "a bounded device-side wait expired");
  return PHYAI_OK;
}
