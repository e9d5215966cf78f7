// fp32 kernels for few token rows (the CUDA-core path: true fp32 FMA, no TF32): projections with the preceding RMSNorm
// folded in, and attention of one (row, head) per block.  At these sizes nothing is throughput: a 64 x 64-tile GEMM runs on
// 4 - 16 SMs and walks K = 1024 in 64 dependent steps (27 us per launch at 17 rows).  So a block takes RM rows x 32 columns,
// sixteen warps share the contraction, every warp has sixteen weight rows in flight (the first ones requested before the
// dependency wait: they are constants), and the partial sums meet in shared memory in a fixed order: 4.6 us per
// launch in the captured loop of the tiny expert, hand-over to the next one included.
#include "kernels.h"

namespace phyai {
namespace {

constexpr int RW = 16;            // warps of a block: ranges of the contraction
constexpr int RK = 16;            // weight rows a warp has in flight

template <int RM, bool DUAL>
__global__ void __launch_bounds__(RW * 32) k_rows_f32(const int* status, const SimtGemm g) {
  extern __shared__ float As[];                              // [RM][K]
  __shared__ float red[DUAL ? 2 : 1][RW][RM][32];
  __shared__ float ssp[RW];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = blockIdx.x * 32 + lane, m0 = blockIdx.y * RM;
  const int kper = ((g.K + RW - 1) / RW + 3) & ~3, k_lo = min(g.K, warp * kper), k_hi = min(g.K, k_lo + kper);
  const bool col = n < g.N;
  pdl_launch_dependents();
  float b[RK], b2[DUAL ? RK : 1];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < RK; ++i) {
      const bool in = col && k0 + i < k_hi;
      b[i] = in ? __ldg(g.B + (size_t)(k0 + i) * g.N + n) : 0.f;
      if (DUAL) b2[i] = in ? __ldg(g.B2 + (size_t)(k0 + i) * g.N + n) : 0.f;
    }
  };
  fetch(k_lo);
  // Every load is asked for as early as its address allows (the norm's and the epilogue's constants ahead of the dependency
  // wait, the row and what the result is added to right after it): each one left where it is used costs a round trip to the L2
  // (55 launches of the tiny expert 274 -> 254 us).  Eight rows per block are for grids of several blocks per SM, which hide
  // the trips themselves and need the registers: there the norm's constants stay where they are used.
  constexpr int WPR = RW / RM, RU = RM == 4 ? 8 : 4, RG = RM == 4 ? RU : 0;
  const int row = warp / WPR, t = (warp % WPR) * 32 + lane, m = m0 + row;
  float gn[RG + 1], sf[RG + 1];
#pragma unroll
  for (int u = 0; u < RG; ++u) {
    const int k = t + u * WPR * 32;
    gn[u] = g.norm_gain && k < g.K ? g.norm_gain[k] : 0.f;
    sf[u] = g.norm_gain && g.norm_shift && k < g.K ? g.norm_shift[k] : 0.f;
  }
  const int mm = m0 + warp, orow = (mm / g.rows_in) * g.rows_out + g.row_off + mm % g.rows_in;
  const bool mine = warp < RM && col && mm < g.M;           // one output per thread of the first RM warps
  float* const o = g.out + (size_t)orow * g.ldo + n;
  float cst = 0.f, old = 0.f;
  if (mine && !DUAL) {
    if (g.epi == EPI_RESID) cst = g.gate ? g.gate[n] : 1.f;
    else if (g.bias) cst = g.bias[n];
  }
  pdl_wait();
  if (mine && !DUAL && g.epi == EPI_RESID) old = *o;
  // ---- the rows (RW / RM warps each), with the norm applied in place
  const float* a = g.A + (size_t)min(m, g.M - 1) * g.lda;
  float ss = 0.f;
  for (int k0 = t; k0 < g.K; k0 += RU * WPR * 32) {
    float x[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) x[u] = k0 + u * WPR * 32 < g.K ? a[k0 + u * WPR * 32] : 0.f;
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      if (k0 + u * WPR * 32 < g.K) As[row * g.K + k0 + u * WPR * 32] = x[u];
      ss = fmaf(x[u], x[u], ss);
    }
  }
  if (status_set(status)) return;
  if (g.norm_gain) {
    ss = warp_sum(ss);
    if (lane == 0) ssp[warp] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < WPR; ++w) tot += ssp[row * WPR + w];
    const float r = 1.0f / sqrtf(tot / (float)g.K + g.eps);
#pragma unroll
    for (int u = 0; u < RG; ++u) {
      const int k = t + u * WPR * 32;
      if (k < g.K) As[row * g.K + k] = fmaf(As[row * g.K + k] * r, gn[u], sf[u]);
    }
    for (int k = t + RG * WPR * 32; k < g.K; k += WPR * 32) {
      float v = As[row * g.K + k] * r * g.norm_gain[k];
      if (g.norm_shift) v += g.norm_shift[k];
      As[row * g.K + k] = v;
    }
  }
  __syncthreads();
  // ---- this warp's range of the contraction
  float acc[RM], acc2[DUAL ? RM : 1];
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    acc[r] = 0.f;
    if (DUAL) acc2[r] = 0.f;
  }
  for (int k0 = k_lo; k0 < k_hi; k0 += RK) {
    float c[RK], c2[DUAL ? RK : 1];
#pragma unroll
    for (int i = 0; i < RK; ++i) {
      c[i] = b[i];
      if (DUAL) c2[i] = b2[i];
    }
    if (k0 + RK < k_hi) fetch(k0 + RK);
#pragma unroll
    for (int i = 0; i < RK; i += 4) {
      if (k0 + i >= k_hi) break;                             // (ranges are multiples of four long unless K ends)
#pragma unroll
      for (int r = 0; r < RM; ++r) {
        float x[4];
        if (k0 + i + 4 <= g.K && !(g.K & 3)) {
          *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(As + r * g.K + k0 + i);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = k0 + i + e < g.K ? As[r * g.K + k0 + i + e] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[r] = fmaf(x[e], c[i + e], acc[r]);
          if (DUAL) acc2[r] = fmaf(x[e], c2[i + e], acc2[r]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    red[0][warp][r][lane] = acc[r];
    if (DUAL) red[DUAL ? 1 : 0][warp][r][lane] = acc2[r];
  }
  __syncthreads();
  // ---- one output per thread: the partial sums in range order, epilogue
  if (!mine) return;
  float v = 0.f, v2 = 0.f;
#pragma unroll
  for (int w = 0; w < RW; ++w) {
    v += red[0][w][warp][lane];
    if (DUAL) v2 += red[DUAL ? 1 : 0][w][warp][lane];
  }
  if (DUAL) *o = gelu_f(v, g.gelu_exact) * v2;
  else if (g.epi == EPI_RESID) *o = fmaf(cst, v, old);
  else if (g.epi == EPI_SWISH) *o = swish_precise(v + cst);
  else *o = v + cst;
}

// One (suffix row, query head) per block of eight warps.  Scores: a lane takes a key and its whole dot product (the key's
// head_dim values in 16-byte loads, all in flight); probabilities in shared memory; output: a lane takes channels, a warp
// every eighth key.  (One key per warp with a shuffle reduction per key walked 20 keys in 20 dependent round trips.)
constexpr int AW = 8;

template <typename KV> __device__ __forceinline__ float4 load4(const KV* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&u.x), b = *reinterpret_cast<const __nv_bfloat162*>(&u.y);
  return make_float4(__low2float(a), __high2float(a), __low2float(b), __high2float(b));
}

template <typename KV>
__global__ void __launch_bounds__(AW * 32) k_attention_row(const Request* rq, const int* status, const float* qkv, const float2* rope,
                                                           int layer, float* out, const Dims d, int max_keys) {
  extern __shared__ __align__(16) float sm[];
  float* const qs = sm;                       // [dh] rotated, scaled query
  float* const ps = sm + d.dh;                // [max_keys] scores, then probabilities
  float* const part = ps + max_keys;          // [AW][dh]
  __shared__ float wred[AW];
  pdl_launch_dependents();
  const int row = blockIdx.x, head = blockIdx.y, b = row / d.S, i = row - b * d.S, hk = head / (d.Hq / d.Hkv);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int half = d.dh >> 1;
  const Request r = *rq;
  pdl_wait();
  if (status_set(status)) return;
  const int p0 = r.cu_lens[b], P = r.cu_lens[b + 1] - p0;
  const float* qrow = qkv + (size_t)row * d.Nqkv + head * d.dh;
  const float scale = rsqrtf((float)d.dh);
  for (int t = tid; t < d.dh; t += AW * 32) {
    float v = qrow[t];
    if (rope) {
      const int j = t < half ? t : t - half;
      const float2 cs = rope[(size_t)(P + i) * half + j];
      const float other = qrow[t < half ? t + half : t - half];
      v = t < half ? v * cs.x - other * cs.y : v * cs.x + other * cs.y;
    }
    qs[t] = v * scale;
  }
  __syncthreads();
  const size_t kv_stride = (size_t)d.Hkv * d.dh;
  const KV* Kp = reinterpret_cast<const KV*>(r.prefix_kv) + ((size_t)(layer * 2) * r.kv_tokens + p0) * kv_stride + (size_t)hk * d.dh;
  const KV* Vp = Kp + (size_t)r.kv_tokens * kv_stride;
  const float* Ks = qkv + (size_t)(b * d.S) * d.Nqkv + d.Nq + hk * d.dh;
  const float* Vs = Ks + (size_t)d.Hkv * d.dh;
  const int nkeys = (d.block_causal && d.ns && i == 0) ? P + 1 : P + d.S;      // (the state token sees, of the suffix, itself)
  float mx = -INFINITY;
  for (int j = tid; j < nkeys; j += AW * 32) {
    float dot = 0.f;
    if (j < P) {
      const KV* k = Kp + (size_t)j * kv_stride;
#pragma unroll 8
      for (int c = 0; c < d.dh; c += 4) {
        const float4 x = load4<KV>(k + c), q = *reinterpret_cast<const float4*>(qs + c);
        dot = fmaf(x.x, q.x, fmaf(x.y, q.y, fmaf(x.z, q.z, fmaf(x.w, q.w, dot))));
      }
    } else {
      const float* k = Ks + (size_t)(j - P) * d.Nqkv;
      const float2* cs = rope + (size_t)j * half;             // (suffix key j - P sits at position j)
#pragma unroll 4
      for (int c = 0; c < half; ++c) {
        float lo = k[c], hi = k[c + half];
        if (rope) {
          const float2 w = cs[c];
          const float l = lo * w.x - hi * w.y;
          hi = hi * w.x + lo * w.y, lo = l;
        }
        dot = fmaf(lo, qs[c], fmaf(hi, qs[c + half], dot));
      }
    }
    ps[j] = dot;
    mx = fmaxf(mx, dot);
  }
  mx = warp_max(mx);
  if (lane == 0) wred[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < AW; ++w) mx = fmaxf(mx, wred[w]);
  __syncthreads();
  float sum = 0.f;
  for (int j = tid; j < nkeys; j += AW * 32) {
    const float p = __expf(ps[j] - mx);
    ps[j] = p;
    sum += p;
  }
  sum = warp_sum(sum);
  if (lane == 0) wred[warp] = sum;
  __syncthreads();
  sum = 0.f;
#pragma unroll
  for (int w = 0; w < AW; ++w) sum += wred[w];
  for (int c = lane; c < d.dh; c += 32) {
    float acc = 0.f;
    int j = warp;
#pragma unroll 8
    for (; j < min(P, nkeys); j += AW) acc = fmaf(ps[j], to_float<KV>(Vp[(size_t)j * kv_stride + c]), acc);
#pragma unroll 4
    for (; j < nkeys; j += AW) acc = fmaf(ps[j], Vs[(size_t)(j - P) * d.Nqkv + c], acc);
    part[warp * d.dh + c] = acc;
  }
  __syncthreads();
  const float inv = 1.0f / sum;
  for (int c = tid; c < d.dh; c += AW * 32) {
    float o = 0.f;
#pragma unroll
    for (int w = 0; w < AW; ++w) o += part[w * d.dh + c];
    out[(size_t)row * d.Nq + head * d.dh + c] = o * inv;
  }
}

}  // namespace

// Up to 512 rows (beyond, the tiled kernel's reuse of the weights wins) and rows that fit the shared memory of a block.
bool simt_rows_supported(int M, int K) { return M <= 512 && K <= 4096; }

cudaError_t launch_simt_rows(const int* status, const SimtGemm& g, cudaStream_t st) {
  // (few rows: four per block, so that the blocks cover the SMs; more rows: eight, half the weight reads)
  const int rm = g.M <= 64 || g.K > 2048 ? 4 : 8;
  const dim3 grid((g.N + 31) / 32, (g.M + rm - 1) / rm);
  const size_t smem = (size_t)rm * g.K * sizeof(float);
  auto k = g.epi == EPI_GEGLU ? (rm == 4 ? k_rows_f32<4, true> : k_rows_f32<8, true>) : (rm == 4 ? k_rows_f32<4, false> : k_rows_f32<8, false>);
  static PerDeviceOnce once;
  if (once.needed()) {
    for (auto f : {k_rows_f32<4, true>, k_rows_f32<8, true>, k_rows_f32<4, false>, k_rows_f32<8, false>}) {
      const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * 4096 * (int)sizeof(float));
      if (e != cudaSuccess) return e;
    }
    once.done();
  }
  return launch_pdl(k, grid, dim3(RW * 32), smem, st, status, g);
}

bool attention_row_supported(const Dims& d, int max_prefix) { return d.dh % 4 == 0 && d.dh <= 256 && max_prefix + d.S <= 8192; }

cudaError_t launch_attention_row(const Request* rq, const int* status, const float* qkv, const float2* rope, int layer, int kv_is_bf16,
                                 float* out, const Dims& d, int batch, int max_prefix, cudaStream_t st) {
  const int max_keys = (max_prefix + d.S + 3) & ~3;
  const size_t smem = (size_t)(d.dh + max_keys + AW * d.dh) * sizeof(float);
  return kv_is_bf16 ? launch_pdl(k_attention_row<__nv_bfloat16>, dim3(batch * d.S, d.Hq), dim3(AW * 32), smem, st, rq, status, qkv, rope, layer, out, d, max_keys)
                    : launch_pdl(k_attention_row<float>, dim3(batch * d.S, d.Hq), dim3(AW * 32), smem, st, rq, status, qkv, rope, layer, out, d, max_keys);
}

}  // namespace phyai
