// fp32 kernels for few token rows (the CUDA-core path: true fp32 FMA, no TF32): projections with the preceding RMSNorm
// folded in, attention of one (row, head) per block, the step boundary of one action row per block.  At these sizes nothing is
// throughput: what a launch costs is the hand-over, its trips to the L2 one after the other, and the fetch of its code.  So a block of
// a projection takes RM rows x 32 columns, sixteen warps share the contraction, the weights are requested before the dependency
// wait (they are constants), the partial sums meet in shared memory in a fixed order, and loops are rolled: 3.7 us per
// launch in the captured loop of the tiny expert, hand-over to the next one included.
#include <algorithm>

#include "kernels.h"

namespace phyai {
namespace {

constexpr int RW = 16;            // warps of a block: ranges of the contraction
constexpr int RK = 16;            // weight rows a warp has in flight

// The form with the least code, because code is what bounds it: between two layers the instruction caches lose it, and a first pass
// costs about 11 clocks per instruction.  Nothing is unrolled: the weight tile [K][32] (gate / up: two) goes to shared memory with
// 16-byte asynchronous copies, ahead of the dependency wait, and rolled loops walk it.  RM = 4 rows for up to 48 token rows (more
// blocks), else 8 (half the weight reads).  A call of the tiny expert, unrolled kernel below -> this one (with an attention that gives
// a key eight lanes): 17 rows 256 -> 208 us, 68: 376 -> 269 (four rows to a block 282), 136: 524 -> 375 (444), 200: 705 -> 508 (597).
template <int RM, bool DUAL>
__global__ void __launch_bounds__(RW * 32) k_rows_small(const int* status, const SimtGemm g) {
  constexpr int WPR = RW / RM, TPR = WPR * 32;
  extern __shared__ __align__(16) float sm[];
  __shared__ float red[DUAL ? 2 : 1][RW][RM][32];
  __shared__ float ssp[RW];
  float* const As = sm;                                      // [RM][K]
  float* const Ws = sm + RM * g.K;                           // [K][32], then the second matrix
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = blockIdx.x * 32, n = n0 + lane, m0 = blockIdx.y * RM, K = g.K;
  pdl_launch_dependents();
  {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Ws);
    const int c4 = (tid & 7) * 4;
#pragma unroll 1
    for (int k = tid >> 3; k < K; k += RW * 4) {
      const size_t src = (size_t)k * g.N + n0 + c4;
      const uint32_t sz = n0 + c4 < g.N ? 16u : 0u;          // (N is a multiple of four)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)(k * 32 + c4) * 4u), "l"(g.B + (sz ? src : 0)), "r"(sz) : "memory");
      if (DUAL) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + (uint32_t)((K + k) * 32 + c4) * 4u), "l"(g.B2 + (sz ? src : 0)), "r"(sz) : "memory");
    }
  }
  // constants of this thread: the norm's (its first four elements of the row), the epilogue's
  const int row = warp / WPR, t = tid & (TPR - 1), mm = m0 + warp;
  const bool mine = warp < RM && n < g.N && mm < g.M;        // one output per thread of the first RM warps
  const float4* const gain4 = reinterpret_cast<const float4*>(g.norm_gain);
  const float4* const shift4 = reinterpret_cast<const float4*>(g.norm_shift);
  float4 gn = make_float4(0.f, 0.f, 0.f, 0.f), sf = gn;
  if (gain4 && t < K / 4) {
    gn = __ldg(gain4 + t);
    if (shift4) sf = __ldg(shift4 + t);
  }
  float cst = g.epi == EPI_RESID ? 1.f : 0.f, old = 0.f;
  float* o = g.out + n;
  if (mine) {
    o += (size_t)((mm / g.rows_in) * g.rows_out + g.row_off + mm % g.rows_in) * g.ldo;
    const float* cp = g.epi == EPI_RESID ? g.gate : g.bias;
    if (!DUAL && cp) cst = cp[n];
  }
  pdl_wait();
  if (mine && !DUAL && g.epi == EPI_RESID) old = *o;
  // ---- the rows (WPR warps each), with the norm applied in place
  const float4* a = reinterpret_cast<const float4*>(g.A + (size_t)min(m0 + row, g.M - 1) * g.lda);
  float4* const as = reinterpret_cast<float4*>(As + row * K);
  float ss = 0.f;
#pragma unroll 2
  for (int k = t; k < K / 4; k += TPR) {
    const float4 x = a[k];
    as[k] = x;
    ss = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, ss))));
  }
  if (status_set(status)) return;
  if (gain4) {
    ss = warp_sum(ss);
    if (lane == 0) ssp[warp] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < WPR; ++w) tot += ssp[row * WPR + w];
    const float r = 1.0f / sqrtf(tot / (float)K + g.eps);
#pragma unroll 1
    for (int k = t; k < K / 4; k += TPR) {
      if (k != t) gn = __ldg(gain4 + k), sf = shift4 ? __ldg(shift4 + k) : sf;
      const float4 x = as[k];
      as[k] = make_float4(fmaf(x.x * r, gn.x, sf.x), fmaf(x.y * r, gn.y, sf.y), fmaf(x.z * r, gn.z, sf.z), fmaf(x.w * r, gn.w, sf.w));
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // ---- this warp's range of the contraction (a multiple of four long)
  const int kper = ((K + RW - 1) / RW + 3) & ~3, k_hi = min(K, (warp + 1) * kper);
  float acc[RM] = {}, acc2[DUAL ? RM : 1] = {};
#pragma unroll 1
  for (int k = warp * kper; k < k_hi; k += 4) {
    const float* w = Ws + k * 32 + lane;
    float w1[4], w2[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w1[e] = w[e * 32], w2[e] = DUAL ? w[(K + e) * 32] : 0.f;
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      const float4 x = *reinterpret_cast<const float4*>(As + r * K + k);
      acc[r] = fmaf(x.x, w1[0], acc[r]), acc[r] = fmaf(x.y, w1[1], acc[r]), acc[r] = fmaf(x.z, w1[2], acc[r]), acc[r] = fmaf(x.w, w1[3], acc[r]);
      if (DUAL) acc2[r] = fmaf(x.x, w2[0], acc2[r]), acc2[r] = fmaf(x.y, w2[1], acc2[r]), acc2[r] = fmaf(x.z, w2[2], acc2[r]), acc2[r] = fmaf(x.w, w2[3], acc2[r]);
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
#pragma unroll 4
  for (int w = 0; w < RW; ++w) {
    v += red[0][w][warp][lane];
    if (DUAL) v2 += red[DUAL ? 1 : 0][w][warp][lane];
  }
  if (DUAL) *o = gelu_f(v, g.gelu_exact) * v2;
  else if (g.epi == EPI_RESID) *o = fmaf(cst, v, old);
  else if (g.epi == EPI_SWISH) *o = swish_precise(v + cst);
  else *o = v + cst;
}
size_t rows_small_smem(const SimtGemm& g, int rm) { return ((size_t)rm + 32 * (g.epi == EPI_GEGLU ? 2 : 1)) * g.K * sizeof(float); }
bool rows_small_ok(const SimtGemm& g) {
  const auto a16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  return g.K % 4 == 0 && g.N % 4 == 0 && g.lda % 4 == 0 && rows_small_smem(g, 8) <= 190 * 1024 && a16(g.A) && a16(g.B) && a16(g.B2) &&
         a16(g.norm_gain) && a16(g.norm_shift);
}

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

// One (suffix row, query head) per block of sixteen warps.  Scores: eight lanes to a key, two keys of a lane in flight; output: a
// thread takes four channels of every (4 x 512 / head_dim)-th key, four of them in flight.  The loops are rolled and batch their loads
// (short code, and no remainder loop that walks its keys in dependent trips to the L2: eight warps, a key per lane and a warp per
// eighth key took 12 us by itself, this 7; calls of the tiny expert 204 -> 188 us at 17 rows, 508 -> 471 at 200).
constexpr int AW = 16;

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
  float* const part = ps + max_keys;          // [key sets][dh + 4]: partial outputs, their sum of probabilities
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
  const int sub = tid & 7;
  float mx = -INFINITY;
#pragma unroll 1
  for (int j0 = tid >> 3; j0 < ((nkeys + 3) & ~3); j0 += AW * 8) {      // (a warp's four keys together: the shuffles are full)
    float dot[2] = {0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = j0 + u * AW * 4;
      if (j < P && j < nkeys) {
        const KV* k = Kp + (size_t)j * kv_stride;
#pragma unroll 2
        for (int c = sub * 4; c < d.dh; c += 32) {
          const float4 x = load4<KV>(k + c), q = *reinterpret_cast<const float4*>(qs + c);
          dot[u] = fmaf(x.x, q.x, fmaf(x.y, q.y, fmaf(x.z, q.z, fmaf(x.w, q.w, dot[u]))));
        }
      } else if (j < nkeys) {
        const float* k = Ks + (size_t)(j - P) * d.Nqkv;
        const float2* cs = rope + (size_t)j * half;             // (suffix key j - P sits at position j)
#pragma unroll 4
        for (int c = sub; c < half; c += 8) {
          float lo = k[c], hi = k[c + half];
          if (rope) {
            const float2 w = cs[c];
            const float l = lo * w.x - hi * w.y;
            hi = hi * w.x + lo * w.y, lo = l;
          }
          dot[u] = fmaf(lo, qs[c], fmaf(hi, qs[c + half], dot[u]));
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = j0 + u * AW * 4;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
      if (j < nkeys) {
        if (sub == 0) ps[j] = dot[u];
        mx = fmaxf(mx, dot[u]);
      }
    }
  }
  mx = warp_max(mx);
  if (lane == 0) wred[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < AW; ++w) mx = fmaxf(mx, wred[w]);
  // groups of dh / 4 threads take every n_sets-th key; each forms the probabilities of its own keys, their sum joins the outputs
  const int n_cg = d.dh >> 2, n_sets = min(128, AW * 32 / n_cg), set = tid / n_cg, c4 = (tid - set * n_cg) * 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float sum = 0.f;
  if (set < n_sets) {
#pragma unroll 1
    for (int j0 = set; j0 < nkeys; j0 += 4 * n_sets) {
      float4 v[4];
      float pj[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u * n_sets, jc = min(j, nkeys - 1);
        if (jc < P) v[u] = load4<KV>(Vp + (size_t)jc * kv_stride + c4);
        else v[u] = load4<float>(Vs + (size_t)(jc - P) * d.Nqkv + c4);
        pj[u] = j < nkeys ? __expf(ps[jc] - mx) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc.x = fmaf(pj[u], v[u].x, acc.x), acc.y = fmaf(pj[u], v[u].y, acc.y), acc.z = fmaf(pj[u], v[u].z, acc.z), acc.w = fmaf(pj[u], v[u].w, acc.w);
        sum += pj[u];
      }
    }
    *reinterpret_cast<float4*>(part + set * (d.dh + 4) + c4) = acc;
    if (c4 == 0) part[set * (d.dh + 4) + d.dh] = sum;
  }
  __syncthreads();
  for (int c = tid; c < d.dh; c += AW * 32) {
    float o = 0.f, tot = 0.f;
#pragma unroll 4
    for (int w = 0; w < n_sets; ++w) o += part[w * (d.dh + 4) + c], tot += part[w * (d.dh + 4) + d.dh];
    out[(size_t)row * d.Nq + head * d.dh + c] = o / tot;
  }
}

// Step boundary of one action row per block: velocity head and Euler update of the step that ends (gain != null), embedding of the one
// that begins (Wc != null): pi0 u = swish(x Wc + bias), pi0.5 h = x Wc + bias; the request's state token with its first row.  Rolled
// loops, as above; the constants are asked for ahead of the dependency wait where there is one value per thread.  (Against a head and
// an embedding kernel: 208 -> 204 us per call of the tiny expert at 17 rows, 234 -> 221 at 34.)
constexpr int BW = 16;
__global__ void __launch_bounds__(BW * 32) k_step_row(const Request* rq, const int* status, const StepRow p) {
  extern __shared__ __align__(16) float sm[];
  float* const nrm = sm;                        // [D] normalised row
  float* const xs = nrm + p.D;                  // [A] actions
  __shared__ float red[BW][32];
  __shared__ float wred[BW];
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x, D = p.D, A = p.A;
  const int ar = blockIdx.x, b = ar / p.H, i = ar - b * p.H;
  float* const h = p.h + (size_t)(b * p.S + p.ns + i) * D;
  float* const x = rq->x + (size_t)ar * A;      // (the request block is written before the captured loop starts)
  const float g0 = p.gain && tid < D ? __ldg(p.gain + tid) : 0.f, s0 = p.gain && p.shift && tid < D ? __ldg(p.shift + tid) : 0.f;
  const float bo = p.gain && tid < A ? __ldg(p.bout + tid) : 0.f;
  pdl_wait();
  if (status_set(status)) return;
  float xv = tid < A ? x[tid] : 0.f;            // (A <= 256)
  if (p.gain) {
    float ss = 0.f;
    for (int e = tid; e < D; e += BW * 32) {
      const float v = h[e];
      nrm[e] = v;
      ss = fmaf(v, v, ss);
    }
    ss = warp_sum(ss);
    if (lane == 0) wred[warp] = ss;
    __syncthreads();
    ss = 0.f;
#pragma unroll
    for (int w = 0; w < BW; ++w) ss += wred[w];
    const float rs = 1.0f / sqrtf(ss / (float)D + p.eps);
    for (int e = tid; e < D; e += BW * 32) {
      const float gn = e == tid ? g0 : __ldg(p.gain + e), sf = e == tid ? s0 : (p.shift ? __ldg(p.shift + e) : 0.f);
      nrm[e] = fmaf(nrm[e] * rs, gn, sf);
    }
    __syncthreads();
    const int dper = (D + BW - 1) / BW;
    for (int a0 = 0; a0 < A; a0 += 32) {
      const int a = a0 + lane;
      float acc = 0.f;
#pragma unroll 8
      for (int e = warp * dper; e < min(D, (warp + 1) * dper); ++e) acc = fmaf(nrm[e], a < A ? __ldg(p.Wout + (size_t)e * A + a) : 0.f, acc);
      red[warp][lane] = acc;
      __syncthreads();
      if (tid >= a0 && tid < a0 + 32 && tid < A) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < BW; ++w) v += red[w][lane];
        xv += p.dt * (v + bo);
        x[tid] = xv;
      }
      __syncthreads();
    }
  }
  if (!p.Wc) return;
  if (tid < A) xs[tid] = xv;
  __syncthreads();
  for (int e = tid; e < D; e += BW * 32) {
    float acc = 0.f;
#pragma unroll 8
    for (int a = 0; a < A; ++a) acc = fmaf(xs[a], __ldg(p.Wc + (size_t)a * D + e), acc);
    const float v = acc + __ldg(p.bias + e);
    if (p.u) p.u[(size_t)ar * D + e] = swish_precise(v);
    else h[e] = v;
    if (p.ns && i == 0) p.h[(size_t)(b * p.S) * D + e] = p.state_tok[(size_t)b * D + e];
  }
}

}  // namespace

// Up to 512 rows (beyond, the tiled kernel's reuse of the weights wins) and rows that fit the shared memory of a block.
bool simt_rows_supported(int M, int K) { return M <= 512 && K <= 4096; }

cudaError_t launch_simt_rows(const int* status, const SimtGemm& g, cudaStream_t st) {
  if (rows_small_ok(g)) {
    static PerDeviceOnce small;
    if (small.needed()) {
      for (auto f : {k_rows_small<4, true>, k_rows_small<4, false>, k_rows_small<8, true>, k_rows_small<8, false>}) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 190 * 1024);
        if (e != cudaSuccess) return e;
      }
      small.done();
    }
    const int rm = g.M <= 48 ? 4 : 8;
    auto k = g.epi == EPI_GEGLU ? (rm == 4 ? k_rows_small<4, true> : k_rows_small<8, true>) : (rm == 4 ? k_rows_small<4, false> : k_rows_small<8, false>);
    return launch_pdl(k, dim3((g.N + 31) / 32, (g.M + rm - 1) / rm), dim3(RW * 32), rows_small_smem(g, rm), st, status, g);
  }
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

// (one row per block: few rows; more of them share their reads of the weights in the kernels of their own)
bool step_row_supported(const Dims& d, int batch) { return batch * d.H <= 256 && d.A <= 256 && d.D + d.A <= 11 * 1024; }

cudaError_t launch_step_row(const Request* rq, const int* status, const StepRow& p, int rows, cudaStream_t st) {
  return launch_pdl(k_step_row, dim3(rows), dim3(BW * 32), (size_t)(p.D + p.A) * sizeof(float), st, rq, status, p);
}

bool attention_row_supported(const Dims& d, int max_prefix) { return d.dh % 4 == 0 && d.dh <= 256 && max_prefix + d.S <= 8192; }

cudaError_t launch_attention_row(const Request* rq, const int* status, const float* qkv, const float2* rope, int layer, int kv_is_bf16,
                                 float* out, const Dims& d, int batch, int max_prefix, cudaStream_t st) {
  const int max_keys = (max_prefix + d.S + 3) & ~3;
  const int sets = std::min(128, AW * 32 / (d.dh / 4));
  const size_t smem = (size_t)(d.dh + max_keys + sets * (d.dh + 4)) * sizeof(float);
  return kv_is_bf16 ? launch_pdl(k_attention_row<__nv_bfloat16>, dim3(batch * d.S, d.Hq), dim3(AW * 32), smem, st, rq, status, qkv, rope, layer, out, d, max_keys)
                    : launch_pdl(k_attention_row<float>, dim3(batch * d.S, d.Hq), dim3(AW * 32), smem, st, rq, status, qkv, rope, layer, out, d, max_keys);
}

}  // namespace phyai
