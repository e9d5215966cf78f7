// Projections of calls with a single 64-token tile on CTA pairs (tcgen05 cta_group::2): the chain of a layer without a
// cluster reduce where the contraction fits one pair, and with a four-way instead of an eight-way one where it does not.
//
// What bounds them is the length of a dependent chain, per kernel: activations from L2 (about 0.8 us of latency plus their
// bytes at 62 bytes per clock and SM), the reduce over a cluster (1.5 - 1.9 us in gemm_b1.cu: staging, bulk copies, the
// slowest peer), the epilogue.  A CTA of gemm_b1.cu holds 128 channels of a k-range and all 64 tokens.  A CTA of a pair
// holds 64 channels of a range twice as long and half of the tokens (the tensor cores read the other half from the peer):
// the same bytes before and after the dependency, but one k-range for K = 1024 (16 chunks of 8 KB of weights and 4 KB of
// activations, all resident), so QKV and gate / up have no reduce at all, and half as many and half as large partials for
// the others (down: 4 ranges of 16 chunks).
//
// Roles: warp 16 issues the copies (weights ahead of the dependency wait, activations after it), warp 17 the MMAs (leader
// CTA), warps 0 - 15 decode weight codes, hold an item's constants in registers (four channels and their rotary or gate / up
// partners of one token: every item has its own thread) and run the epilogue through a staging tile [token][64 channels].
// Norms are folded in as in gemm_b1.cu, with one partial sum of squares per 64 channels.  Waits are bounded; after a
// give-up copies, MMAs, commits and barriers go on and only the stores are skipped.
//
// Measured inside the captured pi0 loop of one request, dependency to last store, gemm_b1.cu -> this: QKV 4.0 -> 2.8 us,
// gate / up 3.9 -> 2.8, down 4.5 -> 3.9, O 3.6 -> 3.6; the loop of ten steps 5.67 -> 5.11 ms.
#include "decode.cuh"
#include "kernels.h"
#include "ptx.cuh"
#include "tc.cuh"
#include "tc_pair.cuh"

namespace phyai {
namespace {

constexpr int BP_EPI = 512, BP_THREADS = BP_EPI + 64;     // 16 epilogue warps, copies, MMAs
constexpr int BP_MAXK = 16;                               // k-chunks of a CTA, all resident
constexpr int BP_A = 64 * 128;                            // 64 weight rows x 64 k
constexpr int BP_GROUP = 4, BP_NG = BP_MAXK / BP_GROUP;   // chunks that signal one barrier (a wait per chunk would set the pace)
constexpr int BP_MAXKP = 4;                               // k-ranges (pairs of a cluster)
constexpr size_t BP_SMEM_MAX = 227 * 1024 - 1024;

__device__ __forceinline__ float4 lds4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint2 pack4(float4 v) { return make_uint2(pack2(v.x, v.y), pack2(v.z, v.w)); }
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
// accumulator -> projection output: weight scale, the folded norm's per-token factor, the folded shift row
__device__ __forceinline__ float4 fin4(float4 x, float4 s, float r, float4 h) {
  return make_float4(fmaf(x.x * s.x, r, h.x), fmaf(x.y * s.y, r, h.y), fmaf(x.z * s.z, r, h.z), fmaf(x.w * s.w, r, h.w));
}

template <int EPI, int WB>
__global__ void __launch_bounds__(BP_THREADS, 1)
    k_gemm_b1_pair(int* status, const B1Gemm g, const __grid_constant__ CUtensorMap tmw, const __grid_constant__ CUtensorMap tmx) {
  constexpr int CODE_ROW = WB == 4 ? 32 : 64;               // bytes of a row of codes (64 weights)
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[BP_NG];         // leader: operands of both CTAs (WB: activations)
  __shared__ __align__(8) uint64_t bar_codes[BP_MAXK];      // WB: a chunk's codes have landed here
  __shared__ __align__(8) uint64_t bar_dec;                 // WB, leader: a decoding warp of either CTA is done
  __shared__ __align__(8) uint64_t bar_accum, bar_recv;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31, tid = threadIdx.x;
  const int rank = (int)blockIdx.x, r = rank & 1, kp = rank >> 1, KP = (int)(gridDim.x >> 1), tile = blockIdx.y;
  const int KC = g.K >> 6, kc_begin = (KC * kp) / KP, nk = (KC * (kp + 1)) / KP - kc_begin;
  const int M = g.M, HN = ((M + 15) >> 4) << 3;             // tokens of a CTA's activation tile: half of M rounded up to 16
  const uint32_t chunk = (uint32_t)(BP_A + HN * 128);
  const int tok_lo = (M * kp) / KP, ntok = (M * (kp + 1)) / KP - tok_lo;    // tokens this CTA finishes

  pdl_launch_dependents();
  unsigned long long* tr = nullptr;
  if (g.trace && tid == 0) {
    if (g.trace_all) tr = g.trace + (size_t)(blockIdx.y * gridDim.x + blockIdx.x) * 16;
    else if (blockIdx.x == 0 && blockIdx.y == 0) tr = g.trace;
  }
  trace_stamp(tr, 0);
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t stage = tiles;                             // [tokens][64] fp32, over the consumed operands
  const uint32_t recv = tiles + max((uint32_t)g.nk_max * chunk, 2u * HN * 256u);
  const uint32_t slot = (uint32_t)((M + KP - 1) / KP) * 256u;              // one peer's partial of my tokens

  if (tid == BP_EPI) prefetch_tmap(&tmw), prefetch_tmap(&tmx);
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < BP_NG; ++i) mbar_init(smem_u32(&bar_full[i]), 1);
    for (int i = 0; i < BP_MAXK; ++i) mbar_init(smem_u32(&bar_codes[i]), 1);
    mbar_init(smem_u32(&bar_dec), 2 * nk);                  // (one warp per chunk decodes; both CTAs of a pair have nk)
    mbar_init(smem_u32(&bar_accum), 1);
    mbar_init(smem_u32(&bar_recv), 1);
    if (KP > 1 && ntok > 0) mbar_expect_tx(smem_u32(&bar_recv), (uint32_t)(KP - 1) * (uint32_t)ntok * 256u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 17) {
    tmem_alloc2(smem_u32(&tmem_slot), 32);
    tc_fence_before();
  }
  pair_sync();                                              // every barrier of the cluster exists before anything signals it
  trace_stamp(tr, 1);
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&tmem_slot), 0);
  const WaitCtx wc{status, &abort_flag, g.wait_limit};

  if (warp == 16) {
    // ---------------- copies -------------------------------------------------------------------------------------
    if (lane == 0) {
      // this CTA's 64 rows of the 128-row block: 32 and their rotary / gate-up partners 64 further on, or (residual) a half
      const int lo = EPI == B1_RESID ? 64 * r : 32 * r, hi = EPI == B1_RESID ? 64 * r + 32 : 64 + 32 * r;
      for (int s = 0; s < nk; ++s) {
        const uint32_t dst = tiles + (uint32_t)s * chunk, full = smem_u32(&bar_full[s / BP_GROUP]);
        if (r == 0 && s % BP_GROUP == 0) mbar_expect_tx(full, 2u * (uint32_t)min(BP_GROUP, nk - s) * (WB ? (uint32_t)HN * 128u : chunk));
        const size_t blk = (size_t)tile * KC + kc_begin + s;
        if constexpr (WB != 0) {
          const uint8_t* src = g.W8 + blk * 128 * CODE_ROW;
          const uint32_t cd = dst + BP_A - 64 * CODE_ROW, bar = smem_u32(&bar_codes[s]);
          mbar_expect_tx(bar, 64 * CODE_ROW);
          bulk_g2s(cd, src + lo * CODE_ROW, 32 * CODE_ROW, bar);
          bulk_g2s(cd + 32 * CODE_ROW, src + hi * CODE_ROW, 32 * CODE_ROW, bar);
        } else {
          tma2d(dst, &tmw, (int)blk * 128 + lo, full & LEADER_MASK);
          tma2d(dst + 32 * 128, &tmw, (int)blk * 128 + hi, full & LEADER_MASK);
        }
      }
      pdl_wait();
      for (int s = 0; s < nk; ++s)
        tma2d(tiles + (uint32_t)s * chunk + BP_A, &tmx, (kc_begin + s) * 64 + r * HN, smem_u32(&bar_full[s / BP_GROUP]) & LEADER_MASK);
    }
    __syncwarp();
    cluster_arrive_relaxed();
  } else if (warp == 17) {
    // ---------------- MMAs: whole warp in the loop, one elected lane issues -----------------------------------------
    if (r == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(HN >> 2) << 17) | (128u >> 4) << 24;
      bool dead = false;
      if constexpr (WB != 0) dead = mbar_wait_drain(smem_u32(&bar_dec), 0u, wc) < 0;
      for (int s = 0; s < nk && !dead; ++s) {
        if (s % BP_GROUP == 0) {
          if (mbar_wait_drain(smem_u32(&bar_full[s / BP_GROUP]), 0u, wc) < 0) break;
          tc_fence_after();
        }
        const uint32_t a0 = tiles + (uint32_t)s * chunk;
        const uint64_t da = make_desc(a0), db = make_desc(a0 + BP_A);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (elect_one()) umma2_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (s > 0 || k > 0) ? 1u : 0u);
        __syncwarp();
      }
      if (elect_one()) umma2_commit(smem_u32(&bar_accum), 3u << (rank & ~1));
      __syncwarp();
    }
    cluster_arrive_relaxed();
  } else {
    // ---------------- epilogue warps ---------------------------------------------------------------------------------
    // an item: four channels (QKV, gate / up: and their partners) of one token; item i belongs to thread i
    constexpr int IT = EPI == B1_RESID ? 16 : 8;            // items per token
    const int tl = tid / IT, c4 = tid % IT, tok = tok_lo + tl;
    const bool mine = tl < ntok;
    const int j0 = EPI == B1_RESID ? 64 * r + 4 * c4 : 32 * r + 4 * c4, n0 = tile * 128;      // first channel, within the block
    const float4 one = make_float4(1.f, 1.f, 1.f, 1.f), zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 s0 = one, s1 = one, h0 = zero, h1 = zero;        // scales and folded shifts; RESID: scale, gain_next in s1
    if (EPI == B1_GEGLU) {
      if (g.wscale) s0 = ld4(g.wscale + tile * 64 + j0);
      if (g.wscale2) s1 = ld4(g.wscale2 + tile * 64 + j0);
    } else if (g.wscale) {
      s0 = ld4(g.wscale + n0 + j0);
      if (EPI == B1_QKV) s1 = ld4(g.wscale + n0 + 64 + j0);
    }
    if (EPI != B1_RESID && g.shift_row) h0 = ld4(g.shift_row + n0 + j0), h1 = ld4(g.shift_row + n0 + 64 + j0);
    if (EPI == B1_RESID) {
      if (g.gate) {
        const float4 t = ld4(g.gate + n0 + j0);
        s0 = make_float4(s0.x * t.x, s0.y * t.y, s0.z * t.z, s0.w * t.w);
      }
      if (g.gain_next) s1 = ld4(g.gain_next + n0 + j0);
    }
    // QKV: where the token sits (the request block is written before the captured loop starts) and its rotary factors
    const int Nq = g.Hq * g.dh, Nk = g.Hkv * g.dh;
    const bool rot_tile = EPI == B1_QKV && n0 < Nq + Nk, isq = n0 < Nq;
    int b = 0, row = 0;
    float4 cs0 = make_float4(1.f, 0.f, 1.f, 0.f), cs1 = cs0;   // (cos, sin) of channels j0, j0 + 1 and j0 + 2, j0 + 3
    if (EPI == B1_QKV && mine) {
      b = tok / g.S, row = tok - b * g.S;
      if (rot_tile && g.rope) {
        const int* cu = g.rq->cu_lens;
        const int pos = cu[b + 1] - cu[b] + g.koff + row, t64 = ((isq ? n0 : n0 - Nq) % g.dh) >> 7;
        const float* rp = reinterpret_cast<const float*>(g.rope + (size_t)pos * (g.dh >> 1) + t64 * 64 + j0);
        cs0 = ld4(rp), cs1 = ld4(rp + 4);
      }
    }
    if constexpr (WB != 0) {
      // a warp decodes a chunk; its generic writes become visible to the tensor core's reads before the leader is told
      if (warp < nk) {
        mbar_wait_drain(smem_u32(&bar_codes[warp]), 0u, wc);
        const uint32_t a0 = tiles + (uint32_t)warp * chunk;
        decode_rows64<WB>(a0 + BP_A - 64 * CODE_ROW, a0, 0, lane, [] { __syncwarp(); });
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          uint32_t bar;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(smem_u32(&bar_dec)), "r"(rank & ~1));
          asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
        }
      }
      trace_stamp(tr, 10);
    }
    pdl_wait();
    trace_stamp(tr, 2);
    const bool suppress = status_set(status);
    float rstd = 1.0f;
    float4 old = zero;
    bool state_row = false;
    if (EPI != B1_RESID) {
      if (g.ss_part) {                                      // the eight threads of a token add the partial sums
        float ss = 0.f;
        if (mine)
          for (int i = c4; i < g.ss_n; i += 8) ss += g.ss_part[i * 64 + tok];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        rstd = 1.0f / sqrtf(ss * g.inv_D + g.eps);
      }
    } else if (mine) {
      // what the projection is added to: the residual stream, or (MLP second layer) the bias / the state token's embedding
      const float* src = g.h + (size_t)tok * g.ldh + n0 + j0;
      if (g.bias) {
        const int rb = tok / g.S;
        state_row = tok - rb * g.S < g.ns;
        src = state_row ? g.state_tok + (size_t)rb * g.N + n0 + j0 : g.bias + n0 + j0;
      }
      old = *reinterpret_cast<const float4*>(src);
    }
    // ---- accumulator -> staging: rows of this CTA in lanes 0 - 63 (tokens 0 .. HN - 1) and 64 - 127 (HN .. 2 HN - 1)
    int ok_r = 0;
    if (lane == 0) ok_r = mbar_wait_drain(smem_u32(&bar_accum), 0u, wc);
    ok_r = __shfl_sync(0xffffffffu, ok_r, 0);
    tc_fence_after();
    trace_stamp(tr, 3);
    {
      const int q = warp & 3, c0 = (warp >> 2) * 8;
      if (c0 < HN && ok_r >= 0) {
        float v[8];
        tmem_ld8(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
        const uint32_t dst = stage + (uint32_t)((q >> 1) * HN + c0) * 256u + (uint32_t)((q & 1) * 32 + lane) * 4u;
#pragma unroll
        for (int j = 0; j < 8; ++j) asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + (uint32_t)j * 256u), "f"(v[j]) : "memory");
      }
    }
    tc_fence_before();
    if (KP > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("bar.sync 1, %0;" ::"n"(BP_EPI) : "memory");
    if (KP > 1) {
      // every peer of the same channels gets its tokens of this partial; the ranges are then added in order
      if (lane == 0 && warp < KP && warp != kp) {
        const int lo = (M * warp) / KP, n = (M * (warp + 1)) / KP - lo;
        if (n > 0) {
          uint32_t dst, bar;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(recv + (uint32_t)kp * slot), "r"(2 * warp + r));
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(smem_u32(&bar_recv)), "r"(2 * warp + r));
          asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                       "r"(stage + (uint32_t)lo * 256u), "r"((uint32_t)n * 256u), "r"(bar)
                       : "memory");
        }
      }
      if (ntok > 0) {
        int rr = 0;
        if (lane == 0) rr = mbar_wait_drain(smem_u32(&bar_recv), 0u, wc);
        rr = __shfl_sync(0xffffffffu, rr, 0);
        ok_r = min(ok_r, rr);
      }
    }
    // what the peers sent has landed; this CTA leaves once they say the same
    cluster_arrive_relaxed();
    trace_stamp(tr, 4);
    const bool store = mine && !suppress && ok_r > 0 && !*reinterpret_cast<volatile int*>(&abort_flag);
    if constexpr (EPI == B1_RESID) {
      float4 a = zero;
      if (mine && !state_row)
        for (int c = 0; c < KP; ++c) {
          const float4 v = lds4((c == kp ? stage + (uint32_t)tok * 256u : recv + (uint32_t)c * slot + (uint32_t)tl * 256u) + (uint32_t)c4 * 16u);
          a.x += v.x, a.y += v.y, a.z += v.z, a.w += v.w;
        }
      const float4 hv = make_float4(fmaf(a.x, s0.x, old.x), fmaf(a.y, s0.y, old.y), fmaf(a.z, s0.z, old.z), fmaf(a.w, s0.w, old.w));
      float ss = hv.x * hv.x + hv.y * hv.y + hv.z * hv.z + hv.w * hv.w;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (store) {
        *reinterpret_cast<float4*>(g.h + (size_t)tok * g.ldh + n0 + j0) = hv;
        if (g.xn_out) {
          *reinterpret_cast<uint2*>(g.xn_out + tiled_index(tok, n0 + j0, 64)) = pack4(make_float4(hv.x * s1.x, hv.y * s1.y, hv.z * s1.z, hv.w * s1.w));
          if (c4 == 0) g.ss_out[(tile * 2 + r) * 64 + tok] = ss;
        }
      }
    } else if (store) {
      const uint32_t sp = stage + (uint32_t)tok * 256u + (uint32_t)c4 * 16u;
      float4 lo = fin4(lds4(sp), s0, rstd, h0), hi = fin4(lds4(sp + 128), s1, rstd, h1);
      if constexpr (EPI == B1_GEGLU) {
        // one 64-wide k-chunk (`tile`) of the down projection's activation tile, in halves of its swizzled 16-byte groups
        float m[4] = {lo.x, lo.y, lo.z, lo.w};
        const float up[4] = {hi.x, hi.y, hi.z, hi.w};
        gelu_mul(m, up, g.gelu_exact);
        *reinterpret_cast<uint2*>(g.out_tiled + ((size_t)tile * 64 + tok) * 64 + (((j0 >> 3) ^ (tok & 7)) << 3) + (j0 & 7)) = make_uint2(pack2(m[0], m[1]), pack2(m[2], m[3]));
      } else if (rot_tile) {
        const int nn = isq ? n0 : n0 - Nq, head = nn / g.dh, t64 = (nn - head * g.dh) >> 7, half = g.dh >> 1;
        const float osc = isq ? rsqrtf((float)g.dh) : 1.0f;
        const float4 l = lo, h = hi;
        lo = make_float4(l.x * cs0.x - h.x * cs0.y, l.y * cs0.z - h.y * cs0.w, l.z * cs1.x - h.z * cs1.y, l.w * cs1.z - h.w * cs1.w);
        hi = make_float4(h.x * cs0.x + l.x * cs0.y, h.y * cs0.z + l.y * cs0.w, h.z * cs1.x + l.z * cs1.y, h.w * cs1.z + l.w * cs1.w);
        const uint2 vlo = pack4(make_float4(lo.x * osc, lo.y * osc, lo.z * osc, lo.w * osc));
        const uint2 vhi = pack4(make_float4(hi.x * osc, hi.y * osc, hi.z * osc, hi.w * osc));
        const int c_lo = t64 * 64 + j0, c_hi = c_lo + half;
        if (isq && g.q_tiles) {
          // the attention kernel's operand tiles (see gemm_b1.cu)
          const int rw = (head & 1) * 64 + row;
          __nv_bfloat16* tb = g.q_tiles + (size_t)(b * (g.Hq >> 1) + (head >> 1)) * (size_t)(128 * g.dh);
          *reinterpret_cast<uint2*>(tb + (size_t)(c_lo >> 6) * 8192 + rw * 64 + ((((c_lo & 63) >> 3) ^ (rw & 7)) << 3) + (c_lo & 7)) = vlo;
          *reinterpret_cast<uint2*>(tb + (size_t)(c_hi >> 6) * 8192 + rw * 64 + ((((c_hi & 63) >> 3) ^ (rw & 7)) << 3) + (c_hi & 7)) = vhi;
        } else {
          __nv_bfloat16* dst = isq ? g.qr + ((size_t)(b * g.Hq + head) * g.S + row) * g.dh
                                   : g.kr + ((size_t)(b * g.Hkv + head) * g.Sk_stride + g.koff + row) * g.dh;
          *reinterpret_cast<uint2*>(dst + c_lo) = vlo;
          *reinterpret_cast<uint2*>(dst + c_hi) = vhi;
        }
      } else {
        const int nn = n0 - Nq - Nk, head = nn / g.dh;
        __nv_bfloat16* dst = g.vr + ((size_t)(b * g.Hkv + head) * g.Sk_stride + g.koff + row) * g.dh + (nn - head * g.dh) + j0;
        *reinterpret_cast<uint2*>(dst) = pack4(lo);
        *reinterpret_cast<uint2*>(dst + 64) = pack4(hi);
      }
    }
    trace_stamp(tr, 5);
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  trace_stamp(tr, 6);
  if (warp == 17) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, 32);
  }
}

size_t bp_smem(int nk, int KP, int M) {
  const int HN = (M + 15) / 16 * 8;
  const size_t ops = (size_t)nk * (BP_A + HN * 128), stg = (size_t)2 * HN * 256;
  return 1024 + (ops > stg ? ops : stg) + (KP > 1 ? (size_t)KP * ((M + KP - 1) / KP) * 256 : 0);
}

template <int EPI, int WB>
cudaError_t launch_one(int* status, const B1Gemm& g, int KP, cudaStream_t st) {
  static PerDeviceOnce once;
  if (once.needed()) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_b1_pair<EPI, WB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BP_SMEM_MAX);
    if (e != cudaSuccess) return e;
    once.done();
  }
  CUtensorMap tw{}, tx;
  if ((WB == 0 && !row_map(&tw, g.W, (uint64_t)g.N * (g.K / 64), 32)) ||
      !row_map(&tx, g.X, (uint64_t)g.K, (uint32_t)((g.M + 15) / 16 * 8)))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * KP, g.N / 128, 1), cfg.blockDim = dim3(BP_THREADS), cfg.dynamicSmemBytes = bp_smem(g.nk_max, KP, g.M), cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2 * KP, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at, cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_gemm_b1_pair<EPI, WB>, status, g, tw, tx);
}

}  // namespace

// k-ranges (CTA pairs per cluster) for a projection, or 0 if it does not fit: the chunks of a range stay resident, the grid
// has at most one CTA per SM.  One range where the contraction fits it (no reduce); otherwise as many as the cluster takes
// (the activations of a range, latency-bound, get fewer; four ranges leave a CTA of 51 tokens 13 to finish).
int b1_pair_ranges(int N, int K, int n_sm, int epi) {
  if (N % 128 || K % 64 || K < 64) return 0;
  const int tiles = N / 128, KC = K / 64;
  int KP = 1;
  if (epi == B1_RESID) {
    KP = KC < BP_MAXKP ? KC : BP_MAXKP;
    while (KP > 1 && 2 * KP * tiles > n_sm) --KP;
  }
  const int nk = (KC + KP - 1) / KP;
  if (epi == B1_RESID && KP < 2) return 0;         // (16 items of up to 64 tokens for 512 threads)
  return nk <= BP_MAXK && 2 * KP * tiles <= n_sm && bp_smem(nk, KP, 64) <= BP_SMEM_MAX ? KP : 0;
}

cudaError_t launch_b1_pair_gemm(int* status, const B1Gemm& g_in, int KP, cudaStream_t st) {
  B1Gemm g = g_in;
  g.nk_max = (g.K / 64 + KP - 1) / KP;
  if (g.M < 1 || g.M > 64 || g.nk_max > BP_MAXK || bp_smem(g.nk_max, KP, g.M) > BP_SMEM_MAX) return cudaErrorInvalidConfiguration;
  const int wb = g.W8 ? (g.w_bits == 4 ? 4 : 8) : 0;
  switch (g.epi) {
    case B1_QKV: return wb == 8 ? launch_one<B1_QKV, 8>(status, g, KP, st) : wb == 4 ? launch_one<B1_QKV, 4>(status, g, KP, st) : launch_one<B1_QKV, 0>(status, g, KP, st);
    case B1_GEGLU: return wb == 8 ? launch_one<B1_GEGLU, 8>(status, g, KP, st) : wb == 4 ? launch_one<B1_GEGLU, 4>(status, g, KP, st) : launch_one<B1_GEGLU, 0>(status, g, KP, st);
    default: return wb == 8 ? launch_one<B1_RESID, 8>(status, g, KP, st) : wb == 4 ? launch_one<B1_RESID, 4>(status, g, KP, st) : launch_one<B1_RESID, 0>(status, g, KP, st);
  }
}

}  // namespace phyai
