// bf16 tile GEMM on CTA pairs (tcgen05 cta_group::2) for calls of more than 64 tokens: a pair of SMs works on one tile of
// 256 output channels x NT tokens, a persistent grid of pairs walks all tiles, the epilogue of a tile runs under the
// main loop of the next.
//
// What bounds it.  An SM takes in about 62 bytes per clock from the L2 while all SMs stream (measured), its tensor
// core multiplies 128 x 256 x 16 in 128 clocks.  A 64-element k-chunk of a 128-row x 256-token tile is 48 KB for 512
// clocks of tensor work: 96 bytes per clock, ingest bound.  A 256 x 256 tile per SM needs 64 bytes per clock, but its
// accumulators fill the 512 tensor-memory columns, so that nothing overlaps its epilogue.  The pair has both: every SM
// holds 128 of the 256 weight rows and half of the tokens (the tensor cores read the other half from the peer's
// shared memory): 32 KB per k-chunk and SM at NT = 256, 64 bytes per clock, and 256 accumulator columns per tile, two
// tiles in tensor memory.
//
// Operands: the packed 128 x 64 weight blocks and the tiled activations are contiguous runs of 128-byte rows in their
// final (128-byte-swizzled) image, so two-dimensional tensor maps of 64-element rows fetch them; the copies of both
// SMs signal the leader's barrier (.cta_group::2), which alone issues the MMAs.
//
// Norms are folded into the projections either side, as in gemm_b1.cu: X holds bf16(h * gain), the accumulator columns
// are multiplied by rsqrt(mean h^2 + eps) of their token (from partial sums of squares), a shift enters as the
// per-channel constant shift . W; the residual epilogue writes h, the next projection's operand and its partial sums of
// squares (one per 64 channels and token).  No split-K and no atomics: a request gives the same bits every time.
//
// Measured in the captured ten-step loops of the pi0 shape, against the one-CTA tile GEMMs and their norm launches (with the
// pair attention's part): 4 requests of 816 tokens 11.3 -> 9.4 ms, 8: 12.9 -> 10.8, 64 ragged: 33.1 -> 29.9 (power-capped, SM
// clock 1.73 GHz), 256: 119.6 -> 107.7 (1.55 GHz).  With cluster arrivals that do not release at cluster scope, shorter epilogues and the
// persistent pair attention since: 8.3, 9.4, 28.0 (1.65 GHz), 100 (1.4 - 1.5 GHz).
//
// Roles: warps 0-3 issue the copies (k-step i by warp i % 4), warp 4 issues the MMAs (leader CTA), the 16 warps from 5
// on are the epilogue (tensor-memory lane quarter = warp % 4).  Every wait is
// bounded; after a give-up copies, MMAs, commits and barriers go on and only the stores are skipped.
#include <algorithm>

#include "kernels.h"
#include "ptx.cuh"
#include "tc.cuh"
#include "tc_pair.cuh"

namespace phyai {
namespace {

constexpr int PG_PROD = 4;
constexpr int PG_EPI = 512, PG_THREADS = (PG_PROD + 1) * 32 + PG_EPI;
// tokens an epilogue warp takes at a time: 16, so that the body of the loop is short (its code is fetched once per launch: with 32 in
// the GeGLU epilogue 2 / 4 requests 7.65 / 8.34 ms, with 16 7.59 / 8.31) and the rotary epilogue has the registers to hold the (cos, sin)
// of the next two blocks (one 32-token block ahead on 8 warps: 7 us per tile, bound by the table's latency)
constexpr int PG_TB = 16;
constexpr int PG_MAXST = 20;
// one CTA's weight block: 128 rows x 64 k; 64 rows in the half-height form (residual projections of few tokens)
template <bool HALF> constexpr int PG_A_BYTES = (HALF ? 64 : 128) * 128;
constexpr int BAR_EPI = 1;
constexpr int PG_PITCH = 36, PG_STG = 16 * PG_PITCH;      // staging block of an epilogue warp: [16 tokens][32 rows + 4] floats
constexpr size_t PG_STG_BYTES = (size_t)16 * PG_STG * 4;
constexpr size_t PG_SMEM_MAX = 227 * 1024 - 11 * 1024;   // dynamic shared memory (the static tables take the rest)

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}
// 16 columns of 16 tensor-memory lanes in the fragment order of the matrix instructions: registers 4 k .. 4 k + 3 of lane T
// hold (row T / 4, columns 8 k + 2 (T % 4), + 1) and the same columns of row T / 4 + 8
__device__ __forceinline__ void tmem_ld_frag16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait16(float* a, float* b) {    // the registers pass through, so that no use moves up
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]), "+f"(b[0]), "+f"(b[1]),
                 "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
               :
               : "memory");
}
// four 8 x 8 bf16 matrices in fragment order -> shared memory, transposed (a memory row = a fragment column)
__device__ __forceinline__ void stmatrix4_t(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}

// CPS: k-chunks of 64 per ring stage.  A stage costs the MMA issuer a wait and a commit on top of the chunks' copies; with few
// tokens per tile that, not bytes or tensor time, set the pace (290 clocks per chunk whatever its size; with four chunks per
// stage 165, the ingest of the SM: down projection of 204 tokens 9.9 -> 5.6 us).
// EPI PG_EMBED (internal): PG_RESID of the action MLP, whose rows start from a bias or the state token instead of h.  (A kernel of its
// own, and the addresses of the residual epilogue as increments: its code is fetched once per launch, between the accumulator and
// the stores; ten-step loops of 2 / 4 / 8 / 16 requests 7.88 / 8.54 / 9.72 / 11.31 ms before, 7.70 / 8.37 / 9.54 / 11.20 after.)
constexpr int PG_EMBED = 4;

template <int EPI, bool HALF, int CPS>
__global__ void __launch_bounds__(PG_THREADS, 1) __cluster_dims__(2, 1, 1)
    k_gemm_pair(int* status, const PairGemm g, const __grid_constant__ CUtensorMap tmw, const __grid_constant__ CUtensorMap tmx) {
  constexpr bool RESID = EPI == PG_RESID || EPI == PG_EMBED;
  constexpr int EPIW = PG_EPI / 32, TB = PG_TB, K8 = TB / 8, A_BYTES = PG_A_BYTES<HALF>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[PG_MAXST];    // leader: both CTAs' operands of a stage have landed
  __shared__ __align__(8) uint64_t bar_empty[PG_MAXST];   // each CTA: the MMAs have read the stage
  __shared__ __align__(8) uint64_t bar_tfull[2];          // each CTA: accumulator complete
  __shared__ __align__(8) uint64_t bar_tempty[2];         // leader: accumulator read out by the epilogue warps of both
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ __align__(16) float rs_tab[2][256];                        // per token: the folded norm's 1 / rms
  // QKV: (position x dh / 2, element offset of the token's row in q without the head term, the same in k / v, suffix row)
  __shared__ int4 tok_tab[EPI == PG_QKV ? 2 : 1][EPI == PG_QKV ? 256 : 1];
  __shared__ float ss_tab[RESID ? 4 : 1][RESID ? 256 : 1];   // partial sums of squares per lane quarter

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int KC = g.K >> 6, NT = g.NT, ST = g.stages, KS = KC / CPS;   // CPS k-chunks per stage, KS stages per tile
  const int n_n = HALF ? g.N >> 7 : g.N >> 8;             // tiles of 256 (128) channels
  const int n_tiles = n_n * ((g.M + NT - 1) / NT);
  const int n_my = pair < n_tiles ? (n_tiles - pair + n_pairs - 1) / n_pairs : 0;
  const int steps = n_my * KS;
  const uint32_t chunk_bytes = (uint32_t)(A_BYTES + NT * 64), stage_bytes = chunk_bytes * (uint32_t)CPS;

  pdl_launch_dependents();
  unsigned long long* const trc = g.trace ? g.trace + (size_t)blockIdx.x * 16 : nullptr;
  if (threadIdx.x == 0) trace_stamp(trc, 0);
  if (threadIdx.x == 32) {      // (the first copy would otherwise wait for its map)
    prefetch_tmap(&tmw), prefetch_tmap(&tmx);
  }
  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < ST; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bar_tfull[b]), 1);
      mbar_init(smem_u32(&bar_tempty[b]), 2 * EPIW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == PG_PROD) {
    tmem_alloc2(smem_u32(&tmem_slot), 512);
    tc_fence_before();
  }
  __syncthreads();
  pair_sync();                                            // the peer's barriers exist before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&tmem_slot), 0);
  const WaitCtx wc{status, &abort_flag, g.wait_limit, true};
  if (threadIdx.x == 0) trace_stamp(trc, 1);

  if (warp < PG_PROD) {
    // ---------------- copy issuers -------------------------------------------------------------------------------
    if (lane == 0) {
      auto load_w = [&](int gi, int s) {
        const int ct = ((pair + (gi / KS) * n_pairs) % n_n) * 2 + rank, kc = (gi % KS) * CPS;      // this CTA's 128-row (64-row) weight tile
        const uint32_t full = smem_u32(&bar_full[s]);
        if (rank == 0) mbar_expect_tx(full, 2 * stage_bytes);
        const int row = g.w_row0 + (HALF ? ((ct >> 1) * KC + kc) * 128 + rank * 64 : (ct * KC + kc) * 128);
        for (int c = 0; c < CPS; ++c) tma2d(tiles + (uint32_t)s * stage_bytes + (uint32_t)c * chunk_bytes, &tmw, row + c * 128, full & LEADER_MASK);
      };
      auto load_x = [&](int gi, int s) {
        const int row = (gi % KS) * CPS * g.rows_pad + (pair + (gi / KS) * n_pairs) / n_n * NT + rank * (NT >> 1);
        for (int c = 0; c < CPS; ++c)
          tma2d(tiles + (uint32_t)s * stage_bytes + (uint32_t)c * chunk_bytes + A_BYTES, &tmx, row + c * g.rows_pad, smem_u32(&bar_full[s]) & LEADER_MASK);
      };
      // Programmatic dependent launch: the weight blocks of the first stages are on their way before the kernel that
      // produces the activations has finished.
      const int n_early = steps < ST ? steps : ST;
      for (int gi = warp; gi < n_early; gi += PG_PROD) load_w(gi, gi);
      pdl_wait();
      if (warp == 0) {
        trace_stamp(trc, 2);
        if (rank == 1) trace_stamp(trc, 3), trace_stamp(trc, 4);             // (only the leader issues MMAs)
      }
      for (int gi = warp; gi < n_early; gi += PG_PROD) load_x(gi, gi);
      for (int gi = warp; gi < steps; gi += PG_PROD) {
        if (gi < n_early) continue;
        const int s = gi % ST;
        if (mbar_wait_drain(smem_u32(&bar_empty[s]), ((uint32_t)(gi / ST) & 1u) ^ 1u, wc) < 0) break;
        load_w(gi, s);
        load_x(gi, s);
      }
    }
  } else if (warp == PG_PROD) {
    const WaitCtx wm{status, &abort_flag, g.wait_limit};
    // ---------------- MMA issuer (whole warp in the loop, one elected lane issues) --------------------------------
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((HALF ? 128u : 256u) >> 4) << 24;
      int s = 0, gi = 0;
      uint32_t ph = 0;
      bool dead = false;
      for (int i = 0; i < n_my && !dead; ++i) {
        const int buf = i & 1;
        // the epilogue warps of both CTAs have read the accumulator that this tile overwrites (two tiles ago)
        if (mbar_wait_drain(smem_u32(&bar_tempty[buf]), (((uint32_t)i >> 1) & 1u) ^ 1u, wm) < 0) break;
        tc_fence_after();
        const uint32_t tacc = tmem_base + (uint32_t)buf * 256u;
        for (int k = 0; k < KS; ++k, ++gi) {
          if (mbar_wait_drain(smem_u32(&bar_full[s]), ph, wm) < 0) {
            dead = true;   // (copies that never landed: nothing more can be done with this pipeline)
            break;
          }
          if (gi == 0 && lane == 0) trace_stamp(trc, 3);
          uint32_t a0 = tiles + (uint32_t)s * stage_bytes;
          // (two chunks per turn: unrolled further, more code to fetch at the start of every layer's kernel than the issue rate gains;
          // ten-step loops of 2 / 8 requests 7.69 / 9.55 ms with all four, 7.64 / 9.47 with two, 7.72 / 9.44 with one, which costs 16 requests 1 %)
#pragma unroll 2
          for (int c = 0; c < CPS; ++c, a0 += chunk_bytes) {
            const uint64_t da = make_desc(a0), db = make_desc(a0 + A_BYTES);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              if (elect_one()) umma2_bf16(tacc, da + 2 * kk, db + 2 * kk, idesc, (k > 0 || c > 0 || kk > 0) ? 1u : 0u);
          }
          if (elect_one()) umma2_commit(smem_u32(&bar_empty[s]));
          __syncwarp();
          if (++s == ST) s = 0, ph ^= 1u;
        }
        if (!dead && elect_one()) umma2_commit(smem_u32(&bar_tfull[buf]));
        __syncwarp();
      }
      if (lane == 0) trace_stamp(trc, 4);
    }
  } else {
    // ---------------- epilogue: tensor memory -> registers -> global ---------------------------------------------
    // The code is kept short: in a captured loop a kernel's code has left the instruction caches by the next layer, and a
    // first version, unrolled per element (one row per thread, 2- and 4-byte stores), spent 14 us on a residual tile.
    // Shared memory is used sparingly: while the main loop runs, the tensor core's operand reads and the copies take most
    // of its bandwidth.
    const int ew = warp - (PG_PROD + 1);
    const int q = warp & 3, cg = ew >> 2;    // tensor-memory lane quarter; column blocks cg, cg + 4, ...
    const int et = ew * 32 + lane;
    const uint32_t tl_addr = tmem_base + ((uint32_t)(q * 32) << 16);
    float* const stg = reinterpret_cast<float*>(smem_raw + (tiles - smem_u32(smem_raw)) + (size_t)ST * stage_bytes) + ew * PG_STG;
    uint32_t tempty0;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(tempty0) : "r"(smem_u32(&bar_tempty[0])));
    bool dead = false;
    pdl_wait();
    const bool skip = status_set(status);
    for (int i = 0; i < n_my; ++i) {
      const int buf = i & 1;
      const int t = pair + i * n_pairs;
      const int ct = (t % n_n) * 2 + rank, tok_base = (t / n_n) * NT;      // this CTA's 128 channels; first token
      const int n_tok = min(NT, g.M - tok_base), n0 = ct * (HALF ? 64 : 128);
      // half height: 64 rows, the second half of the token columns in lanes 64..127
      const int th = HALF ? (q >> 1) * (NT >> 1) : 0, tl_end = HALF ? min(n_tok, th + (NT >> 1)) : n_tok;
      // ---- before the accumulator is complete: per-token and per-channel factors
      if (EPI == PG_GEGLU || EPI == PG_QKV) {
        if (et < NT) {      // (NT <= 256 <= threads of the epilogue)
          float ss = 0.f;
#pragma unroll 8
          for (int j = 0; j < g.ss_n; ++j) ss += __ldg(g.ss_in + (size_t)j * g.rows_pad + min(tok_base + et, g.M - 1));
          rs_tab[buf][et] = 1.0f / sqrtf(ss * g.inv_D + g.eps);
        }
      }
      if constexpr (EPI == PG_QKV) {
        if (et < n_tok) {
          const int tok = tok_base + et, b = tok / g.S, ii = tok - b * g.S;
          const int* cu = g.rq->cu_lens;
          const int qo = g.q_tiles ? b * g.Hq * 64 * g.dh + ii * 64 : (b * g.Hq * g.S + ii) * g.dh;
          tok_tab[buf][et] = make_int4((cu[b + 1] - cu[b] + ii) * (g.dh >> 1), qo, (b * g.Hkv * g.S + ii) * g.dh, ii);
        }
      }
      // (a warp can be at most one tile ahead of the slowest: it passes this barrier only after every warp has left the
      // tile before, so the tables of the tile before that are free to be overwritten)
      asm volatile("bar.sync %0, %1;" ::"n"(BAR_EPI), "n"(PG_EPI) : "memory");
      // GEGLU / QKV / PLANES: a warp's 32 rows are two groups of 16: gate (first-half, first) rows and the up (partner, next)
      // rows; in fragment order a lane holds channels lane / 4 and + 8 of both groups, i.e. the pairs that are combined.
      // Their weight scales and shifts: [group][channel lane / 4 or + 8]
      float sc[2][2] = {{1.f, 1.f}, {1.f, 1.f}}, sh[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, scr = 1.0f;
      if constexpr (EPI == PG_GEGLU || EPI == PG_QKV) {
        const float osc = (EPI == PG_QKV && n0 < g.Hq * g.dh) ? rsqrtf((float)g.dh) : 1.0f;   // q leaves scaled by 1 / sqrt(dh)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int gr = e >> 1, cl = 16 * q + (lane >> 2) + 8 * (e & 1), row = n0 + 64 * gr + cl;
          const float* sp = EPI == PG_QKV ? g.scale : (gr ? g.scale2 : g.scale);
          if (sp) sc[gr][e & 1] = sp[EPI == PG_QKV ? row : ct * 64 + cl];
          if (g.shift) sh[gr][e & 1] = g.shift[row] * osc;
          sc[gr][e & 1] *= osc;
        }
      } else if constexpr (RESID) {
        const int n = n0 + (HALF ? q & 1 : q) * 32 + lane;
        if (g.scale) scr = g.scale[n];
        if (g.gate) scr *= g.gate[n];
      }
      // where a lane's 16-byte pieces go: tokens lane / 2 and + 16 of a 32-token block, channels 8 (lane & 1) .. of a group
      const int p8 = 16 * q + 8 * (lane & 1);
      __nv_bfloat16* obase = nullptr;
      int off2 = 0, rope_c = 0;
      bool isq = false, rot = false, qt = false;
      if constexpr (EPI == PG_GEGLU) {
        obase = g.out + (size_t)ct * g.rows_pad * 64;
      } else if constexpr (EPI == PG_QKV) {
        const int Nq = g.Hq * g.dh, Nqk = Nq + g.Hkv * g.dh;
        isq = n0 < Nq, rot = n0 < Nqk;
        const int nn = isq ? n0 : (rot ? n0 - Nq : n0 - Nqk), head = nn / g.dh, coff = nn - head * g.dh;
        // q / k: channels coff / 2 + .. and their partners dh / 2 further; v: coff + .. and + 64
        rope_c = (coff >> 1) + 16 * q + 2 * (lane >> 2), off2 = rot ? g.dh >> 1 : 64;
        obase = (isq ? g.qr : (rot ? g.kr : g.vr)) + (size_t)head * g.S * g.dh + (rot ? coff >> 1 : coff) + p8;
        qt = isq && g.q_tiles;
        if (qt) {     // operand tiles: (request, head pair) -> dh / 64 blocks of [64 (head & 1) + row][64 channels], swizzled
          obase = g.q_tiles + (size_t)(head >> 1) * 128 * g.dh + (head & 1) * 4096 + (size_t)(coff >> 7) * 8192;
          off2 = (g.dh >> 7) * 8192;
        }
      } else if constexpr (EPI == PG_PLANES) {
        // K | V projections of all layers: row n belongs to plane n / nkv (a warp's 32 rows to one: nkv is a multiple of 64)
        const int n = n0 + 32 * q, plane = n / g.nkv;
        if (plane < g.n_planes) obase = g.out + (size_t)plane * g.plane_rows * g.nkv + (n - plane * g.nkv) + 8 * (lane & 1);
        off2 = 16;
      }
      // RESID: in the transposed view a lane takes 4 channels of tokens lane / 8, + 4, + 8, + 12 of the chunk; what is added
      // to (the residual stream, or the MLP's bias / the state token) is requested one chunk ahead
      const int n4 = n0 + (HALF ? q & 1 : q) * 32 + (lane & 7) * 4;
      const float* const hrow = g.h + (size_t)(tok_base + (lane >> 3)) * g.N + n4;
      float4 old[2][4], gain4 = make_float4(0.f, 0.f, 0.f, 0.f);
      auto fetch_old = [&](int c0, float4* o) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int tl = c0 + 4 * u + (lane >> 3), tok = tok_base + tl;
          const float* src = hrow + (size_t)(c0 + 4 * u) * g.N;
          if (EPI == PG_EMBED) src = (tok % g.S) < g.ns ? g.state_tok + (size_t)(tok / g.S) * g.N + n4 : g.bias + n4;
          o[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (tl < n_tok) o[u] = *reinterpret_cast<const float4*>(src);
        }
      };
      if constexpr (RESID) {
        if (g.gain_next) gain4 = __ldg(reinterpret_cast<const float4*>(g.gain_next + n4));
        if (th + cg * 16 < tl_end) fetch_old(th + cg * 16, old[0]);
        if (th + cg * 16 + 64 < tl_end) fetch_old(th + cg * 16 + 64, old[1]);
      }
      // q / k: (cos, sin) of this lane's rotary pairs at its tokens, two 16-token blocks ahead
      float2 cs[2][EPI == PG_QKV ? 8 : 1];
      auto fetch_cs = [&](int c0, float2* o) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(g.rope + tok_tab[buf][min(c0 + 2 * (lane & 3) + 8 * k + e, n_tok - 1)].x + rope_c));
            o[4 * k + e] = make_float2(x.x, x.y), o[4 * k + 2 + e] = make_float2(x.z, x.w);
          }
      };
      const bool do_rot = EPI == PG_QKV && rot && g.rope && !skip;
      if constexpr (EPI == PG_QKV) {
        if (do_rot) fetch_cs(cg * 16, cs[0]), fetch_cs(cg * 16 + 64, cs[1]);
      }
      // ---- the accumulator
      int r = 0;
      if (!dead) {
        if (lane == 0) r = mbar_wait_drain(smem_u32(&bar_tfull[buf]), ((uint32_t)i >> 1) & 1u, wc);
        r = __shfl_sync(0xffffffffu, r, 0);
        if (r < 0) dead = true;
      }
      const bool ok = !skip && !dead && r > 0 && !*reinterpret_cast<volatile int*>(&abort_flag);
      tc_fence_after();
      if (i == 0 && et == 0) trace_stamp(trc, 5);
      __nv_bfloat16* const orow = RESID ? g.out + ((size_t)(n4 >> 6) * g.rows_pad + tok_base + (lane >> 3)) * 64 + (n4 & 7) : nullptr;
      if constexpr (RESID) {
        // 16 token columns at a time: the lane that holds a row scales it and puts it into the warp's staging block [16
        // tokens][32 rows + 4]; then 8 lanes take the 32 channels (128 bytes of h) of one token
#pragma unroll 1
        for (int c0 = th + cg * 16; c0 < tl_end; c0 += 64) {
          float v[16];
          tmem_ld16(tl_addr + (uint32_t)(buf * 256 + c0 - th), v);
#pragma unroll
          for (int j = 0; j < 16; ++j) stg[j * PG_PITCH + lane] = v[j] * scr;
          __syncwarp();
          const float* sp = stg + (lane >> 3) * PG_PITCH + (lane & 7) * 4;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int tl = c0 + 4 * u + (lane >> 3), tok = tok_base + tl;
            const float4 a = *reinterpret_cast<const float4*>(sp + 4 * u * PG_PITCH);
            const bool live = EPI != PG_EMBED || (tok % g.S) >= g.ns;       // (state rows do not pass through the MLP)
            float4 hv = old[0][u];
            if (live) hv.x += a.x, hv.y += a.y, hv.z += a.z, hv.w += a.w;
            if (ok && tl < tl_end) {
              *reinterpret_cast<float4*>(const_cast<float*>(hrow) + (size_t)(c0 + 4 * u) * g.N) = hv;
              if (g.gain_next)
                *reinterpret_cast<uint2*>(orow + (c0 + 4 * u) * 64 + ((((n4 & 63) >> 3) ^ (tok & 7)) << 3)) =
                    make_uint2(pack_bf16x2(hv.x * gain4.x, hv.y * gain4.y), pack_bf16x2(hv.z * gain4.z, hv.w * gain4.w));
            }
            float s2 = hv.x * hv.x + hv.y * hv.y + hv.z * hv.z + hv.w * hv.w;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            if ((lane & 7) == 0 && tl < tl_end) ss_tab[q][tl] = s2;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) old[0][u] = old[1][u];
          if (c0 + 128 < tl_end) fetch_old(c0 + 128, old[1]);
          __syncwarp();
        }
      } else {
        // TB token columns at a time, both row groups in fragment order; the bf16 results go through the warp's staging
        // block [TB tokens][16 channels] (16-byte chunks swapped in every other group of four tokens against bank
        // conflicts) by transposing matrix stores and leave as 16-byte pieces, two lanes to a 32-byte sector
        const uint32_t st_s = smem_u32(stg);
        const uint32_t st_w = st_s + (uint32_t)((8 * (lane >> 4) + (lane & 7)) * 32 + ((((lane >> 3) & 1) ^ ((lane >> 2) & 1)) << 4));
        const uint32_t st_r = st_s + (uint32_t)((lane >> 1) * 32 + (((lane & 1) ^ ((lane >> 3) & 1)) << 4));
#pragma unroll 1
        for (int c0 = cg * TB; c0 < n_tok; c0 += 4 * TB) {
          float a[4 * K8], b[4 * K8];
          const uint32_t ta = tl_addr + (uint32_t)(buf * 256 + c0), tb = ta + (16u << 16);
          tmem_ld_frag16(ta, a), tmem_ld_frag16(tb, b);
          tmem_ld_wait16(a, b);
          const int t2 = c0 + 2 * (lane & 3);            // this lane's tokens: t2 + 8 k and + 1
          if (EPI == PG_GEGLU || EPI == PG_QKV) {
#pragma unroll
            for (int k = 0; k < K8; ++k) {
              const float2 rs = *reinterpret_cast<const float2*>(&rs_tab[buf][t2 + 8 * k]);
#pragma unroll
              for (int e = 0; e < 4; ++e) {              // e: channel e / 2, token e % 2
                const float r1 = (e & 1) ? rs.y : rs.x;
                a[4 * k + e] = fmaf(a[4 * k + e] * sc[0][e >> 1], r1, sh[0][e >> 1]);
                b[4 * k + e] = fmaf(b[4 * k + e] * sc[1][e >> 1], r1, sh[1][e >> 1]);
              }
            }
          }
          if constexpr (EPI == PG_GEGLU) {
            gelu_mul(a, b, g.gelu_exact);
          } else if constexpr (EPI == PG_QKV) {
            if (do_rot) {
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                const float l0 = a[e], u0 = b[e];
                a[e] = l0 * cs[0][e].x - u0 * cs[0][e].y, b[e] = u0 * cs[0][e].x + l0 * cs[0][e].y;
                cs[0][e] = cs[1][e];
              }
              if (c0 + 128 < n_tok) fetch_cs(c0 + 128, cs[1]);
            }
          }
#pragma unroll
          for (int m = 0; m < (EPI == PG_GEGLU ? 1 : 2); ++m) {      // the two row groups one after the other
            const float* x = m ? b : a;
#pragma unroll
            for (int k = 0; k < K8; k += 2)
              stmatrix4_t(st_w + (uint32_t)k * 256, pack_bf16x2(x[4 * k], x[4 * k + 1]), pack_bf16x2(x[4 * k + 2], x[4 * k + 3]),
                          pack_bf16x2(x[4 * k + 4], x[4 * k + 5]), pack_bf16x2(x[4 * k + 6], x[4 * k + 7]));
            __syncwarp();
#pragma unroll
            for (int it = 0; it < TB / 16; ++it) {
              const int tl = c0 + (lane >> 1) + 16 * it, tok = tok_base + tl;
              uint4 w;
              asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "r"(st_r + (uint32_t)it * 512) : "memory");
              if (ok && tl < n_tok && (EPI != PG_PLANES || obase)) {
                __nv_bfloat16* dst = obase;
                if constexpr (EPI == PG_GEGLU) dst += (size_t)tok * 64 + (((p8 >> 3) ^ (tok & 7)) << 3);
                else if constexpr (EPI == PG_QKV) {
                  const int4 e4 = tok_tab[buf][tl];
                  dst += (isq ? e4.y : e4.z) + m * off2 + (qt ? ((p8 >> 3) ^ (e4.w & 7)) << 3 : 0);
                }
                else dst += (size_t)tok * g.nkv + m * off2;
                if (EPI == PG_PLANES && (reinterpret_cast<uintptr_t>(dst) & 15u)) {      // (planes at a caller's address)
                  reinterpret_cast<uint2*>(dst)[0] = make_uint2(w.x, w.y), reinterpret_cast<uint2*>(dst)[1] = make_uint2(w.z, w.w);
                } else {
                  *reinterpret_cast<uint4*>(dst) = w;
                }
              }
            }
            __syncwarp();
          }
        }
      }
      // this warp has read its part of the accumulator: the MMAs of the tile after next may overwrite it
      tc_fence_before();
      if (lane == 0)
        remote_arrive(tempty0 + (uint32_t)buf * 8u);
      if constexpr (RESID) {
        if (g.ss_out) {
          asm volatile("bar.sync %0, %1;" ::"n"(BAR_EPI + 1), "n"(PG_EPI) : "memory");
          if (ok && et < n_tok) {     // one partial sum per 64 channels and token
            float* so = g.ss_out + tok_base + et;
            const int q0 = HALF && et >= (NT >> 1) ? 2 : 0;
            so[(size_t)(HALF ? ct : 2 * ct) * g.rows_pad] = ss_tab[q0][et] + ss_tab[q0 + 1][et];
            if (!HALF) so[(size_t)(2 * ct + 1) * g.rows_pad] = ss_tab[2][et] + ss_tab[3][et];
          }
        }
      }
    }
    if (et == 0 && trc) {
      unsigned long long tt;
      unsigned sm;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(tt)::"memory");
      asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
      trc[6] = tt, trc[7] = sm, trc[9] = (unsigned long long)n_my;
    }
  }

  __syncthreads();
  // Neither CTA leaves (or gives its tensor memory back) while the other still works: the leader's MMAs read both CTAs'
  // shared memory and write both tensor memories.
  cluster_arrive_relaxed();
  cluster_wait();
  if (warp == PG_PROD) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, 512);
    if (lane == 0 && trc) {
      unsigned long long tt;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(tt)::"memory");
      trc[8] = tt;
    }
  }
}

template <int EPI, bool HALF, int CPS>
cudaError_t launch_cps(int* status, const PairGemm& g, int grid, size_t smem, const CUtensorMap& tw, const CUtensorMap& tx, cudaStream_t st) {
  static PerDeviceOnce once;
  if (once.needed()) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_pair<EPI, HALF, CPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM_MAX);
    if (e != cudaSuccess) return e;
    once.done();
  }
  return launch_pdl(k_gemm_pair<EPI, HALF, CPS>, dim3(grid), dim3(PG_THREADS), smem, st, status, g, tw, tx);
}

template <int EPI, bool HALF = false>
cudaError_t launch_one(int* status, const PairGemm& g, int grid, size_t smem, const CUtensorMap& tw, const CUtensorMap& tx, cudaStream_t st) {
  if (g.cps == 4) return launch_cps<EPI, HALF, 4>(status, g, grid, smem, tw, tx, st);
  if (g.cps == 2) return launch_cps<EPI, HALF, 2>(status, g, grid, smem, tw, tx, st);
  return launch_cps<EPI, HALF, 1>(status, g, grid, smem, tw, tx, st);
}

}  // namespace

bool pair_gemm_supported(int N, int K) { return N % 256 == 0 && K % 64 == 0 && K > 0; }

// Tile of a projection: the token width and, for residual projections, the height (256 or 128 channels per pair) with the
// least work on the busiest pair, in clocks.  A k-chunk of a tile costs the larger of the tensor time (2 NT: four MMAs of
// NT / 2) and the ingest of an SM (16 or 8 KB of weights + 64 NT bytes of activations at 62 bytes per clock); the last tile's
// epilogue is exposed (30 - 60 per token column).  A grid that does not fit beside the kernel before it (`busy` CTAs, one per
// SM) has CTAs that start only when that one ends, and then pay their set-up and the first weights' latency: about 3600
// (measured: 1.9 us).  The half-height tile: few tokens against a long contraction leave 40 - 60 pairs whose SMs are bound
// by the 16 KB of weights per chunk (down projection at 408 tokens: 10.2 us of main loop, 6.2 at half height).
struct PairTile {
  int nt;
  bool half;
};
PairTile pick_tile(const PairGemm& g, int n_sm, int busy) {
  double best = 1e30;
  PairTile t{256, false};
  for (int half = 0; half <= (g.epi == PG_RESID ? 1 : 0); ++half)
    for (int nt = 256; nt >= 32; nt -= 16) {
      const int tiles = g.N / (half ? 128 : 256) * ((g.M + nt - 1) / nt), pairs = n_sm / 2;
      const double chunk = std::max(2.0 * nt, ((half ? PG_A_BYTES<true> : PG_A_BYTES<false>) + 64.0 * nt) / 62.0);
      const double epi = g.epi != PG_RESID ? 30.0 : half ? 30.0 : 60.0;
      const double cost = (double)((tiles + pairs - 1) / pairs) * (g.K / 64) * chunk + epi * nt + (2 * std::min(tiles, pairs) + busy > n_sm ? 3600.0 : 0.0);
      if (cost < best * 0.999) best = cost, t = PairTile{nt, half != 0};
    }
  return t;
}

cudaError_t launch_pair_gemm(int* status, const PairGemm& g_in, int n_sm, int* busy, cudaStream_t st) {
  PairGemm g = g_in;
  if (!pair_gemm_supported(g.N, g.K) || g.M < 1) return cudaErrorInvalidValue;
  const PairTile t = pick_tile(g, n_sm, *busy);
  g.NT = t.nt;
  const size_t chunk = (size_t)(t.half ? PG_A_BYTES<true> : PG_A_BYTES<false>) + 64 * g.NT, ring = PG_SMEM_MAX - 1024 - PG_STG_BYTES;
  // As many chunks per stage as leave a stage to each copy issuer (PG_PROD: with fewer, two issuers would meet in one stage
  // and its parity could not tell their turns apart).
  g.cps = 1;
  while (g.cps < 4 && (g.K / 64) % (2 * g.cps) == 0 && 2 * g.cps * PG_PROD * chunk <= ring) g.cps *= 2;
  const size_t stage = g.cps * chunk;
  g.stages = (int)std::min<size_t>(ring / stage, PG_MAXST);
  CUtensorMap tw, tx;
  if (!row_map(&tw, g.W, g.w_rows, t.half ? 64 : 128) || !row_map(&tx, g.X, (uint64_t)(g.K / 64) * g.rows_pad, (uint32_t)(g.NT / 2)))
    return cudaErrorInvalidValue;
  const int n_tiles = g.N / (t.half ? 128 : 256) * ((g.M + g.NT - 1) / g.NT);
  const int grid = 2 * std::min(n_tiles, n_sm / 2);
  *busy = grid;
  const size_t smem = (size_t)g.stages * stage + 1024 + PG_STG_BYTES;
  if (g.bias) return t.half ? launch_one<PG_EMBED, true>(status, g, grid, smem, tw, tx, st) : launch_one<PG_EMBED>(status, g, grid, smem, tw, tx, st);
  if (t.half) return launch_one<PG_RESID, true>(status, g, grid, smem, tw, tx, st);
  switch (g.epi) {
    case PG_QKV: return launch_one<PG_QKV>(status, g, grid, smem, tw, tx, st);
    case PG_GEGLU: return launch_one<PG_GEGLU>(status, g, grid, smem, tw, tx, st);
    case PG_RESID: return launch_one<PG_RESID>(status, g, grid, smem, tw, tx, st);
    default: return launch_one<PG_PLANES>(status, g, grid, smem, tw, tx, st);
  }
}

}  // namespace phyai
