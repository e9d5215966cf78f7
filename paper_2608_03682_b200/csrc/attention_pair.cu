// Suffix -> (prefix U suffix) attention on CTA pairs (tcgen05 cta_group::2), for calls of several requests.
//
// A pair of SMs takes four query heads of one request that share a kv head (each CTA two of them: 2 x 64 padded rows = its
// 128 rows of the 256-row MMAs).  What bounds the one-CTA form of this kernel (attention_tc.cu) is the key / value stream
// -- every CTA reads all of K and V of its request -- and the tensor pipe at N = 64, which runs at half rate.  In a pair
// every CTA fetches half: of a 128-key tile its 64 keys of K and its DH / 2 channels of all 128 rows of V; the tensor cores
// read the other half from the peer's shared memory, and both products run at N = 128 / DH.  64 KB per CTA and tile of
// 2048 tensor clocks (head_dim 256): 32 bytes per clock, half of what an SM takes in.
//   S = Q K^T   M = 256, N = 128 keys, K = head_dim; Q (the QKV projection wrote it as this kernel's operand tile) and K in
//               shared memory; two S buffers in tensor memory, so that the logits of the next tile exist before the
//               softmax of this one is done
//   softmax     two threads per row (half of the columns each), straight from tensor memory; P (bf16) over the S buffer
//   O += P V    M = 256, N = head_dim, K = 128 keys; P is the tensor-memory A operand, V an MN-major B operand; rescaled
//               only when a row's maximum grows by more than 2^8
// The keys of a request are split over C = 2 to 4 pairs of one cluster (without a split: attention_persist.cu; each range: its share of the prefix and of
// the suffix keys); the fp32 partial results are merged over distributed shared memory: row range p of every head belongs to
// pair p, which is sent its rows of the other C - 1 partials and adds the C in range order.  No partials in global memory, no
// merge launch.  (Owners that read the partials from the other CTAs instead of being sent them: 4.2 us per launch more.)
//
// Measured at 8 requests of 816 + 51 keys and 8 heads (C = 3), from the projection's end to the merged output: 11.3 us (with
// arrivals that release at cluster scope 15; split ranges of the one-CTA kernel 21, their merge launch 8): operands 1.2 - 3, first
// tile 2.9, 1.25 per further tile, merge and output 4.2.  What bounds
// the merge is the way between SMs, 28 bytes per ns for one: a CTA sends (C - 1) / C of its 102 KB, in two pieces, the first
// while the second is staged (in one piece 0.7 us per launch more; as bf16, half the bytes, the merge took 3.7; through
// global memory, which all clusters share, 3 us more at 8 requests).
//
// Warps of a CTA: 0-1 load K, 2-3 load V (full prefix tiles with tensor-map copies -- the map of the call's cache sits in
// the request block --, the rest row by row with cp.async; prefix rows before the dependency wait), 4 issues the MMAs
// (leader CTA), 5-12 fetch Q, softmax, correction, output.  Every wait is bounded; after a give-up the protocol runs to its
// end and only the global stores are skipped.
#include "attention.cuh"
#include "attention_choice.h"
#include "tc.cuh"
#include "tc_pair.cuh"

namespace phyai {
namespace {

constexpr int KB = PAIR_TILE;                 // keys per tile
constexpr int AP_THREADS = 13 * 32;
constexpr int BAR_ROWS = 1, BAR_K = 2, BAR_V = 3;

template <int DH, int C>
struct ApLayout {
  static constexpr int KBLOCK = 64 * 128;                    // one 64-channel block of this CTA's 64 keys
  static constexpr int KTILE = (DH / 64) * KBLOCK;
  static constexpr int PIECE = (DH / 128) * KBLOCK;          // one tensor-map copy: 64 keys x DH / 2 channels
  static constexpr int VTILE = 2 * PIECE;                    // V: two halves of 64 keys, this CTA's DH / 2 channels
  static constexpr int QTILE = 128 * DH * 2;
  static constexpr int KV = 2 * (KTILE + VTILE);             // two buffers each
  // Partials: staged over the (by then dead) K / V buffers in blocks by owner (2 heads x own rows of O, then their (max, sum)
  // entries of 16 bytes: a bulk copy moves multiples of 16 bytes); behind them and behind K / V the blocks of the C - 1 peers,
  // over Q and past it.  Of 256 channels three ranges fit up to 63 suffix rows, four up to 60.
  static constexpr int S_MAX = DH != 256 || C < 3 ? 64 : (C == 3 ? 63 : 60);
  static constexpr int OWN = (S_MAX + C - 1) / C;            // most rows per head a pair finishes
  static constexpr int NP = DH / 128;                        // a block in pieces of 2 x 64 columns, sent as they are staged
  static constexpr int PITCH = 512 + 16;                     // fp32 row of a piece, padded against bank conflicts
  static constexpr int ROW = NP * PITCH + 16;
  static constexpr int STG = 2 * C * OWN * ROW, RECV = (STG > KV ? STG : KV), PEERS = 2 * (C - 1) * OWN * ROW;
  static constexpr size_t SMEM = 1024 + (size_t)(RECV + PEERS > KV + QTILE ? RECV + PEERS : KV + QTILE);
  static_assert(SMEM + 3072 <= 227 * 1024, "partials exceed the shared memory");
};

template <int DH, int C>
__global__ void __launch_bounds__(AP_THREADS, 1) k_attn_pair(const AttnArgs a, const __grid_constant__ CUtensorMap tmq) {
  using L = ApLayout<DH, C>;
  constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(KB >> 3) << 17) | ((256u >> 4) << 24);
  constexpr uint32_t IDESC_PV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((256u >> 4) << 24);

  extern __shared__ uint8_t smem_raw[];
  // leader: operands of a buffer, Q, P of a buffer complete in both CTAs.  Each CTA: logits / P V complete.
  __shared__ __align__(8) uint64_t k_full[2], v_full[2], p_full[2][2], s_full[2], pv_done[2], mrg_bar, q_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag, mrg_ok;
  __shared__ float xch[2][2][128];       // the two half-row threads of a row exchange their maximum (by tile parity) and, at the end, sum

  const Dims& d = a.d;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int crank = blockIdx.x, pr = crank >> 1, half = crank & 1;     // key range, CTA of the pair
  const int b = a.order ? a.order[blockIdx.z] : (int)blockIdx.z;       // longest requests first
  const int head0 = (int)blockIdx.y * 4 + half * 2;
  const int hk = head0 / (d.Hq / d.Hkv);
  const int S = d.S;
  unsigned long long* const trc = a.trace ? a.trace + (size_t)((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * 16 : nullptr;
  if (tid == 0) trace_stamp(trc, 0);
  if (tid == 5 * 32) prefetch_tmap(&tmq);
  pdl_launch_dependents();

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t Ks = base, Vs = base + 2 * L::KTILE, Qs = base + L::KV;
  const int own = (S + C - 1) / C, own_lo = pr * own, n_me = max(0, min(own, S - own_lo));   // suffix rows (per head) this CTA finishes
  const uint32_t slot = (uint32_t)(2 * own * L::ROW);
  const uint32_t stg = base, recv = base + max((uint32_t)C * slot, (uint32_t)L::KV);   // merge: blocks by owner; [C - 1 peers] mine

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&k_full[i]), 2), mbar_init(smem_u32(&v_full[i]), 2), mbar_init(smem_u32(&p_full[i][0]), 8), mbar_init(smem_u32(&p_full[i][1]), 8);
      mbar_init(smem_u32(&s_full[i]), 1), mbar_init(smem_u32(&pv_done[i]), 1);
    }
    mbar_init(smem_u32(&mrg_bar), 1), mbar_init(smem_u32(&q_bar), 1);
    if (n_me > 0) mbar_expect_tx(smem_u32(&mrg_bar), (uint32_t)((C - 1) * 2 * n_me * L::ROW));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 4) {
    tmem_alloc2(smem_u32(&tmem_slot), 512);
    tc_fence_before();
  }
  __syncthreads();
  pair_sync();                                      // every CTA's barriers exist before a peer can signal them
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&tmem_slot), 0);
  const uint32_t tmem_s = tmem_base, tmem_o = tmem_base + 2 * KB;
  const WaitCtx wc{a.status, &abort_flag, a.wait_limit};

  // Keys of this range: a share of the prefix keys followed by a share of the request's own (suffix) keys.  (The request
  // block is written before the captured loop starts: safe to read ahead of the dependency wait.  A call whose lengths are
  // invalid stores nothing; the clamps keep its loads inside the cache.)
  const Request r = *a.rq;
  const int kvt = (int)r.kv_tokens;
  const int p0 = min(max(r.cu_lens[b], 0), kvt), P = min(max(r.cu_lens[b + 1] - p0, 0), kvt - p0);
  const int pre_lo = (int)(((long long)P * pr) / C), n_pre = (int)(((long long)P * (pr + 1)) / C) - pre_lo;
  const int suf_lo = (S * pr) / C, n_suf = (S * (pr + 1)) / C - suf_lo;
  // Tiles: mixed ones (the last n_pre % 128 prefix keys, then the suffix keys; at most two tiles, gathered row by row) among
  // the first two, and the full prefix tiles (tensor-map copies).  A single mixed tile comes second, so that only Q stands
  // between the projection and the first logits (as the first tile 2 us later; as the last one, its gather was exposed: +1.5 %
  // on a loop of 16 requests).  Softmax does not care about the order.
  const int n_full = n_pre / KB, rem = n_pre - n_full * KB, n_mix = (rem + n_suf + KB - 1) / KB;
  const int T = n_mix + n_full, m0 = n_mix == 1 && n_full > 0 ? 1 : 0;      // mixed tiles: m0 .. m0 + n_mix - 1
  const int lead_rank = crank & ~1;
  const uint32_t pair_mask = 3u << lead_rank;

  if (warp < 4) {
    // =========================== loaders: warps 0-1 K, 2-3 V =======================================================
    // Buffer t & 1 is free again once the logits of tile t (K), P V of tile t (V) exist: both commits reach both CTAs.
    // (16-byte cp.async for every row, the first form of this loader, took 3 us to issue 64 KB: the requests of a tile did
    // not fit the load / store unit's queue.)
    const bool is_v = warp >= 2;
    const int lt = tid & 63;
    const uint32_t buf0 = is_v ? Vs : Ks, tile_bytes = is_v ? L::VTILE : L::KTILE;
    const uint32_t full_own = smem_u32(is_v ? &v_full[0] : &k_full[0]);
    const uint32_t full0 = map_rank(full_own, lead_rank);
    // ---- full prefix tiles: two tensor-map copies per stream and CTA, counted on the leader's barrier
    auto issue_full = [&](int t) {
      const int row0 = p0 + pre_lo + (t < m0 ? t : t - n_mix) * KB, plane = a.layer * 2 + (is_v ? 1 : 0);
      const uint32_t bar = full_own + (uint32_t)(t & 1) * 8u, dst = buf0 + (uint32_t)(t & 1) * tile_bytes;
      if (half == 0) mbar_expect_tx(bar, 4u * L::PIECE);
      else remote_arrive(full0 + (uint32_t)(t & 1) * 8u);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        // K: my 64 keys, channel halves u; V: key halves u, my channel half
        const int row = row0 + 64 * (is_v ? u : half), blk = hk * (DH / 64) + (is_v ? half : u) * (DH / 128);
        asm volatile(
            "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
                dst + (uint32_t)u * L::PIECE),
            "l"(a.rq->kv_map), "r"(0), "r"(row), "r"(blk), "r"(plane), "r"(bar & LEADER_MASK)
            : "memory");
      }
    };
    // ---- mixed tiles: row by row
    const int chunks = is_v ? DH / 16 : DH / 8, rstep = 64 / chunks;     // 16-byte chunks per row of this stream
    const int lc = lt % chunks, r0 = lt / chunks;
    const int rows = is_v ? KB : 64, key0 = is_v ? 0 : half * 64;        // my rows are keys key0 .. key0 + rows - 1 of a tile
    const uint32_t src_off = (uint32_t)(is_v ? half * DH : 0) + (uint32_t)lc * 16;
    const size_t kv_stride = (size_t)d.Hkv * DH * 2;
    const uint8_t* Gp = reinterpret_cast<const uint8_t*>(r.prefix_kv) +
                        (((size_t)(a.layer * 2 + (is_v ? 1 : 0)) * r.kv_tokens + p0 + pre_lo + n_full * KB) * d.Hkv + hk) * (DH * 2) + src_off;
    const uint8_t* Gs = reinterpret_cast<const uint8_t*>(is_v ? a.vr : a.kr) + ((size_t)(b * d.Hkv + hk) * S + suf_lo) * (DH * 2) + src_off;
    auto dst_of = [&](int t, int row) {
      return buf0 + (uint32_t)(m0 + t) * tile_bytes + (is_v ? (uint32_t)(row >> 6) * L::PIECE : 0u) + (uint32_t)(lc >> 3) * L::KBLOCK +
             (uint32_t)(row & 63) * 128 + (uint32_t)(((lc & 7) ^ (row & 7)) << 4);
    };
    // the prefix rows of the t-th mixed tile, or its suffix rows and, for V, zeros past the range (their probabilities are 0, but
    // 0 x stale shared memory must stay 0; K rows past the range only give logits that the softmax masks)
    auto gather = [&](int t, bool prefix) {
      const int k0 = t * KB + key0;                                      // first key of my rows within the mixed keys
      const int np = max(0, min(rows, rem - k0)), nv = max(0, min(rows, rem + n_suf - k0));
      if (prefix) {
        const uint8_t* src = Gp + (size_t)(k0 + r0) * kv_stride;
#pragma unroll 4
        for (int row = r0; row < np; row += rstep, src += (size_t)rstep * kv_stride) cp_async16(dst_of(t, row), src, 16u);
      } else {
        int row = r0 + (np > r0 ? (np - r0 + rstep - 1) / rstep * rstep : 0);      // my first row >= np
        for (; row < nv; row += rstep) cp_async16(dst_of(t, row), Gs + (size_t)(k0 + row - rem) * (DH * 2), 16u);
        if (is_v)
          for (; row < rows; row += rstep) asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(dst_of(t, row)), "r"(0u) : "memory");
      }
    };
    // Constants of the call, ahead of the dependency wait, in the order of their use (an SM takes in 64 KB per 0.55 us: what
    // is asked for first arrives first).
    // (the map was written into the request block by the kernel at the head of the call)
    if (lt == 0) {
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(a.rq->kv_map) : "memory");
      if (m0 > 0) issue_full(0);
    }
    __syncwarp();
    for (int t = 0; t < n_mix; ++t) gather(t, true);
    if (lt == 0)
      for (int t = m0 + n_mix; t < 2 && t < T; ++t) issue_full(t);
    __syncwarp();
    pdl_wait();
    if (T > 0) {
      for (int t = 0; t < n_mix; ++t) gather(t, false);
      if (n_mix > 0) {
        cp_async_commit();
        cp_async_wait<0>();
        fence_async_smem();                    // generic-proxy writes, read next by the tensor cores
        if (is_v) group_sync<BAR_V, 64>(); else group_sync<BAR_K, 64>();
      }
      if (lt == 0) {
        for (int t = m0; t < m0 + n_mix; ++t) remote_arrive_stores(full0 + (uint32_t)t * 8u);
        for (int t = 2; t < T; ++t) {
          mbar_wait_drain(smem_u32(is_v ? &pv_done[t & 1] : &s_full[t & 1]), (uint32_t)((t - 2) >> 1) & 1u, wc);
          issue_full(t);
        }
      }
      __syncwarp();
    }
    cluster_arrive_relaxed();
  } else if (warp == 4) {
    // =========================== MMA issuer (leader CTA): S(0), S(1), then P(t) V(t), S(t + 2) ======================
    pdl_wait();
    if (lane == 0) {
      trace_stamp(trc, 1), trace_stamp(trc, 2);
      if (half == 1) trace_stamp(trc, 3), trace_stamp(trc, 4), trace_stamp(trc, 5);
    }
    if (half == 0) {
      // operands of tile t; the rows of a mixed tile were stored by threads of both CTAs
      auto wait_tile = [&](const uint64_t* full, int t) {
        mbar_wait_drain(smem_u32(&full[t & 1]), (uint32_t)(t >> 1) & 1u, wc);
        if (t >= m0 && t < m0 + n_mix) pair_acquire(smem_u32(&full[t & 1]), (uint32_t)(t >> 1) & 1u);
      };
      auto issue_s = [&](int t) {
        wait_tile(k_full, t);
        tc_fence_after();
        const uint32_t kb = Ks + (uint32_t)(t & 1) * L::KTILE;
        // (rolled loops: most of the time of a first pass is the fetch of its code, which has left the instruction caches since the
        // last layer: ten-step loops of 4 / 16 requests 8.76 / 11.64 ms unrolled, 8.54 / 11.30 rolled)
        uint64_t da = make_desc(Qs), db = make_desc(kb);
#pragma unroll 1
        for (int c = 0; c < DH / 64; ++c, da += (128 * 128) >> 4, db += L::KBLOCK >> 4) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            if (elect_one()) umma2_bf16(tmem_s + (uint32_t)(t & 1) * KB, da + 2 * kk, db + 2 * kk, IDESC_S, (c > 0 || kk > 0) ? 1u : 0u);
        }
        if (elect_one()) umma2_commit(smem_u32(&s_full[t & 1]), pair_mask);
        __syncwarp();
      };
      if (T > 0) {
        mbar_wait_drain(smem_u32(&q_bar), 0u, wc);        // both CTAs' Q tiles have landed
        issue_s(0);
      }
      if (lane == 0) trace_stamp(trc, 3);
      if (T > 1) issue_s(1);
      for (int t = 0; t < T; ++t) {
        wait_tile(v_full, t);
        const uint32_t vb = Vs + (uint32_t)(t & 1) * L::VTILE;
        // (the first 64 keys' probabilities are ready before the others': their half of the product hides under the rest of
        // the softmax)
#pragma unroll 1
        for (int kh = 0; kh < 2; ++kh) {
          mbar_wait_drain(smem_u32(&p_full[t & 1][kh]), (uint32_t)(t >> 1) & 1u, wc);
          tc_fence_after();
          // A = P of this tile: bf16 pairs in the first 64 columns of its S buffer
          const uint64_t db = make_desc_mn(vb + (uint32_t)kh * L::PIECE, L::KBLOCK, 1024);
          const uint32_t ta = tmem_s + (uint32_t)(t & 1) * KB + (uint32_t)kh * 32;
#pragma unroll
          for (int kj = 0; kj < KB / 32; ++kj)
            if (elect_one()) umma2_ts(tmem_o, ta + (uint32_t)kj * 8, db + (uint64_t)(kj * ((16 * 128) >> 4)), IDESC_PV, (t > 0 || kh > 0 || kj > 0) ? 1u : 0u);
        }
        if (elect_one()) umma2_commit(smem_u32(&pv_done[t & 1]), pair_mask);
        __syncwarp();
        if (t + 2 < T) issue_s(t + 2);
        if (t == 0 && lane == 0) trace_stamp(trc, 4);
      }
      if (lane == 0) trace_stamp(trc, 5);
    }
    __syncwarp();
    cluster_arrive_relaxed();
  } else {
    // =========================== softmax / correction / output =====================================================
    const int g = (warp - 5) >> 2;            // which half of a row's columns
    const int q = warp & 3;
    const int row = q * 32 + lane;            // accumulator row = tensor-memory lane
    const int hl = row >> 6, i = row & 63;
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const bool causal_row = d.block_causal && d.ns && i == 0;
    const uint32_t pfull0 = map_rank(smem_u32(&p_full[0][g]), lead_rank);
    float m = -INFINITY, l = 0.f;             // running maximum (log2 units) and sum (of this thread's half of the columns)
    pdl_wait();
    if (T > 0 && lane == 0) {
      // Q (rotated, scaled) was written by the QKV projection as this CTA's operand tile: an eighth per warp (the copies of
      // one warp complete one after the other), both CTAs' counted on the leader's barrier (with own
      // barriers and a relay ten-step loops of 2 / 8 / 16 requests 7.61 / 9.45 / 11.14 ms, so 7.57 / 9.42 / 11.06)
      const uint32_t bar = smem_u32(&q_bar);
      if (half == 0 && warp == 5) mbar_expect_tx(bar, 2u * L::QTILE);
      tma2d(Qs + (uint32_t)(warp - 5) * (L::QTILE / 8), &tmq, (b * (d.Hq >> 1) + (head0 >> 1)) * (DH * 2) + (warp - 5) * (DH / 4), bar & LEADER_MASK);
    }
    __syncwarp();
    const bool skip = status_set(a.status);
    // Turn -1 is a rehearsal, without effect, in the 3 - 4 us until the first logits exist: in a captured loop a kernel's code
    // has left the instruction caches by the next layer, and the first softmax took 3.4 us instead of 1.7.
    for (int t = T > 0 ? -1 : 0; t < T; ++t) {
      const uint32_t sb = tmem_s + (uint32_t)(t & 1) * KB + lane_addr;
      // the visible keys of a row form a prefix of a mixed tile: the keys that exist, and for the state-token row under the
      // block-causal mask the prefix keys and its own key (suffix key 0, in the first range)
      const int nvis = t >= m0 && t < m0 + n_mix ? min(KB, (causal_row ? rem + (suf_lo == 0 && n_suf > 0 ? 1 : 0) : rem + n_suf) - (t - m0) * KB) : KB;
      const uint64_t vis = first_columns(nvis - g * 64);
      if (t >= 0) {
        if (lane == 0) mbar_wait_drain(smem_u32(&s_full[t & 1]), (uint32_t)(t >> 1) & 1u, wc);
        __syncwarp();
      }
      tc_fence_after();
      if (t >= 0 && t == T - 1) cluster_arrive_relaxed();     // (the last logits exist: Q is dead, its area may receive partials)
      pair_softmax_tile<DH>(m, l, xch[t & 1], sb, tmem_o + lane_addr, g, q, row, vis, t >= 0, [&] {
        if (lane == 0) mbar_wait_drain(smem_u32(&pv_done[(t - 1) & 1]), (uint32_t)((t - 1) >> 1) & 1u, wc);
      });
      if (t >= 0 && lane == 0) remote_arrive(pfull0 + (uint32_t)(t & 1) * 16u);
    }
    if (T == 0) cluster_arrive_relaxed();
    xch[T & 1][g][row] = l;
    quarter_sync(q);
    l = xch[T & 1][0][row] + xch[T & 1][1][row];
    if (T > 0 && warp == 5) mbar_wait_drain(smem_u32(&pv_done[(T - 1) & 1]), (uint32_t)((T - 1) >> 1) & 1u, wc);
    group_sync<BAR_ROWS, 256>();
    tc_fence_after();
    if (warp == 5 && lane == 0) trace_stamp(trc, 6);
    // ---- partial out: half an O row into the owner's block of the staging area; half 0 adds (max, sum) ----------------
    const int c = i / own, il = i - c * own, n_c = max(0, min(own, S - c * own));
    const bool wr = i < S;
    const uint32_t blk = stg + (uint32_t)c * slot;
    constexpr int PARTS = 8 / (C - 1);       // warps per peer: the bulk copies of one warp complete one after the other
    const int w8 = warp - 5, pi = w8 % (C - 1), peer = pi < pr ? pi : pi + 1, part = w8 / (C - 1);
    const int n_p = max(0, min(own, S - peer * own));
#pragma unroll 1
    for (int k = 0; k < L::NP; ++k) {
      float o[64];
      if (T > 0) {
        tmem_ld64(tmem_o + lane_addr + (uint32_t)(g * (DH / 2) + k * 64), o);
      } else {
#pragma unroll
        for (int e = 0; e < 64; ++e) o[e] = 0.f;
      }
      const uint32_t rowp = blk + (uint32_t)((k * 2 * n_c + hl * n_c + il) * L::PITCH + g * 256);
      if (wr) {
#pragma unroll
        for (int e = 0; e < 64; e += 4)
          asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(rowp + (uint32_t)e * 4), "f"(o[e]), "f"(o[e + 1]), "f"(o[e + 2]), "f"(o[e + 3])
                       : "memory");
        if (k == 0 && g == 0)
          asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(blk + (uint32_t)(L::NP * 2 * n_c * L::PITCH + (hl * n_c + il) * 16)), "f"(m), "f"(l)
                       : "memory");
      }
      fence_async_smem();                    // generic writes -> visible to the bulk-copy engine
      group_sync<BAR_ROWS, 256>();
      if (k == 0) cluster_wait();            // every CTA's Q is dead
      if (lane == 0 && part < PARTS && n_p > 0) {
        const uint32_t bytes = (uint32_t)(2 * n_p * (L::PITCH + (k == L::NP - 1 ? 16 : 0))), chunk = (bytes / PARTS + 15) & ~15u;
        const uint32_t lo = (uint32_t)part * chunk, off = (uint32_t)(k * 2 * n_p * L::PITCH) + lo;
        if (lo < bytes)
          asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                           map_rank(recv + (uint32_t)(pr < peer ? pr : pr - 1) * slot + off, peer * 2 + half)),
                       "r"(stg + (uint32_t)peer * slot + off), "r"(min(chunk, bytes - lo)), "r"(map_rank(smem_u32(&mrg_bar), peer * 2 + half))
                       : "memory");
      }
      __syncwarp();
    }
    if (warp == 5) {
      bool ok = true;
      if (n_me > 0) ok = mbar_wait_drain(smem_u32(&mrg_bar), 0u, wc) > 0;
      if (lane == 0) mrg_ok = ok && !skip ? 1 : 0;
    }
    tc_fence_before();
  }
  if (warp < 5) cluster_wait();
  __syncthreads();
  // From here on this CTA no longer needs its peers; it may leave once every peer says the same (the leader's MMAs have
  // read both CTAs' shared memory, every partial copied out of its staging area has landed).
  cluster_arrive_relaxed();
  {
    // ---- merge my rows: the C partials in range order, normalise, store as the output projection's operand ------------
    // A warp per row (rr = hl * n_me + il, every 13th), lane l the four columns of every piece that its l-th 16 bytes hold;
    // before that the weights of the warp's rows, a row per lane.
    constexpr int NW = AP_THREADS / 32;
    static_assert((2 * L::OWN + NW - 1) / NW <= 32, "more rows per warp than lanes");
    const bool store = !*reinterpret_cast<volatile int*>(&abort_flag) && *reinterpret_cast<volatile int*>(&mrg_ok);
    uint32_t blk[C];
    float w[C], ls[C], mm = -INFINITY, ll = 0.f;
    const int my = min(warp + NW * lane, max(0, 2 * n_me - 1));
#pragma unroll
    for (int s = 0; s < C; ++s) {
      blk[s] = s == pr ? stg + (uint32_t)pr * slot : recv + (uint32_t)(s < pr ? s : s - 1) * slot;
      asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(w[s]), "=f"(ls[s]) : "r"(blk[s] + (uint32_t)(L::NP * 2 * n_me * L::PITCH + my * 16)) : "memory");
      mm = fmaxf(mm, w[s]);
    }
#pragma unroll
    for (int s = 0; s < C; ++s) {
      w[s] = w[s] == -INFINITY ? 0.f : exp2f(w[s] - mm);
      ll = fmaf(w[s], ls[s], ll);
    }
    const float inv = 1.0f / ll;
#pragma unroll
    for (int s = 0; s < C; ++s) w[s] *= inv, blk[s] += (uint32_t)(warp * L::PITCH + lane * 16);
    const int col = head0 * DH + (lane >> 4) * (DH / 2) + (lane & 15) * 4;
    const bool tiled = a.rows_pad > 0;
    const size_t kc = (size_t)(tiled ? a.rows_pad : 1) * 64;             // elements from one 64-column chunk to the next
    __nv_bfloat16* const o0 = a.out + (tiled ? (size_t)(col >> 6) * kc + (col & 7) : (size_t)col);
#pragma unroll 1
    for (int j = 0, rr = warp; rr < 2 * n_me; ++j, rr += NW) {
      const int hl = rr >= n_me ? 1 : 0, orow = b * S + own_lo + rr - hl * n_me;
      float acc[L::NP][4] = {};
#pragma unroll
      for (int s = 0; s < C; ++s) {
        const float ws = __shfl_sync(0xffffffffu, w[s], j);
#pragma unroll
        for (int k = 0; k < L::NP; ++k) {
          float x[4];
          asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
                       : "r"(blk[s] + (uint32_t)((k * 2 * n_me + j * NW) * L::PITCH)) : "memory");
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[k][e] = fmaf(ws, x[e], acc[k][e]);
        }
      }
      __nv_bfloat16* const o = o0 + (tiled ? (size_t)orow * 64 + ((((col & 63) >> 3) ^ (orow & 7)) << 3) : (size_t)orow * d.Nq) + hl * (DH / 64) * kc;
      if (store) {
#pragma unroll
        for (int k = 0; k < L::NP; ++k) *reinterpret_cast<uint2*>(o + k * kc) = make_uint2(pack_bf16(acc[k][0], acc[k][1]), pack_bf16(acc[k][2], acc[k][3]));
      }
    }
  }
  cluster_wait();
  if (warp == 4) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, 512);
    if (lane == 0 && trc) {
      unsigned long long t;
      unsigned sm;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");
      asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
      trc[8] = t, trc[7] = sm, trc[9] = (unsigned long long)T, trc[10] = 1;   // ([10]: marks an attention slot)
    }
  }
}

template <int DH, int C>
cudaError_t setup_one() {
  static PerDeviceOnce once;
  if (!once.needed()) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_attn_pair<DH, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ApLayout<DH, C>::SMEM);
  if (e == cudaSuccess) once.done();
  return e;
}
// clusters of this kernel that are resident at a time (0 on an error)
template <int DH, int C>
int max_clusters_one() {
  if (setup_one<DH, C>() != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * C, 1, 64), cfg.blockDim = dim3(AP_THREADS), cfg.dynamicSmemBytes = ApLayout<DH, C>::SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2 * C, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
  cfg.attrs = at, cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, k_attn_pair<DH, C>, &cfg) == cudaSuccess ? n : 0;
}
int max_clusters(int dh, int c) {
  if (dh == 256) return c == 2 ? max_clusters_one<256, 2>() : c == 3 ? max_clusters_one<256, 3>() : max_clusters_one<256, 4>();
  return c == 2 ? max_clusters_one<128, 2>() : c == 3 ? max_clusters_one<128, 3>() : max_clusters_one<128, 4>();
}

template <int DH, int C>
cudaError_t launch_one(const AttnArgs& a, int batch, cudaStream_t st, bool pdl) {
  cudaError_t e = setup_one<DH, C>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * C, a.d.Hq / 4, batch), cfg.blockDim = dim3(AP_THREADS), cfg.dynamicSmemBytes = ApLayout<DH, C>::SMEM, cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2 * C, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at, cfg.numAttrs = pdl ? 2 : 1;
  CUtensorMap tq;      // q tiles: rows of 64 channels, an eighth of a CTA's tile at a time
  if (!row_map(&tq, a.qr, (uint64_t)batch * (a.d.Hq / 2) * (DH * 2), DH / 4)) return cudaErrorInvalidValue;
  return cudaLaunchKernelEx(&cfg, k_attn_pair<DH, C>, a, tq);
}

}  // namespace

// Tensor map over a prefix cache [planes][tokens][Hkv * dh / 64 blocks][64]: copies of 64 tokens x dh / 128 blocks (64-channel
// blocks of 128-byte rows, 128-byte swizzle: the operand layout of the MMAs).
bool prefix_kv_map(unsigned char* map, const void* kv, uint64_t kv_tokens, const Dims& d) {
  const EncodeTiled enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t row = (cuuint64_t)d.Hkv * d.dh * 2;
  const cuuint64_t dims[4] = {64, kv_tokens, (cuuint64_t)(d.Hkv * d.dh / 64), (cuuint64_t)(2 * d.L)}, strides[3] = {row, 128, kv_tokens * row};
  const cuuint32_t box[4] = {64, 64, (cuuint32_t)(d.dh / 128), 1}, es[4] = {1, 1, 1, 1};
  return enc(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(kv), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool attention_pair_supported(const Dims& d) {
  return (d.dh == 256 || d.dh == 128) && d.S <= 64 && d.Hq % 4 == 0 && (d.Hq / d.Hkv) % 4 == 0;
}

// (most ranges whose fp32 partials fit the shared memory)
int attention_pair_max_ranges(const Dims& d) {
  return d.dh != 256 || d.S <= ApLayout<256, 4>::S_MAX ? 4 : (d.S <= ApLayout<256, 3>::S_MAX ? 3 : 2);
}

// clusters of `ranges` pairs that are resident at a time; <= 0: none
int attention_pair_resident(const Dims& d, int ranges) {
  static PerDeviceCount resident[2][MAX_PAIR_RANGES + 1];
  if (ranges == 1) return attention_persist_pairs(d);
  return resident[d.dh == 256 ? 1 : 0][ranges].get([&] { return max_clusters(d.dh, ranges); });
}

// Key ranges per request (see choose_pair_ranges), 0 if no kernel on pairs can run.  A cluster of 8 CTAs needs 8 free SMs in one
// GPC: 15 on a B200, not 18.  One range: the persistent kernel.  Against every other choice, ten-step loops of 4 / 8 / 12 / 16 / 20
// requests: chosen 8.35 / 9.47 / 10.51 / 11.18 / 12.40 ms with 816-token prefixes (best 8.33 / 9.47 / 10.51 / 11.13 / 12.40), 8.19 /
// 8.89 / 9.90 / 10.55 / 11.72 with 400 (best 8.01, two ranges instead of four / 8.89 / 9.90 / 10.52 / 11.72).
int attention_pair_ranges(const Dims& d, int batch, int max_prefix) {
  int resident[MAX_PAIR_RANGES + 1] = {};
  for (int c = 1; c <= MAX_PAIR_RANGES; ++c) resident[c] = attention_pair_resident(d, c);
  return choose_pair_ranges(resident, batch * (d.Hq / 4), max_prefix + d.S, attention_pair_max_ranges(d));
}

cudaError_t launch_attention_pair(const Request* rq, int* status, const __nv_bfloat16* q_tiles, const __nv_bfloat16* kr,
                                  const __nv_bfloat16* vr, int layer, __nv_bfloat16* out_tiled, int rows_pad, const Dims& d, int batch,
                                  int ranges, const int* order, unsigned wait_limit, cudaStream_t st, unsigned long long* trace, bool pdl) {
  if (ranges > attention_pair_max_ranges(d)) return cudaErrorInvalidValue;
  if (ranges == 1) return launch_attention_persist(rq, status, q_tiles, kr, vr, layer, out_tiled, rows_pad, d, batch, order, wait_limit, st, trace, pdl);
  AttnArgs a{};
  a.rq = rq, a.status = status, a.qr = q_tiles, a.kr = kr, a.vr = vr, a.layer = layer, a.out = out_tiled, a.rows_pad = rows_pad;
  a.num_splits = ranges, a.d = d, a.wait_limit = wait_limit, a.order = order, a.trace = trace;
  switch (ranges + (d.dh == 256 ? 4 : 0)) {
    case 2: return launch_one<128, 2>(a, batch, st, pdl);
    case 3: return launch_one<128, 3>(a, batch, st, pdl);
    case 4: return launch_one<128, 4>(a, batch, st, pdl);
    case 6: return launch_one<256, 2>(a, batch, st, pdl);
    case 7: return launch_one<256, 3>(a, batch, st, pdl);
    default: return launch_one<256, 4>(a, batch, st, pdl);
  }
}

}  // namespace phyai
