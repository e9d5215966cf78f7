// Suffix -> (prefix U suffix) attention of many requests: a persistent grid of CTA pairs (tcgen05 cta_group::2).
//
// A pair of SMs takes four query heads of one request that share a kv head (each CTA two of them: 2 x 64 padded rows = its 128
// rows of the 256-row MMAs) over all its keys, as in attention_pair.cu, and then goes on to its next item without leaving the
// pipeline: keys, values and queries of the next item are on their way, its first logits are computed and go through the softmax
// while the accumulator of the last one is still being read out.  Items (request, head group) come longest first and are dealt to
// the pairs back and forth, so that a pair with a long one gets a short one next.
//   S = Q K^T   M = 256, N = 128 keys, K = head_dim; Q (the QKV projection wrote it as this kernel's operand tile) and K in
//               shared memory; two S buffers in tensor memory
//   softmax     two threads per row (half of the columns each), straight from tensor memory; P (bf16) over the S buffer
//   O += P V    M = 256, N = head_dim, K = 128 keys; P is the tensor-memory A operand, V an MN-major B operand
// A tile is two blocks of 64 keys.  The blocks of an item are its prefix (the last one possibly in part) and, at the end, the
// request's own keys; all come by tensor-map copies.  K: block h of a tile belongs to CTA h of the pair (the tensor cores read the
// other half of the tile from the peer); V: each CTA fetches its half of the channels of both blocks.  No row past the end of a
// prefix is read: a partial last block is the 64 rows that end there, behind keys of the block before (or, of a prefix of fewer than
// 64 keys, behind what lies before it): those rows' logits are masked, their values overwritten with zeros (0 x infinity, 0 x NaN).
//
// What bounds it is the tensor pipe (2048 clocks per tile of 128 keys) and, close behind, the chain logits -> softmax (MUFU: 1024
// clocks) -> P V, which the second S buffer overlaps with the other products.
// The other bound is code: a kernel's instructions have left the caches by the next layer, about 11 clocks for each on its first
// pass.  Rolled loops for the MMAs and the output, and a rehearsal of the softmax and output code before the dependency wait.
//
// Measured in ten-step loops with 816-token prefixes, against one CTA per pair of heads (attention_tc.cu: 64-key tiles, logits at
// N = 64, K and V read by every CTA): 20 requests 13.24 -> 12.52 ms, 32: 17.49 -> 16.82, 64: 30.0 -> 28.3, 128: 57.5 -> 53.3 (power
// capped, 1.65 and 1.53 GHz); attention of 64 ragged requests 39 -> 26 us a layer.  The same with unrolled MMA and output loops
// 64: 28.8; with two groups of four softmax warps that take a tile each (less exposed, but twice the code) 30.7.
// Warps of a CTA: 0 fetches K, 1 V, 2 Q, 3 issues the MMAs (leader CTA), 4-11 softmax, correction, output.  Every wait is
// bounded; after a give-up the protocol runs to its end and only the global stores are skipped.
#include "attention.cuh"
#include "attention_choice.h"
#include "tc.cuh"
#include "tc_pair.cuh"

namespace phyai {
namespace {

constexpr int KB = PAIR_TILE;                 // keys per tile: two blocks of 64
constexpr int AS_THREADS = 12 * 32;

template <int DH>
struct AsLayout {
  static constexpr int KBLOCK = 64 * 128;                    // 64 channels of 64 keys
  static constexpr int PIECE = (DH / 128) * KBLOCK;          // one copy: 64 keys x DH / 2 channels
  static constexpr int TILE = 2 * PIECE;                     // K: this CTA's block, both channel halves; V: both blocks, its channel half
  static constexpr int QTILE = 128 * DH * 2;
  static constexpr int STG = 2048;                           // output staging of a warp: 32 rows x 32 columns
  static constexpr size_t SMEM = 1024 + 4 * (size_t)TILE + QTILE + 8 * STG;
};

__device__ __forceinline__ void kv_copy(uint32_t dst, const void* map, int row, int blk, int plane, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(map), "r"(0), "r"(row), "r"(blk), "r"(plane), "r"(bar)
      : "memory");
}

struct Item {
  int b, group;        // request, group of four query heads
  int p0, P;           // prefix rows of the cache
  int nsp, T;          // blocks of 64 prefix keys; tiles (one more block: the request's own keys)
};

template <int DH>
__global__ void __launch_bounds__(AS_THREADS, 1) __cluster_dims__(2, 1, 1)
    k_attn_persist(const AttnArgs a, const int n_items, const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                   const __grid_constant__ CUtensorMap tmv) {
  using L = AsLayout<DH>;
  constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(KB >> 3) << 17) | ((256u >> 4) << 24);
  constexpr uint32_t IDESC_PV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((256u >> 4) << 24);

  extern __shared__ uint8_t smem_raw[];
  // leader: operands of a buffer complete in both CTAs, P of a buffer (by column half) complete in both, Q complete in both,
  // accumulator read out in both.  Each CTA: logits / P V complete, all logits of an item complete; own V
  // blocks that are cleared in part.  (A wait on a parity must never be more than one phase ahead: hence q_free beside s_full.)
  __shared__ __align__(8) uint64_t k_full[2], v_full[2], p_full[2][2], q_full, o_free, s_full[2], pv_done[2], q_free, v_own;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  // what the two half-row threads of a row exchange: maximum (by tile parity), sum of an item (by item parity: after a last item of one
  // tile two outputs follow one another with no barrier between the reading of one's sums and the writing of the other's)
  __shared__ float xch[2][2][128], xsum[2][2][128];

  const Dims& d = a.d;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int half = blockIdx.x & 1, pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1, groups = d.Hq >> 2;
  const int S = d.S;
  unsigned long long* const trc = a.trace ? a.trace + (size_t)blockIdx.x * 16 : nullptr;
  if (tid == 0) trace_stamp(trc, 0);
  pdl_launch_dependents();
  if (tid == 32) prefetch_tmap(&tmk), prefetch_tmap(&tmv), prefetch_tmap(&tmq);

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t Ks = base, Vs = base + 2 * L::TILE, Qs = base + 4 * L::TILE;
  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&k_full[i]), 1), mbar_init(smem_u32(&v_full[i]), 2), mbar_init(smem_u32(&p_full[i][0]), 8), mbar_init(smem_u32(&p_full[i][1]), 8);
      mbar_init(smem_u32(&s_full[i]), 1), mbar_init(smem_u32(&pv_done[i]), 1);
    }
    mbar_init(smem_u32(&q_full), 1), mbar_init(smem_u32(&o_free), 16), mbar_init(smem_u32(&q_free), 1), mbar_init(smem_u32(&v_own), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 3) {
    tmem_alloc2(smem_u32(&tmem_slot), 512);
    tc_fence_before();
  }
  __syncthreads();
  pair_sync();                                      // both CTAs' barriers exist before the peer can signal them
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(&tmem_slot), 0);
  const uint32_t tmem_s = tmem_base, tmem_o = tmem_base + 2 * KB;
  const WaitCtx wc{a.status, &abort_flag, a.wait_limit}, wl{a.status, &abort_flag, a.wait_limit, true};

  // Items of this pair: of every round of n_pairs items one, rounds dealt back and forth.  (The request block is written before
  // the captured loop starts: safe to read ahead of the dependency wait.  A call whose lengths are invalid stores nothing; the
  // clamps keep its loads inside the cache.)
  const int kvt = (int)a.rq->kv_tokens;
  const int* const cu = a.rq->cu_lens;
  auto index_of = [&](int k) { return k * n_pairs + ((k & 1) ? n_pairs - 1 - pair : pair); };
  const int rounds = n_items / n_pairs, n_my = rounds + (index_of(rounds) < n_items ? 1 : 0);
  auto item = [&](int k) {
    Item it;
    const int j = index_of(min(k, n_my - 1)), pos = j / groups;
    it.b = a.order ? a.order[pos] : pos, it.group = j - pos * groups;
    it.p0 = min(max(cu[it.b], 0), kvt), it.P = min(max(cu[it.b + 1] - it.p0, 0), kvt - it.p0);
    it.nsp = (it.P + 63) >> 6, it.T = (it.nsp + 2) >> 1;
    return it;
  };

  if (warp == 0) {
    // =========================== K: a buffer is free again once the logits of the tile two before exist ==================
    if (lane == 0) {
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(a.rq->kv_map) : "memory");
      bool waited = false;
      Item it = item(0);
      for (int k = 0, n = 0; k < n_my; ++k) {
        const Item nx = item(k + 1);
        const int hk = it.group * 4 / (d.Hq / d.Hkv);
        for (int t = 0; t < it.T; ++t, ++n) {
          // (these products need what the kernel before writes: its time is not to count against the limit of the wait)
          if (n >= 2 && !waited) pdl_wait(), waited = true;
          if (n >= 2) mbar_wait_drain(smem_u32(&s_full[n & 1]), (uint32_t)((n - 2) >> 1) & 1u, wl);
          const int sb = 2 * t + half;
          const uint32_t bar = smem_u32(&k_full[n & 1]), dst = Ks + (uint32_t)(n & 1) * L::TILE;
          if (half == 0) mbar_expect_tx(bar, (uint32_t)L::TILE * (2 * t + 1 <= it.nsp ? 2 : 1));
          if (sb > it.nsp) continue;
          const bool own = sb == it.nsp;
          if (own && !waited) pdl_wait(), waited = true;
          const void* map = own ? (const void*)&tmk : (const void*)a.rq->kv_map;
#pragma unroll
          for (int u = 0; u < 2; ++u)
            kv_copy(dst + (uint32_t)u * L::PIECE, map, own ? 0 : it.p0 + prefix_block(it.P, sb).row, (own ? 0 : hk * (DH / 64)) + u * (DH / 128),
                    own ? it.b * d.Hkv + hk : a.layer * 2, bar & LEADER_MASK);
        }
        it = nx;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // =========================== V: a buffer is free again once P V of the tile two before has completed ==================
    if (lane == 0) asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(a.rq->kv_map) : "memory");
    const uint32_t full_lead = map_rank(smem_u32(&v_full[0]), 0);
    bool waited = false;
    uint32_t ph_own = 0;
    Item it = item(0);
    for (int k = 0, n = 0; k < n_my; ++k) {
      const Item nx = item(k + 1);
      const int hk = it.group * 4 / (d.Hq / d.Hkv), rem = it.P & 63;
      for (int t = 0; t < it.T; ++t, ++n) {
        const int nb = min(2, it.nsp + 1 - 2 * t);                       // blocks of this tile
        const int part = rem ? it.nsp - 1 - 2 * t : -1;                  // its block that is not full, if 0 or 1
        const bool clear = part == 0 || part == 1;
        const uint32_t dst = Vs + (uint32_t)(n & 1) * L::TILE;
        if (lane == 0) {
          if (n >= 2 && !waited) pdl_wait(), waited = true;
          if (n >= 2) mbar_wait_drain(smem_u32(&pv_done[n & 1]), (uint32_t)((n - 2) >> 1) & 1u, wl);
          uint32_t bar = smem_u32(&v_full[n & 1]);
          if (clear) {
            bar = smem_u32(&v_own);
            mbar_expect_tx(bar, (uint32_t)(nb * L::PIECE));
          } else {
            if (half == 0) mbar_expect_tx(bar, (uint32_t)(2 * nb * L::PIECE));
            else remote_arrive(full_lead + (uint32_t)(n & 1) * 8u);
            bar &= LEADER_MASK;
          }
          for (int u = 0; u < nb; ++u) {
            const int sb = 2 * t + u;
            const bool own = sb == it.nsp;
            if (own && !waited) pdl_wait(), waited = true;
            kv_copy(dst + (uint32_t)u * L::PIECE, own ? (const void*)&tmv : (const void*)a.rq->kv_map, own ? 0 : it.p0 + prefix_block(it.P, sb).row,
                    (own ? 0 : hk * (DH / 64)) + half * (DH / 128), own ? it.b * d.Hkv + hk : a.layer * 2 + 1, bar);
          }
          if (clear) mbar_wait_drain(bar, ph_own, wl);
        }
        __syncwarp();
        if (clear) {
          ph_own ^= 1u;
          const uint32_t z = dst + (uint32_t)part * L::PIECE;
          for (int i = lane; i < (64 - rem) * (DH / 16); i += 32) {      // (a row: 8 x 16 bytes in each of DH / 128 blocks)
            const int row = i / (DH / 16), c = i % (DH / 16);
            asm volatile("st.shared.v4.b32 [%0], {%1,%1,%1,%1};" ::"r"(z + (uint32_t)((c >> 3) * L::KBLOCK + row * 128 + (c & 7) * 16)), "r"(0u) : "memory");
          }
          fence_async_smem();                    // generic-proxy writes, read next by the tensor cores
          __syncwarp();
          if (lane == 0) remote_arrive_stores(full_lead + (uint32_t)(n & 1) * 8u);
        }
      }
      it = nx;
    }
  } else if (warp == 2) {
    // =========================== Q: its tile is free again once the last logits of the item before exist ==================
    if (lane == 0) {
      pdl_wait();
      Item it = item(0);
      for (int k = 0; k < n_my; ++k) {
        const Item nx = item(k + 1);
        if (k > 0) mbar_wait_drain(smem_u32(&q_free), (uint32_t)(k - 1) & 1u, wl);
        const uint32_t bar = smem_u32(&q_full);
        if (half == 0) mbar_expect_tx(bar, 2 * L::QTILE);
        const int row = (it.b * (d.Hq >> 1) + it.group * 2 + half) * (DH / 64) * 128;
#pragma unroll
        for (int u = 0; u < DH / 64; ++u) tma2d(Qs + (uint32_t)u * (128 * 128), &tmq, row + u * 128, bar & LEADER_MASK);
        it = nx;
      }
    }
    __syncwarp();
  } else if (warp == 3) {
    // =========================== MMA issuer (leader CTA): S(0), S(1), then P(n) V(n), S(n + 2), across the items ==========
    if (lane == 0) {
      pdl_wait();
      trace_stamp(trc, 1);
      if (half == 1) trace_stamp(trc, 2), trace_stamp(trc, 3), trace_stamp(trc, 4), trace_stamp(trc, 5);
    }
    __syncwarp();
    if (half == 0) {
      // S(n) may be issued once P V of tile n - 2 has been (its S buffer holds P of that tile).  Of the next logits and the next
      // P V whichever has its operands goes first; logits when both have.
      int ns = 0, ks = 0, ts = 0, Ts = item(0).T, Tn = item(1).T;       // next logits: tile of the call, item, tile of the item
      int np = 0, kp = 0, tp = 0;                                       // next P V
      Item it = item(0), nx = item(1);
      uint32_t spins = 0;
      while (kp < n_my) {
        const bool s_next = ks < n_my && ns < np + 2;
        if (s_next) {
          bool go = mbar_test(smem_u32(&k_full[ns & 1]), (uint32_t)(ns >> 1) & 1u) && (ts > 0 || mbar_test(smem_u32(&q_full), (uint32_t)ks & 1u));
          if (spins >= a.wait_limit) {             // given up: the protocol goes on in a fixed order
            mbar_wait_drain(smem_u32(&k_full[ns & 1]), (uint32_t)(ns >> 1) & 1u, wc);
            if (ts == 0) mbar_wait_drain(smem_u32(&q_full), (uint32_t)ks & 1u, wc);
            go = true;
          }
          if (__all_sync(0xffffffffu, go)) {
            if (ns == 0 && lane == 0) trace_stamp(trc, 2);
            tc_fence_after();
            const uint32_t kb = Ks + (uint32_t)(ns & 1) * L::TILE;
            uint64_t da = make_desc(Qs), db = make_desc(kb);      // (a 64-channel block further: 128 x 128 and 64 x 128 bytes)
#pragma unroll 1
            for (int c = 0; c < DH / 64; ++c, da += (128 * 128) >> 4, db += L::KBLOCK >> 4) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                if (elect_one()) umma2_bf16(tmem_s + (uint32_t)(ns & 1) * KB, da + 2 * kk, db + 2 * kk, IDESC_S, (c > 0 || kk > 0) ? 1u : 0u);
            }
            if (elect_one()) umma2_commit(smem_u32(&s_full[ns & 1]));
            if (ts + 1 == Ts && elect_one()) umma2_commit(smem_u32(&q_free));
            __syncwarp();
            if (ns == 0 && lane == 0) trace_stamp(trc, 3);
            ++ns;
            if (++ts == Ts) ts = 0, ++ks, Ts = Tn, Tn = item(ks + 1).T;
            if (spins < a.wait_limit) spins = 0;
            continue;
          }
        }
        if (np < ns) {
          const uint32_t pf = smem_u32(&p_full[np & 1][0]), par = (uint32_t)(np >> 1) & 1u;
          bool go = mbar_test(smem_u32(&v_full[np & 1]), par) && mbar_test(pf, par) && (tp > 0 || kp == 0 || mbar_test(smem_u32(&o_free), (uint32_t)(kp - 1) & 1u));
          if (spins >= a.wait_limit) {
            mbar_wait_drain(smem_u32(&v_full[np & 1]), par, wc);
            mbar_wait_drain(pf, par, wc);
            if (tp == 0 && kp > 0) mbar_wait_drain(smem_u32(&o_free), (uint32_t)(kp - 1) & 1u, wc);
            go = true;
          }
          if (__all_sync(0xffffffffu, go)) {
            // (the tile with the block that is not full: rows of it were cleared by a warp of each CTA)
            if ((it.P & 63) && tp == (it.nsp - 1) >> 1) pair_acquire(smem_u32(&v_full[np & 1]), par);
            const uint32_t vb = Vs + (uint32_t)(np & 1) * L::TILE;
#pragma unroll 1
            for (int kh = 0; kh < 2; ++kh) {
              if (kh == 1) mbar_wait_drain(pf + 8u, par, wc);
              tc_fence_after();
              if (2 * tp + kh > it.nsp) continue;              // (a tile of one block)
              // A = P of this tile: bf16 pairs in the first 64 columns of its S buffer
              const uint64_t db = make_desc_mn(vb + (uint32_t)kh * L::PIECE, L::KBLOCK, 1024);
              const uint32_t tp_ = tmem_s + (uint32_t)(np & 1) * KB + (uint32_t)kh * 32;
#pragma unroll
              for (int kj = 0; kj < KB / 32; ++kj)
                if (elect_one()) umma2_ts(tmem_o, tp_ + (uint32_t)kj * 8, db + kj * ((16 * 128) >> 4), IDESC_PV, (tp > 0 || kh > 0 || kj > 0) ? 1u : 0u);
            }
            if (elect_one()) umma2_commit(smem_u32(&pv_done[np & 1]));
            __syncwarp();
            if (np == 0 && lane == 0) trace_stamp(trc, 4);
            ++np;
            if (++tp == it.T) tp = 0, ++kp, it = nx, nx = item(kp + 1);
            if (spins < a.wait_limit) spins = 0;
            continue;
          }
        }
        ++spins;
      }
      if (lane == 0) trace_stamp(trc, 5);
    }
    __syncwarp();
  } else {
    // =========================== softmax / correction / output ==============================================================
    const int g = (warp - 4) >> 2;            // which half of a row's columns: block g of a tile
    const int q = warp & 3;
    const int row = q * 32 + lane;            // accumulator row = tensor-memory lane
    const int hl = row >> 6, i = row & 63;
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const bool causal_row = d.block_causal && d.ns && i == 0;
    const uint32_t pfull0 = map_rank(smem_u32(&p_full[0][g]), 0), ofree0 = map_rank(smem_u32(&o_free), 0);
    const int i0 = (q * 32) & 63;
    const uint32_t ostage = Qs + L::QTILE + (uint32_t)(warp - 4) * L::STG;
    float m = -INFINITY, l = 0.f, l_prev = 0.f;             // running maximum (log2 units) and sum (of this thread's columns)
    bool skip = true;
    Item it = item(0), nx = item(1);
    int orow0 = 0, ocol0 = 0;                               // of the item before: first row and column of this warp's output
    // The first turn is a rehearsal without effect, while the first operands are on their way (see attention_pair.cu).
    bool rehearsal = true;
    for (int k = 0, t = 0, n = 0;;) {
      if (k < n_my) {
        const uint32_t sb = tmem_s + (uint32_t)(n & 1) * KB + lane_addr;
        // the visible keys of a block: its own of the prefix's; of the request's own keys the state-token row under the block-causal
        // mask sees only the first
        const int blk = 2 * t + g;
        const uint64_t vis = blk < it.nsp ? prefix_block(it.P, blk).keys : blk == it.nsp ? first_columns(causal_row ? 1 : S) : 0;
        if (!rehearsal) {
          if (lane == 0) mbar_wait_drain(smem_u32(&s_full[n & 1]), (uint32_t)(n >> 1) & 1u, wc);
          __syncwarp();
        }
        tc_fence_after();
        pair_softmax_tile<DH>(m, l, xch[n & 1], sb, tmem_o + lane_addr, g, q, row, vis, !rehearsal, [&] {
          if (lane == 0) mbar_wait_drain(smem_u32(&pv_done[(n - 1) & 1]), (uint32_t)((n - 1) >> 1) & 1u, wc);
        });
        if (!rehearsal && lane == 0) remote_arrive(pfull0 + (uint32_t)(n & 1) * 16u);
      }
      if ((t == 0 && k > 0) || rehearsal) {
        // ---- the item before: O / l -> bf16, 32 columns at a time through a staging block of the warp, out with coalesced stores
        // (tiled: the chunk's place as staged; row-major, for the operator: the swizzle undone)
        xsum[k & 1][g][row] = l_prev;
        quarter_sync(q);
        const float inv = 1.0f / (xsum[k & 1][0][row] + xsum[k & 1][1][row]);
        if (lane == 0 && !rehearsal) mbar_wait_drain(smem_u32(&pv_done[(n - 1) & 1]), (uint32_t)((n - 1) >> 1) & 1u, wc);
        __syncwarp();
        tc_fence_after();
        if (k == n_my && warp == 4 && lane == 0) trace_stamp(trc, 6);
        const bool okf = !skip && !*reinterpret_cast<volatile int*>(&abort_flag);
        const int nrow = okf ? max(0, min(32, S - i0)) : 0;
        const uint32_t rowp = ostage + (uint32_t)lane * 64u;
        // (a rolled loop: most of its time is the fetch of its code, which has left the instruction caches since the last layer)
#pragma unroll 1
        for (int c = 0; c < DH / 2; c += 32) {
          float o[32];
          tmem_ld32(tmem_o + lane_addr + (uint32_t)(g * (DH / 2) + c), o);
          if (c + 32 == DH / 2 && !rehearsal) {     // the accumulator may be overwritten
            tc_fence_before();
            __syncwarp();
            if (lane == 0) remote_arrive(ofree0);
          }
#pragma unroll
          for (int e = 0; e < 32; e += 8)
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(rowp + (uint32_t)(((e >> 3) ^ ((lane >> 1) & 3)) << 4)),
                         "r"(pack_bf16(o[e] * inv, o[e + 1] * inv)), "r"(pack_bf16(o[e + 2] * inv, o[e + 3] * inv)),
                         "r"(pack_bf16(o[e + 4] * inv, o[e + 5] * inv)), "r"(pack_bf16(o[e + 6] * inv, o[e + 7] * inv))
                         : "memory");
          __syncwarp();
#pragma unroll 1
          for (int idx = lane; idx < 32 * 4; idx += 32) {
            const int rr = idx >> 2, ch = idx & 3;
            uint4 v;
            asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                         : "r"(ostage + (uint32_t)(rr * 64 + ((ch ^ ((rr >> 1) & 3)) << 4))) : "memory");
            if (rr < nrow) *reinterpret_cast<uint4*>(a.out + out_index(orow0 + rr, ocol0 + c + ch * 8, a.rows_pad, d.Nq)) = v;
          }
          __syncwarp();
        }
        if (rehearsal) {
          rehearsal = false;
          pdl_wait();
          skip = status_set(a.status);
          continue;
        }
      }
      if (k == n_my) break;
      ++n;
      if (++t == it.T) {
        l_prev = l, m = -INFINITY, l = 0.f;
        orow0 = it.b * S + i0, ocol0 = (it.group * 4 + half * 2 + hl) * DH + g * (DH / 2);
        t = 0, ++k, it = nx, nx = item(k + 1);
      }
    }
    tc_fence_before();
  }
  __syncthreads();
  // Neither CTA leaves (or gives its tensor memory back) while the other still works: the leader's MMAs read both CTAs'
  // shared memory and write both tensor memories.
  cluster_arrive_relaxed();
  cluster_wait();
  if (warp == 3) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, 512);
    if (lane == 0 && trc) {
      unsigned long long t;
      unsigned sm;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)::"memory");
      asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
      int tiles = 0;
      for (int k = 0; k < n_my; ++k) tiles += item(k).T;
      trc[8] = t, trc[7] = sm, trc[9] = (unsigned long long)tiles, trc[10] = 1;   // ([10]: marks an attention slot)
    }
  }
}

// rotated suffix keys or values [planes][S][dh]: copies of 64 rows x dh / 128 blocks of 64 channels, rows past S read as zeros
bool own_map(CUtensorMap* m, const void* p, const Dims& d, int batch) {
  const EncodeTiled enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t dims[4] = {64, (cuuint64_t)d.S, (cuuint64_t)(d.dh / 64), (cuuint64_t)batch * d.Hkv};
  const cuuint64_t strides[3] = {(cuuint64_t)d.dh * 2, 128, (cuuint64_t)d.S * d.dh * 2};
  const cuuint32_t box[4] = {64, 64, (cuuint32_t)(d.dh / 128), 1}, es[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int DH>
cudaError_t setup_one() {
  static PerDeviceOnce once;
  if (!once.needed()) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_attn_persist<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AsLayout<DH>::SMEM);
  if (e == cudaSuccess) once.done();
  return e;
}
template <int DH>
int max_pairs_one() {
  if (setup_one<DH>() != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1024), cfg.blockDim = dim3(AS_THREADS), cfg.dynamicSmemBytes = AsLayout<DH>::SMEM;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
  cfg.attrs = at, cfg.numAttrs = 1;
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, k_attn_persist<DH>, &cfg) == cudaSuccess ? n : 0;
}

template <int DH>
cudaError_t launch_one(const AttnArgs& a, int batch, int pairs, cudaStream_t st, bool pdl) {
  cudaError_t e = setup_one<DH>();
  if (e != cudaSuccess) return e;
  CUtensorMap tq, tk, tv;
  if (!row_map(&tq, a.qr, (uint64_t)batch * (a.d.Hq / 2) * (DH / 64) * 128, 128) || !own_map(&tk, a.kr, a.d, batch) || !own_map(&tv, a.vr, a.d, batch))
    return cudaErrorInvalidValue;
  const int items = batch * (a.d.Hq / 4);
  if (items < 1 || pairs < 1) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * (items < pairs ? items : pairs)), cfg.blockDim = dim3(AS_THREADS), cfg.dynamicSmemBytes = AsLayout<DH>::SMEM, cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at, cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_attn_persist<DH>, a, items, tq, tk, tv);
}

}  // namespace

// pairs of this kernel that are resident at a time (0 on an error)
int attention_persist_pairs(const Dims& d) {
  static PerDeviceCount resident[2];
  return d.dh == 256 ? resident[1].get(max_pairs_one<256>) : resident[0].get(max_pairs_one<128>);
}

cudaError_t launch_attention_persist(const Request* rq, int* status, const __nv_bfloat16* q_tiles, const __nv_bfloat16* kr,
                                     const __nv_bfloat16* vr, int layer, __nv_bfloat16* out, int rows_pad, const Dims& d, int batch,
                                     const int* order, unsigned wait_limit, cudaStream_t st, unsigned long long* trace, bool pdl) {
  AttnArgs a{};
  a.rq = rq, a.status = status, a.qr = q_tiles, a.kr = kr, a.vr = vr, a.layer = layer, a.out = out, a.rows_pad = rows_pad;
  a.d = d, a.wait_limit = wait_limit, a.order = order, a.trace = trace;
  const int pairs = attention_persist_pairs(d);
  return d.dh == 256 ? launch_one<256>(a, batch, pairs, st, pdl) : launch_one<128>(a, batch, pairs, st, pdl);
}

}  // namespace phyai
