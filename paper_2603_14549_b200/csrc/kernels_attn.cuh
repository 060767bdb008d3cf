// The layer's attention under the salience-guided bidirectional mask (Eq. 4 applied to the
// values):  O^h = Softmax(W^h + M_bidir) V^h,  W^h = Q^h K^h^T / sqrt(d).
//
//   attn_kernel  persistent blocks; a work item is (two tiles of 128 query rows, head, sequence).  The
//                two row tiles share every key / value tile and take turns on the tensor pipe.
//                For every tile of 128 keys:  S = Q K^T on tcgen05 into tensor memory; the row tile's
//                softmax warpgroup (one thread per row) reads S once, adds Eq. 3's m_j for the future
//                keys of the image span on rows of the image span (nothing else above the diagonal is
//                admitted), turns the logits into probabilities relative to a reference maximum and
//                stores them as bf16 in tensor memory; O += P V then runs with P read from tensor
//                memory and O accumulated in tensor memory.  The final division by the row sum makes
//                the result independent of the reference.  M_bidir is never materialised: it is the
//                vector m_j plus position tests.
//
// V tiles are loaded as they lie in memory (rows = keys) and multiplied as an MN-major operand.
//
// Per (row tile, key tile) the tensor pipe needs 1024 clocks (16 MMAs of 64) and the exponentials 1024 as well (128 x 128,
// 16 per clock and SM), so two row tiles cannot take less than 2048 per key tile; see the figures at attn_kernel.
#pragma once

#include "common.cuh"
#include "kernels_stream.cuh"

namespace asap {

enum : uint32_t { STATUS_ATTN_TIMEOUT = 16u };   // a bounded wait ran out in the attention kernel

constexpr int AT_THREADS = 384;                 // warp 0: items and copies, warp 1: MMA issue, warp 2: Eq. 3's addends, rows past the sequence, warps 4-11: two softmax warpgroups
constexpr int AT_TILE_BYTES = 128 * 128 * 2;    // 128 rows x 128 bf16 as two 64-column blocks of 16 KB
constexpr int AT_BLOCK_BYTES = AT_TILE_BYTES / 2;
constexpr int AT_SLOTS = 4;                     // ring of key and value tiles in the order K0 V0 K1 V1 ...
constexpr int AT_STAGE_BYTES = 32 * 64;         // per softmax warp: 32 rows x 32 columns of the result
constexpr int AT_EXT_BYTES = 128 * 32;          // one k-step: 128 rows x 16 bf16
constexpr int AT_EXT_BUFS = 2;                  // key-side addend tiles in flight
constexpr int AT_EXT_OFF = (2 + AT_SLOTS) * AT_TILE_BYTES;
constexpr int AT_STAGE_OFF = AT_EXT_OFF + (2 + AT_EXT_BUFS) * AT_EXT_BYTES;
constexpr int AT_MAIN_BYTES = AT_STAGE_OFF + 8 * AT_STAGE_BYTES;
constexpr int AT_BOOK_BYTES = 2048;
constexpr int AT_SMEM_BYTES = AT_MAIN_BYTES + AT_BOOK_BYTES;
// Tensor memory: O of both row tiles (2 x 128 columns), ONE S (128) that the row tiles use in turn, P of both (2 x 64).
// A row tile's logits are in registers soon after they are complete, so the next S can be multiplied while their
// exponentials are taken; with an S per row tile P has to lie over it, and softmax, P V and the next S form a chain.
constexpr uint32_t AT_TMEM_COLS = 512, AT_S_COL = 256, AT_P_COL = 384;
constexpr long long AT_WAIT_LIMIT = 2000000000LL;
constexpr float AT_SUM_LIMIT = 1.0995116e12f;   // 2^40: a key tile's sum relative to the reference at which the reference moves
constexpr float AT_NEVER = -1e30f;              // addend of a key that is not admitted (finite: it is a factor of an MMA)
constexpr int AT_ITEM_SLOTS = 4;
static_assert((AT_SLOTS & (AT_SLOTS - 1)) == 0, "ring slots are taken by masking");

struct AttnArgs {
  PrepareArgs pa;              // the blocks derive the descriptors themselves
  int H, pairs;                // pairs: row-tile pairs of the longest sequence
  int n_items, max_vis, mask_enable;
  float scale_log2;            // log2(e) / sqrt(head_dim)
  const float *mask_log;       // [B, max_vis] m_j (natural log) or [B, H, max_vis]; may be null with the mask off
  int mask_b_stride, mask_h_stride;   // max_vis, 0   or   H * max_vis, max_vis
  __nv_bfloat16 *out;          // [tokens, H, 128]
  unsigned int *work;          // [2] items drawn / blocks that have finished; both zero between launches
  uint32_t *status;
  long long wait_limit;        // clock cycles a wait may take before the block gives up
};

struct AttnItem {
  int b;                       // sequence, -1: no more items
  int h, q_base;               // head, first query row (sequence-relative) of the pair
  int n_kt[2];                 // key tiles each row tile looks at (0: no rows)
  int sees[2];                 // the row tile holds rows of the image span and the mask is on
  int row0, n, v0, v_end;
};

struct AttnBook {
  uint64_t full[AT_SLOTS], empty[AT_SLOTS], q_full[2], q_empty[2], s_full[2], s_empty, p_ready[2], pv_done[2];
  uint64_t m_full[2], m_empty[2], ext_full[AT_EXT_BUFS], ext_empty[AT_EXT_BUFS], rows_full[2], rows_empty[2];
  uint64_t item_full[AT_ITEM_SLOTS], item_empty[AT_ITEM_SLOTS], mma_done;
  uint64_t raw[AT_SLOTS];      // a tile that reaches past its sequence lands here; warp 2 passes it on
  AttnItem item[AT_ITEM_SLOTS];
  uint32_t tmem_base;
  int abort_flag;
  alignas(16) float m_tile[2][128];   // [row tile][key]: Eq. 3's addends for the key tile that the diagonal crosses, in the
                                      // units of q.k: m_j inside the span, AT_NEVER outside
};
static_assert(sizeof(AttnBook) <= AT_BOOK_BYTES, "attention kernel bookkeeping exceeds its shared-memory slot");
static_assert(AT_SMEM_BYTES <= 227 * 1024, "attention kernel exceeds an SM's shared memory");

// keys a tile of query rows [q_lo, q_lo + 128) can see: up to its last row (causal), and to the end
// of the image span if one of its rows lies inside the span and the mask is on
__device__ __forceinline__ int attn_key_end(const SampleDesc &d, int q_lo, int mask_enable, int &sees_span) {
  const int q_hi = min(q_lo + 128, d.n);
  sees_span = mask_enable && q_lo < d.v0 + d.nv && q_hi > d.v0;
  return min(d.n, sees_span ? max(q_hi, d.v0 + d.nv) : q_hi);
}

// What Eq. 3's mask does to key tile kt for a row tile that starts at row q_lo.
struct AttnTileKind {
  bool above;    // the row tile holds rows of the span and all keys of the tile lie after all of its rows: every row needs an
                 // addend for every key (m_j for a row of the span, AT_NEVER for any other): one more k-step of the S MMA
  bool crossed;  // the row tile holds rows of the span and the diagonal crosses the key tile: the softmax warps add m_j
};
__device__ __forceinline__ AttnTileKind attn_tile_kind(int sees, int q_lo, int kt) {
  AttnTileKind k;
  k.above = sees && kt * 128 > q_lo + 127;
  k.crossed = sees && !k.above && kt * 128 + 127 > q_lo;
  return k;
}

// The item's last key tile lies above the diagonal of one of its row tiles (see attn_tile_kind).
__device__ __forceinline__ bool attn_last_above(const int (&n_kt)[2], const int (&sees)[2], int q_base) {
  const int kt = max(n_kt[0], n_kt[1]) - 1;
  return (kt < n_kt[0] && attn_tile_kind(sees[0], q_base, kt).above) || (kt < n_kt[1] && attn_tile_kind(sees[1], q_base + 128, kt).above);
}

// What bounds it: at the largest size the power cap (1.04 PFLOP/s algorithmic, 75 % of what a library GEMM sustains under
// the same cap); below that the hand-overs between the tensor pipe and the softmax warps: a key tile of both row tiles takes
// about 3000 clocks where either alone needs 2048.  Measured per call (before: a block per pair of row tiles, a kernel that
// transposed V, a validation kernel, two threads per query row with a shared running maximum, S and P on the same columns):
//   1 x 643 rows, 32 heads            29.0 ->   19.6 us
//   16 x 627-739 rows, 32 heads        304 ->    173 us
//   64 x 2947-3171 rows, 32 heads     14.2 ->    8.7 ms   (9.3 TFLOP)
// Of that on the largest: persistent blocks with V as an MN-major operand 14.1 -> 12.3, an S of its own 11.7 -> 9.8, the mask
// above the diagonal as one more k-step and the issuing warp converged -> 9.0 ms.  A polynomial for an eighth or a quarter of
// the exponentials changed nothing (8.9-9.0), for three eighths it cost 4 %.
__global__ void __launch_bounds__(AT_THREADS, 1)
attn_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
            const __grid_constant__ CUtensorMap tmap_v, AttnArgs a) {
  extern __shared__ __align__(1024) uint8_t at_smem[];
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = smem_u32(at_smem);
  const uint32_t q_smem = base, ring = base + 2 * AT_TILE_BYTES;
  AttnBook *bk = reinterpret_cast<AttnBook *>(at_smem + AT_MAIN_BYTES);

  if (threadIdx.x == 0) {
    for (int s = 0; s < AT_SLOTS; ++s) {
      mbar_init(smem_u32(&bk->full[s]), 1);
      mbar_init(smem_u32(&bk->empty[s]), 1);
      mbar_init(smem_u32(&bk->raw[s]), 1);
    }
    for (int g = 0; g < 2; ++g) {
      mbar_init(smem_u32(&bk->q_full[g]), 1);
      mbar_init(smem_u32(&bk->q_empty[g]), 1);
      mbar_init(smem_u32(&bk->s_full[g]), 1);
      mbar_init(smem_u32(&bk->p_ready[g]), 4);            // the row tile's four softmax warps
      mbar_init(smem_u32(&bk->pv_done[g]), 1);
      mbar_init(smem_u32(&bk->m_full[g]), 1);
      mbar_init(smem_u32(&bk->m_empty[g]), 4);
      mbar_init(smem_u32(&bk->rows_full[g]), 1);
      mbar_init(smem_u32(&bk->rows_empty[g]), 1);
    }
    for (int i = 0; i < AT_EXT_BUFS; ++i) {
      mbar_init(smem_u32(&bk->ext_full[i]), 1);
      mbar_init(smem_u32(&bk->ext_empty[i]), 1);
    }
    for (int i = 0; i < AT_ITEM_SLOTS; ++i) {
      mbar_init(smem_u32(&bk->item_full[i]), 1);
      mbar_init(smem_u32(&bk->item_empty[i]), 10);        // the MMA issuer, the addend warp, every softmax warp
    }
    mbar_init(smem_u32(&bk->mma_done), 1);
    mbar_init(smem_u32(&bk->s_empty), 4);                 // the softmax warps that have taken an S into registers
    bk->abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_q);
    tma_prefetch_desc(&tmap_k);
    tma_prefetch_desc(&tmap_v);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bk->tmem_base), AT_TMEM_COLS);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bk->tmem_base;
  WaitCtx wc{&bk->abort_flag, a.status, STATUS_ATTN_TIMEOUT, a.wait_limit};
  pdl_enter();
  if (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_ATTN_TIMEOUT) bk->abort_flag = 1;   // benign race: same value
  __syncthreads();

  // The launch gives every thread 168 registers; a softmax thread holds its row's 128 logits and needs more, the first
  // warpgroup needs few: 128 x 72 + 256 x 216 = 384 x 168.
  if (warp < 4) {
    reg_dec<72>();
    if (warp == 0) {
      // ---------------------------------------------------------------- items, query / key / value tiles
      // (the whole warp walks the loop and stays converged, see tma_load_2d_w; lane 0 draws the items)
      const uint32_t leader = warp_leader();
      int ic = 0;                                 // items published
      bool first = true;                          // every block's first item is its own number, the others are drawn
      // Draws the next item that has rows and publishes it.  The item queue keeps working after an abort (its waits
      // ignore the flag and are bounded on their own): every consumer must see the same sequence, ending with -1.
      auto draw = [&](AttnItem &it) {
        const int slot = ic % AT_ITEM_SLOTS;
        bool room = true;
        if (ic >= AT_ITEM_SLOTS)
          room = mbar_wait_drain(smem_u32(&bk->item_empty[slot]), ((ic / AT_ITEM_SLOTS) - 1) & 1, AT_WAIT_LIMIT);
        __syncwarp();
        if (!__shfl_sync(0xffffffffu, room ? 1 : 0, 0)) {
          it.b = -1;
          return;
        }
        if (lane == 0) {
          while (true) {
            const int item = bk->abort_flag ? a.n_items : (first ? (int)blockIdx.x : (int)(gridDim.x + atomicAdd(a.work, 1u)));
            first = false;
            it.b = -1;
            if (item >= a.n_items) break;
            const int bh = item / a.pairs;
            it.q_base = (a.pairs - 1 - (item - bh * a.pairs)) * 256;       // long rows first
            it.b = bh / a.H;
            it.h = bh - it.b * a.H;
            const SampleDesc d = make_desc(a.pa, it.b);
            if (!d.valid || it.q_base >= d.n) continue;
            it.row0 = d.row0; it.n = d.n; it.v0 = d.v0; it.v_end = d.v0 + d.nv;
            it.n_kt[0] = (attn_key_end(d, it.q_base, a.mask_enable, it.sees[0]) + 127) / 128;
            it.n_kt[1] = 0; it.sees[1] = 0;
            if (it.q_base + 128 < d.n) it.n_kt[1] = (attn_key_end(d, it.q_base + 128, a.mask_enable, it.sees[1]) + 127) / 128;
            break;
          }
          bk->item[slot] = it;
          mbar_arrive(smem_u32(&bk->item_full[slot]));      // release: the slot's content is visible to the waiters
        }
        __syncwarp();
        it = bk->item[slot];                      // (the slot is not reused before this warp draws four more)
        ++ic;
      };
      AttnItem cur, nxt;
      int tc = 0, qc[2] = {0, 0};                 // key / value tiles and query tiles so far
      int t_issued = 0, q_issued[2] = {0, 0};     // copies actually issued
      uint32_t raw_any = 0u, raw_odd = 0u, raw_last = 0u;     // per ring slot: copies through `raw`: any, an odd number, the latest one
      auto stopped = [&]() { return __shfl_sync(0xffffffffu, bk->abort_flag, 0) != 0; };
      draw(cur);
      while (cur.b >= 0) {
        auto load_q = [&](int g) {
          if (cur.n_kt[g] == 0) return;
          if (qc[g] >= 1) mbar_wait_warp(smem_u32(&bk->q_empty[g]), (qc[g] - 1) & 1, wc);
          if (!stopped()) {
            const uint32_t bar = smem_u32(&bk->q_full[g]);
            const int row = cur.row0 + cur.q_base + g * 128;
            mbar_expect_tx_w(bar, AT_TILE_BYTES, leader);
            tma_load_2d_w(q_smem + g * AT_TILE_BYTES, &tmap_q, bar, cur.h * 128, row, leader);
            tma_load_2d_w(q_smem + g * AT_TILE_BYTES + AT_BLOCK_BYTES, &tmap_q, bar, cur.h * 128 + 64, row, leader);
            q_issued[g] = qc[g] + 1;
          }
          ++qc[g];
        };
        auto load_tile = [&](const CUtensorMap *map, int kt, bool past) {
          const int s = tc % AT_SLOTS;
          if (tc >= AT_SLOTS) mbar_wait_warp(smem_u32(&bk->empty[s]), ((tc / AT_SLOTS) - 1) & 1, wc);
          if (!stopped()) {
            const uint32_t bar = smem_u32(past ? &bk->raw[s] : &bk->full[s]), dst = ring + s * AT_TILE_BYTES, bit = 1u << s;
            const int row = cur.row0 + kt * 128;
            raw_last = past ? raw_last | bit : raw_last & ~bit;
            if (past) { raw_any |= bit; raw_odd ^= bit; }
            mbar_expect_tx_w(bar, AT_TILE_BYTES, leader);
            tma_load_2d_w(dst, map, bar, cur.h * 128, row, leader);
            tma_load_2d_w(dst + AT_BLOCK_BYTES, map, bar, cur.h * 128 + 64, row, leader);
            t_issued = tc + 1;
          }
          ++tc;
        };
        const int n_max = max(cur.n_kt[0], cur.n_kt[1]);
        const bool ragged = n_max * 128 > cur.n, clear_k = ragged && attn_last_above(cur.n_kt, cur.sees, cur.q_base);
        load_q(0);
#pragma unroll 1
        for (int kt = 0; kt < n_max; ++kt) {
          load_tile(&tmap_k, kt, clear_k && kt == n_max - 1);
          if (kt == 0) load_q(1);
          load_tile(&tmap_v, kt, ragged && kt == n_max - 1);
          if (kt == 0) draw(nxt);                 // its look-ups overlap this item's work
        }
        cur = nxt;
      }
      // drain: every copy issued must have landed before the block leaves
      for (int g = 0; g < 2; ++g)
        if (q_issued[g] > 0) mbar_wait_drain(smem_u32(&bk->q_full[g]), (q_issued[g] - 1) & 1, AT_WAIT_LIMIT);
      for (int s = 0; s < AT_SLOTS; ++s) {
        const int fills = t_issued > s ? (t_issued - s + AT_SLOTS - 1) / AT_SLOTS : 0;
        if ((raw_any >> s) & 1u) mbar_wait_drain(smem_u32(&bk->raw[s]), ((raw_odd >> s) & 1u) ^ 1u, AT_WAIT_LIMIT);
        if (fills > 0 && !((raw_last >> s) & 1u)) mbar_wait_drain(smem_u32(&bk->full[s]), (fills - 1) & 1, AT_WAIT_LIMIT);
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer
      // Per key tile and row tile: S of this key tile, then P V of the PREVIOUS one.  In that order an S never waits in the
      // pipe behind a P V that could as well run after it, and no P V is late: its P has been ready for half a turn.
      // The whole warp walks the loop and stays converged (see warp_leader).  After an abort its waits return at once and it
      // goes on multiplying whatever lies in the block's own memory: nothing of it is used.
      const uint32_t leader = warp_leader();
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
      const uint32_t idesc_s = umma_idesc_bf16(128, 128), idesc_o = idesc_s | UMMA_IDESC_B_MN;
      const uint64_t qdesc = umma_desc_sw128(q_smem), tile0 = umma_desc_sw128(ring), vtile0 = umma_desc_sw128_mn(ring, AT_BLOCK_BYTES);
      int t0 = 0;                                 // first tile of the item in the ring: K0 V0 K1 V1 ...
      int qc[2] = {0, 0}, pc[2] = {0, 0}, sn = 0;             // query tiles, P tiles and S so far
      int rc[2] = {0, 0}, ec = 0;                 // row-side and key-side addend tiles so far
      for (int ic = 0;; ++ic) {
        const int slot = ic % AT_ITEM_SLOTS;
        const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / AT_ITEM_SLOTS) & 1, AT_WAIT_LIMIT);
        __syncwarp();
        auto field = [&](const int &f) { return __shfl_sync(0xffffffffu, f, 0); };
        const AttnItem &it = bk->item[slot];
        const int b = field(got ? it.b : -1);
        const int n[2] = {field(it.n_kt[0]), field(it.n_kt[1])}, sees[2] = {field(it.sees[0]), field(it.sees[1])}, q_base = field(it.q_base);
        if (leader) mbar_arrive(smem_u32(&bk->item_empty[slot]));
        if (b < 0) break;
        const int n_max = max(n[0], n[1]);
        for (int kt = 0; kt <= n_max; ++kt) {
          const int tk = t0 + 2 * kt, tv = tk - 1;            // ring tiles: K of this key tile, V of the previous one
          const int sk = tk & (AT_SLOTS - 1), sv = tv & (AT_SLOTS - 1);
          bool above[2] = {false, false};
          const int eb = ec % AT_EXT_BUFS;
          if (kt < n_max) {
            above[0] = kt < n[0] && attn_tile_kind(sees[0], q_base, kt).above;
            above[1] = kt < n[1] && attn_tile_kind(sees[1], q_base + 128, kt).above;
            mbar_wait_warp(smem_u32(&bk->full[sk]), (tk / AT_SLOTS) & 1, wc);
            if (above[0] || above[1]) mbar_wait_warp(smem_u32(&bk->ext_full[eb]), (ec / AT_EXT_BUFS) & 1, wc);
          }
          if (kt > 0) mbar_wait_warp(smem_u32(&bk->full[sv]), (tv / AT_SLOTS) & 1, wc);
          const uint64_t kdesc = tile0 + sk * (AT_TILE_BYTES >> 4), vdesc = vtile0 + sv * (AT_TILE_BYTES >> 4);
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            if (kt < n[g]) {
              if (kt == 0) {
                mbar_wait_warp(smem_u32(&bk->q_full[g]), qc[g] & 1, wc);
                ++qc[g];
                if (sees[g]) {
                  mbar_wait_warp(smem_u32(&bk->rows_full[g]), rc[g] & 1, wc);
                  ++rc[g];
                }
              }
              if (sn > 0) mbar_wait_warp(smem_u32(&bk->s_empty), (sn - 1) & 1, wc);     // the previous S is in registers
              ++sn;
              tc_fence_after();
              tc_mma_bf16_k128_w(tm + AT_S_COL, qdesc + g * (AT_TILE_BYTES >> 4), kdesc, AT_BLOCK_BYTES, AT_BLOCK_BYTES, idesc_s, leader);
              if (above[g])
                tc_mma_bf16_w(tm + AT_S_COL, umma_desc_sw32(base + AT_EXT_OFF + g * AT_EXT_BYTES),
                              umma_desc_sw32(base + AT_EXT_OFF + (2 + eb) * AT_EXT_BYTES), idesc_s, 1u, leader);
              tc_commit_w(smem_u32(&bk->s_full[g]), leader);
              if (g == (kt < n[1] ? 1 : 0)) {                 // the last row tile that looks at this key tile
                tc_commit_w(smem_u32(&bk->empty[sk]), leader);
                if (above[0] || above[1]) tc_commit_w(smem_u32(&bk->ext_empty[eb]), leader);
              }
              if (kt == n[g] - 1) {
                tc_commit_w(smem_u32(&bk->q_empty[g]), leader);
                if (sees[g]) tc_commit_w(smem_u32(&bk->rows_empty[g]), leader);
              }
            }
            if (kt > 0 && kt - 1 < n[g]) {
              mbar_wait_warp(smem_u32(&bk->p_ready[g]), pc[g] & 1, wc);
              ++pc[g];
              tc_fence_after();
#pragma unroll
              for (int kk = 0; kk < 8; ++kk)
                tc_mma_bf16_ta_w(tm + g * 128, tm + AT_P_COL + g * 64 + kk * 8, vdesc + kk * (2048 >> 4), idesc_o,
                                 (kt > 1 || kk > 0) ? 1u : 0u, leader);
              tc_commit_w(smem_u32(&bk->pv_done[g]), leader);
              if (g == (kt - 1 < n[1] ? 1 : 0)) tc_commit_w(smem_u32(&bk->empty[sv]), leader);
            }
          }
          if (above[0] || above[1]) ++ec;
        }
        t0 += 2 * n_max;
      }
      // every MMA this warp issued has completed before tensor memory is given back: after an abort the
      // softmax warps no longer wait for S or P V, so nothing else would hold the block until then
      tc_commit_w(smem_u32(&bk->mma_done), leader);
      mbar_wait_drain(smem_u32(&bk->mma_done), 0, AT_WAIT_LIMIT);
      __syncwarp();
    } else if (warp == 2) {
      // ---------------------------------------------------------------- Eq. 3's addends, one key tile at a time, per row tile
      // (written by the softmax warps themselves they cost those a barrier and a global load per key tile)
      if (blockIdx.x == 0)                        // ... and the validation of the batch
        for (int b = lane; b < a.pa.B; b += 32)
          if (!make_desc(a.pa, b).valid) atomicOr(a.status, (uint32_t)STATUS_BAD_SAMPLE);
      const float m_to_raw = LOG2E_F / a.scale_log2;
      // 16-byte chunk 0 of row r of a one-k-step operand tile; chunk 1 (columns 8-15) stays zero
      auto ext_row = [&](int tile, int r) {
        return reinterpret_cast<uint4 *>(at_smem + AT_EXT_OFF + tile * AT_EXT_BYTES + r * 32 + (((r >> 2) & 1) << 4));
      };
      for (int t = lane; t < (2 + AT_EXT_BUFS) * AT_EXT_BYTES / 16; t += 32)
        reinterpret_cast<uint4 *>(at_smem + AT_EXT_OFF)[t] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
      // The last key and value tile of a sequence reaches into the next one (or past the tensors).  Its probabilities there are
      // exactly zero, but 0 * NaN and an addend on a NaN are NaN: value rows there, and key rows where the mask is an addend, are
      // cleared before the tiles are multiplied.  Such tiles land on `raw` and are handed on here.  (A warp of its own for this
      // cost 2 % on short sequences: it polls beside the softmax warps of its scheduler.)
      int t0 = 0;                                 // first tile of the item in the ring
      uint32_t raw_phase = 0u;                    // per ring slot
      auto clear_past = [&](const AttnItem &it) {
        const int n_max = max(it.n_kt[0], it.n_kt[1]), rows = it.n - (n_max - 1) * 128;     // rows inside the sequence
        for (int v = rows >= 128 ? 2 : (attn_last_above(it.n_kt, it.sees, it.q_base) ? 0 : 1); v < 2; ++v) {
          const int s = (t0 + 2 * n_max - 2 + v) & (AT_SLOTS - 1);
          const bool landed = mbar_wait(smem_u32(&bk->raw[s]), (raw_phase >> s) & 1u, wc);
          raw_phase ^= 1u << s;
          if (!__all_sync(0xffffffffu, landed)) continue;     // (gave up: the copy may not have been issued)
          uint8_t *tile = at_smem + (2 + s) * AT_TILE_BYTES;
          for (int i = rows * 8 + lane; i < 128 * 8; i += 32) {
            reinterpret_cast<uint4 *>(tile)[i] = make_uint4(0u, 0u, 0u, 0u);
            reinterpret_cast<uint4 *>(tile + AT_BLOCK_BYTES)[i] = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bk->full[s]));
        }
        t0 += 2 * n_max;
      };
      int rc[2] = {0, 0}, mc[2] = {0, 0}, ec = 0;             // row-side, diagonal and key-side addend tiles so far
      for (int ic = 0;; ++ic) {
        const int slot = ic % AT_ITEM_SLOTS;
        const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / AT_ITEM_SLOTS) & 1, AT_WAIT_LIMIT);
        AttnItem it;
        if (got) it = bk->item[slot];
        else it.b = -1;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bk->item_empty[slot]));
        if (it.b < 0) break;
        if (it.sees[0] || it.sees[1]) {
          const float *mlog = a.mask_log + (size_t)it.b * a.mask_b_stride + (size_t)it.h * a.mask_h_stride - it.v0;
          // row side: columns 0-2 are 1 for a row of the span (they meet the three pieces of m_j), column 3 for any other row
          // (it meets AT_NEVER)
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            if (!it.sees[g]) continue;
            if (rc[g] >= 1) mbar_wait_warp(smem_u32(&bk->rows_empty[g]), (rc[g] - 1) & 1, wc);
            for (int r = lane; r < 128; r += 32) {
              const int i = it.q_base + g * 128 + r;
              const bool vis = i >= it.v0 && i < it.v_end;
              *ext_row(g, r) = vis ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0u, 0x3f800000u, 0u, 0u);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bk->rows_full[g]));
            ++rc[g];
          }
          const int n_max = max(it.n_kt[0], it.n_kt[1]);
          for (int kt = 0; kt < n_max; ++kt) {
            AttnTileKind kind[2];
#pragma unroll
            for (int g = 0; g < 2; ++g) kind[g] = attn_tile_kind(kt < it.n_kt[g] ? it.sees[g] : 0, it.q_base + g * 128, kt);
            if (!kind[0].above && !kind[1].above && !kind[0].crossed && !kind[1].crossed) continue;
            float m[4];                                         // keys kt * 128 + lane + 32 e
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int j = kt * 128 + lane + 32 * e;
              m[e] = j >= it.v0 && j < it.v_end ? fmaxf(__ldg(mlog + j) * m_to_raw, AT_NEVER) : AT_NEVER;
            }
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              if (!kind[g].crossed) continue;
              if (mc[g] >= 1) mbar_wait_warp(smem_u32(&bk->m_empty[g]), (mc[g] - 1) & 1, wc);
#pragma unroll
              for (int e = 0; e < 4; ++e) bk->m_tile[g][lane + 32 * e] = m[e];
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&bk->m_full[g]));
              ++mc[g];
            }
            if (kind[0].above || kind[1].above) {
              const int eb = ec % AT_EXT_BUFS;
              if (ec >= AT_EXT_BUFS) mbar_wait_warp(smem_u32(&bk->ext_empty[eb]), ((ec / AT_EXT_BUFS) - 1) & 1, wc);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                // the addend as three bf16 pieces: 24 bits of mantissa, all of fp32's
                float piece[3], rest = m[e];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                  piece[k] = __bfloat162float(__float2bfloat16_rn(rest));
                  rest -= piece[k];
                }
                *ext_row(2 + eb, lane + 32 * e) = make_uint4(pack2_rn(piece[0], piece[1]), pack2_rn(piece[2], AT_NEVER), 0u, 0u);
              }
              fence_proxy_async();
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&bk->ext_full[eb]));
              ++ec;
            }
          }
        }
        clear_past(it);
      }
    }
  } else {
    reg_inc<216>();
    // ------------------------------------------------------------------ softmax: one thread per query row
    const int g = (warp - 4) >> 2;                // row tile of this warpgroup
    const int quarter = warp & 3;                 // the TMEM lanes this warp may read
    const int lrow = quarter * 32 + lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t s_addr = lane_addr + AT_S_COL, p_addr = lane_addr + AT_P_COL + g * 64, o_addr = lane_addr + g * 128;
    const float scale = a.scale_log2;
    const uint64_t scale2 = f2_pack(scale, scale);
    int ic = 0, sc = 0, mc = 0;                   // items / key tiles / addend tiles so far
    while (true) {
      const int slot = ic % AT_ITEM_SLOTS;
      const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / AT_ITEM_SLOTS) & 1, AT_WAIT_LIMIT);
      AttnItem it;
      if (got) it = bk->item[slot];
      else it.b = -1;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bk->item_empty[slot]));
      ++ic;
      if (it.b < 0) break;
      const int my_kt = g == 0 ? it.n_kt[0] : it.n_kt[1];
      if (my_kt == 0) continue;
      const int my_sees = g == 0 ? it.sees[0] : it.sees[1];
      const int q_lo = it.q_base + g * 128;
      const int i = q_lo + lrow;                    // sequence-relative query row
      const int i_lo = q_lo + quarter * 32;         // first row of this warp
      const bool vis_row = a.mask_enable && i >= it.v0 && i < it.v_end;
      const int hi_adm = min(it.n - 1, vis_row ? max(i, it.v_end - 1) : i);   // last admitted key
      // p = 2^((x - ref) * scale), x = q.k + addend.  The reference is the maximum of the row's first key tile and then
      // stays: a reference below the running maximum only scales the sums.  Should a tile's sum outgrow AT_SUM_LIMIT in some
      // row of the warp, that tile is done again with the row's true maximum as the new reference (O and the sum so far
      // are rescaled), so no tile but the first needs a pass for its maximum.
      // The code of a key tile is straight-line (its logits are in registers), and its size matters: with an own version
      // per kind of mask it outgrew the instruction cache and ran at half the speed.  So the masks only change x.
      float neg_ref = 0.f, l_run = 0.f;             // -ref * scale
      for (int kt = 0; kt < my_kt; ++kt, ++sc) {
        const int j0 = kt * 128;                    // key of column 0
        const AttnTileKind kind = attn_tile_kind(my_sees, q_lo, kt);
        mbar_wait(smem_u32(&bk->s_full[g]), sc & 1, wc);
        tc_fence_after();
        if (!kind.above && (j0 + 127 > i_lo || j0 + 127 >= it.n)) {
          // Some row of the warp does not admit every key, or needs an addend for a later one: the logits are put right
          // in tensor memory, 32 keys at a time (a loop: once per row tile or twice, and straight-line code of that length
          // would run from outside the instruction cache).  Where no addend belongs to the key tile nothing above the
          // diagonal is admitted, and c > hi hides whatever m_tile holds.
          if (kind.crossed) mbar_wait(smem_u32(&bk->m_full[g]), mc & 1, wc);
          const int di = i - j0, hi = hi_adm - j0;  // columns of the diagonal and of the last admitted key
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += 32) {
            if (j0 + c0 + 31 < it.n && (j0 + c0 + 31 <= i_lo || (kind.crossed && j0 + c0 > i_lo))) continue;   // nothing to do, or done below
            uint32_t r[32];
            tmem_ld32(s_addr + c0, r);
            tmem_wait_ld();
#pragma unroll
            for (int c4 = 0; c4 < 32; c4 += 4) {
              const float4 m4 = *reinterpret_cast<const float4 *>(bk->m_tile[g] + c0 + c4);
              const float add[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int c = c0 + c4 + e;
                const float v = __uint_as_float(r[c4 + e]) + (c > di ? add[e] : 0.f);
                r[c4 + e] = __float_as_uint(c > hi ? -INFINITY : v);
              }
            }
            tmem_st32(s_addr + c0, r);
          }
          tmem_wait_st();
        }
        // ---- this row's 128 logits, once
        uint32_t xr[128];
#pragma unroll
        for (int c = 0; c < 128; c += 32) tmem_ld32p(s_addr + c, xr + c);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bk->s_empty));
        if (kind.crossed) {
          // columns past all rows of the warp (the tile lies on the diagonal, so its first 32 never do): m_j for a row of the span,
          // AT_NEVER for any other (see `chosen` below for logits that are not finite).  Put right in tensor memory like the 32 columns that the diagonal crosses, 450 clocks per 32, they
          // held up the S that both row tiles share for 2000 to 2600 clocks (per call 1 x 643 rows 20.1 -> 19.5 us, 16 x 627-739 174.7 -> 171.3).
          const float off = vis_row ? 0.f : AT_NEVER, in = vis_row ? 1.f : 0.f;
          const uint64_t off2 = f2_pack(off, off), in2 = f2_pack(in, in);
#pragma unroll
          for (int c0 = 32; c0 < 128; c0 += 32) {
            if (j0 + c0 <= i_lo || j0 + c0 + 31 >= it.n) continue;
#pragma unroll
            for (int c = c0; c < c0 + 32; c += 4) {
              const ulonglong2 m4 = *reinterpret_cast<const ulonglong2 *>(bk->m_tile[g] + c);
              float x[4];
              f2_unpack(f2_add(f2_fma(in2, m4.x, f2_pack(__uint_as_float(xr[c]), __uint_as_float(xr[c + 1]))), off2), x[0], x[1]);
              f2_unpack(f2_add(f2_fma(in2, m4.y, f2_pack(__uint_as_float(xr[c + 2]), __uint_as_float(xr[c + 3]))), off2), x[2], x[3]);
#pragma unroll
              for (int e = 0; e < 4; ++e) xr[c + e] = __float_as_uint(x[e]);
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bk->m_empty[g]));
          ++mc;
        }
        if (kt > 0) {
          mbar_wait(smem_u32(&bk->pv_done[g]), (sc - 1) & 1, wc);      // O is complete up to here, and P may be overwritten
          tc_fence_after();
        }
        bool move = kt == 0, again = kt == 0, chosen = !kind.crossed;
        float tile_sum;
#pragma unroll 1
        while (true) {
          if (again) {
            // ---- the row's true maximum becomes the reference of the rows that need it
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};       // four independent chains
#pragma unroll
            for (int c = 0; c < 128; c += 8)
#pragma unroll
              for (int e = 0; e < 4; ++e) mx4[e] = max3(mx4[e], __uint_as_float(xr[c + e]), __uint_as_float(xr[c + 4 + e]));
            const float neg = -fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * scale;   // (key 0 is admitted by every row: finite)
            if (kt > 0) {
              const float f = move ? fast_exp2(neg - neg_ref) : 1.0f;
#pragma unroll 1
              for (int c0 = 0; c0 < 128; c0 += 16) {
                uint32_t r[16];
                tmem_ld16(o_addr + c0, r);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * f);
                tmem_st16(o_addr + c0, r);
              }
              l_run *= f;
            }
            if (move) neg_ref = neg;
          }
          // ---- probabilities relative to the reference, stored as bf16
          const uint64_t neg2 = f2_pack(neg_ref, neg_ref);
          uint64_t sum2[2] = {0ull, 0ull};          // even and odd keys apart, two chains
#pragma unroll
          for (int c0 = 0; c0 < 128; c0 += 32) {
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              float p0, p1;
              f2_unpack(f2_fma(f2_pack(__uint_as_float(xr[c0 + 2 * e]), __uint_as_float(xr[c0 + 2 * e + 1])), scale2, neg2), p0, p1);
              p0 = fast_exp2(p0);
              p1 = fast_exp2(p1);
              sum2[e & 1] = f2_add(sum2[e & 1], f2_pack(p0, p1));
              w[e] = pack2_rn(p0, p1);
            }
            tmem_st16(p_addr + (c0 >> 1), w);
          }
          float s0, s1;
          f2_unpack(f2_add(sum2[0], sum2[1]), s0, s1);
          tile_sum = s0 + s1;
          move = !(tile_sum < AT_SUM_LIMIT);
          if (!__any_sync(0xffffffffu, move)) break;
          if (!chosen) {
            // An addend hides the logit of a key that the row does not admit only if that logit is finite.  The tile is done again
            // with -inf in its place.  (Per call, 16 x 627-739 rows: without this 172.3 us, with it 173.1, with the choice in every tile,
            // two instructions a column, 178.4.)
            chosen = true;
            move = kt == 0;                         // the first tile's reference is taken again, other references stay
            const int hi = hi_adm - j0;
#pragma unroll
            for (int c = 32; c < 128; ++c)
              if (c > hi) xr[c] = __float_as_uint(-INFINITY);
            continue;
          }
          if (again) break;                         // (relative to the true maximum no sum exceeds 128)
          again = true;
        }
        l_run += tile_sum;
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bk->p_ready[g]));
      }
      // ---- normalisation and store
      mbar_wait(smem_u32(&bk->pv_done[g]), (sc - 1) & 1, wc);
      tc_fence_after();
      const float inv_l = l_run > 0.f ? 1.0f / l_run : 0.f;
      // Through shared memory (32 columns at a time, 16-byte chunk c of row r at c ^ ((r >> 1) & 3)), so that a store
      // instruction covers eight pieces of 64 bytes: with one row per lane it touches 32 lines, and the eight warps'
      // stores of an item took 2100 clocks.
      uint8_t *stage = at_smem + AT_STAGE_OFF + (warp - 4) * AT_STAGE_BYTES;
      __nv_bfloat16 *orow = a.out + ((size_t)(it.row0 + i_lo) * a.H + it.h) * 128;
      const int rows = bk->abort_flag ? 0 : it.n - i_lo;       // rows of this warp inside the sequence
#pragma unroll 1
      for (int c0 = 0; c0 < 128; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(o_addr + c0, r);
        tmem_wait_ld();
        __syncwarp();                               // the previous piece has been read
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            w[e] = pack2_rn(__uint_as_float(r[8 * c + 2 * e]) * inv_l, __uint_as_float(r[8 * c + 2 * e + 1]) * inv_l);
          *reinterpret_cast<uint4 *>(stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        __syncwarp();
#pragma unroll
        for (int r8 = 0; r8 < 32; r8 += 8) {
          const int rr = r8 + (lane >> 2), c = lane & 3;
          const uint4 x = *reinterpret_cast<const uint4 *>(stage + rr * 64 + ((c ^ ((rr >> 1) & 3)) << 4));
          if (rr < rows) *reinterpret_cast<uint4 *>(orow + (size_t)rr * a.H * 128 + c0 + c * 8) = x;
        }
      }
      tc_fence_before();                            // the next item's first P (and so its first P V) comes after these loads
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, AT_TMEM_COLS);
  }
  // the block that leaves last puts the work counters back to zero for the next launch (every block has drawn its
  // last item by then)
  if (threadIdx.x == 0) {
    const unsigned int done = atomicAdd(a.work + 1, 1u);
    if (done == gridDim.x - 1) {
      a.work[0] = 0u;
      a.work[1] = 0u;
      __threadfence();
    }
  }
}

}  // namespace asap
