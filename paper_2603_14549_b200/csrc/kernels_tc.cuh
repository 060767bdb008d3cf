// The two dense contractions of the ASAP prune step on the sm_100a tensor cores
// (tcgen05.mma, operands staged by TMA into 128-byte-swizzled shared memory, fp32
// accumulators in tensor memory):
//
//   score_kernel  Eq. 3 / Eq. 4: masked softmax of the ranking rows' logits, reduced over
//                 ranking rows; the logits never leave the SM.
//   sim_kernel    Sec. 4.2: cosine similarity of every visual row against the kept rows with
//                 the arg-max over kept slots taken in the epilogue.
//
// Nothing that the directly preceding kernel of the stream writes (mask vectors, inverse norms) is read by __ldg: these kernels
// start while that one runs, and such a load promises that its data never change.
//
// All use one TMA-producer warp and one MMA-issuer warp, both walking their loops converged with one elected lane issuing
// (see warp_leader), and one or two groups of four epilogue warps that read tensor memory (warp w may touch lanes
// 32*(w%4) .. 32*(w%4)+31).
// Every mbarrier wait is bounded (see WaitCtx); after an abort the block keeps walking its
// uniform control flow so that every named barrier and the final teardown are still reached.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "kernels_stream.cuh"

namespace asap {

constexpr long long TC_WAIT_LIMIT = 1500000000LL;   // clock cycles, roughly one second

// named barriers of the score kernel: 2 = all eight epilogue
// warps; 3 / 4 = one of its two epilogue groups
__device__ __forceinline__ void epi_bar_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }
__device__ __forceinline__ void group_bar_sync(int group) {
  asm volatile("bar.sync %0, 128;" ::"r"(3 + group) : "memory");
}

// =======================================================================================
// score_kernel
//
// Persistent blocks; a work item is one (sample b, head h); blocks draw items from a global
// counter (the ranking rows per sample differ by up to 8x, so a fixed deal leaves blocks idle).
// The ranking rows of an item are taken 256 at a time (a row pair: two row tiles of 128).  For
// each row pair, every key tile is brought to shared memory once per pass and serves both row tiles:
//   pass 1  D = Q_rows K_tile^T   (M = 128 rows, N = 128 keys, one accumulator per row tile):
//           thread-per-row running max / sum over all admitted keys -> off_i = max_i + log2(sum_i)
//   pass 2  D = K_tile Q_rows^T   (M = 128 keys, N = all rows of the pair, up to 256): thread-per-key
//           sum over rows of exp2(logit + mask - off_i), i.e. of the Eq. 4 probabilities A[i, j]
// Key tiles stream through a shared-memory ring in one linear order (pass 1 ascending, pass 2
// over the tiles that hold visual keys, coming back from L2).  Tensor memory holds four accumulators of 128 columns, two per
// epilogue group: an operation is one such accumulator (a pass-2 accumulator wider than 128 columns is two operations), a group
// alternates between its two, and the MMA issuer runs one operation ahead of each group.
// Epilogue: two groups of four warps.  Pass 1 with two row tiles: group g owns row tile g of every
// key tile.  Pass 1 with one row tile, and pass 2: the groups take alternate key tiles.  A group waits for and gives back only
// its own operations; issuer and groups derive the same deal from the item's shape.
// Additive mask (Eq. 3), logits in log2 units: 0 for key j <= row position p; m_j*log2(e) for
// j > p when both are in the image span (mask enabled); -inf otherwise.
// The per-head sums over ranking rows go to `partial`; head_sum_kernel adds them in head order.
// Attention mass on the way (a.mass_heads given; ranking rows after the image span): Eq. 1 with the sum over
// the queries taken first is qbar^h . k_j^h, and pass 2 already multiplies every visual key tile by the
// row pair's queries.  The visual queries stream through the same ring, one tile behind every key tile of pass 1; two warps of
// their own add them up (the pipes that bound the kernel are the exponentials' and the epilogue's: memory, shared memory and
// issue slots have room) and write the sum as ten more "query rows" (its bf16 value, dealt to eight rows by k-step, the
// bf16 value of what that rounding lost, and again: 24 bits of mantissa together, all that fp32 holds)
// behind the pair's rows in shared memory, so the first row pair's pass-2 accumulators get ten
// more columns whose sum is the key's mass for this head.  Row pairs then hold at most 240 rows (the
// accumulator grows by the 16 columns an MMA's width moves in).
// =======================================================================================
constexpr int SC_THREADS = 384;          // producer warp, MMA warp, 2 x 4 epilogue warps, two query-sum warps
constexpr int SC_EPI_THREADS = 256;
constexpr int SC_STAGES = 4;
constexpr int SC_HALF_BYTES = 128 * 128;        // 128 rows x 64 bf16
constexpr int SC_TILE_BYTES = 2 * SC_HALF_BYTES;
constexpr int SC_Q_HALF_BYTES = 256 * 128;      // 256 rows x 64 bf16: one 64-column half of a row pair
constexpr int SC_Q_BYTES = 2 * SC_Q_HALF_BYTES;
constexpr int SC_SMEM_MAIN = SC_Q_BYTES + SC_STAGES * SC_TILE_BYTES;
// Total dynamic shared memory stays at 195 KB: with the 1 KB the system reserves per block that
// is the 196 KB carve-out; one byte more selects the 228 KB carve-out, and an SM that changes its carve-out between this
// kernel and its neighbours delays the next launch by about 10 us.
constexpr int SC_BOOK_BYTES = 3072;
constexpr int SC_SMEM_BYTES = SC_SMEM_MAIN + SC_BOOK_BYTES;
constexpr uint32_t SC_TMEM_COLS = 512;     // four accumulators of 128 columns
constexpr int SC_ITEM_SLOTS = 4;
constexpr int SC_ORDER_MAX = 64;            // sequences up to which items are drawn by size

struct ScoreArgs {
  PrepareArgs pa;             // every block derives its descriptors itself: the kernel does not wait
                              // for the validation kernel (it writes nothing but scratch)
  int B, H, max_vis, mask_enable;
  float scale_log2;           // log2(e) / sqrt(head_dim)
  const float *mask_log;      // [B, max_vis] m_j (natural log), or [B, H, max_vis] with a mask per head
  int mask_b_stride, mask_h_stride;   // max_vis, 0   or   H * max_vis, max_vis
  float *partial;             // [B, H, max_vis] per-head sums over ranking rows
  float *mass_heads;          // [B, H, max_vis] qbar^h . k_j^h for every visual key j (unscaled), qbar^h the sum of the visual
                              // queries (Eq. 1, queries first); nullptr: not wanted.  Given: the kernel also
                              // validates the batch and writes the descriptors (pa.write_desc)
  unsigned int *work;         // [2] next item (score_kernel<true>: past the blocks' first ones) / blocks that have finished; both zero between launches
  uint32_t *status;
  long long wait_limit;       // clock cycles a wait may take before the block gives up
};

struct ScoreBook {             // bookkeeping block placed after the tiles in shared memory
  uint64_t full[SC_STAGES], empty[SC_STAGES], q_full, q_empty, acc_full[4], acc_empty[4];
  uint64_t item_full[SC_ITEM_SLOTS], item_empty[SC_ITEM_SLOTS], mma_done, qbar_ready, qt_full[2], order_ready;
  int item_q[SC_ITEM_SLOTS];   // items drawn by the producer, -1 = no more
  alignas(16) float noff[256]; // per ranking row of the pair: -(max + log2(sum)), -inf for rows past its end
                               // (with one row tile, noff[128..255] carries group 1's partial sums)
  alignas(16) float soft[2][128];   // per epilogue group, per key of its current tile: m_j*log2(e) or -inf
                               // (soft[1] also carries group 1's partial maxima at the end of pass 1)
  alignas(16) int work[SC_ORDER_MAX];   // per sequence (see score_order)
  uint8_t order[SC_ORDER_MAX]; // sequences whose items are drawn by size
  int place;                   // of the first of them in that order
  uint32_t tmem_base;
  int abort_flag;
};

static_assert(sizeof(ScoreBook) <= SC_BOOK_BYTES, "score kernel bookkeeping exceeds its shared-memory slot");

struct RowPair {
  int R0, nrows, nrt, n2, n_kt, t_lo, t_hi, n_p2;
  bool use_soft;
  bool past;                   // -inf is added to logits of the last key tile, which reaches past the sequence
};

// Row pair rp of a sample's ranking rows: rows R0 .. R0 + nrows - 1 (sequence-relative positions).
__device__ __forceinline__ RowPair score_row_pair(const SampleDesc &d, int rp, int mask_enable, int pair_rows) {
  RowPair r;
  r.R0 = d.r0 + rp * pair_rows;
  r.nrows = min(pair_rows, d.nr - rp * pair_rows);
  r.nrt = (r.nrows + 127) >> 7;
  r.n2 = (r.nrows + 15) & ~15;
  const int p_max = r.R0 + r.nrows - 1;
  r.use_soft = mask_enable && (r.R0 < d.v0 + d.nv) && (p_max >= d.v0);
  int jmax = p_max;
  if (r.use_soft) jmax = max(jmax, d.v0 + d.nv - 1);
  r.n_kt = jmax / 128 + 1;
  r.past = r.use_soft && r.n_kt * 128 > d.n;
  r.t_lo = d.v0 / 128;
  r.t_hi = min((d.v0 + d.nv - 1) / 128, r.n_kt - 1);
  r.n_p2 = r.t_hi >= r.t_lo ? r.t_hi - r.t_lo + 1 : 0;
  return r;
}

// Work of one item: the exponentials of pass 1 (a row tile counts whole) and of pass 2, for each pair of row tiles.  In 64 bits and then
// capped: half a million ranking rows over as many keys are past 31 bits, and score_order leaves out what is negative.
__host__ __device__ constexpr int score_work(int n_kt, int nrt, int n_p2, int n2, int n_rp) {
  const long long w = ((long long)n_kt * nrt * 128 + (long long)n_p2 * (n2 + 16)) * n_rp;
  return w < 0x7fffffff ? (int)w : 0x7fffffff;
}
static_assert(score_work(5, 1, 4, 64, 1) == 960 && score_work(4096, 2, 448, 240, 2185) == 0x7fffffff &&
              score_work(1 << 24, 2, 449, 240, 0x7fffffff / 240 + 1) == 0x7fffffff, "a sequence's work is positive at every length");

// Sequences first .. B - 1 (at most SC_ORDER_MAX in all) by descending work of one of their items, a stable order, by one warp;
// returns the place of sequence `first`.
__device__ __forceinline__ int score_order(const ScoreArgs &a, int first, int *work, uint8_t *order, int pair_rows, int lane) {
  int mine[SC_ORDER_MAX / 32];
#pragma unroll
  for (int e = 0; e < SC_ORDER_MAX / 32; ++e) {
    const int b = lane + 32 * e;
    mine[e] = -1;
    if (b >= first && b < a.B) {
      const SampleDesc d = make_desc(a.pa, b);
      if (d.valid) {
        const RowPair T = score_row_pair(d, 0, a.mask_enable, pair_rows);
        mine[e] = score_work(T.n_kt, T.nrt, T.n_p2, T.n2, (d.nr + pair_rows - 1) / pair_rows);
      } else {
        mine[e] = 0;
      }
    }
    work[b] = mine[e];                         // (-1: not among them, never ahead of one that is)
  }
  __syncwarp();
  int place = 0;
#pragma unroll
  for (int e = 0; e < SC_ORDER_MAX / 32; ++e) {
    const int b = lane + 32 * e;
    if (32 * e >= a.B) break;
    int rank = 0;
#pragma unroll 2
    for (int t = 0; t < a.B; t += 8) {         // (entries past the last sequence are -1)
      const int4 u = *reinterpret_cast<const int4 *>(work + t), v = *reinterpret_cast<const int4 *>(work + t + 4);
      const int w[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 8; ++k) rank += w[k] > mine[e] || (w[k] == mine[e] && t + k < b);
    }
    if (mine[e] >= 0) order[rank] = (uint8_t)b;
    if (first / 32 == e) place = __shfl_sync(0xffffffffu, rank, first & 31);
  }
  __syncwarp();
  return place;
}

// SORTED: items past the first round are drawn by size, so that the blocks end together (score of 12 images of 577 to 2881 rows
// 109 -> 97 us, of 64 of 280 to 1400 rows with 16 heads 157 -> 149).  Taken for image spans of different lengths in more items than blocks,
// up to 64 sequences: beyond, a block has so many items that the last one counts little (in order against by size: 96 of 280 to 1400
// rows 220 and 224 us, 128 of them 283 and 286, 128 of 140 to 700 rows with 32 heads 352 and 364).  A block's first item is its own number, see
// the draw.  The order is worked out by a query-sum
// warp that has its first item behind it: by the copy warp it cost 2 to 4 us, and in the kernel for batches that do not want
// it, its code alone 1 to 3 us (1 x 576 39.5 -> 40.6 us, 16 x 576 110.3 -> 113.4).
template <bool SORTED>
__global__ void __launch_bounds__(SC_THREADS, 1)
score_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
             ScoreArgs a) {
  // (the wait for the preceding kernel comes after the block's set-up, which reads nothing that kernel writes)
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int n_items = a.B * a.H;
  const bool with_mass = a.mass_heads != nullptr;
  const int pair_rows = with_mass ? 240 : 256;           // ranking rows per row pair
  // drawn in the first round: all items of `first` sequences, `part` of the next one's
  const int round = (int)gridDim.x, first = SORTED ? round / a.H : 0, part = round - first * a.H;

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
  if ((base - smem_u32(smem_raw)) + SC_SMEM_MAIN + sizeof(ScoreBook) > (uint32_t)SC_SMEM_BYTES) {
    // the tiles need a 1024-byte aligned start; the window is expected to provide it
    if (threadIdx.x == 0) atomicOr(a.status, STATUS_SCORE_TIMEOUT);
    return;
  }
  const uint32_t q_smem = base;                          // the row pair's queries
  const uint32_t k_smem = base + SC_Q_BYTES;             // ring of key tiles
  ScoreBook *bk = reinterpret_cast<ScoreBook *>(base_ptr + SC_SMEM_MAIN);

  if (threadIdx.x == 0) {
    for (int s = 0; s < SC_STAGES; ++s) {
      mbar_init(smem_u32(&bk->full[s]), 1);
      mbar_init(smem_u32(&bk->empty[s]), 2);             // a key tile: the MMAs and their issuer; a query tile: the sum warps
    }
    mbar_init(smem_u32(&bk->q_full), 1);
    mbar_init(smem_u32(&bk->q_empty), 3);                    // the MMAs and both sum warps
    for (int i = 0; i < 4; ++i) {
      mbar_init(smem_u32(&bk->acc_full[i]), 1);
      mbar_init(smem_u32(&bk->acc_empty[i]), 4);          // the epilogue warps of the group that owns the buffer
    }
    for (int i = 0; i < SC_ITEM_SLOTS; ++i) {
      mbar_init(smem_u32(&bk->item_full[i]), 1);
      mbar_init(smem_u32(&bk->item_empty[i]), 11);   // the MMA issuer, every epilogue warp, the sum warps
    }
    mbar_init(smem_u32(&bk->mma_done), 1);
    mbar_init(smem_u32(&bk->qbar_ready), 2);
    mbar_init(smem_u32(&bk->order_ready), 1);
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&bk->qt_full[i]), 1);
    bk->abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bk->tmem_base), SC_TMEM_COLS);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bk->tmem_base;
  WaitCtx wc{&bk->abort_flag, a.status, STATUS_SCORE_TIMEOUT, a.wait_limit};
  if (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_SCORE_TIMEOUT) bk->abort_flag = 1;   // benign race: same value
  __syncthreads();
  pdl_enter();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer: items, queries, key tiles
    // (converged, see tma_load_2d_w)
    const uint32_t leader = warp_leader();
    if (leader) {
      tma_prefetch_desc(&tmap_q);
      tma_prefetch_desc(&tmap_k);
    }
    int kc = 0, qc = 0, ic = 0;               // key tiles / row pairs / items so far
    // query tiles and the second visit of a key tile are the last use of their lines: leaving L2 to the keys of the items in
    // work (and to the hidden rows the next kernels read) is worth 1 to 2 % of the step (16 x 576 121.5 -> 119.1 us, 64 x 2880
    // 2378 -> 2350 us)
    const uint64_t keep = l2_evict_normal(), drop = l2_evict_first();
    int qt = 0;                               // tiles issued for the sum warps
    uint32_t last_past = 0u;                  // ring slots whose latest tile is to be cleared
    int k_issued = 0, q_issued = 0;           // copies actually issued (an abort is sticky, so
                                              // these are prefixes of the two sequences)
    while (true) {
      const int slot = ic % SC_ITEM_SLOTS;
      // The item queue keeps working after an abort (its waits ignore the flag and are bounded on their
      // own): every consumer must see the same sequence of items, ending with -1, or the epilogue warps'
      // named barriers would no longer match.  After an abort that sequence ends at once.
      bool room = true;
      if (ic >= SC_ITEM_SLOTS) room = mbar_wait_drain(smem_u32(&bk->item_empty[slot]), ((ic / SC_ITEM_SLOTS) - 1) & 1, TC_WAIT_LIMIT);
      __syncwarp();
      if (!__shfl_sync(0xffffffffu, room ? 1 : 0, 0)) break;
      int item = 0;
      if (lane == 0) {
        // SORTED: a block's first item is its own number, however late the block starts: an item past the first round waits for the
        // order, which a warp of this block works out behind its own first item.  (Dealt so in the other form too: 1 x 576 39.4 ->
        // 38.9 us, 16 x 576 108.4 -> 109.0.)
        item = bk->abort_flag ? n_items : SORTED && ic == 0 ? (int)blockIdx.x : (SORTED ? round : 0) + (int)atomicAdd(a.work, 1u);
        if (item >= n_items) item = -1;
        if (SORTED && item >= round) {
          if (mbar_wait(smem_u32(&bk->order_ready), 0, wc)) {
            int m = item - round;              // `part` heads of sequence `first` are gone: as if they had come first of it
            if (m >= bk->place * a.H) m += part;
            item = bk->order[m / a.H] * a.H + m % a.H;
          } else {
            item = -1;
          }
        }
        bk->item_q[slot] = item;
        mbar_arrive(smem_u32(&bk->item_full[slot]));      // release: the slot's content is visible to the waiters
      }
      item = __shfl_sync(0xffffffffu, item, 0);
      ++ic;
      if (item < 0) break;
      const int b = item / a.H, h = item - b * a.H;
      const SampleDesc d = make_desc(a.pa, b);
      if (!d.valid) continue;
      const int n_rp = (d.nr + pair_rows - 1) / pair_rows;
      for (int rp = 0; rp < n_rp; ++rp, ++qc) {
        const RowPair T = score_row_pair(d, rp, a.mask_enable, pair_rows);
        auto load_queries = [&]() {
          if (qc >= 1) mbar_wait_warp(smem_u32(&bk->q_empty), (qc - 1) & 1, wc);
          if (!__shfl_sync(0xffffffffu, bk->abort_flag, 0)) {
            mbar_expect_tx_w(smem_u32(&bk->q_full), T.nrt * SC_TILE_BYTES, leader);
            for (int hf = 0; hf < 2; ++hf)
              for (int rt = 0; rt < T.nrt; ++rt)
                tma_load_2d_w(q_smem + hf * SC_Q_HALF_BYTES + rt * SC_HALF_BYTES, &tmap_q, smem_u32(&bk->q_full),
                              h * 128 + hf * 64, d.row0 + T.R0 + rt * 128, leader);
            q_issued = qc + 1;
          }
        };
        const int nq = with_mass && rp == 0 ? (d.nv + 127) / 128 : 0;      // tiles of visual queries (never more than n_kt)
        // A query tile lands on a barrier of its own (alternating: the sum warps see only these, in order, so they cannot
        // mistake a ring slot's phase; two query tiles are never in flight on the same one, see below) and its slot's
        // barrier is passed at once, which keeps that barrier's phases in step with the ring.
        // A key tile that needs rows cleared first (`past`; never in a kernel with query tiles) uses the same barriers, and the
        // clearing warp passes its slot's barrier.
        auto load_tile = [&](bool query, bool past, int row, uint64_t policy) {
          const int s = kc % SC_STAGES;
          if (kc >= SC_STAGES) mbar_wait_warp(smem_u32(&bk->empty[s]), ((kc / SC_STAGES) - 1) & 1, wc);
          if (!__shfl_sync(0xffffffffu, bk->abort_flag, 0)) {
            const uint32_t dst = k_smem + s * SC_TILE_BYTES;
            const uint32_t bar = smem_u32(query || past ? &bk->qt_full[qt & 1] : &bk->full[s]);
            const CUtensorMap *map = query ? &tmap_q : &tmap_k;
            mbar_expect_tx_w(bar, SC_TILE_BYTES, leader);
            tma_load_2d_hint_w(dst, map, bar, h * 128, row, policy, leader);
            tma_load_2d_hint_w(dst + SC_HALF_BYTES, map, bar, h * 128 + 64, row, policy, leader);
            if (query && leader) mbar_arrive(smem_u32(&bk->full[s]));
            if (query || past) ++qt;
            last_past = past ? last_past | (1u << s) : last_past & ~(1u << s);
            k_issued = kc + 1;
          }
          ++kc;
        };
        // The pair's queries overwrite the last pair's, whose MMAs must have ended; the ring's tiles only wait for their slots.
        // Two key tiles and what follows them go first, no more: four tiles find a slot without these queries' products (16 x 576
        // 110.2 -> 108.9 us, 8 x 1536 with a mask per head 189.7 -> 188.1, score of 64 x 2880 986 -> 966).  A block's first pair waits for nothing.
        const int q_at = qc == 0 ? 0 : min(2, T.n_kt + T.n_p2 - 1);
        for (int u = 0; u < T.n_kt + T.n_p2; ++u) {
          if (u == q_at) load_queries();
          load_tile(false, T.past && u == T.n_kt - 1, d.row0 + (u < T.n_kt ? u : T.t_hi - (u - T.n_kt)) * 128, u < T.n_kt ? keep : drop);
          // (query tiles are two ring positions apart, so the one after the next takes the slot of this one, whose
          // release says that it has been added up; between two items at least four other tiles pass)
          if (u < nq) load_tile(true, false, d.row0 + d.v0 + u * 128, drop);
        }
      }
    }
    // every copy this warp issued must have landed before the block may leave
    for (int s = 0; s < SC_STAGES; ++s) {
      const int fills = k_issued > s ? (k_issued - s + SC_STAGES - 1) / SC_STAGES : 0;
      if (fills > 0 && !((last_past >> s) & 1u)) mbar_wait_drain(smem_u32(&bk->full[s]), (fills - 1) & 1, TC_WAIT_LIMIT);
    }
    if (q_issued > 0) mbar_wait_drain(smem_u32(&bk->q_full), (q_issued - 1) & 1, TC_WAIT_LIMIT);
    for (int i = 0; i < 2; ++i)
      if (qt > i) mbar_wait_drain(smem_u32(&bk->qt_full[i]), (((qt - 1 - i) >> 1) & 1), TC_WAIT_LIMIT);
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // (the whole warp walks the loop and stays converged, see warp_leader: 64 sequences of 2880 visual tokens 1043 -> 1000 us,
    // 16 of 576 57.8 -> 54.7 us against one lane under a branch.  After an abort its waits return at once and it
    // goes on multiplying whatever lies in the block's own memory: nothing of it is used)
    const uint32_t leader = warp_leader();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
    int kc = 0, qc = 0, ic = 0, mc = 0;               // mc: row pairs whose query tile the sum warps complete
    int ops0 = 0, ops1 = 0;                           // operations given to either epilogue group
    const uint32_t idesc1 = umma_idesc_bf16(128, 128);
    const uint64_t qdesc = umma_desc_sw128(q_smem), kdesc0 = umma_desc_sw128(k_smem);   // (every tile lies below 256 KB: offsets never carry out of the address field)
    while (true) {
      const int slot = ic % SC_ITEM_SLOTS;
      const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / SC_ITEM_SLOTS) & 1, TC_WAIT_LIMIT);
      __syncwarp();
      const int item = __shfl_sync(0xffffffffu, got ? bk->item_q[slot] : -1, 0);
      if (leader) mbar_arrive(smem_u32(&bk->item_empty[slot]));
      ++ic;
      if (item < 0) break;
      SampleDesc d = make_desc(a.pa, item / a.H);
      d.v0 = __shfl_sync(0xffffffffu, d.v0, 0); d.nv = __shfl_sync(0xffffffffu, d.nv, 0);
      d.r0 = __shfl_sync(0xffffffffu, d.r0, 0); d.nr = __shfl_sync(0xffffffffu, d.nr, 0);
      if (!__shfl_sync(0xffffffffu, d.valid, 0)) continue;
      const int n_rp = (d.nr + pair_rows - 1) / pair_rows;
      for (int rp = 0; rp < n_rp; ++rp, ++qc) {
        const RowPair T = score_row_pair(d, rp, a.mask_enable, pair_rows);
        const bool mass_here = with_mass && rp == 0;         // ten more columns (16 with padding): the summed query
        const int n2 = T.n2 + (mass_here ? 16 : 0);          // columns of a pass-2 accumulator
        const bool fixed = mass_here || T.nrows < T.n2;
        mbar_wait_warp(smem_u32(&bk->q_full), qc & 1, wc);
        // the accumulator of group gr's next operation, once the group has given it back
        auto acc = [&](int gr) -> int {
          const int n = gr ? ops1 : ops0, buf = 2 * gr + (n & 1);
          if (gr) ++ops1;
          else ++ops0;
          if (n >= 2) mbar_wait_warp(smem_u32(&bk->acc_empty[buf]), ((n >> 1) - 1) & 1, wc);
          tc_fence_after();
          return buf;
        };
        const int nq = mass_here ? (d.nv + 127) / 128 : 0;    // every key tile below nq is followed by a query tile (the sum warps')
        for (int u = 0; u < T.n_kt + T.n_p2; kc += u < nq ? 2 : 1, ++u) {
          const int s = kc % SC_STAGES;
          if (fixed && u == T.n_kt) {                        // the sum warps have written their rows
            mbar_wait_warp(smem_u32(&bk->qbar_ready), mc & 1, wc);
            ++mc;
          }
          mbar_wait_warp(smem_u32(&bk->full[s]), (kc / SC_STAGES) & 1, wc);
          const uint64_t kdesc = kdesc0 + s * (SC_TILE_BYTES >> 4);
          if (u < T.n_kt) {
            for (int rt = 0; rt < T.nrt; ++rt) {
              const int buf = acc(T.nrt == 2 ? rt : u & 1);
              tc_mma_bf16_k128_w(tm + buf * 128, qdesc + rt * (SC_HALF_BYTES >> 4), kdesc, SC_Q_HALF_BYTES, SC_HALF_BYTES, idesc1, leader);
              tc_commit_w(smem_u32(&bk->acc_full[buf]), leader);
            }
          } else {
            for (int c0 = 0; c0 < n2; c0 += 128) {
              const int buf = acc((u - T.n_kt + 1) & 1);
              tc_mma_bf16_k128_w(tm + buf * 128, kdesc, qdesc + (c0 >> 7) * (SC_HALF_BYTES >> 4), SC_HALF_BYTES, SC_Q_HALF_BYTES,
                                 umma_idesc_bf16(128, min(128, n2 - c0)), leader);
              tc_commit_w(smem_u32(&bk->acc_full[buf]), leader);
            }
          }
          tc_commit_w(smem_u32(&bk->empty[s]), leader);
          if (leader) mbar_arrive(smem_u32(&bk->empty[s]));
        }
        if (fixed && T.n_p2 == 0) {                          // (no visual key tile: keep the barrier's phases in step)
          mbar_wait_warp(smem_u32(&bk->qbar_ready), mc & 1, wc);
          ++mc;
        }
        tc_commit_w(smem_u32(&bk->q_empty), leader);
      }
    }
    // every MMA this warp issued has completed before tensor memory is given back: after an abort the
    // epilogue warps no longer wait for the accumulators, so nothing else would hold the block until then
    tc_commit_w(smem_u32(&bk->mma_done), leader);
    mbar_wait_drain(smem_u32(&bk->mma_done), 0, TC_WAIT_LIMIT);
    __syncwarp();
  } else if (warp < 10) {
    // ------------------------------------------------------------------ epilogue (2 groups x 4 warps)
    // Warp q of a group reads tensor-memory lanes 32q .. 32q+31.
    const int group = (warp - 2) >> 2;
    const int quarter = warp & 3;
    const int lrow = quarter * 32 + lane;          // tensor-memory lane owned by this thread
    const int et = (warp - 2) * 32 + lane;         // 0..255 among the epilogue threads
    const float scale = a.scale_log2;
    const uint32_t tlane0 = tmem_base + ((uint32_t)(quarter * 32) << 16);
    float *soft = bk->soft[group];
    float *pm = bk->soft[1], *pl = bk->noff + 128; // group 1's (max, sum) when both groups share one row tile
    const uint64_t scale2 = f2_pack(scale, scale);
    int ops = 0, ic = 0, qc = 0;                   // ops: operations of this group so far
    while (true) {
      const int slot = ic % SC_ITEM_SLOTS;
      const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / SC_ITEM_SLOTS) & 1, TC_WAIT_LIMIT);
      const int item = got ? bk->item_q[slot] : -1;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bk->item_empty[slot]));
      ++ic;
      if (item < 0) break;
      const int b = item / a.H, h = item - b * a.H;
      const SampleDesc d = make_desc(a.pa, b);
      if (!d.valid) continue;
      const int n_rp = (d.nr + pair_rows - 1) / pair_rows;
      float *part = a.partial + ((size_t)b * a.H + h) * a.max_vis;
      const float *mlog = a.mask_log + (size_t)b * a.mask_b_stride + (size_t)h * a.mask_h_stride;
      const int v_end = d.v0 + d.nv;
      {
        // visual keys beyond the tiles the first row pair visits in pass 2 (possible only when
        // ranking rows lie before the end of the image span) start from zero; the epilogue-wide
        // barrier that ends every pass 1 orders these stores before any later add
        const RowPair T0 = score_row_pair(d, 0, a.mask_enable, pair_rows);
        const int first = T0.n_p2 > 0 ? max((T0.t_hi + 1) * 128 - d.v0, 0) : 0;
        for (int j = first + et; j < d.nv; j += SC_EPI_THREADS) part[j] = 0.f;
      }
      for (int rp = 0; rp < n_rp; ++rp, ++qc) {
        const RowPair T = score_row_pair(d, rp, a.mask_enable, pair_rows);
        // ---------------- pass 1: thread = ranking row.  Two row tiles: group g owns tile g of every key
        // tile; one row tile: the groups take alternate key tiles
        const bool two = T.nrt == 2;
        const int my_row = (two ? group * 128 : 0) + lrow;             // row of the pair
        const bool row_ok = my_row < T.nrows;
        const bool warp_rows = (two ? group * 128 : 0) + quarter * 32 < T.nrows;
        const int p_i = T.R0 + my_row;
        const bool row_vis = T.use_soft && p_i >= d.v0 && p_i < v_end;
        float m = -INFINITY, l = 0.f;
        for (int t = two ? 0 : group; t < T.n_kt; t += two ? 1 : 2, ++ops) {
          const int buf = 2 * group + (ops & 1);
          const int j0 = t * 128;
          const bool fast = (j0 + 127 <= T.R0 + (two ? group * 128 : 0));
          const bool stage_soft = T.use_soft && !fast;
          if (stage_soft) {
            const int j = j0 + lrow;
            soft[lrow] = (j >= d.v0 && j < v_end) ? mlog[j - d.v0] * LOG2E_F : -INFINITY;
            group_bar_sync(group);
          }
          const uint32_t tlane = tlane0 + buf * 128;
          mbar_wait(smem_u32(&bk->acc_full[buf]), (ops >> 1) & 1, wc);
          tc_fence_after();
          if (warp_rows && !bk->abort_flag) {
            bool summed = false;
            if (fast && __all_sync(0xffffffffu, !row_ok || m > -INFINITY)) {
              // every key admitted, no mask, and the rows already have a reference maximum: add
              // exp2(dot * scale - m) without looking for a new maximum (a stale reference only scales
              // the sum; off_i = m + log2(l) comes out the same), the next 32 columns on their way meanwhile.  Should a
              // row's sum outgrow fp32's range the tile is done again below, with true maxima as new references.
              const float neg_m = row_ok ? -m : 0.f;
              const uint64_t negm2 = f2_pack(neg_m, neg_m);
              uint64_t sm2[4] = {0ull, 0ull, 0ull, 0ull};
              auto add32 = [&](const uint32_t (&r)[32]) {
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                  float x0, x1;
                  f2_unpack(f2_fma(f2_pack(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), scale2, negm2), x0, x1);
                  sm2[(e >> 1) & 3] = f2_add(sm2[(e >> 1) & 3], f2_pack(fast_exp2(x0), fast_exp2(x1)));
                }
              };
              uint32_t ra[32], rb[32];
              tmem_ld32(tlane, ra);
              tmem_wait_ld();
#pragma unroll 1
              for (int c = 0; c < 128; c += 64) {
                tmem_ld32(tlane + c + 32, rb);
                add32(ra);
                tmem_wait_ld();
                if (c == 0) tmem_ld32(tlane + 64, ra);
                add32(rb);
                tmem_wait_ld();
              }
              float cs, c1;
              f2_unpack(f2_add(f2_add(sm2[0], sm2[1]), f2_add(sm2[2], sm2[3])), cs, c1);
              cs += c1;
              if (!__any_sync(0xffffffffu, row_ok && !(cs < 1e30f))) {
                if (row_ok) l += cs;
                summed = true;
              }
            }
#pragma unroll 1
            for (int c = summed ? 128 : 0; c < 128; c += 32) {
              // with a new maximum per chunk: the first tile of a row pair, tiles that cross a row's own position (selects only,
              // no branches), and the rare second try.  `lim` = last column of this chunk the row may attend to without
              // the soft mask
              uint32_t r[32];
              tmem_ld32(tlane + c, r);
              tmem_wait_ld();
              const int lim = p_i - (j0 + c);
              float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
              if (!stage_soft) {
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                  const float x = (e <= lim) ? __uint_as_float(r[e]) * scale : -INFINITY;
                  r[e] = __float_as_uint(x);
                  mx[e & 3] = fmaxf(mx[e & 3], x);
                }
              } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                  const float sv = row_vis ? soft[c + e] : -INFINITY;
                  const float x = fmaf(__uint_as_float(r[e]), scale, (e <= lim) ? 0.f : sv);
                  r[e] = __float_as_uint(x);
                  mx[e & 3] = fmaxf(mx[e & 3], x);
                }
              }
              const float m_new = fmaxf(m, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])));
              if (row_ok && m_new > -INFINITY) {
                float sm[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 32; ++e) sm[e & 3] += fast_exp2(__uint_as_float(r[e]) - m_new);
                l = l * fast_exp2(m - m_new) + ((sm[0] + sm[1]) + (sm[2] + sm[3]));
                m = m_new;
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bk->acc_empty[buf]));
          if (stage_soft) group_bar_sync(group);   // soft[] is rewritten by this group's next masked tile
        }
        // off_i = max_i + log2(sum_i), so that exp2(x - off_i) = exp2(x - max_i) / sum_i.  With one row
        // tile the two groups saw disjoint key tiles: their (max, sum) per row are merged first
        epi_bar_sync();                             // both groups are past the previous row pair's offsets and the last soft[1]
        if (two) {
          bk->noff[my_row] = row_ok ? -(m + __log2f(l)) : -INFINITY;
        } else {
          if (group == 1) { pm[lrow] = m; pl[lrow] = l; }
          epi_bar_sync();
          if (group == 0) {
            const float m1 = pm[lrow], l1 = pl[lrow];
            const float mm = fmaxf(m, m1);
            float ll = 0.f;
            if (m > -INFINITY) ll += l * fast_exp2(m - mm);
            if (m1 > -INFINITY) ll += l1 * fast_exp2(m1 - mm);
            bk->noff[lrow] = row_ok ? -(mm + __log2f(ll)) : -INFINITY;
          }
        }
        epi_bar_sync();
        // ---------------- pass 2: thread = key; the groups take alternate visual key tiles
        const int n2 = T.n2 + (with_mass && rp == 0 ? 16 : 0);
        for (int u = group ^ 1; u < T.n_p2; u += 2) {
          const int t = T.t_hi - u, j0 = t * 128;
          const int j = j0 + lrow;
          const bool key_ok = j >= d.v0 && j < v_end;
          const bool fast = (j0 + 127 <= T.R0);
          const bool warp_keys = (j0 + quarter * 32 + 31 >= d.v0) && (j0 + quarter * 32 < v_end);
          const float soft_j = (T.use_soft && key_ok) ? mlog[j - d.v0] * LOG2E_F : -INFINITY;
          uint64_t sm2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 1
          for (int h0 = 0; h0 < n2; h0 += 128, ++ops) {
            const int buf = 2 * group + (ops & 1);
            const uint32_t tlane = tlane0 + buf * 128;
            mbar_wait(smem_u32(&bk->acc_full[buf]), (ops >> 1) & 1, wc);
            tc_fence_after();
            if (warp_keys && !bk->abort_flag) {
              const int n_here = min(128, T.n2 - h0);       // (a multiple of 16)
              // rows past the pair's end have the offset -inf (every entry up to the next multiple of 128 is
              // written), so their terms vanish; four offsets per shared-memory load
              auto add32 = [&](const uint32_t (&r)[32], int c) {
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                  const ulonglong2 o = *reinterpret_cast<const ulonglong2 *>(bk->noff + h0 + c + e);
                  float x0, x1, x2, x3;
                  f2_unpack(f2_fma(f2_pack(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), scale2, o.x), x0, x1);
                  f2_unpack(f2_fma(f2_pack(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), scale2, o.y), x2, x3);
                  sm2[(e >> 1) & 3] = f2_add(sm2[(e >> 1) & 3], f2_pack(fast_exp2(x0), fast_exp2(x1)));
                  sm2[((e >> 1) + 1) & 3] = f2_add(sm2[((e >> 1) + 1) & 3], f2_pack(fast_exp2(x2), fast_exp2(x3)));
                }
              };
              int c = 0;
              if (fast && n_here >= 32) {
                // the next 32 columns are on their way while these are exponentiated
                const int last = (n_here & ~31) - 32;
                uint32_t ra[32], rb[32];
                tmem_ld32(tlane, ra);
                tmem_wait_ld();
#pragma unroll 1
                for (; c <= last; c += 64) {
                  if (c < last) tmem_ld32(tlane + c + 32, rb);
                  add32(ra, c);
                  tmem_wait_ld();
                  if (c < last) {
                    if (c + 32 < last) tmem_ld32(tlane + c + 64, ra);
                    add32(rb, c + 32);
                    tmem_wait_ld();
                  }
                }
                c = last + 32;
              }
#pragma unroll 1
              for (; c < n_here; c += 16) {
                uint32_t r[16];
                tmem_ld16(tlane + c, r);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; e += 2) {
                  const float2 o = *reinterpret_cast<const float2 *>(bk->noff + h0 + c + e);
                  float x[2];
#pragma unroll
                  for (int k = 0; k < 2; ++k) {
                    const int p = T.R0 + h0 + c + e + k;
                    const float above = (p >= d.v0 && p < v_end) ? soft_j : -INFINITY;
                    x[k] = fast_exp2(fmaf(__uint_as_float(r[e + k]), scale, (j <= p) ? 0.f : above) + (k ? o.y : o.x));
                  }
                  sm2[(e >> 1) & 3] = f2_add(sm2[(e >> 1) & 3], f2_pack(x[0], x[1]));
                }
              }
              if (with_mass && rp == 0 && T.n2 - h0 >= 0 && T.n2 - h0 < 128) {
                // columns n2 .. n2 + 9: the pieces of the summed query against this key
                uint32_t r[16];
                tmem_ld16(tlane + (T.n2 - h0), r);
                tmem_wait_ld();
                auto g = [&](int e) { return __uint_as_float(r[e]); };
                if (key_ok)
                  a.mass_heads[((size_t)b * a.H + h) * a.max_vis + (j - d.v0)] =
                      (((g(0) + g(1)) + (g(2) + g(3))) + ((g(4) + g(5)) + (g(6) + g(7)))) + (g(8) + g(9));
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bk->acc_empty[buf]));
          }
          if (key_ok && !bk->abort_flag) {
            float s0, s1;
            f2_unpack(f2_add(f2_add(sm2[0], sm2[1]), f2_add(sm2[2], sm2[3])), s0, s1);
            // the first row pair initialises the slots it covers; later row pairs add (the barriers between their passes
            // make the earlier pair's sums visible, whichever group wrote them)
            if (rp == 0) part[j - d.v0] = s0 + s1;
            else part[j - d.v0] += s0 + s1;
          }
        }
      }
    }
    __threadfence();
  } else {
    // ------------------------------------------------------------------ query-sum warps: one 64-column half of the head each
    // They also clear the query rows between a pair's last row and the next multiple of 16: those belong to whatever lies behind
    // the ranking rows, the next sequence perhaps, and a NaN there would pass through the offset of -inf into every key's sum.
    if (warp == 11 && blockIdx.x == 0 && a.pa.write_desc) prepare_warp(a.pa);
    const int half = warp - 10;
    const int c = lane & 7, r0 = lane >> 3;        // a lane adds 16-byte chunk c of rows r0, r0 + 4, ...
    int kc = 0, qc = 0, qt = 0;                    // ring positions, row pairs, query tiles so far
    for (int ic = 0;; ++ic) {
      const int slot = ic % SC_ITEM_SLOTS;
      const bool got = mbar_wait_drain(smem_u32(&bk->item_full[slot]), (ic / SC_ITEM_SLOTS) & 1, TC_WAIT_LIMIT);
      __syncwarp();
      const int item = __shfl_sync(0xffffffffu, got ? bk->item_q[slot] : -1, 0);
      if (lane == 0) mbar_arrive(smem_u32(&bk->item_empty[slot]));
      if (item < 0) break;
      const SampleDesc d = make_desc(a.pa, item / a.H);
      const int n_rp = d.valid ? (d.nr + pair_rows - 1) / pair_rows : 0;
      for (int rp = 0; rp < n_rp; ++rp, ++qc) {
        const RowPair T = score_row_pair(d, rp, a.mask_enable, pair_rows);
        const bool mass_here = with_mass && rp == 0, fixed = mass_here || T.nrows < T.n2;
        float f[8];
        if (mass_here) {
          const int nq = (d.nv + 127) / 128;
          uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
          for (int u = 0; u < nq; ++u, ++qt) {
            const int s = (kc + 2 * u + 1) % SC_STAGES;
            mbar_wait_warp(smem_u32(&bk->qt_full[qt & 1]), (qt >> 1) & 1, wc);
            const uint8_t *tile = base_ptr + SC_Q_BYTES + s * SC_TILE_BYTES + half * SC_HALF_BYTES;
            const int rows = min(128, d.nv - u * 128);
#pragma unroll 8
            for (int r = r0; r < rows; r += 4) {
              const uint4 x = *reinterpret_cast<const uint4 *>(tile + r * 128 + ((c ^ (r & 7)) << 4));
              acc[0] = f2_add(acc[0], f2_pack(bf16_lo(x.x), bf16_hi(x.x)));
              acc[1] = f2_add(acc[1], f2_pack(bf16_lo(x.y), bf16_hi(x.y)));
              acc[2] = f2_add(acc[2], f2_pack(bf16_lo(x.z), bf16_hi(x.z)));
              acc[3] = f2_add(acc[3], f2_pack(bf16_lo(x.w), bf16_hi(x.w)));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bk->empty[s]));
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) f2_unpack(acc[e], f[2 * e], f[2 * e + 1]);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            f[e] += __shfl_xor_sync(0xffffffffu, f[e], 8);
            f[e] += __shfl_xor_sync(0xffffffffu, f[e], 16);
          }
          kc += nq;
        }
        mbar_wait_warp(smem_u32(&bk->q_full), qc & 1, wc);    // (of every row pair, in order: its phases cannot be mistaken)
        if (fixed) {
          // The summed query of this head as rows n2 .. n2 + 9 of the pair's query tile (row r of a 64-column half is 128
          // bytes at r * 128, chunk c at c ^ (r & 7)), once the tiled copy of the queries has landed: the value as three bf16
          // pieces, 24 bits of mantissa, all of fp32's.  The first piece is dealt to eight rows, one per k-step, zero elsewhere: the
          // accumulator drops bits at every k-step that adds to it, so each step gets an accumulator of its own and
          // the epilogue adds them up with rounding.  The other two pieces are small enough for a row each.
          uint8_t *qrows = base_ptr + half * SC_Q_HALF_BYTES;
          for (int i = T.nrows * 8 + lane; i < T.n2 * 8; i += 32) reinterpret_cast<uint4 *>(qrows)[i] = make_uint4(0u, 0u, 0u, 0u);
          if (mass_here) {
            uint32_t w[3][4];                               // [piece][two elements of this lane's chunk]
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float rest[2] = {f[2 * e], f[2 * e + 1]};
#pragma unroll
              for (int k = 0; k < 3; ++k) {
                w[k][e] = pack2_rn(rest[0], rest[1]);
                rest[0] -= bf16_lo(w[k][e]);
                rest[1] -= bf16_hi(w[k][e]);
              }
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              const int j = r0 + 4 * i;                     // lanes 8 r0 .. 8 r0 + 7 write rows r0, r0 + 4 and r0 + 8 of the ten
              const bool step = i < 2 && (j >> 2) == half && (j & 3) == c >> 1;
              uint4 x = make_uint4(0u, 0u, 0u, 0u);
              if (i < 2 && step) x = make_uint4(w[0][0], w[0][1], w[0][2], w[0][3]);
              if (i == 2) x = r0 == 0 ? make_uint4(w[1][0], w[1][1], w[1][2], w[1][3]) : make_uint4(w[2][0], w[2][1], w[2][2], w[2][3]);
              const int row = T.n2 + j;
              if (j < 10) *reinterpret_cast<uint4 *>(qrows + row * 128 + ((c ^ (row & 7)) << 4)) = x;
            }
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&bk->qbar_ready));
        }
        if (lane == 0) mbar_arrive(smem_u32(&bk->q_empty));
        if (T.past) {
          // key rows of the next sequence (see RowPair), by one of the two warps
          const int s = (kc + T.n_kt - 1) % SC_STAGES, end = d.n - (T.n_kt - 1) * 128;
          if (half == 0 && __all_sync(0xffffffffu, mbar_wait(smem_u32(&bk->qt_full[qt & 1]), (qt >> 1) & 1, wc))) {
            uint8_t *tile = base_ptr + SC_Q_BYTES + s * SC_TILE_BYTES;
            for (int i = end * 8 + lane; i < 128 * 8; i += 32) {
              reinterpret_cast<uint4 *>(tile)[i] = make_uint4(0u, 0u, 0u, 0u);
              reinterpret_cast<uint4 *>(tile + SC_HALF_BYTES)[i] = make_uint4(0u, 0u, 0u, 0u);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bk->full[s]));
          }
          ++qt;
        }
        kc += T.n_kt + T.n_p2;
      }
      if (SORTED && ic == 0 && half == 0) {
        const int place = score_order(a, first, bk->work, bk->order, pair_rows, lane);
        if (lane == 0) {
          bk->place = place;
          mbar_arrive(smem_u32(&bk->order_ready));
        }
      }
    }
  }

  // ---------------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, SC_TMEM_COLS);
  }
  // the block that leaves last puts the work counters back to zero for the next launch (every block
  // has drawn its last item by then: a block only gets here after a draw past the end)
  if (threadIdx.x == 0) {
    const unsigned int done = atomicAdd(a.work + 1, 1u);
    if (done == gridDim.x - 1) {
      a.work[0] = 0u;
      a.work[1] = 0u;
      __threadfence();
    }
  }
}

// r_j = (1 / (H |R|)) sum_h partial[b, h, j]: the mean over heads and ranking rows of the Eq. 4
// probabilities, heads added in ascending order.  grid (ceil(max_vis / 256), B).
__global__ void __launch_bounds__(256)
head_sum_kernel(const SampleDesc *__restrict__ desc, int H, int max_vis,
                const float *__restrict__ partial, float *__restrict__ rank_score) {
  pdl_enter();
  const int b = blockIdx.y;
  const SampleDesc d = desc[b];
  const int j = blockIdx.x * 256 + threadIdx.x;
  if (j >= max_vis) return;
  float tot = 0.f;
  if (d.valid && j < d.nv) {
    const float *p = partial + (size_t)b * H * max_vis + j;
    int hh = 0;
    for (; hh + 8 <= H; hh += 8) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = __ldcg(p + (size_t)(hh + e) * max_vis);
#pragma unroll
      for (int e = 0; e < 8; ++e) tot += v[e];
    }
    for (; hh < H; ++hh) tot += __ldcg(p + (size_t)hh * max_vis);
    tot *= 1.0f / ((float)H * (float)d.nr);
  }
  rank_score[(size_t)b * max_vis + j] = tot;
}

// =======================================================================================
// sim_kernel
//
// One block per (128 rows, sample, slice of the hidden dimension).  D = Row_tile Kept^T
// with M = 128 rows (see "row operand" below), N = n_tile kept slots per accumulator, K = this block's slice of
// the hidden size in steps of 64.
//   row operand:    either the dropped rows alone, fetched where they lie in `hidden` by the gather
//                   warps (16-byte asynchronous copies, written in the 128-byte-swizzled layout the
//                   tiled copies produce), so that only rows whose result is used are multiplied; or
//                   every visual row by plain tiled copies, the kept rows' results being thrown away.
//                   A gathered row costs the gather warps' 16-byte copies (their requests in flight bound them) what
//                   several rows cost the tiled path, so the host gathers only from a quarter of the span kept on, where the
//                   products saved outweigh it (the line and both sides' times stand at the rule in asap_api.cu).
// While the first
// accumulator is being built the epilogue warps also read every row tile from shared memory and
// add up the squares (the row norms of Sec. 4.2's cosine similarity).
//   one slice:      the epilogue scales column s by 1/||kept_s||, keeps the running maximum
//                   and the first slot attaining it, and writes, for rows that were dropped,
//                   the slot (or -1 if the cosine similarity is not above the threshold) and
//                   the similarity.
//   several slices: (small problems, to fill the machine) every block stores its partial dot
//                   products and partial squared norms; the block that finishes last for the
//                   row tile adds the slices in slice order and does the same epilogue.
// Rows past the last dropped token (the ragged tail of the last tile) repeat that token and are
// not written.  The thread that assigns a token sets its bit in the slot's row of member bits (a.member_bits), or, where
// those have no room, the block that finishes a sample's last row tile groups the dropped tokens by destination.
//   one pass:       (a.wide, gathered rows, or up to 384 slots of a batch too large for sim_pair_kernel) the accumulators of
//                   all slot tiles are live at once and a stage is one 64-column block of the rows
//                   plus the matching block of EVERY slot tile, so the visual rows are read from
//                   memory once instead of once per slot tile.
//   slot groups:    (a.groups > 1, one-pass layout, blockIdx.x = row tile * groups + group) more kept slots than tensor memory
//                   holds at once: every block takes one group of slot tiles in ONE pass over the hidden
//                   dimension and publishes its rows' best (value, slot); the block that finishes a row
//                   tile last takes the maximum over the groups (lowest slot among equals).  The blocks
//                   of a row tile are neighbours in launch order and stream the same rows at the same
//                   time, so the rows come from memory once and from L2 afterwards -- several passes in
//                   one block read them from memory every time, because the rows of all resident
//                   blocks together do not fit L2.
//   matrix mode:    (a.smat set) the row operand is the dense kept-row array too, and
//                   the epilogue writes the whole keep_k x keep_k cosine matrix of the sample,
//                   S[p][q] = <h_p, h_q> * (1/||h_p|| * 1/||h_q||), for the routing inside the
//                   kept set; `tmap_h` is then a map of the kept rows with a 128-row box (plain
//                   tiled copies, no gather).
// =======================================================================================
#ifndef SIM_GWARPS_N
#define SIM_GWARPS_N 4
#endif
constexpr int SIM_GWARPS = SIM_GWARPS_N;                // gather warps
constexpr int SIM_THREADS = 192 + 32 * SIM_GWARPS;      // copy warp, MMA warp, four epilogue warps, the gather warps
constexpr int SIM_A_BYTES = 128 * 128;           // 128 rows x 64 bf16
constexpr int SIM_BOOK_BYTES = 2048;
constexpr int SIM_MAX_STAGES = 8;
constexpr int SIM_B_STAGES = 4;

struct SimArgs {
  const SampleDesc *desc;
  int D, max_vis, keep_k, n_tile, n_nt, stages, splits, max_mt;
  int a_stages;              // gathered form and pair kernel: slots of the row ring (`stages` counts those of the kept-row ring)
  int wide;                  // 1: one pass, all slot tiles' accumulators live at once
  int groups;                // > 1: slot tiles dealt to `groups` blocks per row tile (n_nt counts one group's tiles)
  int cluster;               // 1: the `splits` slices of a row tile form a thread-block cluster (grid z) and add their
                             // partial products through distributed shared memory instead of `part`
  uint32_t tmem_cols;        // power of two >= 2 * n_tile: two accumulators
  float threshold;
  const int32_t *drop_idx;   // [B, max_vis-keep_k] dropped tokens, ascending: the row operand is gathered from them;
                             // nullptr: the row operand is every visual row (tiled copies), kept rows' results unused
  const int32_t *role;       // [B, max_vis] kept slot / -(dropped position + 1) of every visual token (all-rows form)
  const int32_t *drop_all;   // [B, max_vis-keep_k] the dropped tokens whatever the form (for member_meta), or nullptr
  const __nv_bfloat16 *hidden;   // [tokens, D] (the gather warps read the dropped rows from here)
  const float *kept_inv;     // [B*keep_k]   1/||kept row||, 0 for a zero row
  int32_t *assign;           // [B, max_vis-keep_k]
  float *best_sim;           // [B, max_vis-keep_k] or nullptr
  int32_t *seg;              // [B, keep_k+1]       CSR of assign, built by the last block of a sample; nullptr: not wanted
  int32_t *members;          // [B, max_vis-keep_k]
  unsigned int *counters;    // [B]            finished row tiles per sample
  unsigned int *tile_counters;  // [B, max_mt] finished slices per row tile
  float *part;               // [B, max_mt, splits, keep_k, 128] partial dot products (several slices only)
  float *ss_part;            // [B, max_mt, splits, 128]         partial squared norms
  float *smat;               // [B, keep_k, keep_k] or nullptr: matrix mode
  uint16_t *mask16;          // (pair kernel, matrix mode) [B, keep_k, mask_pitch] or nullptr: bit q of row p set where S[p][q] > threshold, q != p
  int mask_pitch;            // halfwords per row, even
  const float *salience;     // [B, max_vis] or nullptr: with member_meta, the merge weights the grouping copies
  int2 *member_meta;         // [B, max_vis-keep_k] or nullptr (see csr_block)
  uint32_t *member_bits;     // [B, keep_k, bit_words], zero, or nullptr: bit j of a slot's row is set where visual token j merges into it
  int bit_words;
  uint32_t *status;
  long long wait_limit;      // clock cycles a wait may take before the block gives up
};

__device__ __forceinline__ void set_member_bit(const SimArgs &a, int b, int slot, int v) {
  atomicOr(a.member_bits + ((size_t)b * a.keep_k + slot) * a.bit_words + (v >> 5), 1u << (v & 31));
}

struct SimBook {
  uint64_t full[SIM_MAX_STAGES], empty[SIM_MAX_STAGES], acc_full[2], acc_empty[2], mma_done;
  uint64_t full_b[SIM_B_STAGES], empty_b[SIM_B_STAGES];   // gathered form: the kept rows' own ring
  uint32_t tmem_base;
  int abort_flag;
  int is_last;
  int skip;                  // cluster form: an earlier similarity kernel of this call gave up
  int scan[33];
  int rows[128];             // packed row of each of the tile's dropped tokens (main mode)
};

static_assert(sizeof(SimBook) <= SIM_BOOK_BYTES, "similarity kernel bookkeeping exceeds its shared-memory slot");

__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}

// Running first-argmax of one tensor-memory lane over 32 accumulator columns, column e scaled by kinv[e] (shared memory,
// 16-byte aligned).  The chunk's maximum first (packed products, three-way maxima), then, only where some row of the warp has
// a new maximum, the lowest column that attains it: about three instructions per column instead of a chain of four and a
// global load (176 columns: 6000 -> 1600 clocks, on the path of a block that nothing overlaps).
__device__ __forceinline__ void sim_scan32(uint32_t taddr, const float *kinv, int slot0, float &best, int &best_slot) {
  uint32_t r[32];
  tmem_ld32(taddr, r);
  tmem_wait_ld();
  float v[32];
#pragma unroll
  for (int e = 0; e < 32; e += 4) {
    const ulonglong2 k = *reinterpret_cast<const ulonglong2 *>(kinv + e);
    f2_unpack(f2_mul(f2_pack(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), k.x), v[e], v[e + 1]);
    f2_unpack(f2_mul(f2_pack(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), k.y), v[e + 2], v[e + 3]);
  }
  float m[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) m[e] = max3(v[e], v[e + 4], v[e + 8]);
#pragma unroll
  for (int c = 12; c < 28; c += 8)
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = max3(m[e], v[c + e], v[c + 4 + e]);
#pragma unroll
  for (int e = 0; e < 4; ++e) m[e] = fmaxf(m[e], v[28 + e]);
  const float mx = fmaxf(max3(m[0], m[1], m[2]), m[3]);
  if (__any_sync(0xffffffffu, mx > best)) {
    int at = 31;
#pragma unroll
    for (int e = 30; e >= 0; --e) at = v[e] == mx ? e : at;
    if (mx > best) { best = mx; best_slot = slot0 + at; }
  }
}

template <int V>
struct IntC {
  static constexpr int value = V;
};

constexpr int SIM_THREADS_TILED = 192;                  // without gather warps: two such blocks fit an SM

template <bool GATHER>
__global__ void __launch_bounds__(GATHER ? SIM_THREADS : SIM_THREADS_TILED, 1)
sim_kernel(const __grid_constant__ CUtensorMap tmap_h, const __grid_constant__ CUtensorMap tmap_kept,
           SimArgs a) {
  // (the wait for the preceding kernel comes after this block's set-up, which reads nothing that kernel
  // writes: descriptors and status word are older; barriers, tensor memory and the cluster's first barrier
  // are then ready when the kept rows are)
  extern __shared__ uint8_t smem_raw[];
  // the groups of a row tile are neighbours in launch order (blockIdx.x = row tile * groups + group)
  const int mt = blockIdx.x / a.groups, b = blockIdx.y;
  const int z = blockIdx.z;                              // slice of the hidden dimension
  const int gz = blockIdx.x - mt * a.groups;             // group of slot tiles
  const int tile0 = gz * a.n_nt;                         // first slot tile of this block
  const SampleDesc d = a.desc[b];
  if (!d.valid) {
    pdl_wait();         // (should all blocks leave here, the grid must not complete before the preceding one)
    return;
  }
  const int nd = d.nv - a.keep_k;                        // dropped tokens of this sample
  constexpr bool gather = GATHER;                        // a.drop_idx given, not matrix mode
  const int n_rows = a.smat ? a.keep_k : (gather ? nd : d.nv);   // rows of the row operand
  if (mt * 128 >= max(n_rows, 1)) return;
  // (in the cluster form the blocks of a cluster must leave together: decided below, by the cluster's first block)
  if (!a.cluster && (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_SIM_TIMEOUT)) {
    pdl_wait();
    return;
  }
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
  // a stage holds two adjacent 64-column blocks (256 contiguous bytes of every row):
  // [ rows, block 0 | rows, block 1 | kept, block 0 | kept, block 1 ]
  const int b_bytes = a.n_tile * 128;
  const int stage_bytes = a.wide ? SIM_A_BYTES + a.n_nt * b_bytes : 2 * (SIM_A_BYTES + b_bytes);
  // (gathered form: a ring of a_stages row tiles, then one of `stages` kept-row tiles, one 64-column block each)
  const int ring_bytes = GATHER ? a.a_stages * SIM_A_BYTES + a.stages * a.n_nt * b_bytes : a.stages * stage_bytes;
  SimBook *bk = reinterpret_cast<SimBook *>(base_ptr + (size_t)ring_bytes);
  if (n_rows <= 0) {
    // nothing was dropped in this sample: only the (empty) grouping has to be written
    pdl_enter();
    if (z == 0 && gz == 0 && a.seg) csr_block(d, b, a.max_vis, a.keep_k, a.assign, a.seg, a.members, reinterpret_cast<int *>(base_ptr), bk->scan, a.drop_all, a.salience, a.member_meta);
    return;
  }

  if (threadIdx.x == 0) {
    if (GATHER) {
      for (int s = 0; s < a.stages; ++s) {
        mbar_init(smem_u32(&bk->full_b[s]), 1);
        mbar_init(smem_u32(&bk->empty_b[s]), 1);
      }
    }
    for (int s = 0; s < (GATHER ? a.a_stages : a.stages); ++s) {
      mbar_init(smem_u32(&bk->full[s]), GATHER ? 32 * SIM_GWARPS : 1);      // every gather thread, or the copy warp's announcement
      mbar_init(smem_u32(&bk->empty[s]), 5);      // the MMAs that read the stage + four epilogue warps
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&bk->acc_full[i]), 1);
      mbar_init(smem_u32(&bk->acc_empty[i]), 4);
    }
    mbar_init(smem_u32(&bk->mma_done), 1);
    bk->abort_flag = 0;
    bk->is_last = 0;
    bk->skip = (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_SIM_TIMEOUT) ? 1 : 0;
    fence_barrier_init();
  }
  if (a.cluster) {
    cluster_sync_all();
    if (ld_cluster_s32(cluster_map(smem_u32(&bk->skip), 0))) {
      cluster_sync_all();                                // the first block's shared memory has been read by all
      pdl_wait();
      return;
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bk->tmem_base), a.tmem_cols);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  pdl_enter();
  const uint32_t tmem_base = bk->tmem_base;
  WaitCtx wc{&bk->abort_flag, a.status, STATUS_SIM_TIMEOUT, a.wait_limit};
  // cluster form, in the tile ring once it is free: this slice's partial products [keep_k][128]; per quarter
  // of this block's share of the slots the rows' best (value [4][128], slot [4][128]); this slice's partial squared
  // norms [128]; and, filled by all blocks in the cluster's first block, every block's best (value, slot)
  // ([splits][128] each)
  const int cl_per = (a.keep_k + a.splits - 1) / a.splits;
  float *cl_p = reinterpret_cast<float *>(base_ptr);
  float *cl_wv = cl_p + (size_t)a.keep_k * 128;
  int *cl_ws = reinterpret_cast<int *>(cl_wv + 4 * 128);
  float *cl_ss = reinterpret_cast<float *>(cl_ws + 4 * 128);
  float *cl_bv = cl_ss + 128;
  int *cl_bs = reinterpret_cast<int *>(cl_bv + a.splits * 128);
  // steps of this slice: 128 columns each, or 64 in the one-pass layout
  const int n_kb = a.wide ? (a.D / 64) / a.splits : (a.D / 128) / a.splits;
  const int kb0 = z * n_kb;
  const int total_it = a.wide ? n_kb : a.n_nt * n_kb;

  if (warp == 0) {
    // ---- copy warp: the kept-row tiles (and, in matrix mode, the row operand) by tiled copies (converged, see tma_load_2d_w)
    const uint32_t leader = warp_leader();
    if (leader) {
      tma_prefetch_desc(&tmap_h);
      tma_prefetch_desc(&tmap_kept);
    }
    const int row_b = b * a.keep_k;
    // tiled row operand: rows of the dense kept array (matrix mode) or of the image span
    const int row_a = a.smat ? row_b + mt * 128 : d.row0 + d.v0 + mt * 128;
    const int tx_bytes = gather ? a.n_nt * b_bytes : stage_bytes;
    // every block walks its k-blocks from a different starting point, so that at any moment
    // the blocks read different 128-byte columns of the rows and spread over the memory channels
    const int rot = (mt * 5 + b * 3) % n_kb;
    int issued = 0, nt = 0, kr = 0, kb = kb0 + rot;           // slot tile, step of its pass, column step
    RingPos r;
    for (int it = 0; it < total_it; ++it) {
      const uint32_t full = smem_u32(GATHER ? &bk->full_b[r.slot] : &bk->full[r.slot]);
      if (it >= a.stages) mbar_wait_warp(smem_u32(GATHER ? &bk->empty_b[r.slot] : &bk->empty[r.slot]), r.phase ^ 1u, wc);
      if (__shfl_sync(0xffffffffu, bk->abort_flag, 0)) break;
      const uint32_t dst = GATHER ? base + a.a_stages * SIM_A_BYTES + r.slot * a.n_nt * b_bytes - SIM_A_BYTES : base + r.slot * stage_bytes;
      mbar_expect_tx_w(full, tx_bytes, leader);
      if (GATHER || a.wide) {
        if (!gather) tma_load_2d_w(dst, &tmap_h, full, kb * 64, row_a, leader);
        for (int t = 0; t < a.n_nt; ++t)
          tma_load_2d_w(dst + SIM_A_BYTES + t * b_bytes, &tmap_kept, full, kb * 64, row_b + (tile0 + t) * a.n_tile, leader);
      } else {
        tma_load_2d_w(dst, &tmap_h, full, kb * 128, row_a, leader);
        tma_load_2d_w(dst + SIM_A_BYTES, &tmap_h, full, kb * 128 + 64, row_a, leader);
        tma_load_2d_w(dst + 2 * SIM_A_BYTES, &tmap_kept, full, kb * 128, row_b + nt * a.n_tile, leader);
        tma_load_2d_w(dst + 2 * SIM_A_BYTES + b_bytes, &tmap_kept, full, kb * 128 + 64, row_b + nt * a.n_tile, leader);
      }
      issued = it + 1;
      r.step(a.stages);
      if (++kb == kb0 + n_kb) kb = kb0;
      if (++kr == n_kb) { kr = 0; ++nt; kb = kb0 + rot; }
    }
    // drain: the last fill of every stage must have landed before the block leaves
    for (int s = 0; s < a.stages; ++s) {
      if (issued > s) {
        const int last = ((issued - 1 - s) / a.stages) * a.stages + s;
        mbar_wait_drain(smem_u32(GATHER ? &bk->full_b[s] : &bk->full[s]), (last / a.stages) & 1, TC_WAIT_LIMIT);
      }
    }
    __syncwarp();
    if (a.cluster) { cluster_sync_all(); cluster_sync_all(); }   // the two barriers of the epilogue warps' reduction
  } else if (warp >= 6) {
    // ---- gather warps (main mode): warp g fetches its share of the tile's rows (128 / SIM_GWARPS hidden rows
    // of dropped tokens), one stage's columns at a time.  A warp instruction covers whole rows
    // (2 rows x 256 bytes, or 4 rows x 128 bytes in the one-pass layout), each lane one 16-byte chunk,
    // written where the tiled copies would put it: row r of a 64-column block is 128 bytes at
    // r * 128, its chunk c at position c ^ (r & 7).  Every lane's copies of a stage arrive on the stage's
    // barrier by themselves when they have landed, so the warps only ever wait for a free stage.  Few
    // threads with many copies each: every thread costs the barrier one arrival per stage, and 128
    // arrivals per stage were measured to hold the whole pipeline back.
    if (gather) {
      const int g = warp - 6;
      constexpr int RW = 128 / SIM_GWARPS;                // rows of the tile per gather warp
      const int c = lane & 7, rsub = lane >> 3;           // 16-byte chunk of the 128-byte piece, row of the group of four
      const int32_t *drop_b = a.drop_idx + (size_t)b * (a.max_vis - a.keep_k);
      for (int r = g * RW + lane; r < (g + 1) * RW; r += 32) {
        const int dp = min(mt * 128 + r, nd - 1);        // the ragged tail repeats the last dropped token
        bk->rows[r] = d.row0 + d.v0 + min(max(__ldg(drop_b + dp), 0), d.nv - 1);
      }
      __syncwarp();
      const uint8_t *src[RW / 4];
#pragma unroll
      for (int i = 0; i < RW / 4; ++i)
        src[i] = reinterpret_cast<const uint8_t *>(a.hidden) + (size_t)bk->rows[g * RW + i * 4 + rsub] * ((size_t)a.D * 2) + c * 16;
      const uint32_t dst0 = base + (g * RW + rsub) * 128;
      int kb = kb0 + (mt * 5 + b * 3) % n_kb;
      RingPos r;
      for (int it = 0; it < total_it; ++it) {
        // (every lane waits: each overwrites rows that the epilogue warps have read and the MMAs multiplied)
        if (it >= a.a_stages) mbar_wait_warp(smem_u32(&bk->empty[r.slot]), r.phase ^ 1u, wc);
        if (__shfl_sync(0xffffffffu, bk->abort_flag, 0)) break;
        const uint32_t dst = dst0 + r.slot * SIM_A_BYTES;
#pragma unroll
        for (int i = 0; i < RW / 4; ++i)                   // (row r of a block: its chunk c at position c ^ (r & 7))
          cp_async16(dst + i * 512 + (((c ^ ((i * 4 + rsub) & 7))) << 4), src[i] + (size_t)kb * 128);
        cp_async_arrive_on(smem_u32(&bk->full[r.slot]));  // this lane's share of the tile, once it has landed
        r.step(a.a_stages);
        if (++kb == kb0 + n_kb) kb = kb0;
      }
      cp_async_commit();
      cp_async_wait<0>();                                 // nothing of this thread's is in flight when the block leaves
    }
  } else if (warp == 1) {
    // ---- MMA issuer: the whole warp walks the loop and stays converged (see warp_leader).  After an abort its waits return
    // at once and it goes on multiplying whatever lies in the block's own memory: nothing of it is used.
    const uint32_t leader = warp_leader();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
    const uint32_t idesc = umma_idesc_bf16(128, a.n_tile);
    const uint64_t desc0 = umma_desc_sw128(base);
    int it = 0;
    if (GATHER) {
      const uint64_t bdesc0 = umma_desc_sw128(base + a.a_stages * SIM_A_BYTES);
      RingPos ra, rb;
      for (int kb = 0; kb < n_kb; ++kb) {
        mbar_wait_warp(smem_u32(&bk->full[ra.slot]), ra.phase, wc);
        mbar_wait_warp(smem_u32(&bk->full_b[rb.slot]), rb.phase, wc);
        fence_proxy_async();                   // the gathered rows were written by ordinary asynchronous copies
        tc_fence_after();
        const uint64_t da = desc0 + (uint32_t)(ra.slot * SIM_A_BYTES) / 16, db = bdesc0 + (uint32_t)(rb.slot * a.n_nt * b_bytes) / 16;
        for (int t = 0; t < a.n_nt; ++t)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc_mma_bf16_w(tm + t * a.n_tile, da + kk * 2, db + t * (b_bytes / 16) + kk * 2, idesc, (kb > 0 || kk > 0) ? 1u : 0u, leader);
        tc_commit_w(smem_u32(&bk->empty_b[rb.slot]), leader);
        tc_commit_w(smem_u32(&bk->empty[ra.slot]), leader);
        ra.step(a.a_stages);
        rb.step(a.stages);
      }
      tc_commit_w(smem_u32(&bk->acc_full[0]), leader);
    } else {
      if (a.wide) {
        for (int kb = 0; kb < n_kb; ++kb) {
          const int s = kb % a.stages;
          mbar_wait_warp(smem_u32(&bk->full[s]), (kb / a.stages) & 1, wc);
          tc_fence_after();
          const uint64_t da = desc0 + (uint32_t)(s * stage_bytes) / 16, db = da + SIM_A_BYTES / 16;
          for (int t = 0; t < a.n_nt; ++t)
  #pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              tc_mma_bf16_w(tm + t * a.n_tile, da + kk * 2, db + t * (b_bytes / 16) + kk * 2, idesc, (kb > 0 || kk > 0) ? 1u : 0u, leader);
          tc_commit_w(smem_u32(&bk->empty[s]), leader);
          if (a.smat && leader) mbar_arrive_n(smem_u32(&bk->empty[s]), 4);
        }
        tc_commit_w(smem_u32(&bk->acc_full[0]), leader);
      }
      for (int nt = 0; nt < (a.wide ? 0 : a.n_nt); ++nt) {
        const int buf = nt & 1;
        if (nt >= 2) mbar_wait_warp(smem_u32(&bk->acc_empty[buf]), ((nt >> 1) - 1) & 1, wc);
        const uint32_t dcol = tm + buf * (a.tmem_cols >> 1);
        for (int kb = 0; kb < n_kb; ++kb, ++it) {
          const int s = it % a.stages;
          mbar_wait_warp(smem_u32(&bk->full[s]), (it / a.stages) & 1, wc);
          tc_fence_after();
          const uint64_t da = desc0 + (uint32_t)(s * stage_bytes) / 16, db = da + 2 * SIM_A_BYTES / 16;
  #pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            tc_mma_bf16_w(dcol, da + (kk >> 2) * (SIM_A_BYTES / 16) + (kk & 3) * 2, db + (kk >> 2) * (b_bytes / 16) + (kk & 3) * 2, idesc,
                          (kb > 0 || kk > 0) ? 1u : 0u, leader);
          tc_commit_w(smem_u32(&bk->empty[s]), leader);
          // after the first accumulator the epilogue warps no longer read the stages
          if ((nt > 0 || a.smat) && leader) mbar_arrive_n(smem_u32(&bk->empty[s]), 4);
        }
        tc_commit_w(smem_u32(&bk->acc_full[buf]), leader);
      }
    }
    // every MMA this warp issued has completed before tensor memory is given back: after an abort the
    // epilogue warps no longer wait for the accumulators, so nothing else would hold the block until then
    tc_commit_w(smem_u32(&bk->mma_done), leader);
    mbar_wait_drain(smem_u32(&bk->mma_done), 0, TC_WAIT_LIMIT);
    __syncwarp();
    if (a.cluster) { cluster_sync_all(); cluster_sync_all(); }
  } else {
    const int quarter = warp & 3;
    const int lrow = quarter * 32 + lane;
    const int v = mt * 128 + lrow;                       // this thread's row: dropped position (kept slot in matrix mode)
    const float *kinv = a.kept_inv + (size_t)b * a.keep_k;
    // ---- squared norm of this thread's row, from the row tiles of the first accumulator's pass.
    // Row r of a tile is 128 bytes; its 16-byte chunk c sits at chunk position c ^ (r & 7).
    float ssq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int it = 0; it < (a.smat ? 0 : n_kb); ++it) {
      const int ring = GATHER ? a.a_stages : a.stages, s = it % ring;
      mbar_wait(smem_u32(&bk->full[s]), (it / ring) & 1, wc);
      if (!bk->abort_flag) {
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {
          if (hb == 1 && (GATHER || a.wide)) break;      // one 64-column block of the rows per stage
          const uint4 *row = reinterpret_cast<const uint4 *>(base_ptr + (size_t)s * (GATHER ? SIM_A_BYTES : stage_bytes) +
                                                             hb * SIM_A_BYTES + lrow * 128);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const uint4 x = row[c ^ (lrow & 7)];
            float f[8];
            unpack8(x, f);
#pragma unroll
            for (int e = 0; e < 8; ++e) ssq[c] = fmaf(f[e], f[e], ssq[c]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bk->empty[s]));
    }
    const float ss = ((ssq[0] + ssq[1]) + (ssq[2] + ssq[3])) + ((ssq[4] + ssq[5]) + (ssq[6] + ssq[7]));

    float best = -INFINITY;
    int best_slot = 0;
    float *part = nullptr;
    if (a.cluster) {
      // the four epilogue warps are done reading the row tiles for the norms: from here on the ring only
      // holds stages the MMAs still read, and those are complete once acc_full has been passed
      asm volatile("bar.sync 1, 128;" ::: "memory");
      part = cl_p;
    } else if (a.splits > 1) {
      const size_t tile = ((size_t)b * a.max_mt + mt) * a.splits + z;
      part = a.part + tile * (size_t)a.keep_k * 128;
      a.ss_part[tile * 128 + lrow] = ss;
    }
    // one pass over the rows and no partial sums: the inverse norms of the slots wait in registers and go to the tile ring
    // once the last MMA has read it
    const bool scan_smem = !part && !a.smat && (a.wide || a.n_nt == 1);
    float *sk = reinterpret_cast<float *>(base_ptr);
    float kreg[4] = {0.f, 0.f, 0.f, 0.f};
    if (scan_smem) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int c = e * 128 + lrow, slot = tile0 * a.n_tile + c;
        if (c < a.n_nt * a.n_tile && slot < a.keep_k) kreg[e] = kinv[slot];
      }
    }
    for (int nt = 0; nt < a.n_nt; ++nt) {
      const int buf = a.wide ? 0 : (nt & 1);
      mbar_wait(smem_u32(&bk->acc_full[buf]), a.wide ? 0 : ((nt >> 1) & 1), wc);
      tc_fence_after();
      if (scan_smem && nt == 0) {
        asm volatile("bar.sync 1, 128;" ::: "memory");     // the other warps have read their rows for the norms
#pragma unroll
        for (int e = 0; e < 4; ++e) sk[e * 128 + lrow] = kreg[e];
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) +
                             (a.wide ? nt * a.n_tile : buf * (a.tmem_cols >> 1));
      const int slot0 = (tile0 + nt) * a.n_tile;
      const int ncol = min(a.n_tile, a.keep_k - slot0);   // kept slots in this accumulator (none in a group's ragged end)
      int c0 = 0;
      if (!a.smat || part) {
        // 32 columns per tensor-memory wait while they last (see sim_pair_kernel)
#pragma unroll 1
        for (; c0 + 32 <= ncol; c0 += 32) {
          if (scan_smem) {
            sim_scan32(taddr + c0, sk + nt * a.n_tile + c0, slot0 + c0, best, best_slot);
            continue;
          }
          uint32_t r[32];
          tmem_ld32(taddr + c0, r);
          tmem_wait_ld();
          if (part) {
#pragma unroll
            for (int e = 0; e < 32; ++e) part[(size_t)(slot0 + c0 + e) * 128 + lrow] = __uint_as_float(r[e]);
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              const int slot = slot0 + c0 + e;
              const float val = __uint_as_float(r[e]) * kinv[slot];
              if (val > best) { best = val; best_slot = slot; }
            }
          }
        }
      }
#pragma unroll 1
      for (int c = c0; c < ncol; c += 16) {
        uint32_t r[16];
        tmem_ld16(taddr + c, r);
        tmem_wait_ld();
        if (a.smat && !part) {
          if (v < a.keep_k && !bk->abort_flag) {
            const float inv_p = kinv[v];
            float *srow = a.smat + ((size_t)b * a.keep_k + v) * a.keep_k + slot0 + c;
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (c + e < ncol) srow[e] = __uint_as_float(r[e]) * (inv_p * kinv[slot0 + c + e]);
          }
        } else if (part) {
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (c + e < ncol) part[(size_t)(slot0 + c + e) * 128 + lrow] = __uint_as_float(r[e]);
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int slot = slot0 + c + e;
            if (c + e < ncol) {
              const float val = __uint_as_float(r[e]) * kinv[slot];
              if (val > best) { best = val; best_slot = slot; }
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bk->acc_empty[buf]));
    }
    float ss_tot = ss;
    bool finalize = true;
    if (a.cluster) {
      // ---- the slices of this row tile are the blocks of one cluster.  Block r adds, in slice order, the
      // partial products of ITS share of the kept slots, read from every block's shared memory: warp q takes
      // every fourth slot of the share, a lane four neighbouring rows (one 16-byte load per slice).  The
      // warps' bests per row are merged (larger value, lower slot among equals), handed to the cluster's
      // first block, and that block takes the maximum over the blocks in ascending slots.
      const int rank = (int)cluster_cta_rank(), S = a.splits;
      // (every block keeps its own norms until the barrier: the first block's ring may still be multiplied from)
      cl_ss[lrow] = ss;
      cluster_sync_all();
      if (rank == 0) {
        ss_tot = 0.f;
        for (int r2 = 0; r2 < S; ++r2) ss_tot += ld_cluster_f32(cluster_map(smem_u32(cl_ss), (uint32_t)r2) + (uint32_t)lrow * 4u);
      }
      const int s_lo = min(a.keep_k, rank * cl_per), n_mine = min(a.keep_k, s_lo + cl_per) - s_lo;
      uint32_t pz[8];
#pragma unroll
      for (int zz = 0; zz < 8; ++zz)
        pz[zz] = cluster_map(smem_u32(cl_p), (uint32_t)min(zz, S - 1)) + (uint32_t)lane * 16u;
      float wb[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      int wsl[4] = {0, 0, 0, 0};
      // (the loads of U slots are in flight together: with one slot's loads at a time the adding was a chain of round
      // trips of 700 clocks, 6000-7000 in all)
      auto add_slots = [&](auto uc, int i0) {
        constexpr int U = decltype(uc)::value, Z = 8 / U;      // slots in flight, slices at most
        float4 x[U][Z];
        float ks[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int slot = min(s_lo + i0 + 4 * u, a.keep_k - 1);
          ks[u] = kinv[slot];
#pragma unroll
          for (int zz = 0; zz < Z; ++zz)
            if (zz < S) x[u][zz] = ld_cluster_v4f32(pz[zz] + (uint32_t)slot * 512u);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (i0 + 4 * u >= n_mine) continue;
          const int slot = s_lo + i0 + 4 * u;
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int zz = 0; zz < Z; ++zz)
            if (zz < S) { acc[0] += x[u][zz].x; acc[1] += x[u][zz].y; acc[2] += x[u][zz].z; acc[3] += x[u][zz].w; }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (a.smat) {
              const int vr = mt * 128 + lane * 4 + j;
              if (vr < a.keep_k && !bk->abort_flag)
                a.smat[((size_t)b * a.keep_k + vr) * a.keep_k + slot] = acc[j] * (kinv[vr] * ks[u]);
            } else {
              const float val = acc[j] * ks[u];
              if (val > wb[j]) { wb[j] = val; wsl[j] = slot; }
            }
          }
        }
      };
      if (S <= 2)
        for (int i = quarter; i < n_mine; i += 16) add_slots(IntC<4>(), i);
      else if (S <= 4)
        for (int i = quarter; i < n_mine; i += 8) add_slots(IntC<2>(), i);
      else
        for (int i = quarter; i < n_mine; i += 4) add_slots(IntC<1>(), i);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        cl_wv[quarter * 128 + lane * 4 + j] = wb[j];
        cl_ws[quarter * 128 + lane * 4 + j] = wsl[j];
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      for (int q2 = 0; q2 < 4; ++q2) {
        const float val = cl_wv[q2 * 128 + lrow];
        const int sl = cl_ws[q2 * 128 + lrow];
        if (val > best || (val == best && val > -INFINITY && sl < best_slot)) { best = val; best_slot = sl; }
      }
      st_cluster_f32(cluster_map(smem_u32(cl_bv), 0) + (uint32_t)(rank * 128 + lrow) * 4u, best);
      st_cluster_s32(cluster_map(smem_u32(cl_bs), 0) + (uint32_t)(rank * 128 + lrow) * 4u, best_slot);
      cluster_sync_all();
      finalize = rank == 0;
      if (finalize) {
        best = -INFINITY;
        best_slot = 0;
        for (int r2 = 0; r2 < S; ++r2) {                    // ascending slots: the first maximum stays
          const float val = cl_bv[r2 * 128 + lrow];
          if (val > best) { best = val; best_slot = cl_bs[r2 * 128 + lrow]; }
        }
      }
    } else if (a.splits > 1) {
      // publish this slice; the last slice to arrive for the row tile reduces all of them
      __threadfence();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 2 && lane == 0) {
        unsigned int *cnt = a.tile_counters + (size_t)b * a.max_mt + mt;
        const unsigned int old = atomicAdd(cnt, 1u);
        bk->is_last = (old == (unsigned int)(a.splits - 1));
        if (bk->is_last) *cnt = 0u;
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      finalize = bk->is_last != 0;
      if (finalize) {
        __threadfence();
        const size_t tile0 = ((size_t)b * a.max_mt + mt) * a.splits;
        ss_tot = 0.f;
        for (int zz = 0; zz < a.splits; ++zz) ss_tot += __ldcg(a.ss_part + (tile0 + zz) * 128 + lrow);
        const float *p0 = a.part + tile0 * (size_t)a.keep_k * 128 + lrow;
        const size_t zstride = (size_t)a.keep_k * 128;
        for (int s0 = 0; s0 < a.keep_k; s0 += 16) {     // 16 slots x all slices in flight per thread
          float acc[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) acc[e] = 0.f;
          for (int zz = 0; zz < a.splits; zz += 4) {    // 64 loads in flight per thread
            float x[4][16];
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
              for (int e = 0; e < 16; ++e)
                x[t][e] = (zz + t < a.splits && s0 + e < a.keep_k)
                              ? __ldcg(p0 + (zz + t) * zstride + (size_t)(s0 + e) * 128) : 0.f;
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
              for (int e = 0; e < 16; ++e) acc[e] += x[t][e];
          }
          if (a.smat) {
            if (v < a.keep_k && !bk->abort_flag) {
              const float inv_p = kinv[v];
              float *srow = a.smat + ((size_t)b * a.keep_k + v) * a.keep_k + s0;
#pragma unroll
              for (int e = 0; e < 16; ++e)
                if (s0 + e < a.keep_k) srow[e] = acc[e] * (inv_p * kinv[s0 + e]);
            }
            continue;
          }
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int slot = s0 + e;
            if (slot < a.keep_k) {
              const float val = acc[e] * kinv[slot];
              if (val > best) { best = val; best_slot = slot; }
            }
          }
        }
      }
    }
    if (a.groups > 1) {
      // publish this group's best (value, slot); the last group to arrive for the row tile combines them
      const size_t tile = ((size_t)b * a.max_mt + mt) * a.groups;
      a.part[(tile + gz) * 256 + lrow] = best;
      reinterpret_cast<int *>(a.part)[(tile + gz) * 256 + 128 + lrow] = best_slot;
      __threadfence();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 2 && lane == 0) {
        unsigned int *cnt = a.tile_counters + (size_t)b * a.max_mt + mt;
        const unsigned int old = atomicAdd(cnt, 1u);
        bk->is_last = (old == (unsigned int)(a.groups - 1));
        if (bk->is_last) *cnt = 0u;
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      finalize = bk->is_last != 0;
      if (finalize) {
        __threadfence();
        best = -INFINITY;
        best_slot = 0;
        for (int g2 = 0; g2 < a.groups; ++g2) {           // ascending slots: the first maximum stays
          const float val = __ldcg(a.part + (tile + g2) * 256 + lrow);
          const int slot = __ldcg(reinterpret_cast<const int *>(a.part) + (tile + g2) * 256 + 128 + lrow);
          if (val > best) { best = val; best_slot = slot; }
        }
      }
    }
    if (a.smat) finalize = false;
    // the dropped position of this thread's row: the row index itself, or looked up for a visual row
    int dp = -1;
    if (finalize && v < n_rows) {
      if (gather) dp = v;
      else { const int role = a.role[(size_t)b * a.max_vis + v]; dp = role < 0 ? -role - 1 : -1; }
    }
    if (dp >= 0 && dp < nd && !bk->abort_flag) {
      const bool zero_row = !(ss_tot >= 1e-24f);        // ||h|| < 1e-12: similarity 0 to every slot
      const float sim = zero_row ? 0.f : best * rsqrtf(ss_tot);
      const int slot = zero_row ? 0 : best_slot;
      const size_t o = (size_t)b * (a.max_vis - a.keep_k) + dp;
      a.assign[o] = (sim > a.threshold) ? slot : -1;
      if (a.best_sim) a.best_sim[o] = sim;
      if (a.member_bits && sim > a.threshold) set_member_bit(a, b, slot, gather ? min(max(__ldg(a.drop_idx + o), 0), d.nv - 1) : v);
    }
    if (warp == 2 && lane == 0) bk->is_last = finalize ? 1 : 0;
    if (a.seg) __threadfence();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, a.tmem_cols);
  }
  if (a.smat) return;
  if (!a.seg || (!bk->is_last && (a.splits > 1 || a.groups > 1))) return;   // (or a slice / group that did not finalize its row tile)
  __syncthreads();
  // (no member bits) the block that finishes the sample's last row tile groups the dropped tokens by destination
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int n_mt = (unsigned int)((n_rows + 127) / 128);
    const unsigned int old = atomicAdd(a.counters + b, 1u);
    bk->is_last = (old == n_mt - 1u);
    if (bk->is_last) a.counters[b] = 0u;
  }
  __syncthreads();
  if (!bk->is_last) return;
  __threadfence();
  // the tile ring is free: every copy has landed and every MMA that read it has completed
  csr_block(d, b, a.max_vis, a.keep_k, a.assign, a.seg, a.members, reinterpret_cast<int *>(base_ptr),
            bk->scan, a.drop_all, a.salience, a.member_meta);
}

// =======================================================================================
// sim_pair_kernel
//
// The all-rows form of sim_kernel for batches large enough to fill the machine without slicing the
// hidden dimension.  A block of sim_kernel streams 128 rows and n_tile kept rows per 64 columns, (128 + n_tile) * 128 bytes
// for 128 * n_tile * 64 products, more than an SM takes in (about 92 bytes per clock with converged issue) while the tensor
// pipe works on them at small n_tile.  This kernel multiplies TWO row tiles against each stage's kept rows -- (256 + n_tile) *
// 128 bytes for twice the products, 30 % fewer bytes per product at n_tile = 192; tensor memory (512 columns = 2 tiles x
// n_tile <= 256) allows no larger block.  (MMAs spanning a pair of CTAs, each loading half of the kept rows, ran 30 % slower
// than this form when both issued from one lane under a branch.)
// It makes a single pass over the hidden dimension: the kept slots are dealt in groups of n_tile <= 256 to `groups` blocks per
// pair of row tiles (blockIdx.x = pair * groups + group).  The blocks of a pair are neighbours in
// launch order and stream the same rows at the same pace, so the rows come from memory once and
// from L2 for the other groups.  Accumulators: row tile t at tensor-memory column t * n_tile.
// Rows and kept rows have rings of their own: the rows come from memory and want as many bytes in flight as there is room for,
// the kept rows come from L2.  Every block adds up its rows' squares over its group's share of the 64-column blocks, and
// publishes its rows' best (value, slot) and that sum (one ring, and all the squares in group 0: 8 x 2304 with 320 kept 58 -> 49.5
// us, 8 x 1536 with 340 56 -> 49, 12 x 577-2881 with 145 56.5 -> 50, 64 x 2880 793 -> 775); the block that finishes a pair last takes the maximum over the
// groups (lowest slot among equals), looks up which rows were dropped and writes their assignment.
// The assignment leaves as member bits or a grouping, as in sim_kernel.
// Matrix mode (a.smat set): the row operand is the dense kept-row array too (`tmap_h` maps it with a 128-row box)
// and every block writes its 256 x n_tile piece of the sample's keep_k x keep_k cosine matrix; nothing else.  The matrix is
// symmetric: blocks that lie below the diagonal as a whole leave, and the blocks of the mirrored places write their pieces too
// (24 x 576 slots: 6 of 9 blocks per sequence are left, one round of blocks instead of two: 100 -> 64 us).
// =======================================================================================
constexpr int SIMP_THREADS = 352;                // copy warp (rows), MMA warp, two groups of four epilogue warps, copy warp (kept rows)
constexpr int SIMP_MAX_ROWS = 12, SIMP_MAX_KEPT = 4;   // slots of the two rings

struct SimPairBook {
  uint64_t full[SIMP_MAX_ROWS], empty[SIMP_MAX_ROWS], full_b[SIMP_MAX_KEPT], empty_b[SIMP_MAX_KEPT], acc_full, mma_done, norm_go;
  uint32_t tmem_base;
  int abort_flag;
  int is_last;
  int scan[33];
  alignas(16) float kinv[256];   // 1/||kept row|| of this block's slots
};

static_assert(sizeof(SimPairBook) <= SIM_BOOK_BYTES, "pair kernel bookkeeping exceeds its shared-memory slot");

__global__ void __launch_bounds__(SIMP_THREADS, 1)
sim_pair_kernel(const __grid_constant__ CUtensorMap tmap_h, const __grid_constant__ CUtensorMap tmap_kept,
                SimArgs a) {
  // (the wait for the preceding kernel comes after the block's set-up, which reads nothing that kernel writes)
  extern __shared__ uint8_t smem_raw[];
  const int pr = blockIdx.x / a.groups, b = blockIdx.y;
  const int gz = blockIdx.x - pr * a.groups;             // group of kept slots
  const SampleDesc d = a.desc[b];
  if (!d.valid) {
    pdl_wait();         // (as in sim_kernel)
    return;
  }
  const int nd = d.nv - a.keep_k;
  const int n_rows = a.smat ? a.keep_k : d.nv;           // matrix mode: the row operand is the dense kept-row array
  if (pr * 256 >= n_rows) return;
  if (a.smat && (gz + 1) * a.n_tile <= pr * 256) {       // below the diagonal: written by the block of the mirrored place
    pdl_wait();
    return;
  }
  if (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_SIM_TIMEOUT) {
    pdl_wait();
    return;
  }
  const bool two = pr * 256 + 128 < n_rows;              // the pair's second row tile holds visual rows
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t *base_ptr = smem_raw + (base - smem_u32(smem_raw));
  // a ring of row tiles (row tile 0, row tile 1, row tile 0 of the next 64 columns, ...) and one of the kept rows' tiles
  const int b_bytes = a.n_tile * 128;
  const int ring_bytes = a.a_stages * SIM_A_BYTES + a.stages * b_bytes;
  const uint32_t base_b = base + a.a_stages * SIM_A_BYTES;
  SimPairBook *bk = reinterpret_cast<SimPairBook *>(base_ptr + (size_t)ring_bytes);

  // the epilogue warps read this group's range of 64-column blocks of their row tile (for the row norms; matrix mode takes them
  // from kept_inv)
  const int n_kb = a.D / 64;
  const int norm_lo = n_kb * gz / a.groups, norm_hi = n_kb * (gz + 1) / a.groups;
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.a_stages; ++s) {
      mbar_init(smem_u32(&bk->full[s]), 1);
      mbar_init(smem_u32(&bk->empty[s]), a.smat ? 1 : 5);  // the MMAs that read the tile + the warps that do, or their issuer for them
    }
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(smem_u32(&bk->full_b[s]), 1);
      mbar_init(smem_u32(&bk->empty_b[s]), 1);
    }
    mbar_init(smem_u32(&bk->acc_full), 1);
    mbar_init(smem_u32(&bk->mma_done), 1);
    mbar_init(smem_u32(&bk->norm_go), 1);
    bk->abort_flag = 0;
    bk->is_last = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bk->tmem_base), a.tmem_cols);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  pdl_enter();
  const uint32_t tmem_base = bk->tmem_base;
  WaitCtx wc{&bk->abort_flag, a.status, STATUS_SIM_TIMEOUT, a.wait_limit};
  // the groups of a pair walk the 64-column blocks from the same starting point (they share the rows
  // through L2); different pairs start elsewhere and spread over the memory channels
  const int rot = (pr * 5 + b * 3) % n_kb;

  const int n_t = two ? 2 : 1;
  if (warp == 0 || warp == 10) {
    // ---- copy warps, one per ring (converged, see tma_load_2d_w)
    const uint32_t leader = warp_leader();
    const bool rows = warp == 0;
    const CUtensorMap *map = rows ? &tmap_h : &tmap_kept;
    if (leader) tma_prefetch_desc(map);
    const int slots = rows ? a.a_stages : a.stages, bytes = rows ? SIM_A_BYTES : b_bytes, tiles = rows ? n_t : 1;
    const int row = !rows ? b * a.keep_k + gz * a.n_tile : a.smat ? b * a.keep_k + pr * 256 : d.row0 + d.v0 + pr * 256;
    const uint32_t ring = rows ? base : base_b;
    uint64_t *full0 = rows ? bk->full : bk->full_b, *empty0 = rows ? bk->empty : bk->empty_b;
    int issued = 0, kb = rot;
    RingPos r;
    for (int it = 0; it < n_kb; ++it) {
      int t = 0;
      for (; t < tiles; ++t) {
        if (issued >= slots) mbar_wait_warp(smem_u32(&empty0[r.slot]), r.phase ^ 1u, wc);
        if (__shfl_sync(0xffffffffu, bk->abort_flag, 0)) break;
        const uint32_t full = smem_u32(&full0[r.slot]);
        mbar_expect_tx_w(full, bytes, leader);
        tma_load_2d_w(ring + r.slot * bytes, map, full, kb * 64, row + t * 128, leader);
        ++issued;
        r.step(slots);
      }
      if (t < tiles) break;
      if (++kb == n_kb) kb = 0;
    }
    // drain: the last fill of every slot must have landed before the block leaves
    for (int s = 0; s < slots; ++s)
      if (issued > s) mbar_wait_drain(smem_u32(&full0[s]), ((issued - 1 - s) / slots) & 1, TC_WAIT_LIMIT);
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer (converged, as in sim_kernel)
    const uint32_t leader = warp_leader();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
    const uint32_t idesc = umma_idesc_bf16(128, a.n_tile);
    const uint64_t desc0 = umma_desc_sw128(base), bdesc0 = umma_desc_sw128(base_b);
    RingPos ra, rb;
    for (int it = 0; it < n_kb; ++it, rb.step(a.stages)) {
      mbar_wait_warp(smem_u32(&bk->full_b[rb.slot]), rb.phase, wc);
      const uint64_t db = bdesc0 + (uint32_t)(rb.slot * b_bytes) / 16;
      for (int t = 0; t < n_t; ++t, ra.step(a.a_stages)) {
        mbar_wait_warp(smem_u32(&bk->full[ra.slot]), ra.phase, wc);
        tc_fence_after();
        if (it == norm_lo && t == 0 && leader) mbar_arrive(smem_u32(&bk->norm_go));
        const uint64_t da = desc0 + ra.slot * (SIM_A_BYTES / 16);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          tc_mma_bf16_w(tm + t * a.n_tile, da + kk * 2, db + kk * 2, idesc, (it > 0 || kk > 0) ? 1u : 0u, leader);
        tc_commit_w(smem_u32(&bk->empty[ra.slot]), leader);
        if (!a.smat && (it < norm_lo || it >= norm_hi) && leader) mbar_arrive_n(smem_u32(&bk->empty[ra.slot]), 4);
      }
      tc_commit_w(smem_u32(&bk->empty_b[rb.slot]), leader);
    }
    tc_commit_w(smem_u32(&bk->acc_full), leader);
    // every MMA this warp issued has completed before tensor memory is given back
    tc_commit_w(smem_u32(&bk->mma_done), leader);
    mbar_wait_drain(smem_u32(&bk->mma_done), 0, TC_WAIT_LIMIT);
    __syncwarp();
  } else {
    const int grp = (warp - 2) >> 2;                     // row tile of the pair
    const int quarter = warp & 3;                        // the tensor-memory lanes a warp may read
    const int lrow = quarter * 32 + lane;
    const int prow = grp * 128 + lrow;                   // row inside the pair
    const int v = pr * 256 + prow;                       // visual token
    const bool active = grp == 0 || two;
    const float *kinv = a.kept_inv + (size_t)b * a.keep_k;
    // ---- squared norm of this thread's row: this group's share of the 64-column blocks
    float ssq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const bool norms = active && !a.smat;
    // (a parity tells two neighbouring fills of a slot apart, no more: the warps join in when the issuer, who waits for every
    // tile, has reached the range, so that all earlier fills are complete)
    if (norms) mbar_wait(smem_u32(&bk->norm_go), 0, wc);
    for (int it = norm_lo; it < (norms ? norm_hi : 0); ++it) {
      const int u = it * n_t + grp, s = u % a.a_stages;
      mbar_wait(smem_u32(&bk->full[s]), (u / a.a_stages) & 1, wc);
      if (!bk->abort_flag) {
        const uint4 *row = reinterpret_cast<const uint4 *>(base_ptr + (size_t)s * SIM_A_BYTES + lrow * 128);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint4 x = row[c ^ (lrow & 7)];
          float f[8];
          unpack8(x, f);
#pragma unroll
          for (int e = 0; e < 8; ++e) ssq[c] = fmaf(f[e], f[e], ssq[c]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bk->empty[s]));
    }
    float ss = ((ssq[0] + ssq[1]) + (ssq[2] + ssq[3])) + ((ssq[4] + ssq[5]) + (ssq[6] + ssq[7]));

    float best = -INFINITY;
    int best_slot = 0;
    const int slot0 = gz * a.n_tile;
    const int ncol = max(0, min(a.n_tile, a.keep_k - slot0));
    bk->kinv[prow] = prow < ncol ? kinv[slot0 + prow] : 0.f;
    asm volatile("bar.sync 1, 256;" ::: "memory");
    mbar_wait(smem_u32(&bk->acc_full), 0, wc);
    tc_fence_after();
    if (active && !bk->abort_flag) {
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + grp * a.n_tile;
      const float inv_p = (a.smat && v < a.keep_k) ? kinv[v] : 0.f;
      int c0 = 0;
      if (!a.smat) {
        // 32 columns per tensor-memory wait while they last: half as many waits on the path every block goes
        // through after its last MMA, which nothing overlaps (c4 881 -> 833 us; 64 columns per wait: the same)
#pragma unroll 1
        for (; c0 + 32 <= ncol; c0 += 32) sim_scan32(taddr + c0, bk->kinv + c0, slot0 + c0, best, best_slot);
      }
#pragma unroll 1
      for (int c = c0; c < ncol; c += 16) {
        uint32_t r[16];
        tmem_ld16(taddr + c, r);
        tmem_wait_ld();
        if (a.smat) {
          // matrix mode: S[p][q] = <h_p, h_q> * (1/||h_p|| * 1/||h_q||) for this thread's kept row p
          float sv[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) sv[e] = __uint_as_float(r[e]) * (inv_p * bk->kinv[c + e]);   // (a column past the last slot has kinv 0 in shared memory)
          if (v < a.keep_k) {
            float *srow = a.smat + ((size_t)b * a.keep_k + v) * a.keep_k + slot0 + c;
            uint32_t above = 0u;
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (c + e < ncol && slot0 + c + e != v && sv[e] > a.threshold) above |= 1u << e;
            if (c + 16 <= ncol && (reinterpret_cast<size_t>(srow) & 15) == 0) {
#pragma unroll
              for (int e = 0; e < 16; e += 4)         // 16-byte stores: a quarter of the store requests
                reinterpret_cast<float4 *>(srow)[e >> 2] = make_float4(sv[e], sv[e + 1], sv[e + 2], sv[e + 3]);
            } else {
#pragma unroll
              for (int e = 0; e < 16; ++e)
                if (c + e < ncol) srow[e] = sv[e];
            }
            if (a.mask16) {
              // the routing's bit matrix on the way (slot0 and c are multiples of 16); the last chunk also
              // clears the other half of its word
              const int hw = (slot0 + c) >> 4;
              uint16_t *mrow = a.mask16 + ((size_t)b * a.keep_k + v) * a.mask_pitch;
              mrow[hw] = (uint16_t)above;
              if (slot0 + c + 16 >= a.keep_k && !(hw & 1)) mrow[hw + 1] = 0;
            }
          }
          // S[q][p] where the block of that place has left it to this one (the same for the 16 columns, and for each half of the
          // warp's rows): a warp's 32 rows are neighbours in row q
          const bool mirrored = (v / a.n_tile + 1) * a.n_tile <= ((slot0 + c) & ~255);
          const uint32_t halves = __ballot_sync(0xffffffffu, mirrored);
          if (halves) {
            uint32_t word = 0u;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              if (mirrored && c + e < ncol) a.smat[((size_t)b * a.keep_k + slot0 + c + e) * a.keep_k + v] = sv[e];
              const uint32_t w = __ballot_sync(0xffffffffu, mirrored && sv[e] > a.threshold);
              if ((lane & 15) == e) word = w;
            }
            const int half = lane >> 4;                   // lane writes its half of the warp's rows for column lane & 15
            if (a.mask16 && ((halves >> (16 * half)) & 1u) && c + (lane & 15) < ncol)
              a.mask16[((size_t)b * a.keep_k + slot0 + c + (lane & 15)) * a.mask_pitch + ((v & ~31) >> 4) + half] = (uint16_t)(word >> (16 * half));
          }
          continue;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int slot = slot0 + c + e;
          if (c + e < ncol) {
            const float val = __uint_as_float(r[e]) * kinv[slot];
            if (val > best) { best = val; best_slot = slot; }
          }
        }
      }
    }
    tc_fence_before();
    bool finalize = !a.smat;
    if (a.groups > 1 && !a.smat) {
      // per pair: [group][best of 256 rows | slot of 256 rows | its share of their squared norms]
      float *pp = a.part + ((size_t)b * a.max_mt + pr) * (size_t)(a.groups * 768);
      pp[gz * 768 + prow] = best;
      reinterpret_cast<int *>(pp)[gz * 768 + 256 + prow] = best_slot;
      pp[gz * 768 + 512 + prow] = ss;
      __threadfence();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (warp == 2 && lane == 0) {
        unsigned int *cnt = a.tile_counters + (size_t)b * a.max_mt + pr;
        const unsigned int old = atomicAdd(cnt, 1u);
        bk->is_last = (old == (unsigned int)(a.groups - 1));
        if (bk->is_last) *cnt = 0u;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      finalize = bk->is_last != 0;
      if (finalize) {
        __threadfence();
        best = -INFINITY;
        best_slot = 0;
        ss = 0.f;
        for (int g2 = 0; g2 < a.groups; ++g2) {           // ascending slots: the first maximum stays
          const float val = __ldcg(pp + g2 * 768 + prow);
          const int slot = __ldcg(reinterpret_cast<const int *>(pp) + g2 * 768 + 256 + prow);
          ss += __ldcg(pp + g2 * 768 + 512 + prow);
          if (val > best) { best = val; best_slot = slot; }
        }
      }
    }
    int dp = -1;
    if (finalize && v < n_rows) {
      const int role = a.role[(size_t)b * a.max_vis + v];
      dp = role < 0 ? -role - 1 : -1;
    }
    if (dp >= 0 && dp < nd && !bk->abort_flag) {
      const bool zero_row = !(ss >= 1e-24f);             // ||h|| < 1e-12: similarity 0 to every slot
      const float sim = zero_row ? 0.f : best * rsqrtf(ss);
      const int slot = zero_row ? 0 : best_slot;
      const size_t o = (size_t)b * (a.max_vis - a.keep_k) + dp;
      a.assign[o] = (sim > a.threshold) ? slot : -1;
      if (a.best_sim) a.best_sim[o] = sim;
      if (a.member_bits && sim > a.threshold) set_member_bit(a, b, slot, v);
    }
    if (warp == 2 && lane == 0) bk->is_last = finalize ? 1 : 0;
    if (a.seg) __threadfence();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, a.tmem_cols);
  }
  if (!a.seg || !bk->is_last) return;                    // (or a group that did not finalize its pair, or matrix mode)
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int n_pr = (unsigned int)((n_rows + 255) / 256);
    const unsigned int old = atomicAdd(a.counters + b, 1u);
    bk->is_last = (old == n_pr - 1u);
    if (bk->is_last) a.counters[b] = 0u;
  }
  __syncthreads();
  if (!bk->is_last) return;
  __threadfence();
  csr_block(d, b, a.max_vis, a.keep_k, a.assign, a.seg, a.members, reinterpret_cast<int *>(base_ptr),
            bk->scan, a.drop_all, a.salience, a.member_meta);
}

}  // namespace asap
