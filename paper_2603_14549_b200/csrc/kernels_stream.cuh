// The memory-bound and latency-bound kernels of the ASAP prune step:
//   prepare        device-side validation, per-sample descriptors, output row offsets (one warp of a kernel that runs anyway)
//   mass           sum of the visual queries, s_j, then s_hat_j and m_j   (Eq. 1, Eq. 2, Eq. 3), with one mask or one per head
//   salience_block s_hat_j from per-head masses the score kernel produced (part of the selection launch)
//   select         stable radix top-k of the ranking scores           (Fig. 3)
//   role_map       kept slot / dropped position of every visual token
//   kept_gather    kept rows gathered for the similarity GEMM, with their inverse norms (Sec. 4.2)
//   csr_block      dropped tokens grouped by destination slot (tail of the similarity kernel where member bits have no room)
//   route          Sec. 4.2 inside the kept set, from the bit matrix of similar pairs
//   merge_compact  Eq. 5 and the hand-off of Fig. 3
//   gather_rows    KV-cache compaction with the row map of the hand-off
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace asap {

// =======================================================================================
// prepare
// =======================================================================================
struct PrepareArgs {
  int32_t B, total_tokens, min_vis, max_vis, max_seq, max_rank, keep_k, out_capacity;
  int32_t write_desc;        // mass and score kernel: the first block also runs prepare_warp
  const int32_t *cu_seqlens, *vis_start, *vis_len, *text_start, *text_len, *rank_start, *rank_len;
  SampleDesc *desc;          // [B]
  int32_t *out_cu_seqlens;   // [B+1] or nullptr
  uint32_t *status;
};

// Descriptor of sequence b with its validity (out_row0 is filled in by prepare_warp).
__device__ __forceinline__ SampleDesc make_desc(const PrepareArgs &a, int b) {
  const int lo = a.cu_seqlens[b], hi = a.cu_seqlens[b + 1];
  const int n = hi - lo;
  const int v0 = a.vis_start[b], nv = a.vis_len[b];
  const int t0 = a.text_start[b], tl = a.text_len[b];
  const int r0 = a.rank_start ? a.rank_start[b] : t0;
  const int nr = a.rank_len ? a.rank_len[b] : tl;
  bool ok = lo >= 0 && n > 0 && n <= a.max_seq && hi <= a.total_tokens;
  ok = ok && v0 >= 0 && nv >= a.min_vis && nv <= a.max_vis && v0 + nv <= n;
  ok = ok && tl >= 0 && t0 >= v0 + nv && t0 + tl <= n;
  ok = ok && r0 >= 0 && nr >= 1 && nr <= a.max_rank && r0 + nr <= n;
  ok = ok && a.keep_k <= nv;
  if (b == 0) ok = ok && lo == 0;
  if (b == a.B - 1) ok = ok && hi == a.total_tokens;
  SampleDesc d;
  d.row0 = lo; d.n = n; d.v0 = v0; d.nv = nv; d.r0 = r0; d.nr = nr; d.out_row0 = 0;
  d.valid = ok ? 1 : 0;
  return d;
}

// Whether the shortened batch fits the output, by one warp: if not, nothing may be written (see prepare_warp).
__device__ __forceinline__ bool output_fits(const PrepareArgs &a) {
  int len = 0;
  for (int b = threadIdx.x & 31; b < a.B; b += 32) {
    const SampleDesc d = make_desc(a, b);
    if (d.valid) len += d.n - d.nv + a.keep_k;
  }
  return __reduce_add_sync(0xffffffffu, len) <= a.out_capacity;
}

// Run by one warp: validates every sequence, writes the descriptors, the output row offsets and the status bits.
// (A whole block with one thread adding the offsets up took 6 us for 8 sequences: a chain of round trips.)
__device__ __forceinline__ void prepare_warp(const PrepareArgs &a) {
  const int lane = threadIdx.x & 31;
  int carry = 0;
  bool bad = false;
  for (int b0 = 0; b0 < a.B; b0 += 32) {
    const int b = b0 + lane;
    SampleDesc d;
    int len = 0;
    if (b < a.B) {
      d = make_desc(a, b);
      if (d.valid) len = d.n - d.nv + a.keep_k;
      else bad = true;
    }
    int inc = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (b < a.B) {
      d.out_row0 = carry + inc - len;
      a.desc[b] = d;
      if (a.out_cu_seqlens) a.out_cu_seqlens[b] = d.out_row0;
    }
    carry += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (a.out_cu_seqlens && lane == 0) a.out_cu_seqlens[a.B] = carry;
  uint32_t bits = __any_sync(0xffffffffu, bad) ? STATUS_BAD_SAMPLE : 0u;
  if (carry > a.out_capacity) {
    bits |= STATUS_OUT_CAPACITY;
    __syncwarp();
    for (int b = lane; b < a.B; b += 32) a.desc[b].valid = 0;   // nothing may be written
  }
  if (bits && lane == 0) atomicOr(a.status, bits);
  __syncwarp();
}

__global__ void prepare_kernel(PrepareArgs a) {
  pdl_enter();
  prepare_warp(a);
}

// =======================================================================================
// mass_kernel: Eq. 1 with the sum over the queries taken first, per head:  s_j^h = qbar^h . k_j^h,  qbar^h = sum of the visual
// queries of head h.  Persistent blocks, an item is one (sample, head): a copy warp streams the head's visual queries and then
// its keys, 128 rows a tile, through a ring of shared memory and runs ahead into the next item; eight warps add the query rows up,
// exchange their sums and multiply the key rows.  A half-warp holds a row of the head (256 bytes).
//   PER_HEAD   (one salience and one mask per head) heads gets s_j^h / sqrt(d); then Eq. 2 and Eq. 3 of the head, whose
//              (minimum, 1 / range) stay in `norm` [B, H, 2] for the head means.
//   otherwise  heads gets the masses as they are, for salience_kernel.  (As the tail of the block that finishes a sample's last
//              head it held that block's ring up: 31 samples of 611 rows 108 us.)
// Bound by memory: queries and keys are read once and nothing else of size moves.  Three kernels did this (a query sum with
// partial rows through memory, masses with all heads of a row per warp, masks; per step, before -> now): 8 x 1536 rows, 32 heads, a
// mask per head 70 -> 45 us of kernels (4.5 TB/s), the step 206.5 -> 189; 31 x 611 83 -> 70 (5.2 TB/s without the salience), the step
// 270 -> 252; 3 x 174-186 with 16 heads, a mask per head 49.5 -> 39.7.  The same work with rows held in registers, eight in flight per
// thread, and a cluster of blocks per item: 59 us on the first (loads, sums and exchanges in turn).
// =======================================================================================
constexpr int MASS_THREADS = 288;                // copy warp, eight adding warps
constexpr int MASS_ADDERS = 256;
constexpr int MASS_STAGES = 5;                   // (with the rest below the 195 KB that the neighbouring kernels use)
constexpr int MASS_TILE_BYTES = 2 * 128 * 128;   // 128 rows x 128 bf16 as two 64-column blocks
constexpr int MASS_SMEM_BYTES = MASS_STAGES * MASS_TILE_BYTES + 1024;
constexpr long long MASS_WAIT_LIMIT = 1500000000LL;   // clock cycles, roughly one second

struct SalienceArgs {
  int H;
  double scale;                             // 1 / (H sqrt(head_dim))
  float lambda_max, eps;
  const float *heads;                       // [B, H, max_vis]
  const float *norm;                        // [B, H, 2] or nullptr: a salience per head (salience_heads_block)
  float *mass, *salience, *mask_log, *rank_score;   // [B, max_vis]
};

struct MassArgs {
  PrepareArgs pa;            // write_desc: the first block validates the batch and writes the descriptors
  int max_vis;
  float scale;               // of `heads`
  float *heads;              // [B, H, max_vis]
  float *mask_log_heads;     // PER_HEAD: [B, H, max_vis]
  float *norm;               // PER_HEAD: [B, H, 2]
  int H;
  float lambda_max, eps;
  uint32_t *status;
  long long wait_limit;
};

// barrier of the adding warps alone
__device__ __forceinline__ void mass_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// The masses' own sums over the heads: sixteen in pairs, the sixteens and the scale in 64 bits.  One after the other in 32 bits, 32
// heads lose more than the masses themselves do (error against 64 bits 9.3e-8 instead of 5.0e-8 with their exact sum).
template <int N>
__device__ __forceinline__ float pair_sum(float (&v)[N]) {
#pragma unroll
  for (int o = 1; o < N; o <<= 1)
#pragma unroll
    for (int e = 0; e < N; e += 2 * o) v[e] += v[e + o];
  return v[0];
}

// Column j of `p` [H, max_vis]: the sum over the heads, scaled.
__device__ __forceinline__ float head_total(const float *p, int H, int max_vis, double scale) {
  double sum = 0.0;
  int hh = 0;
  for (; hh + 16 <= H; hh += 16) {          // sixteen loads in flight
    float v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = __ldcg(p + (size_t)(hh + e) * max_vis);
    sum += (double)pair_sum(v);
  }
  if (hh < H) {
    float v[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = hh + e < H ? __ldcg(p + (size_t)(hh + e) * max_vis) : 0.f;
    sum += (double)pair_sum(v);
  }
  return (float)(sum * scale);
}
// salience_heads_block: one block per sample: mass = mean_h s^h (equal to the default mass), salience =
// mean_h s_hat^h (the Eq. 5 weight), mask_log = Eq. 3 of that mean.
__device__ __forceinline__ void salience_heads_block(const SampleDesc &d, int b, int max_vis, const SalienceArgs &a) {
  float *mass_b = a.mass + (size_t)b * max_vis, *sal_b = a.salience + (size_t)b * max_vis, *msk_b = a.mask_log + (size_t)b * max_vis;
  const float *sh_b = a.heads + (size_t)b * a.H * max_vis, *norm = a.norm + (size_t)b * a.H * 2;
  __shared__ float2 s_norm[64];             // (H <= 64: D <= 8192)
  if ((int)threadIdx.x < a.H) s_norm[threadIdx.x] = make_float2(__ldcg(norm + 2 * threadIdx.x), __ldcg(norm + 2 * threadIdx.x + 1));
  __syncthreads();
  const float inv_h = 1.0f / (float)a.H;
  for (int j = threadIdx.x; j < max_vis; j += blockDim.x) {
    float acc_s = 0.f, acc_sh = 0.f, sal = 0.f;
    if (d.valid && j < d.nv) {
      for (int h0 = 0; h0 < a.H; h0 += 16) {                        // heads in order, sixteen loads in flight
        float v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = h0 + e < a.H ? __ldcg(sh_b + (size_t)(h0 + e) * max_vis + j) : 0.f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          if (h0 + e >= a.H) break;
          const float2 n = s_norm[h0 + e];
          acc_s += v[e];
          acc_sh += (v[e] - n.x) * n.y;
        }
      }
      sal = acc_sh * inv_h;
    }
    const bool in = d.valid && j < d.nv;
    mass_b[j] = in ? acc_s * inv_h : 0.f;
    sal_b[j] = in ? sal : 0.f;
    msk_b[j] = in ? logf(fmaxf(a.lambda_max * sal, a.eps)) : 0.f;
    if (!d.valid) a.rank_score[(size_t)b * max_vis + j] = 0.f;      // the score kernel and the selection skip the sample
  }
}

__global__ void __launch_bounds__(MASS_THREADS)
salience_heads_kernel(const SampleDesc *__restrict__ desc, int max_vis, SalienceArgs a) {
  pdl_enter();
  salience_heads_block(desc[blockIdx.x], blockIdx.x, max_vis, a);
}

// =======================================================================================
// salience_block: the tail of Eq. 1 and Eq. 2-3 when the per-head masses qbar^h . k_j^h were
// produced by the score kernel (from the query and key tiles it streams).  One block per sample, beside
// the block that selects (grid y of the selection launch): s_j = scale * sum_h heads[b, h, j], then the min-max normalisation and
// the mask vector over the image span; padding past the span is zeroed.
// =======================================================================================
constexpr int SAL_THREADS = 1024;

// Sums over the heads, in head order, of four neighbouring columns (max_vis a multiple of four): 16-byte loads, sixteen in
// flight.  With 4-byte loads the request rate of one SM bound this (2880 columns x 32 heads: 18 thousand clocks).
__device__ __forceinline__ bool wide_columns(int max_vis, int nv) { return (max_vis & 3) == 0 && nv > SAL_THREADS; }
__device__ __forceinline__ float4 head_sum4(const float *p, int H, int max_vis) {
  float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
  int hh = 0;
  for (; hh + 8 <= H; hh += 8) {
    float4 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __ldcg(reinterpret_cast<const float4 *>(p + (size_t)(hh + e) * max_vis));
#pragma unroll
    for (int e = 0; e < 8; ++e) { t.x += v[e].x; t.y += v[e].y; t.z += v[e].z; t.w += v[e].w; }
  }
  for (; hh < H; ++hh) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p + (size_t)hh * max_vis));
    t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
  }
  return t;
}

__device__ __forceinline__ void salience_block(const SampleDesc &d, int b, int max_vis, const SalienceArgs &a) {
  __shared__ float s_red[2 * (SAL_THREADS / 32)];
  float *mass_b = a.mass + (size_t)b * max_vis, *sal_b = a.salience + (size_t)b * max_vis, *msk_b = a.mask_log + (size_t)b * max_vis;
  const int H = a.H;
  const float lambda_max = a.lambda_max, eps = a.eps;
  if (!d.valid) {
    for (int j = threadIdx.x; j < max_vis; j += SAL_THREADS) {
      mass_b[j] = 0.f; sal_b[j] = 0.f; msk_b[j] = 0.f;
      a.rank_score[(size_t)b * max_vis + j] = 0.f;     // the score kernel and the selection skip the sample
    }
    return;
  }
  const float *hb = a.heads + (size_t)b * H * max_vis;
  float lo = INFINITY, hi = -INFINITY;
  const bool vec = wide_columns(max_vis, d.nv);
  if (vec) {
    for (int j = threadIdx.x * 4; j < d.nv; j += SAL_THREADS * 4) {
      double tot[4] = {0.0, 0.0, 0.0, 0.0};
      for (int h0 = 0; h0 < H; h0 += 8) {
        float v[4][8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 x = h0 + e < H ? __ldcg(reinterpret_cast<const float4 *>(hb + (size_t)(h0 + e) * max_vis + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
          v[0][e] = x.x; v[1][e] = x.y; v[2][e] = x.z; v[3][e] = x.w;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) tot[c] += (double)pair_sum(v[c]);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (j + e >= d.nv) break;
        const float m = (float)(tot[e] * a.scale);
        mass_b[j + e] = m;
        lo = fminf(lo, m); hi = fmaxf(hi, m);
      }
    }
  }
  for (int j = vec ? d.nv : (int)threadIdx.x; j < d.nv; j += SAL_THREADS) {
    const float tot = head_total(hb + j, H, max_vis, a.scale);
    mass_b[j] = tot;
    lo = fminf(lo, tot); hi = fmaxf(hi, tot);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) { s_red[warp] = lo; s_red[SAL_THREADS / 32 + warp] = hi; }
  __syncthreads();
  lo = s_red[0]; hi = s_red[SAL_THREADS / 32];
#pragma unroll
  for (int w = 1; w < SAL_THREADS / 32; ++w) {
    lo = fminf(lo, s_red[w]); hi = fmaxf(hi, s_red[SAL_THREADS / 32 + w]);
  }
  const float inv = 1.0f / ((hi - lo) + eps);
  for (int j = threadIdx.x; j < max_vis; j += SAL_THREADS) {
    if (j < d.nv) {
      const float sh = (mass_b[j] - lo) * inv;      // (stored above, before the block's barrier)
      sal_b[j] = sh;
      msk_b[j] = logf(fmaxf(lambda_max * sh, eps));
    } else {
      mass_b[j] = 0.f; sal_b[j] = 0.f; msk_b[j] = 0.f;
    }
  }
}

// one block per sample, where the score kernel needs the mask vector (ranking rows in the image span)
__global__ void __launch_bounds__(SAL_THREADS)
salience_kernel(const SampleDesc *desc, int max_vis, SalienceArgs a) {
  pdl_enter();
  salience_block(ld_prev(desc + blockIdx.x), blockIdx.x, max_vis, a);
}

template <bool PER_HEAD>
__global__ void __launch_bounds__(MASS_THREADS, 1)
mass_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k, MassArgs a) {
  extern __shared__ __align__(1024) uint8_t m_smem[];
  __shared__ uint64_t s_full[MASS_STAGES], s_empty[MASS_STAGES];
  __shared__ float s_part[MASS_ADDERS / 32][128], s_sum[128], s_red[2 * (MASS_ADDERS / 32)];
  __shared__ int s_abort;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(m_smem) + 1023u) & ~1023u;
  const uint8_t *tiles = m_smem + (base - smem_u32(m_smem));
  if (threadIdx.x == 0) {
    for (int s = 0; s < MASS_STAGES; ++s) {
      mbar_init(smem_u32(&s_full[s]), 1);
      mbar_init(smem_u32(&s_empty[s]), MASS_ADDERS / 32);
    }
    s_abort = 0;
    fence_barrier_init();
  }
  __syncthreads();
  pdl_enter();
  if (threadIdx.x == 0 && (*reinterpret_cast<volatile uint32_t *>(a.status) & STATUS_MASS_TIMEOUT)) s_abort = 1;
  __syncthreads();
  WaitCtx wc{&s_abort, a.status, STATUS_MASS_TIMEOUT, a.wait_limit};
  const int H = a.H, n_items = a.pa.B * H;
  if (warp == 0) {
    // ---- copies (converged, see tma_load_2d_w)
    const uint32_t leader = warp_leader();
    const uint64_t keep = l2_evict_normal(), drop = l2_evict_first();     // (the score kernel comes for the keys)
    if (leader) {
      tma_prefetch_desc(&tmap_q);
      tma_prefetch_desc(&tmap_k);
    }
    RingPos r;
    int issued = 0;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
      const int b = item / H, h = item - b * H;
      const SampleDesc d = make_desc(a.pa, b);
      const int n = d.valid ? (d.nv + 127) / 128 : 0;
      int u = 0;
      for (; u < 2 * n; ++u) {
        if (issued >= MASS_STAGES) mbar_wait_warp(smem_u32(&s_empty[r.slot]), r.phase ^ 1u, wc);
        if (__shfl_sync(0xffffffffu, s_abort, 0)) break;
        const uint32_t bar = smem_u32(&s_full[r.slot]), dst = base + r.slot * MASS_TILE_BYTES;
        const int row = d.row0 + d.v0 + (u < n ? u : u - n) * 128;
        const CUtensorMap *map = u < n ? &tmap_q : &tmap_k;
        mbar_expect_tx_w(bar, MASS_TILE_BYTES, leader);
        tma_load_2d_hint_w(dst, map, bar, h * 128, row, u < n ? drop : keep, leader);
        tma_load_2d_hint_w(dst + MASS_TILE_BYTES / 2, map, bar, h * 128 + 64, row, u < n ? drop : keep, leader);
        ++issued;
        r.step(MASS_STAGES);
      }
      if (u < 2 * n) break;
    }
    for (int s = 0; s < MASS_STAGES; ++s)                 // every copy has landed before the block may leave
      if (issued > s) mbar_wait_drain(smem_u32(&s_full[s]), ((issued - 1 - s) / MASS_STAGES) & 1, MASS_WAIT_LIMIT);
    __syncwarp();
    return;
  }
  const int tid = threadIdx.x - 32, aw = warp - 1;        // among the adding warps
  if (a.pa.write_desc && blockIdx.x == 0 && aw == 0) prepare_warp(a.pa);
  const bool fits = !PER_HEAD || output_fits(a.pa);       // (the masks of the heads are outputs; the first tiles are on their way)
  const int c = lane & 15, row0 = (tid >> 4) * 8;         // this thread's 16-byte chunk of the head, its half-warp's eight rows of a tile
  const bool up8 = lane & 8, up4 = lane & 4, up2 = lane & 2;
  RingPos r;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int b = item / H, h = item - b * H;
    const SampleDesc d = make_desc(a.pa, b);
    float *mh = PER_HEAD ? a.mask_log_heads + (size_t)item * a.max_vis : nullptr;
    float *out = a.heads + (size_t)item * a.max_vis;
    if (!d.valid) {
      if (PER_HEAD)
        for (int j = tid; j < a.max_vis; j += MASS_ADDERS) mh[j] = 0.f;
      continue;
    }
    const int n = (d.nv + 127) / 128;
    auto chunk = [&](int row) {                            // (row r of a block: its chunk c at position c ^ (r & 7))
      return *reinterpret_cast<const uint4 *>(tiles + r.slot * MASS_TILE_BYTES + (c >> 3) * (MASS_TILE_BYTES / 2) + row * 128 + (((c & 7) ^ (row & 7)) << 4));
    };
    auto release = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_empty[r.slot]));
      r.step(MASS_STAGES);
    };
    // ---- the queries' sum
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
    for (int u = 0; u < n; ++u) {
      mbar_wait(smem_u32(&s_full[r.slot]), r.phase, wc);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        uint4 x = chunk(row0 + i);
        if (u * 128 + row0 + i >= d.nv) x = make_uint4(0u, 0u, 0u, 0u);
        acc[0] = f2_add(acc[0], f2_pack(bf16_lo(x.x), bf16_hi(x.x)));
        acc[1] = f2_add(acc[1], f2_pack(bf16_lo(x.y), bf16_hi(x.y)));
        acc[2] = f2_add(acc[2], f2_pack(bf16_lo(x.z), bf16_hi(x.z)));
        acc[3] = f2_add(acc[3], f2_pack(bf16_lo(x.w), bf16_hi(x.w)));
      }
      release();
    }
    float f[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) f2_unpack(acc[e], f[2 * e], f[2 * e + 1]);
#pragma unroll
    for (int e = 0; e < 8; ++e) f[e] += __shfl_xor_sync(0xffffffffu, f[e], 16);
    if (lane < 16) {
#pragma unroll
      for (int e = 0; e < 8; ++e) s_part[aw][c * 8 + e] = f[e];
    }
    mass_bar();
    if (tid < 128) {
      float t = 0.f;
#pragma unroll
      for (int w = 0; w < MASS_ADDERS / 32; ++w) t += s_part[w][tid];
      s_sum[tid] = t;
    }
    mass_bar();
    float qs[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) qs[e] = s_sum[c * 8 + e];
    // ---- the keys
    float lo = INFINITY, hi = -INFINITY;
    for (int u = 0; u < n; ++u) {
      mbar_wait(smem_u32(&s_full[r.slot]), r.phase, wc);
      float s[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float g[8];
        unpack8(chunk(row0 + i), g);
        s[i] = (g[0] * qs[0] + g[1] * qs[1] + g[2] * qs[2] + g[3] * qs[3]) + (g[4] * qs[4] + g[5] * qs[5] + g[6] * qs[6] + g[7] * qs[7]);
      }
      release();
      // sums over 16 lanes, the rows dealt out on the way: eight shuffles for eight rows
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] = (up8 ? s[4 + i] : s[i]) + __shfl_xor_sync(0xffffffffu, up8 ? s[i] : s[4 + i], 8);
#pragma unroll
      for (int i = 0; i < 2; ++i) s[i] = (up4 ? s[2 + i] : s[i]) + __shfl_xor_sync(0xffffffffu, up4 ? s[i] : s[2 + i], 4);
      float t = (up2 ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, up2 ? s[0] : s[1], 2);
      t += __shfl_xor_sync(0xffffffffu, t, 1);
      const int j = u * 128 + row0 + (up8 ? 4 : 0) + (up4 ? 2 : 0) + (up2 ? 1 : 0);
      if (j < d.nv) {
        t *= a.scale;
        if (!(lane & 1)) out[j] = t;
        lo = fminf(lo, t); hi = fmaxf(hi, t);
      }
    }
    if (PER_HEAD) {
      // ---- Eq. 2 and Eq. 3 of the head
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      }
      if (lane == 0) { s_red[aw] = lo; s_red[MASS_ADDERS / 32 + aw] = hi; }
      mass_bar();
#pragma unroll
      for (int w = 0; w < MASS_ADDERS / 32; ++w) {
        lo = fminf(lo, s_red[w]); hi = fmaxf(hi, s_red[MASS_ADDERS / 32 + w]);
      }
      const float inv = 1.0f / ((hi - lo) + a.eps);
      if (tid == 0) {
        a.norm[(size_t)item * 2] = lo;
        a.norm[(size_t)item * 2 + 1] = inv;
      }
      for (int j = tid; j < a.max_vis; j += MASS_ADDERS)
        mh[j] = fits && j < d.nv ? logf(fmaxf(a.lambda_max * ((out[j] - lo) * inv), a.eps)) : 0.f;
      // (two barriers come before s_red is written again)
    }
  }
}

// =======================================================================================
// select: exact top-k by radix select over order-preserving 32-bit keys, equal scores resolved
// toward the lower index, outputs in ascending index order.  One block per sample.
// =======================================================================================
constexpr int SELECT_THREADS = 1024;

__device__ __forceinline__ uint32_t score_key(float f) {
  if (f != f) return 0u;                       // NaN ranks below everything
  uint32_t u = __float_as_uint(f);
  if (f == 0.f) u = 0u;                        // -0.0 and +0.0 are one score: they tie, the lower index wins
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// exclusive prefix sum of one int per thread across the block; returns the block total in `total`
__device__ __forceinline__ int block_exclusive_scan(int v, int *s_warp /*[32]*/, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();   // s_warp may still be read from a previous scan
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0;
    int winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += t;
    }
    s_warp[lane] = winc - w;             // exclusive warp offsets
    if (lane == 31) s_warp[32] = winc;   // block total
  }
  __syncthreads();
  total = s_warp[32];
  return s_warp[warp] + inc - v;
}

__global__ void __launch_bounds__(SELECT_THREADS)
select_kernel(const float *__restrict__ rank_score, const SampleDesc *desc,
              int max_vis, int keep_k, int32_t *__restrict__ keep_idx, int32_t *__restrict__ drop_idx,
              int32_t *__restrict__ role /*[B, max_vis]*/, int32_t *__restrict__ assign /*nullable*/,
              float *__restrict__ best_sim /*nullable*/, int sim_follows,
              const float *__restrict__ head_partial /*nullable: [B, H, max_vis]*/, int H,
              float *__restrict__ rank_out /*[B, max_vis], written when head_partial is given*/,
              SalienceArgs sal /* blockIdx.y == 1 */) {
  pdl_enter();
  if (blockIdx.y == 1) {
    const SampleDesc d = ld_prev(desc + blockIdx.x);
    if (sal.norm) salience_heads_block(d, blockIdx.x, max_vis, sal);
    else salience_block(d, blockIdx.x, max_vis, sal);
    return;
  }
  extern __shared__ uint32_t s_key[];   // [max_vis]
  __shared__ int s_hist[256];
  __shared__ int s_scan[33];
  __shared__ uint32_t s_prefix, s_lo[32], s_hi[32];
  __shared__ int s_remaining, s_bucket;
  const int b = blockIdx.x;
  const SampleDesc d = ld_prev(desc + b);
  const int nd_max = max_vis - keep_k;
  int32_t *keep_b = keep_idx + (size_t)b * keep_k;
  int32_t *drop_b = drop_idx + (size_t)b * nd_max;
  int32_t *role_b = role + (size_t)b * max_vis;
  // assign / best_sim entries the similarity kernel will not write: the padding past the last
  // dropped token, and everything when no similarity kernel follows or the sample is skipped
  if (assign) {
    const int first = (d.valid && sim_follows) ? d.nv - keep_k : 0;
    for (int j = first + threadIdx.x; j < nd_max; j += blockDim.x) {
      assign[(size_t)b * nd_max + j] = -1;
      if (best_sim) best_sim[(size_t)b * nd_max + j] = 0.f;
    }
  }
  if (!d.valid) {
    for (int j = threadIdx.x; j < keep_k; j += blockDim.x) keep_b[j] = -1;
    for (int j = threadIdx.x; j < nd_max; j += blockDim.x) drop_b[j] = -1;
    for (int j = threadIdx.x; j < max_vis; j += blockDim.x) role_b[j] = 0;
    return;
  }
  const int nv = d.nv;
  if (head_partial) {
    // r_j = mean over heads and ranking rows of the Eq. 4 probabilities: the per-head sums
    // over ranking rows are added here in head order, and r is also written out
    const float inv = 1.0f / ((float)H * (float)d.nr);
    const bool vec = wide_columns(max_vis, nv);
    if (vec) {
      for (int j = threadIdx.x * 4; j < max_vis; j += SELECT_THREADS * 4) {
        const float4 t4 = j < nv ? head_sum4(head_partial + (size_t)b * H * max_vis + j, H, max_vis) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float tot = j + e < nv ? tv[e] * inv : 0.f;
          if (j + e < nv) s_key[j + e] = score_key(tot);
          rank_out[(size_t)b * max_vis + j + e] = tot;
        }
      }
    }
    for (int j = vec ? max_vis : (int)threadIdx.x; j < max_vis; j += blockDim.x) {
      float tot = 0.f;
      if (j < nv) {
        const float *p = head_partial + (size_t)b * H * max_vis + j;
        int hh = 0;
        for (; hh + 32 <= H; hh += 32) {         // 32 loads in flight: one round trip for 32 heads
          float v[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) v[e] = __ldcg(p + (size_t)(hh + e) * max_vis);
#pragma unroll
          for (int e = 0; e < 32; ++e) tot += v[e];
        }
        for (; hh + 8 <= H; hh += 8) {
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = __ldcg(p + (size_t)(hh + e) * max_vis);
#pragma unroll
          for (int e = 0; e < 8; ++e) tot += v[e];
        }
        for (; hh < H; ++hh) tot += __ldcg(p + (size_t)hh * max_vis);
        tot *= inv;
        s_key[j] = score_key(tot);
      }
      rank_out[(size_t)b * max_vis + j] = tot;
    }
  } else {
    for (int j = threadIdx.x; j < nv; j += blockDim.x)
      s_key[j] = score_key(rank_score[(size_t)b * max_vis + j]);
  }
  __syncthreads();
  // The bits in which the keys differ at all: scores of one sequence share their sign and most of their exponent, and a digit
  // that all keys have in common costs a pass of atomics on one counter.
  uint32_t k_lo = 0xffffffffu, k_hi = 0u;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) { k_lo = min(k_lo, s_key[j]); k_hi = max(k_hi, s_key[j]); }
  k_lo = __reduce_min_sync(0xffffffffu, k_lo);
  k_hi = __reduce_max_sync(0xffffffffu, k_hi);
  if ((threadIdx.x & 31) == 0) { s_lo[threadIdx.x >> 5] = k_lo; s_hi[threadIdx.x >> 5] = k_hi; }
  for (int i = threadIdx.x; i < 256; i += blockDim.x) s_hist[i] = 0;
  __syncthreads();
  k_lo = __reduce_min_sync(0xffffffffu, s_lo[threadIdx.x & 31]);
  k_hi = __reduce_max_sync(0xffffffffu, s_hi[threadIdx.x & 31]);
  const int top = k_lo == k_hi ? 0 : 32 - __clz(k_lo ^ k_hi);        // the keys agree in all bits from `top` up

  // 8-bit digits, most significant first, until the bucket of the keep_k-th largest score is kept whole: that score's key
  // (or, when the pass ends early, the key just below the bucket)
  uint32_t known = top >= 32 ? 0u : ~((1u << top) - 1u);   // mask of the digits fixed so far
  uint32_t prefix = k_lo & known;
  int remaining = keep_k;
  for (int hi_bit = top; hi_bit > 0;) {
    const int shift = max(hi_bit - 8, 0);
    for (int j = threadIdx.x; j < nv; j += blockDim.x) {
      const uint32_t key = s_key[j];
      if ((key & known) == prefix) atomicAdd(&s_hist[(key >> shift) & ((1u << (hi_bit - shift)) - 1u)], 1);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      // lane L owns digits 255-8L .. 248-8L (descending); find where the running count reaches `remaining`
      int c[8], mine = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) { c[e] = s_hist[255 - 8 * lane - e]; mine += c[e]; }
      int inc = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      const int before = inc - mine;
      if (before < remaining && remaining <= inc) {
        int run = before;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (run < remaining && run + c[e] >= remaining) {
            s_prefix = prefix | ((uint32_t)(255 - 8 * lane - e) << shift);
            s_remaining = remaining - run;
            s_bucket = c[e];
          }
          run += c[e];
        }
      }
      // the counters of the next pass
      __syncwarp();
#pragma unroll
      for (int e = 0; e < 8; ++e) s_hist[255 - 8 * lane - e] = 0;
    }
    known |= ((1u << (hi_bit - shift)) - 1u) << shift;
    hi_bit = shift;
    __syncthreads();
    prefix = s_prefix;
    remaining = s_remaining;
    if (remaining == s_bucket) {            // the whole bucket is kept: everything above the key just below it
      if (prefix != 0u) { prefix -= 1u; remaining = 0; break; }
    }
  }
  const uint32_t kth = prefix;        // key of the keep_k-th largest score
  const int take_equal = remaining;   // how many tokens with exactly that key are kept (lowest indices)

  // ordered emission: thread t owns the contiguous indices [t*per, (t+1)*per)
  const int per = (nv + blockDim.x - 1) / blockDim.x;
  const int lo = min(nv, (int)threadIdx.x * per), hi = min(nv, lo + per);
  int n_eq = 0;
  for (int j = lo; j < hi; ++j) n_eq += (s_key[j] == kth);
  int tot;
  int eq_before = block_exclusive_scan(n_eq, s_scan, tot);
  int n_keep = 0;
  {
    int e = eq_before;
    for (int j = lo; j < hi; ++j) {
      const uint32_t key = s_key[j];
      n_keep += (key > kth) || (key == kth && e < take_equal);
      e += (key == kth);
    }
  }
  int keep_before = block_exclusive_scan(n_keep, s_scan, tot);
  {
    int e = eq_before, kp = keep_before;
    for (int j = lo; j < hi; ++j) {
      const uint32_t key = s_key[j];
      const bool kept = (key > kth) || (key == kth && e < take_equal);
      e += (key == kth);
      if (kept) {
        keep_b[kp] = j; role_b[j] = kp; ++kp;
      } else {
        const int dp = j - kp;
        drop_b[dp] = j; role_b[j] = -(dp + 1);
      }
    }
  }
  for (int j = nv - keep_k + threadIdx.x; j < nd_max; j += blockDim.x) drop_b[j] = -1;
  for (int j = nv + threadIdx.x; j < max_vis; j += blockDim.x) role_b[j] = 0;
}

// role map from caller-provided keep / drop lists (entry point asap_merge)
__global__ void role_map_kernel(const SampleDesc *desc, int max_vis, int keep_k,
                                const int32_t *__restrict__ keep_idx,
                                const int32_t *__restrict__ drop_idx, int32_t *__restrict__ role,
                                int32_t *__restrict__ assign, float *__restrict__ best_sim,
                                int sim_follows) {
  pdl_enter();
  const int b = blockIdx.y;
  const SampleDesc d = ld_prev(desc + b);
  const int nd_max = max_vis - keep_k;
  {
    const int first = (d.valid && sim_follows) ? d.nv - keep_k : 0;
    for (int j = first + blockIdx.x * blockDim.x + threadIdx.x; j < nd_max; j += gridDim.x * blockDim.x) {
      assign[(size_t)b * nd_max + j] = -1;
      if (best_sim) best_sim[(size_t)b * nd_max + j] = 0.f;
    }
  }
  if (!d.valid) return;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < d.nv; t += gridDim.x * blockDim.x) {
    if (t < keep_k) {
      const int j = keep_idx[(size_t)b * keep_k + t];
      if (j >= 0 && j < d.nv) role[(size_t)b * max_vis + j] = t;
    } else {
      const int dp = t - keep_k;
      const int j = drop_idx[(size_t)b * nd_max + dp];
      if (j >= 0 && j < d.nv) role[(size_t)b * max_vis + j] = -(dp + 1);
    }
  }
}

// =======================================================================================
// kept_gather: one warp per kept slot.  The kept row is copied to its slot of the dense
// [B*keep_k, D] operand of the similarity GEMM and its inverse norm 1/||h|| is stored (0 if
// ||h|| < 1e-12, which makes every similarity to that slot 0)   (Sec. 4.2).  With member_bits the slot's row of
// member bits is cleared for the similarity kernel.
// =======================================================================================
constexpr int GATHER_THREADS = 256;

__global__ void __launch_bounds__(GATHER_THREADS)
kept_gather_kernel(const __nv_bfloat16 *__restrict__ hidden, const SampleDesc *desc,
                   int D, int keep_k, const int32_t *__restrict__ keep_idx,
                   __nv_bfloat16 *__restrict__ kept_rows /*[B*keep_k, D]*/,
                   float *__restrict__ kept_inv /*[B*keep_k]*/, uint32_t *__restrict__ member_bits /*[B*keep_k, bit_words], nullable*/,
                   int bit_words) {
  pdl_enter();
  const int b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = blockIdx.x * (GATHER_THREADS / 32) + warp;
  if (slot >= keep_k) return;
  const int kept = ld_prev(keep_idx + (size_t)b * keep_k + slot);      // (beside the descriptor, not behind it)
  const SampleDesc d = ld_prev(desc + b);
  if (!d.valid) return;
  const int j = min(max(kept, 0), d.nv - 1);
  const uint4 *src = reinterpret_cast<const uint4 *>(hidden + (size_t)(d.row0 + d.v0 + j) * D);
  uint4 *dst = reinterpret_cast<uint4 *>(kept_rows + ((size_t)b * keep_k + slot) * D);
  const int nvec = D / 8;
  if (member_bits)
    for (int w = lane; w < bit_words; w += 32) member_bits[((size_t)b * keep_k + slot) * bit_words + w] = 0u;
  float ss = 0.f;
  for (int v = lane; v < nvec; v += 256) {
    uint4 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v + 32 * u < nvec) x[u] = __ldg(src + v + 32 * u);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v + 32 * u < nvec) {
        float f[8];
        unpack8(x[u], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) ss += f[e] * f[e];
        dst[v + 32 * u] = x[u];
      }
  }
  ss = warp_sum(ss);
  if (lane == 0) {
    const float nrm = sqrtf(ss);
    kept_inv[(size_t)b * keep_k + slot] = nrm >= 1e-12f ? 1.0f / nrm : 0.f;
  }
}

// =======================================================================================
// csr_block: group the dropped tokens of one sample by destination slot (counting sort, stable
// in dropped order so the merge adds its members in a fixed order).  Run by one whole block of W
// warps (six, ten in the gathered and eleven in the two-row-tile form): warp w owns the w-th contiguous
// chunk of dropped positions, counts its chunk into its own histogram, and after a scan over (slot,
// warp) writes its chunk's positions behind those of the warps before it.  s_cnt needs (W + 1) * keep_k ints, s_scan 33 ints.
// seg [B, keep_k+1], members [B, max_vis-keep_k] (dropped POSITIONS, ascending inside a slot).
// With drop_idx, salience and member_meta given, member_meta [B, max_vis-keep_k] receives, beside every
// entry of `members`, the member's visual index and its merge weight (the salience, as bits): the
// merge kernel then reaches a member's row in two dependent loads instead of four.
// =======================================================================================
constexpr int CSR_BATCH = 6;      // 2736 dropped tokens: one warp's chunk of 288 positions is two batches instead of nine round trips

__device__ __forceinline__ void csr_block(const SampleDesc &d, int b, int max_vis, int keep_k,
                                          const int32_t *__restrict__ assign,
                                          int32_t *__restrict__ seg, int32_t *__restrict__ members,
                                          int *s_cnt, int *s_scan,
                                          const int32_t *__restrict__ drop_idx = nullptr,
                                          const float *__restrict__ salience = nullptr,
                                          int2 *__restrict__ member_meta = nullptr) {
  int32_t *seg_b = seg + (size_t)b * (keep_k + 1);
  const int nd_max = max_vis - keep_k, nd = d.nv - keep_k;
  const int32_t *as_b = assign + (size_t)b * nd_max;
  int32_t *mem_b = members + (size_t)b * nd_max;
  const int W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = (((nd + W - 1) / W) + 31) & ~31;        // positions per warp, a multiple of 32
  int *hist = s_cnt;                                         // [W][keep_k]
  int *tot = s_cnt + W * keep_k;                             // [keep_k] members per slot
  for (int i = threadIdx.x; i < (W + 1) * keep_k; i += blockDim.x) s_cnt[i] = 0;
  __syncthreads();
  const int p_lo = min(nd, warp * chunk), p_hi = min(nd, p_lo + chunk);
  // (CSR_BATCH groups of 32 positions at a time, here and below, so that their loads are in flight together)
  for (int base = p_lo; base < p_hi; base += 32 * CSR_BATCH) {
    int a[CSR_BATCH];
#pragma unroll
    for (int t = 0; t < CSR_BATCH; ++t) {
      const int p = base + 32 * t + lane;
      a[t] = p < p_hi ? __ldcg(as_b + p) : -1;
    }
#pragma unroll
    for (int t = 0; t < CSR_BATCH; ++t)
      if (a[t] >= 0 && a[t] < keep_k) atomicAdd(&hist[warp * keep_k + a[t]], 1);
  }
  __syncthreads();
  // per slot: turn the per-warp counts into per-warp offsets inside the slot, and total them
  for (int i = threadIdx.x; i < keep_k; i += blockDim.x) {
    int run = 0;
    for (int w = 0; w < W; ++w) {
      const int c = hist[w * keep_k + i];
      hist[w * keep_k + i] = run;
      run += c;
    }
    tot[i] = run;
  }
  __syncthreads();
  // exclusive scan over slots; thread t owns a contiguous range of slots
  const int per = (keep_k + blockDim.x - 1) / blockDim.x;
  const int lo = min(keep_k, (int)threadIdx.x * per), hi = min(keep_k, lo + per);
  int mine = 0;
  for (int i = lo; i < hi; ++i) mine += tot[i];
  int total;
  int run = block_exclusive_scan(mine, s_scan, total);
  for (int i = lo; i < hi; ++i) {
    const int c = tot[i];
    seg_b[i] = run;
    tot[i] = run;        // becomes the slot's base
    run += c;
  }
  if (threadIdx.x == 0) seg_b[keep_k] = total;
  __syncthreads();
  // stable fill: every warp walks its chunk 32 positions at a time in ascending order
  const bool meta = drop_idx && salience && member_meta;
  for (int base0 = p_lo; base0 < p_hi; base0 += 32 * CSR_BATCH) {
    int av[CSR_BATCH];
    int2 mv[CSR_BATCH];
#pragma unroll
    for (int t = 0; t < CSR_BATCH; ++t) {
      const int p = base0 + 32 * t + lane;
      av[t] = p < p_hi ? __ldcg(as_b + p) : -1;
      mv[t] = make_int2((meta && p < p_hi) ? __ldg(drop_idx + (size_t)b * nd_max + p) : 0, 0);
    }
    if (meta) {
#pragma unroll
      for (int t = 0; t < CSR_BATCH; ++t) {
        mv[t].x = min(max(mv[t].x, 0), d.nv - 1);
        mv[t].y = __float_as_int(__ldcg(salience + (size_t)b * max_vis + mv[t].x));
      }
    }
#pragma unroll
    for (int t = 0; t < CSR_BATCH; ++t) {
      const int p = base0 + 32 * t + lane;
      if (base0 + 32 * t >= p_hi) break;
      int a = av[t];
      if (a >= keep_k) a = -1;
      const unsigned peers = __match_any_sync(0xffffffffu, a);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      int cur = 0;
      if (a >= 0) cur = hist[warp * keep_k + a];
      __syncwarp();
      if (a >= 0) {
        mem_b[tot[a] + cur + rank] = p;
        if (meta) member_meta[(size_t)b * nd_max + tot[a] + cur + rank] = mv[t];
        if (rank == 0) hist[warp * keep_k + a] = cur + __popc(peers);
      }
      __syncwarp();
    }
  }
}

// =======================================================================================
// route: Sec. 4.2 inside the kept set, one block per sample.  Input: the keep_k x keep_k cosine
// matrix S of the kept rows, the salience, the attention mass, stage 1's kept / pruned lists.
//   A  visiting order of the kept slots: salience descending, sequence index ascending.
//   B  bit matrix  M[p] = { q : S[p][q] > t }, from the similarity kernel where that form writes it.
//   C  A slot is absorbed if an anchor that was visited before it is similar to it (while the pruned pool can still refill a
//      slot, i.e. at most nv - keep_k times); any other slot becomes an anchor.  This is the greedy
//      rule "join the most similar earlier anchor if that similarity exceeds t, else become an anchor" with the question
//      WHICH anchor left to step D.  Decided in rounds by all threads: as many as the longest chain of slots each of which
//      waits for the one before, two to four on clustered rows; after some rounds that decide few slots the rest is taken in order
//      (route_walk).  (One warp walking the order took 38 of the kernel's 174 us on 24 x 576 slots, reading the similarities a
//      second time for D 50, forming the bit matrix here 30; 174 -> 48 us in all, 43 with D's loads after its scan.
//      Rounds alone: 0.57 ms on a chain through 576 slots and 9.5 ms through 1024; with the walk 62 and 270 us.)
//   D  every absorbed slot finds the most similar anchor that was visited before it (lowest slot
//      among equals), looking only at the anchors in its row of the bit matrix.
//   E  the vacated slots are refilled with the pruned tokens of largest attention mass (radix
//      select, lower index first among equals).
//   F  anchors and refilled tokens, in sequence order, form the final kept list; the absorbed
//      tokens, ascending, form the source list with their anchor's FINAL slot; CSR of that list.
// Outputs use the layouts of the merge kernel: final_keep [B, keep_k], src_idx / src_assign /
// src_sim [B, max_vis - keep_k] (padding -1 / 0), seg [B, keep_k + 1], members [B, max_vis - keep_k].
// =======================================================================================
constexpr int ROUTE_THREADS = 1024;
constexpr int ROUTE_MAX_WORDS = 128;                    // keep_k <= 32 * 128
constexpr int ROUTE_WALK_BELOW = 32;                    // threads that decide something in a round, below which it is a slow one
constexpr int ROUTE_SLOW_ROUNDS = 8;

struct RouteArgs {
  const SampleDesc *desc;
  int max_vis, keep_k, kw;        // kw = ceil(keep_k / 32)
  float threshold;
  const float *smat;              // [B, keep_k, keep_k]
  uint32_t *mask_g;               // [B, keep_k, kw] bit matrix in global memory
  int mask_in_smem;               // the bit matrix fits shared memory (else mask_g is used where it lies)
  int mask_written;               // mask_g was filled by the similarity kernel
  int union_words;                // 32-bit words of the last region of shared memory
  const float *salience, *mass;   // [B, max_vis]
  const int32_t *keep_idx;        // [B, keep_k]            stage 1
  const int32_t *drop_idx;        // [B, max_vis - keep_k]  stage 1
  int32_t *final_keep, *src_idx, *src_assign, *seg, *members, *n_absorbed;
  float *src_sim;                 // nullable
  const uint32_t *status;
};

// The undecided slots in visiting order, 32 at a time, by the whole block.  Rows hold earlier slots only, and those before the group
// are all decided: warp w looks whether the group's w-th slot has an anchor among them and which of the group come before
// it; one warp then decides the 32 one after the other out of registers.
__device__ __forceinline__ void route_walk(const int *s_order, const uint32_t *mask, uint32_t *s_anchor, const uint32_t *s_gone,
                                           int *s_flag, uint32_t *s_before, int k, int kw) {
  static_assert(ROUTE_THREADS == 1024, "a warp per slot of a group");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r0 = 0; r0 < k; r0 += 32) {
    const int q = r0 + lane < k ? s_order[r0 + lane] : -1;
    const uint32_t todo = __ballot_sync(0xffffffffu, q >= 0 && !(((s_anchor[q >> 5] | s_gone[q >> 5]) >> (q & 31)) & 1u));
    if (todo == 0u) continue;                             // (the same in every warp)
    if ((todo >> warp) & 1u) {
      const uint32_t *row = mask + (size_t)__shfl_sync(0xffffffffu, q, warp) * kw;
      uint32_t hit = 0u;
      for (int w = lane; w < kw; w += 32) hit |= row[w] & s_anchor[w];
      const uint32_t before = __ballot_sync(0xffffffffu, q >= 0 && ((row[q >> 5] >> (q & 31)) & 1u));
      const bool by_anchor = __any_sync(0xffffffffu, hit != 0u);
      if (lane == 0) s_before[warp] = by_anchor ? before | (1u << warp) : before & ~(1u << warp);
    }
    __syncthreads();
    if (warp == 0) {
      const uint32_t before = s_before[lane];
      uint32_t anchors = 0u;
#pragma unroll 4
      for (int t = 0; t < 32; ++t)
        if (!(__shfl_sync(0xffffffffu, before, t) & (anchors | (1u << t)))) anchors |= (1u << t) & todo;
      if ((anchors >> lane) & 1u) {
        atomicOr(&s_anchor[q >> 5], 1u << (q & 31));
        s_flag[q] = 1;
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(ROUTE_THREADS)
route_kernel(RouteArgs a) {
  pdl_enter();
  extern __shared__ uint32_t r_smem[];
  __shared__ int s_hist[256];
  __shared__ int s_scan[33];
  __shared__ uint32_t s_prefix;
  __shared__ int s_remaining, s_nabs;
  __shared__ uint32_t s_anchor[ROUTE_MAX_WORDS], s_gone[ROUTE_MAX_WORDS];   // decided slots: anchors, absorbed
  const int b = blockIdx.x;
  const SampleDesc d = a.desc[b];
  const int k = a.keep_k, kw = a.kw, nd_max = a.max_vis - k;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x;
  int32_t *fk_b = a.final_keep + (size_t)b * k;
  int32_t *si_b = a.src_idx + (size_t)b * nd_max;
  int32_t *sa_b = a.src_assign + (size_t)b * nd_max;
  float *ss_b = a.src_sim ? a.src_sim + (size_t)b * nd_max : nullptr;
  int32_t *seg_b = a.seg + (size_t)b * (k + 1);
  int32_t *mem_b = a.members + (size_t)b * nd_max;
  // (a similarity kernel that gave up has left the matrices unwritten: they hold whatever the caller's scratch held.  Nothing
  // writes the status word while this kernel runs)
  if (!d.valid || (__ldcg(a.status) & STATUS_SIM_TIMEOUT)) {
    for (int j = tid; j < k; j += nthr) fk_b[j] = -1;
    for (int j = tid; j < nd_max; j += nthr) { si_b[j] = -1; sa_b[j] = -1; if (ss_b) ss_b[j] = 0.f; }
    for (int j = tid; j <= k; j += nthr) seg_b[j] = 0;
    if (tid == 0 && a.n_absorbed) a.n_absorbed[b] = 0;
    return;
  }
  const int nv = d.nv, nd = nv - k;
  // shared memory: [tmp k][order k][rank k][flag k][dest k] [union: bit matrix k*kw | key nd_max + pos max_vis]
  uint32_t *s_tmp = r_smem;
  int *s_order = reinterpret_cast<int *>(r_smem + k);
  int *s_rank = s_order + k;
  int *s_flag = s_rank + k;
  int *s_dest = s_flag + k;
  uint32_t *s_union = r_smem + 5 * (size_t)k;
  uint32_t *mask = a.mask_in_smem ? s_union : a.mask_g + (size_t)b * k * kw;
  const int32_t *keep_b = a.keep_idx + (size_t)b * k;
  const int32_t *drop_b = a.drop_idx + (size_t)b * nd_max;
  const float *sal_b = a.salience + (size_t)b * a.max_vis;
  const float *S = a.smat + (size_t)b * k * k;

  // ---- A: visiting order.  Keys are order-preserving integers, so NaN cannot break the permutation.
  for (int p = tid; p < k; p += nthr) {
    const int j = min(max(keep_b[p], 0), nv - 1);
    s_tmp[p] = score_key(sal_b[j]);
  }
  // the attention mass of this thread's first pruned tokens, for E: two dependent loads that end long before they are needed
  uint32_t mass_key[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int i = tid + t * nthr;
    mass_key[t] = i < nd ? score_key(__ldg(a.mass + (size_t)b * a.max_vis + min(max(__ldg(drop_b + i), 0), nv - 1))) : 0u;
  }
  __syncthreads();
  for (int p = tid; p < k; p += nthr) {
    const uint32_t mine = s_tmp[p];
    // the kept list is ascending: an equal key before p is the lower index.  Four keys per (broadcast) load
    int r = 0;
    const uint4 *t4 = reinterpret_cast<const uint4 *>(s_tmp);
    const int pc = p >> 2, nc = k >> 2;
#pragma unroll 4
    for (int c = 0; c < pc; ++c) {
      const uint4 o = t4[c];
      r += (o.x >= mine) + (o.y >= mine) + (o.z >= mine) + (o.w >= mine);
    }
    uint32_t own[4], last[4];                           // p's own four, and the up to three past the last whole four
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      own[e] = pc * 4 + e < k ? s_tmp[pc * 4 + e] : 0u;
      last[e] = pc < nc && nc * 4 + e < k ? s_tmp[nc * 4 + e] : 0u;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) r += (own[e] > mine || (own[e] == mine && pc * 4 + e < p)) + (last[e] > mine);
#pragma unroll 4
    for (int c = pc + 1; c < nc; ++c) {
      const uint4 o = t4[c];
      r += (o.x > mine) + (o.y > mine) + (o.z > mine) + (o.w > mine);
    }
    s_rank[p] = r;
    s_order[r] = p;
    s_flag[p] = 0;
  }
  for (int w = tid; w < kw; w += nthr) { s_anchor[w] = 0u; s_gone[w] = 0u; }
  // ---- B: bit matrix  M[p] = { q : S[p][q] > t }
  if (!a.mask_written) {
    for (int p = warp; p < k; p += (nthr >> 5)) {     // one warp per row, coalesced
      const float *row = S + (size_t)p * k;
      for (int w0 = 0; w0 < kw; w0 += 16) {             // sixteen loads in flight per lane
        float v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int q = (w0 + e) * 32 + lane;
          v[e] = q < k ? __ldcg(row + q) : -INFINITY;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int q = (w0 + e) * 32 + lane;
          const unsigned bits = __ballot_sync(0xffffffffu, q < k && q != p && v[e] > a.threshold);
          if (lane == 0 && w0 + e < kw) mask[(size_t)p * kw + w0 + e] = bits;
        }
      }
    }
  } else if (a.mask_in_smem) {
    const uint32_t *src = a.mask_g + (size_t)b * k * kw;
#pragma unroll 8
    for (int i = tid; i < k * kw; i += nthr) mask[i] = __ldcg(src + i);
  }
  __syncthreads();
  // ---- C: rounds.  A slot with an earlier anchor among its neighbours is absorbed; one whose earlier neighbours are all
  // absorbed is an anchor; any other waits.  The first undecided slot of the visiting order is decided in every round, and the
  // outcome is that of walking the slots in that order (a slot's fate depends on earlier slots alone).
  // First every row of the matrix loses the slots that come after its own (a thread works on its own rows only): from then on
  // a round is a few words of bit operations per slot.
  // (the loops over a thread's slots tid, tid + nthr, ... are not unrolled: up to 1024 slots make one trip, and the kernel is short
  // enough for the fetching of its code to count)
  uint32_t open = 0u;                                 // bit t: slot tid + t * nthr is undecided (k <= 4096)
#pragma unroll 1
  for (int t = 0; tid + t * nthr < k; ++t) {
    const int p = tid + t * nthr;
    open |= 1u << t;
    const int rp = s_rank[p];
    uint32_t *row = mask + (size_t)p * kw;
#pragma unroll 4
    for (int w = 0; w < kw; ++w) {
      uint32_t word = row[w], rest = word;
      while (rest) {
        const int bit = __ffs(rest) - 1;
        rest &= rest - 1;
        if (s_rank[w * 32 + bit] > rp) word &= ~(1u << bit);
      }
      row[w] = word;
    }
  }
  // A round costs the same whether it decides one slot or all.  After ROUTE_SLOW_ROUNDS in a row that decide fewer slots than the
  // walk does in their time (one such round says nothing: the next may absorb all others) the rest is taken in order, so the
  // rounds are bounded whatever the matrix holds.
  for (int slow = 0;;) {
    uint32_t anchors = 0u, absorbed = 0u;             // this round's verdicts, like `open`
#pragma unroll 1
    for (int t = 0; tid + t * nthr < k; ++t) {
      if (!((open >> t) & 1u)) continue;
      const uint32_t *row = mask + (size_t)(tid + t * nthr) * kw;
      uint32_t by_anchor = 0u, left = 0u;
#pragma unroll 4
      for (int w = 0; w < kw; ++w) {
        const uint32_t word = row[w];
        by_anchor |= word & s_anchor[w];
        left |= word & ~s_gone[w];
      }
      if (by_anchor) absorbed |= 1u << t;
      else if (!left) anchors |= 1u << t;
    }
    open &= ~(anchors | absorbed);
    const int progress = __syncthreads_count((anchors | absorbed) != 0u);   // (and every slot has looked at the last round's decisions)
#pragma unroll 1
    for (uint32_t rest = anchors | absorbed; rest; rest &= rest - 1) {
      const int t = __ffs(rest) - 1, p = tid + t * nthr;
      const bool anchor = (anchors >> t) & 1u;
      atomicOr(anchor ? &s_anchor[p >> 5] : &s_gone[p >> 5], 1u << (p & 31));
      if (anchor) s_flag[p] = 1;
    }
    if (!__syncthreads_or(open != 0u)) break;
    slow = progress < ROUTE_WALK_BELOW ? slow + 1 : 0;
    if (slow == ROUTE_SLOW_ROUNDS) {
      route_walk(s_order, mask, s_anchor, s_gone, s_flag, reinterpret_cast<uint32_t *>(s_hist), k, kw);
      break;
    }
  }
  // at most nd slots are absorbed, the first ones of the visiting order: later ones stay anchors
  {
    const int per = (k + nthr - 1) / nthr;
    const int lo = min(k, tid * per), hi = min(k, lo + per);
    int cnt = 0;
    for (int r = lo; r < hi; ++r) cnt += !s_flag[s_order[r]];
    int tot;
    int run = block_exclusive_scan(cnt, s_scan, tot);
    if (tot > nd) {
      for (int r = lo; r < hi; ++r) {
        const int p = s_order[r];
        if (!s_flag[p] && run++ >= nd) {
          s_flag[p] = 1;
          atomicOr(&s_anchor[p >> 5], 1u << (p & 31));
        }
      }
    }
    if (tid == 0) s_nabs = min(tot, nd);
  }
  __syncthreads();
  const int n_abs = s_nabs;
  // ---- D: destination of every absorbed slot: the most similar earlier anchor (it lies above the threshold, since one
  // of them does), the lowest slot among equals
  for (int p = tid; p < k; p += nthr) {
    int best_q = -1;
    float best = -INFINITY;
    if (!s_flag[p]) {
      const float *row = S + (size_t)p * k;
      // (a few such anchors are the rule: their similarities are loaded after the scan, by all lanes together.  Inside the scan
      // the lanes come upon theirs in different words, a trip to memory each)
      constexpr int FEW = 6;
      int c[FEW], n_words = 0, n_cand = 0;              // the latest words' lowest candidates, c[0] the last
#pragma unroll
      for (int e = 0; e < FEW; ++e) c[e] = 0;
#pragma unroll 4
      for (int w = 0; w < kw; ++w) {
        const uint32_t cand = mask[(size_t)p * kw + w] & s_anchor[w];
        if (cand) {
#pragma unroll
          for (int e = FEW - 1; e > 0; --e) c[e] = c[e - 1];
          c[0] = w * 32 + __ffs(cand) - 1;
          ++n_words;
        }
        n_cand += __popc(cand);
      }
      if (n_words == n_cand && n_cand <= FEW) {
        float v[FEW];
#pragma unroll
        for (int e = 0; e < FEW; ++e) v[e] = e < n_cand ? __ldcg(row + c[e]) : -INFINITY;
#pragma unroll
        for (int e = FEW - 1; e >= 0; --e)              // ascending slots: the first maximum stays
          if (v[e] > best) { best = v[e]; best_q = c[e]; }
      } else {
#pragma unroll 4
        for (int w = 0; w < kw; ++w) {
          uint32_t cand = mask[(size_t)p * kw + w] & s_anchor[w];
          while (cand) {
            const int q = w * 32 + __ffs(cand) - 1;
            cand &= cand - 1;
            const float v = __ldcg(row + q);
            if (v > best) { best = v; best_q = q; }
          }
        }
      }
    }
    s_dest[p] = best_q;
    s_tmp[p] = __float_as_uint(best);
  }
  __syncthreads();      // the bit matrix is dead from here on: its space is reused
  uint32_t *s_key = s_union;                                  // [nd]
  int *s_pos = reinterpret_cast<int *>(s_union + nd_max);     // [nv] 1 + final slot, 0 = not in the final list
  // ---- E: the n_abs pruned tokens of largest attention mass
  const float *mass_b = a.mass + (size_t)b * a.max_vis;
  for (int v = tid; v < nv; v += nthr) s_pos[v] = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (tid + t * nthr < nd) s_key[tid + t * nthr] = mass_key[t];
  for (int i = tid + 4 * nthr; i < nd; i += nthr) {
    const int j = min(max(drop_b[i], 0), nv - 1);
    s_key[i] = score_key(mass_b[j]);
  }
  if (tid == 0) { s_prefix = 0u; s_remaining = n_abs; }
  __syncthreads();
  if (n_abs > 0) {
    uint32_t known = 0u;
    for (int shift = 24; shift >= 0; shift -= 8) {
      for (int i = tid; i < 256; i += nthr) s_hist[i] = 0;
      __syncthreads();
      const uint32_t prefix = s_prefix;
      for (int i = tid; i < nd; i += nthr) {
        const uint32_t key = s_key[i];
        if ((key & known) == prefix) atomicAdd(&s_hist[(key >> shift) & 255u], 1);
      }
      __syncthreads();
      if (tid < 32) {
        int mine = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) mine += s_hist[255 - 8 * lane - e];
        int inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += t;
        }
        const int remaining = s_remaining;
        __syncwarp();
        const int before = inc - mine;
        if (before < remaining && remaining <= inc) {
          int run = before;
          for (int e = 0; e < 8; ++e) {
            const int digit = 255 - 8 * lane - e;
            const int c = s_hist[digit];
            if (run + c >= remaining) {
              s_prefix = prefix | ((uint32_t)digit << shift);
              s_remaining = remaining - run;
              break;
            }
            run += c;
          }
        }
      }
      known |= 255u << shift;
      __syncthreads();
    }
    const uint32_t kth = s_prefix;
    const int take_equal = s_remaining;
    const int per = (nd + nthr - 1) / nthr;
    const int lo = min(nd, tid * per), hi = min(nd, lo + per);
    int n_eq = 0;
    for (int i = lo; i < hi; ++i) n_eq += (s_key[i] == kth);
    int tot;
    int e = block_exclusive_scan(n_eq, s_scan, tot);
    for (int i = lo; i < hi; ++i) {
      const uint32_t key = s_key[i];
      if (key > kth || (key == kth && e < take_equal)) s_pos[min(max(drop_b[i], 0), nv - 1)] = 1;
      e += (key == kth);
    }
  }
  for (int p = tid; p < k; p += nthr)
    if (s_flag[p]) s_pos[min(max(keep_b[p], 0), nv - 1)] = 1;
  __syncthreads();
  // ---- F: final kept list in sequence order
  {
    const int per = (nv + nthr - 1) / nthr;
    const int lo = min(nv, tid * per), hi = min(nv, lo + per);
    int cnt = 0;
    for (int v = lo; v < hi; ++v) cnt += s_pos[v];
    int tot;
    int run = block_exclusive_scan(cnt, s_scan, tot);
    for (int v = lo; v < hi; ++v) {
      if (s_pos[v]) {
        if (run < k) fk_b[run] = v;
        s_pos[v] = ++run;
      }
    }
    // fewer than keep_k can only come from malformed input lists: pad
    for (int j = tot + tid; j < k; j += nthr) fk_b[j] = -1;
  }
  __syncthreads();
  // source list: absorbed slots in ascending order, with the final slot of their anchor
  {
    const int per = (k + nthr - 1) / nthr;
    const int lo = min(k, tid * per), hi = min(k, lo + per);
    int cnt = 0;
    for (int p = lo; p < hi; ++p) cnt += !s_flag[p];
    int tot;
    int run = block_exclusive_scan(cnt, s_scan, tot);
    for (int p = lo; p < hi; ++p) {
      if (!s_flag[p] && run < nd_max) {
        const int q = s_dest[p];
        const int slot = q >= 0 ? s_pos[min(max(keep_b[q], 0), nv - 1)] - 1 : -1;
        si_b[run] = keep_b[p];
        sa_b[run] = (slot >= 0 && slot < k) ? slot : -1;
        if (ss_b) ss_b[run] = __uint_as_float(s_tmp[p]);
        s_key[run] = (uint32_t)((slot >= 0 && slot < k) ? slot : -1);     // for the grouping below
        ++run;
      }
    }
    for (int j = n_abs + tid; j < nd_max; j += nthr) { si_b[j] = -1; sa_b[j] = -1; if (ss_b) ss_b[j] = 0.f; }
  }
  if (tid == 0 && a.n_absorbed) a.n_absorbed[b] = n_abs;
  __syncthreads();
  // grouping by destination (counting sort, stable in source order): as many warps as there is room for a histogram each, up to
  // eight, take a contiguous chunk of the sources (the region holds max_vis - k sources and max_vis words more: one at least)
  {
    int *s_cnt = s_order;                     // reuse: the visiting order is no longer needed
    int *hist = reinterpret_cast<int *>(s_union) + n_abs;      // [W][k] behind the sources' slots
    const int W = min(8, (a.union_words - n_abs) / k);
    const int chunk = (((n_abs + W - 1) / W) + 31) & ~31;
    const int p_lo = min(n_abs, warp * chunk), p_hi = warp < W ? min(n_abs, p_lo + chunk) : p_lo;
    for (int i = tid; i < W * k; i += nthr) hist[i] = 0;
    __syncthreads();
    for (int i = p_lo + lane; i < p_hi; i += 32) {
      const int sl = (int)s_key[i];
      if (sl >= 0 && sl < k) atomicAdd(&hist[warp * k + sl], 1);
    }
    __syncthreads();
    const int per = (k + nthr - 1) / nthr;
    const int lo = min(k, tid * per), hi = min(k, lo + per);
    int mine = 0;
    for (int sl = lo; sl < hi; ++sl) {
      int run = 0;
      for (int w = 0; w < W; ++w) {
        const int c = hist[w * k + sl];
        hist[w * k + sl] = run;               // this warp's offset inside the slot
        run += c;
      }
      s_cnt[sl] = run;
      mine += run;
    }
    int tot;
    int run = block_exclusive_scan(mine, s_scan, tot);
    for (int sl = lo; sl < hi; ++sl) {
      const int c = s_cnt[sl];
      seg_b[sl] = run;
      s_cnt[sl] = run;
      run += c;
    }
    if (tid == 0) seg_b[k] = tot;
    __syncthreads();
    // every warp walks its chunk 32 sources at a time in ascending order, so members stay ascending inside a slot
    for (int base = p_lo; base < p_hi; base += 32) {
      const int i = base + lane;
      int sl = i < p_hi ? (int)s_key[i] : -1;
      if (sl >= k) sl = -1;
      const unsigned peers = __match_any_sync(0xffffffffu, sl);
      const int rank = __popc(peers & ((1u << lane) - 1u));
      int at = 0;
      if (sl >= 0) at = hist[warp * k + sl];
      __syncwarp();
      if (sl >= 0) {
        mem_b[s_cnt[sl] + at + rank] = i;
        if (rank == 0) hist[warp * k + sl] = at + __popc(peers);
      }
      __syncwarp();
    }
  }
}

// =======================================================================================
// merge_compact: grid (keep_k, or an eighth of it, + copy-row groups, B).
//   blockIdx.x <  keep_k : the block owns one kept visual row (or eight, see below).  Its members (the dropped tokens
//                          assigned to that slot) are first listed in shared memory, then their rows are streamed
//                          up to four at a time and accumulated in fp32 in ascending order:  (s_hat_i h_i + sum_j s_hat_j h_j) / (s_hat_i +
//                          sum_j s_hat_j)   (Eq. 5), rounded to bf16 once.  No members, merging
//                          off, or total weight <= eps: the row is copied.
//   blockIdx.x >= keep_k : each warp copies one prefix / suffix row.
// Every output row also gets its gathered position id and its source row (hand-off of Fig. 3).
// =======================================================================================
constexpr int MERGE_THREADS = 256;
constexpr int MERGE_COPY_ROWS = MERGE_THREADS / 32;   // copy rows per block
constexpr int MERGE_LIST = 256;                        // members listed per pass
constexpr int MERGE_BATCH = 4;                         // member rows in flight per thread
constexpr int MERGE_WARP_LIST = 64;                    // BITS: members listed per warp and pass
constexpr int MERGE_BIT_WORDS = 4;                     // BITS: words of a slot's bits per lane and pass (4096 visual tokens)

struct MergeArgs {
  const __nv_bfloat16 *hidden;
  const int32_t *pos_ids;
  const SampleDesc *desc;
  int D, max_vis, keep_k, merge_enable;
  float eps;
  const float *salience;
  const int32_t *keep_idx, *drop_idx, *seg, *members;
  const int2 *member_meta;   // [B, max_vis-keep_k] (visual index, weight bits) beside `members`, or nullptr
  const uint32_t *member_bits;   // (BITS only) [B, keep_k, bit_words]: bit j of a slot's row set where visual token j merges into it
  int bit_words;
  int block_rows;            // (not BITS) kept rows per block: 1, or one per warp
  __nv_bfloat16 *out_hidden;
  int32_t *out_pos, *src_row;
};

// NV: 16-byte vectors per thread (D <= NV * 256 * 8); wide rows keep fewer member rows in flight per thread
// so that three or four blocks still fit the register file of an SM.
// LEAN (rows of at most 4096 elements, launches of many waves): two member rows in flight as well, 60 registers,
// four blocks per SM -- more blocks in their dependent look-ups at any time (c4 398 -> 369 us); on launches of a
// few waves the shorter batches cost more than the occupancy gives (c2 24.8 -> 26.6 us), so those keep four rows.
// Rows of 4097-6144 elements (NV = 3): one member row in flight, 64 registers, four blocks per SM as well
// (D = 5120, 1152 of 2304 kept: 280 -> 241 us; 576 of 1152: 151 -> 133 us; 288 of 576: 85 -> 75 us).
// BITS: the similarity kernel left a row of bits per slot instead of a grouping.  Every warp lists the slot's members for itself,
// in ascending order, so the block needs no barrier at all.
template <int NV, bool LEAN = false, bool BITS = false>
__global__ void __launch_bounds__(MERGE_THREADS, NV >= 4 ? 2 : ((LEAN || NV == 3) ? 4 : 3))
merge_compact_kernel(MergeArgs a) {
  constexpr int BATCH = NV == 3 ? 1 : ((NV >= 4 || LEAN) ? 2 : MERGE_BATCH);
  pdl_enter();
  __shared__ int s_j[BITS ? (MERGE_THREADS / 32) * MERGE_WARP_LIST : MERGE_LIST];
  __shared__ float s_w[BITS ? 1 : MERGE_LIST];
  const int b = blockIdx.y;
  const int nvec = a.D / 8;
  const int k = a.keep_k;
  // The look-ups of a kept row that need no other are under way together with the descriptor: behind it they cost every block another
  // round trip before its first row.
  const int lane = threadIdx.x & 31;
  // a block's slots: one, or eight, of which every warp looks its own up
  const int warp = threadIdx.x >> 5, rows = BITS ? 1 : a.block_rows, n_blocks = BITS ? k : (k + rows - 1) / rows;
  const int slot = BITS ? (int)blockIdx.x : (int)blockIdx.x * rows + (rows > 1 ? warp : 0);
  int kept = 0, m_lo = 0, m_hi = 0;
  // BITS: the lanes of a warp own neighbouring words, so that one scan over the lanes gives every member's place
  const uint32_t *bit_row = BITS ? a.member_bits + ((size_t)b * k + slot) * a.bit_words : nullptr;
  uint32_t mw[MERGE_BIT_WORDS];
  int per = 0;
  auto load_words = [&](int w0) {
    per = (min(a.bit_words - w0, 32 * MERGE_BIT_WORDS) + 31) >> 5;
#pragma unroll
    for (int g = 0; g < MERGE_BIT_WORDS; ++g) {
      const int w = w0 + lane * per + g;
      mw[g] = g < per && w < a.bit_words ? (uint32_t)ld_prev(reinterpret_cast<const int *>(bit_row + w)) : 0u;
    }
  };
  if (slot < k) {
    kept = ld_prev(a.keep_idx + (size_t)b * k + slot);
    if (BITS) {
      load_words(0);
    } else if (a.merge_enable) {
      m_lo = ld_prev(a.seg + (size_t)b * (k + 1) + slot);
      m_hi = ld_prev(a.seg + (size_t)b * (k + 1) + slot + 1);
    }
  }
  const SampleDesc d = a.desc[b];
  if (!d.valid) return;
  // a row without members, by one warp
  auto copy_row = [&](size_t grow, int orow) {
    if (lane == 0) {
      a.out_pos[orow] = a.pos_ids[grow];
      a.src_row[orow] = (int32_t)grow;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(a.hidden + grow * a.D);
    uint4 *dst = reinterpret_cast<uint4 *>(a.out_hidden + (size_t)orow * a.D);
    for (int v = lane; v < nvec; v += 32 * 8) {
      uint4 x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (v + 32 * u < nvec) x[u] = __ldg(src + v + 32 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (v + 32 * u < nvec) dst[v + 32 * u] = x[u];
    }
  };
  if ((int)blockIdx.x >= n_blocks) {
    if (blockIdx.z) return;
    // ---------------------------------------------------------------- copy rows, one per warp
    const int c = ((int)blockIdx.x - n_blocks) * MERGE_COPY_ROWS + warp;   // index among prefix + suffix rows
    if (c >= d.n - d.nv) return;
    copy_row((size_t)(d.row0 + (c < d.v0 ? c : c + d.nv)), d.out_row0 + (c < d.v0 ? c : c + k));
    return;
  }
  // ------------------------------------------------------------------ one kept row, by the block
  auto kept_row = [&](int slot, int kept, int m_lo, int m_hi) {
    const int vi = min(max(kept, 0), d.nv - 1);           // visual index
    const size_t grow = (size_t)(d.row0 + d.v0 + vi);
    const int orow = d.out_row0 + d.v0 + slot;
    const int v0 = blockIdx.z * (NV * MERGE_THREADS) + threadIdx.x;       // grid z: pieces of NV * 256 vectors of the row
    if (threadIdx.x == 0 && blockIdx.z == 0) {
      a.out_pos[orow] = a.pos_ids[grow];
      a.src_row[orow] = (int32_t)grow;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(a.hidden + grow * a.D);
    uint4 *dst = reinterpret_cast<uint4 *>(a.out_hidden + (size_t)orow * a.D);
    const int nd_max = a.max_vis - k;
    m_lo = min(max(m_lo, 0), nd_max);
    m_hi = min(max(m_hi, m_lo), nd_max);
    uint4 self[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = v0 + u * MERGE_THREADS;
      if (v < nvec) self[u] = __ldg(src + v);
    }
    if (!BITS && m_hi <= m_lo) {
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = v0 + u * MERGE_THREADS;
        if (v < nvec) dst[v] = self[u];
      }
      return;
    }
    const float *sal_b = a.salience + (size_t)b * a.max_vis;
    const int32_t *mem_b = a.members + (size_t)b * nd_max;
    const int32_t *drop_b = a.drop_idx + (size_t)b * nd_max;
    const float w_self = sal_b[vi];
    float acc[NV][8];
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      float f[8];
      unpack8(self[u], f);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[u][e] = w_self * f[e];
    }
    float den = w_self;
    bool merged = !BITS;
    const __nv_bfloat16 *vis0 = a.hidden + (size_t)(d.row0 + d.v0) * a.D;
    // adds the members listed in s_j (and s_w, unless BITS) at `at`
    auto add_members = [&](int at, int cnt) {
      for (int m0 = 0; m0 < cnt; m0 += BATCH) {
        uint4 x[BATCH][NV];
        float wt[BATCH];
#pragma unroll
        for (int t = 0; t < BATCH; ++t) {
          if (m0 + t < cnt) {
            const int j = s_j[at + m0 + t];
            wt[t] = BITS ? __ldg(sal_b + j) : s_w[at + m0 + t];
            const uint4 *msrc = reinterpret_cast<const uint4 *>(vis0 + (size_t)j * a.D);
#pragma unroll
            for (int u = 0; u < NV; ++u) {
              const int v = v0 + u * MERGE_THREADS;
              if (v < nvec) x[t][u] = __ldg(msrc + v);
            }
          }
        }
#pragma unroll
        for (int t = 0; t < BATCH; ++t) {
          if (m0 + t < cnt) {
            const float w = wt[t];
            den += w;
#pragma unroll
            for (int u = 0; u < NV; ++u) {
              float f[8];
              unpack8(x[t][u], f);
#pragma unroll
              for (int e = 0; e < 8; ++e) acc[u][e] += w * f[e];
            }
          }
        }
      }
    };
    if (BITS) {
      const int list0 = (threadIdx.x >> 5) * MERGE_WARP_LIST;
      // (a pass over more members than the list holds reads the words again: kept, they cost the pass its registers)
      for (int w0 = 0, c0 = 0; w0 < a.bit_words;) {
        if (w0 | c0) load_words(w0);
        int mine = 0;
#pragma unroll
        for (int g = 0; g < MERGE_BIT_WORDS; ++g) mine += __popc(mw[g]);
        int at = mine;                          // inclusive, then exclusive sum over the lanes
        if (__any_sync(0xffffffffu, mine)) {
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += t;
          }
        }
        const int left = __shfl_sync(0xffffffffu, at, 31) - c0;      // members of these words not yet added
        if (left > 0) {
          merged = true;
          int r = at - mine - c0;
#pragma unroll
          for (int g = 0; g < MERGE_BIT_WORDS; ++g)
            for (uint32_t m = mw[g]; m; m &= m - 1, ++r)
              if (r >= 0 && r < MERGE_WARP_LIST) s_j[list0 + r] = (w0 + lane * per + g) * 32 + __ffs(m) - 1;
          __syncwarp();
          add_members(list0, min(MERGE_WARP_LIST, left));
          __syncwarp();                         // the list has been read
        }
        if (left > MERGE_WARP_LIST) c0 += MERGE_WARP_LIST;
        else { c0 = 0; w0 += 32 * MERGE_BIT_WORDS; }
      }
    } else {
      for (int base = m_lo; base < m_hi; base += MERGE_LIST) {
        const int cnt = min(MERGE_LIST, m_hi - base);
        __syncthreads();                      // the previous list has been consumed
        if ((int)threadIdx.x < cnt) {
          if (a.member_meta) {
            const int2 mm = ld_prev(a.member_meta + (size_t)b * nd_max + base + threadIdx.x);
            s_j[threadIdx.x] = min(max(mm.x, 0), d.nv - 1);
            s_w[threadIdx.x] = __int_as_float(mm.y);
          } else {
            const int j = min(max(drop_b[min(max(mem_b[base + threadIdx.x], 0), nd_max - 1)], 0), d.nv - 1);
            s_j[threadIdx.x] = j;
            s_w[threadIdx.x] = sal_b[j];
          }
        }
        __syncthreads();
        add_members(0, cnt);
      }
    }
    if (den <= a.eps || !merged) {
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = v0 + u * MERGE_THREADS;
        if (v < nvec) dst[v] = self[u];
      }
    } else {
      const float inv = 1.0f / den;
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = v0 + u * MERGE_THREADS;
        if (v < nvec) {
          uint4 o;
          o.x = pack2_rn(acc[u][0] * inv, acc[u][1] * inv);
          o.y = pack2_rn(acc[u][2] * inv, acc[u][3] * inv);
          o.z = pack2_rn(acc[u][4] * inv, acc[u][5] * inv);
          o.w = pack2_rn(acc[u][6] * inv, acc[u][7] * inv);
          dst[v] = o;
        }
      }
    }
  };
  if (rows == 1) {
    kept_row(slot, kept, m_lo, m_hi);
    return;
  }
  // Eight slots: those without members are copied by the warp that looked them up (4 KB on their way per warp, where the
  // block together has one row), the others by the block, one after the other (24 x 576 slots, 512 of them copies: 88.6 -> 85.6 us).
  __shared__ int s_slot[3][MERGE_THREADS / 32];
  if (lane == 0) { s_slot[0][warp] = kept; s_slot[1][warp] = m_lo; s_slot[2][warp] = m_hi; }
  if (slot < k && m_hi <= m_lo) copy_row((size_t)(d.row0 + d.v0 + min(max(kept, 0), d.nv - 1)), d.out_row0 + d.v0 + slot);
  __syncthreads();
  for (int s = 0; s < rows && (int)blockIdx.x * rows + s < k; ++s)
    if (s_slot[2][s] > s_slot[1][s]) kept_row((int)blockIdx.x * rows + s, s_slot[0][s], s_slot[1][s], s_slot[2][s]);
}

// =======================================================================================
// gather_rows: KV-cache compaction.  Output row r of every tensor is input row src_row[r] (the
// row map the prune step wrote); one warp per (row, tensor), 16-byte vectors, eight in flight.
// Rows at or past *n_rows (a device-side count, e.g. out_cu_seqlens[B]) are left untouched.
// =======================================================================================
constexpr int KV_MAX_TENSORS = 64;
constexpr int KV_THREADS = 256;

struct GatherArgs {
  const void *src[KV_MAX_TENSORS];
  void *dst[KV_MAX_TENSORS];
  const int32_t *src_row;
  const int32_t *n_rows;      // device scalar
  int32_t rows_capacity, src_rows, row_vecs;   // row_vecs = row bytes / 16
};

__global__ void __launch_bounds__(KV_THREADS)
gather_rows_kernel(GatherArgs a) {
  pdl_enter();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * (KV_THREADS / 32) + warp;
  if (r >= a.rows_capacity || r >= *a.n_rows) return;
  const int sr = a.src_row[r];
  if (sr < 0 || sr >= a.src_rows) return;                 // not a valid source row: leave the output row alone
  const uint4 *src = reinterpret_cast<const uint4 *>(a.src[blockIdx.y]) + (size_t)sr * a.row_vecs;
  uint4 *dst = reinterpret_cast<uint4 *>(a.dst[blockIdx.y]) + (size_t)r * a.row_vecs;
  for (int v = lane; v < a.row_vecs; v += 32 * 8) {
    uint4 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v + 32 * u < a.row_vecs) x[u] = __ldg(src + v + 32 * u);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (v + 32 * u < a.row_vecs) dst[v + 32 * u] = x[u];
  }
}

}  // namespace asap
