// Hybrid-mask paged-KV attention (Eq. 1 over a shared prefix), split over KV ranges, plus the combine.
//
// A work item is (request, kv head, row tile of <=128 query rows = tokens x GQA group, KV block range).
// One producer warp streams the item's 64-token KV blocks page by page with 1-D bulk copies into a
// shared-memory ring (the pool tiles are stored pre-swizzled, so a linear copy lands fragment-ready);
// eight consumer warps hold 16 query rows each and, when the tile has fewer than 128 rows, share the
// rows and split the KV blocks among themselves instead.  Only blocks that reach past the committed
// context apply the visibility test; the prefix loop is mask-free.
#include <cstdlib>
#include "common.cuh"
#include "kernels.h"

namespace recg {

namespace {

constexpr int kStages = 4;
constexpr int kConsumerWarps = 8;
constexpr int kAttnThreads = (kConsumerWarps + 1) * 32;
constexpr int kBlockTokens = 64;
constexpr int kPagesPerBlock = kBlockTokens / kPageSize;
constexpr uint32_t kSpinLimit = 1u << 22;

template <int D>
struct AttnSmem {
  static constexpr int kPageBytes = 2 * kPageSize * D * 2;          // K tile + V tile
  static constexpr int kStageBytes = kPagesPerBlock * kPageBytes;
  static constexpr int kRingBytes = kStages * kStageBytes;
  static constexpr int kMergeFloats = (D / 8 * 4 + 4) * 32;         // per warp: o frags + m[2] + l[2]
  static constexpr int kMergeBytes = kConsumerWarps * kMergeFloats * 4;
  static constexpr int kBarOffset = kRingBytes + kMergeBytes;
  static constexpr int kTotal = kBarOffset + 2 * kStages * 8 + 16;
};

struct AttnParams {
  const AttnItem* items;
  const int* cta_off;
  const int* page_table;
  int pt_stride;
  const int* tok_climit;
  const int* tok_lo;
  const int* tok_hi;
  const __nv_bfloat16* q;
  __nv_bfloat16* o;
  const __nv_bfloat16* pool;
  int64_t n_pages;
  int layer, n_q, n_kv, group;
  float scale_log2;   // log2(e) / sqrt(d)
  float* part_o;      // [part][128][D]
  float* part_ml;     // [part][128][2]
  int* status;
};

__device__ __forceinline__ void consumer_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

template <int D>
__global__ void __launch_bounds__(kAttnThreads, 1) attention_kernel(AttnParams P) {
  using SM = AttnSmem<D>;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + SM::kBarOffset);
  uint64_t* empty_bar = full_bar + kStages;
  float* merge = reinterpret_cast<float*>(smem + SM::kRingBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_launch();

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], kConsumerWarps);
    }
    fence_barrier_init();
  }
  __syncthreads();
  griddep_wait();

  // the CTA walks two ranges of the item list one after the other (see the layout kernel)
  const int4 r4 = *reinterpret_cast<const int4*>(P.cta_off + 4 * blockIdx.x);
  const int range_n0 = r4.y - r4.x;
  const int item_begin = 0, item_end = range_n0 + (r4.w - r4.z);
  auto item_at = [&](int i) { return i < range_n0 ? r4.x + i : r4.z + (i - range_n0); };
  uint32_t it = 0;  // running block counter, identical in producer and consumers
  bool aborted = false;

  if (warp == kConsumerWarps) {
    // ------------------------------ producer ------------------------------
    for (int item = item_begin; item < item_end && !aborted; ++item) {
      const AttnItem w = P.items[item_at(item)];
      const int n_req_pages = (w.kv_len + kPageSize - 1) / kPageSize;
      const int* pt = P.page_table + (size_t)w.req * P.pt_stride;
      // lanes 0..3 each own one page of the block; ids are fetched one block ahead of their use
      auto fetch_page = [&](int n) -> int {
        int pg = -1;
        if (lane < kPagesPerBlock && n < w.blk_end) {
          const int lp = n * kPagesPerBlock + lane;
          if (lp < n_req_pages) pg = __ldg(pt + lp);   // validated when used
        }
        return pg;
      };
      int pg_next = fetch_page(w.blk_begin);
      for (int n = w.blk_begin; n < w.blk_end; ++n, ++it) {
        const int s = it % kStages;
        int my_pg = pg_next;
        pg_next = fetch_page(n + 1);                   // in flight during this iteration
        if (my_pg >= P.n_pages) {
          set_status(P.status, DEV_BAD_INDEX);
          my_pg = -1;
        }
        if (!mbar_wait(&empty_bar[s], ((it / kStages) & 1) ^ 1, kSpinLimit)) {
          set_status(P.status, DEV_TIMEOUT_EMPTY);
          aborted = true;
          break;
        }
        const unsigned valid = __ballot_sync(0xffffffffu, my_pg >= 0);
        if (lane == 0) {
          if (valid == 0) mbar_arrive(&full_bar[s]);
          else mbar_arrive_expect_tx(&full_bar[s], __popc(valid) * SM::kPageBytes);
        }
        __syncwarp();
        if (my_pg >= 0) {
          const __nv_bfloat16* src = P.pool + kv_tile_base(P.n_pages, P.n_kv, D, P.layer, my_pg, w.kv_head);
          bulk_g2s(smem + s * SM::kStageBytes + lane * SM::kPageBytes, src, SM::kPageBytes, &full_bar[s]);
        }
        __syncwarp();
      }
    }
    if (aborted && lane == 0) {
      // let copies already in flight land before the CTA may exit
      for (int s = 0; s < kStages; ++s) {
        for (uint32_t i = 0; i < (1u << 16); ++i) {
          if (mbar_try_wait(&full_bar[s], 0) || mbar_try_wait(&full_bar[s], 1)) break;
          __nanosleep(64);
        }
      }
    }
    return;
  }

  // ------------------------------ consumers ------------------------------
  const int g = lane >> 2, q4 = lane & 3;
  const uint32_t ring = smem_u32(smem);

  for (int item = item_begin; item < item_end; ++item) {
    const AttnItem w = P.items[item_at(item)];
    const int R = w.ntok * P.group;
    const int RW = (R + 15) >> 4;
    const int KW = RW == 1 ? 8 : (RW == 2 ? 4 : (RW <= 4 ? 2 : 1));
    const int rw = warp % RW, kw = warp / RW;
    const bool active = kw < KW;

    // Q fragments and per-row visibility for this thread's two rows (g and g + 8 of the warp's 16)
    uint32_t qf[D / 16][4];
    int climit[2], vlo[2], vhi[2];
    int qrow_tok[2], qrow_head[2];
    bool rvalid[2];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int rho = rw * 16 + g + hh * 8;
      rvalid[hh] = active && rho < R;
      const int j = rho / P.group, hg = rho % P.group;
      const int t = w.tok0 + (rvalid[hh] ? j : 0);
      qrow_tok[hh] = t;
      qrow_head[hh] = w.kv_head * P.group + hg;
      climit[hh] = rvalid[hh] ? P.tok_climit[t] : -1;
      vlo[hh] = rvalid[hh] ? P.tok_lo[t] : 0;
      vhi[hh] = rvalid[hh] ? P.tok_hi[t] : 0;
    }
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(
            P.q + ((size_t)qrow_tok[hh] * P.n_q + qrow_head[hh]) * D + k * 16 + q4 * 2);
        qf[k][hh] = rvalid[hh] ? __ldg(src) : 0u;
        qf[k][hh + 2] = rvalid[hh] ? __ldg(src + 4) : 0u;
      }
    }

    float o[D / 8][4];
#pragma unroll
    for (int i = 0; i < D / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    float m_run[2] = {-1e30f, -1e30f};
    float l_run[2] = {0.f, 0.f};
    const int ctx_first_new = w.kv_len;  // positions >= kv_len never exist

    for (int n = w.blk_begin; n < w.blk_end; ++n, ++it) {
      const int s = it % kStages;
      if (!aborted && !mbar_wait(&full_bar[s], (it / kStages) & 1, kSpinLimit)) {
        set_status(P.status, DEV_TIMEOUT_FULL);
        aborted = true;
      }
      if (!aborted && active && ((n - w.blk_begin) % KW) == kw) {
        const uint32_t stage = ring + s * SM::kStageBytes;
        // ---- S = Q K^T over the 64 tokens of the block ----
        float sc[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
        for (int j = 0; j < D / 32; ++j) {
#pragma unroll
          for (int nt = 0; nt < 8; ++nt) {
            const int token = nt * 8 + (lane & 7);
            const int pg = token >> 4, tok = token & 15;
            const int c = 4 * j + (lane >> 3);
            const uint32_t addr = stage + pg * SM::kPageBytes + ((tok >> 3) * (D / 64) + (c >> 3)) * 1024 +
                                  (tok & 7) * 128 + (((c & 7) ^ (tok & 7)) << 4);
            uint32_t b0, b1, b2, b3;
            ldmatrix_x4(b0, b1, b2, b3, addr);
            mma_bf16_16816(sc[nt], qf[2 * j], b0, b1);
            mma_bf16_16816(sc[nt], qf[2 * j + 1], b2, b3);
          }
        }
        // ---- visibility (only blocks that reach past the mask-free prefix) ----
        const int pos0 = n * kBlockTokens;
        const int min_limit = min(climit[0], climit[1]);
        // every row of the tile sees all positions <= its climit; the block is mask-free when it ends
        // at or before the smallest climit of the warp's rows (invalid rows carry -1 and force the test)
        const bool need_mask = __any_sync(0xffffffffu, pos0 + kBlockTokens - 1 > min_limit);
        if (need_mask) {
#pragma unroll
          for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int hh = e >> 1;
              const int pos = pos0 + nt * 8 + q4 * 2 + (e & 1);
              const bool vis = pos <= climit[hh] || (pos >= vlo[hh] && pos < vhi[hh]);
              if (!vis) sc[nt][e] = -INFINITY;
            }
          }
        }
        // ---- online softmax in the log2 domain ----
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          float mx = -INFINITY;
#pragma unroll
          for (int nt = 0; nt < 8; ++nt) mx = fmaxf(mx, fmaxf(sc[nt][2 * hh], sc[nt][2 * hh + 1]));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
          const float m_new = fmaxf(m_run[hh], mx * P.scale_log2);
          const float alpha = exp2f(m_run[hh] - m_new);
          m_run[hh] = m_new;
          float ls = 0.f;
#pragma unroll
          for (int nt = 0; nt < 8; ++nt) {
            const float p0 = exp2f(sc[nt][2 * hh] * P.scale_log2 - m_new);
            const float p1 = exp2f(sc[nt][2 * hh + 1] * P.scale_log2 - m_new);
            sc[nt][2 * hh] = p0;
            sc[nt][2 * hh + 1] = p1;
            ls += p0 + p1;
          }
          l_run[hh] = l_run[hh] * alpha + ls;
#pragma unroll
          for (int i = 0; i < D / 8; ++i) {
            o[i][2 * hh] *= alpha;
            o[i][2 * hh + 1] *= alpha;
          }
        }
        // ---- O += P V ----
        const bool sanitize = pos0 + kBlockTokens > ctx_first_new;  // stale or unwritten V rows in the block
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          uint32_t a[4];
          a[0] = pack_bf16(sc[2 * kk][0], sc[2 * kk][1]);
          a[1] = pack_bf16(sc[2 * kk][2], sc[2 * kk][3]);
          a[2] = pack_bf16(sc[2 * kk + 1][0], sc[2 * kk + 1][1]);
          a[3] = pack_bf16(sc[2 * kk + 1][2], sc[2 * kk + 1][3]);
          uint32_t keep0 = 0xffffffffu, keep1 = 0xffffffffu;
          if (sanitize) {
            const int tb = pos0 + kk * 16 + q4 * 2;
            keep0 = (tb < ctx_first_new ? 0x0000ffffu : 0u) | (tb + 1 < ctx_first_new ? 0xffff0000u : 0u);
            keep1 = (tb + 8 < ctx_first_new ? 0x0000ffffu : 0u) | (tb + 9 < ctx_first_new ? 0xffff0000u : 0u);
          }
          const int mi = lane >> 3, r8 = lane & 7;
          const int tok = (mi & 1) * 8 + r8;
#pragma unroll
          for (int jj = 0; jj < D / 16; ++jj) {
            const int c = 2 * jj + (mi >> 1);
            const uint32_t addr = stage + kk * SM::kPageBytes + kPageSize * D * 2 +
                                  ((tok >> 3) * (D / 64) + (c >> 3)) * 1024 + (tok & 7) * 128 +
                                  (((c & 7) ^ (tok & 7)) << 4);
            uint32_t b0, b1, b2, b3;
            ldmatrix_x4_trans(b0, b1, b2, b3, addr);
            if (sanitize) {
              b0 &= keep0; b1 &= keep1; b2 &= keep0; b3 &= keep1;
            }
            mma_bf16_16816(o[2 * jj], a, b0, b1);
            mma_bf16_16816(o[2 * jj + 1], a, b2, b3);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_bar[s]);
    }

    // quad-reduce the row sums
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 1);
      l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 2);
    }

    // ---- merge the KV-split warps of the CTA ----
    if (KW > 1) {
      float* mine = merge + warp * SM::kMergeFloats;
      if (active && kw > 0) {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) mine[(i * 4 + e) * 32 + lane] = o[i][e];
        mine[(D / 2 + 0) * 32 + lane] = m_run[0];
        mine[(D / 2 + 1) * 32 + lane] = m_run[1];
        mine[(D / 2 + 2) * 32 + lane] = l_run[0];
        mine[(D / 2 + 3) * 32 + lane] = l_run[1];
      }
      consumer_bar();
      if (active && kw == 0) {
        for (int k2 = 1; k2 < KW; ++k2) {
          const float* oth = merge + (k2 * RW + rw) * SM::kMergeFloats;
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            const float mo = oth[(D / 2 + hh) * 32 + lane];
            const float lo_ = oth[(D / 2 + 2 + hh) * 32 + lane];
            const float m_new = fmaxf(m_run[hh], mo);
            const float fa = exp2f(m_run[hh] - m_new), fb = exp2f(mo - m_new);
            m_run[hh] = m_new;
            l_run[hh] = l_run[hh] * fa + lo_ * fb;
#pragma unroll
            for (int i = 0; i < D / 8; ++i) {
              o[i][2 * hh] = o[i][2 * hh] * fa + oth[(i * 4 + 2 * hh) * 32 + lane] * fb;
              o[i][2 * hh + 1] = o[i][2 * hh + 1] * fa + oth[(i * 4 + 2 * hh + 1) * 32 + lane] * fb;
            }
          }
        }
      }
      consumer_bar();  // scratch may be rewritten by the next item only after everyone has read it
    }

    // ---- write out ----
    if (active && kw == 0 && !aborted) {
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        if (!rvalid[hh]) continue;
        const int rho = rw * 16 + g + hh * 8;
        if (w.part < 0) {
          const float inv = l_run[hh] > 0.f ? 1.f / l_run[hh] : 0.f;
          uint32_t* dst = reinterpret_cast<uint32_t*>(P.o + ((size_t)qrow_tok[hh] * P.n_q + qrow_head[hh]) * D);
#pragma unroll
          for (int i = 0; i < D / 8; ++i)
            dst[i * 4 + q4] = pack_bf16(o[i][2 * hh] * inv, o[i][2 * hh + 1] * inv);
        } else {
          float2* dst = reinterpret_cast<float2*>(P.part_o + ((size_t)w.part * 128 + rho) * D);
#pragma unroll
          for (int i = 0; i < D / 8; ++i) dst[i * 4 + q4] = make_float2(o[i][2 * hh], o[i][2 * hh + 1]);
          if (q4 == 0) {
            P.part_ml[((size_t)w.part * 128 + rho) * 2 + 0] = m_run[hh];
            P.part_ml[((size_t)w.part * 128 + rho) * 2 + 1] = l_run[hh];
          }
        }
      }
    }
  }
}

// How many warps merge a row and how many of its partial rows are on their way at once (see combine_split and few_tiles):
// kManyTiles one warp, six rows; kSplitRows two or four warps, which merge their sums through shared memory; kDeepRows one warp,
// 18 rows, for which a CTA has the registers of an SM to itself (117 of 128 a thread at head_dim 128).
enum CombineMode { kManyTiles, kSplitRows, kDeepRows };
// Merges the KV-range partials of the tiles that were split (`tiles` lists no others: tiles with a single part were written by
// the attention kernel itself).  Work unit = 16 rows of a tile (8 or 4 where rows are split), each lane D/32
// consecutive dims.  Bound by latency, not by its bytes (a tile entry, the (max, sum) pairs and the partial rows are
// dependent reads): the tile entry is read ahead of the wait where the work list is settled, lane p fetches the pair of part
// p, so that one read and a few shuffles give all weights of up to 32 parts, and the rows of the first kRows parts are on
// their way at the same time.  Attention and combine kernel of a layer together, one request of 18 parts per row: 19.5 us with
// four parts fetched at a time, each with its own pair, 16.1 with six and one read for all pairs; 13.9 now, with four warps a row.
template <int D, CombineMode MODE>
__global__ void __launch_bounds__(512, MODE == kDeepRows ? 1 : 2) attention_combine_kernel(const AttnTile* __restrict__ tiles,
                                                                const int* __restrict__ counts, int n_q, int group,
                                                                const float* __restrict__ part_o,
                                                                const float* __restrict__ part_ml,
                                                                __nv_bfloat16* __restrict__ o, int list_settled, int log_split) {
  constexpr int E = D / 32;
  constexpr bool SPLIT = MODE == kSplitRows;
  constexpr int kRows = MODE == kDeepRows ? 18 : 6;     // partial rows in flight
  __shared__ float s_acc[SPLIT ? 16 : 1][D + 2];
  griddep_launch();
  if (!list_settled) griddep_wait();
  const int n_tiles = counts[1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int log_s = SPLIT ? log_split : 0, S = 1 << log_s;
  const int n_units = n_tiles << (3 + log_s), my = warp & (S - 1);
  AttnTile tl = {};
  if ((int)blockIdx.x < n_units) tl = tiles[blockIdx.x >> (3 + log_s)];
  if (list_settled) griddep_wait();
  for (int wu = blockIdx.x; wu < n_units; wu += gridDim.x) {
    if (wu != (int)blockIdx.x) tl = tiles[wu >> (3 + log_s)];
    const int rho = (((wu & ((8 << log_s) - 1)) << 4) + warp) >> log_s;
    const bool live = rho < tl.ntok * group;
    const int n_mine = live ? (tl.n_parts - my + S - 1) >> log_s : 0;       // parts my, my + S, ...
    const size_t first = tl.part_begin + my;
    const float* rows = part_o + (first * 128 + rho) * D + lane * E;
    auto fetch = [&](int p, float (&v)[E]) {
      if constexpr (E == 4) {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(rows + (size_t)(p << log_s) * 128 * D));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
      } else {
        const float2 t = __ldcg(reinterpret_cast<const float2*>(rows + (size_t)(p << log_s) * 128 * D));
        v[0] = t.x; v[1] = t.y;
      }
    };
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    float m = -1e30f, l = 0.f;
    for (int p0 = 0; p0 < n_mine; p0 += 32) {
      const int np = min(32, n_mine - p0);
      float2 ml = make_float2(-1e30f, 0.f);
      if (lane < np) ml = __ldcg(reinterpret_cast<const float2*>(part_ml) + (first + ((p0 + lane) << log_s)) * 128 + rho);
      float v[kRows][E];
#pragma unroll
      for (int k = 0; k < kRows; ++k)
        if (k < np) fetch(p0 + k, v[k]);
      float m_new = ml.x;
#pragma unroll
      for (int s = 16; s; s >>= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xffffffffu, m_new, s));
      m_new = fmaxf(m_new, m);
      const float f = exp2f(m - m_new), wgt = exp2f(ml.x - m_new);   // (a lane without a part: sum 0)
      m = m_new;
      float ls = wgt * ml.y;
#pragma unroll
      for (int s = 16; s; s >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, s);
      l = l * f + ls;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] *= f;
      for (int k0 = 0; k0 < np; k0 += kRows) {
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
          if (k0 + k >= np) continue;
          const float wk = __shfl_sync(0xffffffffu, wgt, k0 + k);
#pragma unroll
          for (int e = 0; e < E; ++e) acc[e] += wk * v[k][e];
          if (k0 + kRows + k < np) fetch(p0 + k0 + kRows + k, v[k]);      // the slot's next row follows at once
        }
      }
    }
    if constexpr (SPLIT) {
      if (my) {
#pragma unroll
        for (int e = 0; e < E; ++e) s_acc[warp][lane * E + e] = acc[e];
        if (lane == 0) {
          s_acc[warp][D] = m;
          s_acc[warp][D + 1] = l;
        }
      }
      __syncthreads();
      for (int k = 1; my == 0 && k < S; ++k) {
        const float* other = s_acc[warp + k];
        const float m_k = other[D], m_new = fmaxf(m, m_k), f = exp2f(m - m_new), g = exp2f(m_k - m_new);
        m = m_new;
        l = l * f + other[D + 1] * g;
#pragma unroll
        for (int e = 0; e < E; ++e) acc[e] = acc[e] * f + other[lane * E + e] * g;
      }
      __syncthreads();
    }
    if (live && my == 0) {
      const float inv = l > 0.f ? 1.f / l : 0.f;
      const int j = rho / group, hg = rho % group;
      __nv_bfloat16* dst = o + ((size_t)(tl.tok0 + j) * n_q + tl.kv_head * group + hg) * D + lane * E;
      if constexpr (E == 4) {
        uint2 pk;
        pk.x = pack_bf16(acc[0] * inv, acc[1] * inv);
        pk.y = pack_bf16(acc[2] * inv, acc[3] * inv);
        *reinterpret_cast<uint2*>(dst) = pk;
      } else {
        *reinterpret_cast<uint32_t*>(dst) = pack_bf16(acc[0] * inv, acc[1] * inv);
      }
    }
  }
}

// Few row tiles (at most `tiles`, 0: not known) are merged by few warps, each with many parts: a chain of dependent reads while most
// SMs are idle.
// By itself (recg_attention) two or four warps share a row: one request over 4096 tokens (8 tiles of 18 parts), 32 layers, 479 us
// with one warp per row, 446 with four.  The line lies where that many warps per row are resident at once, two CTAs per SM.
// Inside a step the idle SMs are worth more to the next projection, whose CTAs come in early and request weights (a round of that
// request 3548 us with one warp per row, 3600 with four): there a row keeps its warp, in as many CTAs as there is work, and up to
// 18 of its parts are on their way at once (six at once: 3553).  18 are the parts of a row where one request's 8 tiles share all
// CTAs; fewer tiles have more parts and take more turns.  Rounds with kManyTiles and with kDeepRows, us (runs differ by up to 0.4 %):
//   8 tiles: contexts of 900, 4096 and 8192 tokens 3415 -> 3382, 3555 -> 3515, 3686 -> 3641; 14B class, 3000 tokens, 5533 -> 5424
//   16 tiles: two requests of 4096 tokens 3888 -> 3882, one of 64 rows 3826 -> 3820; two of 1000 3697 -> 3698 (4.7 %), two of 200
//     to 8000 3756 -> 3655 (6 %), two of the 14B class 5781 -> 5609 (3.4 %)
//   2 layers of hidden size 512, 4000 tokens: 2, 10 and 18 tiles 124 -> 116, 130 -> 125 (6 %), 148 -> 134 (24 %)
// The line lies where all CTAs of kDeepRows are resident at once, one per SM (18 tiles: 144); nothing below it is slower.
int combine_split(int tiles, int n_sm, bool step) {
  return tiles <= 0 || step ? 0 : (tiles * 32 <= 2 * n_sm ? 2 : (tiles * 16 <= 2 * n_sm ? 1 : 0));
}
bool few_tiles(int tiles, int n_sm) { return tiles > 0 && tiles * 16 <= 2 * n_sm; }
unsigned combine_ctas(int tiles, int log_s, int n_sm) { return few_tiles(tiles, n_sm) ? (unsigned)tiles << (3 + log_s) : 4u * n_sm; }
template <int D>
auto combine_kernel(int tiles, int log_s, int n_sm) {
  return log_s ? attention_combine_kernel<D, kSplitRows>
               : (few_tiles(tiles, n_sm) ? attention_combine_kernel<D, kDeepRows> : attention_combine_kernel<D, kManyTiles>);
}

template <int D>
void launch_attention_t(const BatchLayout& bl, const Dims& dm, int layer, const void* q, void* o, const void* kv_pool,
                        int64_t n_pages, float* part_o, float* part_ml, int tok_per_tile, int n_sm, int* status,
                        cudaStream_t st, bool whole, int tiles, bool step) {
  static bool configured[kMaxDevices] = {false};
  if (first_use_on_device(configured))
    cudaFuncSetAttribute(attention_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem<D>::kTotal);

  AttnParams P;
  P.items = bl.items;
  P.cta_off = bl.cta_off;
  P.page_table = bl.page_table;
  P.pt_stride = bl.pt_stride;
  P.tok_climit = bl.tok_climit;
  P.tok_lo = bl.tok_lo;
  P.tok_hi = bl.tok_hi;
  P.q = static_cast<const __nv_bfloat16*>(q);
  P.o = static_cast<__nv_bfloat16*>(o);
  P.pool = static_cast<const __nv_bfloat16*>(kv_pool);
  P.n_pages = n_pages;
  P.layer = layer;
  P.n_q = dm.n_q;
  P.n_kv = dm.n_kv;
  P.group = dm.n_q / dm.n_kv;
  P.scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  P.part_o = part_o;
  P.part_ml = part_ml;
  P.status = status;
  launch_pdl(attention_kernel<D>, dim3(n_sm), dim3(kAttnThreads), AttnSmem<D>::kTotal, st, P);
  if (whole) return;
  const int log_s = combine_split(tiles, n_sm, step);
  launch_pdl(combine_kernel<D>(tiles, log_s, n_sm), dim3(combine_ctas(tiles, log_s, n_sm)), dim3(512), 0, st,
             (const AttnTile*)bl.tiles, (const int*)bl.counts, dm.n_q, P.group, (const float*)part_o, (const float*)part_ml,
             static_cast<__nv_bfloat16*>(o), 0, log_s);
}

}  // namespace

size_t attention_smem_bytes(int head_dim) {
  return head_dim == 64 ? AttnSmem<64>::kTotal : AttnSmem<128>::kTotal;
}

void launch_attention(const BatchLayout& bl, const Dims& dm, int layer, const void* q, void* o, const void* kv_pool,
                      int64_t n_pages, float* part_o, float* part_ml, int tok_per_tile, int n_sm, int* status,
                      cudaStream_t st, bool use_tc, bool layout_settled, bool whole, int tiles, bool step) {
  if (use_tc && dm.head_dim == 128) {
    launch_attention_tc_main(bl, dm, layer, q, o, kv_pool, n_pages, part_o, part_ml, n_sm, status, st, layout_settled);
    if (whole) return;
    const int log_s = combine_split(tiles, n_sm, step);
    launch_pdl(combine_kernel<128>(tiles, log_s, n_sm), dim3(combine_ctas(tiles, log_s, n_sm)), dim3(512), 0, st,
               (const AttnTile*)bl.tiles, (const int*)bl.counts, dm.n_q, dm.n_q / dm.n_kv, (const float*)part_o, (const float*)part_ml,
               static_cast<__nv_bfloat16*>(o), 1, log_s);    // (the kernel in front signals its dependents when the list is settled)
    return;
  }
  if (dm.head_dim == 64)
    launch_attention_t<64>(bl, dm, layer, q, o, kv_pool, n_pages, part_o, part_ml, tok_per_tile, n_sm, status, st, whole, tiles, step);
  else
    launch_attention_t<128>(bl, dm, layer, q, o, kv_pool, n_pages, part_o, part_ml, tok_per_tile, n_sm, status, st, whole, tiles, step);
}

}  // namespace recg
