// Projection GEMM on the 5th-generation tensor cores: y = x . w^T, bf16 in, fp32 accumulate in TMEM.
//
// The WEIGHTS are the M operand (128 output features per CTA) and the tokens the N operand of the tensor core: the N extent
// of an instruction is any multiple of 16 up to 256, so a batch of T rows is cut into ceil(T / 256) or a few more equal token
// tiles and next to nothing is computed for padding (with the tokens on the M side 376 rows cost as much as 512), and an
// accumulator tile is spread over all four epilogue warps however few tokens there are (TMEM lane = output feature).
//
// Persistent, warp-specialised CTA of 6 warps:
//   warp 0   producer: TMA loads (128-byte swizzle) of the w tile [128 x 64] and the x tile [tokens x 64] into a
//            shared-memory ring, completion on mbarriers;
//   warp 1   one elected lane issues tcgen05.mma (M = 128, N = tokens, K = 16) from shared-memory descriptors
//            into one of two TMEM accumulators and commits to the ring's empty barriers;
//   warps 2-5  epilogue: tcgen05.ld of the finished accumulator (each warp its 32 lanes = features, 32 tokens at a time),
//            then the fused epilogue straight from registers (residual add with the next norm's input, SwiGLU, rotary +
//            paged KV append, or plain store) while the MMA warp already fills the other accumulator.  One warp per
//            scheduler runs it, so what counts is its instructions: the 16x256b form of tcgen05.ld hands out 8 x 8 fragments,
//            stmatrix.trans turns them into rows of tokens, and stores are whole 32-byte sectors.  32 tokens take .6 us to
//            1 us, and 3.5 us more when the code is not in the SM's instruction cache, which is so for the projections
//            behind an attention kernel: all ways of finishing a tile share one instance of it, and the warps run it once
//            without effect while they wait for the kernels in front of this one.
// Operands of an epilogue that belong together sit in the same thread: the tensor map over w lists its rows 16 by 16 in the
// order the tile wants them (16 gate rows, their 16 up rows, ...; 16 low dims of a head, their 16 rotation partners, ...), and
// a thread holds the same row of both halves of a 32-row quadrant.
// Tiles are walked token-fastest so that CTAs running together share the same weight tile through L2.
// Tiles can be cut over K: stream-K (partial tiles are parked in a workspace and reduced by the last part to arrive), or the
// parts of a tile form a thread-block cluster and reduce it through distributed shared memory, each member finishing its share
// of the tokens.
// Every wait is bounded; on a timeout the kernel records a status code, drains and frees TMEM.
//
// What bounds it (B200): a k-block (64 of K) costs max(operand bytes / 115 GB/s per SM (64 bytes per clock from L2), token
// columns x 1.5 ns (the tensor pipe at the clock that the power cap leaves), weight bytes / its share of HBM).  Figures at
// the choice of the configuration (choose_config below).
#include <cuda.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cmath>
#include <functional>
#include <mutex>
#include <unordered_map>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace recg {

namespace {

constexpr int FT = 128, BK = 64;            // output features per CTA, k-block
constexpr int kTcThreads = 192;
constexpr int kMaxTok = 256;                // widest token tile
constexpr int kRingBytes = 210 * 1024;      // operand ring
constexpr int kMaxStages = 16;
constexpr int kABytes = FT * BK * 2;
constexpr int kChunkBytes = 32 * FT * 4;    // 32 tokens of a partial tile
constexpr int kAccStride = kMaxTok;         // TMEM columns between the two accumulators
constexpr int kTmemCols = 2 * kMaxTok;
constexpr int kOffBar = kRingBytes;
constexpr int kBarBytes = (2 * kMaxStages + 2 + 2 + 1 + 1) * 8 + 16;
constexpr int kOffRstd = kOffBar + ((kBarBytes + 15) & ~15);      // float [256] row factors of the token tile
constexpr int kOffSlot = kOffRstd + kMaxTok * 4;                   // int [256] cache slots of the token tile
constexpr int kOffSs = kOffSlot + kMaxTok * 4;                     // float [4][256] sums of squares per epilogue warp
constexpr int kOffStage = kOffSs + 4 * kMaxTok * 4;                // per epilogue warp: 32 tokens x 32 bf16 on their way out
constexpr int kSmemBytes = kOffStage + 4 * 2048 + 1024;            // + slack for 1024-byte alignment
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
constexpr uint32_t kSpin = 1u << 22;

using namespace tc;   // the tcgen05 / TMA wrappers (tc_ptx.cuh)

// ---- CTA pairs (tcgen05 cta_group::2) ----------------------------------------------------------------
// With PAIR two CTAs of a cluster compute tiles of 256 features: each CTA loads its own 128 rows of w and its own half of the
// token tile per k-block (28 KB for 192 tokens instead of the 40 KB of a single CTA, so more stages fit and fewer operand
// bytes cross L2 -> shared memory per flop); the tensor cores of the pair read both halves of the token tile, each CTA
// accumulates its 128 features in its own TMEM.  Only the pair's leader (even cluster rank) issues MMAs.
//   full barrier  (leader's):   the leader's producer arrives with the byte count of BOTH CTAs' loads; both CTAs'
//                               TMA loads (cta_group::2 form, no multicast) complete on it
//   empty barrier (per CTA):    tcgen05.commit multicast to both CTAs frees the stage in each
//   accumulator full (per CTA): commit multicast; accumulator empty (leader's): all eight epilogue warps of the
//                               pair arrive (the other CTA's remotely)
// The scheduling unit becomes the pair; its two CTAs park, hand over and reduce their halves of a cut tile independently.
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the shared::cluster address of the same location in the CTA of rank `rank`
__device__ __forceinline__ uint32_t mapa_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t smem_dst, const CUtensorMap* map, int x, int y, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
               :
               : "r"(smem_dst), "l"(map), "r"(bar_cluster), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void tma_load_w_pair(uint32_t smem_dst, const CUtensorMap* map, int k, int c3, int c4, uint32_t bar_cluster) {
  const int z = 0;
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %6, %6, %4, %5}], [%2];"
      :
      : "r"(smem_dst), "l"(map), "r"(bar_cluster), "r"(k), "r"(c3), "r"(c4), "r"(z)
      : "memory");
}
__device__ __forceinline__ void tma_load_w(uint32_t smem_dst, const CUtensorMap* map, int k, int c3, int c4, uint64_t* bar) {
  const int z = 0;
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %6, %6, %4, %5}], [%2];"
      :
      : "r"(smem_dst), "l"(map), "r"(smem_u32(bar)), "r"(k), "r"(c3), "r"(c4), "r"(z)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                               uint32_t accumulate) {
  const uint32_t z = 0;
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, {%5, %5, %5, %5, %5, %5, %5, %5}, p;\n}"
      :
      : "r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate), "r"(z)
      : "memory");
}
// arrives on this barrier in both CTAs of the pair (mask: their cluster ranks)
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"(mask)
               : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_slot)), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(smem_u32(bar)), "r"(parity)
               : "memory");
  return ok != 0;
}
__device__ __forceinline__ void st_cluster_f4(uint32_t addr_cluster, const float4& v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr_cluster), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

// ---- where the epilogue takes its accumulator values (32 features x 32 tokens per warp) from --------------------------------
// Thread `lane` holds features rg + 8 q (rg = lane / 4, q = 0 .. 3 within the warp's 32) of tokens 8 k + 2 (lane % 4) + e (k = 0 .. 3,
// e = 0, 1) of the chunk: value (q, k, e) at index 16 (q / 2) + 4 k + 2 (q % 2) + e.
__device__ __forceinline__ int vidx(int q, int k, int e) { return 16 * (q >> 1) + 4 * k + 2 * (q & 1) + e; }
__device__ __forceinline__ void tmem_ld_chunk(uint32_t taddr, float (&v)[32]) {   // taddr: (lane quadrant, first column)
  uint32_t r[32];
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[16 * h]), "=r"(r[16 * h + 1]), "=r"(r[16 * h + 2]), "=r"(r[16 * h + 3]), "=r"(r[16 * h + 4]), "=r"(r[16 * h + 5]),
          "=r"(r[16 * h + 6]), "=r"(r[16 * h + 7]), "=r"(r[16 * h + 8]), "=r"(r[16 * h + 9]), "=r"(r[16 * h + 10]),
          "=r"(r[16 * h + 11]), "=r"(r[16 * h + 12]), "=r"(r[16 * h + 13]), "=r"(r[16 * h + 14]), "=r"(r[16 * h + 15])
        : "r"(taddr + ((uint32_t)(16 * h) << 16)));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ float4 ld_volatile_f4(const float4* p) {   // generic address: shared or global memory
  float4 t;
  asm volatile("ld.volatile.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "l"(p) : "memory");
  return t;
}
// Partial tiles hold the values as the threads hold them, [chunk][8][128 threads][4] fp32: a warp's access is 512 contiguous
// bytes.  Parts are added in part order starting from zero, so the result does not depend on who arrived last.
struct Source {
  uint32_t tacc;          // TMEM address of (lane quadrant, column 0): the only part, or part `own`
  int n_parts, own;
  bool cluster;           // the copies are of this member's chunks only, the parts of a chunk one after the other
  const float4* first;    // part 0 where it lies apart from the others (workspace), else null
  const float4* rest;     // the other parts (+ this thread): from part 1 on if `first`, else without part `own`
  size_t stride;          // from one part to the next
  // chunk c, the nth one that this CTA finishes
  __device__ __forceinline__ void load(int c, int nth, float (&v)[32]) const {
    if (n_parts == 1) {
      tmem_ld_chunk(tacc + c * 32, v);
      return;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = 0.f;
    const size_t at = (size_t)(cluster ? nth * (n_parts - 1) : c) * (kChunkBytes / 16);
#pragma unroll 1
    for (int p = 0; p < n_parts; ++p) {
      if (p == own) {
        float t[32];
        tmem_ld_chunk(tacc + c * 32, t);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] += t[i];
      } else {
        const float4* q = (first && p == 0 ? first : rest + (size_t)(p - ((first || p > own) ? 1 : 0)) * stride) + at;
        float4 t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = ld_volatile_f4(q + (size_t)i * FT);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[4 * i] += t[i].x; v[4 * i + 1] += t[i].y; v[4 * i + 2] += t[i].z; v[4 * i + 3] += t[i].w;
        }
      }
    }
  }
};

// ---- work decomposition -----------------------------------------------------------------------------------------------------
// The rows of the batch in equal token tiles: as few as tmax allows, each a multiple of gran wide (tmax is one too).
__host__ __device__ inline void token_tiles(int M, int tmax, int gran, int* width, int* count) {
  const int n = (M + tmax - 1) / tmax;
  const int per = (M + n - 1) / n;
  *width = (per + gran - 1) / gran * gran;
  *count = (M + *width - 1) / *width;
}

// Whole tiles, token-fastest, strided over the units; and "stream-K" for the last columns (all of them, or the ragged end of the
// whole tiles), done per COLUMN of output tiles (the mt token tiles that share one weight tile; the cut columns may have
// narrower token tiles of their own): the k-blocks of the columns form one line of cut_cols * KB units, column after column; a
// TEAM of mt units (unit team * mt + i works on token tile i) owns the contiguous range [team * per, (team + 1) * per) and walks
// it in step, so that the members read the same weight k-blocks at the same time and share them through L2, exactly like the
// CTAs of a wave of whole tiles.  A column may be cut by team boundaries; each owner computes its K range of its token tile
// ("part").  Part p >= 1 of a tile is always the FIRST piece of its unit, part 0 the last piece (or the first, when the range
// starts exactly at the column): that decides the workspace slot, 2 * unit + (first piece ? 0 : 1).
// K-blocks per team for a line of `cols` columns.
__host__ __device__ inline int cut_range(int cols, int mt, int KB, int n_units) {
  const int total = cols * KB, n_teams = n_units / mt;       // (launch_gemm_tc keeps the line within int; mt <= n_units)
  const int per = (total + n_teams - 1) / n_teams;
  return per < 4 && total >= 4 ? 4 : per;                    // pieces long enough to amortise their hand-over
}

// Row count on the device: the token tiles and the columns that are cut over K for every 32 rows up to kPlanRows * 32, as the
// host's estimate chooses them (device_plan); more rows come in whole tiles of the widest kind.  Widths in units of 32 tokens.
// (28672 x 4096 weights at 320, 512, 848 and 1024 rows: 67.7, 99, 158 and 179 us; when any choice of cut columns cut all of
// them, 94, 131, 238 and 243.)
constexpr int kPlanRows = 64;
struct DevPlan {
  uint8_t tmax[kPlanRows], cut_tmax[kPlanRows];
  uint16_t cut_cols[kPlanRows];
};
struct Tiling {
  int width, mt;                       // tokens per tile, token tiles
  int cut_cols, cut_width, cut_mt;     // last columns whose tiles are cut, their token tiles (never wider than the others)
  int per;                             // k-blocks of a team's range
};
__host__ __device__ inline Tiling tiling(int M, int tmax, int gran, int cut_cols, int cut_tmax, int KB, int n_units) {
  Tiling t;
  token_tiles(M, tmax, gran, &t.width, &t.mt);
  t.cut_cols = cut_cols;
  t.cut_width = t.width;
  t.cut_mt = t.mt;
  t.per = 1;
  if (cut_cols) {
    token_tiles(M, cut_tmax < t.width ? cut_tmax : t.width, gran, &t.cut_width, &t.cut_mt);
    if (t.cut_mt <= n_units) t.per = cut_range(cut_cols, t.cut_mt, KB, n_units);      // (else refused by the host)
  }
  return t;
}
__host__ __device__ inline Tiling planned(const DevPlan& p, int M, int KB, int n_units) {
  const int i = (M - 1) / 32;
  return i < kPlanRows ? tiling(M, 32 * p.tmax[i], 32, p.cut_cols[i], 32 * p.cut_tmax[i], KB, n_units)
                       : tiling(M, kMaxTok, 32, 0, 0, KB, n_units);
}

struct Piece {
  int col, tm;            // column of tiles and token tile
  int kb0, kb1;           // k-block range
  bool cut;               // of the stream-K line: token tiles of the cut columns
  int part, n_parts;      // which part of the tile this is
  int slot;               // workspace slot if n_parts > 1
  int slot0, slot_next;   // slots of part 0 and part 1 (for the reducing CTA)
  int counter;            // arrival counter of the tile
};
struct Schedule {
  int KB, n_units;
  int whole, mt;          // whole tiles, token tiles of their columns
  int cut_col0, cut_mt;   // first cut column, token tiles of the cut columns
  int per;                // k-blocks of a team's range
};
// Next piece of this unit: first its range of the stream-K line (pos advances by reference), then its whole tiles
// (jd counts them).  The cut tiles come first so that parking and reducing their partials overlaps the main loop
// of the whole tiles that follow, instead of happening in every CTA at once at the end of the kernel.
__device__ __forceinline__ Piece make_piece(const Schedule& S, int& jd, int& pos, int hi, int unit) {
  Piece p;
  if (pos >= hi) {
    const int tile = unit + jd * S.n_units;
    ++jd;
    p.col = tile / S.mt;
    p.tm = tile - p.col * S.mt;
    p.kb0 = 0;
    p.kb1 = S.KB;
    p.cut = false;
    p.part = 0;
    p.n_parts = 1;
    p.slot = p.slot0 = p.slot_next = p.counter = 0;
    return p;
  }
  const int team = unit / S.cut_mt, member = unit - team * S.cut_mt;
  const int col = pos / S.KB;
  p.kb0 = pos - col * S.KB;
  const int room = hi - pos;
  p.kb1 = room < S.KB - p.kb0 ? p.kb0 + room : S.KB;
  const int t0 = col * S.KB, t1 = t0 + S.KB;
  const int c_first = t0 / S.per, c_last = (t1 - 1) / S.per;    // first and last team on this column
  p.cut = true;
  p.n_parts = c_last - c_first + 1;
  p.part = team - c_first;
  const bool first_piece = pos == team * S.per;
  p.slot = 2 * unit + (first_piece ? 0 : 1);
  p.slot0 = 2 * (c_first * S.cut_mt + member) + (c_first * S.per >= t0 ? 0 : 1);
  p.slot_next = 2 * ((c_first + 1) * S.cut_mt + member);
  p.counter = col * S.cut_mt + member;
  p.col = S.cut_col0 + col;
  p.tm = member;
  pos += p.kb1 - p.kb0;
  return p;
}

// ---- epilogues --------------------------------------------------------------------------------------------------------------
struct TileOut {
  int tile;              // 128-feature tile
  int t0, nv;            // first token, tokens of the tile that exist
  int quad, lane;
  const float* rstd;     // shared: row factors (ss_in given)
  const int* slot;       // shared: cache slots (rotary epilogue)
  float* ss;             // shared: [4][256]
  uint8_t* stage;        // shared: this warp's 2 KB
};
// What the epilogue of a chunk reads besides the accumulator: the old residual values (index as the accumulator's), or the
// rotary factors: (cos, sin) of (q = 0 / 1, k, e) at 2 vidx(q, k, e).  Fetched ahead: for the first chunk while the accumulator is
// still being computed, like the next norm's gains of the thread's four features.
__device__ __forceinline__ void load_gain(const EpiParams& ep, int tile, int quad, int lane, float (&gain)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int f = tile * FT + quad * 32 + (lane >> 2) + 8 * q;
    gain[q] = ep.epi == EPI_RESIDUAL_NORM && f < ep.N ? __bfloat162float(ep.gain[f]) : 0.f;
  }
}
__device__ __forceinline__ void prefetch_chunk(const EpiParams& ep, const TileOut& o, int c, float (&pre)[32]) {
  const int rg = o.lane >> 2, tok = c * 32 + 2 * (o.lane & 3), nv = o.nv;
  if (ep.epi == EPI_RESIDUAL_NORM) {
    const int f = o.tile * FT + o.quad * 32 + rg;
    const float* h = static_cast<const float*>(ep.out) + (size_t)(o.t0 + tok) * ep.N + f;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          pre[vidx(q, k, e)] = (tok + 8 * k + e < nv && f + 8 * q < ep.N) ? __ldcg(h + (size_t)(8 * k + e) * ep.N + 8 * q) : 0.f;
  } else if (ep.epi == EPI_QKV_ROPE) {
    const int half = ep.head_dim / 2, g = ep.head_dim == 128 ? o.quad : (o.quad & 1);
    const float2* tab = ep.rope_cs + (size_t)(o.t0 + tok) * half + g * 16 + rg;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float2 cs = tok + 8 * k + e < nv ? __ldcg(tab + (size_t)(8 * k + e) * half + 8 * q) : make_float2(1.f, 0.f);
          pre[2 * vidx(q, k, e)] = cs.x;
          pre[2 * vidx(q, k, e) + 1] = cs.y;
        }
  }
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
// The chunk as bf16 rows [32 tokens][32 features] in the warp's staging: 16-byte piece p of token t at piece p ^ ((t >> 1) & 3)
// of its 64 bytes (conflict free both ways).
__device__ __forceinline__ void stage_rows32(const TileOut& o, const float (&v)[32]) {
  const int m = o.lane >> 3;             // this lane gives the address of row lane % 8 of matrix m = 8 features
  __syncwarp();                          // the previous chunk has been read
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int t = 8 * k + (o.lane & 7);
    stmatrix_x4_trans(smem_u32(o.stage) + t * 64 + ((m ^ ((t >> 1) & 3)) << 4), pack_bf16(v[vidx(0, k, 0)], v[vidx(0, k, 1)]),
                      pack_bf16(v[vidx(1, k, 0)], v[vidx(1, k, 1)]), pack_bf16(v[vidx(2, k, 0)], v[vidx(2, k, 1)]),
                      pack_bf16(v[vidx(3, k, 0)], v[vidx(3, k, 1)]));
  }
  __syncwarp();
}
// ... and the pieces handed to put(token, piece, 16 bytes), eight tokens x four pieces at a time
template <typename Put>
__device__ __forceinline__ void unstage_rows32(const TileOut& o, int nv, const Put& put) {
  const int p = o.lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int t = 8 * i + (o.lane >> 2);
    const uint4 w = *reinterpret_cast<const uint4*>(o.stage + t * 64 + ((p ^ ((t >> 1) & 3)) << 4));
    if (t < nv) put(t, p, w);
  }
}
// Epilogue of the token chunks c0, c0 + step, ... < c1 (32 tokens each) of an accumulator tile; the four epilogue warps call
// together.  pre: what prefetch_chunk brings for chunk c0.
__device__ __forceinline__ void tile_out(const EpiParams& ep, const Source& src, const TileOut& o, int c0, int c1, int step,
                                         float (&pre)[32], const float (&gain)[4]) {
  const int lane = o.lane, rg = lane >> 2, tq = lane & 3;
  const int f0 = o.tile * FT + o.quad * 32;    // first feature of the warp (not of SwiGLU and the rotary epilogue)
  auto scale = [&](int c, float (&v)[32]) {    // the row factors of a normalised input
    if (!ep.ss_in) return;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 s = *reinterpret_cast<const float2*>(o.rstd + c * 32 + 8 * k + 2 * tq);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[vidx(q, k, 0)] *= s.x;
        v[vidx(q, k, 1)] *= s.y;
      }
    }
  };
  if (ep.epi == EPI_RESIDUAL_NORM) {
    // every element has one writer, so the residual add is a load (ahead of the accumulator) and a store; the new value also
    // gives the next norm's input x = bf16(h * gain) and the row's sum of squares over this tile's features
#pragma unroll 1
    for (int c = c0, nth = 0; c < c1; c += step, ++nth) {
      const int nv = o.nv - c * 32;
      float* h = static_cast<float*>(ep.out) + (size_t)(o.t0 + c * 32 + 2 * tq) * ep.N + f0 + rg;
      float v[32], sq[8];
      src.load(c, nth, v);
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float s = 0.f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float& x = v[vidx(q, k, e)];
            x += pre[vidx(q, k, e)];
            if (2 * tq + 8 * k + e < nv && f0 + rg + 8 * q < ep.N) h[(size_t)(8 * k + e) * ep.N + 8 * q] = x;
            else x = 0.f;
            s = fmaf(x, x, s);
            x *= gain[q];
          }
          sq[2 * k + e] = s;
        }
      if (c + step < c1) prefetch_chunk(ep, o, c + step, pre);
      stage_rows32(o, v);
      __nv_bfloat16* xp = ep.x_out + (size_t)(o.t0 + c * 32) * ep.N + f0;
      unstage_rows32(o, nv, [&](int t, int p, const uint4& w) {
        if (f0 + 8 * p < ep.N) *reinterpret_cast<uint4*>(xp + (size_t)t * ep.N + 8 * p) = w;
      });
      // sums of squares over the warp's 32 features: the eight lanes of a token column (lane / 4) halve the tokens at each step
#pragma unroll
      for (int s = 4; s; s >>= 1) {           // lane bits 4, 3, 2 <-> token index bits 2, 1, 0 of the thread's eight
        const bool up = lane & (4 * s);
#pragma unroll
        for (int j = 0; j < s; ++j) {
          const float keep = up ? sq[j + s] : sq[j], send = up ? sq[j] : sq[j + s];
          sq[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * s);
        }
      }
      // thread holds index rg = 2 k + e
      o.ss[o.quad * kMaxTok + c * 32 + 8 * (rg >> 1) + 2 * tq + (rg & 1)] = sq[0];
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    for (int t = (c0 + o.quad * step) * 32 + lane; t < o.nv; t += 128 * step)       // warp w sums the chunks c0 + w step, ...
      ep.ss_out[(size_t)o.tile * ep.ss_stride + o.t0 + t] =
          (o.ss[t] + o.ss[kMaxTok + t]) + (o.ss[2 * kMaxTok + t] + o.ss[3 * kMaxTok + t]);
    asm volatile("bar.sync 1, 128;" ::: "memory");      // (the sums may be overwritten)
    return;
  }
  if (ep.epi == EPI_SWIGLU) {
    // features 0-15 of the warp: gate, 16-31: the up features that belong to them
    const int fo = o.tile * (FT / 2) + o.quad * 16;
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(ep.out) + (size_t)o.t0 * ep.N + fo;
#pragma unroll 1
    for (int c = c0, nth = 0; c < c1; c += step, ++nth) {
      float v[32];
      src.load(c, nth, v);
      scale(c, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = silu_f(v[i]) * v[16 + i];
      // rows [32 tokens][16 features] of 32 bytes
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 4; k += 2) {
        const int m = lane >> 3, t = 8 * (k + (m >> 1)) + (lane & 7);
        stmatrix_x4_trans(smem_u32(o.stage) + t * 32 + (m & 1) * 16, pack_bf16(v[vidx(0, k, 0)], v[vidx(0, k, 1)]),
                          pack_bf16(v[vidx(1, k, 0)], v[vidx(1, k, 1)]), pack_bf16(v[vidx(0, k + 1, 0)], v[vidx(0, k + 1, 1)]),
                          pack_bf16(v[vidx(1, k + 1, 0)], v[vidx(1, k + 1, 1)]));
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = 16 * i + (lane >> 1);
        const uint4 w = *reinterpret_cast<const uint4*>(o.stage + t * 32 + (lane & 1) * 16);
        if (fo < ep.N && c * 32 + t < o.nv) *reinterpret_cast<uint4*>(out + (size_t)(c * 32 + t) * ep.N + (lane & 1) * 8) = w;
      }
    }
    return;
  }
  if (ep.epi == EPI_QKV_ROPE) {
    // features 0-15 of the warp: 16 low dims of a head, 16-31: their rotation partners half a head away
    const int D = ep.head_dim, half = D / 2;
    const int head = D == 128 ? o.tile : 2 * o.tile + (o.quad >> 1), g = D == 128 ? o.quad : (o.quad & 1);
    const bool is_q = head < ep.n_q, is_v = head >= ep.n_q + ep.n_kv, live = head < ep.n_q + 2 * ep.n_kv;
    const int kvh = is_v ? head - ep.n_q - ep.n_kv : head - ep.n_q;
    __nv_bfloat16* layer = ep.kv_pool + kv_tile_base(ep.n_pages, ep.n_kv, D, ep.layer, 0, is_q ? 0 : kvh) + (is_v ? kv_tile_elems(D) : 0);
    const size_t page_elems = kv_tile_base(ep.n_pages, ep.n_kv, D, 0, 1, 0);
#pragma unroll 1
    for (int c = c0, nth = 0; c < c1; c += step, ++nth) {
      float v[32];
      src.load(c, nth, v);
      scale(c, v);
      if (!is_v) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float lo = v[i], hi = v[16 + i];
          v[i] = lo * pre[2 * i] - hi * pre[2 * i + 1];
          v[16 + i] = hi * pre[2 * i] + lo * pre[2 * i + 1];
        }
        if (c + step < c1) prefetch_chunk(ep, o, c + step, pre);
      }
      stage_rows32(o, v);
      unstage_rows32(o, o.nv - c * 32, [&](int t, int p, const uint4& w) {
        if (!live) return;
        const int dim = (p >> 1) * half + g * 16 + (p & 1) * 8;
        if (is_q) {
          *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(ep.out) + ((size_t)(o.t0 + c * 32 + t) * ep.n_q + head) * D + dim) = w;
          return;
        }
        const int slot = o.slot[c * 32 + t];
        if (slot < 0) return;
        const int64_t page = slot / kPageSize;
        if (page >= ep.n_pages) {
          set_status(ep.status, DEV_BAD_INDEX);
          return;
        }
        *reinterpret_cast<uint4*>(layer + page * page_elems + kv_tile_offset(slot % kPageSize, dim, D)) = w;
      });
    }
    return;
  }
#pragma unroll 1
  for (int c = c0, nth = 0; c < c1; c += step, ++nth) {
    const int nv = o.nv - c * 32;
    float v[32];
    src.load(c, nth, v);
    scale(c, v);
    if (ep.epi == EPI_PLAIN_BF16) {
      stage_rows32(o, v);
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(ep.out) + (size_t)(o.t0 + c * 32) * ep.N + f0;
      unstage_rows32(o, nv, [&](int t, int p, const uint4& w) {
        if (f0 + 8 * p < ep.N) *reinterpret_cast<uint4*>(out + (size_t)t * ep.N + 8 * p) = w;
      });
    } else {
      float* out = static_cast<float*>(ep.out) + (size_t)(o.t0 + c * 32 + 2 * tq) * ep.N + f0 + rg;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (2 * tq + 8 * k + e < nv && f0 + rg + 8 * q < ep.N) out[(size_t)(8 * k + e) * ep.N + 8 * q] = v[vidx(q, k, e)];
    }
  }
}

struct GemmLaunch {
  int m_cap;                 // rows the maps cover
  int n_cols;                // columns of tiles: feature tiles of 128, or of 256 for pairs
  int K;
  Tiling tiles;              // (row count on the device: of the capacity; the kernel takes its own from the plan)
  int tmax;                  // widest token tile
  int cl;                    // parts per tile that form a cluster (0: no clusters)
  int w_step3, w_step4;      // what a 128-feature tile advances in dimensions 3 and 4 of w's tensor map
  float* split_ws;
  int* split_counters;
  const int* m_dev;
  int m_dev_wait;
};

// x: one load per k-block whatever the width of the token tile.  With the row count on the device that is any multiple of 32, and
// there is a map for each: 4096 x 4096 weights at 376, 848 and 1024 rows 34.1, 54.6 and 59.9 us, with loads of 32 rows (a pair's
// CTAs 16) 37.4, 63.2 and 65.6.
template <bool DEV> struct XMaps;
template <> struct XMaps<false> {
  CUtensorMap whole, cut;              // boxes of a token tile's rows (of a pair's CTA: half of them)
};
template <> struct XMaps<true> {
  CUtensorMap wide[kMaxTok / 32];      // likewise, by width / 32 - 1
  DevPlan plan;
};

template <bool PAIR, bool DEV>
__global__ void __launch_bounds__(kTcThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ XMaps<DEV> X, GemmLaunch G, EpiParams ep) {
  // Device-resident rounds: the row count comes from device memory; the tensor maps cover the capacity, and rows
  // between the count and the capacity hold stale data and are computed but never used.  The count is written by the
  // first kernel of the step, and the small kernels between it and the first projection signal their dependents before
  // they wait themselves, so the FIRST projection of a step can be running before that one has finished: it has to wait
  // for its predecessors before it reads the count (m_dev_wait; it gives up the early weight requests).  The first
  // projection signals its own dependents only after that wait, so for every kernel behind it the count is settled.
  if (DEV && G.m_dev_wait) griddep_wait();
  const int M = DEV ? *reinterpret_cast<const volatile int*>(G.m_dev) : G.m_cap;
  if (M <= 0) {                // an empty round (the same for every thread of the grid): nothing to do, nothing was set up yet
    griddep_wait();            // (this grid must not count as complete before the ones it follows are)
    return;
  }
  constexpr int kMul = PAIR ? 2 : 1;                     // CTAs of a scheduling unit; they use separate slots and counters
  const uint32_t crank = (PAIR || G.cl) ? cluster_ctarank() : 0u;
  const uint32_t rank = PAIR ? (crank & 1u) : 0u;        // within the pair
  const uint32_t lead_rank = crank & ~1u;                // cluster rank of the pair's leader (PAIR)
  const int cl = G.cl;
  const uint32_t part_rank = cl ? crank / kMul : 0u;     // which part of the cluster's tile this unit computes
  const int unit = (int)blockIdx.x / kMul;               // scheduling unit: CTA or pair
  const int n_units = (int)gridDim.x / kMul;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

  const int KB = G.K / BK;
  Tiling tl = G.tiles;
  if constexpr (DEV) tl = cl ? tiling(M, G.tmax, 32, 0, 0, KB, n_units) : planned(X.plan, M, KB, n_units);
  const int nt_tok = tl.width, mt = tl.mt, cut_cols = tl.cut_cols, cut_tok = tl.cut_width, cut_mt = tl.cut_mt, per = tl.per;
  // (the cut columns' token tiles are never wider than the others: one stage layout serves both)
  const int stage_bytes = kABytes + nt_tok / kMul * BK * 2;
  const int part_bytes = (cut_tok + 31) / 32 * kChunkBytes;   // a partial tile in the workspace
  // Clusters: chunk c of the tile (32 tokens) is finished by member c % cl, into whose shared memory the others write their
  // partial sums of it (16 KB each).  A tile of one chunk has a reserve for them at the top of the ring; else they go into the
  // ring itself, once its owner says that its own products have read it.
  const bool reserve = cl && nt_tok <= 32;
  const int ring_bytes = kRingBytes - (reserve ? (cl - 1) * kChunkBytes : 0);
  const int n_stages = ring_bytes / stage_bytes > kMaxStages ? kMaxStages : ring_bytes / stage_bytes;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
  uint64_t* empty_bar = full_bar + kMaxStages;
  uint64_t* tfull_bar = empty_bar + kMaxStages;
  uint64_t* tempty_bar = tfull_bar + 2;
  uint64_t* red_bar = tempty_bar + 2;      // the parts of the others have landed (bulk copies, or the cluster's peers)
  uint64_t* go_bar = red_bar + 1;          // clusters: the other members' rings may be written
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(go_bar + 1);
  float* s_rstd = reinterpret_cast<float*>(smem + kOffRstd);
  int* s_slot = reinterpret_cast<int*>(smem + kOffSlot);
  float* s_ss = reinterpret_cast<float*>(smem + kOffSs);

  // Bounded waits.  The producer and the MMA issuer leave their loops when a wait runs out.  The four epilogue warps
  // must all keep meeting at the named barriers and must keep counting the arrivals of cut tiles (so that the counters
  // stay consistent for the next launch), so they never leave their loop: a wait of theirs that runs out records why
  // and raises a CTA-wide flag, after which their waits return at once; the outputs of such a launch are garbage and
  // the status word says so.  (The flag is only looked at between waits: polling it inside the producer's and the
  // issuer's per-k-block waits cost up to 40 % on narrow tiles.)
  __shared__ volatile int s_abort;
  auto wait_bar = [&](uint64_t* bar, uint32_t parity) -> bool {
    for (uint32_t i = 0; i < kSpin; ++i) {
      if (PAIR ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
      if (i > 64) __nanosleep(32);
    }
    return false;
  };
  auto wait_or_abort = [&](uint64_t* bar, uint32_t parity, int code, bool cluster = false) {   // epilogue warps only
    if (s_abort) return;
    bool ok = false;
    if (cluster) {
      for (uint32_t i = 0; i < kSpin && !ok; ++i) {
        ok = mbar_try_wait_cluster(bar, parity);
        if (!ok && i > 64) __nanosleep(32);
      }
    } else {
      ok = wait_bar(bar, parity);
    }
    if (!ok) {
      set_status(ep.status, code);
      s_abort = 1;
    }
  };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tiles = mt * G.n_cols;
  const Schedule S{KB, n_units, (G.n_cols - cut_cols) * mt, mt, G.n_cols - cut_cols, cut_mt, per};
  // the unit's range of the stream-K line, and its whole tiles
  const int total = cut_cols * KB;
  const int lo_raw = cut_cols ? unit / cut_mt * per : 0;
  const bool cl_live = cl && unit / cl < n_tiles;          // (the grid of a device-resident step is sized for the capacity)
  const int range_lo = cl ? 0 : (lo_raw < total ? lo_raw : total);
  const int range_hi = cl ? (cl_live ? 1 : 0) : (range_lo + per < total ? range_lo + per : total);
  const int dp_count = cl ? 0 : (unit < S.whole ? (S.whole - 1 - unit) / n_units + 1 : 0);
  // the next piece of this unit (a cluster member has exactly one)
  auto next_piece = [&](int& jd, int& pos) -> Piece {
    if (cl) {
      Piece p;
      const int tile = unit / cl;
      p.col = tile / mt;
      p.tm = tile - p.col * mt;
      p.cut = false;
      p.kb0 = (int)part_rank * KB / cl;
      p.kb1 = ((int)part_rank + 1) * KB / cl;
      p.part = (int)part_rank;
      p.n_parts = cl;
      p.slot = p.slot0 = p.slot_next = p.counter = 0;
      pos = range_hi;
      return p;
    }
    return make_piece(S, jd, pos, range_hi, unit);
  };

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull_bar[a], 1);
      mbar_init(&tempty_bar[a], PAIR ? 8 : 4);
    }
    mbar_init(red_bar, cl ? (cl - 1) * 4 : 1);             // (clusters: one arrival per other member and epilogue warp)
    mbar_init(go_bar, cl > 1 ? cl - 1 : 1);
    fence_barrier_init();
    if constexpr (DEV) prefetch_tmap(&X.wide[nt_tok / 32 - 1]);
    else prefetch_tmap(&X.whole);
    prefetch_tmap(&map_w);
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR || cl) cluster_sync_all();       // all CTAs' barriers are initialised before anyone signals across
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // (each role waits for the kernels before this one where it first needs their results)

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    if (elect_one()) {
      // of a pair, rank r loads the weight rows of feature tile 2 c + r and half r of the token tile; all loads of the pair
      // complete on the leader's barrier
      auto expect = [&](int s, bool cut) {
        const int bytes = kMul * kABytes + (cut ? cut_tok : nt_tok) * BK * 2;
        if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], bytes);
      };
      auto load_w = [&](int s, int kb, int col) {
        const uint32_t dst = smem_u32(smem + s * stage_bytes);
        const int ft = col * kMul + (int)rank;
        if constexpr (PAIR) tma_load_w_pair(dst, &map_w, kb * BK, ft * G.w_step3, ft * G.w_step4, mapa_rank(smem_u32(&full_bar[s]), lead_rank));
        else tma_load_w(dst, &map_w, kb * BK, ft * G.w_step3, ft * G.w_step4, &full_bar[s]);
      };
      auto load_x = [&](int s, int kb, int tm, bool cut) {
        uint8_t* dst = smem + s * stage_bytes + kABytes;
        const int tok = cut ? cut_tok : nt_tok, row = tm * tok + (int)rank * (tok / kMul);
        const CUtensorMap* map;
        if constexpr (DEV) map = &X.wide[tok / 32 - 1];
        else map = cut ? &X.cut : &X.whole;
        if constexpr (PAIR) tma_load_2d_pair(smem_u32(dst), map, kb * BK, row, mapa_rank(smem_u32(&full_bar[s]), lead_rank));
        else tma_load_2d(dst, map, kb * BK, row, &full_bar[s]);
      };
      // The weights do not depend on the kernels before this one: the weight tiles of the first stages are requested
      // BEFORE waiting for those kernels, so the ring fills while they drain (or while a short kernel runs); the x tiles of
      // those stages follow right after the wait.
      int n_pre = 0, pre_kb0 = 0, pre_tm = 0;
      bool pre_cut = false;
      if (dp_count > 0 || range_lo < range_hi) {
        int p0 = range_lo;
        int j0 = 0;
        const Piece pc = next_piece(j0, p0);
        n_pre = pc.kb1 - pc.kb0 < n_stages ? pc.kb1 - pc.kb0 : n_stages;
        pre_kb0 = pc.kb0;
        pre_tm = pc.tm;
        pre_cut = pc.cut;
        for (int i = 0; i < n_pre; ++i) {
          expect(i, pre_cut);
          load_w(i, pre_kb0 + i, pc.col);
        }
      }
      griddep_wait();
      for (int i = 0; i < n_pre; ++i) load_x(i, pre_kb0 + i, pre_tm, pre_cut);
      int st_idx = 0, issued = 0;
      uint32_t st_phase = 0;
      bool ok = true;
      int pos = range_lo;
      for (int jd = 0; (jd < dp_count || pos < range_hi) && ok;) {
        const Piece pc = next_piece(jd, pos);
        const int kb0 = pc.kb0, kb1 = pc.kb1;
        for (int kb = kb0; kb < kb1; ++kb) {
          const int s = st_idx;
          const uint32_t ph = st_phase;
          if (++st_idx == n_stages) { st_idx = 0; st_phase ^= 1; }
          if (issued < n_pre) {       // requested above
            ++issued;
            continue;
          }
          if (!wait_bar(&empty_bar[s], ph ^ 1)) {
            set_status(ep.status, DEV_TIMEOUT_EMPTY);
            ok = false;
            break;
          }
          expect(s, pc.cut);
          load_x(s, kb, pc.tm, pc.cut);
          load_w(s, kb, pc.col);
        }
      }
      if (!ok) {  // let loads already issued land before the CTA may exit
        for (int s = 0; s < n_stages; ++s)
          for (uint32_t i = 0; i < (1u << 14); ++i) {
            if (mbar_try_wait(&full_bar[s], 0) || mbar_try_wait(&full_bar[s], 1)) break;
            __nanosleep(64);
          }
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (rank == 0 && elect_one()) {         // of a pair only the leader issues (it touches shared memory and TMEM only)
      const uint32_t idesc_whole = make_idesc(nt_tok, FT * kMul), idesc_cut = make_idesc(cut_cols ? cut_tok : nt_tok, FT * kMul);
      const uint64_t desc0 = make_smem_desc(smem_u32(smem));
      const uint16_t pair_mask = (uint16_t)(3u << lead_rank);
      int st_idx = 0;
      uint32_t st_phase = 0, tcount = 0;
      bool ok = true;
      int pos = range_lo;
      for (int jd = 0; (jd < dp_count || pos < range_hi) && ok; ++tcount) {
        const Piece pc = next_piece(jd, pos);
        const int kb0 = pc.kb0, kb1 = pc.kb1;
        const int acc = tcount & 1;
        if (!wait_bar(&tempty_bar[acc], ((tcount >> 1) & 1) ^ 1)) {
          set_status(ep.status, DEV_TIMEOUT_MMA);
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * kAccStride, idesc = pc.cut ? idesc_cut : idesc_whole;
        for (int kb = kb0; kb < kb1; ++kb) {
          const int s = st_idx;
          const uint32_t ph = st_phase;
          if (++st_idx == n_stages) { st_idx = 0; st_phase ^= 1; }
          if (!wait_bar(&full_bar[s], ph)) {
            set_status(ep.status, DEV_TIMEOUT_FULL);
            ok = false;
            break;
          }
          tc_fence_after();
          // descriptors are linear in the address (the ring lies inside the 14-bit address field without carry), so
          // the descriptor of a 16-column slice is the stage's descriptor plus 32 bytes >> 4
          const uint64_t da0 = desc0 + (uint64_t)((s * stage_bytes) >> 4);
          const uint64_t db0 = da0 + (uint64_t)(kABytes >> 4);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            if constexpr (PAIR) umma_bf16_pair(d_tmem, da0 + 2 * k, db0 + 2 * k, idesc, ((kb - kb0) | k) ? 1u : 0u);
            else umma_bf16(d_tmem, da0 + 2 * k, db0 + 2 * k, idesc, ((kb - kb0) | k) ? 1u : 0u);
          }
          // frees the stage (in both CTAs of a pair) when these MMAs have read it
          if constexpr (PAIR) umma_commit_pair(&empty_bar[s], pair_mask);
          else umma_commit(&empty_bar[s]);
        }
        if (ok) {                            // accumulator complete
          if constexpr (PAIR) umma_commit_pair(&tfull_bar[acc], pair_mask);
          else umma_commit(&tfull_bar[acc]);
        }
      }
    }
  } else {
    // ------------------------------ epilogue warps ------------------------------
    const int quad = warp & 3;             // TMEM lane quadrant this warp may read
    const int row = quad * 32 + lane;      // this thread among the 128 of the epilogue
    const uint32_t tmem_quad = tmem_base + ((uint32_t)(quad * 32) << 16);
    uint32_t tcount = 0;
    int prep_tm = -1;                      // the token tile whose row factors and slots are in shared memory
    __shared__ int s_last;
    TileOut o{0, 0, 0, quad, lane, s_rstd, s_slot, s_ss, smem + kOffStage + quad * 2048};
    float pre[32], gain[4] = {0.f, 0.f, 0.f, 0.f};
    int pos = range_lo;
    bool dry = true;                       // first pass: the epilogue's code without effect (no token exists, values are arbitrary)
    for (int jd = 0; jd < dp_count || pos < range_hi;) {
      Source src{tmem_quad + kAccStride, 1, 0, false, nullptr, nullptr, 0};
      int c_begin = 0, c_end = 1, c_step = 1;     // the chunks that are finished here
      int acc = 0;
      // hands the accumulator back to the MMA issuer (of a pair: the leader's barrier collects both CTAs' warps)
      auto release_acc = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) mbar_arrive_cluster(mapa_rank(smem_u32(&tempty_bar[acc]), lead_rank));
          else mbar_arrive(&tempty_bar[acc]);
        }
      };
      bool release = false, last_sync = false;
      if (dry) {
        if (cl) {
          src.n_parts = cl;
          src.own = (int)part_rank;
          src.rest = reinterpret_cast<const float4*>(smem) + row;
          src.stride = kChunkBytes / 16;
        }
      } else {
        const Piece pc = next_piece(jd, pos);
        const int n_splits = pc.n_parts, width = pc.cut ? cut_tok : nt_tok;
        o.tile = pc.col * kMul + (int)rank;
        o.t0 = pc.tm * width;
        o.nv = M - o.t0 < width ? M - o.t0 : width;
        acc = tcount & 1;
        src.tacc = tmem_quad + acc * kAccStride;
        const int n_chunks = (o.nv + 31) / 32;
        // What the epilogue needs per token, fetched while the accumulator is still being computed: the row factors of a
        // normalised input (the partial sums of squares in slot order: the same bits in every tile of the row) and the slots.
        const int prep = 2 * pc.tm + (pc.cut ? 1 : 0);
        if (prep != prep_tm && (ep.ss_in || ep.epi == EPI_QKV_ROPE)) {
          if (prep_tm >= 0) asm volatile("bar.sync 1, 128;" ::: "memory");
          for (int t = (int)threadIdx.x - 64; t < o.nv; t += 128) {
            if (ep.ss_in) {
              float sq = 0.f;
              const float* p = ep.ss_in + o.t0 + t;
#pragma unroll 8
              for (int k = 0; k < ep.ss_slots; ++k) sq += __ldcg(p + (size_t)k * ep.ss_stride);
              s_rstd[t] = rsqrtf(sq * ep.norm_inv_n + ep.norm_eps);
            }
            if (ep.epi == EPI_QKV_ROPE) s_slot[t] = ep.tok_slot[o.t0 + t];
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
          prep_tm = prep;
        }
        c_end = n_chunks;
        if (cl) {
          c_begin = (int)part_rank;
          c_step = cl;
        }
        // (likewise, where this CTA is sure to finish the tile, what its first tokens need)
        load_gain(ep, o.tile, quad, lane, gain);
        if ((n_splits == 1 || cl) && c_begin < c_end) prefetch_chunk(ep, o, c_begin, pre);
        wait_or_abort(&tfull_bar[acc], (tcount >> 1) & 1, DEV_TIMEOUT_MMA);   // after a timeout: carry on without blocking
        tc_fence_after();
        ++tcount;
        if (n_splits == 1) {
          release = true;
        } else if (cl) {
          uint8_t* land = smem + (reserve ? ring_bytes : 0);
          if (!reserve) {            // this CTA's products are complete and have read its ring (its accumulator is)
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (warp == 2 && lane < cl && lane != (int)part_rank) mbar_arrive_cluster(mapa_rank(smem_u32(go_bar), lane * kMul + rank));
            wait_or_abort(go_bar, 0, DEV_TIMEOUT_EMPTY, true);
          }
#pragma unroll 1
          for (int c = 0; c < n_chunks; ++c) {
            const int owner = c % cl;
            if (owner == (int)part_rank) continue;
            const int at = (c / cl) * (cl - 1) + ((int)part_rank < owner ? (int)part_rank : (int)part_rank - 1);
            const uint32_t dst = mapa_rank(smem_u32(land + at * kChunkBytes), owner * kMul + rank) + row * 16;
            float v[32];
            tmem_ld_chunk(src.tacc + c * 32, v);
#pragma unroll
            for (int i = 0; i < 8; ++i)
              st_cluster_f4(dst + (uint32_t)i * (FT * 16), make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
          }
          __syncwarp();
          if (lane < cl && lane != (int)part_rank && lane < n_chunks)    // release: the warp's stores are visible
            mbar_arrive_cluster(mapa_rank(smem_u32(red_bar), lane * kMul + rank));
          if (c_begin < c_end) wait_or_abort(red_bar, 0, DEV_TIMEOUT_FULL, true);  // the others' parts have landed (acquire at cluster scope)
          src.n_parts = cl;
          src.own = (int)part_rank;
          src.cluster = true;
          src.rest = reinterpret_cast<const float4*>(land) + row;
          src.stride = kChunkBytes / 16;
          release = true;
        } else {
          // park this split's partial tile and let the LAST split to arrive reduce all partials in split order
          // (deterministic) and run the fused epilogue
          // (the two CTAs of a pair park and reduce their 128 features independently: slot and counter index are
          // doubled and offset by the rank)
          const int slot_mine = pc.slot * kMul + (int)rank, slot0 = pc.slot0 * kMul + (int)rank;
          const int slot_next = pc.slot_next * kMul + (int)rank, slot_stride = 2 * cut_mt * kMul;
          const int counter = pc.counter * kMul + (int)rank;
          const size_t part_f4 = part_bytes / 16;
          float4* mine = reinterpret_cast<float4*>(G.split_ws) + slot_mine * part_f4 + row;
#pragma unroll 1
          for (int c = 0; c < n_chunks; ++c) {
            float v[32];
            tmem_ld_chunk(src.tacc + c * 32, v);
#pragma unroll
            for (int i = 0; i < 8; ++i)
              __stcg(mine + (size_t)(c * 8 + i) * FT, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
          }
          // the accumulator may be handed back at once: the own part is read from TMEM again only when nothing follows
          // in this CTA, and then nobody overwrites it
          release_acc();
          asm volatile("bar.sync 1, 128;" ::: "memory");
          if (warp == 2 && lane == 0) {
            __threadfence();   // cumulative: orders the partial rows all 128 threads wrote before the barrier
            const int old = atomicAdd(&G.split_counters[counter], 1);
            s_last = (old == n_splits - 1);
            if (old == n_splits - 1) G.split_counters[counter] = 0;   // ready for the next launch
            __threadfence();
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
          last_sync = true;
          if (!s_last) {
            c_end = 0;
          } else {
            prefetch_chunk(ep, o, 0, pre);
            src.n_parts = n_splits;
            // When nothing follows in this CTA the operand ring is idle (every load was consumed before the accumulator
            // completed): the other parts are fetched into it with bulk copies at full bandwidth and the own part is
            // taken from TMEM.  Otherwise the parts are read from global memory while the next piece's main loop runs.
            const bool final_piece = !(jd < dp_count || pos < range_hi);
            if (final_piece && (n_splits - 1) * part_bytes <= kRingBytes) {
              if (warp == 2 && lane == 0) {
                asm volatile("fence.proxy.async;" ::: "memory");   // the parts were written with ordinary stores
                mbar_arrive_expect_tx(red_bar, (uint32_t)((n_splits - 1) * part_bytes));
                int k = 0;
                for (int p = 0; p < n_splits; ++p) {
                  if (p == pc.part) continue;
                  const int slot = p == 0 ? slot0 : slot_next + slot_stride * (p - 1);
                  const uint8_t* from = reinterpret_cast<const uint8_t*>(G.split_ws) + (size_t)slot * part_bytes;
                  for (int off = 0; off < part_bytes; off += kChunkBytes)
                    bulk_g2s(smem + (size_t)k * part_bytes + off, from + off, kChunkBytes, red_bar);
                  ++k;
                }
              }
              wait_or_abort(red_bar, 0, DEV_TIMEOUT_FULL);
              src.own = pc.part;
              src.rest = reinterpret_cast<const float4*>(smem) + row;
              src.stride = part_f4;
            } else {
              src.own = -1;
              src.first = reinterpret_cast<const float4*>(G.split_ws) + slot0 * part_f4 + row;
              src.rest = reinterpret_cast<const float4*>(G.split_ws) + slot_next * part_f4 + row;
              src.stride = slot_stride * part_f4;
            }
          }
        }
      }
      if (c_begin < c_end) tile_out(ep, src, o, c_begin, c_end, c_step, pre, gain);
      if (release) release_acc();
      if (last_sync) asm volatile("bar.sync 1, 128;" ::: "memory");       // s_last is reused by the next unit
      if (dry) griddep_wait();             // from here on the epilogue reads and writes what earlier kernels produced
      dry = false;
    }
  }

  griddep_launch();   // this CTA's work is done: the next kernel's CTAs may be scheduled onto freed SMs
  tc_fence_before();
  __syncthreads();
  // of a pair, the other CTA may read this CTA's operands and signal its barriers until here; in a cluster without a reserve
  // every member signals and writes the others.  (With a reserve only the shared memory of member 0 is written by others, and
  // it has waited for those stores: they are free to leave.)
  if (PAIR || (cl && !reserve)) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---- host side -------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct MapKey {
  const void* ptr;
  uint64_t rows, cols;
  uint32_t box_rows;     // rows of the box (x), or 0x10000 + the order of w's rows (WeightOrder)
  bool operator==(const MapKey& o) const { return ptr == o.ptr && rows == o.rows && cols == o.cols && box_rows == o.box_rows; }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    return std::hash<const void*>()(k.ptr) ^ (k.rows * 1000003u) ^ (k.cols * 7919u) ^ (size_t)k.box_rows << 40;
  }
};

constexpr size_t kSplitWsBytes = 96ull << 20;   // partial tiles of split-K launches
constexpr int kSplitCounters = 1 << 16;
constexpr size_t kMapCacheMax = 4096;           // entries; the keys include the row count, so a serving loop keeps adding

// How a projection runs: single CTAs or CTA pairs, the widest token tile, clusters of cl parts per tile or the last cut_cols
// columns cut over K in token tiles of at most cut_tmax.
struct Config {
  bool pair;
  int tmax, cl, cut_cols, cut_tmax;
};
struct Shape {
  int M, n_feat, K;       // n_feat: rows of w
  int cap;                // 0, or (row count on the device) the rows that the launch has to cover
  bool operator==(const Shape& o) const { return M == o.M && n_feat == o.n_feat && K == o.K && cap == o.cap; }
};
struct ShapeHash {
  size_t operator()(const Shape& s) const { return (size_t)s.M * 1000003u ^ (size_t)s.n_feat * 7919u ^ (size_t)s.K << 32 ^ (size_t)s.cap << 20; }
};
struct TcState {
  int n_sm = 0;
  int force_tile = 0, force_s = 0;
  float* split_ws = nullptr;
  int* split_counters = nullptr;
  EncodeTiledFn encode = nullptr;
  std::unordered_map<MapKey, CUtensorMap, MapKeyHash> maps;
  size_t evictions = 0;
  std::unordered_map<Shape, Config, ShapeHash> configs;    // choose_config's answers (emptied when there are kMapCacheMax)
  std::unordered_map<Shape, DevPlan, ShapeHash> plans;     // device_plan's, with `pair` in the place of the rows
  bool configured[2][2] = {{false, false}, {false, false}};
  bool clusters = true;       // tiles cut over K may be handed over inside clusters
  int max_clusters[2][9];     // cached occupancy answers, single CTAs / pairs and cluster size in CTAs (-1: not asked yet)
  TcState() {
    for (auto& row : max_clusters)
      for (int& v : row) v = -1;
  }
};

// Cache of encoded tensor maps (TcState::maps).  Maps are handed out BY VALUE: a launch needs several at once,
// and a miss on a later lookup may empty the full cache, so nothing may point into it.
template <typename Encode>
bool cached_map(TcState* st, const MapKey& key, CUtensorMap* out, Encode&& encode) {
  auto it = st->maps.find(key);
  if (it != st->maps.end()) {
    *out = it->second;
    return true;
  }
  CUtensorMap m;
  if (!encode(&m)) return false;
  if (st->maps.size() >= kMapCacheMax) {   // emptied, never trimmed behind a caller's back: maps leave by value
    st->maps.clear();
    ++st->evictions;
  }
  st->maps.emplace(key, m);
  *out = m;
  return true;
}

// x [rows, cols] bf16 row-major, box = [box_rows, 64 columns], 128-byte swizzle, zero fill out of bounds
bool get_x_map(TcState* st, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, CUtensorMap* out) {
  return cached_map(st, MapKey{ptr, rows, cols, box_rows}, out, [&](CUtensorMap* m) {
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {BK, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return st->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  });
}

// w [rows, K] as five dimensions (k, 16 rows, halves, groups, heads); one box is the 128 rows of a feature tile in the order
// the epilogue wants them in the TMEM lanes:
//   plain   rows as they are
//   SwiGLU  16 gate rows, the 16 up rows that belong to them, the next 16 gate rows ... (rows = 2 F)
//   rotary  per head: 16 low dims, their 16 partners half a head away, the next 16 low dims ...
enum WeightOrder { kWPlain = 0, kWSwiglu = 1, kWRope128 = 2, kWRope64 = 3 };
bool get_w_map(TcState* st, const void* ptr, uint64_t rows, uint64_t K, WeightOrder order, CUtensorMap* out, int* step3, int* step4) {
  *step3 = order == kWPlain ? 8 : (order == kWSwiglu ? 4 : 0);
  *step4 = order == kWRope128 ? 1 : (order == kWRope64 ? 2 : 0);
  return cached_map(st, MapKey{ptr, rows, K, 0x10000u + (uint32_t)order}, out, [&](CUtensorMap* m) {
    const cuuint64_t r = K * 2;      // bytes of a row
    cuuint64_t dims[5] = {K, 16, 1, rows / 16, 1}, strides[4] = {r, 16 * r, 16 * r, 128 * r};
    cuuint32_t box[5] = {BK, 16, 1, 8, 1}, estr[5] = {1, 1, 1, 1, 1};
    if (order == kWSwiglu) {
      dims[2] = 2; dims[3] = rows / 32;
      strides[1] = rows / 2 * r;
      box[2] = 2; box[3] = 4;
    } else if (order == kWRope128 || order == kWRope64) {
      const int D = order == kWRope128 ? 128 : 64;
      dims[2] = 2; dims[3] = D / 32; dims[4] = rows / D;
      strides[1] = D / 2 * r; strides[3] = D * r;
      box[2] = 2; box[3] = D / 32; box[4] = 128 / D;
    }
    return st->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptr), dims, strides, box, estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  });
}

typedef void (*KernelHost)(CUtensorMap, XMaps<false>, GemmLaunch, EpiParams);
typedef void (*KernelDev)(CUtensorMap, XMaps<true>, GemmLaunch, EpiParams);
KernelHost kernel_host(bool pair) { return pair ? gemm_tc_kernel<true, false> : gemm_tc_kernel<false, false>; }
KernelDev kernel_dev(bool pair) { return pair ? gemm_tc_kernel<true, true> : gemm_tc_kernel<false, true>; }

bool configure(TcState* st, bool pair, bool dev) {
  if (st->configured[pair][dev]) return true;
  const void* k = dev ? reinterpret_cast<const void*>(kernel_dev(pair)) : reinterpret_cast<const void*>(kernel_host(pair));
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) return false;
  return st->configured[pair][dev] = true;
}

// Whether n clusters of `size` CTAs are resident at once (the occupancy query's answer is kept).
bool clusters_fit(TcState* st, bool pair, int size, int n) {
  if (size > 8 || !configure(st, pair, false)) return false;
  int& cached = st->max_clusters[pair][size];
  if (cached < 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size * n);
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int got = 0;
    if (cudaOccupancyMaxActiveClusters(&got, kernel_host(pair), &cfg) != cudaSuccess) {
      cudaGetLastError();
      got = 0;
    }
    cached = got;
  }
  return cached >= n;
}

// Estimated time in microseconds, fitted to B200 measurements of the five 8B-class projections at 8 to 1864 rows (single calls
// back to back, weights from HBM; within about 10 %).
// A k-block of a tile costs (.075 + .001 x tokens) us alone and a third more when all SMs pull operands through L2; a CTA pair
// .085 + .00085 x tokens and a quarter more.  Examples, all SMs busy: 128 features x 256 tokens .44 us, 256 x 256 .37, 256 x 128
// .24.  Below .18 us a CTA is bound by the latency of its loads.
// The weights come from HBM once, at 6.7 TB/s when 105 CTAs or more stream them, .093 TB/s per CTA for a few, 2.2 TB/s + .043 per
// CTA in between (so four parts per tile and not two: 5120 x 17408 weights at 80 rows 39.7 us on 80 CTAs, 34.9 on 120).  The
// shorter of the two, products and stream, shows through by a tenth (128256 x 4096 at 128 rows 180 us on single CTAs, 174 on
// pairs, with 121 and 104 us of products under 157 us of stream).
// On top come the ends (launch, first loads, last tile's epilogue; more for pairs): 4.5 us + .003 x tokens for whole tiles; 5.6 us when
// clusters reduce tiles of one chunk, 6 us + 1 us per chunk that a member sends for wider ones, .4 us per further token tile;
// 11.5 us + .05 x tokens when all tiles are cut and go through the workspace (parking, counting, fetching, the epilogue in the
// last part to arrive).
// A ragged last wave of whole tiles: its columns can be cut over all units and done first, in narrower token tiles so that a tile
// has few parts; their hand-over hides under the whole tiles behind them.  28672 x 4096
// weights at 320, 376, 416 and 1024 rows: 65.5, 72.6, 79.9 and 161.9 us, all tiles whole 69.8, 77.6, 85.1 and 167.3; 4096 x 14336
// at 1331 rows 111.4 instead of 118.9 with the cut tiles as wide as the others.
double est_kblock(bool pair, int width, double busy) {
  if (busy > 1.0) busy = 1.0;
  const double t = pair ? (.085 + .00085 * width) * (.95 + .25 * busy) : (.075 + .001 * width) * (.92 + .40 * busy);
  return fmax(t, .18);
}

// kinds: which of single CTAs (1) and pairs (2) to look at, and whether clusters may be chosen (4)
Config estimate(TcState* st, const Shape& s, int kinds) {
  const int KB = s.K / BK;
  const auto with_stream = [&](double products, double ctas) {
    const double t = 2.0 * s.n_feat * s.K / fmin(6.7e6, fmin(93e3 * ctas, 2.2e6 + 43e3 * ctas));
    return fmax(products, t) + .1 * fmin(products, t);
  };
  Config best{false, kMaxTok, 0, 0, 0};
  double best_t = 1e30;
  for (int pair = 0; pair < 2; ++pair) {
    if (!(kinds & (pair + 1))) continue;
    const int gran = pair || s.cap ? 32 : 16, units = pair ? st->n_sm / 2 : st->n_sm;
    const int cols = (s.n_feat + FT * (pair + 1) - 1) / (FT * (pair + 1));
    const int fewest = (s.M + kMaxTok - 1) / kMaxTok;
    const double pair_end = pair ? .3 : 0.0;
    int last = 0;
    // (few k-blocks: the epilogue is what takes time, so as many and narrow tiles as one wave holds.  256 x 256 weights at 1024
    // rows, fp32 results, 3.7 us, 4.9 with a few more tiles than the fewest; 16 x 64 at 4000 rows 4.7 and 5.2; a prefill of the
    // 2-layer model of width 256 at 1024 rows 103 and 118)
    const int most = fewest + 3 + fewest / 4, wave = KB <= 4 ? units / cols : 0;
    for (int want = fewest; want <= (wave > most ? wave : most); ++want) {
      const int tmax = ((s.M + want - 1) / want + gran - 1) / gran * gran;    // the widest tile that gives `want` tiles
      if (tmax == last || tmax < gran) continue;
      last = tmax;
      int width, mt;
      token_tiles(s.M, tmax, gran, &width, &mt);
      const long long tiles = (long long)mt * cols;
      if (want > fewest && width < 32) continue;
      auto consider = [&](double t, int cl, int cut_cols, int cut_tmax) {
        if (t < best_t) {
          best_t = t;
          best = Config{pair != 0, tmax, cl, cut_cols, cut_tmax};
        }
      };
      const long long full = tiles / units, rem = tiles % units;      // full waves, and a last one that has the machine to itself
      const double ends = 4.5 + .003 * width + pair_end, t_full = full * KB * est_kblock(pair, width, 1.0);
      consider(with_stream(t_full + (rem ? KB * est_kblock(pair, width, (double)rem / units) : 0.0), (full ? units : rem) * (pair + 1.0)) + ends,
               0, 0, 0);
      if (full == 0) {
        // all tiles cut over K through the workspace
        if (mt <= units)
          consider(with_stream((double)tiles * KB / ((units / mt) * mt) * est_kblock(pair, width, 1.0), st->n_sm) + 11.5 + .05 * width, 0,
                   cols, tmax);
      } else if (rem) {
        const int cut = cols - (int)(full * units / mt);
        int cut_last = 0;
        for (int cw = fewest; cw <= s.M / 16 && cw <= units; ++cw) {     // token tiles of the cut columns
          const int ctmax = ((s.M + cw - 1) / cw + gran - 1) / gran * gran;
          if (ctmax == cut_last || ctmax > width) continue;
          cut_last = ctmax;
          int c_width, c_mt;
          token_tiles(s.M, ctmax, gran, &c_width, &c_mt);
          if (c_mt > units || c_mt * cut * (pair + 1) > kSplitCounters) continue;
          const int per = cut_range(cut, c_mt, KB, units), parts = (KB + per - 1) / per + 1;
          // (6 %: below that the cut lost as often as it won; under the power limit a ragged wave's idle time is given back as
          // clock.  28672 features, 256 tokens: 60 us cut, 56 whole; the LM head at 480: 384 and 375.)
          // reducing (the parts of a chunk fetched one after the other) holds the reducing unit's epilogue; what exceeds the main
          // loop of its next tile holds its products, too
          const double hand = (c_width + 31) / 32 * (.6 + 1.3 * parts);
          const double t = t_full + per * est_kblock(pair, c_width, 1.0) + 3.0 + fmax(0.0, hand - KB * est_kblock(pair, width, 1.0));
          consider(1.06 * (with_stream(t, st->n_sm) + ends), 0, cut, ctmax);
        }
      }
      // clusters of 2 to 4 parts per tile, all resident at once
      const int chunks = (width + 31) / 32;
      for (int cl = 2; cl <= 4 && st->clusters && (kinds & 4); ++cl) {
        if (tiles * cl > units || cl * 4 > KB || !clusters_fit(st, pair, cl * (pair + 1), (int)tiles)) break;
        const double cl_ends = (chunks == 1 ? 5.6 : 6.0 + (double)chunks * (cl - 1) / cl) + .4 * (mt - 1) + pair_end;
        consider(with_stream((KB + cl - 1) / cl * est_kblock(pair, width, (double)tiles * cl / units), tiles * cl * (pair + 1.0)) + cl_ends,
                 cl, 0, 0);
      }
    }
  }
  return best;
}

Config choose_config(TcState* st, const Shape& s) {
  const auto known = st->configs.find(s);
  if (known != st->configs.end()) return known->second;
  Config c = estimate(st, s, 7);
  // With the row count on the device one token tile takes any of them, so that of a cluster is as wide as the capacity allows:
  // there are no clusters for tiles that turn out not to exist, which take SMs from the others.
  if (s.cap && c.cl && s.M <= c.tmax) c.tmax = s.cap < kMaxTok ? (s.cap + 31) / 32 * 32 : kMaxTok;
  if (st->configs.size() >= kMapCacheMax) st->configs.clear();
  st->configs.emplace(s, c);
  return c;
}

// The division for every row count that a launch may find on the device: the caller's hint decides between single CTAs, pairs and
// clusters, everything else is chosen as if the row count were known.  All rows of an entry have the same token tiles (tile
// widths and entries are multiples of 32 rows).
DevPlan make_plan(const std::function<Config(int)>& config_of, int cap, int n_feat, int K, bool pair, int n_sm) {
  const int mul = pair ? 2 : 1, n_units = n_sm / mul, n_cols = (n_feat + FT * mul - 1) / (FT * mul);
  DevPlan p;
  for (int i = 0; i < kPlanRows; ++i) {
    const int rows = 32 * (i + 1) < cap ? 32 * (i + 1) : cap;      // (entries behind the capacity are not read)
    if (i > 0 && 32 * i >= cap) {
      p.tmax[i] = p.tmax[i - 1];
      p.cut_tmax[i] = p.cut_tmax[i - 1];
      p.cut_cols[i] = p.cut_cols[i - 1];
      continue;
    }
    const Config c = config_of(rows);
    p.tmax[i] = (uint8_t)((c.tmax + 31) / 32);
    p.cut_tmax[i] = (uint8_t)((c.cut_tmax + 31) / 32);
    const Tiling t = tiling(rows, 32 * p.tmax[i], 32, c.cut_cols, 32 * p.cut_tmax[i], K / BK, n_units);
    const bool fits = c.cut_cols <= n_cols && c.cut_cols < 65536 && t.cut_mt <= n_units && (long long)t.cut_mt * c.cut_cols * mul <= kSplitCounters;
    p.cut_cols[i] = (uint16_t)(fits ? c.cut_cols : 0);
  }
  return p;
}
DevPlan device_plan(TcState* st, const Shape& s, bool pair) {
  const Shape key{pair ? 2 : 1, s.n_feat, s.K, s.cap};
  const auto known = st->plans.find(key);
  if (known != st->plans.end()) return known->second;
  const DevPlan p = make_plan([&](int rows) { return estimate(st, Shape{rows, s.n_feat, s.K, s.cap}, pair ? 2 : 1); }, s.cap, s.n_feat,
                              s.K, pair, st->n_sm);
  if (st->plans.size() >= kMapCacheMax) st->plans.clear();
  st->plans.emplace(key, p);
  return p;
}

// What a launch of M rows (row count on the device, cap > 0: of any number up to cap, M of them expected) runs: the estimate's
// choice, or what the debugging aid forces: single CTAs (64, 128, 256 tokens) or pairs (384: 128, 512: 256 tokens), tiles whole
// or cut over K.  *plan: with the row count on the device and no clusters, the division for every row count.
Config configuration(TcState* st, int M, int n_feat, int K, int cap, DevPlan* plan) {
  const Shape s{M, n_feat, K, cap};
  const Config chosen = choose_config(st, s);
  const int f = st->force_tile;
  if (!f && st->force_s != 1) {
    if (cap && !chosen.cl) *plan = device_plan(st, s, chosen.pair);
    return chosen;
  }
  auto forced = [&](int rows) {
    Config c = f ? Config{f > 256, f == 384 ? 128 : (f == 512 ? 256 : f), 0, 0, 0} : chosen;
    const int gran = c.pair || cap ? 32 : 16, units = c.pair ? st->n_sm / 2 : st->n_sm, mul = c.pair ? 2 : 1;
    const int cols = (n_feat + FT * mul - 1) / (FT * mul);
    int width, mt;
    token_tiles(rows, c.tmax, gran, &width, &mt);
    const int tiles = mt * cols;
    c.cl = 0;
    c.cut_cols = 0;
    c.cut_tmax = c.tmax;
    if (!st->force_s) return c;
    for (int cl = 4; cl >= 2 && st->clusters && !c.cl; --cl)
      if (tiles * cl <= units && cl * 4 <= K / BK && clusters_fit(st, c.pair, cl * mul, tiles)) c.cl = cl;
    // else all columns of less than two waves, or the last one-to-two waves of more
    const int cut = tiles < 2 * units ? cols : cols - (tiles / units - 1) * units / mt;
    if (!c.cl && mt <= units && mt * cut * mul <= kSplitCounters) c.cut_cols = cut;
    return c;
  };
  const Config c = forced(cap ? cap : M);
  const int mul = c.pair ? 2 : 1;
  if (cap && !c.cl)
    *plan = make_plan([&](int rows) {
      Config r = forced(rows);
      if (r.cl) r.cut_cols = (n_feat + FT * mul - 1) / (FT * mul);       // (no clusters in this launch)
      return r;
    }, cap, n_feat, K, c.pair, st->n_sm);
  return c;
}

bool launch_config(TcState* st, const GemmArgs& a, const EpiParams& ep, const Config& c, const DevPlan* plan, cudaStream_t stream) {
  const bool dev = a.m_dev != nullptr;
  if (!configure(st, c.pair, dev)) return false;
  const bool swiglu = a.epi == EPI_SWIGLU;
  const int mul = c.pair ? 2 : 1;
  const uint64_t w_rows = swiglu ? 2ull * a.N : (uint64_t)a.N;
  GemmLaunch g{};
  g.m_cap = a.M;
  g.K = a.K;
  g.n_cols = (int)((w_rows + FT * mul - 1) / (FT * mul));
  const int gran = c.pair || dev ? 32 : 16, n_units = c.pair ? st->n_sm / 2 : st->n_sm;       // scheduling units: CTAs or pairs
  const int KB = a.K / BK;
  g.tmax = (c.tmax + gran - 1) / gran * gran;
  g.tiles = tiling(a.M, g.tmax, gran, dev ? 0 : c.cut_cols, (c.cut_tmax + gran - 1) / gran * gran, KB, n_units);
  const Tiling& t = g.tiles;
  const int n_tiles = t.mt * g.n_cols;
  int units = n_tiles < n_units ? n_tiles : n_units;
  g.cl = c.cl;
  if (c.cl) {
    units = n_tiles * c.cl;   // one cluster per tile; the kernel derives each member's k-blocks from its rank
  } else if (dev) {
    units = n_units;          // (units without work leave at once)
  } else if (t.cut_cols) {
    if (t.cut_mt > n_units || t.cut_mt * t.cut_cols * mul > kSplitCounters) return false;
    const int whole = (g.n_cols - t.cut_cols) * t.mt, used = (t.cut_cols * KB + t.per - 1) / t.per * t.cut_mt;
    units = whole > used ? (whole < n_units ? whole : n_units) : used;
  }
  CUtensorMap mw;              // copies: see cached_map
  XMaps<false> xh;
  XMaps<true> xd;
  const WeightOrder order = swiglu ? kWSwiglu : (a.epi == EPI_QKV_ROPE ? (a.head_dim == 128 ? kWRope128 : kWRope64) : kWPlain);
  if (!get_w_map(st, a.w, w_rows, a.K, order, &mw, &g.w_step3, &g.w_step4)) return false;
  if (dev) {
    for (int i = 0; i < kMaxTok / 32; ++i)
      if (!get_x_map(st, a.x, a.M, a.K, 32 * (i + 1) / mul, &xd.wide[i])) return false;
    if (plan) xd.plan = *plan;
  } else if (!get_x_map(st, a.x, a.M, a.K, t.width / mul, &xh.whole) || !get_x_map(st, a.x, a.M, a.K, t.cut_width / mul, &xh.cut)) {
    return false;
  }
  g.split_ws = st->split_ws;
  g.split_counters = st->split_counters;
  g.m_dev = a.m_dev;
  g.m_dev_wait = a.m_dev_settled ? 0 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(mul * units);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (c.pair || c.cl) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = mul * (c.cl ? c.cl : 1);
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr].val.clusterDim.z = 1;
    ++n_attr;
  }
  // programmatic dependent launch, except inside a stream capture (see launch_pdl)
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  return (dev ? cudaLaunchKernelEx(&cfg, kernel_dev(c.pair), mw, xd, g, ep)
              : cudaLaunchKernelEx(&cfg, kernel_host(c.pair), mw, xh, g, ep)) == cudaSuccess;
}

}  // namespace

void* tc_state_create(int n_sm) {
  TcState* st = new TcState();
  st->n_sm = n_sm;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || !fn) {
    delete st;
    return nullptr;
  }
  st->encode = reinterpret_cast<EncodeTiledFn>(fn);
  if (cudaMalloc(reinterpret_cast<void**>(&st->split_ws), kSplitWsBytes) != cudaSuccess ||
      cudaMalloc(reinterpret_cast<void**>(&st->split_counters), kSplitCounters * sizeof(int)) != cudaSuccess ||
      cudaMemset(st->split_counters, 0, kSplitCounters * sizeof(int)) != cudaSuccess) {
    if (st->split_ws) cudaFree(st->split_ws);
    if (st->split_counters) cudaFree(st->split_counters);
    delete st;
    return nullptr;
  }
  return st;
}

void tc_state_force(void* s, int tile, int stream_k) {
  TcState* st = static_cast<TcState*>(s);
  if (!st) return;
  st->force_tile = tile;
  st->force_s = stream_k;
  st->clusters = stream_k != 2;     // 2: cut tiles always go through the partial-tile workspace
  st->configs.clear();
  st->plans.clear();
}

// debugging aid: what a launch of `rows` rows runs (cap > 0: row count on the device, `hint` rows expected and at most cap)
bool tc_state_plan(void* s, int rows, int n_feat, int K, int hint, int cap, int (&out)[8]) {
  TcState* st = static_cast<TcState*>(s);
  if (!st || rows <= 0 || n_feat <= 0 || n_feat % 16 || K <= 0 || K % BK || (cap && (rows > cap || hint <= 0 || hint > cap))) return false;
  DevPlan plan;
  const Config c = configuration(st, cap ? hint : rows, n_feat, K, cap, &plan);
  const int mul = c.pair ? 2 : 1, gran = c.pair || cap ? 32 : 16, n_units = st->n_sm / mul;
  const Tiling t = cap && !c.cl ? planned(plan, rows, K / BK, n_units)
                                : tiling(rows, (c.tmax + gran - 1) / gran * gran, gran, cap ? 0 : c.cut_cols, (c.cut_tmax + gran - 1) / gran * gran, K / BK, n_units);
  const int got[8] = {c.pair, t.width, t.mt, c.cl, (n_feat + FT * mul - 1) / (FT * mul), t.cut_cols, t.cut_width, t.per};
  memcpy(out, got, sizeof(got));
  return true;
}

void tc_state_reset(void* s, cudaStream_t stream) {
  TcState* st = static_cast<TcState*>(s);
  if (st && st->split_counters) cudaMemsetAsync(st->split_counters, 0, kSplitCounters * sizeof(int), stream);
}

// Host-only check of the map cache: n_keys distinct keys go through it three at a time, the way a launch takes its
// maps, with an encoder that writes the key into the map; every map handed out must still carry its own key after
// the later lookups of the same launch (which may have emptied the cache).  Returns the number of wrong maps.
int tc_map_cache_selftest(int n_keys, int* evictions) {
  TcState st;
  auto fake = [](const MapKey& k) {
    return [k](CUtensorMap* m) {
      memset(m, 0, sizeof(*m));
      memcpy(m, &k, sizeof(k));
      return true;
    };
  };
  auto key_of = [](int i) { return MapKey{reinterpret_cast<const void*>(static_cast<uintptr_t>(4096) * (i + 1)), (uint64_t)i, 64, 128}; };
  int bad = 0;
  for (int i = 0; i + 2 < n_keys; i += 3) {
    CUtensorMap m[3];
    for (int j = 0; j < 3; ++j)
      if (!cached_map(&st, key_of(i + j), &m[j], fake(key_of(i + j)))) ++bad;
    auto carries = [](const CUtensorMap& m, const MapKey& k) {   // (field by field: the key has padding bytes)
      MapKey got;
      memcpy(&got, &m, sizeof(got));
      return got == k;
    };
    for (int j = 0; j < 3; ++j)
      if (!carries(m[j], key_of(i + j))) ++bad;
    // an old key again: a hit, or a miss that re-encodes; either way the right map
    CUtensorMap again;
    const MapKey k0 = key_of(i / 2);
    if (!cached_map(&st, k0, &again, fake(k0)) || !carries(again, k0)) ++bad;
  }
  if (st.maps.size() > kMapCacheMax) ++bad;
  if (evictions) *evictions = (int)st.evictions;
  return bad;
}

void tc_state_destroy(void* s) {
  TcState* st = static_cast<TcState*>(s);
  if (!st) return;
  if (st->split_ws) cudaFree(st->split_ws);
  if (st->split_counters) cudaFree(st->split_counters);
  delete st;
}

bool launch_gemm_tc(const GemmArgs& a, void* tc_state, int* status, cudaStream_t stream, int* ss_slots_out) {
  TcState* st = static_cast<TcState*>(tc_state);
  if (!st || a.M <= 0 || a.K % BK || a.N % 16) return false;
  if ((reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.w)) & 15) return false;
  // (bf16 rows leave in pieces of 16 bytes, fp32 ones element by element)
  if (reinterpret_cast<uintptr_t>(a.out) & (a.epi == EPI_PLAIN_F32 || a.epi == EPI_RESIDUAL_NORM ? 3 : 15)) return false;
  if (a.epi == EPI_RESIDUAL || (a.epi == EPI_RESIDUAL_NORM && (!a.x_out || !a.gain || !a.ss_out))) return false;
  if (a.epi == EPI_SWIGLU && a.N % 64) return false;
  if (((int64_t)a.N * 2 / FT + 2) * (a.K / BK) > (1 << 30)) return false;      // the line of k-blocks is counted in int
  if (a.epi == EPI_QKV_ROPE && (a.N % 128 || (a.head_dim != 64 && a.head_dim != 128))) return false;
  EpiParams ep;
  ep.epi = a.epi;
  ep.out = a.out;
  ep.x_out = static_cast<__nv_bfloat16*>(a.x_out);
  ep.M = a.M;
  ep.N = a.N;
  ep.tok_slot = a.tok_slot;
  ep.rope_cs = static_cast<const float2*>(a.rope_cs);
  ep.kv_pool = static_cast<__nv_bfloat16*>(a.kv_pool);
  ep.n_pages = a.n_pages;
  ep.layer = a.layer;
  ep.n_q = a.n_q;
  ep.n_kv = a.n_kv;
  ep.head_dim = a.head_dim;
  ep.status = status;
  ep.ss_in = a.ss_in;
  ep.ss_slots = a.ss_slots;
  ep.ss_stride = a.ss_stride;
  ep.norm_inv_n = 1.f / (float)a.K;
  ep.norm_eps = a.norm_eps;
  ep.gain = static_cast<const __nv_bfloat16*>(a.gain);
  ep.ss_out = a.ss_out;
  const int n_feat = a.epi == EPI_SWIGLU ? 2 * a.N : a.N;
  // (device-resident rounds: the configuration is chosen for the caller's hint of the row count, the launch covers the capacity)
  const int Mc = (a.m_dev && a.m_hint > 0 && a.m_hint < a.M) ? a.m_hint : a.M;
  DevPlan plan;
  const Config c = configuration(st, Mc, n_feat, a.K, a.m_dev ? a.M : 0, &plan);
  if (ss_slots_out) *ss_slots_out = (a.N + FT - 1) / FT;
  return launch_config(st, a, ep, c, a.m_dev && !c.cl ? &plan : nullptr, stream);
}

}  // namespace recg
