// Ragged layout (per-token arrays + attention work list), embedding gather, RMSNorm, KV import/export.
#include "common.cuh"
#include "kernels.h"

namespace recg {

namespace {

__device__ __forceinline__ int upper_request(const int* cu, int n_req, int t) {
  // largest r with cu[r] <= t  (cu is an exclusive prefix sum with cu[n_req] = total)
  int lo = 0, hi = n_req;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (cu[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// CTA 0 builds the attention work list, every further CTA the per-token arrays of kLayoutThreads tokens.  In a forward pass the
// embedding kernel, which does not need the work list and runs beside this kernel's one CTA, fills those arrays
// (a step of a 2-layer model of width 256, three requests: 91.7 us one behind the other, 87.9 us side by side).
//
// Attention work list.  A request with n new tokens has ceil(n / tok_per_tile) row tiles per kv head.  Row tiles
// 2 j and 2 j + 1 of a kv head are "siblings": they read the same K/V.  A tile reads the 64-token KV blocks up to the last
// position that one of its rows may see (verify rows are causal, so the early tiles of a long chunk of prompt need fewer
// blocks than the late ones; siblings share the range of the later one).  Two lines of KV blocks are built, every tile
// preceded by virtual blocks that stand for the fixed cost of starting an item (fetching Q, refilling and draining the
// pipeline; kItemCostPair, kItemCostSingle, in blocks: the blocks of a pair take less time, every second one comes from L2.
// Attention of a layer with 4 for both / 6 and 4 / 8 and 4: two chunks of 1000 prompt tokens 158 / 143 / 143 us, eight requests
// with two branches each 79.9 / 73.9 / 72.6, sixteen requests 66.7 / 66.7 / 68.0; 6 for both: the last one 67.5):
//   line A holds one segment per sibling PAIR and is cut into equal contiguous ranges, one per pair of CTAs
//          (2 p, 2 p + 1): the even CTA works on the first sibling and the odd CTA on the second sibling of the SAME
//          block ranges, at the same time, so that the second reader of a K/V block finds it in L2;
//   line B holds the tiles without a sibling and is cut into equal ranges, one per CTA.
// The CTAs are divided between the two lines in proportion to their work (line A: the first 2 n_pairs_a CTAs), so
// that every CTA walks ONE range and all carry about the same load.  Each piece that holds real blocks is an item;
// a tile whose blocks are cut by range boundaries gets one partial slot per piece.
// Small work lists are not cut at all (`whole`, decided on the host from the same lengths): every tile is one item of a CTA of
// its own, and no combine kernel follows.
// Items: [line A, first siblings | line A, second siblings (same order) | line B]; cta_off holds, per CTA, two
// index ranges it walks one after the other (the second one is empty in this division).
//
// The kernel is a chain of dependent steps on little data, so it is bound by latency: one thread handles one segment (all
// per-request sums are block-wide scans), and descriptors are read into shared memory once.  Measured before, with one
// thread per request and sums over the requests in one thread: 5.6 us for one request, 13 us with its attention work list,
// 58 us for 8448 rows of 256 requests.
constexpr int kItemCostPair = 6, kItemCostSingle = 4;
constexpr int kLayoutThreads = 1024;
constexpr int kWholeBlocks = 5;

// exclusive prefix sums over the threads of the CTA, and the totals; `carry` scratch: 3 x 33 ints of shared memory
struct Scan3 { int a, b, c; };
__device__ __forceinline__ Scan3 block_scan(Scan3 x, Scan3* total, int (*sm)[33]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Scan3 s = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ya = __shfl_up_sync(0xffffffffu, s.a, o), yb = __shfl_up_sync(0xffffffffu, s.b, o), yc = __shfl_up_sync(0xffffffffu, s.c, o);
    if (lane >= o) { s.a += ya; s.b += yb; s.c += yc; }
  }
  if (lane == 31) { sm[0][warp] = s.a; sm[1][warp] = s.b; sm[2][warp] = s.c; }
  __syncthreads();
  if (warp < 3) {                       // warp k scans the warps' sums of component k
    const int v = sm[warp][lane];
    int t = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    sm[warp][lane] = t - v;
    if (lane == 31) sm[warp][32] = t;
  }
  __syncthreads();
  s.a += sm[0][warp] - x.a;
  s.b += sm[1][warp] - x.b;
  s.c += sm[2][warp] - x.c;
  *total = Scan3{sm[0][32], sm[1][32], sm[2][32]};
  __syncthreads();                      // the scratch may be reused
  return s;
}

struct TokenPos { int id, pos; };
__device__ __forceinline__ TokenPos layout_token(const BatchLayout& bl, int r, int j, int mask_id, int t, int64_t n_pages, int* status) {
  const int L = bl.ctx_len[r], v = bl.verify_len[r], b = bl.block_size[r];
  const int idx = L + j;   // cache position of the token's K/V
  int pos, id, climit, lo, hi;
  if (j < v) {             // verifier: causal
    pos = idx; id = bl.verify_tokens[bl.cu_ver[r] + j]; climit = idx; lo = 0; hi = 0;
  } else if (j < v + b) {  // continuation block: the whole prefix and the block
    pos = idx; id = mask_id; climit = L + v - 1; lo = L + v; hi = L + v + b;
  } else {                 // correction branch k: replacement token, then its mask tokens
    const int* cr = bl.corr + 6 * r;
    const int span = 1 + cr[1], jj = j - v - b, k = jj / span, q = jj - k * span;
    const int i = cr[2 + k], first = L + v + b + k * span;
    pos = L + i + q;
    id = q == 0 ? cr[4 + k] : mask_id;
    climit = L + i - 1;
    lo = first;
    hi = q == 0 ? first + 1 : first + span;
  }
  bl.tok_req[t] = r;
  bl.tok_pos[t] = pos;
  bl.tok_id[t] = id;
  bl.tok_climit[t] = climit;
  bl.tok_lo[t] = lo;
  bl.tok_hi[t] = hi;
  const int page = bl.page_table[(size_t)r * bl.pt_stride + idx / kPageSize];
  int slot = -1;
  if (page < 0 || page >= n_pages) set_status(status, DEV_BAD_INDEX);
  else slot = page * kPageSize + idx % kPageSize;
  bl.tok_slot[t] = slot;
  return TokenPos{id, pos};
}

__global__ void __launch_bounds__(kLayoutThreads) layout_kernel(BatchLayout bl, int n_kv, int mask_id, int tok_per_tile,
                                                                int n_ctas, int whole, int64_t n_pages, int* status, int* desc_dev,
                                                                const __grid_constant__ SmallDesc desc) {
  extern __shared__ int sm[];
  const int C = bl.n_req;
  const int max_pairs = n_ctas / 2;
  int* cu_tok = sm;                      // [C + 1] rows of the batch in front of request r
  int* seg_a = sm + (C + 1);             // [C + 1] line-A segments in front of request r
  int* seg_b = sm + 2 * (C + 1);         // [C + 1] line-B segments
  int* ctx = sm + 3 * (C + 1);           // [C]
  int* vis = sm + 4 * (C + 1);           // [C] verify rows (causal) of request r
  int* a_off = sm + 5 * (C + 1);         // [max_pairs + 1] first line-A piece of every CTA pair
  int* b_off = a_off + (max_pairs + 1);  // [n_ctas + 1]  first line-B piece of every line-B CTA
  __shared__ int scratch[3][33];
  __shared__ long long s_cost[2];
  const int tid = threadIdx.x;
  griddep_wait();   // the previous step's kernels may still be reading the arrays this kernel rewrites
  griddep_launch(); // (after the wait: an embedding kernel behind this one does not wait itself)
  if (desc.n) {     // (no copy went ahead of this kernel: it reads the descriptor from its parameters and leaves it for the others)
    bl.rebase(desc_dev, desc.v);
    if (blockIdx.x == 0)
      for (int i = tid; i < desc.n; i += kLayoutThreads) desc_dev[i] = desc.v[i];
  }
  for (int r = tid; r <= C; r += kLayoutThreads) cu_tok[r] = bl.cu_tok[r];

  // ---- per-token arrays ----
  if (blockIdx.x > 0) {
    __syncthreads();
    const int t = (blockIdx.x - 1) * kLayoutThreads + tid;
    if (t < cu_tok[C]) {
      const int r = upper_request(cu_tok, C, t);
      layout_token(bl, r, t - cu_tok[r], mask_id, t, n_pages, status);
    }
    return;
  }

  // ---- attention work list ----
  for (int r = tid; r < C; r += kLayoutThreads) {
    ctx[r] = bl.ctx_len[r];
    vis[r] = bl.verify_len[r];
  }
  if (tid < 2) s_cost[tid] = 0;
  __syncthreads();
  Scan3 carry{0, 0, 0};
  for (int r0 = 0; r0 < C; r0 += kLayoutThreads) {
    const int r = r0 + tid;
    const int rt = r < C ? (cu_tok[r + 1] - cu_tok[r] + tok_per_tile - 1) / tok_per_tile : 0;
    Scan3 tot;
    const Scan3 e = block_scan(Scan3{n_kv * (rt / 2), n_kv * (rt & 1), 0}, &tot, scratch);
    if (r < C) {
      seg_a[r] = carry.a + e.a;
      seg_b[r] = carry.b + e.b;
    }
    carry.a += tot.a;
    carry.b += tot.b;
  }
  const int n_seg_a = carry.a, n_seg_b = carry.b;
  if (tid == 0) {
    seg_a[C] = n_seg_a;
    seg_b[C] = n_seg_b;
  }
  __syncthreads();
  // segment s of a line: its request, kv head, (first) tile and KV blocks
  struct Seg { int r, kvh, tile, nb; };
  auto segment = [&](const int* first, int s, bool pair) {
    Seg g;
    g.r = upper_request(first, C, s);
    const int n = cu_tok[g.r + 1] - cu_tok[g.r], rt = (n + tok_per_tile - 1) / tok_per_tile;
    const int per_head = pair ? rt / 2 : 1, i = s - first[g.r];
    g.kvh = i / per_head;
    g.tile = pair ? 2 * (i - g.kvh * per_head) : rt - 1;
    // the last of the segment's rows: causal up to itself if it is a verify row, else anything up to the request's end
    const int last_row = min(n, (g.tile + (pair ? 2 : 1)) * tok_per_tile);
    g.nb = (ctx[g.r] + (last_row <= vis[g.r] ? last_row : n) + 63) / 64;
    return g;
  };
  for (int line = 0; line < 2; ++line) {
    const int n_seg = line ? n_seg_b : n_seg_a;
    for (int s0 = 0; s0 < n_seg; s0 += kLayoutThreads) {
      const int s = s0 + tid;
      int cost = 0;
      if (s < n_seg) cost = line ? segment(seg_b, s, false).nb + kItemCostSingle : segment(seg_a, s, true).nb + kItemCostPair;
      cost = __reduce_add_sync(0xffffffffu, cost);
      if ((tid & 31) == 0 && cost) atomicAdd(reinterpret_cast<unsigned long long*>(&s_cost[line]), (unsigned long long)cost);
    }
  }
  __syncthreads();
  const long long wa = s_cost[0], wb = s_cost[1];
  const bool too_long = wa > 0x3fffffff || wb > 0x3fffffff;      // far beyond any pool; the arithmetic below is in int
  // CTAs for line A in proportion to its CTA time (two CTAs work on every unit of it)
  int pairs_a = (2 * wa + wb) > 0 ? (int)(0.5 * n_ctas * (2.0 * wa) / (2.0 * wa + wb) + 0.5) : 0;
  if (wa > 0 && pairs_a < 1) pairs_a = 1;
  if (pairs_a > max_pairs) pairs_a = max_pairs;
  if (wb > 0 && n_ctas - 2 * pairs_a < 1) pairs_a = (n_ctas - 1) / 2;
  if (wa == 0) pairs_a = 0;
  if (whole) pairs_a = n_seg_a;            // (2 n_seg_a + n_seg_b <= n_ctas)
  const int n_ctas_b = n_ctas - 2 * pairs_a;
  const int per_a = pairs_a > 0 && wa > 0 ? (int)((wa + pairs_a - 1) / pairs_a) : 0x3fffffff;
  const int per_b = n_ctas_b > 0 && wb > 0 ? (int)((wb + n_ctas_b - 1) / n_ctas_b) : 0x3fffffff;

  // Lines A, then B: offsets by scans over the segments, then every thread emits the pieces of its segment.
  // The tiles that are cut are listed one behind the other for the combine kernel: with all tiles in the list it took 23 us per
  // layer of 128 requests, 27 dependent reads of entries of which one in ten was cut.
  int n_pieces_a = 0, n_pieces_b = 0, parts = 0, n_cut = 0;
  bool overflow = too_long;
  // pass 0 counts line A's pieces (the second siblings' items lie behind all first ones), passes 1 and 2 emit
  for (int pass = too_long ? 3 : 0; pass < 3; ++pass) {
    const bool pair = pass < 2;
    const int item_cost = pair ? kItemCostPair : kItemCostSingle;
    const int n_seg = pair ? n_seg_a : n_seg_b, per = pair ? per_a : per_b;
    const int* first = pair ? seg_a : seg_b;
    int* owner_off = pair ? a_off : b_off;
    const int n_owners = pair ? max_pairs : n_ctas;
    int off = 0, pieces = 0;             // cost units and pieces of the line so far
    for (int s0 = 0; s0 < n_seg; s0 += kLayoutThreads) {
      const int s = s0 + tid;
      Seg g{0, 0, 0, 0};
      if (s < n_seg) g = segment(first, s, pair);
      Scan3 tot;
      const Scan3 e1 = block_scan(Scan3{s < n_seg ? g.nb + item_cost : 0, 0, 0}, &tot, scratch);
      const int g0 = off + e1.a + item_cost;              // cost range of the real blocks: [g0, g0 + nb)
      off += tot.a;
      const int c_first = whole ? s : g0 / per, c_last = whole ? s : (g0 + g.nb - 1) / per;
      const int np = s < n_seg ? c_last - c_first + 1 : 0;
      const int cut_tiles = np > 1 ? (pair ? 2 : 1) : 0;
      const Scan3 e2 = block_scan(Scan3{np, cut_tiles * np, cut_tiles}, &tot, scratch);
      const int item0 = pieces + e2.a, cut0 = n_cut + e2.c;
      int part = parts + e2.b;
      pieces += tot.a;
      if (pass > 0) {
        parts += tot.b;
        n_cut += tot.c;
      }
      if (pass == 0 || s >= n_seg) continue;
      // first piece of every owner: an owner without pieces starts where the next one does
      const int c_prev = s == 0 || whole ? s - 1 : (g0 - item_cost - 1) / per;     // owner of the last block of the segment before
      for (int c = c_prev + 1; c <= c_last && c <= n_owners; ++c) owner_off[c] = c <= c_first ? item0 : item0 + (c - c_first);
      if (s == n_seg - 1)
        for (int c = c_last + 1; c <= n_owners; ++c) owner_off[c] = item0 + np;
      const int n = cu_tok[g.r + 1] - cu_tok[g.r], kv_len = ctx[g.r] + n;
      for (int sib = 0; sib < (pair ? 2 : 1); ++sib) {
        AttnTile tl;
        tl.part_begin = part;
        tl.n_parts = np;
        tl.tok0 = cu_tok[g.r] + (g.tile + sib) * tok_per_tile;
        tl.ntok = min(tok_per_tile, n - (g.tile + sib) * tok_per_tile);
        tl.kv_head = g.kvh;
        if (np > 1) bl.tiles[cut0 + sib] = tl;
        const int at = pair ? (sib ? n_pieces_a : 0) + item0 : 2 * n_pieces_a + item0;
        for (int c = c_first; c <= c_last; ++c) {
          AttnItem a;
          a.req = g.r;
          a.kv_head = g.kvh;
          a.tok0 = tl.tok0;
          a.ntok = tl.ntok;
          a.blk_begin = whole ? 0 : max(g0, c * per) - g0;
          a.blk_end = whole ? g.nb : min(g0 + g.nb, (c + 1) * per) - g0;
          a.part = np > 1 ? part++ : -1;
          a.kv_len = kv_len;
          if (at + (c - c_first) < bl.max_items && a.part < bl.max_parts) bl.items[at + (c - c_first)] = a;
        }
      }
    }
    if (pass == 0) n_pieces_a = pieces;
    if (pass == 2) n_pieces_b = pieces;
    if (pass > 0 && n_seg == 0)
      for (int c = tid; c <= n_owners; c += kLayoutThreads) owner_off[c] = 0;
  }
  overflow = overflow || 2 * n_pieces_a + n_pieces_b > bl.max_items || parts > bl.max_parts;
  if (tid == 0) {
    if (overflow) set_status(status, DEV_BAD_INDEX);
    bl.counts[0] = overflow ? 0 : 2 * n_pieces_a + n_pieces_b;
    bl.counts[1] = overflow ? 0 : n_cut;
    bl.counts[2] = per_b;
    bl.counts[3] = per_a;
  }
  __syncthreads();
  // the ranges of item indices every CTA walks: a CTA of line A its pair's pieces (first or second siblings), a CTA of
  // line B its own pieces
  for (int c = tid; c < n_ctas; c += kLayoutThreads) {
    int a0 = 0, a1 = 0, b0 = 0, b1 = 0;
    if (!overflow) {
      if (c < 2 * pairs_a) {
        const int p = c >> 1;
        a0 = ((c & 1) ? n_pieces_a : 0) + a_off[p];
        a1 = ((c & 1) ? n_pieces_a : 0) + a_off[p + 1];
      } else if (c - 2 * pairs_a < n_ctas_b) {
        b0 = 2 * n_pieces_a + b_off[c - 2 * pairs_a];
        b1 = 2 * n_pieces_a + b_off[c - 2 * pairs_a + 1];
      }
    }
    *reinterpret_cast<int4*>(bl.cta_off + 4 * c) = make_int4(a0, a1, b0, b1);
  }
}

// One CTA per row; fp32 in, bf16 out.  hidden a multiple of 4.  The row is read once and kept in registers
// when it fits (hidden <= 256 threads x kRegVecs float4), otherwise it is read a second time.
constexpr int kRegVecs = 8;
__device__ __forceinline__ float row_sum(float ss) {     // over the 256 threads of the CTA, the same bits in every thread
  __shared__ float red[8];
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) tot += red[i];
  return tot;
}
// four elements of x = bf16(h * rstd * gain); rstd = 1: x = bf16(h * gain)
__device__ __forceinline__ uint2 norm_vec(const float4& t, float rstd, const uint2* __restrict__ gain, int i) {
  const uint2 gv = __ldg(gain + i);
  const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gv.x));
  const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gv.y));
  uint2 o;
  o.x = pack_bf16(t.x * rstd * g0.x, t.y * rstd * g0.y);
  o.y = pack_bf16(t.z * rstd * g1.x, t.w * rstd * g1.y);
  return o;
}

// One CTA per token: the token's entries of the per-token arrays, the residual row h = embed[tok_id], the rotary table's column
// of the token, and the input of the first
// projection: x = rmsnorm(h) * gain, or (ss given: folded RMSNorm) x = h * gain and the row's sum of squares.  All of it
// follows from the token alone and each part by itself is one launch latency (2.5 us each at any size up to a few hundred
// rows), so one launch does the three.
__global__ void __launch_bounds__(256) embed_kernel(BatchLayout bl, int mask_id, int64_t n_pages, int* status,
                                                    const __nv_bfloat16* __restrict__ embed, float* __restrict__ h, int hidden,
                                                    int vocab, const __nv_bfloat16* __restrict__ gain,
                                                    __nv_bfloat16* __restrict__ x, float* __restrict__ ss, float eps,
                                                    float2* __restrict__ cs, int half, double log_base,
                                                    const int* desc_dev, const __grid_constant__ SmallDesc desc) {
  __shared__ TokenPos s_token;
  griddep_launch();      // (no wait: the layout kernel in front signals when the kernels before it are done, and nothing of it is needed)
  if (desc.n) bl.rebase(desc_dev, desc.v);
  const int t = blockIdx.x;
  const auto end = [&] { if (t == 0) griddep_wait(); };    // this grid must not count as complete before the layout kernel is
  if (bl.dyn && t >= bl.dyn[0]) return end();              // (the grid was sized for the capacity)
  int r = 0;                               // requests whose successor does not start behind this token
  for (int r0 = 1; r0 < bl.n_req; r0 += 256) {
    const int i = r0 + threadIdx.x;
    r += __syncthreads_count(i < bl.n_req && bl.cu_tok[i] <= t);
  }
  if (threadIdx.x == 0) s_token = layout_token(bl, r, t - bl.cu_tok[r], mask_id, t, n_pages, status);
  __syncthreads();
  int id = s_token.id;
  const int pos = s_token.pos;
  id = id < 0 ? 0 : (id >= vocab ? vocab - 1 : id);
  const uint2* src = reinterpret_cast<const uint2*>(embed + (size_t)id * hidden);
  float4* dst = reinterpret_cast<float4*>(h + (size_t)t * hidden);
  const int nvec = hidden / 4;
  auto load = [&](int i) {
    const uint2 u = __ldg(src + i);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
  };
  const bool in_regs = nvec <= 256 * kRegVecs;
  float4 v[kRegVecs];
  float sq = 0.f;
  if (in_regs) {
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) {
      const int i = threadIdx.x + u * 256;
      v[u] = i < nvec ? load(i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) {
      const int i = threadIdx.x + u * 256;
      if (i < nvec) dst[i] = v[u];
      sq += v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
    }
  } else {
    for (int i = threadIdx.x; i < nvec; i += 256) {
      const float4 f = load(i);
      dst[i] = f;
      sq += f.x * f.x + f.y * f.y + f.z * f.z + f.w * f.w;
    }
  }
  // rotary factors [token][half]: in the projection epilogue a lane has one frequency, so a warp reads a token's 16
  // consecutive frequencies in one 128-byte request.  Angles in double.
  for (int i = threadIdx.x; i < half; i += 256) {
    const double ang = (double)pos * exp(-log_base * (double)i / (double)half);  // pos * base^(-2i/d)
    cs[(size_t)t * half + i] = make_float2((float)cos(ang), (float)sin(ang));
  }
  const float tot = row_sum(sq);
  const float rstd = ss ? 1.f : rsqrtf(tot / hidden + eps);
  if (ss && threadIdx.x == 0) ss[t] = tot;
  uint2* xo = reinterpret_cast<uint2*>(x + (size_t)t * hidden);
  const uint2* gg = reinterpret_cast<const uint2*>(gain);
  if (in_regs) {
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) {
      const int i = threadIdx.x + u * 256;
      if (i < nvec) xo[i] = norm_vec(v[u], rstd, gg, i);
    }
  } else {
    for (int i = threadIdx.x; i < nvec; i += 256) xo[i] = norm_vec(load(i), rstd, gg, i);
  }
  end();
}

__global__ void __launch_bounds__(256) rmsnorm_kernel(const float* __restrict__ h, const __nv_bfloat16* __restrict__ g,
                                                      __nv_bfloat16* __restrict__ x, int hidden, float eps,
                                                      const int* __restrict__ rows_dev) {
  griddep_launch();
  griddep_wait();
  const int row = blockIdx.x;
  if (rows_dev && row >= rows_dev[0]) return;
  const int nvec = hidden / 4;
  const float4* src = reinterpret_cast<const float4*>(h + (size_t)row * hidden);
  const bool in_regs = nvec <= 256 * kRegVecs;
  float4 v[kRegVecs];
  float ss = 0.f;
  if (in_regs) {
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) {
      const int i = threadIdx.x + u * 256;
      v[u] = i < nvec ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) ss += v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
  } else {
    for (int i = threadIdx.x; i < nvec; i += 256) {
      const float4 t = src[i];
      ss += t.x * t.x + t.y * t.y + t.z * t.z + t.w * t.w;
    }
  }
  const float rstd = rsqrtf(row_sum(ss) / hidden + eps);
  uint2* dst = reinterpret_cast<uint2*>(x + (size_t)row * hidden);
  const uint2* gg = reinterpret_cast<const uint2*>(g);
  if (in_regs) {
#pragma unroll
    for (int u = 0; u < kRegVecs; ++u) {
      const int i = threadIdx.x + u * 256;
      if (i < nvec) dst[i] = norm_vec(v[u], rstd, gg, i);
    }
  } else {
    for (int i = threadIdx.x; i < nvec; i += 256) dst[i] = norm_vec(src[i], rstd, gg, i);
  }
}

// Moves logical K/V rows [n_pos, n_kv, head_dim] into or out of the pool.  Nothing but bytes: bound by HBM.  A thread takes
// kKvIoUnroll 16-byte chunks of K and the same of V, all loads in flight before the first store; consecutive threads take
// consecutive chunks, so the logical side is one contiguous stream and the pool side whole 128-byte rows of the swizzled
// tiles.  The page ids come with the launch (constant bank: a warp covers few positions), so no upload goes ahead of it.
// Calls for one layer after the other follow on each other's heels: the addresses are ready before the wait for the kernel in
// front, and two chunks a thread (32 registers: eight CTAs per SM) let more of the next kernel's CTAs move in early than four (48).
// 8000 positions of 8 heads x 128 (66 MB in and out), write / read of a layer: four chunks, addresses behind the wait 13.0 /
// 12.5 us, ahead of it 12.5 / 11.8, two chunks 11.5 / 11.6, eight 12.7 / 12.7.  Up to 4001 positions the host's calls bound it
// (8.1 us; 22.5 with one 16-thread CTA per (position, head) and a page row copied ahead of it).
constexpr int kKvIoPages = 896;       // page ids per launch: 3.5 of the 4 KB of kernel parameters
constexpr int kKvIoPagesFew = 256;    // up to 4081 positions: fewer parameters for the host to copy, 8.5 -> 8.1 us a call (16 positions)
constexpr int kKvIoThreads = 256, kKvIoUnroll = 2;
template <int N>
struct KvIoPages {
  int first;                          // logical page of ids[0]
  int ids[N];
};
template <bool WRITE, int N>
__global__ void __launch_bounds__(kKvIoThreads) kv_io_kernel(__nv_bfloat16* pool, int64_t n_pages, int layer, int n_kv, int log2_cpr,
                                                             const __grid_constant__ KvIoPages<N> pages, int pos0, int n_pos,
                                                             uint4* __restrict__ k, uint4* __restrict__ v) {
  griddep_launch();
  const int cpr = 1 << log2_cpr, head_dim = cpr * 8;          // 16-byte chunks per row
  const int total = (n_pos * n_kv) << log2_cpr;
  const int base = blockIdx.x * (kKvIoThreads * kKvIoUnroll) + threadIdx.x;
  uint4* at[kKvIoUnroll];
  uint4 a[kKvIoUnroll], b[kKvIoUnroll];
  const int v_off = (int)kv_tile_elems(head_dim) / 8;
#pragma unroll
  for (int u = 0; u < kKvIoUnroll; ++u) {
    const int i = base + u * kKvIoThreads;
    at[u] = nullptr;
    if (i >= total) continue;
    const int row = i >> log2_cpr, c = i & (cpr - 1);
    const int p = row / n_kv, hk = row - p * n_kv, pos = pos0 + p;
    const int page = pages.ids[pos / kPageSize - pages.first];
    at[u] = reinterpret_cast<uint4*>(pool + kv_tile_base(n_pages, n_kv, head_dim, layer, page, hk) +
                                     kv_tile_offset(pos % kPageSize, c * 8, head_dim));
  }
  griddep_wait();
#pragma unroll
  for (int u = 0; u < kKvIoUnroll; ++u) {
    if (!at[u]) continue;
    const int i = base + u * kKvIoThreads;
    a[u] = WRITE ? k[i] : at[u][0];
    b[u] = WRITE ? v[i] : at[u][v_off];
  }
#pragma unroll
  for (int u = 0; u < kKvIoUnroll; ++u) {
    if (!at[u]) continue;
    const int i = base + u * kKvIoThreads;
    if (WRITE) {
      at[u][0] = a[u];
      at[u][v_off] = b[u];
    } else {
      k[i] = a[u];
      v[i] = b[u];
    }
  }
}

// one launch: positions [pos0, pos0 + n), whose pages are page_row[first], ... (at most N)
template <int N>
void kv_io_part(bool write, __nv_bfloat16* pool, int64_t n_pages, int layer, const Dims& dm, const int* page_row, int pos0, int n,
                uint4* k, uint4* v, cudaStream_t st) {
  const int log2_cpr = dm.head_dim == 128 ? 4 : 3;
  KvIoPages<N> pg;
  pg.first = pos0 / kPageSize;
  const int last = (pos0 + n - 1) / kPageSize;
  for (int i = pg.first; i <= last; ++i) pg.ids[i - pg.first] = page_row[i];
  constexpr size_t kPer = (size_t)kKvIoThreads * kKvIoUnroll;
  const dim3 grid((unsigned)((((size_t)n * dm.n_kv << log2_cpr) + kPer - 1) / kPer));
  launch_pdl(write ? kv_io_kernel<true, N> : kv_io_kernel<false, N>, grid, dim3(kKvIoThreads), 0, st, pool, n_pages, layer, dm.n_kv,
             log2_cpr, pg, pos0, n, k, v);
}

}  // namespace

size_t layout_smem_bytes(int n_req, int n_ctas) {
  return (5 * (size_t)(n_req + 1) + (size_t)(n_ctas / 2 + 1) + (size_t)(n_ctas + 1)) * sizeof(int);
}

// Whole tiles against work cut evenly.  A tile's 64-token block takes about .5 us of its CTA; cutting costs the write of the
// partial results, the combine kernel and its boundary, about 2.5 us.  Measured (one request, 16 rows, a layer's attention): 64
// tokens of context 6.3 us whole, 8.8 cut; 256 tokens 8.7 and 9.1; 512 tokens 10.8 and 10.3; with head_dim 64 4.3 and 5.8, 5.8
// and 6.0, 7.8 and 6.4.
bool attention_whole_tiles(int n_req, const int* ctx_len, const int* rows, int n_kv, int tok_per_tile, int n_ctas) {
  long long tiles = 0, cost = 0;
  int longest = 0;
  for (int r = 0; r < n_req; ++r) {
    const int rt = (rows[r] + tok_per_tile - 1) / tok_per_tile, nb = (ctx_len[r] + rows[r] + 63) / 64;
    tiles += (long long)n_kv * rt;
    cost += (long long)n_kv * (rt * nb + (rt & ~1) * kItemCostPair + (rt & 1) * kItemCostSingle);
    if (nb > longest) longest = nb;
  }
  return tiles <= n_ctas && longest - (cost + n_ctas - 1) / n_ctas <= kWholeBlocks;
}

void launch_layout(const BatchLayout& bl, const Dims& dm, int tok_per_tile, int n_ctas, bool whole, int64_t n_pages,
                   int* status, bool tokens, int* desc_dev, const SmallDesc* desc, cudaStream_t st) {
  static const SmallDesc none{};
  const size_t smem = layout_smem_bytes(bl.n_req, n_ctas);
  static bool configured[kMaxDevices] = {false};
  if (first_use_on_device(configured))    // room for kMaxLayoutRequests requests (the default limit is 48 KB)
    cudaFuncSetAttribute(layout_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)layout_smem_bytes(kMaxLayoutRequests, 1024));
  const int token_ctas = tokens ? (bl.n_tok + kLayoutThreads - 1) / kLayoutThreads : 0;
  launch_pdl(layout_kernel, dim3(1 + token_ctas), dim3(kLayoutThreads), smem, st, bl, dm.n_kv, dm.mask_id, tok_per_tile, n_ctas,
             whole ? 1 : 0, n_pages, status, desc_dev, desc ? *desc : none);
}

void launch_embed(const BatchLayout& bl, const Dims& dm, const void* embed, float* h, const void* gain, void* x, float* ss,
                  void* rope_cs, int64_t n_pages, int* status, const int* desc_dev, const SmallDesc* desc, cudaStream_t st) {
  static const SmallDesc none{};
  launch_pdl(embed_kernel, dim3(bl.n_tok), dim3(256), 0, st, bl, dm.mask_id, n_pages, status, static_cast<const __nv_bfloat16*>(embed), h, dm.hidden, dm.vocab, static_cast<const __nv_bfloat16*>(gain),
             static_cast<__nv_bfloat16*>(x), ss, dm.rms_eps, static_cast<float2*>(rope_cs), dm.head_dim / 2,
             log((double)dm.rope_base), desc_dev, desc ? *desc : none);
}

void launch_rmsnorm(const float* h, const void* gain, void* x, int rows, int hidden, float eps, cudaStream_t st,
                    const int* rows_dev) {
  launch_pdl(rmsnorm_kernel, dim3(rows), dim3(256), 0, st, h, static_cast<const __nv_bfloat16*>(gain),
             static_cast<__nv_bfloat16*>(x), hidden, eps, rows_dev);
}

void launch_kv_io(bool write, void* pool, int64_t n_pages, int layer, const Dims& dm, const int* page_row, int pos0, int n_pos,
                  void* k, void* v, cudaStream_t st) {
  const size_t row = (size_t)dm.n_kv * (dm.head_dim / 8);     // chunks per position
  __nv_bfloat16* to = static_cast<__nv_bfloat16*>(pool);
  while (n_pos > 0) {
    const int first = pos0 / kPageSize;
    int n = (first + kKvIoPages) * kPageSize - pos0;          // positions that a launch's page ids cover
    if (n > n_pos) n = n_pos;
    uint4 *kp = static_cast<uint4*>(k), *vp = static_cast<uint4*>(v);
    if ((pos0 + n - 1) / kPageSize - first < kKvIoPagesFew)
      kv_io_part<kKvIoPagesFew>(write, to, n_pages, layer, dm, page_row, pos0, n, kp, vp, st);
    else
      kv_io_part<kKvIoPages>(write, to, n_pages, layer, dm, page_row, pos0, n, kp, vp, st);
    pos0 += n;
    n_pos -= n;
    k = kp + n * row;
    v = vp + n * row;
  }
}

}  // namespace recg

// ---------------------------------------------------------------------------------------------------
// Debug checks: guard bands behind the workspace regions, and a wait that is meant to run out.
// ---------------------------------------------------------------------------------------------------
namespace recg {
namespace {
constexpr uint32_t kGuardWord = 0x5ca1ab1eu;

// grid = bands, 64 threads: 256 bytes each
__global__ void guard_fill_kernel(uint8_t* base, const size_t* __restrict__ offs) {
  reinterpret_cast<uint32_t*>(base + offs[blockIdx.x])[threadIdx.x] = kGuardWord;
}
__global__ void guard_check_kernel(const uint8_t* base, const size_t* __restrict__ offs, int* status) {
  if (reinterpret_cast<const uint32_t*>(base + offs[blockIdx.x])[threadIdx.x] != kGuardWord) set_status(status, DEV_GUARD);
}

// One CTA, one thread: waits on an mbarrier that nobody ever arrives on, with the same bounded wait the kernels
// use; when the polls are used up it records the timeout in the status word and returns.  Nothing else happens:
// no trap, no fault, the context stays usable.
__global__ void wait_timeout_kernel(uint32_t max_polls, int* status) {
  __shared__ uint64_t bar;
  mbar_init(&bar, 1);
  fence_barrier_init();
  if (!mbar_wait(&bar, 0, max_polls)) set_status(status, DEV_TIMEOUT_FULL);
}
}  // namespace

void launch_guard_fill(void* base, const size_t* offs_dev, int n, cudaStream_t st) {
  if (n > 0) guard_fill_kernel<<<n, 64, 0, st>>>(static_cast<uint8_t*>(base), offs_dev);
}
void launch_guard_check(const void* base, const size_t* offs_dev, int n, int* status, cudaStream_t st) {
  if (n > 0) guard_check_kernel<<<n, 64, 0, st>>>(static_cast<const uint8_t*>(base), offs_dev, status);
}
void launch_wait_timeout(uint32_t max_polls, int* status, cudaStream_t st) {
  wait_timeout_kernel<<<1, 1, 0, st>>>(max_polls, status);
}
}  // namespace recg

// ---------------------------------------------------------------------------------------------------
// Device-resident rounds (Sec. 5.2): descriptor of a round from device arrays, and the step from one round to the next.
// ---------------------------------------------------------------------------------------------------
namespace recg {
namespace {

// One CTA.  Writes the packed descriptor [ctx_len | verify_len | block_size | corr (all zero: no correction branches in
// this mode) | cu_tok | cu_ver | verify_tokens (ragged)] and {n_tok, n_ver}.  A request whose lengths break a capacity
// (negative, no rows, more verify tokens than max_verify, rows beyond its page-table row, or a total beyond max_tokens)
// flags the status word and the round becomes empty (n_tok = 0): later kernels then do nothing.
__global__ void __launch_bounds__(256) pack_device_kernel(DeviceRound dr, int* __restrict__ desc, int* __restrict__ dyn,
                                                          int* status) {
  griddep_launch();
  griddep_wait();
  const int C = dr.n_req;
  int* ctx = desc;
  int* ver = desc + C;
  int* blk = desc + 2 * C;
  int* corr = desc + 3 * C;
  int* cu_tok = desc + 9 * C;
  int* cu_ver = cu_tok + (C + 1);
  int* vt = cu_ver + (C + 1);
  __shared__ int s_bad, s_tok, s_ver;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int r = threadIdx.x; r < C; r += blockDim.x) {
    const int L = dr.ctx_len[r], v = dr.verify_len[r], b = dr.block_size[r];
    if (L < 0 || v < 0 || b < 0 || v + b < 1 || v > dr.max_verify ||
        ((long long)L + v + b + kPageSize - 1) / kPageSize > dr.pt_stride)
      s_bad = 1;
    ctx[r] = L;
    ver[r] = v;
    blk[r] = b;
    for (int k = 0; k < 6; ++k) corr[6 * r + k] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0, tv = 0;
    cu_tok[0] = cu_ver[0] = 0;
    for (int r = 0; r < C; ++r) {
      t += ver[r] + blk[r];
      tv += ver[r];
      if (t > dr.max_tokens || t < 0) {
        s_bad = 1;
        t = tv = 0;
      }
      cu_tok[r + 1] = t;
      cu_ver[r + 1] = tv;
    }
    if (s_bad) {
      set_status(status, DEV_BAD_INDEX);
      t = tv = 0;
      for (int r = 0; r <= C; ++r) cu_tok[r] = cu_ver[r] = 0;
    }
    s_tok = t;
    s_ver = tv;
    dyn[0] = t;
    dyn[1] = tv;
  }
  __syncthreads();
  if (s_tok == 0) return;
  for (int r = threadIdx.x; r < C; r += blockDim.x)
    for (int j = 0; j < ver[r]; ++j) vt[cu_ver[r] + j] = dr.verify_tokens[(size_t)r * dr.max_verify + j];
}

// One thread per request: the bookkeeping between two rounds (Sec. 3.1, 5.1) from the verification results that are
// still on the device.  planted_emitted (may be null): synthetic acceptance -- the round is taken to have emitted
// min(planted_emitted[r], v) tokens, and its continuation block to be reusable exactly when all drafts were accepted.
__global__ void next_round_kernel(DeviceRound dr, BatchLayout bl, VerifyBuffers vb, const int* __restrict__ next_block,
                                  const int* __restrict__ planted_emitted, RoundLog log, int round, int* status) {
  griddep_launch();
  griddep_wait();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < dr.n_req) {
    const int L = bl.ctx_len[r], v = bl.verify_len[r], b = bl.block_size[r];
    const int t0 = bl.cu_tok[r], tv0 = bl.cu_ver[r];
    const bool ran = bl.cu_tok[dr.n_req] > 0;       // an empty round (a capacity was broken) changes nothing
    int a = 0, emitted = 0, cont = 0;
    if (ran && v > 0) {
      a = vb.accept_len[r];
      cont = vb.cont_hit[r];
      if (planted_emitted) {
        const int e = planted_emitted[r] < 1 ? 1 : (planted_emitted[r] > v ? v : planted_emitted[r]);
        a = e - 1;
        cont = (b > 0 && a == v - 1) ? 1 : 0;
      }
      emitted = a + 1;
    }
    if (log.accept_len && round < log.max_rounds) {
      log.accept_len[(size_t)round * dr.n_req + r] = a;
      log.block_size[(size_t)round * dr.n_req + r] = b;
      log.verify_len[(size_t)round * dr.n_req + r] = v;
      if (log.entropy_mean) log.entropy_mean[(size_t)round * dr.n_req + r] = (ran && v > 0) ? vb.entropy_mean[r] : 0.f;
    }
    if (ran && v > 0) {
      // emitted tokens: the accepted drafts y_1 .. y_a, then the verifier's token at row a
      const int last = vb.top1[t0 + a];
      if (log.tokens) {
        int n = log.n_tokens[r];
        for (int i = 1; i <= a && n < log.max_out; ++i) log.tokens[(size_t)r * log.max_out + n++] = bl.verify_tokens[tv0 + i];
        if (n < log.max_out) log.tokens[(size_t)r * log.max_out + n++] = last;
        log.n_tokens[r] = n;
      }
      int nb = next_block ? next_block[r] : b;
      int nv = 1;
      int* y = dr.verify_tokens + (size_t)r * dr.max_verify;
      y[0] = last;
      if (cont) {                      // the drafted block becomes the next verify tokens (its first token only
        nv = b < dr.max_verify ? b : dr.max_verify;   // confirmed the one just emitted)
        const int tb0 = t0 - tv0;      // offset of the request's draft rows in next_draft
        for (int j = 1; j < nv; ++j) y[j] = vb.next_draft[tb0 + j];
      }
      const int nL = L + emitted;
      // the next round must fit the page-table row; a request that has run out of room stops growing
      if (((long long)nL + nv + nb + kPageSize - 1) / kPageSize > dr.pt_stride) {
        nb = 0;
        nv = 1;
        if (((long long)nL + 1 + kPageSize - 1) / kPageSize > dr.pt_stride) set_status(status, DEV_BAD_INDEX);
      }
      dr.ctx_len[r] = nL;
      dr.verify_len[r] = nv;
      dr.block_size[r] = nb;
    } else if (ran && next_block) {
      dr.block_size[r] = next_block[r];
    }
  }
  if (r == 0 && log.n_rounds) log.n_rounds[0] = round + 1;     // rounds logged so far
}

}  // namespace

void launch_pack_device(const DeviceRound& dr, int* desc, int* dyn, int* status, cudaStream_t st) {
  launch_pdl(pack_device_kernel, dim3(1), dim3(256), 0, st, dr, desc, dyn, status);
}

void launch_next_round(const DeviceRound& dr, const BatchLayout& bl, const VerifyBuffers& vb, const int* next_block,
                       const int* planted_emitted, const RoundLog& log, int round, int* status, cudaStream_t st) {
  launch_pdl(next_round_kernel, dim3((dr.n_req + 127) / 128), dim3(128), 0, st, dr, bl, vb, next_block, planted_emitted, log,
             round, status);
}
}  // namespace recg
