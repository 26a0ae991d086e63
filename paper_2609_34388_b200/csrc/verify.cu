// Fused greedy verification: one pass over the logits (top-2 ids, softmax mass, entropy) split over
// vocab chunks, then a per-request finalize (accept-length scan, emitted tokens, continuation rule,
// mean verifier entropy, KV commit / rollback indices).
#include <cstddef>
#include <string>

#include "../../include/recg.h"
#include "common.cuh"
#include "kernels.h"

namespace recg {

namespace {

constexpr int kVerifyThreads = 256;

struct Top2 {
  float m1, m2;
  int i1, i2;
};
__device__ __forceinline__ bool better(float av, int ai, float bv, int bi) { return av > bv || (av == bv && ai < bi); }
__device__ __forceinline__ void top2_insert(Top2& t, float x, int i) {
  if (better(x, i, t.m1, t.i1)) {
    t.m2 = t.m1; t.i2 = t.i1; t.m1 = x; t.i1 = i;
  } else if (better(x, i, t.m2, t.i2)) {
    t.m2 = x; t.i2 = i;
  }
}

// running softmax mass relative to a moving maximum m: s = sum e^(x-m), t = sum x e^(x-m)
// (entropy = ln s - t/s + m).  Logits of -inf contribute nothing: they are clamped to a finite value whose
// exponential underflows to zero, so that x * 0 stays 0.
struct Mass {
  float m, s, t;
};
constexpr float kLog2e = 1.4426950408889634f;
// The moving maximum starts no lower than this: masked logits (-inf, the type's lowest value, -1e30) then underflow to zero while
// a thread or a chunk has seen nothing else, where x log2(e) - m log2(e) would overflow or cancel to anything.  (Below it the
// product's rounding error reaches the exponent's range; no logit that counts lies there.)
constexpr float kMassFloor = -1.0e9f;
__device__ __forceinline__ void mass_rebase(Mass& a, float m_new) {
  if (m_new > a.m) {
    const float f = a.s > 0.f ? exp2f((a.m - m_new) * kLog2e) : 0.f;   // a.m may be -inf with s = t = 0
    a.s *= f;
    a.t *= f;
    a.m = m_new;
  }
}
// neg_m2 = -m * log2(e), hoisted by the caller
__device__ __forceinline__ void mass_add(Mass& a, float x, float neg_m2) {
  const float xc = fmaxf(x, -3.0e38f);
  const float e = exp2f(fmaf(xc, kLog2e, neg_m2));
  a.s += e;
  a.t = fmaf(xc, e, a.t);
}
__device__ __forceinline__ void mass_merge(Mass& a, const Mass& b) {
  if (b.s <= 0.f) return;
  Mass bb = b;
  const float m = fmaxf(a.m, b.m);
  mass_rebase(a, m);
  mass_rebase(bb, m);
  a.s += bb.s;
  a.t += bb.t;
}

// One 16-byte vector of logits as words; fill = -inf in every element.
template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  static constexpr uint32_t kFill = 0xff80ff80u;
  __device__ static float one(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  // largest element of four vectors
  __device__ static float max_of(const uint4 (&r)[4]) {
    __nv_bfloat162 m = word(r[0].x);
#pragma unroll
    for (int u = 0; u < 4; ++u) m = __hmax2(__hmax2(m, __hmax2(word(r[u].x), word(r[u].y))), __hmax2(word(r[u].z), word(r[u].w)));
    return fmaxf(__low2float(m), __high2float(m));
  }
  __device__ static __nv_bfloat162 word(uint32_t w) { return *reinterpret_cast<__nv_bfloat162*>(&w); }
  __device__ static void elements(const uint4& r, float (&x)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = __uint_as_float(w[i] << 16);
      x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
  static constexpr int kPairs = 4;       // pairs of elements per vector
  __device__ static float2 pair(const uint4& r, int i) {
    const uint32_t w = i == 0 ? r.x : (i == 1 ? r.y : (i == 2 ? r.z : r.w));
    const __nv_bfloat162 c = __hmax2(word(w), word(0xff7fff7fu));      // -inf -> the lowest finite value
    const uint32_t cw = *reinterpret_cast<const uint32_t*>(&c);
    return make_float2(__uint_as_float(cw << 16), __uint_as_float(cw & 0xffff0000u));
  }
};
template <> struct Vec<float> {
  static constexpr int N = 4;
  static constexpr uint32_t kFill = 0xff800000u;
  __device__ static float one(const float* p) { return *p; }
  __device__ static float max_of(const uint4 (&r)[4]) {
    float m = -INFINITY;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(r[u].x), __uint_as_float(r[u].y)), fmaxf(__uint_as_float(r[u].z), __uint_as_float(r[u].w))));
    return m;
  }
  __device__ static void elements(const uint4& r, float (&x)[4]) {
    x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y); x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
  }
  static constexpr int kPairs = 2;
  __device__ static float2 pair(const uint4& r, int i) {
    return i == 0 ? make_float2(fmaxf(__uint_as_float(r.x), -3.0e38f), fmaxf(__uint_as_float(r.y), -3.0e38f))
                  : make_float2(fmaxf(__uint_as_float(r.z), -3.0e38f), fmaxf(__uint_as_float(r.w), -3.0e38f));
  }
};
__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 u;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "l"(p));
  return u;
}
// One-dimensional grid of rows x chunks_per_row CTAs, chunk-fastest (consecutive CTAs read consecutive memory; the
// row count is not bound by the 65535 limit of the other grid dimensions).  Each CTA scans [c0, c1) of one row.
// Bound by HBM for bf16 logits only if little else is done per element (6.4 TB/s is 11 elements per SM and clock: two thirds of
// what the 2^x unit gives, and the issue slots leave 11 instructions for each): vectors stay packed (maxima and the clamp of
// -inf on two bf16 at a time), sums use two-element instructions, the next four vectors of a thread are on their way while it
// works on four, and the search for the two largest elements remembers only the two best GROUPS of four vectors per thread, of
// which the CTA afterwards re-reads those that reach its second-largest group maximum (two, as a rule).  8448 rows x 128256
// bf16, the kernel: 435 us with unpacked arithmetic, loads behind the arithmetic and a search per thread, 358 us (6.05 TB/s)
// like this.
template <typename T>
__global__ void __launch_bounds__(kVerifyThreads, 4) verify_partial_kernel(const T* __restrict__ logits, int vocab,
                                                                           int chunk_len, int chunks_per_row,
                                                                           RowPartial* __restrict__ partials,
                                                                           const int* __restrict__ rows_dev) {
  constexpr int N = Vec<T>::N, kWarps = kVerifyThreads / 32;
  __shared__ float2 s_g[kWarps];
  __shared__ Top2 s_tp[kWarps];
  __shared__ float2 s_st[kWarps];
  griddep_launch();
  griddep_wait();
  const int row = blockIdx.x / chunks_per_row, chunk = blockIdx.x - row * chunks_per_row;
  if (rows_dev && row >= rows_dev[0]) return;      // (the grid was sized for the capacity)
  const T* base = logits + (size_t)row * vocab;
  const int c0 = chunk * chunk_len;
  const int c1 = min(vocab, c0 + chunk_len);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool vec_ok = ((reinterpret_cast<uintptr_t>(base + c0) & 15) == 0);
  const int nvec = vec_ok ? (c1 - c0) / N : 0;
  Top2 tp = {-INFINITY, -INFINITY, 0x7fffffff, 0x7fffffff};
  Mass ms = {-INFINITY, 0.f, 0.f};
  float g1 = -INFINITY, g2 = -INFINITY;      // the two largest group maxima of this thread ...
  int i1 = -1, i2 = -1;                      // ... and the first vector of those groups (the earlier one on ties)
  const uint4* vec = reinterpret_cast<const uint4*>(base + c0);
  auto fetch = [&](int i, uint4 (&r)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = i + u * kVerifyThreads;
      r[u] = k < nvec ? ld_stream(vec + k) : make_uint4(Vec<T>::kFill, Vec<T>::kFill, Vec<T>::kFill, Vec<T>::kFill);
    }
  };
  if (nvec > 0) {
    uint4 cur[4], nxt[4];
    float2 s2 = make_float2(0.f, 0.f), t2 = make_float2(0.f, 0.f);
    const float2 log2e = make_float2(kLog2e, kLog2e);
    fetch(tid, cur);
    for (int i = tid; i < nvec; i += 4 * kVerifyThreads) {
      fetch(i + 4 * kVerifyThreads, nxt);
      const float gm = Vec<T>::max_of(cur);
      if (gm > ms.m) {
        const float m = fmaxf(gm, kMassFloor), f = exp2f((ms.m - m) * kLog2e);      // 0 the first time
        s2.x *= f; s2.y *= f; t2.x *= f; t2.y *= f;
        ms.m = m;
      }
      const bool b1 = gm > g1, b2 = gm > g2;
      i2 = b1 ? i1 : (b2 ? i : i2);
      g2 = b1 ? g1 : (b2 ? gm : g2);
      i1 = b1 ? i : i1;
      g1 = b1 ? gm : g1;
      const float neg = ms.m > -INFINITY ? -ms.m * kLog2e : 0.f;   // all -inf so far: every term underflows to 0
      const float2 neg2 = make_float2(neg, neg);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < Vec<T>::kPairs; ++k) {
          const float2 x = Vec<T>::pair(cur[u], k);
          const float2 y = fma2(x, log2e, neg2);
          const float2 e = make_float2(exp2f(y.x), exp2f(y.y));
          s2 = add2(s2, e);
          t2 = fma2(x, e, t2);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u) cur[u] = nxt[u];
    }
    ms.s = s2.x + s2.y;
    ms.t = t2.x + t2.y;
  }
  // elements outside whole vectors (unaligned rows: all of them), four loads in flight per thread: 5000 x 50257 fp32 379 us, one
  // by one 743
  for (int i = c0 + nvec * N + tid; i < c1; i += 4 * kVerifyThreads) {
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = i + u * kVerifyThreads < c1 ? Vec<T>::one(base + i + u * kVerifyThreads) : -INFINITY;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i + u * kVerifyThreads >= c1) break;
      mass_rebase(ms, fmaxf(x[u], kMassFloor));
      mass_add(ms, x[u], ms.m > -INFINITY ? -ms.m * kLog2e : 0.f);
      if (x[u] >= tp.m2) top2_insert(tp, x[u], i + u * kVerifyThreads);
    }
  }
  const float e1 = tp.m1, e2 = tp.m2;
  // the CTA's largest and second-largest of the groups' maxima and the single elements
  float h1 = fmaxf(g1, e1), h2 = fmaxf(fminf(g1, e1), fmaxf(g2, e2));
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float a = __shfl_xor_sync(0xffffffffu, h1, o), b = __shfl_xor_sync(0xffffffffu, h2, o);
    h2 = fmaxf(fminf(h1, a), fmaxf(h2, b));
    h1 = fmaxf(h1, a);
  }
  if (lane == 0) s_g[warp] = make_float2(h1, h2);
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const float2 g = s_g[w];
    if (w == 0) { h1 = g.x; h2 = g.y; continue; }
    h2 = fmaxf(fminf(h1, g.x), fmaxf(h2, g.y));
    h1 = fmaxf(h1, g.x);
  }
  // The two largest elements are not below the second-largest group maximum: only groups that reach it are searched element
  // by element (in index order; ties resolve to the lowest index).
  const int lo = i2 < 0 ? i1 : min(i1, i2), hi = i2 < 0 ? -1 : max(i1, i2);
  const float g_lo = lo == i1 ? g1 : g2, g_hi = hi == i2 ? g2 : g1;
#pragma unroll 1
  for (int q = 0; q < 2; ++q) {
    const int i = q ? hi : lo;
    if (i < 0 || (q ? g_hi : g_lo) < h2) continue;
    uint4 r[4];
    fetch(i, r);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float x[N];
      Vec<T>::elements(r[u], x);
      if (i + u * kVerifyThreads < nvec)
#pragma unroll
        for (int k = 0; k < N; ++k)
          if (x[k] >= tp.m2) top2_insert(tp, x[k], c0 + (i + u * kVerifyThreads) * N + k);
    }
  }
  const float f = ms.m > -INFINITY ? exp2f((ms.m - fmaxf(h1, kMassFloor)) * kLog2e) : 0.f;
  ms.s *= f;
  ms.t *= f;
  const bool any = __any_sync(0xffffffffu, tp.i1 != 0x7fffffff);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    ms.s += __shfl_xor_sync(0xffffffffu, ms.s, o);
    ms.t += __shfl_xor_sync(0xffffffffu, ms.t, o);
    if (!any) continue;
    const Top2 ot = {__shfl_xor_sync(0xffffffffu, tp.m1, o), __shfl_xor_sync(0xffffffffu, tp.m2, o),
                     __shfl_xor_sync(0xffffffffu, tp.i1, o), __shfl_xor_sync(0xffffffffu, tp.i2, o)};
    top2_insert(tp, ot.m1, ot.i1);
    top2_insert(tp, ot.m2, ot.i2);
  }
  if (lane == 0) {
    s_tp[warp] = tp;
    s_st[warp] = make_float2(ms.s, ms.t);
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kWarps; ++w) {
      top2_insert(tp, s_tp[w].m1, s_tp[w].i1);
      top2_insert(tp, s_tp[w].m2, s_tp[w].i2);
      ms.s += s_st[w].x;
      ms.t += s_st[w].y;
    }
    RowPartial p;
    p.m1 = tp.m1; p.m2 = tp.m2; p.i1 = tp.i1; p.i2 = tp.i2;
    p.s = ms.s; p.t = ms.t;               // relative to the chunk's maximum
    partials[(size_t)row * chunks_per_row + chunk] = p;
  }
}

// Statistics of one row from its chunk partials: `lanes` consecutive lanes (a power of two) share the row, every lane of the
// warp takes part, and all lanes of a group return the row's result.
struct RowStats {
  int top1, top2;
  float p1, p2, entropy;
};
__device__ __forceinline__ RowStats row_stats(const RowPartial* __restrict__ p, int chunks, int lanes, bool valid) {
  Top2 tp = {-INFINITY, -INFINITY, 0x7fffffff, 0x7fffffff};
  Mass ms = {-INFINITY, 0.f, 0.f};
  for (int c = threadIdx.x & (lanes - 1); valid && c < chunks; c += lanes) {
    const RowPartial q = p[c];
    top2_insert(tp, q.m1, q.i1);
    top2_insert(tp, q.m2, q.i2);
    mass_merge(ms, Mass{q.m1, q.s, q.t});
  }
  for (int o = lanes >> 1; o; o >>= 1) {
    const Top2 ot = {__shfl_xor_sync(0xffffffffu, tp.m1, o), __shfl_xor_sync(0xffffffffu, tp.m2, o),
                     __shfl_xor_sync(0xffffffffu, tp.i1, o), __shfl_xor_sync(0xffffffffu, tp.i2, o)};
    top2_insert(tp, ot.m1, ot.i1);
    top2_insert(tp, ot.m2, ot.i2);
    mass_merge(ms, Mass{__shfl_xor_sync(0xffffffffu, ms.m, o), __shfl_xor_sync(0xffffffffu, ms.s, o), __shfl_xor_sync(0xffffffffu, ms.t, o)});
  }
  const float inv = 1.f / ms.s;
  return RowStats{tp.i1, tp.i2, inv,                               // e^(m1 - m1) / S
                  __expf(tp.m2 - tp.m1) * inv, logf(ms.s) - ms.t * inv + ms.m};   // ln S - (1/S) sum x e^(x-M) + M
}
// lanes per row: the smallest power of two that covers the chunks, at most a warp
__host__ __device__ inline int stat_lanes(int chunks) {
  int g = 1;
  while (g < chunks && g < 32) g *= 2;
  return g;
}

// One CTA per request: merge the chunk partials of its rows, then the accept scan and the index work.  A handful of values
// per row and several dependent decisions: bound by latency, so the rows' chunk partials are merged by groups of lanes, the
// statistics the decisions need stay in shared memory (kFinalRows rows; a longer request reads them back from its output
// arrays), the scans over rows are ballots, and the descriptor is read ahead of the wait for the vocabulary scan where it is
// settled (desc_settled).  Every result also goes to the host's mirror of the output arrays (`mirror` bytes further on, in
// mapped pinned memory; 0: none), so that no copy has to follow.  One request with four drafts: 20.8 us of the call with one
// thread per row and serial scans plus 13.8 us for the copy, 7.9 us with this kernel.
constexpr int kFinalThreads = 256, kFinalRows = 256;
__global__ void __launch_bounds__(kFinalThreads) verify_finalize_kernel(BatchLayout bl, const RowPartial* __restrict__ partials,
                                                                        int chunks_per_row, VerifyBuffers vb, int desc_settled,
                                                                        ptrdiff_t mirror, int* desc_dev,
                                                                        const __grid_constant__ SmallDesc desc) {
  __shared__ int s_top1[kFinalRows], s_top2[kFinalRows], s_vt[kFinalRows];
  __shared__ float s_p1[kFinalRows], s_p2[kFinalRows], s_ent[kFinalRows];
  __shared__ int s_a, s_first_free, s_last;
  griddep_launch();
  if (!desc_settled) griddep_wait();
  if (desc.n) bl.rebase(desc_dev, desc.v);
  const int r = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t0 = bl.cu_tok[r], tv0 = bl.cu_ver[r];
  const int n = bl.cu_tok[r + 1] - t0;          // v + b + n_corr * span; 0 in a round that broke a capacity on the device,
  // whose lengths come as they were given: v and b must name rows of the request in any case
  const int v = max(0, min(bl.verify_len[r], n)), b = max(0, min(bl.block_size[r], n - v)), L = bl.ctx_len[r];
  const int* cr = bl.corr + 6 * r;              // correction branches: count, mask tokens per branch, indices, tokens
  const int n_corr = n > 0 ? cr[0] : 0, span = 1 + cr[1];
  const bool small = n <= kFinalRows;
  if (small)
    for (int j = tid; j < v; j += kFinalThreads) s_vt[j] = bl.verify_tokens[tv0 + j];
  if (desc_settled) griddep_wait();
  if (desc.n && r == 0 && !bl.page_table)      // for the kernels that may follow (the layout kernel has not written it)
    for (int i = tid; i < desc.n; i += kFinalThreads) desc_dev[i] = desc.v[i];
  auto put = [&](auto* p, auto x) {
    *p = x;
    if (mirror) *reinterpret_cast<decltype(p)>(reinterpret_cast<char*>(p) + mirror) = x;
  };
  const int lanes = stat_lanes(chunks_per_row), group = tid / lanes, groups = kFinalThreads / lanes;
  for (int j0 = 0; j0 < n; j0 += groups) {
    const int j = j0 + group;
    const RowStats st = row_stats(partials + (size_t)(t0 + j) * chunks_per_row, chunks_per_row, lanes, j < n);
    if (j < n && (tid & (lanes - 1)) == 0) {
      if (small) {
        s_top1[j] = st.top1; s_top2[j] = st.top2; s_p1[j] = st.p1; s_p2[j] = st.p2; s_ent[j] = st.entropy;
      } else {
        put(vb.top1 + t0 + j, st.top1); put(vb.top2 + t0 + j, st.top2);
        put(vb.p1 + t0 + j, st.p1); put(vb.p2 + t0 + j, st.p2); put(vb.entropy + t0 + j, st.entropy);
      }
    }
  }
  __syncthreads();
  const int* top1 = small ? s_top1 : vb.top1 + t0;
  const int* top2 = small ? s_top2 : vb.top2 + t0;
  const int* vt = small ? s_vt : bl.verify_tokens + tv0;
  const float* p1 = small ? s_p1 : vb.p1 + t0;
  const float* p2 = small ? s_p2 : vb.p2 + t0;
  const float* ent = small ? s_ent : vb.entropy + t0;
  if (warp == 0) {
    int a = v > 0 ? v - 1 : 0;           // drafts accepted: up to the first one that differs from the verifier's token
    for (int j0 = 0; j0 < v - 1; j0 += 32) {
      const int j = j0 + lane;
      const unsigned diff = __ballot_sync(0xffffffffu, j < v - 1 && vt[j + 1] != top1[j]);
      if (diff) {
        a = j0 + __ffs(diff) - 1;
        break;
      }
    }
    if (lane == 0) {
      float es = 0.f;
      if (v > 0) {
        for (int i = 0; i <= a; ++i) es += ent[i];
        es /= (a + 1);
      }
      put(vb.entropy_mean + r, es);
      put(vb.accept_len + r, a);
      put(vb.n_emitted + r, v > 0 ? a + 1 : 0);
      const int new_L = L + (v > 0 ? a + 1 : 0);
      put(vb.new_ctx_len + r, new_L);
      put(vb.cont_hit + r, (v > 0 && b > 0 && a == v - 1 && top1[v] == top1[v - 1]) ? 1 : 0);
      const int first_free = (new_L + kPageSize - 1) / kPageSize;
      const int last = (L + n + kPageSize - 1) / kPageSize;
      put(vb.freed_pages + r, bl.page_table ? last - first_free : 0);
      s_first_free = first_free;
      s_last = bl.page_table ? last : first_free;
      // a correction branch is confirmed when the verifier rejected exactly the draft it replaced and emitted the
      // replacement token there (Sec. 5.1)
      for (int k = 0; k < 2; ++k)
        put(vb.corr_hit + 2 * r + k, (k < n_corr && v > 0 && a == cr[2 + k] - 1 && top1[a] == cr[4 + k]) ? 1 : 0);
      s_a = a;
    }
  } else if (warp <= 3) {
    // risky drafts of every draft block, indexed as the verify tokens the block would become: the continuation's
    // mask row m is y'_m (row 0 only confirms the bonus token), a correction's mask row m is y'_{m+1}
    const int blk = warp - 1;
    int row0 = 0, rows = 0;
    if (blk == 0) { row0 = v + 1; rows = b > 0 ? b - 1 : 0; }
    else if (blk - 1 < n_corr) { row0 = v + b + (blk - 1) * span + 1; rows = span - 1; }
    int cnt = 0, at[2] = {-1, -1};       // (the same in every lane)
    for (int m0 = 0; m0 < rows; m0 += 32) {
      const int m = m0 + lane;
      unsigned risky = __ballot_sync(0xffffffffu, m < rows && p1[row0 + m] - p2[row0 + m] < bl.risk_delta);
      while (risky && cnt < 2) {
        at[cnt++] = m0 + __ffs(risky) - 1;
        risky &= risky - 1;
      }
      cnt += __popc(risky);
    }
    if (lane == 0) put(vb.risky_n + 3 * r + blk, cnt);
    if (lane < 2) {
      put(vb.risky_index + 6 * r + 2 * blk + lane, at[lane] < 0 ? -1 : 1 + at[lane]);
      put(vb.risky_token + 6 * r + 2 * blk + lane, at[lane] < 0 ? -1 : top2[row0 + at[lane]]);
    }
  }
  __syncthreads();
  const int a = s_a;
  const int tb0 = t0 - tv0;  // draft-token offset of this request: sum of b over earlier requests
  for (int j = tid; j < n; j += kFinalThreads) {
    if (small) {
      put(vb.top1 + t0 + j, top1[j]); put(vb.top2 + t0 + j, top2[j]);
      put(vb.p1 + t0 + j, p1[j]); put(vb.p2 + t0 + j, p2[j]); put(vb.entropy + t0 + j, ent[j]);
    }
    if (j < v) put(vb.emitted + tv0 + j, j < a ? vt[j + 1] : (j == a ? top1[a] : -1));
    else put(vb.next_draft + tb0 + (j - v), top1[j]);
    int state = 0;
    if (bl.page_table) {
      const int slot = bl.tok_slot[t0 + j];
      state = slot < 0 ? 0 : ((j < v && j <= a) ? slot : -(slot + 1));
    }
    put(vb.slot_state + t0 + j, state);
    // ids of the pages that hold no committed token any more, at the request's row offset (there are never more
    // of them than rows: each starts at a position of a row that was rolled back)
    if (vb.freed_page_ids) {
      const int e = s_first_free + j;
      put(vb.freed_page_ids + t0 + j, e < s_last ? bl.page_table[(size_t)r * bl.pt_stride + e] : -1);
    }
  }
}

}  // namespace

int verify_chunks_per_row(int rows, int vocab, int n_sm) {
  int by_size = (vocab + 4095) / 4096;
  int by_rows = rows > 0 ? (n_sm * 4 + rows - 1) / rows : 1;
  int c = by_size < by_rows ? by_size : by_rows;
  if (c < 1) c = 1;
  if (c > 64) c = 64;
  return c;
}

void launch_verify(const BatchLayout& bl, const void* logits, int logits_dtype, int vocab, RowPartial* partials,
                   int max_chunks_total, const VerifyBuffers& vb, int* desc_dev, const SmallDesc* desc, int n_sm, cudaStream_t st,
                   ptrdiff_t mirror) {
  static const SmallDesc none{};
  const int rows = bl.n_tok;
  if (rows <= 0) return;
  int chunks = verify_chunks_per_row(rows, vocab, n_sm);
  while (chunks > 1 && (long long)chunks * rows > max_chunks_total) --chunks;
  int chunk_len = (vocab + chunks - 1) / chunks;
  chunk_len = (chunk_len + 63) / 64 * 64;  // keeps every chunk start 16-byte aligned relative to the row
  chunks = (vocab + chunk_len - 1) / chunk_len;
  dim3 grid((unsigned)chunks * (unsigned)rows);
  if (logits_dtype == 0)
    launch_pdl(verify_partial_kernel<__nv_bfloat16>, grid, dim3(kVerifyThreads), 0, st,
               static_cast<const __nv_bfloat16*>(logits), vocab, chunk_len, chunks, partials, bl.dyn);
  else
    launch_pdl(verify_partial_kernel<float>, grid, dim3(kVerifyThreads), 0, st, static_cast<const float*>(logits), vocab,
               chunk_len, chunks, partials, bl.dyn);
  // (a descriptor that the host uploaded was in place before the vocabulary scan could start, and a small one comes with this
  // launch; one that a kernel of this round packs on the device is not settled before the wait)
  launch_pdl(verify_finalize_kernel, dim3(bl.n_req), dim3(kFinalThreads), 0, st, bl, (const RowPartial*)partials, chunks, vb,
             bl.dyn ? 0 : 1, mirror, desc_dev, desc ? *desc : none);
}

}  // namespace recg

// ---------------------------------------------------------------------------------------------------
// Block-size rule of verification-guided drafting (Sec. 5.2): one thread per request.
// ---------------------------------------------------------------------------------------------------
namespace recg {
namespace {

__global__ void policy_kernel(BatchLayout bl, PolicyTable tb, float* __restrict__ e1, float* __restrict__ e2,
                              int* __restrict__ block_index, int* __restrict__ full,
                              const float* __restrict__ entropy_mean, const int* __restrict__ accept_len,
                              int* __restrict__ next_block) {
  griddep_launch();
  griddep_wait();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= bl.n_req) return;
  const int v = bl.verify_len[r];
  float a1 = e1[r], a2 = e2[r];
  int f = full[r];
  if (v > 0) {   // the finished round verified something: shift its mean verifier entropy into the history
    a2 = a1;
    a1 = entropy_mean[r];
    f = (v > 1 && accept_len[r] == v - 1) ? 1 : 0;
    e1[r] = a1;
    e2[r] = a2;
    full[r] = f;
  }
  const float s = __fmul_rn(__fadd_rn(a1, a2), -0.5f);   // Eq. 2
  int k = 0;
  for (int i = 0; i < tb.n_bins - 1; ++i) k += tb.edges[i] <= s ? 1 : 0;
  int jp = block_index[r];
  jp = jp < 0 ? 0 : (jp >= tb.n_blocks ? tb.n_blocks - 1 : jp);
  int best = 0;
  float best_score = 0.f;
  for (int j = 0; j < tb.n_blocks; ++j) {   // Eq. 3; the first maximum wins
    const float score = __fsub_rn(tb.value[((j * tb.n_bins + k) * tb.n_blocks + jp) * 2 + f], tb.cost[j]);
    if (j == 0 || score > best_score) { best = j; best_score = score; }
  }
  block_index[r] = best;
  next_block[r] = tb.blocks[best];
}

}  // namespace

void launch_policy(const BatchLayout& bl, const PolicyTable& tb, float* e1, float* e2, int* block_index, int* full,
                   const float* entropy_mean, const int* accept_len, int* next_block, cudaStream_t st) {
  if (bl.n_req <= 0) return;
  launch_pdl(policy_kernel, dim3((bl.n_req + 127) / 128), dim3(128), 0, st, bl, tb, e1, e2, block_index, full,
             entropy_mean, accept_len, next_block);
}

}  // namespace recg

// ---------------------------------------------------------------------------------------------------
// Row statistics without any allocation: the chunk partials live in a file-scope device array.
// ---------------------------------------------------------------------------------------------------
namespace recg {
namespace {

constexpr int kStaticMaxPartials = 1 << 16;   // 65536 x 24 bytes = 1.5 MiB held by every GPU that loads the library
static __device__ __align__(256) RowPartial g_static_partials[kStaticMaxPartials];

RowPartial* g_static_ptr[kMaxDevices] = {nullptr};   // device address of the array, per device, set on first use
int g_static_sm[kMaxDevices] = {0};

thread_local std::string g_static_error;

// merges the rows' chunk partials into the five per-row outputs, stat_lanes(chunks) lanes per row
__global__ void row_stats_finalize_kernel(const RowPartial* __restrict__ partials, int rows, int chunks_per_row, int lanes,
                                          int* __restrict__ top1, int* __restrict__ top2, float* __restrict__ p1,
                                          float* __restrict__ p2, float* __restrict__ entropy) {
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) / lanes;
  const RowStats s = row_stats(partials + (size_t)r * chunks_per_row, chunks_per_row, lanes, r < rows);
  if (r >= rows || (threadIdx.x & (lanes - 1))) return;
  if (top1) top1[r] = s.top1;
  if (top2) top2[r] = s.top2;
  if (p1) p1[r] = s.p1;
  if (p2) p2[r] = s.p2;
  if (entropy) entropy[r] = s.entropy;
}

}  // namespace

const char* static_entry_error() { return g_static_error.c_str(); }

}  // namespace recg

extern "C" const char* recg_row_stats_static_error(void) { return recg::static_entry_error(); }

extern "C" recg_status recg_row_stats_static(const void* logits, int32_t logits_dtype, int32_t rows, int32_t vocab,
                                             int32_t* top1, int32_t* top2, float* p1, float* p2, float* entropy,
                                             void* cuda_stream) {
  using namespace recg;
  auto fail = [](recg_status s, const std::string& m) { g_static_error = m; return s; };
  if (!logits || rows < 0 || vocab <= 1) return fail(RECG_ERR_INVALID_ARG, "recg_row_stats_static: null logits or bad extent");
  if (logits_dtype != RECG_DTYPE_BF16 && logits_dtype != RECG_DTYPE_F32)
    return fail(RECG_ERR_INVALID_ARG, "recg_row_stats_static: unknown logits dtype");
  if (rows == 0) return RECG_OK;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(RECG_ERR_CUDA, "recg_row_stats_static: no current CUDA device");
  if (!g_static_ptr[dev]) {
    // first call on this device: the array's name is only a host-side handle, so ask the runtime for the
    // device address (with this device current) and remember it
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_partials);
    if (e != cudaSuccess || !ptr)
      return fail(RECG_ERR_CUDA, std::string("recg_row_stats_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    int n_sm = 0;
    e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || n_sm <= 0)
      return fail(RECG_ERR_CUDA, std::string("recg_row_stats_static: SM count: ") + cudaGetErrorString(e));
    g_static_sm[dev] = n_sm;
    g_static_ptr[dev] = static_cast<RowPartial*>(ptr);
  }
  if (rows > kStaticMaxPartials)
    return fail(RECG_ERR_CAPACITY, "recg_row_stats_static: more than 65536 rows; use recg_verify with a context");
  int chunks = verify_chunks_per_row(rows, vocab, g_static_sm[dev]);
  while (chunks > 1 && (long long)chunks * rows > kStaticMaxPartials) --chunks;
  int chunk_len = (vocab + chunks - 1) / chunks;
  chunk_len = (chunk_len + 63) / 64 * 64;
  chunks = (vocab + chunk_len - 1) / chunk_len;
  if ((long long)chunks * rows > kStaticMaxPartials)
    return fail(RECG_ERR_CAPACITY, "recg_row_stats_static: rows x vocab chunks exceed the static scratch (65536 partials)");
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  RowPartial* scratch = g_static_ptr[dev];
  dim3 grid((unsigned)chunks * (unsigned)rows);
  if (logits_dtype == RECG_DTYPE_BF16)
    verify_partial_kernel<__nv_bfloat16>
        <<<grid, kVerifyThreads, 0, st>>>(static_cast<const __nv_bfloat16*>(logits), vocab, chunk_len, chunks, scratch, nullptr);
  else
    verify_partial_kernel<float><<<grid, kVerifyThreads, 0, st>>>(static_cast<const float*>(logits), vocab, chunk_len,
                                                                  chunks, scratch, nullptr);
  cudaError_t e = cudaGetLastError();   // nothing reads the scratch unless the scan was launched
  if (e != cudaSuccess) return fail(RECG_ERR_CUDA, std::string("recg_row_stats_static: launch: ") + cudaGetErrorString(e));
  const int lanes = stat_lanes(chunks);
  row_stats_finalize_kernel<<<(unsigned)(((size_t)rows * lanes + 127) / 128), 128, 0, st>>>(scratch, rows, chunks, lanes, top1, top2,
                                                                                         p1, p2, entropy);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(RECG_ERR_CUDA, std::string("recg_row_stats_static: launch: ") + cudaGetErrorString(e));
  return RECG_OK;
}
