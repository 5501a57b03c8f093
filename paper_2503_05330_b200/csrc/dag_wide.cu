// Follower gather, DAG aggregation (Eq. 5) and the greedy walk for queries with many matches on prompts that do not take the
// single-launch build, spread over the whole device.
//
// One CTA that aggregates a query of thousands of matches by itself takes hundreds of microseconds while the other SMs idle,
// so dag_kernel hands such queries over (wide_register).  First all CTAs lay the followers of all candidates out layer by layer.
// Then (query, layer) pairs are tasks that come from a counter, heavy queries first, each done by one CTA in its shared memory:
//   sums    followers and probabilities of the layer, summed up per token in a hash table
//   offers  a second table, by the token of the layer before: the heaviest node among its successors, found in three 32-bit
//           maxima (upper and lower word of the weight, then the smaller token), and the sums of the edge to it
// so that every candidate has the best successor of the node it comes from, as the index of one candidate on it, and the CTA
// that completes the last layer of a query walks it with one dependent load per layer.  Queries above wide_alone() matches: the
// sums only, a task per class of tokens (a table holds at most 16 384), and a walk that picks the candidates on the current node
// out of each layer's row.  Sums are integers and every choice has a tie rule, so the order in which things happen cannot show
// in a result.
//
// What bounds a task: the latency of its chain of shared-memory steps up to a few hundred candidates (8 K cycles), the shared-
// memory atomics beyond (a layer of 7300 candidates: 55 K cycles, of these 18 K claims and sums, 20 K offers).  The form before
// (node tables in global memory, five passes with grid barriers between them) took 32 us for one query of 200 matches and
// D = 16 against 22 here, 165 against 50 for one of 8000, and 1.3 to 2.6 KB of tables per match, so that 16 prompts of
// 128 x 4096 tokens, 420 000 matches at k = 1, overran the area and kept one CTA each for their largest queries (1.2 ms).
// Also measured: a task for all queries above wide_alone() by a cluster of 8 CTAs with the table in distributed shared memory
// (26 270 matches: 187 us against 250, but 8 times slower than classes as soon as there are tasks for all CTAs, and 3 us for every
// launch that has nothing to do); slots, tokens and weights of 64 candidates per thread (spills; 546 us); N table accesses of a
// thread on their way together, predicated (no change: the atomics' throughput is what counts).
#include <climits>
#include "sdms_internal.h"
#include "wide_dev.cuh"

namespace sdms {

namespace {

constexpr int kWideSmem = kWideSlots * 12;
constexpr int kWideWarps = kWideThreads / 32;
constexpr long long kWideWait = 1ll << 32;            // cycles, about two seconds
constexpr int kSortFrom = 256;                       // more queries than this balance without an order

__device__ __forceinline__ u64 ld_u64(const u64* p) { return __ldcg(p); }

// A wait for a count, bounded in cycles.
__device__ __forceinline__ bool wait_for_count(const u64* ctr, u64 target, long long cycles) {
  const long long t0 = clock64();
  while (ld_u64(ctr) < target) {
    if (clock64() - t0 > cycles) return false;
    __nanosleep(20);
  }
  return true;
}

// sdms_debug_wait_timeout: a bounded wait on a count that nobody raises.
__global__ void wait_timeout_kernel(Dev s, long long cycles) {
  if (threadIdx.x == 0 && !wait_for_count(s.b_ctl + kBeamNever, ~0ull, cycles)) atomicOr(s.status, SDMS_STATUS_TIMEOUT);
}

// What is kept for a query, in rows of `pitch` entries, one for every layer:
//   tok    the candidates' followers (-1: ended), from dag_rows_kernel
//   out    first their probabilities (32 bits each, the first half of the row), then node weights, in the end for those
//          candidates that are named by others what the draft says of them (score, weight of the edge from the node before)
//   succ   the best successor of the node that the candidate was on at the layer before (a candidate on it; -1: none).  Queries
//          of more than wide_alone() matches have no such row.
struct WideItems { u64* out; int* tok; int* succ; int pitch; };
__device__ __forceinline__ WideItems wide_items(const Dev& s, int first, int M) {
  WideItems w;
  w.pitch = wide_pitch(M);
  const size_t n = (size_t)s.D * w.pitch;
  w.out = reinterpret_cast<u64*>(s.w_tab + (unsigned)first);
  w.tok = reinterpret_cast<int*>(w.out + n);
  w.succ = w.tok + n;
  return w;
}
__device__ __forceinline__ u64 wide_out(const Dev& s, u64 weight, u64 edge_sum, unsigned edge_count) {
  const float score = s.alpha == 1.0 ? (float)eq5_weight(1.0, weight, 0u) : (float)__longlong_as_double((long long)weight);
  const float edge = s.mode == 1 ? 0.0f : (float)eq5_weight(s.alpha, edge_sum, edge_count);
  return (u64)__float_as_uint(edge) << 32 | __float_as_uint(score);
}
__device__ __forceinline__ unsigned wide_class(int v) { return ((unsigned)v * 0x85ebca6bu) >> 8; }

// The table of one layer in shared memory.
struct WideTable { int* key; unsigned* lo; unsigned* hi; unsigned* cnt; int mask, shift; };   // sums of the lower 15 bits, of the rest, counts
__device__ __forceinline__ WideTable wide_table(unsigned char* smem, int cap) {
  WideTable t;
  t.key = reinterpret_cast<int*>(smem);
  t.lo = reinterpret_cast<unsigned*>(t.key + cap); t.hi = t.lo + cap; t.cnt = t.hi + cap;
  t.mask = cap - 1; t.shift = __clz(cap) + 1;
  return t;
}
__device__ __forceinline__ void wide_table_empty(unsigned char* smem, int cap, bool counts) {
  int4* const z = reinterpret_cast<int4*>(smem);
  const int k4 = cap / 4, end = (counts ? 4 : 3) * k4;
  for (int x = threadIdx.x; x < k4; x += kWideThreads) z[x] = make_int4(-1, -1, -1, -1);
  for (int x = k4 + threadIdx.x; x < end; x += kWideThreads) z[x] = make_int4(0, 0, 0, 0);
}
// Slot of token v, claimed if need be; -1: the table is full.
__device__ __forceinline__ int wide_claim(const WideTable& t, int v) {
  unsigned h = ((unsigned)v * 2654435761u) >> t.shift;
#pragma unroll 1
  for (int probe = 0; probe <= t.mask; ++probe) {
    int k = *(volatile int*)&t.key[h];
    if (k == -1) k = atomicCAS(&t.key[h], -1, v);
    if (k == -1 || k == v) return (int)h;
    h = (h + 1) & t.mask;
  }
  return -1;
}
__device__ __forceinline__ void wide_add(const WideTable& t, int h, unsigned p, bool counts) {
  atomicAdd(&t.lo[h], p & 0x7fffu);
  atomicAdd(&t.hi[h], p >> 15);
  if (counts) atomicAdd(&t.cnt[h], 1u);
}
__device__ __forceinline__ u64 wide_weight(const Dev& s, const WideTable& t, int h, bool counts) {
  const u64 S = ((u64)t.hi[h] << 15) + t.lo[h];
  return counts ? (u64)__double_as_longlong(eq5_weight(s.alpha, S, t.cnt[h])) : S;
}
// (The match list is read past L1 throughout: the kernel before this one still cuts it down in place, with a cap on the
// matches per path, while CTAs of this one are resident.  Tokens, probabilities and lengths are older and go through __ldg.)
// Entries m0, m0 + kWideThreads, ... of a row (`none` where there is no candidate).
template <int N>
__device__ __forceinline__ void wide_row(const int* row, int M, int m0, int none, int (&v)[N]) {
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = m0 + r * kWideThreads < M ? __ldcg(row + m0 + r * kWideThreads) : none;
}

// ---- the followers of all candidates, layer by layer ---------------------------------------------------------------
// A candidate's followers lie next to each other in the store, a task wants one of each candidate.  Fetched by the tasks, each
// layer and each step on its own, they were 3 to 4 sectors of 32 bytes per (candidate, layer), and those were what a task
// waited for (40 of the 90 K cycles of a layer of 7300 candidates).  Here a thread reads a candidate's followers and
// probabilities, 16 aligned bytes at a time, and lays them out in rows.
__device__ __forceinline__ int4 shifted(int4 a, int4 b, int off) {      // words off .. off + 3 of a, b
  if (off & 2) { a.x = a.z; a.y = a.w; a.z = b.x; a.w = b.y; b.x = b.z; }
  if (off & 1) { a.x = a.y; a.y = a.z; a.z = a.w; a.w = b.x; }
  return a;
}
// Candidates c0 .. c0 + kWideThreads of a query, their followers l0 .. l1 (a multiple of 4 each, or D).  The loads of 16 layers go out
// together: one after the other they were 32 K cycles out of a cold cache, for 13 chunks of a few hundred candidates.
__device__ __forceinline__ void wide_lay_out(const Dev& s, const int4 de, int c0, int l0, int l1) {
  const int M = de.y, m = c0 + threadIdx.x;
  if (m >= M) return;
  const WideItems items = wide_items(s, de.z, M);
  const int g = __ldcg(s.matches + s.q_off[de.x] + m), j = path_of(s, g);
  const int n = min(l1, __ldg(s.len + j) - 1 - (g - j * s.L));         // followers
  const int off = (g + 1) & 3;
  const int4* const st = reinterpret_cast<const int4*>(s.tok) + ((g + 1) >> 2);
  const int4* const sp = reinterpret_cast<const int4*>(s.pq) + ((g + 1) >> 2);
#pragma unroll 1
  for (int lb = l0; lb < l1; lb += 16) {
    int4 a[5], c[5];                                                   // 16 bytes each of tokens and probabilities
#pragma unroll
    for (int x = 0; x < 5; ++x) {
      a[x] = make_int4(0, 0, 0, 0); c[x] = a[x];
      const int at = lb + 4 * x - off;                                 // the first follower in them
      if (at < n && at < lb + 16) { a[x] = __ldg(st + (lb >> 2) + x); c[x] = __ldg(sp + (lb >> 2) + x); }   // (only what holds a follower)
    }
    int* tok = items.tok + (size_t)lb * items.pitch + m;
    int* p = reinterpret_cast<int*>(items.out + (size_t)lb * items.pitch) + m;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int4 v = shifted(a[x], a[x + 1], off), q = shifted(c[x], c[x + 1], off);
      const int vs[4] = {v.x, v.y, v.z, v.w}, ps[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int l = lb + 4 * x + y;
        if (l < l1) { *tok = l < n ? vs[y] : -1; *p = ps[y]; }
        tok += items.pitch; p += 2 * items.pitch;
      }
    }
  }
}

// Layer d of a query with at most N * CH * kWideThreads candidates.  Slots and tokens stay in registers, with KEEP weights too
// (else they are read again from where they were left).
template <int N, int CH, bool KEEP>
__device__ __forceinline__ void wide_layer(const Dev& s, const int4 de, int d) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  static_assert(N * CH <= 32, "one bit per candidate");
  const int tid = threadIdx.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems items = wide_items(s, de.z, M);
  u64* const weight = items.out + (size_t)(d - 1) * items.pitch;
  const int* const row = items.tok + (size_t)(d - 1) * items.pitch;
  const int* const row_p = reinterpret_cast<const int*>(weight);
  const bool counts = s.alpha != 1.0;                  // with alpha = 1 a weight does not depend on the count
  // At most half full where there is room for that, in any case 7/8: a CTA waits for its unluckiest lane's probe sequence (a layer
  // of 862 candidates: 47 to 58 K cycles in 1024 slots, 16 K in 2048).
  const int most = counts ? kWideSlots / 2 : kWideSlots;
  int cap = 64;
  while (cap < 2 * M && cap < most) cap *= 2;
  const WideTable t = wide_table(wide_smem, cap);
  int v[N], p[N];
  wide_row<N>(row, M, tid, -1, v);                     // on its way while the table is emptied
  wide_row<N>(row_p, M, tid, 0, p);
  wide_table_empty(wide_smem, cap, counts);
  __syncthreads();
  // ---- sums
  int slot[CH][N];
  int kt[CH][N];                                       // tokens and weights
  u64 kw[KEEP ? CH : 1][N];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int m0 = c * N * kWideThreads + tid;
    if (c > 0) { wide_row<N>(row, M, m0, -1, v); wide_row<N>(row_p, M, m0, 0, p); }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      kt[c][r] = v[r];
      slot[c][r] = -1;
      if (v[r] < 0) continue;
      slot[c][r] = wide_claim(t, v[r]);
      wide_add(t, slot[c][r], p[r], counts);
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r) {
      if (KEEP) kw[KEEP ? c : 0][r] = 0ull;
      if (slot[c][r] < 0) continue;
      const u64 w = wide_weight(s, t, slot[c][r], counts);
      if (KEEP) kw[KEEP ? c : 0][r] = w;
      else weight[(c * N + r) * kWideThreads + tid] = w;
    }
  __syncthreads();
  // ---- offers.  slot becomes that of the node before (-1: the candidate was not on one)
  const bool single = d == 1 || s.mode == 1;           // all successors of the root / of no node in particular
  for (int x = tid; x < (single ? 1 : cap); x += kWideThreads) { t.key[x] = -1; t.lo[x] = 0u; t.hi[x] = 0u; }
  __syncthreads();
  unsigned alive = 0u, best = 0u, named = 0u;         // bit c * N + r: has a token; is on the best successor; is the one that is named
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int m0 = c * N * kWideThreads + tid;
    if (!single) wide_row<N>(row - items.pitch, M, m0, -1, v);
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int m = m0 + r * kWideThreads;
      alive |= (unsigned)(slot[c][r] >= 0) << (c * N + r);
      slot[c][r] = m >= M || (!single && v[r] < 0) ? -1 : single ? 0 : wide_claim(t, v[r]);
    }
  }
  __syncthreads();
  auto weight_of = [&](int c, int r) { return KEEP ? kw[KEEP ? c : 0][r] : weight[(c * N + r) * kWideThreads + tid]; };
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (alive >> (c * N + r) & 1u) {
        const unsigned x = (unsigned)(weight_of(c, r) >> 32);
        if (*(volatile unsigned*)&t.hi[slot[c][r]] < x) atomicMax(&t.hi[slot[c][r]], x);
      }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (alive >> (c * N + r) & 1u) {
        const u64 w = weight_of(c, r);
        if (t.hi[slot[c][r]] == (unsigned)(w >> 32) && *(volatile unsigned*)&t.lo[slot[c][r]] < (unsigned)w) atomicMax(&t.lo[slot[c][r]], (unsigned)w);
      }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (alive >> (c * N + r) & 1u) {
        const u64 w = weight_of(c, r);
        best |= (unsigned)(t.hi[slot[c][r]] == (unsigned)(w >> 32) && t.lo[slot[c][r]] == (unsigned)w) << (c * N + r);
      }
  __syncthreads();
  for (int x = tid; x < (single ? 1 : cap); x += kWideThreads) { t.hi[x] = 0u; t.lo[x] = ~0u; }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (best >> (c * N + r) & 1u) {
        const unsigned x = ~(unsigned)kt[c][r];   // the smallest token is the largest complement
        if (*(volatile unsigned*)&t.hi[slot[c][r]] < x) atomicMax(&t.hi[slot[c][r]], x);
      }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (best >> (c * N + r) & 1u) {
        if (t.hi[slot[c][r]] == ~(unsigned)kt[c][r]) t.lo[slot[c][r]] = (unsigned)((c * N + r) * kWideThreads + tid);   // any one of them
        else best &= ~(1u << (c * N + r));
      }
  __syncthreads();
  int* const succ = items.succ + (size_t)(d - 1) * items.pitch;
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (slot[c][r] >= 0) {
        const int m = (c * N + r) * kWideThreads + tid, to = (int)t.lo[slot[c][r]];
        succ[m] = to;
        named |= (unsigned)(to == m) << (c * N + r);
      }
  __syncthreads();
  for (int x = tid; x < (single ? 1 : cap); x += kWideThreads) { t.hi[x] = 0u; t.lo[x] = 0u; t.key[x] = 0; }
  __syncthreads();
  // the edge to the best successor: in layer-wise search it counts only for candidates that were on the winner's own node, which
  // is not known here: the walk adds it up
  if (s.mode != 1) {
    unsigned lo = 0u, hi = 0u;
#pragma unroll
    for (int c = 0; c < CH; ++c)
#pragma unroll
      for (int r = 0; r < N; ++r)
        if (best >> (c * N + r) & 1u) {
          const int m = (c * N + r) * kWideThreads + tid;
          const unsigned q = (unsigned)(KEEP ? __ldcg(row_p + m) : __ldg(s.pq + __ldcg(list + m) + d));
          if (single) { lo += q & 0x7fffu; hi += q >> 15; }
          else {
            atomicAdd(&t.lo[slot[c][r]], q & 0x7fffu);
            atomicAdd(&t.hi[slot[c][r]], q >> 15);
            atomicAdd(&t.key[slot[c][r]], 1);
          }
        }
    if (single) {                                      // one edge for all
      lo = __reduce_add_sync(FULL, lo); hi = __reduce_add_sync(FULL, hi);
      const unsigned n = __reduce_add_sync(FULL, (unsigned)__popc(best));
      if ((tid & 31) == 0 && n) { atomicAdd(&t.lo[0], lo); atomicAdd(&t.hi[0], hi); atomicAdd(&t.key[0], (int)n); }
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (named >> (c * N + r) & 1u) {
        const int x = slot[c][r], m = (c * N + r) * kWideThreads + tid;
        const u64 w = weight_of(c, r);
        weight[m] = wide_out(s, w, ((u64)t.hi[x] << 15) + t.lo[x], (unsigned)t.key[x]);
      }
}

__device__ __forceinline__ void wide_task(const Dev& s, const int4 de, int d) {
  const int M = de.y;
  if (M <= 4 * kWideThreads) wide_layer<4, 1, true>(s, de, d);
  else if (M <= 16 * kWideThreads) wide_layer<8, 2, true>(s, de, d);
  else wide_layer<7, 4, false>(s, de, d);
}

// ---- larger queries: sums only, one task per class of tokens ------------------------------------------------------
// Classes (a power of two): tables at most 7/8 full.
__device__ __forceinline__ int wide_classes(const Dev& s, int M) {
  if (M <= wide_alone(s)) return 1;
  int c = 2;
  while ((long long)c * wide_alone(s) < M) c *= 2;
  return c;
}
// Weights of the nodes of layer d with tokens of class `cls`.  A table that overruns all the same is done again in sub-classes.
__device__ __forceinline__ void wide_sums(const Dev& s, const int4 de, int d, unsigned cls, unsigned classes) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  __shared__ int sh_over;
  constexpr int N = 16;
  const int tid = threadIdx.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems rows = wide_items(s, de.z, M);
  u64* const weight = rows.out + (size_t)(d - 1) * rows.pitch;
  const int* const tok = rows.tok + (size_t)(d - 1) * rows.pitch;
  const bool counts = s.alpha != 1.0;
  const int cap = counts ? kWideSlots / 2 : kWideSlots;
  const WideTable t = wide_table(wide_smem, cap);
  unsigned subs = 1;
#pragma unroll 1
  for (unsigned sub = 0; sub < subs; ++sub) {
    const unsigned others = classes * subs - 1u, mine = cls + classes * sub;
    if (tid == 0) sh_over = 0;
    wide_table_empty(wide_smem, cap, counts);
    __syncthreads();
#pragma unroll 1
    for (int m0 = tid; m0 < M; m0 += N * kWideThreads) {
      int v[N];
      unsigned p[N];
      wide_row<N>(tok, M, m0, -1, v);
      if (cls == 0u) {
#pragma unroll
        for (int r = 0; r < N; ++r)
          if (v[r] < 0 && m0 + r * kWideThreads < M) weight[m0 + r * kWideThreads] = 0ull;   // (ended)
      }
#pragma unroll
      for (int r = 0; r < N; ++r)
        if ((wide_class(v[r]) & others) != mine) v[r] = -1;
      // (from the store: other classes write their weights over the row of probabilities)
#pragma unroll
      for (int r = 0; r < N; ++r) p[r] = v[r] >= 0 ? (unsigned)__ldcg(list + m0 + r * kWideThreads) : 0u;
#pragma unroll
      for (int r = 0; r < N; ++r) p[r] = v[r] >= 0 ? (unsigned)__ldg(s.pq + (int)p[r] + d) : 0u;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (v[r] < 0) continue;
        const int h = wide_claim(t, v[r]);
        if (h < 0) sh_over = 1;
        else wide_add(t, h, p[r], counts);
      }
    }
    __syncthreads();
    if (sh_over) {                                     // (the same for everybody)
      __syncthreads();
      subs *= 2; sub = ~0u;
      continue;
    }
#pragma unroll 1
    for (int m0 = tid; m0 < M; m0 += N * kWideThreads) {
      int v[N];
      wide_row<N>(tok, M, m0, -1, v);
#pragma unroll
      for (int r = 0; r < N; ++r)
        if (v[r] >= 0 && (wide_class(v[r]) & others) == mine) weight[m0 + r * kWideThreads] = wide_weight(s, t, wide_claim(t, v[r]), counts);
    }
    __syncthreads();
  }
}

// ---- the walk over a query whose layers are all done --------------------------------------------------------------
struct WideOut { int32_t* tok; int32_t* len; float* score; float* edge_w; };

__device__ __forceinline__ u64 warp_max64(u64 x) {
  const unsigned hi = (unsigned)(x >> 32), top = __reduce_max_sync(FULL, hi);
  const unsigned lo = __reduce_max_sync(FULL, hi == top ? (unsigned)x : 0u);
  return (u64)top << 32 | lo;
}
struct WideWalk {                        // what the walk over rows keeps in shared memory
  u64 best[kWideWarps];
  int tok[kWideWarps];
  int draft[SDMS_MAX_DRAFT];
  u64 weight[SDMS_MAX_DRAFT];
  unsigned e[SDMS_MAX_DRAFT][3];         // edge sums: lower 15 bits, rest, count
  int hits[2];
};

// Sums only: layer by layer the candidates on the current node are picked from its row into a list in shared memory (whose
// length does not depend on M, and is short for most nodes), their successors compared and the candidates on the edge
// taken weighed.  A list that overflows, and layer 1, where all are on the root, go over the rows instead.
__device__ __forceinline__ void wide_walk_rows(const Dev& s, const int4 de, const WideOut out) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  __shared__ WideWalk sh;
  constexpr int B = 8, kHits = kWideSmem / 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D, i = de.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[i];
  const WideItems rows = wide_items(s, de.z, M);
  int* const hit = reinterpret_cast<int*>(wide_smem);
  if (tid < SDMS_MAX_DRAFT) { sh.e[tid][0] = 0u; sh.e[tid][1] = 0u; sh.e[tid][2] = 0u; }
  if (tid == 0) { sh.hits[0] = 0; sh.hits[1] = 0; }
  __syncthreads();
  int cur = -1, emitted = 0;
#pragma unroll 1
  for (int d = 1; d <= D; ++d) {
    const int* const row = rows.tok + (size_t)(d - 1) * rows.pitch;
    const int* const before = row - rows.pitch;
    const u64* const row_w = rows.out + (size_t)(d - 1) * rows.pitch;
    const bool all = d == 1 || s.mode == 1;            // successors of the root / of no node in particular
    if (!all) {
#pragma unroll 1
      for (int x0 = 4 * tid; x0 < M; x0 += B * 4 * kWideThreads) {
        int4 u[B];
#pragma unroll
        for (int r = 0; r < B; ++r) {
          const int x = x0 + r * 4 * kWideThreads;
          u[r] = x < M ? __ldcg(reinterpret_cast<const int4*>(before + x)) : make_int4(-1, -1, -1, -1);
          if (x + 1 >= M) u[r].y = -1;
          if (x + 2 >= M) u[r].z = -1;
          if (x + 3 >= M) u[r].w = -1;
        }
        unsigned on = 0u;
#pragma unroll
        for (int r = 0; r < B; ++r)
          on |= ((unsigned)(u[r].x == cur) | (unsigned)(u[r].y == cur) << 1 | (unsigned)(u[r].z == cur) << 2 | (unsigned)(u[r].w == cur) << 3) << (4 * r);
        if (on == 0u) continue;
        int at = atomicAdd(&sh.hits[d & 1], __popc(on));
        for (; on && at < kHits; on &= on - 1u, ++at) {
          const int bit = __ffs(on) - 1;
          hit[at] = x0 + (bit >> 2) * 4 * kWideThreads + (bit & 3);
        }
      }
      __syncthreads();
    }
    const int hits = all ? M : sh.hits[d & 1];
    const bool listed = !all && hits <= kHits;
    const int n = listed ? hits : M;
    if (tid == 0) sh.hits[(d + 1) & 1] = 0;
    // The heaviest successor, the smallest token of those, the edge to it: weights of all hits, tokens only of the heaviest,
    // probabilities only on the edge (what a CTA gathers from L2 takes 2 cycles per sector).  Read again for each step if there
    // are more hits than are kept in registers.
    const bool again = n > B * kWideThreads;
    int m[B], t[B];
    u64 w[B];
    auto load_weights = [&](int x0) {
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const int x = x0 + r * kWideThreads;
        m[r] = x >= n ? -1 : listed ? hit[x] : x;
        if (!all && !listed && m[r] >= 0 && __ldcg(before + m[r]) != cur) m[r] = -1;
        w[r] = m[r] >= 0 ? ld_u64(row_w + m[r]) : 0ull;
      }
    };
    u64 best = 0ull;
    auto load_tokens = [&]() {
#pragma unroll
      for (int r = 0; r < B; ++r) t[r] = m[r] >= 0 && w[r] == best ? __ldcg(row + m[r]) : -1;
    };
#pragma unroll 1
    for (int x0 = tid; x0 - tid < n; x0 += B * kWideThreads) {
      load_weights(x0);
#pragma unroll
      for (int r = 0; r < B; ++r) best = w[r] > best ? w[r] : best;
    }
    best = warp_max64(best);
    if (lane == 0) sh.best[warp] = best;
    __syncthreads();
    best = warp_max64(lane < kWideWarps ? sh.best[lane] : 0ull);
    int tok = INT_MAX;
#pragma unroll 1
    for (int x0 = tid; x0 - tid < n; x0 += B * kWideThreads) {
      if (again) load_weights(x0);
      load_tokens();
#pragma unroll
      for (int r = 0; r < B; ++r) tok = t[r] >= 0 && t[r] < tok ? t[r] : tok;        // (a candidate that has ended weighs nothing)
    }
    tok = (int)__reduce_min_sync(FULL, (unsigned)tok);
    if (lane == 0) sh.tok[warp] = tok;
    __syncthreads();
    tok = (int)__reduce_min_sync(FULL, (unsigned)(lane < kWideWarps ? sh.tok[lane] : INT_MAX));
    if (tok == INT_MAX) break;                         // no successor: the draft ends here
    unsigned lo = 0u, hi = 0u, count = 0u;
#pragma unroll 1
    for (int x0 = tid; x0 - tid < n; x0 += B * kWideThreads) {
      if (again) { load_weights(x0); load_tokens(); }
      int g[B];
      unsigned p[B];
#pragma unroll
      for (int r = 0; r < B; ++r) {
        // (layer-wise search looks at all candidates, but the edge is from the node before)
        const bool on = t[r] == tok && (!all || d == 1 || __ldcg(before + m[r]) == cur);
        g[r] = on ? __ldcg(list + m[r]) : -1;
      }
#pragma unroll
      for (int r = 0; r < B; ++r) p[r] = g[r] >= 0 ? (unsigned)__ldg(s.pq + g[r] + d) : 0u;
#pragma unroll
      for (int r = 0; r < B; ++r) { lo += p[r] & 0x7fffu; hi += p[r] >> 15; count += g[r] >= 0; }
    }
    lo = __reduce_add_sync(FULL, lo); hi = __reduce_add_sync(FULL, hi); count = __reduce_add_sync(FULL, count);
    if (lane == 0 && count) { atomicAdd(&sh.e[d - 1][0], lo); atomicAdd(&sh.e[d - 1][1], hi); atomicAdd(&sh.e[d - 1][2], count); }
    if (tid == 0) { sh.draft[d - 1] = tok; sh.weight[d - 1] = best; }
    cur = tok; emitted = d;
    __syncthreads();                                   // before the next layer's list
  }
  __syncthreads();
  if (tid < D) {
    const size_t x = (size_t)i * D + tid;
    const bool on = tid < emitted;
    out.tok[x] = on ? sh.draft[tid] : -1;
    if (out.score)
      out.score[x] = !on ? 0.0f : s.alpha == 1.0 ? (float)eq5_weight(1.0, sh.weight[tid], 0u)
                                                 : (float)__longlong_as_double((long long)sh.weight[tid]);
    if (out.edge_w) out.edge_w[x] = on ? (float)eq5_weight(s.alpha, ((u64)sh.e[tid][1] << 15) + sh.e[tid][0], sh.e[tid][2]) : 0.0f;
  }
  if (tid == 0) out.len[i] = emitted;
}
// Successors known: one dependent load per layer.

__device__ __forceinline__ void wide_walk_known(const Dev& s, const int4 de, const WideOut out) {
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_e[SDMS_MAX_DRAFT][3];         // layer-wise search: edge sums (lower 15 bits, rest) and counts
  static_assert(SDMS_MAX_DRAFT <= 32, "a lane per layer");
  const int tid = threadIdx.x, D = s.D, i = de.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[i];
  const WideItems items = wide_items(s, de.z, M);
  if (s.mode == 1 && out.edge_w) {                     // the edges are known only now
    if (tid < 32) { sh_draft[tid] = -1; sh_e[tid][0] = 0u; sh_e[tid][1] = 0u; sh_e[tid][2] = 0u; }
    __syncthreads();
    if (tid < D) { const int at = __ldcg(items.succ + (size_t)tid * items.pitch); if (at >= 0) sh_draft[tid] = __ldcg(items.tok + (size_t)tid * items.pitch + at); }
    __syncthreads();
    for (int m = tid; m < M; m += kWideThreads) {
      const int g = __ldcg(list + m), j = path_of(s, g), n = min(D, __ldg(s.len + j) - 1 - (g - j * s.L));
      bool on = true;                                  // this candidate is on the draft's node so far
      for (int l = 0; l < n && sh_draft[l] >= 0; ++l) {
        const bool here = __ldg(s.tok + g + l + 1) == sh_draft[l];
        if (on && here) {
          const unsigned q = (unsigned)__ldg(s.pq + g + l + 1);
          atomicAdd(&sh_e[l][0], q & 0x7fffu); atomicAdd(&sh_e[l][1], q >> 15); atomicAdd(&sh_e[l][2], 1u);
        }
        on = here;
      }
    }
    __syncthreads();
  }
  if (tid < 32) {
    int at = __ldcg(items.succ), emitted = 0, mine = -1;               // every candidate of layer 1 names the root's best
#pragma unroll 1
    for (int d = 1; d <= D && at >= 0; ++d) {
      if (tid == d - 1) mine = at;
      emitted = d;
      at = d < D ? __ldcg(items.succ + (size_t)d * items.pitch + at) : -1;
    }
    if (tid < D) {
      const size_t x = (size_t)i * D + tid, y = (size_t)tid * items.pitch + max(mine, 0);
      const bool on = mine >= 0;
      const int v = on ? __ldcg(items.tok + y) : -1;
      const u64 o = ld_u64(items.out + y);
      out.tok[x] = v;
      if (out.score) out.score[x] = on ? __uint_as_float((unsigned)o) : 0.0f;
      if (out.edge_w)
        out.edge_w[x] = !on ? 0.0f
                        : s.mode == 1 ? (float)eq5_weight(s.alpha, ((u64)sh_e[tid][1] << 15) + sh_e[tid][0], sh_e[tid][2])
                                      : __uint_as_float((unsigned)(o >> 32));
    }
    if (tid == 0) out.len[i] = emitted;
  }
}

__device__ __forceinline__ void wide_walk(const Dev& s, const int4 de, const WideOut out) {
  if (de.y <= wide_alone(s)) wide_walk_known(s, de, out);
  else wide_walk_rows(s, de, out);
  if (s.beam_stride > 0) {                             // the beams want the table area empty
    __syncthreads();
    uint4* const z = reinterpret_cast<uint4*>(s.w_tab + (unsigned)de.z);
    for (size_t x = threadIdx.x; x < (size_t)wide_slots(s, de.y) * 2; x += kWideThreads) z[x] = make_uint4(0u, 0u, 0u, 0u);
  }
}

__global__ void __launch_bounds__(kWideThreads, 1)
dag_wide_kernel(Dev s, int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  grid_wait();                                         // scheduled while dag_kernel drains; its list is complete from here on
  const u64 registered = ld_u64(&s.w_ctl[0]);
  if (registered == 0) return;
  const int nq = (int)(registered < (u64)kMaxWide ? registered : (u64)kMaxWide);
  __shared__ int4 sh_desc[kMaxWide];
  __shared__ int sh_base[kMaxWide + 1];                // first task of each query
  __shared__ int sh_unit[kMaxWide + 1];                // first chunk of kWideThreads candidates of each query
  __shared__ int sh_warp[kWideWarps];
  __shared__ int sh_task, sh_last, sh_large;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D;
  int spread;
  if (tid == 0) sh_large = 0;
  static_assert(kMaxWide == 2 * kWideThreads, "two list entries per thread");
  // the list of queries, the largest first, and by prefix sums the first task and the first chunk of each
  {
    int4 de[2];
    int rank[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int q = 2 * tid + r;
      de[r] = q < nq ? __ldcg(&s.w_desc[q]) : make_int4(0, 0, 0, 0);
      if (q < nq) sh_desc[q] = de[r];
      rank[r] = q;
    }
    __syncthreads();
    if (nq > 1 && nq <= kSortFrom) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int q = 2 * tid + r;
        if (q >= nq) continue;
        rank[r] = 0;
        for (int x = 0; x < nq; ++x) {
          const int m = sh_desc[x].y;
          rank[r] += m > de[r].y || (m == de[r].y && x < q);
        }
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (2 * tid + r < nq) sh_desc[rank[r]] = make_int4(de[r].x, de[r].y, de[r].z, 2 * tid + r);
    } else {
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (2 * tid + r < nq) sh_desc[2 * tid + r].w = 2 * tid + r;
    }
    __syncthreads();
    int c[2], large = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int M = 2 * tid + r < nq ? sh_desc[2 * tid + r].y : 0;
      c[r] = M > 0 ? D * wide_classes(s, M) : 0;
      if (M > wide_alone(s)) large += c[r];
    }
    if (large) atomicAdd(&sh_large, large);
    __syncthreads();
    // more and smaller classes while the large queries' tasks leave most of the CTAs without work (one query of 26 270 matches,
    // D = 16: 333 us with 32 tasks, 250 with 128; where there are tasks for all CTAs four times the classes are 1.4 to 1.8 times the
    // work: 16 prompts of 128 x 4096 tokens, k = 1, 1.39 against 2.44 ms)
    spread = 1;
    while (spread < 4 && sh_large > 0 && 2 * spread * sh_large <= (int)gridDim.x) spread *= 2;
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (2 * tid + r < nq && sh_desc[2 * tid + r].y > wide_alone(s)) c[r] *= spread;
    auto prefix = [&](int c0, int c1, int* first) {    // first[q] = sum of the counts before q, for two queries per thread
      int x = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(FULL, x, o); if (lane >= o) x += y; }
      if (lane == 31) sh_warp[warp] = x;
      __syncthreads();
      if (warp == 0) {
        int w = lane < kWideWarps ? sh_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(FULL, w, o); if (lane >= o) w += y; }
        if (lane < kWideWarps) sh_warp[lane] = w;
      }
      __syncthreads();
      const int ahead = (warp ? sh_warp[warp - 1] : 0) + x - c0 - c1;
      first[2 * tid] = ahead;
      first[2 * tid + 1] = ahead + c0;
      if (tid == kWideThreads - 1) first[kMaxWide] = ahead + c0 + c1;
      __syncthreads();
    };
    prefix(c[0], c[1], sh_base);
#pragma unroll
    for (int r = 0; r < 2; ++r) c[r] = 2 * tid + r < nq ? (sh_desc[2 * tid + r].y + kWideThreads - 1) / kWideThreads : 0;
    prefix(c[0], c[1], sh_unit);
  }
  auto owner = [&](const int* first, int x) {          // first[owner] <= x < first[owner + 1], of those that are not empty
    int a = 0, b = nq;
    while (b - a > 1) { const int mid = (a + b) >> 1; if (first[mid] <= x) a = mid; else b = mid; }
    return a;
  };
  // Everybody lays out rows, then waits until all rows are there.  Chunks come from a counter, so that the wait is for running
  // CTAs only, whatever else is on the device; it is bounded all the same.
  const int whole = sh_unit[nq], quads = (D + 3) >> 2;
  int parts = 1;                                       // a chunk is split by layers while that gives more CTAs something to do
  while (parts < quads && 2 * parts * whole <= (int)gridDim.x) parts *= 2;
  const int units = whole * parts, span = 4 * ((quads + parts - 1) / parts);
  if (tid == 0) sh_task = (int)atomicAdd(&s.w_ctl[3], 1ull);
  __syncthreads();
#pragma unroll 1
  for (int unit = sh_task; unit < units;) {
    __syncthreads();
    if (tid == 0) sh_task = (int)atomicAdd(&s.w_ctl[3], 1ull);         // (on its way during this one)
    const int chunk = unit / parts, l0 = (unit - chunk * parts) * span;
    const int q = owner(sh_unit, chunk);
    if (l0 < D) wide_lay_out(s, sh_desc[q], (chunk - sh_unit[q]) * kWideThreads, l0, min(D, l0 + span));
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(&s.w_ctl[4], 1ull);
    unit = sh_task;
  }
  __syncthreads();
  if (tid == 0) {
    sh_last = wait_for_count(s.w_ctl + 4, (u64)units, kWideWait);
    if (sh_last) sh_task = (int)atomicAdd(&s.w_ctl[2], 1ull);          // (whoever gives up here leaves no task undone)
  }
  __syncthreads();
  if (!sh_last) {
    if (tid == 0) atomicOr(s.status, SDMS_STATUS_TIMEOUT);
    return;
  }
  __threadfence();
  const int tasks = sh_base[nq];
  int task = sh_task;
  __syncthreads();
#pragma unroll 1
  while (task < tasks) {
    const int a = owner(sh_base, task);
    const int4 de = sh_desc[a];
    const int classes = wide_classes(s, de.y) * (de.y > wide_alone(s) ? spread : 1), part = task - sh_base[a];
    if (de.y <= wide_alone(s)) wide_task(s, de, part + 1);
    else wide_sums(s, de, part / classes + 1, (unsigned)(part % classes), (unsigned)classes);
    // done with it: its results are out before it is counted, and whoever counts the last one has seen all of them
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      sh_task = (int)atomicAdd(&s.w_ctl[2], 1ull);
      const int total = D * classes;
      sh_last = atomicAdd(&s.w_done[de.w], 1) == total - 1;
      if (sh_last) s.w_done[de.w] = 0;                 // the next build finds it at zero
      __threadfence();
    }
    __syncthreads();
    if (sh_last) wide_walk(s, de, WideOut{draft_tok, draft_len, draft_score, draft_edge_w});
    task = sh_task;
    __syncthreads();
  }
}

}  // namespace

// CTAs of the wide pass on the current device (0: it is not used).
int wide_kernel_grid() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(dag_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return sms;
}

cudaError_t launch_wait_timeout(const Dev& s, long long cycles, cudaStream_t stream) {
  wait_timeout_kernel<<<1, 32, 0, stream>>>(s, cycles);
  return cudaGetLastError();
}

cudaError_t launch_dag_wide(const Dev& s, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                            float* draft_edge_w, cudaStream_t stream) {
  return launch_overlapped(dag_wide_kernel, dim3(s.w_grid), dim3(kWideThreads), kWideSmem, stream, s, draft_tok, draft_len,
                           draft_score, draft_edge_w);
}

}  // namespace sdms
