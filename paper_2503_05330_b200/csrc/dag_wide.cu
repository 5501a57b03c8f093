// Follower gather, DAG aggregation (Eq. 5) and the greedy walk for queries with many matches, spread over the whole device: on prompts that do not
// take the single-launch build, and behind that build or step for its heaviest queries (hand_over_from, dag.cu).
//
// One CTA that aggregates a query of thousands of matches by itself takes hundreds of microseconds while the other SMs idle,
// so dag_kernel and the single-launch kernels hand such queries over (wide_register).  First all CTAs lay the followers of all candidates out layer by layer.
// Then (query, layer) pairs are tasks that come from a counter, heavy queries first, each done by one CTA in its shared memory:
//   sums    followers and probabilities of the layer, summed up per token in a hash table
//   offers  a second table, by the token of the layer before: the heaviest node among its successors, found in three 32-bit
//           maxima (upper and lower word of the weight, then the smaller token), and the sums of the edge to it
// so that every candidate has the best successor of the node it comes from, as the index of one candidate on it, and the CTA
// that completes the last layer of a query walks it with one dependent load per layer.  Queries above wide_alone() matches: a
// task per class of tokens (a table holds at most 8192 nodes) for the sums, and while such queries are few a second one for the
// offers, else a walk that picks the candidates on the current node out of each layer's row.  Sums are integers and every choice
// has a tie rule, so the order in which things happen cannot show in a result.
//
// What bounds a task: the latency of its chain of shared-memory steps up to a few hundred candidates (8 K cycles), the shared-
// memory atomics beyond (a layer of 7300 candidates: 55 K cycles, of these 18 K claims and sums, 20 K offers).  The form before
// (node tables in global memory, five passes with grid barriers between them) took 32 us for one query of 200 matches and
// D = 16 against 22 here, and 1.3 to 2.6 KB of tables per match, so that 16 prompts of 128 x 4096 tokens, 420 000 matches at
// k = 1, overran the area and kept one CTA each for their largest queries (1.2 ms).  k = 1 builds of 256 x 8192 tokens, queries of up to
// 26 236 matches (three inputs): 225 / 227 / 261 us in that form, 291 / 280 / 292 with a walk over rows by one CTA for the
// largest queries (326 K cycles), 174 / 214 / 233 with their offers; layer-wise search 264, 681, 175.
// Also measured: a task for all queries above wide_alone() by a cluster of 8 CTAs with the table in distributed shared memory
// (8 times slower than classes as soon as there are tasks for all CTAs, and 3 us for every launch that has nothing to do); slots,
// tokens and weights of 64 candidates per thread (spills; 546 us); N table accesses of a thread on their way together,
// predicated (no change: the atomics' throughput is what counts); in the class tasks, lanes on one node that add and raise together (sums
// 5.2 -> 6.8, offers 16.7 -> 22 M cycles in all: the ballots and reductions cost more than the atomics they save), 2048 candidates
// per class instead of 4096 (248 for 215 us), all queries from 2048 matches on by classes (40 x 4096 tokens, one query of
// 4773 matches: 90 for 67 us).
#include <climits>
#include "sdms_internal.h"
#include "wide_dev.cuh"

namespace sdms {

namespace {

constexpr int kWideSmem = kWideSlots * 12;
constexpr int kWideWarps = kWideThreads / 32;
constexpr long long kWideWait = 1ll << 32;            // cycles, about two seconds
constexpr int kFewLarge = 4;                         // most tasks of queries split by classes, per CTA, up to which their offers are worked out
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

__device__ __forceinline__ bool wait_for_tasks(const int* ctr, int target, long long cycles) {
  const long long t0 = clock64();
  while (__ldcg(ctr) < target) {
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
//   tok    the candidates' followers (-1: ended), from wide_lay_out
//   out    first their probabilities (32 bits each, the first half of the row), then node weights, in the end for those
//          candidates that are named by others what the draft says of them (score, weight of the edge from the node before)
//   succ   the best successor of the node that the candidate was on at the layer before (a candidate on it; -1: none).  Queries
//          of more than wide_alone() matches have no such row (and no probabilities): see wide_offers.
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
// Slot of token v, claimed if need be; -1: the table is full (or, with `most`, as good as).
__device__ __forceinline__ int wide_claim(const WideTable& t, int v, int most = INT_MAX) {
  unsigned h = ((unsigned)v * 2654435761u) >> t.shift;
  const int end = min(t.mask, most);
#pragma unroll 1
  for (int probe = 0; probe <= end; ++probe) {
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
// (The match list is read past L1 throughout: the kernel before this one still cuts it down in place, with a cap on the matches per
// path, while CTAs of this one are resident.  So it does, if it is a step, with tokens, probabilities and lengths: ldm.)
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
  const int n = min(l1, ldm(s.len + j) - 1 - (g - j * s.L));         // followers
  const bool probs = M <= wide_alone(s);
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
      if (at < n && at < lb + 16) { a[x] = ldm(st + (lb >> 2) + x); c[x] = ldm(sp + (lb >> 2) + x); }   // (only what holds a follower)
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
        if (l < l1) { *tok = l < n ? vs[y] : -1; if (probs) *p = ps[y]; }
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
  // At most half full, 65 % in the largest but one, in any case 7/8: a CTA waits for its unluckiest lane's probe sequence (a layer of 862
  // candidates: 47 to 58 K cycles in 1024 slots, 16 K in 2048), but emptying 192 KB three times is 4 us (4773 candidates, most of
  // them on few nodes: a build of 57 us with 16384 slots, 53 with 8192).
  const int most = counts ? kWideSlots / 2 : kWideSlots;
  int cap = 64;
  while ((cap < 2 * M && cap < most / 2) || (20 * cap < 31 * M && cap < most)) cap *= 2;
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
          const unsigned q = (unsigned)(KEEP ? __ldcg(row_p + m) : ldm(s.pq + __ldcg(list + m) + d));
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

// ---- larger queries: a task per class of tokens --------------------------------------------------------------------
// Sums by class of the layer's own token, then (all sums of the query are waited for) offers by class of the token before.  A task picks
// its candidates out of the row into a list, so that everything else it does is dense.  What a query keeps per candidate and layer is
// one word: the node's weight from the sums, which only one offers task reads, the one whose class the candidate's token before
// is in; that one leaves there where the walk goes from here.  Layers whose nodes all compete with one another (the first one, and
// all of them in layer-wise search) have no offers: each class leaves its heaviest node.
constexpr int kClassSlots = 8192;                      // most slots of a sums task's table (4 words each); of an offers task's (8 words): half
// Candidates per class aimed at.  Without offers few, large classes: each reads the whole row (16 prompts of 128 x 4096: 1322 us, with
// 7168 1389).  With offers what a thread keeps in registers (3072), give or take.
constexpr int kClassMembers = 12288, kOfferMembers = 4096;
constexpr int kClassProbes = 255;                      // a claim that looks further has its part of the class halved
constexpr int kClassList = (kWideSmem - kClassSlots * 16) / 4;
// Classes (a power of two) for `members` candidates each; 1: the layers are one task each.
__device__ __forceinline__ int wide_classes(const Dev& s, int M, int members) {
  int c = 1;
  if (M > wide_alone(s)) while ((long long)c * members < M) c *= 2;
  return c;
}
struct WideBest { u64 weight, sum; int tok, rep; unsigned cnt, unused; };             // a class's heaviest node: a candidate on it
static_assert(sizeof(WideBest) == 32, "four words of the layer's row");
__device__ __forceinline__ WideBest* wide_best(const WideItems& rows, int d) { return reinterpret_cast<WideBest*>(rows.out + (size_t)(d - 1) * rows.pitch); }

struct WideClass {                       // what a task keeps in shared memory beside its table and list
  int count, over, rep;
  u64 best[kWideWarps];
  int tok[kWideWarps];
};
// A class, or the part of one that is being worked on: tokens whose hash has `mine` in the bits of width - 1.  A table that overruns (tokens
// are not known beforehand) is done again with half the class, then the other half.
struct WidePart { unsigned mine, width; };
__device__ __forceinline__ bool wide_next_part(WidePart& c, unsigned classes) {
  while (c.width > classes && (c.mine & (c.width >> 1))) { c.width >>= 1; c.mine &= ~c.width; }
  if (c.width == classes) return false;
  c.mine |= c.width >> 1;
  return true;
}
// Candidates whose token of `row` is in the part, into `list` as far as it goes; how many (in sh.count, zero before).  ended: weights of
// candidates that have ended become zero there.
__device__ __forceinline__ void wide_members(const int* row, int M, const WidePart c, int* list, WideClass& sh, u64* ended = nullptr) {
  constexpr int B = 8;
  const unsigned others = c.width - 1u;
#pragma unroll 1
  for (int x0 = 4 * threadIdx.x; x0 < M; x0 += B * 4 * kWideThreads) {
    int4 u[B];
#pragma unroll
    for (int r = 0; r < B; ++r) {
      const int x = x0 + r * 4 * kWideThreads;
      u[r] = x < M ? __ldcg(reinterpret_cast<const int4*>(row + x)) : make_int4(-1, -1, -1, -1);
      if (x + 1 >= M) u[r].y = -1;
      if (x + 2 >= M) u[r].z = -1;
      if (x + 3 >= M) u[r].w = -1;
    }
    unsigned on = 0u;
    auto in = [&](int v) { return (unsigned)(v >= 0 && (wide_class(v) & others) == c.mine); };
#pragma unroll
    for (int r = 0; r < B; ++r) on |= (in(u[r].x) | in(u[r].y) << 1 | in(u[r].z) << 2 | in(u[r].w) << 3) << (4 * r);
    if (ended) {
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const int v[4] = {u[r].x, u[r].y, u[r].z, u[r].w};
#pragma unroll
        for (int y = 0; y < 4; ++y) if (v[y] < 0 && x0 + r * 4 * kWideThreads + y < M) ended[x0 + r * 4 * kWideThreads + y] = 0ull;
      }
    }
    if (on == 0u) continue;
    int at = atomicAdd(&sh.count, __popc(on));
    for (; on && at < kClassList; on &= on - 1u, ++at) {
      const int bit = __ffs(on) - 1;
      list[at] = x0 + (bit >> 2) * 4 * kWideThreads + (bit & 3);
    }
  }
}
// Members x0, x0 + kWideThreads, ... of the part (-1: no more): from the list, or where that overflowed from the row.
template <int N>
__device__ __forceinline__ void wide_member(const int* list, bool listed, int total, const int* row, const WidePart c, int x0, int (&m)[N]) {
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const int x = x0 + r * kWideThreads;
    m[r] = x >= total ? -1 : listed ? list[x] : x;
    if (!listed && m[r] >= 0) {
      const int v = __ldcg(row + x);
      if (v < 0 || (wide_class(v) & (c.width - 1u)) != c.mine) m[r] = -1;
    }
  }
}

// Weights of the nodes of layer d with tokens of class `cls`.
__device__ __forceinline__ void wide_sums(const Dev& s, const int4 de, int d, unsigned cls, unsigned classes, WideClass& sh) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  constexpr int N = 8;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems rows = wide_items(s, de.z, M);
  u64* const weight = rows.out + (size_t)(d - 1) * rows.pitch;
  const int* const row = rows.tok + (size_t)(d - 1) * rows.pitch;
  int* const mem = reinterpret_cast<int*>(wide_smem + kClassSlots * 16);
  const bool counts = s.alpha != 1.0, single = d == 1 || s.mode == 1;
  WideBest best{0ull, 0ull, INT_MAX, -1, 0u, 0u};      // (single) the same in every thread
  WidePart c{cls, classes};
  for (bool more = true; more;) {
    if (tid == 0) { sh.count = 0; sh.over = 0; }
    __syncthreads();
    wide_members(row, M, c, mem, sh, !single && c.mine == 0u ? weight : nullptr);
    __syncthreads();
    const bool listed = sh.count <= kClassList;
    const int total = listed ? sh.count : M;
    int cap = 64;
    while (cap < 2 * sh.count && cap < kClassSlots) cap *= 2;
    const WideTable t = wide_table(wide_smem, cap);
    wide_table_empty(wide_smem, cap, counts);
    __syncthreads();
#pragma unroll 1
    for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
      int m[N], v[N];
      unsigned p[N];
      wide_member<N>(mem, listed, total, row, c, x0, m);
#pragma unroll
      for (int r = 0; r < N; ++r) { v[r] = m[r] >= 0 ? __ldcg(row + m[r]) : -1; p[r] = m[r] >= 0 ? (unsigned)__ldcg(list + m[r]) : 0u; }
#pragma unroll
      for (int r = 0; r < N; ++r) p[r] = m[r] >= 0 ? (unsigned)ldm(s.pq + (int)p[r] + d) : 0u;
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (x0 - tid + r * kWideThreads >= total) break;               // (the same for everybody)
        if (m[r] < 0 || *(volatile int*)&sh.over) continue;            // (a table that has overrun is done again)
        const int h = wide_claim(t, v[r], kClassProbes);
        if (h < 0) *(volatile int*)&sh.over = 1;
        else wide_add(t, h, p[r], counts);
      }
    }
    __syncthreads();
    if (sh.over) {                                     // (the same for everybody)
      c.width *= 2;
      __syncthreads();
      continue;
    }
    if (!single) {
#pragma unroll 1
      for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
        int m[N], v[N];
        wide_member<N>(mem, listed, total, row, c, x0, m);
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = m[r] >= 0 ? __ldcg(row + m[r]) : -1;
#pragma unroll
        for (int r = 0; r < N; ++r) {
          if (x0 - tid + r * kWideThreads >= total) break;
          if (m[r] >= 0) weight[m[r]] = wide_weight(s, t, wide_claim(t, v[r], kClassProbes), counts);
        }
      }
    } else {
      u64 w = 0ull;
      int v = INT_MAX;
      for (int x = tid; x < cap; x += kWideThreads) {
        const int k = t.key[x];
        if (k < 0) continue;
        const u64 y = wide_weight(s, t, x, counts);
        if (v == INT_MAX || y > w || (y == w && k < v)) { w = y; v = k; }
      }
      u64 top = warp_max64(w);
      int tok = (int)__reduce_min_sync(FULL, (unsigned)(w == top ? v : INT_MAX));
      if (lane == 0) { sh.best[warp] = top; sh.tok[warp] = tok; }
      __syncthreads();
      w = lane < kWideWarps ? sh.best[lane] : 0ull;
      v = lane < kWideWarps ? sh.tok[lane] : INT_MAX;
      top = warp_max64(v == INT_MAX ? 0ull : w);
      tok = (int)__reduce_min_sync(FULL, (unsigned)(w == top ? v : INT_MAX));
      if (tok != INT_MAX && (best.tok == INT_MAX || top > best.weight || (top == best.weight && tok < best.tok))) {
        const int h = wide_claim(t, tok, kClassProbes);
        best = WideBest{top, ((u64)t.hi[h] << 15) + t.lo[h], tok, -1, counts ? t.cnt[h] : 0u, 0u};
#pragma unroll 1
        for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
          int m[N];
          wide_member<N>(mem, listed, total, row, c, x0, m);
#pragma unroll
          for (int r = 0; r < N; ++r)
            if (m[r] >= 0 && __ldcg(row + m[r]) == tok) sh.rep = m[r];   // any one of them
        }
        __syncthreads();
        best.rep = sh.rep;
      }
    }
    __syncthreads();
    more = wide_next_part(c, classes);
  }
  if (single && tid == 0) wide_best(rows, d)[cls] = best;
}

// Layer d, candidates whose token before is of class `cls`: the best successor of the node each of them comes from.  What it leaves for a
// candidate: bit 31 set if it is the one that stands for that successor, then what the draft says of it (score, weight of the edge);
// else the candidate that does, plus one (0: the node has no successor).
__device__ __forceinline__ void wide_offers(const Dev& s, const int4 de, int d, unsigned cls, unsigned classes, WideClass& sh) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  constexpr int N = 6;
  const int tid = threadIdx.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems rows = wide_items(s, de.z, M);
  u64* const word = rows.out + (size_t)(d - 1) * rows.pitch;
  const int* const row = rows.tok + (size_t)(d - 1) * rows.pitch;
  const int* const before = row - rows.pitch;
  int* const mem = reinterpret_cast<int*>(wide_smem + kClassSlots * 16);
  WidePart c{cls, classes};
  for (bool more = true; more;) {
    if (tid == 0) { sh.count = 0; sh.over = 0; }
    __syncthreads();
    wide_members(before, M, c, mem, sh);
    __syncthreads();
    const bool listed = sh.count <= kClassList;
    const int total = listed ? sh.count : M;
    int cap = 64;
    while (cap < 2 * sh.count && cap < kClassSlots / 2) cap *= 2;
    const WideTable t = wide_table(wide_smem, cap);                    // lo, hi: the largest weight's lower and upper word
    unsigned* const best_tok = t.cnt;                                  // the smallest token of that weight, as its complement
    unsigned* const e_lo = best_tok + cap;                             // sums of the edge to it
    unsigned* const e_hi = e_lo + cap;
    unsigned* const e_cnt = e_hi + cap;
    int* const named = reinterpret_cast<int*>(e_cnt + cap);            // a candidate on it, plus one
    {
      int4* const z = reinterpret_cast<int4*>(wide_smem);
      for (int x = tid; x < 2 * cap; x += kWideThreads) z[x] = x < cap / 4 ? make_int4(-1, -1, -1, -1) : make_int4(0, 0, 0, 0);
    }
    __syncthreads();
    // A member in the list: candidate, slot of the node it comes from, whether it can still be the one that is looked for.  Tokens
    // and weights stay in registers, or are fetched again for those that can if there are more members than that.
    constexpr unsigned kRuns = 1u << 29;
    const bool again = total > N * kWideThreads;
    int m[N], h[N], v[N];
    u64 w[N];
    bool runs[N];
    auto fetch = [&](int x0) {
      wide_member<N>(mem, listed, total, before, c, x0, m);
#pragma unroll
      for (int r = 0; r < N; ++r) {
        h[r] = 0; runs[r] = m[r] >= 0;
        if (m[r] < 0) continue;
        if (listed) { const unsigned e = (unsigned)m[r]; m[r] = (int)(e & 0x1ffffu); h[r] = (int)(e >> 17 & 0xfffu); runs[r] = (e & kRuns) != 0u; }
        else h[r] = wide_claim(t, __ldcg(before + m[r]), kClassProbes);
      }
      if (again) {
#pragma unroll
        for (int r = 0; r < N; ++r) { v[r] = runs[r] ? __ldcg(row + m[r]) : -1; w[r] = runs[r] ? ld_u64(word + m[r]) : 0ull; }
      }
    };
    // f(r): does it still?
    auto each = [&](auto f) {
#pragma unroll 1
      for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
        fetch(x0);
#pragma unroll
        for (int r = 0; r < N; ++r) {
          if (x0 - tid + r * kWideThreads >= total) break;             // (the same for everybody)
          if (m[r] >= 0 && runs[r] && !(v[r] >= 0 && f(r)) && listed) mem[x0 + r * kWideThreads] = (int)((unsigned)m[r] | (unsigned)h[r] << 17);
        }
      }
      __syncthreads();
    };
    auto raise = [&](unsigned* at, unsigned x) { if (*(volatile unsigned*)at < x) atomicMax(at, x); };
    auto top_hi = [&](int r) { return t.hi[h[r]] == (unsigned)(w[r] >> 32); };
    auto top = [&](int r) { return top_hi(r) && t.lo[h[r]] == (unsigned)w[r]; };
#pragma unroll 1
    for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
      int u[N];
      wide_member<N>(mem, listed, total, before, c, x0, m);
#pragma unroll
      for (int r = 0; r < N; ++r) {
        u[r] = -1; v[r] = -1; w[r] = 0ull;
        if (m[r] >= 0) { u[r] = __ldcg(before + m[r]); v[r] = __ldcg(row + m[r]); w[r] = ld_u64(word + m[r]); }
      }
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (x0 - tid + r * kWideThreads >= total) break;
        if (m[r] < 0 || *(volatile int*)&sh.over) continue;
        const int slot = wide_claim(t, u[r], kClassProbes);
        if (slot < 0) { *(volatile int*)&sh.over = 1; continue; }
        if (listed) mem[x0 + r * kWideThreads] = (int)((unsigned)m[r] | (unsigned)slot << 17 | kRuns);
        if (v[r] >= 0) raise(&t.hi[slot], (unsigned)(w[r] >> 32));
      }
    }
    __syncthreads();
    if (sh.over) {
      c.width *= 2;
      __syncthreads();
      continue;
    }
    each([&](int r) { if (!top_hi(r)) return false; raise(&t.lo[h[r]], (unsigned)w[r]); return true; });
    each([&](int r) { if (!top(r)) return false; raise(&best_tok[h[r]], ~(unsigned)v[r]); return true; });
    each([&](int r) {
      if (!top(r) || best_tok[h[r]] != ~(unsigned)v[r]) return false;
      named[h[r]] = m[r] + 1;                          // any one of them
      const unsigned q = (unsigned)ldm(s.pq + __ldcg(list + m[r]) + d);
      atomicAdd(&e_lo[h[r]], q & 0x7fffu);
      atomicAdd(&e_hi[h[r]], q >> 15);
      atomicAdd(&e_cnt[h[r]], 1u);
      return true;
    });
#pragma unroll 1
    for (int x0 = tid; x0 < total; x0 += N * kWideThreads) {
      fetch(x0);
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (x0 - tid + r * kWideThreads >= total) break;
        if (m[r] < 0) continue;
        const int to = named[h[r]];
        word[m[r]] = to == m[r] + 1 ? wide_out(s, w[r], ((u64)e_hi[h[r]] << 15) + e_lo[h[r]], e_cnt[h[r]]) | 0x80000000ull : (u64)(unsigned)to;
      }
    }
    __syncthreads();
    more = wide_next_part(c, classes);
  }
}

// ---- the walk over a query whose layers are all done --------------------------------------------------------------
struct WideOut { int32_t* tok; int32_t* len; float* score; float* edge_w; };

// Layer-wise search: sums of the edges between the nodes of a draft, known only now.  A warp per layer.
struct WideEdges { unsigned lo[SDMS_MAX_DRAFT], hi[SDMS_MAX_DRAFT], cnt[SDMS_MAX_DRAFT]; };
__device__ __forceinline__ void wide_edges(const Dev& s, const WideItems& rows, const int32_t* list, int M, const int* draft, WideEdges& e) {
  constexpr int B = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int l = warp; l < s.D; l += kWideWarps) {
    const int to = draft[l], from = l > 0 ? draft[l - 1] : -1;
    unsigned lo = 0u, hi = 0u, cnt = 0u;
    if (to >= 0) {
      const int* const row = rows.tok + (size_t)l * rows.pitch;
#pragma unroll 1
      for (int x0 = 4 * lane; x0 < M; x0 += B * 128) {
        int4 a[B], b[B];
#pragma unroll
        for (int r = 0; r < B; ++r) {
          const int x = x0 + r * 128;
          a[r] = x < M ? __ldcg(reinterpret_cast<const int4*>(row + x)) : make_int4(-1, -1, -1, -1);
          b[r] = l > 0 && x < M ? __ldcg(reinterpret_cast<const int4*>(row - rows.pitch + x)) : make_int4(-1, -1, -1, -1);
        }
        int g[4 * B];
#pragma unroll
        for (int r = 0; r < B; ++r) {
          const int va[4] = {a[r].x, a[r].y, a[r].z, a[r].w}, vb[4] = {b[r].x, b[r].y, b[r].z, b[r].w};
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const int m = x0 + r * 128 + y;
            g[4 * r + y] = m < M && va[y] == to && (l == 0 || vb[y] == from) ? __ldcg(list + m) : -1;
          }
        }
        unsigned p[4 * B];
#pragma unroll
        for (int y = 0; y < 4 * B; ++y) p[y] = g[y] >= 0 ? (unsigned)ldm(s.pq + g[y] + l + 1) : 0u;
#pragma unroll
        for (int y = 0; y < 4 * B; ++y) { lo += p[y] & 0x7fffu; hi += p[y] >> 15; cnt += g[y] >= 0; }
      }
    }
    lo = __reduce_add_sync(FULL, lo); hi = __reduce_add_sync(FULL, hi); cnt = __reduce_add_sync(FULL, cnt);
    if (lane == 0) { e.lo[l] = lo; e.hi[l] = hi; e.cnt[l] = cnt; }
  }
}

// The heaviest of the classes' heaviest nodes of layer d (tok INT_MAX: there is none).  By one warp.
__device__ __forceinline__ WideBest wide_best_of(const WideItems& rows, int d, int classes) {
  const int lane = threadIdx.x & 31;
  WideBest mine{0ull, 0ull, INT_MAX, -1, 0u, 0u};
  for (int c = lane; c < classes; c += 32) {
    const ulonglong2* const p = reinterpret_cast<const ulonglong2*>(wide_best(rows, d) + c);
    const ulonglong2 a = __ldcg(p), b = __ldcg(p + 1);
    const WideBest x{a.x, a.y, (int)(unsigned)b.x, (int)(unsigned)(b.x >> 32), (unsigned)b.y, 0u};
    if (x.tok != INT_MAX && (mine.tok == INT_MAX || x.weight > mine.weight || (x.weight == mine.weight && x.tok < mine.tok))) mine = x;
  }
  const u64 top = warp_max64(mine.tok == INT_MAX ? 0ull : mine.weight);
  const int tok = (int)__reduce_min_sync(FULL, (unsigned)(mine.weight == top ? mine.tok : INT_MAX));
  const int from = max(__ffs(__ballot_sync(FULL, mine.tok == tok)) - 1, 0);
  WideBest b;
  b.weight = __shfl_sync(FULL, mine.weight, from); b.sum = __shfl_sync(FULL, mine.sum, from);
  b.tok = tok; b.rep = __shfl_sync(FULL, mine.rep, from); b.cnt = __shfl_sync(FULL, mine.cnt, from); b.unused = 0u;
  return b;
}

// With offers, and in layer-wise search: one or two dependent loads per layer.
__device__ __forceinline__ void wide_walk_classes(const Dev& s, const int4 de, int classes, const WideOut out) {
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ float sh_score[SDMS_MAX_DRAFT];
  __shared__ WideEdges sh_e;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D, i = de.x, M = de.y;
  const WideItems rows = wide_items(s, de.z, M);
  auto score_of = [&](const WideBest& b) { return __uint_as_float((unsigned)wide_out(s, b.weight, 0ull, 0u)); };
  if (s.mode == 1) {
    for (int l = warp; l < D; l += kWideWarps) {
      const WideBest b = wide_best_of(rows, l + 1, classes);
      if (lane == 0) { sh_draft[l] = b.tok == INT_MAX ? -1 : b.tok; sh_score[l] = score_of(b); }
    }
    __syncthreads();
    if (out.edge_w) wide_edges(s, rows, s.matches + s.q_off[i], M, sh_draft, sh_e);
    __syncthreads();
  }
  if (tid >= 32) return;
  int tok = -1, emitted = 0;                           // lane d - 1 keeps what layer d comes to
  float score = 0.0f, edge = 0.0f;
  if (s.mode == 1) {
    const unsigned none = __ballot_sync(FULL, lane >= D || sh_draft[lane] < 0);
    emitted = none ? __ffs(none) - 1 : 32;
    if (lane < emitted) {
      tok = sh_draft[lane]; score = sh_score[lane];
      edge = (float)eq5_weight(s.alpha, ((u64)sh_e.hi[lane] << 15) + sh_e.lo[lane], sh_e.cnt[lane]);
    }
  } else {
    const WideBest b = wide_best_of(rows, 1, classes);
    int at = b.rep, mine = -1;
    if (at >= 0) {
      emitted = 1;
      if (lane == 0) { mine = at; score = score_of(b); edge = (float)eq5_weight(s.alpha, b.sum, b.cnt); }
    }
#pragma unroll 1
    for (int d = 2; d <= D && at >= 0; ++d) {
      const u64* const word = rows.out + (size_t)(d - 1) * rows.pitch;
      u64 o = ld_u64(word + at);
      if (!(o >> 31 & 1u)) {
        at = (int)(unsigned)o - 1;
        if ((unsigned)at >= (unsigned)M) break;        // no successor: the draft ends here
        o = ld_u64(word + at);
      }
      if (lane == d - 1) { mine = at; score = __uint_as_float((unsigned)o & 0x7fffffffu); edge = __uint_as_float((unsigned)(o >> 32)); }
      emitted = d;
    }
    if (mine >= 0) tok = __ldcg(rows.tok + (size_t)lane * rows.pitch + mine);
  }
  if (lane < D) {
    const size_t x = (size_t)i * D + lane;
    out.tok[x] = tok;
    if (out.score) out.score[x] = score;
    if (out.edge_w) out.edge_w[x] = edge;
  }
  if (lane == 0) out.len[i] = emitted;
}

struct WideWalk {                        // what the walk over rows keeps in shared memory
  u64 best[kWideWarps];
  int tok[kWideWarps];
  int draft[SDMS_MAX_DRAFT];
  float score[SDMS_MAX_DRAFT];
  unsigned e[SDMS_MAX_DRAFT][3];         // edge sums: lower 15 bits, rest, count
  int hits[2], first;
};

// Sums only: layer by layer the candidates on the current node are picked from its row into a list in shared memory (whose
// length does not depend on M, and is short for most nodes), their successors compared and the candidates on the edge
// taken weighed.  A list that overflows goes over the rows instead.
__device__ __forceinline__ void wide_walk_rows(const Dev& s, const int4 de, int classes, const WideOut out) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  __shared__ WideWalk sh;
  constexpr int B = 4, kHits = kWideSmem / 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D, i = de.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[i];
  const WideItems rows = wide_items(s, de.z, M);
  int* const hit = reinterpret_cast<int*>(wide_smem);
  auto score_of = [&](u64 weight) { return __uint_as_float((unsigned)wide_out(s, weight, 0ull, 0u)); };
  if (tid < SDMS_MAX_DRAFT) { sh.e[tid][0] = 0u; sh.e[tid][1] = 0u; sh.e[tid][2] = 0u; }
  if (tid == 0) { sh.hits[0] = 0; sh.hits[1] = 0; }
  __syncthreads();
  if (warp == 0) {
    const WideBest b = wide_best_of(rows, 1, classes);
    if (lane == 0) {
      sh.first = b.tok; sh.draft[0] = b.tok; sh.score[0] = score_of(b.weight);
      sh.e[0][0] = (unsigned)b.sum & 0x7fffu; sh.e[0][1] = (unsigned)(b.sum >> 15); sh.e[0][2] = b.cnt;
    }
  }
  __syncthreads();
  int cur = sh.first, emitted = cur == INT_MAX ? 0 : 1;
#pragma unroll 1
  for (int d = 2; d <= D && emitted > 0; ++d) {
    const int* const row = rows.tok + (size_t)(d - 1) * rows.pitch;
    const int* const before = row - rows.pitch;
    const u64* const row_w = rows.out + (size_t)(d - 1) * rows.pitch;
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
    const int hits = sh.hits[d & 1];
    const bool listed = hits <= kHits;
    const int n = listed ? hits : M;
    if (tid == 0) sh.hits[(d + 1) & 1] = 0;
    // The heaviest successor, the smallest token of those, the edge to it: weights of all hits, tokens only of the heaviest,
    // probabilities only on the edge (what a CTA gathers from L2 takes 2 cycles per sector).  Read again for each step if there
    // are more hits than are kept in registers.
    const bool again = n > B * kWideThreads;
    int m[B], t[B];
    u64 w[B];
    u64 best = 0ull;
    auto load_weights = [&](int x0) {
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const int x = x0 + r * kWideThreads;
        m[r] = x >= n ? -1 : listed ? hit[x] : x;
        if (!listed && m[r] >= 0 && __ldcg(before + m[r]) != cur) m[r] = -1;
        w[r] = m[r] >= 0 ? ld_u64(row_w + m[r]) : 0ull;
      }
    };
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
      for (int r = 0; r < B; ++r) g[r] = t[r] == tok ? __ldcg(list + m[r]) : -1;
#pragma unroll
      for (int r = 0; r < B; ++r) p[r] = g[r] >= 0 ? (unsigned)ldm(s.pq + g[r] + d) : 0u;
#pragma unroll
      for (int r = 0; r < B; ++r) { lo += p[r] & 0x7fffu; hi += p[r] >> 15; count += g[r] >= 0; }
    }
    lo = __reduce_add_sync(FULL, lo); hi = __reduce_add_sync(FULL, hi); count = __reduce_add_sync(FULL, count);
    if (lane == 0 && count) { atomicAdd(&sh.e[d - 1][0], lo); atomicAdd(&sh.e[d - 1][1], hi); atomicAdd(&sh.e[d - 1][2], count); }
    if (tid == 0) { sh.draft[d - 1] = tok; sh.score[d - 1] = score_of(best); }
    cur = tok; emitted = d;
    __syncthreads();                                   // before the next layer's list
  }
  __syncthreads();
  if (tid < D) {
    const size_t x = (size_t)i * D + tid;
    const bool on = tid < emitted;
    out.tok[x] = on ? sh.draft[tid] : -1;
    if (out.score) out.score[x] = on ? sh.score[tid] : 0.0f;
    if (out.edge_w) out.edge_w[x] = on ? (float)eq5_weight(s.alpha, ((u64)sh.e[tid][1] << 15) + sh.e[tid][0], sh.e[tid][2]) : 0.0f;
  }
  if (tid == 0) out.len[i] = emitted;
}

// For queries whose layers are one task each: one dependent load per layer.
__device__ __forceinline__ void wide_walk_known(const Dev& s, const int4 de, const WideOut out) {
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ WideEdges sh_e;
  static_assert(SDMS_MAX_DRAFT <= 32, "a lane per layer");
  const int tid = threadIdx.x, D = s.D, i = de.x, M = de.y;
  const WideItems items = wide_items(s, de.z, M);
  if (s.mode == 1 && out.edge_w) {                     // the edges are known only now
    if (tid < D) { const int at = __ldcg(items.succ + (size_t)tid * items.pitch); sh_draft[tid] = at >= 0 ? __ldcg(items.tok + (size_t)tid * items.pitch + at) : -1; }
    __syncthreads();
    wide_edges(s, items, s.matches + s.q_off[i], M, sh_draft, sh_e);
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
                        : s.mode == 1 ? (float)eq5_weight(s.alpha, ((u64)sh_e.hi[tid] << 15) + sh_e.lo[tid], sh_e.cnt[tid])
                                      : __uint_as_float((unsigned)(o >> 32));
    }
    if (tid == 0) out.len[i] = emitted;
  }
}

__device__ __forceinline__ void wide_walk(const Dev& s, const int4 de, int classes, bool few, const WideOut out) {
  if (de.y <= wide_alone(s)) wide_walk_known(s, de, out);
  else if (few || s.mode == 1) wide_walk_classes(s, de, classes, out);
  else wide_walk_rows(s, de, classes, out);
  if (s.beam_stride > 0) {                             // the beams want the table area empty
    __syncthreads();
    uint4* const z = reinterpret_cast<uint4*>(s.w_tab + (unsigned)de.z);
    for (size_t x = threadIdx.x; x < (size_t)wide_slots(s, de.y) * 2; x += kWideThreads) z[x] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// The launch's last CTA leaves all counts at zero: the single-launch build that registers queries next has no kernel in front of
// it that would.  By one thread of each CTA, once it has its last tickets.
__device__ __forceinline__ void wide_counts_done(const Dev& s) {
  __threadfence();
  if (atomicAdd(&s.w_ctl[kWideLeft], 1ull) == gridDim.x - 1)
    for (int x = 0; x < kWideCtlWords; ++x) s.w_ctl[x] = 0ull;
}

__global__ void __launch_bounds__(kWideThreads, 1)
dag_wide_kernel(Dev s, int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  grid_wait();                                         // scheduled while dag_kernel drains; its list is complete from here on
  const u64 registered = ld_u64(&s.w_ctl[kWideListed]);
  if (registered == 0) {                               // (room may have been asked for in vain)
    if (blockIdx.x == 0 && threadIdx.x == 0) s.w_ctl[kWideTaken] = s.w_ctl[kWideHeavy] = 0ull;
    return;
  }
  const int nq = (int)(registered < (u64)kMaxWide ? registered : (u64)kMaxWide);
  __shared__ int4 sh_desc[kMaxWide];
  __shared__ int sh_base[kMaxWide + 1];                // first task of each query: layers, or sums by classes
  __shared__ int sh_offer[kMaxWide + 1];               // its first task of those that wait for its sums
  __shared__ WideClass sh_class;
  __shared__ int sh_unit[kMaxWide + 1];                // first chunk of kWideThreads candidates of each query
  __shared__ int sh_warp[kWideWarps];
  __shared__ int sh_task, sh_last, sh_large;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D;
  int members;                                         // candidates per class of the large queries
  bool few;                                            // they are few: offers
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
      if (M > wide_alone(s)) large += D * wide_classes(s, M, kClassMembers);
    }
    if (large) atomicAdd(&sh_large, large);
    __syncthreads();
    // Offers work out every node's best successor where a walk by one CTA looks at those on its way only: eighteen times the work (6 M
    // against 326 K cycles for 26 000 matches, D = 16), in a fraction of the time as long as such queries are few.  About eight of them
    // at these sizes; 53 (16 prompts of 128 x 4096 tokens, k = 1) take 1920 us with offers, 1320 without.
    few = sh_large <= kFewLarge * (int)gridDim.x;
    members = few && s.mode != 1 ? kOfferMembers : kClassMembers;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int M = 2 * tid + r < nq ? sh_desc[2 * tid + r].y : 0;
      c[r] = M > 0 ? D * wide_classes(s, M, members) : 0;
    }
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
    for (int r = 0; r < 2; ++r) c[r] = few && s.mode != 1 && 2 * tid + r < nq && sh_desc[2 * tid + r].y > wide_alone(s) ? c[r] / D * (D - 1) : 0;
    prefix(c[0], c[1], sh_offer);
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
  if (tid == 0) sh_task = (int)atomicAdd(&s.w_ctl[kWideChunkNext], 1ull);
  __syncthreads();
#pragma unroll 1
  for (int unit = sh_task; unit < units;) {
    __syncthreads();
    if (tid == 0) sh_task = (int)atomicAdd(&s.w_ctl[kWideChunkNext], 1ull);         // (on its way during this one)
    const int chunk = unit / parts, l0 = (unit - chunk * parts) * span;
    const int q = owner(sh_unit, chunk);
    if (l0 < D) wide_lay_out(s, sh_desc[q], (chunk - sh_unit[q]) * kWideThreads, l0, min(D, l0 + span));
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(&s.w_ctl[kWideChunksDone], 1ull);
    unit = sh_task;
  }
  __syncthreads();
  if (tid == 0) {
    sh_last = wait_for_count(s.w_ctl + kWideChunksDone, (u64)units, kWideWait);
    if (sh_last) sh_task = (int)atomicAdd(&s.w_ctl[kWideTask], 1ull);          // (whoever gives up here leaves no task undone)
  }
  __syncthreads();
  if (!sh_last) {
    if (tid == 0) { atomicOr(s.status, SDMS_STATUS_TIMEOUT); wide_counts_done(s); }
    return;
  }
  __threadfence();
  const int firsts = sh_base[nq], tasks = firsts + sh_offer[nq];
  int task = sh_task;
  __syncthreads();
#pragma unroll 1
  while (task < tasks) {
    const bool offers = task >= firsts;
    const int a = owner(offers ? sh_offer : sh_base, offers ? task - firsts : task);
    const int4 de = sh_desc[a];
    const bool large = de.y > wide_alone(s);
    const int classes = wide_classes(s, de.y, members), part = offers ? task - firsts - sh_offer[a] : task - sh_base[a];
    int* const done = s.w_done + 2 * de.w;             // tasks done, sums done
    if (!large) {
      wide_task(s, de, part + 1);
    } else if (!offers) {
      wide_sums(s, de, part / classes + 1, (unsigned)(part % classes), (unsigned)classes, sh_class);
    } else {
      // the sums were dealt out before and wait for nobody.  (Should the wait run out all the same, the results are wrong but every
      // index stays within the query's rows, and the counts come out right.)
      if (tid == 0 && !wait_for_tasks(done + 1, D * classes, kWideWait)) atomicOr(s.status, SDMS_STATUS_TIMEOUT);
      __syncthreads();
      __threadfence();
      wide_offers(s, de, part / classes + 2, (unsigned)(part % classes), (unsigned)classes, sh_class);
    }
    // done with it: its results are out before it is counted, and whoever counts the last one has seen all of them
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      sh_task = (int)atomicAdd(&s.w_ctl[kWideTask], 1ull);
      const int total = (large && few && s.mode != 1 ? 2 * D - 1 : D) * classes;
      if (large && !offers) atomicAdd(done + 1, 1);
      sh_last = atomicAdd(done, 1) == total - 1;
      if (sh_last) { done[0] = 0; done[1] = 0; }       // the next build finds them at zero
      __threadfence();
    }
    __syncthreads();
    if (sh_last) wide_walk(s, de, classes, few, WideOut{draft_tok, draft_len, draft_score, draft_edge_w});
    task = sh_task;
    __syncthreads();
  }
  if (tid == 0) wide_counts_done(s);
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
