// Follower gather, DAG aggregation (Eq. 5) and the greedy walk for queries with many matches on prompts that do not take the
// single-launch build, spread over the whole device.
//
// One CTA that aggregates a query of thousands of matches by itself takes hundreds of microseconds while the other SMs idle,
// so dag_kernel hands such queries over (wide_register).  Here every (query, layer) pair is a task of its own: a CTA gathers
// the layer's followers, sums them up per token in a hash table in its shared memory and leaves, for every candidate, its
// token and its node's weight in the table area of the workspace.  The CTA that completes the last layer of a query then
// walks it: per layer one coalesced sweep over the candidates' tokens, the weights only of those on the current node.
// Nobody waits for anybody: tasks come from a counter, heavy queries first.  Sums are integers and every choice has a tie
// rule, so the order in which things happen cannot show in a result.
//
// What bounds it: a task the gather (one 32-byte sector per follower and SM at a time) and the shared-memory atomics, both
// around 1.3 cycles per candidate; the walk one round trip to L2 and one barrier per layer.  The form before this one kept all
// nodes in tables in global memory and passed over all items five times with grid barriers in between: 32 us for one query
// of 200 matches and D = 16, 165 us for 12 000 matches, and room for a quarter of the 420 000 matches of 16 prompts of 128 x
// 4096 tokens, whose heaviest queries then kept one CTA each busy for 1.2 ms.
#include <climits>
#include "sdms_internal.h"
#include "wide_dev.cuh"

namespace sdms {

namespace {

constexpr int kWideSlots = 16384;                    // most slots of a task's table (half of them where counts are kept too)
constexpr int kWideSmem = kWideSlots * 12;
constexpr int kWideTableMatches = 16384;             // candidates per table
constexpr int kWideWarps = kWideThreads / 32;
constexpr int kSortFrom = 256;                       // more queries than this balance without an order

__device__ __forceinline__ u64 ld_u64(const u64* p) { return __ldcg(p); }

// A wait for a count, bounded in cycles.
__device__ __forceinline__ bool wait_for_count(const u64* ctr, u64 target, long long cycles) {
  const long long t0 = clock64();
  while (ld_u64(ctr) < target) {
    if (clock64() - t0 > cycles) return false;
    __nanosleep(32);
  }
  return true;
}

// sdms_debug_wait_timeout: a bounded wait on a count that nobody raises.
__global__ void wait_timeout_kernel(Dev s, long long cycles) {
  if (threadIdx.x == 0 && !wait_for_count(s.b_ctl + 1, ~0ull, cycles)) atomicOr(s.status, SDMS_STATUS_TIMEOUT);
}

__device__ __forceinline__ u64 warp_max64(u64 x) {
  const unsigned hi = (unsigned)(x >> 32), top = __reduce_max_sync(FULL, hi);
  const unsigned lo = __reduce_max_sync(FULL, hi == top ? (unsigned)x : 0u);
  return (u64)top << 32 | lo;
}

// Where a query's candidates leave their nodes: weights [D][M], then tokens [D][M] (-1: the candidate has ended).
struct WideItems { u64* weight; int* tok; };
__device__ __forceinline__ WideItems wide_items(const Dev& s, int first, int M) {
  u64* const w = reinterpret_cast<u64*>(s.w_tab + (unsigned)first);
  return WideItems{w, reinterpret_cast<int*>(w + (size_t)s.D * M)};
}

// Number of tables (a power of two) that the tokens of a layer are dealt out to by their hash.
__device__ __forceinline__ int wide_classes(int M) {
  int c = 1;
  while ((long long)c * kWideTableMatches < M) c *= 2;
  return c;
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
__device__ __forceinline__ int wide_claim(const WideTable& t, int v, int cap) {
  unsigned h = ((unsigned)v * 2654435761u) >> t.shift;
#pragma unroll 1
  for (int probe = 0; probe < cap; ++probe) {
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
// Followers d of candidates m0, m0 + kWideThreads, ...: token (-1: none) and probability, all requests on their way together.
template <int N>
__device__ __forceinline__ void wide_gather(const Dev& s, const int32_t* list, int M, int d, int m0, int (&v)[N], unsigned (&p)[N]) {
  int gpos[N];
#pragma unroll
  for (int r = 0; r < N; ++r) gpos[r] = __ldg(list + min(m0 + r * kWideThreads, M - 1));
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const int j = path_of(s, gpos[r]);
    const bool on = m0 + r * kWideThreads < M && gpos[r] - j * s.L + d <= __ldg(s.len + j) - 1;
    v[r] = -1; p[r] = 0u;
    if (on) { v[r] = __ldg(s.tok + gpos[r] + d); p[r] = (unsigned)__ldg(s.pq + gpos[r] + d); }
  }
}

// Layer d of a query with at most N * CH * kWideThreads candidates: node sums, then every candidate's token and node weight.
// The slots stay in registers in between.  false: more distinct tokens than slots, nothing is done.
template <int N, int CH>
__device__ __forceinline__ bool wide_sums_kept(const Dev& s, const int4 de, int d) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  __shared__ int sh_full;
  const int tid = threadIdx.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems items = wide_items(s, de.z, M);
  u64* const weight = items.weight + (size_t)(d - 1) * M;
  int* const tok = items.tok + (size_t)(d - 1) * M;
  const bool counts = s.alpha != 1.0;                  // with alpha = 1 a weight does not depend on the count
  int cap = 64;
  while (cap < (counts ? kWideSlots / 2 : kWideSlots) && 7 * cap < 8 * M) cap *= 2;
  const WideTable t = wide_table(wide_smem, cap);
  if (tid == 0) sh_full = 0;
  int v[N];
  unsigned p[N];
  wide_gather<N>(s, list, M, d, tid, v, p);            // on its way while the table is emptied
  wide_table_empty(wide_smem, cap, counts);
  __syncthreads();
  int slot[CH][N];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int m0 = c * N * kWideThreads + tid;
    if (c > 0) wide_gather<N>(s, list, M, d, m0, v, p);
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int m = m0 + r * kWideThreads;
      if (m < M) tok[m] = v[r];
      slot[c][r] = -1;
      if (v[r] < 0) continue;
      slot[c][r] = wide_claim(t, v[r], cap);
      if (slot[c][r] < 0) sh_full = 1;
      else wide_add(t, slot[c][r], p[r], counts);
    }
  }
  __syncthreads();
  if (sh_full) return false;                           // (the same for everybody)
#pragma unroll
  for (int c = 0; c < CH; ++c)
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (slot[c][r] >= 0) weight[(c * N + r) * kWideThreads + tid] = wide_weight(s, t, slot[c][r], counts);
  return true;
}

// The same for any number of candidates, tokens of class `cls` of `classes`; the followers are fetched twice.  Almost always
// one pass; a table that turns out too small is done again in sub-classes.
__device__ __forceinline__ void wide_sums_any(const Dev& s, const int4 de, int d, unsigned cls, unsigned classes) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  __shared__ int sh_over;
  const int tid = threadIdx.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[de.x];
  const WideItems items = wide_items(s, de.z, M);
  u64* const weight = items.weight + (size_t)(d - 1) * M;
  int* const tok = items.tok + (size_t)(d - 1) * M;
  const bool counts = s.alpha != 1.0;
  const int cap = counts ? kWideSlots / 2 : kWideSlots;
  const WideTable t = wide_table(wide_smem, cap);
  unsigned subs = 1;
#pragma unroll 1
  for (unsigned sub = 0; sub < subs; ++sub) {
    const unsigned all_classes = classes * subs, mine = cls + classes * sub;
    if (tid == 0) sh_over = 0;
    wide_table_empty(wide_smem, cap, counts);
    __syncthreads();
#pragma unroll 1
    for (int sweep = 0; sweep < 2; ++sweep) {
#pragma unroll 1
      for (int m0 = tid; m0 - tid < M; m0 += 8 * kWideThreads) {
        int v[8];
        unsigned p[8];
        wide_gather<8>(s, list, M, d, m0, v, p);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int m = m0 + r * kWideThreads;
          if (sweep == 0 && cls == 0u && sub == 0u && m < M) tok[m] = v[r];
          if (v[r] < 0 || (wide_class(v[r]) & (all_classes - 1u)) != mine) continue;
          const int h = wide_claim(t, v[r], cap);
          if (h < 0) sh_over = 1;
          else if (sweep == 0) wide_add(t, h, p[r], counts);
          else weight[m] = wide_weight(s, t, h, counts);
        }
      }
      __syncthreads();
      if (sh_over) break;                              // (the same for everybody; only sweep 0 claims)
    }
    if (sh_over) {
      __syncthreads();
      subs *= 2; sub = ~0u;
    }
  }
}

__device__ __forceinline__ void wide_sums(const Dev& s, const int4 de, int d, unsigned cls, unsigned classes) {
  const int M = de.y;
  bool done = false;
  if (M <= 4 * kWideThreads) done = wide_sums_kept<4, 1>(s, de, d);
  else if (M <= 32 * kWideThreads) done = wide_sums_kept<8, 4>(s, de, d);
  if (!done) { __syncthreads(); wide_sums_any(s, de, d, cls, classes); }
}

// The walk over a query whose layers are all done.  N > 0: at most N candidates per thread; their tokens of the layer before
// stay in registers, and with AHEAD a layer's tokens and weights are asked for a layer ahead.  N = 0: any number.
template <int N, bool AHEAD>
__device__ __forceinline__ void wide_walk(const Dev& s, const int4 de, int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                                          float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  __shared__ u64 sh_best[2][kWideWarps];
  __shared__ int sh_tok[2][kWideWarps];
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_e[SDMS_MAX_DRAFT][3];
  constexpr int B = N > 0 ? N : 8;                     // candidates of a thread in flight
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D, i = de.x, M = de.y;
  const int32_t* const list = s.matches + s.q_off[i];
  const WideItems items = wide_items(s, de.z, M);
  if (tid < SDMS_MAX_DRAFT) { sh_e[tid][0] = 0u; sh_e[tid][1] = 0u; sh_e[tid][2] = 0u; sh_draft[tid] = -1; }
  int my_tok = -1, cur = -1;                           // lane d - 1 of warp 0 keeps what layer d comes to
  u64 my_weight = 0ull;
  int t[B], u[B];
  u64 w[AHEAD ? B : 1];
  auto fetch = [&](int d, int m0) {
#pragma unroll
    for (int r = 0; r < B; ++r) {
      const int m = m0 + r * kWideThreads;
      t[r] = m < M ? __ldcg(items.tok + (size_t)(d - 1) * M + m) : -1;
      if (AHEAD) w[r] = m < M ? ld_u64(items.weight + (size_t)(d - 1) * M + m) : 0ull;
    }
  };
  if (N > 0) fetch(1, tid);
  int emitted = 0;
#pragma unroll 1
  for (int d = 1; d <= D; ++d) {
    u64 best = 0ull;
    int tok = INT_MAX;
#pragma unroll 1
    for (int m0 = tid; m0 - tid < (N > 0 ? 1 : M); m0 += B * kWideThreads) {
      if (N == 0) {
        fetch(d, m0);
#pragma unroll
        for (int r = 0; r < B; ++r) u[r] = d > 1 && m0 + r * kWideThreads < M ? __ldcg(items.tok + (size_t)(d - 2) * M + m0 + r * kWideThreads) : -1;
      }
      int q[B];
      u64 ww[B];
#pragma unroll
      for (int r = 0; r < B; ++r) {
        q[r] = d == 1 || s.mode == 1 || u[r] == cur ? t[r] : -1;                 // -1: not on the current node
        ww[r] = AHEAD ? w[AHEAD ? r : 0] : q[r] >= 0 ? ld_u64(items.weight + (size_t)(d - 1) * M + m0 + r * kWideThreads) : 0ull;
      }
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const bool better = q[r] >= 0 && (tok == INT_MAX || ww[r] > best || (ww[r] == best && q[r] < tok));
        best = better ? ww[r] : best; tok = better ? q[r] : tok;
      }
    }
    if (N > 0) {
#pragma unroll
      for (int r = 0; r < B; ++r) u[r] = t[r];
      if (AHEAD && d < D) fetch(d + 1, tid);           // arrives during the reduction
    }
    {
      const u64 top = warp_max64(best);
      tok = (int)__reduce_min_sync(FULL, best == top ? (unsigned)tok : (unsigned)INT_MAX);
      if (lane == 0) { sh_best[d & 1][warp] = top; sh_tok[d & 1][warp] = tok; }
    }
    if (N > 0 && !AHEAD && d < D) fetch(d + 1, tid);
    __syncthreads();
    {
      const u64 b = lane < kWideWarps ? sh_best[d & 1][lane] : 0ull;
      const int bt = lane < kWideWarps ? sh_tok[d & 1][lane] : INT_MAX;
      best = warp_max64(b);
      // (a node of weight zero is still a node: what counts is whether there is a token)
      tok = (int)__reduce_min_sync(FULL, b == best ? (unsigned)bt : (unsigned)INT_MAX);
    }
    if (tok == INT_MAX) break;                         // no successor: the draft ends here
    if (lane == d - 1) { my_tok = tok; my_weight = best; }
    if (tid == 0) sh_draft[d - 1] = tok;
    cur = tok; emitted = d;
  }
  __syncthreads();
  // weights of the edges taken: a warp takes 128 candidates of one layer at a time
  const int chunks = (M + 127) >> 7;
#pragma unroll 1
  for (int x = warp, l = 0, c = warp; x < emitted * chunks; x += kWideWarps, c += kWideWarps) {
    while (c >= chunks) { c -= chunks; ++l; }
    const int want = sh_draft[l], from = l > 0 ? sh_draft[l - 1] : -1;
    int a[4], b[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int m = c * 128 + r * 32 + lane;
      a[r] = m < M ? __ldcg(items.tok + (size_t)l * M + m) : -1;
      b[r] = l > 0 && m < M ? __ldcg(items.tok + (size_t)(l - 1) * M + m) : -1;
    }
    unsigned e0 = 0u, e1 = 0u, e2 = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (a[r] != want || b[r] != from) continue;
      const unsigned p = (unsigned)__ldg(s.pq + __ldg(list + c * 128 + r * 32 + lane) + l + 1);
      e0 += p & 0x7fffu; e1 += p >> 15; ++e2;
    }
    if (__any_sync(FULL, e2 != 0u)) {
      e0 = __reduce_add_sync(FULL, e0); e1 = __reduce_add_sync(FULL, e1); e2 = __reduce_add_sync(FULL, e2);
      if (lane < 3) atomicAdd(&sh_e[l][lane], lane == 0 ? e0 : lane == 1 ? e1 : e2);
    }
  }
  __syncthreads();
  if (warp == 0) {
    if (lane < D) {
      const size_t at = (size_t)i * D + lane;
      const bool on = my_tok >= 0;
      draft_tok[at] = my_tok;
      if (draft_score)
        draft_score[at] = !on ? 0.0f : s.alpha == 1.0 ? (float)eq5_weight(1.0, my_weight, 0u)
                                                      : (float)__longlong_as_double((long long)my_weight);
      if (draft_edge_w)
        draft_edge_w[at] = on ? (float)eq5_weight(s.alpha, ((u64)sh_e[lane][1] << 15) + sh_e[lane][0], sh_e[lane][2]) : 0.0f;
    }
    if (lane == 0) draft_len[i] = emitted;
  }
  if (s.beam_stride > 0) {                             // the beams want the table area empty
    __syncthreads();
    uint4* const z = reinterpret_cast<uint4*>(s.w_tab + (unsigned)de.z);
    for (size_t x = tid; x < (size_t)wide_slots(s, M) * 2; x += kWideThreads) z[x] = make_uint4(0u, 0u, 0u, 0u);
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
  __shared__ int sh_warp[kWideWarps];
  __shared__ int sh_task, sh_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, D = s.D;
  static_assert(kMaxWide == 2 * kWideThreads, "two list entries per thread");
  // the list of queries, the largest first, and by a prefix sum the first task of each
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
    int c[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) c[r] = 2 * tid + r < nq ? D * wide_classes(sh_desc[2 * tid + r].y) : 0;
    int x = c[0] + c[1];
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
    const int ahead = (warp ? sh_warp[warp - 1] : 0) + x - c[0] - c[1];
    sh_base[2 * tid] = ahead;
    sh_base[2 * tid + 1] = ahead + c[0];
    if (tid == kWideThreads - 1) sh_base[kMaxWide] = ahead + c[0] + c[1];
    __syncthreads();
  }
  const int tasks = sh_base[nq];
  int task = blockIdx.x;                               // the first one without asking
#pragma unroll 1
  while (task < tasks) {
    int a = 0, b = nq;                                 // sh_base[a] <= task < sh_base[b]
    while (b - a > 1) { const int mid = (a + b) >> 1; if (sh_base[mid] <= task) a = mid; else b = mid; }
    const int4 de = sh_desc[a];
    const int classes = wide_classes(de.y), part = task - sh_base[a];
    wide_sums(s, de, part / classes + 1, (unsigned)(part % classes), (unsigned)classes);
    // done with it: its results are out before it is counted, and whoever counts the last one has seen all of them
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      sh_task = (int)gridDim.x + (int)atomicAdd(&s.w_ctl[2], 1ull);
      const int total = D * classes;
      sh_last = atomicAdd(&s.w_done[de.w], 1) == total - 1;
      if (sh_last) s.w_done[de.w] = 0;                 // the next build finds it at zero
      __threadfence();
    }
    __syncthreads();
    if (sh_last) {
      if (de.y <= 4 * kWideThreads) wide_walk<4, true>(s, de, draft_tok, draft_len, draft_score, draft_edge_w);
      else if (de.y <= 16 * kWideThreads) wide_walk<16, false>(s, de, draft_tok, draft_len, draft_score, draft_edge_w);
      else wide_walk<0, false>(s, de, draft_tok, draft_len, draft_score, draft_edge_w);
    }
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
