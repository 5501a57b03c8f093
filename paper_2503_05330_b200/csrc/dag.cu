// Follower gather, layered DAG aggregation (Eq. 5) and greedy extraction, plus
// the single-launch build for small prompts.
//
// Every match m of query path i contributes, at layer d = 1..D, its d-th
// follower v = tok[e+d] with the fixed-point probability pq[e+d].  A node is a
// distinct token of a layer, an edge a distinct (previous token, token) pair; S
// and cnt of nodes and edges are integer sums, so the order of accumulation
// (atomics, warp shuffles) cannot change a result.
//
// Ways through, all per query path in one CTA:
//   dag_walk_warp (M <= 32 matches, the common case) and dag_walk (up to thousands): the greedy draft alone.  Node
//     sums of all layers first, side by side, then the walk, then the weights of the edges taken.
//   dag_small (M <= 32; export, tree pool, layer-wise search): lane m owns candidate m and each WARP owns a
//     layer.  Lanes with the same follower token (__match_any_sync) form a node, lanes that also share the previous
//     token form an edge; sums run over the lanes of a group, ranks over the group leaders.
//   dag_block (any M): layers in sequence.  Followers are staged in shared memory
//     when they fit; every candidate adds into a shared-memory hash table keyed
//     by token (32-bit atomics with explicit carry).  Unstaged fan-out past the
//     first layer runs in two phases - claim a slot for every successor of the
//     current node, then add only the candidates that land on a claimed slot -
//     so the table holds the successors of one node instead of a whole layer.
//     One warp then picks the best successor.  A layer with more distinct tokens
//     than the table holds is processed in several passes, each over the tokens
//     of one residue class, so any fan-out fits the same tables.
//   The EXPORT instantiation (sdms_get_dag) also keeps an edge table and lets
//   other warps rank the B best nodes of the layer and the Ke best out-edges of
//   the nodes kept one layer up.  tree / list pools reuse the same passes with a
//   prefix filter / a single arg-max over candidates.
#include "sdms_internal.h"
#include "append_dev.cuh"
#include "wide_dev.cuh"

namespace sdms {

namespace {

constexpr int CAP = kDagCap;
constexpr int MAXB = SDMS_MAX_DAG_NODES;
constexpr int MAXKE = SDMS_MAX_DAG_EDGES;
constexpr int kRollMax = 2 * 8192 / 3;   // candidates whose followers are staged layer by layer (three arrays in the staging area)
constexpr int kStageWords = 8192;      // followers (token, pq) of all matches staged in shared memory when M*D fits
constexpr int kLoadBatch = 4;          // candidates a thread loads before it touches the tables
constexpr int kListCap = 2048;         // matches a fused CTA keeps in shared memory besides its global slice
static_assert(kStageWords >= 4 * 32 * SDMS_MAX_DRAFT, "dag_small keeps its per-layer lanes in the staging area");

struct Cand {            // a node or an edge competing in a selection
  double w; u64 S; unsigned cnt; int tok; int valid;
};

// Lane holding the first candidate in rank order (largest weight, then smallest
// token) among the lanes with valid set, or -1.  Weights are non-negative, so
// their bit patterns order like the values: three full-warp reductions settle it.
__device__ __forceinline__ int warp_arg_first(bool valid, double w, int tok) {
  const u64 bits = (u64)__double_as_longlong(w);
  const unsigned hi = (unsigned)(bits >> 32), lo = (unsigned)bits;
  if (__ballot_sync(FULL, valid) == 0) return -1;
  const unsigned mh = __reduce_max_sync(FULL, valid ? hi : 0u);
  const bool c1 = valid && hi == mh;
  const unsigned ml = __reduce_max_sync(FULL, c1 ? lo : 0u);
  const bool c2 = c1 && lo == ml;
  const unsigned mt = __reduce_min_sync(FULL, c2 ? (unsigned)tok : 0xffffffffu);
  return __ffs(__ballot_sync(FULL, c2 && (unsigned)tok == mt)) - 1;
}

__device__ __forceinline__ Cand warp_best(Cand c) {
  const int src = warp_arg_first(c.valid != 0, c.w, c.tok);
  const int from = src < 0 ? 0 : src;
  Cand r;
  r.valid = src >= 0;
  r.w = __shfl_sync(FULL, c.w, from);
  r.S = __shfl_sync(FULL, c.S, from);
  r.cnt = __shfl_sync(FULL, c.cnt, from);
  r.tok = __shfl_sync(FULL, c.tok, from);
  return r;
}

// The K first candidates in rank order among get(0..ncand-1); lane 0 stores them.
// Tokens are distinct among valid candidates, so "strictly after the previous
// pick" enumerates them one by one.  Returns how many were found.
template <class Get>
__device__ int warp_topk(int ncand, Get get, int K, int* out_tok, u64* out_S, unsigned* out_cnt) {
  const int lane = threadIdx.x & 31;
  double prev_w = 0.0; int prev_tok = 0;
  int r = 0;
  for (; r < K; ++r) {
    Cand best; best.valid = 0; best.w = 0.0; best.S = 0; best.cnt = 0; best.tok = 0;
    for (int x = lane; x < ncand; x += 32) {
      const Cand c = get(x);
      if (!c.valid) continue;
      if (r > 0 && !ranks_before(prev_w, prev_tok, c.w, c.tok)) continue;
      if (!best.valid || ranks_before(c.w, c.tok, best.w, best.tok)) best = c;
    }
    best = warp_best(best);
    if (!best.valid) break;
    if (lane == 0) { out_tok[r] = best.tok; out_S[r] = best.S; out_cnt[r] = best.cnt; }
    prev_w = best.w; prev_tok = best.tok;
  }
  __syncwarp();
  return r;
}

// Sums of val over the lanes of group a and of group b; `live` (warp-uniform)
// lists the lanes worth visiting.
__device__ __forceinline__ void group_sums(unsigned live, unsigned a, unsigned b, unsigned val, u64* sa, u64* sb) {
  u64 x = 0, y = 0;
  for (unsigned rem = live; rem; rem &= rem - 1) {
    const int src = __ffs(rem) - 1;
    const unsigned t = __shfl_sync(FULL, val, src);
    if (a >> src & 1) x += t;
    if (b >> src & 1) y += t;
  }
  *sa = x; *sb = y;
}

// 64-bit add on a (lo, hi) pair of shared words with 32-bit atomics: whoever
// makes the low word wrap carries into the high word.
__device__ __forceinline__ void add64(unsigned* lo, unsigned* hi, u64 v) {
  const unsigned l = (unsigned)v;
  unsigned h = (unsigned)(v >> 32);
  const unsigned old = atomicAdd(lo, l);
  if (old + l < old) ++h;
  if (h) atomicAdd(hi, h);
}
__device__ __forceinline__ u64 get64(const unsigned* lo, const unsigned* hi, int x) {
  return ((u64)hi[x] << 32) | lo[x];
}

struct Smem {
  // node table: key = token; sums over all candidates and over those coming from the current node
  int* n_key; unsigned* n_Slo; unsigned* n_Shi; unsigned* n_Clo; unsigned* n_Chi; unsigned* n_call; unsigned* n_ccur;
  int* n_touch;
  // edge table (export): key = token * MAXB + slot of the kept source node
  int* e_key; unsigned* e_Slo; unsigned* e_Shi; unsigned* e_c; int* e_touch;
  // export lists
  u64* r_node_S; int* r_node_tok; unsigned* r_node_cnt;
  u64* r_edge_S; int* r_edge_dst; unsigned* r_edge_cnt;
  u64* t_S; int* t_tok; unsigned* t_cnt;        // per-warp scratch for merging
  int* kept; int* r_nedge; int* r_outdeg;
  int* st_tok; int* st_pq;                      // staged followers [m*D + d-1], token -1 = past the path's end
  int* list;                                    // fused kernel: first kListCap matches
  int pool_words;                               // words from st_tok on (at least kPoolWords): one pool for the aggregations
};

constexpr int kMaxWarps = 32;

template <bool EXPORT>
__host__ __device__ constexpr size_t dag_smem_bytes() {
  size_t b = (size_t)CAP * 8 * 4 + (size_t)kStageWords * 8 + (size_t)kListCap * 4;
  if (EXPORT) {
    b += (size_t)CAP * 5 * 4;
    b += (size_t)MAXB * 16 + (size_t)MAXB * MAXKE * 16 + (size_t)kMaxWarps * 32 * 16 + (size_t)MAXB * 12;
  }
  return b;
}

template <bool EXPORT>
__device__ Smem carve(unsigned char* base) {
  Smem m;
  u64* p8 = reinterpret_cast<u64*>(base);
  if (EXPORT) {
    m.r_node_S = p8; p8 += MAXB;
    m.r_edge_S = p8; p8 += MAXB * MAXKE;
    m.t_S = p8; p8 += kMaxWarps * 32;
  }
  int* p4 = reinterpret_cast<int*>(p8);
  if (!EXPORT) {
    unsigned bytes;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(bytes));
    m.list = p4; p4 += kListCap;
    m.pool_words = (int)(bytes >> 2) - kListCap;
  }
  m.st_tok = p4; p4 += kStageWords;
  m.st_pq = p4; p4 += kStageWords;
  m.n_key = p4; p4 += CAP;
  m.n_Slo = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_Shi = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_Clo = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_Chi = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_call = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_ccur = reinterpret_cast<unsigned*>(p4); p4 += CAP;
  m.n_touch = p4; p4 += CAP;
  if (EXPORT) {
    m.list = p4; p4 += kListCap;
    m.pool_words = 0;
    m.e_key = p4; p4 += CAP;
    m.e_Slo = reinterpret_cast<unsigned*>(p4); p4 += CAP;
    m.e_Shi = reinterpret_cast<unsigned*>(p4); p4 += CAP;
    m.e_c = reinterpret_cast<unsigned*>(p4); p4 += CAP;
    m.e_touch = p4; p4 += CAP;
    m.r_node_tok = p4; p4 += MAXB;
    m.r_node_cnt = reinterpret_cast<unsigned*>(p4); p4 += MAXB;
    m.r_edge_dst = p4; p4 += MAXB * MAXKE;
    m.r_edge_cnt = reinterpret_cast<unsigned*>(p4); p4 += MAXB * MAXKE;
    m.t_tok = p4; p4 += kMaxWarps * 32;
    m.t_cnt = reinterpret_cast<unsigned*>(p4); p4 += kMaxWarps * 32;
    m.kept = p4; p4 += MAXB;
    m.r_nedge = p4; p4 += MAXB;
    m.r_outdeg = p4; p4 += MAXB;
  }
  return m;
}

// 16-bit tag of a token, never 0 (0 marks "no token")
__device__ __forceinline__ unsigned short tag_of(int tok) { return (unsigned short)(0x8000u | (((unsigned)tok * 2654435761u) >> 17)); }
__device__ __forceinline__ unsigned slot_hash(unsigned x) { return (x * 2654435761u) >> 22; }   // 10 bits = CAP
static_assert(CAP == 1024, "slot_hash yields 10 bits");

// Defaults of one query path: no draft, empty export.
template <bool EXPORT>
__device__ void write_defaults(const Dev& s, int i, int32_t* draft_tok, float* draft_score, float* draft_edge_w) {
  const int tid = threadIdx.x, D = s.D, B = s.B, Ke = s.Ke;
  for (int d = tid; d < D; d += blockDim.x) {
    draft_tok[(size_t)i * D + d] = -1;
    if (draft_score) draft_score[(size_t)i * D + d] = 0.0f;
    if (draft_edge_w) draft_edge_w[(size_t)i * D + d] = 0.0f;
  }
  if (EXPORT) {
    for (int x = tid; x < D * B; x += blockDim.x) {
      const size_t nx = (size_t)i * D * B + x;
      s.x_node_tok[nx] = -1; s.x_node_S[nx] = 0; s.x_node_cnt[nx] = 0; s.x_out_degree[nx] = 0;
    }
    for (int x = tid; x < D * B * Ke; x += blockDim.x) {
      const size_t ex = (size_t)i * D * B * Ke + x;
      s.x_edge_dst[ex] = -1; s.x_edge_S[ex] = 0; s.x_edge_cnt[ex] = 0;
    }
    for (int d = tid; d < D; d += blockDim.x) s.x_node_count[(size_t)i * D + d] = 0;
  }
}

// ---------------------------------------------------------------------------
// M <= 32, tree pool, layer-wise search and export: one warp per layer, then (not for the export) one
// warp walks.  The export rows must hold their defaults already (write_defaults followed by a barrier).
// ---------------------------------------------------------------------------
template <bool EXPORT>
__device__ void dag_small(const Dev& s, const Smem& sm, int i, int M, const int32_t* mlist,
                          const int32_t* plen, int poff, int root, int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                          float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int D = s.D, B = s.B, Ke = s.Ke;
  // per layer and lane: follower token, previous token, node score, edge weight; per layer: leader masks
  int* L_v = sm.st_tok;
  int* L_u = sm.st_tok + 32 * SDMS_MAX_DRAFT;
  unsigned* L_lead = reinterpret_cast<unsigned*>(sm.st_tok + 2 * 32 * SDMS_MAX_DRAFT);
  unsigned* L_elead = L_lead + SDMS_MAX_DRAFT;
  unsigned* L_best = L_elead + SDMS_MAX_DRAFT;      // per layer: the best node
  int* L_p = sm.st_tok + 3 * 32 * SDMS_MAX_DRAFT;   // fixed-point probability of the follower (tree pool)
  double* L_W = reinterpret_cast<double*>(sm.st_pq);
  double* L_we = L_W + 32 * SDMS_MAX_DRAFT;

  int gpos = 0, n_m = 0;
  if (lane < M) {
    gpos = mlist[lane];
    const int j = path_of(s, gpos);
    n_m = min(D, plen[j - poff] - 1 - (gpos - j * s.L));
  }
  for (int d = warp + 1; d <= D; d += nwarps) {
    const bool alive = d <= n_m;                        // candidate reaches layer d
    const bool alive_prev = lane < M && d - 1 <= n_m;   // ... reached layer d-1 (layer 0 is the root)
    const int v = alive ? ldm(s.tok + gpos + d) : -1;
    const unsigned p = alive ? (unsigned)ldm(s.pq + gpos + d) : 0u;
    const int u = !alive_prev ? -1 : (d == 1 ? root : ldm(s.tok + gpos + d - 1));
    const unsigned live = __ballot_sync(FULL, alive);
    const unsigned gv = __match_any_sync(FULL, v);                     // lanes on the same node
    const unsigned gu = __match_any_sync(FULL, u);                     // lanes with the same previous node
    const unsigned ge = gv & gu;                                       // lanes on the same edge
    u64 S_all, S_uv;
    group_sums(live, gv, ge, p, &S_all, &S_uv);
    const unsigned c_all = __popc(gv), c_uv = __popc(ge);
    const bool leader = alive && lane == __ffs(gv) - 1;
    const bool eleader = alive && lane == __ffs(ge) - 1;
    const double W = eq5_weight(s.alpha, S_all, c_all);
    const double w_uv = eq5_weight(s.alpha, S_uv, c_uv);
    const unsigned leaders = __ballot_sync(FULL, leader), eleaders = __ballot_sync(FULL, eleader);
    const int top = !EXPORT && s.mode == 1 ? warp_arg_first(leader, W, v) : -1;   // best node of the layer
    L_v[(d - 1) * 32 + lane] = v; L_u[(d - 1) * 32 + lane] = u; L_p[(d - 1) * 32 + lane] = (int)p;
    L_W[(d - 1) * 32 + lane] = W; L_we[(d - 1) * 32 + lane] = w_uv;
    if (lane == 0) {
      L_lead[d - 1] = leaders; L_elead[d - 1] = eleaders;
      L_best[d - 1] = top >= 0 ? 1u << top : 0u;
    }
    if (EXPORT && live) {
      int rank = 0;
      for (unsigned rem = leaders; rem; rem &= rem - 1) {
        const int src = __ffs(rem) - 1;
        const double ow = __shfl_sync(FULL, W, src);
        const int ot = __shfl_sync(FULL, v, src);
        if (ranks_before(ow, ot, W, v)) ++rank;
      }
      if (leader && rank < B) {
        const size_t nx = ((size_t)i * D + (d - 1)) * B + rank;
        s.x_node_tok[nx] = v; s.x_node_S[nx] = (int64_t)S_all; s.x_node_cnt[nx] = (int32_t)c_all;
      }
      if (lane == 0) s.x_node_count[(size_t)i * D + (d - 1)] = __popc(leaders);
      if (d > 1) {
        // rank of each previous-layer node, recomputed here so that layers stay independent
        const unsigned pu = alive_prev ? (unsigned)ldm(s.pq + gpos + d - 1) : 0u;
        const unsigned live_prev = __ballot_sync(FULL, alive_prev);
        u64 S_u, unused;
        group_sums(live_prev, gu, 0u, pu, &S_u, &unused);
        const double W_u = eq5_weight(s.alpha, S_u, __popc(gu));
        const bool uleader = alive_prev && lane == __ffs(gu) - 1;
        const unsigned uleaders = __ballot_sync(FULL, uleader);
        int urank = 0;
        for (unsigned rem = uleaders; rem; rem &= rem - 1) {
          const int src = __ffs(rem) - 1;
          const double ow = __shfl_sync(FULL, W_u, src);
          const int ot = __shfl_sync(FULL, u, src);
          if (ranks_before(ow, ot, W_u, u)) ++urank;
        }
        const int slot_u = __shfl_sync(FULL, urank, __ffs(gu) - 1);     // export slot of this lane's source node
        int erank = 0, deg = 0;
        for (unsigned rem = eleaders; rem; rem &= rem - 1) {
          const int src = __ffs(rem) - 1;
          const double ow = __shfl_sync(FULL, w_uv, src);
          const int ot = __shfl_sync(FULL, v, src);
          const int ou = __shfl_sync(FULL, u, src);
          if (ou == u) { ++deg; if (ranks_before(ow, ot, w_uv, v)) ++erank; }
        }
        if (eleader && slot_u < B) {
          const size_t nb = ((size_t)i * D + (d - 2)) * B + slot_u;
          if (erank < Ke) {
            s.x_edge_dst[nb * Ke + erank] = v; s.x_edge_S[nb * Ke + erank] = (int64_t)S_uv;
            s.x_edge_cnt[nb * Ke + erank] = (int32_t)c_uv;
          }
          if (erank == 0) s.x_out_degree[nb] = deg;
        }
      }
    }
  }
  if (EXPORT) return;
  __syncthreads();
  if (warp != 0) return;
  if (s.pool == 1) {
    // tree pool: only the candidates that spell the draft so far stay in play
    bool in_play = lane < M;
    int emitted = 0;
    for (int d = 1; d <= D; ++d) {
      const int v = L_v[(d - 1) * 32 + lane];
      const bool on = in_play && v >= 0;
      const unsigned live = __ballot_sync(FULL, on);
      if (live == 0) break;
      const unsigned gv = __match_any_sync(FULL, on ? v : -1);
      u64 S, unused;
      group_sums(live, gv, 0u, (unsigned)L_p[(d - 1) * 32 + lane], &S, &unused);
      const double W = eq5_weight(s.alpha, S, __popc(gv));
      const int src = warp_arg_first(on && lane == __ffs(gv) - 1, W, v);
      const int tok = __shfl_sync(FULL, v, src);
      const double Wb = __shfl_sync(FULL, W, src);
      if (lane == 0) {
        draft_tok[(size_t)i * D + (d - 1)] = tok;
        if (draft_score) draft_score[(size_t)i * D + (d - 1)] = (float)Wb;
        if (draft_edge_w) draft_edge_w[(size_t)i * D + (d - 1)] = (float)Wb;
      }
      in_play = on && v == tok;
      ++emitted;
    }
    if (lane == 0) draft_len[i] = emitted;
    return;
  }
  int cur = root, emitted = 0;
  for (int d = 1; d <= D; ++d) {
    const int v = L_v[(d - 1) * 32 + lane], u = L_u[(d - 1) * 32 + lane];
    const unsigned from_cur = __ballot_sync(FULL, u == cur);
    const unsigned pick = L_best[d - 1];
    if (pick == 0) break;
    const int src = __ffs(pick) - 1;
    const int tok = __shfl_sync(FULL, v, src);
    const double W = __shfl_sync(FULL, L_W[(d - 1) * 32 + lane], src);
    // the edge taken may not exist
    const unsigned emask = L_elead[d - 1] & from_cur & __ballot_sync(FULL, v == tok);
    const double we = __shfl_sync(FULL, L_we[(d - 1) * 32 + lane], emask ? __ffs(emask) - 1 : 0);
    if (lane == 0) {
      draft_tok[(size_t)i * D + (d - 1)] = tok;
      if (draft_score) draft_score[(size_t)i * D + (d - 1)] = (float)W;
      if (draft_edge_w) draft_edge_w[(size_t)i * D + (d - 1)] = emask ? (float)we : 0.0f;
    }
    cur = tok;
    ++emitted;
  }
  if (lane == 0) draft_len[i] = emitted;
}

// ---------------------------------------------------------------------------
// any M: layers in sequence, shared-memory hash tables
// ---------------------------------------------------------------------------
template <bool EXPORT>
__device__ void dag_block(const Dev& s, const Smem& sm, int i, int M, const int32_t* mlist,
                          const int32_t* plen, int poff, int root, int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                          float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  __shared__ int sh_nn, sh_ne, sh_overflow, sh_found, sh_cur, sh_nkept, sh_nnode_run, sh_node_total;
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ double sh_best_w, sh_best_ew;
  __shared__ int sh_best_tok, sh_best_valid;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int D = s.D, B = s.B, Ke = s.Ke;

  // stage every follower once: one round trip to memory instead of one per layer
  const bool staged = M * D <= kStageWords;
  if (staged) {
    for (int x = tid; x < M * D; x += blockDim.x) {
      const int m = x / D, dd = x - m * D + 1;
      const int gpos = mlist[m];
      const int j = path_of(s, gpos);
      const int e = gpos - j * s.L;
      const bool on = e + dd <= plen[j - poff] - 1;
      sm.st_tok[x] = on ? ldm(s.tok + gpos + dd) : -1;
      sm.st_pq[x] = on ? ldm(s.pq + gpos + dd) : 0;
    }
  }
  // too many followers to stage them all: stage one layer at a time (token and probability of every
  // candidate; the layer before stays, it holds the edges' sources), so that the passes and phases of
  // a layer read shared memory and only one sweep per layer goes to L2
  const bool rolling = !staged && M <= kRollMax && !(!EXPORT && s.pool == 1);
  // more candidates than that: the staging area is free and keeps a 16-bit tag of every candidate's token
  // of the layer before (written by the last sweep of that layer), so that the sweep that claims the
  // successors of the current node (phase 0 below) reads shared memory and goes to the histories only
  // for the candidates whose tag is the current node's
  const bool tagged = !EXPORT && !staged && !rolling && s.pool == 0 && M <= 4 * kStageWords;
  unsigned short* const tag = reinterpret_cast<unsigned short*>(sm.st_tok);
  int* const roll_odd = sm.st_tok;
  int* const roll_even = sm.st_tok + kRollMax;
  int* const roll_p = sm.st_tok + 2 * kRollMax;
  for (int x = tid; x < CAP; x += blockDim.x) {
    sm.n_key[x] = -1; sm.n_Slo[x] = 0; sm.n_Shi[x] = 0; sm.n_Clo[x] = 0; sm.n_Chi[x] = 0;
    sm.n_call[x] = 0; sm.n_ccur[x] = 0;
    if (EXPORT) { sm.e_key[x] = -1; sm.e_Slo[x] = 0; sm.e_Shi[x] = 0; sm.e_c[x] = 0; }
  }
  if (tid == 0) { sh_nn = 0; sh_ne = 0; sh_overflow = 0; sh_cur = root; sh_nkept = 0; }
  __syncthreads();

  const int npart_max = (int)(((long long)s.V * (EXPORT ? max(1, B) : 1) + CAP / 2 - 1) / (CAP / 2));
  int npart = 1;
  int emitted = 0;
  bool walking = true;

  for (int d = 1; d <= D; ++d) {
    if (!walking && !EXPORT) break;
    const int cur = sh_cur;
    const int nkept = EXPORT ? sh_nkept : 0;
    const bool tree = !EXPORT && s.pool == 1;       // only candidates that spell the draft so far take part
    const bool restricted = !EXPORT && !staged && !tree && s.mode != 1 && d > 1;   // staged candidates are cheap to revisit
    if (!EXPORT) {
      // first layer (or every layer in mode 1): every distinct follower is a node.  The guess is
      // optimistic, one node per 32 candidates (popular n-grams have far fewer distinct followers than
      // occurrences): a sweep that finds the table three quarters full stops at once and the layer is
      // redone with twice the residue classes, so a wrong guess costs a fraction of a sweep, while a
      // cautious one costs a full sweep for every class too many.  Restricted layers only hold the
      // successors of one node.
      npart = 1;
      if (!restricted) while (npart * (CAP / 2) * 32 < M && npart < npart_max) npart *= 2;
    }
    const unsigned short cur_tag = tag_of(cur);
    int* const cur_v = (d & 1) ? roll_odd : roll_even;
    const int* const prev_v = (d & 1) ? roll_even : roll_odd;
    if (rolling) {
      constexpr int kRollBatch = 8;
      for (int m0 = tid; m0 < M; m0 += kRollBatch * blockDim.x) {
        int tv[kRollBatch], tp[kRollBatch];
#pragma unroll
        for (int r = 0; r < kRollBatch; ++r) {
          const int m = m0 + r * blockDim.x;
          tv[r] = -1; tp[r] = 0;
          if (m >= M) continue;
          const int gpos = mlist[m];
          const int j = path_of(s, gpos);
          if (gpos - j * s.L + d <= plen[j - poff] - 1) { tv[r] = ldm(s.tok + gpos + d); tp[r] = ldm(s.pq + gpos + d); }
        }
#pragma unroll
        for (int r = 0; r < kRollBatch; ++r) {
          const int m = m0 + r * blockDim.x;
          if (m < M) { cur_v[m] = tv[r]; roll_p[m] = tp[r]; }
        }
      }
    }
    bool layer_done = false;
    // the tags describe the layer before only until the last residue class of a pass has overwritten them with
    // this layer's: a pass that is given up after that point and done again must not filter by them
    bool tags_fresh = true;
    while (!layer_done) {
      if (tid == 0) { sh_best_valid = 0; sh_nnode_run = 0; sh_node_total = 0; }
      if (EXPORT && tid < MAXB) { sm.r_nedge[tid] = 0; sm.r_outdeg[tid] = 0; }
      __syncthreads();
      bool overflowed = false;
      // while the layer can still be split further, a claim that does not find its slot within 64 probes gives the
      // pass up (it is redone): a first batch of 2048 claims can fill the table before any thread looks at the count
      const int probe_max = npart < npart_max ? 64 : CAP;
      const bool part_pow2 = (npart & (npart - 1)) == 0;        // nearly always: residue and quotient without a division
      const int part_shift = __ffs(npart) - 1;
      for (int part = 0; part < npart && !overflowed; ++part) {
        // ---- accumulate this residue class of follower tokens ----
        // Walking in mode 0 past the first layer, only successors of the current node can be chosen:
        // phase 0 claims a slot for each of them, phase 1 adds every candidate that lands on a claimed
        // slot.  Otherwise one phase claims and adds.
        for (int phase = restricted ? 0 : 1; phase < 2; ++phase) {
          for (int m0 = tid; m0 < M; m0 += kLoadBatch * blockDim.x) {
            if (npart < npart_max && *(volatile int*)&sh_nn > CAP * 3 / 4) break;   // too many nodes for this pass: it is redone
            int v[kLoadBatch], u[kLoadBatch];
            unsigned p[kLoadBatch];
#pragma unroll
            for (int r = 0; r < kLoadBatch; ++r) {                    // loads of the whole batch go out together
              const int m = m0 + r * blockDim.x;
              v[r] = -1; u[r] = -1; p[r] = 0;
              if (m >= M) continue;
              if (staged) {
                v[r] = sm.st_tok[m * D + d - 1];
                if (v[r] >= 0) { u[r] = d == 1 ? root : sm.st_tok[m * D + d - 2]; p[r] = (unsigned)sm.st_pq[m * D + d - 1]; }
                if (tree) for (int x = 1; x < d && v[r] >= 0; ++x) if (sm.st_tok[m * D + x - 1] != sh_draft[x - 1]) v[r] = -1;
              } else if (rolling) {
                v[r] = cur_v[m];
                if (v[r] >= 0) { u[r] = d == 1 ? root : prev_v[m]; p[r] = (unsigned)roll_p[m]; }
              } else {
                if (tagged && phase == 0 && tags_fresh && tag[m] != cur_tag) continue;   // its token of the layer before is not the current node
                const int gpos = mlist[m];
                const int j = path_of(s, gpos);
                if (gpos - j * s.L + d <= plen[j - poff] - 1) {
                  v[r] = ldm(s.tok + gpos + d);
                  u[r] = d == 1 ? root : ldm(s.tok + gpos + d - 1);
                  p[r] = (unsigned)ldm(s.pq + gpos + d);
                  if (tree) for (int x = 1; x < d && v[r] >= 0; ++x) if (ldm(s.tok + gpos + x) != sh_draft[x - 1]) v[r] = -1;
                }
                if (tagged && phase == 1 && part == npart - 1) tag[m] = v[r] >= 0 ? tag_of(v[r]) : (unsigned short)0;
              }
            }
#pragma unroll
            for (int r = 0; r < kLoadBatch; ++r) {
              const int vv = v[r], uu = u[r];
              const unsigned pp = p[r];
              if (vv < 0 || (npart > 1 && (part_pow2 ? (vv & (npart - 1)) : vv % npart) != part)) continue;
              if (phase == 0 && uu != cur) continue;
              const unsigned vq = part_pow2 ? (unsigned)vv >> part_shift : (unsigned)(vv / npart);
              unsigned h = slot_hash(vq);
              int slot = -1;
              if (phase == 1 && restricted) {                          // read-only: is vv a claimed successor?
                for (int probe = 0; probe < CAP; ++probe) {
                  const int key = sm.n_key[h];
                  if (key == vv) { slot = (int)h; break; }
                  if (key == -1) break;
                  h = (h + 1) & (CAP - 1);
                }
                if (slot < 0) continue;
              } else {
                for (int probe = 0; probe < probe_max; ++probe) {
                  const int old = atomicCAS(&sm.n_key[h], -1, vv);
                  if (old == -1) sm.n_touch[atomicAdd(&sh_nn, 1)] = (int)h;
                  if (old == -1 || old == vv) { slot = (int)h; break; }
                  h = (h + 1) & (CAP - 1);
                }
                if (slot < 0) { sh_overflow = 1; continue; }
                if (phase == 0) continue;
              }
              add64(&sm.n_Slo[slot], &sm.n_Shi[slot], pp);
              atomicAdd(&sm.n_call[slot], 1u);
              if (uu == cur) { add64(&sm.n_Clo[slot], &sm.n_Chi[slot], pp); atomicAdd(&sm.n_ccur[slot], 1u); }
              if (EXPORT && d > 1) {
                int b = -1;
                for (int x = 0; x < nkept; ++x) if (sm.kept[x] == uu) { b = x; break; }
                if (b >= 0) {
                  const int ekey = vv * MAXB + b;               // (destination, kept source) in one word
                  unsigned he = slot_hash(vq * 37u + (unsigned)b);
                  int es = -1;
                  for (int probe = 0; probe < CAP; ++probe) {
                    const int old = atomicCAS(&sm.e_key[he], -1, ekey);
                    if (old == -1) sm.e_touch[atomicAdd(&sh_ne, 1)] = (int)he;
                    if (old == -1 || old == ekey) { es = (int)he; break; }
                    he = (he + 1) & (CAP - 1);
                  }
                  if (es < 0) { sh_overflow = 1; continue; }
                  add64(&sm.e_Slo[es], &sm.e_Shi[es], pp);
                  atomicAdd(&sm.e_c[es], 1u);
                }
              }
            }
          }
          if (phase == 0) __syncthreads();
        }
        __syncthreads();
        const int nn = sh_nn, ne = EXPORT ? sh_ne : 0;
        overflowed = sh_overflow || (npart < npart_max && (nn > CAP * 3 / 4 || ne > CAP * 3 / 4));
        if (!overflowed) {
          // ---- selections, one warp each ----
          if (warp == 0 && walking) {
            Cand best; best.valid = 0; best.w = 0; best.tok = 0; best.S = 0; best.cnt = 0;
            for (int x = lane; x < nn; x += 32) {
              const int sl = sm.n_touch[x];
              Cand c;
              c.tok = sm.n_key[sl]; c.S = 0;
              c.valid = s.mode == 1 || tree || sm.n_ccur[sl] > 0;
              c.w = eq5_weight(s.alpha, get64(sm.n_Slo, sm.n_Shi, sl), sm.n_call[sl]);
              c.cnt = (unsigned)sl;                  // carry the slot: the edge weight is read from it below
              if (c.valid && (!best.valid || ranks_before(c.w, c.tok, best.w, best.tok))) best = c;
            }
            best = warp_best(best);
            if (lane == 0 && best.valid &&
                (!sh_best_valid || ranks_before(best.w, best.tok, sh_best_w, sh_best_tok))) {
              const int sl = (int)best.cnt;
              sh_best_valid = 1; sh_best_w = best.w; sh_best_tok = best.tok;
              sh_best_ew = tree ? best.w
                         : sm.n_ccur[sl] ? eq5_weight(s.alpha, get64(sm.n_Clo, sm.n_Chi, sl), sm.n_ccur[sl]) : 0.0;
            }
          }
          if (EXPORT && warp == 1) {
            const int nrun = sh_nnode_run;
            auto get = [&](int x) {
              Cand c; c.valid = 1;
              if (x < nn) { const int sl = sm.n_touch[x]; c.tok = sm.n_key[sl]; c.S = get64(sm.n_Slo, sm.n_Shi, sl); c.cnt = sm.n_call[sl]; }
              else { c.tok = sm.r_node_tok[x - nn]; c.S = sm.r_node_S[x - nn]; c.cnt = sm.r_node_cnt[x - nn]; }
              c.w = eq5_weight(s.alpha, c.S, c.cnt);
              return c;
            };
            int* tt = sm.t_tok + warp * 32; u64* tS = sm.t_S + warp * 32; unsigned* tc = sm.t_cnt + warp * 32;
            const int got = warp_topk(nn + nrun, get, B, tt, tS, tc);
            for (int x = lane; x < got; x += 32) { sm.r_node_tok[x] = tt[x]; sm.r_node_S[x] = tS[x]; sm.r_node_cnt[x] = tc[x]; }
            if (lane == 0) { sh_nnode_run = got; sh_node_total += nn; }
          }
          if (EXPORT && warp >= 2 && d > 1) {
            for (int b = warp - 2; b < nkept; b += nwarps - 2) {
              const int nrun = sm.r_nedge[b];
              int deg = 0;
              for (int x = lane; x < ne; x += 32) deg += sm.e_key[sm.e_touch[x]] % MAXB == b;
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) deg += __shfl_xor_sync(FULL, deg, o);
              auto get = [&](int x) {
                Cand c;
                if (x < ne) {
                  const int sl = sm.e_touch[x];
                  c.valid = sm.e_key[sl] % MAXB == b; c.tok = sm.e_key[sl] / MAXB;
                  c.S = get64(sm.e_Slo, sm.e_Shi, sl); c.cnt = sm.e_c[sl];
                } else {
                  const int y = b * MAXKE + (x - ne);
                  c.valid = 1; c.tok = sm.r_edge_dst[y]; c.S = sm.r_edge_S[y]; c.cnt = sm.r_edge_cnt[y];
                }
                c.w = eq5_weight(s.alpha, c.S, c.cnt);
                return c;
              };
              int* tt = sm.t_tok + warp * 32; u64* tS = sm.t_S + warp * 32; unsigned* tc = sm.t_cnt + warp * 32;
              const int got = warp_topk(ne + nrun, get, Ke, tt, tS, tc);
              for (int x = lane; x < got; x += 32) {
                const int y = b * MAXKE + x;
                sm.r_edge_dst[y] = tt[x]; sm.r_edge_S[y] = tS[x]; sm.r_edge_cnt[y] = tc[x];
              }
              if (lane == 0) { sm.r_nedge[b] = got; sm.r_outdeg[b] += deg; }
              __syncwarp();
            }
          }
        }
        __syncthreads();
        // ---- wipe the touched slots for the next pass ----
        for (int x = tid; x < nn; x += blockDim.x) {
          const int sl = sm.n_touch[x];
          sm.n_key[sl] = -1; sm.n_Slo[sl] = 0; sm.n_Shi[sl] = 0; sm.n_Clo[sl] = 0; sm.n_Chi[sl] = 0;
          sm.n_call[sl] = 0; sm.n_ccur[sl] = 0;
        }
        if (EXPORT)
          for (int x = tid; x < ne; x += blockDim.x) {
            const int sl = sm.e_touch[x];
            sm.e_key[sl] = -1; sm.e_Slo[sl] = 0; sm.e_Shi[sl] = 0; sm.e_c[sl] = 0;
          }
        __syncthreads();
        if (tid == 0) { sh_nn = 0; sh_ne = 0; sh_overflow = 0; }
        __syncthreads();
      }
      if (overflowed && npart < npart_max) {
        npart = min(npart * 2, npart_max);          // redo the layer with smaller residue classes
        tags_fresh = false;
      } else {
        layer_done = true;
      }
    }
    // ---- close the layer ----
    if (tid == 0) {
      sh_found = 0;
      if (walking && sh_best_valid) {
        sh_found = 1;
        draft_tok[(size_t)i * D + (d - 1)] = sh_best_tok;
        sh_draft[d - 1] = sh_best_tok;
        if (draft_score) draft_score[(size_t)i * D + (d - 1)] = (float)sh_best_w;
        if (draft_edge_w) draft_edge_w[(size_t)i * D + (d - 1)] = (float)sh_best_ew;
        sh_cur = sh_best_tok;
      }
    }
    if (EXPORT) {
      const int nrun = sh_nnode_run;
      if (d > 1)
        for (int x = tid; x < nkept * Ke; x += blockDim.x) {
          const int b = x / Ke, r = x % Ke;
          if (r < sm.r_nedge[b]) {
            const size_t ex = (((size_t)i * D + (d - 2)) * B + b) * Ke + r;
            const int y = b * MAXKE + r;
            s.x_edge_dst[ex] = sm.r_edge_dst[y]; s.x_edge_S[ex] = (int64_t)sm.r_edge_S[y];
            s.x_edge_cnt[ex] = (int32_t)sm.r_edge_cnt[y];
          }
          if (r == 0) s.x_out_degree[((size_t)i * D + (d - 2)) * B + b] = sm.r_outdeg[b];
        }
      __syncthreads();
      for (int x = tid; x < nrun; x += blockDim.x) {
        const size_t nx = ((size_t)i * D + (d - 1)) * B + x;
        s.x_node_tok[nx] = sm.r_node_tok[x]; s.x_node_S[nx] = (int64_t)sm.r_node_S[x];
        s.x_node_cnt[nx] = (int32_t)sm.r_node_cnt[x];
        sm.kept[x] = sm.r_node_tok[x];
      }
      if (tid == 0) { s.x_node_count[(size_t)i * D + (d - 1)] = sh_node_total; sh_nkept = nrun; }
    }
    __syncthreads();
    if (walking) {
      if (sh_found) ++emitted; else walking = false;
    }
    // expected growth of the next layer decides where its pass count starts
    if (EXPORT) {
      const int tot = sh_node_total;
      int next = 1;
      while (next * (CAP / 2) < 2 * tot && next < npart_max) next *= 2;
      npart = min(next, npart_max);
      if (tot == 0) { break; }                      // no candidate reaches this depth: nor any deeper one
    }
    __syncthreads();
  }
  if (tid == 0) draft_len[i] = emitted;
}

// List pool (ablation): no merging; the draft is the single candidate that weighs most by Eq. 5 on
// its own tokens (S = sum of its probabilities, Freq = its length), ties to the smaller position.
__device__ void list_pool(const Dev& s, int i, int M, const int32_t* mlist, const int32_t* plen, int poff,
                          int32_t* __restrict__ draft_tok, int32_t* __restrict__ draft_len,
                          float* __restrict__ draft_score, float* __restrict__ draft_edge_w) {
  __shared__ double sh_w[kMaxWarps];
  __shared__ int sh_g[kMaxWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int D = s.D;
  double best_w = 0.0;
  int best_g = -1;
  for (int m = tid; m < M; m += blockDim.x) {
    const int gpos = mlist[m];
    const int j = path_of(s, gpos);
    const int n_m = min(D, plen[j - poff] - 1 - (gpos - j * s.L));
    u64 S = 0;
    for (int d = 1; d <= n_m; ++d) S += (unsigned)ldm(s.pq + gpos + d);
    const double w = eq5_weight(s.alpha, S, (unsigned)n_m);
    if (best_g < 0 || ranks_before(w, gpos, best_w, best_g)) { best_w = w; best_g = gpos; }
  }
  int src = warp_arg_first(best_g >= 0, best_w, best_g);
  if (src < 0) src = 0;
  best_w = __shfl_sync(FULL, best_w, src); best_g = __shfl_sync(FULL, best_g, src);
  if (lane == 0) { sh_w[warp] = best_w; sh_g[warp] = best_g; }
  __syncthreads();
  if (warp != 0) return;
  best_w = lane < nwarps ? sh_w[lane] : 0.0; best_g = lane < nwarps ? sh_g[lane] : -1;
  src = warp_arg_first(best_g >= 0, best_w, best_g);
  best_g = __shfl_sync(FULL, best_g, src < 0 ? 0 : src);
  const int j = best_g / s.L;
  const int n_m = min(D, plen[j - poff] - 1 - (best_g - j * s.L));
  if (lane < n_m) {
    const float w = (float)eq5_weight(s.alpha, (unsigned)ldm(s.pq + best_g + 1 + lane), 1u);
    draft_tok[(size_t)i * D + lane] = ldm(s.tok + best_g + 1 + lane);
    if (draft_score) draft_score[(size_t)i * D + lane] = w;
    if (draft_edge_w) draft_edge_w[(size_t)i * D + lane] = w;
  }
  if (lane == 0) draft_len[i] = n_m;
}

// ---- all layers at once (layer-wise search, a few hundred matches) --------------------------------
// dag_block takes the layers one after the other because the walk decides which node's successors
// count; each layer then costs a few barriers and a chain of shared-memory atomics whatever M is.
// Here every layer is aggregated at the same time into a table of its own (follower token -> sum of
// probabilities, count) and its heaviest node found.  The pool of shared words (staging area and
// dag_block's tables, kPoolWords in a row) holds the staged followers and as many layers' tables as
// fit; more layers take more rounds.
constexpr int kPoolWords = 2 * kStageWords + 8 * CAP;
constexpr int kLayerWords = 4;                    // per table slot: key, low and high part of the sum, count

struct LayerTable { int* key; unsigned* lo; unsigned* hi; unsigned* cnt; };
__device__ __forceinline__ LayerTable layer_table(int* pool, int cap, int l) {
  int* b = pool + (size_t)l * kLayerWords * cap;
  return LayerTable{b, reinterpret_cast<unsigned*>(b + cap), reinterpret_cast<unsigned*>(b + 2 * cap), reinterpret_cast<unsigned*>(b + 3 * cap)};
}
// slot of `key` in an open-addressing table of `cap` (power of two) slots; claims one if INSERT
template <bool INSERT>
__device__ __forceinline__ int table_slot(int* keys, int cap, int shift, int key) {
  unsigned h = ((unsigned)key * 2654435761u) >> shift;
#pragma unroll 1
  for (int probe = 0; probe < cap; ++probe) {
    const int old = INSERT ? atomicCAS(&keys[h], -1, key) : keys[h];
    if (old == key || (INSERT && old == -1)) return (int)h;
    if (!INSERT && old == -1) return -1;
    h = (h + 1) & (cap - 1);
  }
  return -1;
}
// Sums of 30-bit probabilities are kept as two 32-bit sums, of the low 16 bits and of the rest: each
// stays below 2^32 for any number of candidates a CTA handles, and an add needs no result back (no
// carry to pass on), so the adds do not stall their thread.
__device__ __forceinline__ void add_split(unsigned* lo16, unsigned* hi, unsigned* cnt, unsigned pq) {
  atomicAdd(lo16, pq & 0xffffu);
  atomicAdd(hi, pq >> 16);
  atomicAdd(cnt, 1u);
}
__device__ __forceinline__ u64 weight_bits(double alpha, const unsigned* lo16, const unsigned* hi, const unsigned* cnt, int x) {
  return (u64)__double_as_longlong(eq5_weight(alpha, ((u64)hi[x] << 16) + lo16[x], cnt[x]));
}

// How many layers' tables fit beside the staged followers (0: use dag_block).  Three words are staged
// per follower: token, probability, and the table slots found for it (so that no pass probes twice).
__device__ __forceinline__ int layers_per_round(int M, int D, int* cap_out) {
  const int staged = (3 * M * D + 1) & ~1;
  int cap = 64;                                    // more slots than keys: a probe always ends at a free slot
  while (cap <= M) cap *= 2;
  // twice the slots shorten the probe sequences (a warp waits for its longest); taken when all
  // layers still fit in one round
  if ((kPoolWords - staged) / (kLayerWords * 2 * cap) >= D) cap *= 2;
  *cap_out = cap;
  return (kPoolWords - staged) / (kLayerWords * cap);
}

__device__ __forceinline__ bool layers_in_round_ok(int M, int D) {
  int cap;
  return layers_per_round(M, D, &cap) >= min(D, 2);
}

__device__ void dag_layers(const Dev& s, const Smem& sm, int i, int M, const int32_t* mlist, const int32_t* plen,
                           int poff, int32_t* draft_tok, int32_t* draft_len, float* draft_score, float* draft_edge_w) {
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_lwhi[SDMS_MAX_DRAFT], sh_lwlo[SDMS_MAX_DRAFT];   // heaviest node of the layer
  __shared__ int sh_lt[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_eSlo[SDMS_MAX_DRAFT], sh_eShi[SDMS_MAX_DRAFT], sh_ec[SDMS_MAX_DRAFT];
  __shared__ int sh_emitted, sh_walking;
  const int tid = threadIdx.x, D = s.D;
  int cap;
  const int per_round = min(D, layers_per_round(M, D, &cap));
  const int lcap = 31 - __clz(cap), shift = 32 - lcap;
  int* st_tok = sm.st_tok;                         // [m * D + d - 1], -1 past the end of the path
  int* st_pq = sm.st_tok + M * D;
  int* st_slot = sm.st_tok + 2 * M * D;            // slot of each staged follower
  int* pool = sm.st_tok + ((3 * M * D + 1) & ~1);
  const int lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int nchunk = (M + 31) >> 5;                // a warp takes 32 matches of one layer at a time

  if (tid < D) { sh_lwhi[tid] = 0; sh_lwlo[tid] = 0; sh_lt[tid] = INT_MAX; sh_eSlo[tid] = 0; sh_eShi[tid] = 0; sh_ec[tid] = 0; }
  if (tid == 0) { sh_emitted = 0; sh_walking = 1; }
  // stage the followers: a thread asks for four entries before it stores the first
  {
    int lD = 0;
    while ((1 << lD) < D) ++lD;                    // entries are numbered m << lD | d - 1: no division
    constexpr int kBatch = 4;
#pragma unroll 1
    for (int x0 = tid; x0 < (M << lD); x0 += kBatch * blockDim.x) {
      int tk[kBatch], pr[kBatch];
#pragma unroll
      for (int r = 0; r < kBatch; ++r) {
        const int x = x0 + r * blockDim.x;
        const int m = x >> lD, dd = (x & ((1 << lD) - 1)) + 1;
        tk[r] = -1; pr[r] = 0;
        if (m >= M || dd > D) continue;
        const int gpos = mlist[m];
        const int j = path_of(s, gpos);
        if (gpos - j * s.L + dd <= plen[j - poff] - 1) { tk[r] = ldm(s.tok + gpos + dd); pr[r] = ldm(s.pq + gpos + dd); }
      }
#pragma unroll
      for (int r = 0; r < kBatch; ++r) {
        const int x = x0 + r * blockDim.x;
        const int m = x >> lD, dd = (x & ((1 << lD) - 1)) + 1;
        if (m < M && dd <= D) { st_tok[m * D + dd - 1] = tk[r]; st_pq[m * D + dd - 1] = pr[r]; }
      }
    }
  }

#pragma unroll 1
  for (int d0 = 1; d0 <= D; d0 += per_round) {
    const int nl = min(per_round, D - d0 + 1);
    // empty tables: keys -1, sums 0
#pragma unroll 1
    for (int x = tid; x < ((nl * kLayerWords) << lcap); x += blockDim.x) pool[x] = ((x >> lcap) & (kLayerWords - 1)) == 0 ? -1 : 0;
    __syncthreads();
    if (!sh_walking) break;
    // pass 0: node sums; passes 1, 2: the layer's heaviest weight, the upper half of the weight's bit pattern first, then the
    // lower half among those (weights are >= 0, so the patterns order like the values); pass 3: the smallest token that has it
#pragma unroll 1
    for (int pass = 0; pass < 4; ++pass) {
#pragma unroll 1
      for (int task = warp; task < nl * nchunk; task += nwarps) {
        const int l = task / nchunk, m = ((task - l * nchunk) << 5) + lane;
        const int d = d0 + l, at = m * D + d - 1;
        const int v = m < M ? st_tok[at] : -1;
        if (v < 0) continue;
        const LayerTable t = layer_table(pool, cap, l);
        if (pass == 0) {
          const int sl = table_slot<true>(t.key, cap, shift, v);
          st_slot[at] = sl;
          add_split(&t.lo[sl], &t.hi[sl], &t.cnt[sl], (unsigned)st_pq[at]);
          continue;
        }
        const u64 w = weight_bits(s.alpha, t.lo, t.hi, t.cnt, st_slot[at]);
        const unsigned whi = (unsigned)(w >> 32), wlo = (unsigned)w;
        if (pass == 1) atomicMax(&sh_lwhi[d - 1], whi);
        else if (pass == 2) { if (sh_lwhi[d - 1] == whi) atomicMax(&sh_lwlo[d - 1], wlo); }
        else if (sh_lwhi[d - 1] == whi && sh_lwlo[d - 1] == wlo) atomicMin(&sh_lt[d - 1], v);
      }
      __syncthreads();
    }
    // the draft through this round's layers
    if (tid == 0) {
      int emitted = sh_emitted;
#pragma unroll 1
      for (int d = d0; d < d0 + nl; ++d) {
        const int next = sh_lt[d - 1];
        if (next == INT_MAX) { sh_walking = 0; break; }
        draft_tok[(size_t)i * D + d - 1] = next;
        if (draft_score)
          draft_score[(size_t)i * D + d - 1] = (float)__longlong_as_double((long long)((u64)sh_lwhi[d - 1] << 32 | sh_lwlo[d - 1]));
        sh_draft[d - 1] = next;
        ++emitted;
      }
      sh_emitted = emitted;
    }
    __syncthreads();
  }
  // weight of the edges the draft took (Eq. 5 over the candidates that contain the edge)
  const int emitted = sh_emitted;
#pragma unroll 1
  for (int task = warp; task < emitted * nchunk; task += nwarps) {
    const int l = task / nchunk, m = ((task - l * nchunk) << 5) + lane;
    const int d = l + 1, at = m * D + d - 1;
    if (m < M && st_tok[at] == sh_draft[d - 1] && (d == 1 || st_tok[at - 1] == sh_draft[d - 2]))
      add_split(&sh_eSlo[d - 1], &sh_eShi[d - 1], &sh_ec[d - 1], (unsigned)st_pq[at]);
  }
  __syncthreads();
  if (tid < emitted && draft_edge_w)
    draft_edge_w[(size_t)i * D + tid] =
        sh_ec[tid] ? (float)__longlong_as_double((long long)weight_bits(s.alpha, sh_eSlo, sh_eShi, sh_ec, tid)) : 0.0f;
  if (tid == 0) draft_len[i] = emitted;
}

// ---- the greedy walk (search modes 0 and 2) -----------------------------------------------------------
// One CTA is bound here by how many dependent instructions follow one another (4.3 cycles each, 33 for a shared load, 50 to
// 70 for a taken or divergent branch): so items are handled in fixed batches of registers, without branches in between.

__device__ __forceinline__ u64 max64(u64 a, u64 b) { return a > b ? a : b; }

// M <= 32: lane m of a warp holds candidate m.  A warp per layer fetches the followers and forms every candidate's node
// sum (a broadcast read of the layer's row: 32 compares, where __match_any_sync on distinct tokens takes 364 cycles);
// one warp walks.  Where all candidates on a node go on with the same token nothing is compared.
constexpr int kRow = 36;                 // words per layer: 16-byte aligned, rows on different banks

__device__ void dag_walk_warp(const Dev& s, int i, int M, const int32_t* mlist, const int32_t* plen, int poff,
                              int32_t* draft_tok, int32_t* draft_len, float* draft_score, float* draft_edge_w) {
  // (shared memory is named here and not passed in, so that every access is known to be to shared memory: atomics
  // through a generic pointer cost several hundred cycles each)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, D = s.D;
  int* const row_v = reinterpret_cast<int*>(smem_raw) + kListCap;     // [d - 1][kRow] token, -1: the candidate has ended
  int* const row_p = row_v + kRow * SDMS_MAX_DRAFT;
  unsigned* const row_lo = reinterpret_cast<unsigned*>(row_p + kRow * SDMS_MAX_DRAFT);     // node sum of the candidate's token
  unsigned* const row_hi = row_lo + kRow * SDMS_MAX_DRAFT;
  unsigned* const row_c = row_hi + kRow * SDMS_MAX_DRAFT;
  if (warp < D) {
    int gpos = 0, n_m = 0;
    if (lane < M) {
      gpos = mlist[lane];
      const int j = path_of(s, gpos);
      n_m = min(D, plen[j - poff] - 1 - (gpos - j * s.L));
    }
    for (int d = warp + 1; d <= D; d += nwarps) {
      const int v = d <= n_m ? ldm(s.tok + gpos + d) : -1, p = d <= n_m ? ldm(s.pq + gpos + d) : 0;
      int* const rv = row_v + (d - 1) * kRow;
      int* const rp = row_p + (d - 1) * kRow;
      rv[lane] = v; rp[lane] = p;
      __syncwarp();
      u64 S = 0;
      unsigned c = 0;
#pragma unroll 2
      for (int x = 0; x < M; x += 4) {
        const int4 tv = *reinterpret_cast<const int4*>(rv + x), tp = *reinterpret_cast<const int4*>(rp + x);
        if (tv.x == v) { S += (unsigned)tp.x; ++c; }
        if (tv.y == v) { S += (unsigned)tp.y; ++c; }
        if (tv.z == v) { S += (unsigned)tp.z; ++c; }
        if (tv.w == v) { S += (unsigned)tp.w; ++c; }
      }
      row_lo[(d - 1) * kRow + lane] = (unsigned)S; row_hi[(d - 1) * kRow + lane] = (unsigned)(S >> 32);
      row_c[(d - 1) * kRow + lane] = c;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  auto sum_at = [&](int d, int x) { return ((u64)row_hi[(d - 1) * kRow + x] << 32) | row_lo[(d - 1) * kRow + x]; };
  unsigned from = __ballot_sync(FULL, lane < M);       // candidates on the current node
  int emitted = 0;
  int my_tok = -1, my_src = 0;                         // lane d - 1 keeps what was decided for layer d
  unsigned my_node = 0u, my_edge = 0u;
  int v = row_v[lane];
#pragma unroll 1
  for (int d = 1; d <= D; ++d) {
    const int v_next = d < D ? row_v[d * kRow + lane] : -1;
    const bool on = (from >> lane & 1u) && v >= 0;
    const unsigned succ = __ballot_sync(FULL, on);
    if (succ == 0u) break;
    int src = __ffs(succ) - 1;
    int tok = __shfl_sync(FULL, v, src);
    if (__ballot_sync(FULL, on && v != tok)) {         // several successors: the heaviest
      src = warp_arg_first(on, eq5_weight(s.alpha, sum_at(d, lane), row_c[(d - 1) * kRow + lane]), v);
      tok = __shfl_sync(FULL, v, src);
    }
    const unsigned node = __ballot_sync(FULL, v == tok);
    if (lane == d - 1) { my_tok = tok; my_src = src; my_node = node; my_edge = node & from; }
    from = node; v = v_next;
    emitted = d;
  }
  if (lane < D) {
    u64 S = 0, Se = 0;
    if (lane < emitted) {
      S = Se = sum_at(lane + 1, my_src);
      if (my_edge != my_node) {
        Se = 0;
        for (unsigned rem = my_edge; rem; rem &= rem - 1u) Se += (unsigned)row_p[lane * kRow + __ffs(rem) - 1];
      }
    }
    const size_t at = (size_t)i * D + lane;
    draft_tok[at] = my_tok;
    if (draft_score) draft_score[at] = my_tok >= 0 ? (float)eq5_weight(s.alpha, S, __popc(my_node)) : 0.0f;
    if (draft_edge_w) draft_edge_w[at] = my_tok >= 0 ? (float)eq5_weight(s.alpha, Se, __popc(my_edge)) : 0.0f;
  }
  if (lane == 0) draft_len[i] = emitted;
}

// More candidates.  As many layers at once as fit shared memory (all of them up to a hundred-odd candidates), a table per
// layer, all (candidate, layer) items side by side, four of a thread's at a time:
//   sums   an item claims the slot of its token in the layer's table and adds its probability; it notes the slot
//   keys   the slot becomes the item's key: its node's weight and its token in one word that orders by weight, then by
//          smaller token (PACKED: with alpha = 1 the weight is the sum itself; else weight and token stay apart)
//   walk   per layer the largest key among the candidates on the current node, four candidates per lane: one warp, and no
//          barrier, up to 128 candidates; a layer's rows do not depend on the walk and are fetched a layer ahead
constexpr int kWalkMaxCap = 8192;        // most slots of a layer's table

struct WalkPlan { int cap, stride, layers; bool packed; };    // slots per table, words per row of items, layers per round
// layers = 0: does not fit
__device__ __forceinline__ WalkPlan walk_plan(const Dev& s, int M, int pool_words) {
  WalkPlan w;
  w.cap = 64;
  while (7 * w.cap < 8 * M) w.cap *= 2;                // at most 7/8 full
  w.stride = ((M + 31) & ~31) + 4;
  // sum (30 bits and those of the number of candidates) and token side by side in 64 bits
  w.packed = s.alpha == 1.0 && (32 - __clz(M)) + (32 - __clz(s.V)) + 30 <= 64;
  const int per_layer = (w.packed ? 3 : 4) * (w.stride + w.cap), room = pool_words - w.stride;
  w.layers = w.cap > kWalkMaxCap || room < per_layer ? 0 : s.D * per_layer <= room ? s.D : room / per_layer;
  return w;
}

template <bool PACKED>
__device__ void dag_walk(const Dev& s, const WalkPlan w, int i, int M, const int32_t* mlist, const int32_t* plen,
                         int poff, int root, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                         float* draft_edge_w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ u64 sh_best[2][kMaxWarps];
  __shared__ int sh_tok[2][kMaxWarps];
  __shared__ unsigned sh_e[SDMS_MAX_DRAFT][3];          // walk by several warps: edge sum (lower 16 bits, rest), count
  __shared__ int sh_cur;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5, D = s.D;
  const int cap = w.cap, mask = cap - 1, shift = __clz(cap) + 1, stride = w.stride;
  const int all = w.layers * cap, items = w.layers * stride;
  int* const keys = reinterpret_cast<int*>(smem_raw) + kListCap;                 // tables, every array: [layer of the round][slot]
  unsigned* const sum_lo = reinterpret_cast<unsigned*>(keys + all);
  unsigned* const sum_hi = sum_lo + all;
  unsigned* const cnt = sum_hi + all;                   // not packed
  unsigned* const row_prev = reinterpret_cast<unsigned*>(keys + (PACKED ? 3 : 4) * all);     // last layer's tokens of the round before
  unsigned* const rows_t = row_prev + stride;           // items, every array: [layer][candidate]: token, -1: has ended; packed: then lower key word
  unsigned* const rows_p = rows_t + items;              // probability
  unsigned* const rows_h = rows_p + items;              // slot, then upper key word
  unsigned* const rows_l = PACKED ? rows_t : rows_h + items;                     // lower key word
  // the token of an item as the walk compares it: packed, its complement in the lower bits of the key (0: has ended)
  const int tok_bits = 32 - __clz(s.V);
  const unsigned tok_mask = PACKED ? (1u << tok_bits) - 1u : ~0u;
  auto code_of = [&](int tok) { return PACKED ? ~(unsigned)tok & tok_mask : (unsigned)tok; };
  const int walkers = min(nwarps, (M + 127) >> 7), width = walkers * 32;

  if (tid < D) { sh_e[tid][0] = 0u; sh_e[tid][1] = 0u; sh_e[tid][2] = 0u; }
  // lane d - 1 of warp 0 keeps what layer d comes to
  int my_tok = -1;
  u64 my_key = 0ull;
  unsigned my_e0 = 0u, my_e1 = 0u, my_e2 = 0u;
  int cur = root, emitted = 0;
#pragma unroll 1
  for (int d0 = 1; d0 <= D; d0 += w.layers) {
    const int nl = min(w.layers, D - d0 + 1);
    const int lN = nl > 1 ? 32 - __clz(nl - 1) : 0, nN = 1 << lN;       // items are numbered m << lN | layer: no division
    {
      int4* const z = reinterpret_cast<int4*>(keys);
      const int key_end = all / 4, end = key_end * (PACKED ? 3 : 4);
      for (int x = tid; x < key_end; x += blockDim.x) z[x] = make_int4(-1, -1, -1, -1);
      for (int x = key_end + tid; x < end; x += blockDim.x) z[x] = make_int4(0, 0, 0, 0);
    }
    // the followers: four entries of a thread are asked for before the first is stored
#pragma unroll 1
    for (int x0 = tid; x0 < (M << lN); x0 += 4 * blockDim.x) {
      int gpos[4], left[4], tk[4], pr[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) gpos[r] = mlist[min((x0 + r * (int)blockDim.x) >> lN, M - 1)];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int j = path_of(s, gpos[r]);
        left[r] = plen[j - poff] - 1 - (gpos[r] - j * s.L);              // followers of the match
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int l = (x0 + r * (int)blockDim.x) & (nN - 1);
        const bool on = d0 + l <= left[r] && l < nl;
        tk[r] = -1; pr[r] = 0;
        if (on) { tk[r] = ldm(s.tok + gpos[r] + d0 + l); pr[r] = ldm(s.pq + gpos[r] + d0 + l); }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int x = x0 + r * (int)blockDim.x, m = x >> lN, l = x & (nN - 1);
        if (m < M && l < nl) { rows_t[l * stride + m] = (unsigned)tk[r]; rows_p[l * stride + m] = (unsigned)pr[r]; }
      }
    }
    __syncthreads();
    const int ntask = ((M + 31) >> 5) << lN;            // a warp takes 32 candidates of one layer
    // sums
#pragma unroll 1
    for (int t0 = warp; t0 < ntask; t0 += 4 * nwarps) {
      int v[4], at[4], k[4], slot[4];                   // slot: within all layers' tables
      unsigned p[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int t = t0 + r * nwarps, l = t & (nN - 1), m = ((t >> lN) << 5) + lane;
        const bool in = t < ntask && l < nl && m < M;
        at[r] = in ? l * stride + m : -1;
        v[r] = in ? (int)rows_t[at[r]] : -1;
        p[r] = in ? rows_p[at[r]] : 0u;
        slot[r] = (in ? l * cap : 0) + (int)(((unsigned)v[r] * 2654435761u) >> shift);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) k[r] = *(volatile int*)&keys[slot[r]];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (k[r] == -1 && v[r] >= 0) k[r] = atomicCAS(&keys[slot[r]], -1, v[r]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
#pragma unroll 1
        while (v[r] >= 0 && k[r] != -1 && k[r] != v[r]) {                // ends: more slots than candidates
          slot[r] = (slot[r] & ~mask) | ((slot[r] + 1) & mask);
          k[r] = atomicCAS(&keys[slot[r]], -1, v[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (v[r] >= 0) {
          atomicAdd(&sum_lo[slot[r]], p[r] & 0xffffu);
          atomicAdd(&sum_hi[slot[r]], p[r] >> 16);
          if (!PACKED) atomicAdd(&cnt[slot[r]], 1u);
        }
        if (at[r] >= 0) rows_h[at[r]] = (unsigned)slot[r];
      }
    }
    __syncthreads();
    // keys
#pragma unroll 1
    for (int t0 = warp; t0 < ntask; t0 += 4 * nwarps) {
      int at[4], v[4], sl[4];
      u64 key[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int t = t0 + r * nwarps, l = t & (nN - 1), m = ((t >> lN) << 5) + lane;
        const bool in = t < ntask && l < nl && m < M;
        at[r] = in ? l * stride + m : -1;
        v[r] = in ? (int)rows_t[at[r]] : -1;
        sl[r] = in ? (int)rows_h[at[r]] : 0;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const u64 S = ((u64)sum_hi[sl[r]] << 16) + sum_lo[sl[r]];
        key[r] = PACKED ? S << tok_bits | (~(unsigned)v[r] & tok_mask) : (u64)__double_as_longlong(eq5_weight(s.alpha, S, cnt[sl[r]]));
        if (v[r] < 0) key[r] = 0ull;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (at[r] >= 0) { rows_h[at[r]] = (unsigned)(key[r] >> 32); rows_l[at[r]] = (unsigned)key[r]; }
    }
    __syncthreads();
    // walk
    if (tid < width) {
      unsigned u[4], t[4], h[4], lw[4], p[4];           // tokens of the layer before, of this one, key words, probabilities
      // candidates m0 + r * width at layer l; behind the last one: has ended
      auto fetch = [&](int l, int m0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int m = m0 + r * width, at = l * stride + min(m, M - 1);
          const bool in = m < M;
          t[r] = rows_t[at]; h[r] = rows_h[at]; p[r] = rows_p[at];
          lw[r] = PACKED ? 0u : rows_l[at];
          if (!in) { t[r] = PACKED ? 0u : ~0u; h[r] = 0u; }
        }
      };
      auto fetch_before = [&](int l, int m0) {          // (row_prev lies in front of the rows)
#pragma unroll
        for (int r = 0; r < 4; ++r) u[r] = rows_t[l * stride + min(m0 + r * width, M - 1) - stride];
      };
      const bool one = M <= 4 * width;                  // a thread's candidates fit its registers
      fetch(0, tid);
      if (d0 > 1) fetch_before(0, tid);
#pragma unroll 1
      for (int l = 0; l < nl; ++l) {
        const int d = d0 + l;
        const bool first = d == 1;                      // every first token follows the root
        const unsigned from = code_of(cur);
        u64 best = 0ull;
        int tok = INT_MAX;                              // not packed: smallest token of that weight
        auto consider = [&]() {
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const bool on = first || (u[r] & tok_mask) == from;
            if (PACKED) {
              best = max64(best, on ? (u64)h[r] << 32 | t[r] : 0ull);
            } else {
              const u64 key = (u64)h[r] << 32 | lw[r];
              const bool better = on && (int)t[r] >= 0 && (tok == INT_MAX || key > best || (key == best && (int)t[r] < tok));
              best = better ? key : best; tok = better ? (int)t[r] : tok;
            }
          }
        };
        consider();
        if (!one) {
#pragma unroll 1
          for (int m0 = tid + 4 * width; m0 - tid < M; m0 += 4 * width) {
            fetch(l, m0);
            if (!first) fetch_before(l, m0);
            consider();
          }
        }
        if (PACKED) {
          best = warp_max64(best);
        } else {
          const u64 mine = tok == INT_MAX ? 0ull : best;
          best = warp_max64(mine);
          tok = (int)__reduce_min_sync(FULL, tok != INT_MAX && mine == best ? (unsigned)tok : (unsigned)INT_MAX);
        }
        if (walkers > 1) {
          if (lane == 0) { sh_best[l & 1][warp] = best; sh_tok[l & 1][warp] = tok; }
          asm volatile("bar.sync 1, %0;" ::"r"(width) : "memory");
          const u64 b = lane < walkers ? sh_best[l & 1][lane] : 0ull;
          const int bt = lane < walkers ? sh_tok[l & 1][lane] : INT_MAX;
          best = warp_max64(PACKED || bt != INT_MAX ? b : 0ull);
          if (!PACKED) tok = (int)__reduce_min_sync(FULL, bt != INT_MAX && b == best ? (unsigned)bt : (unsigned)INT_MAX);
        }
        if (PACKED ? best == 0ull : tok == INT_MAX) { cur = -1; break; }   // no successor: the draft ends here
        if (PACKED) tok = (int)(~(unsigned)best & tok_mask);
        // weight of the edge taken
        const unsigned want = code_of(tok);
        unsigned e0 = 0u, e1 = 0u, e2 = 0u;
        auto weigh = [&]() {
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const bool on = (t[r] & tok_mask) == want && (first || (u[r] & tok_mask) == from);
            e0 += on ? p[r] & 0xffffu : 0u; e1 += on ? p[r] >> 16 : 0u; e2 += on;
          }
        };
        if (one) {
          weigh();
#pragma unroll
          for (int r = 0; r < 4; ++r) u[r] = t[r];
        } else {
#pragma unroll 1
          for (int m0 = tid; m0 - tid < M; m0 += 4 * width) {
            fetch(l, m0);
            if (!first) fetch_before(l, m0);
            weigh();
          }
        }
        if (l + 1 < nl) {
          fetch(l + 1, tid);                            // in flight during the sums below
          if (!one) fetch_before(l + 1, tid);
        }
        e0 = __reduce_add_sync(FULL, e0); e1 = __reduce_add_sync(FULL, e1); e2 = __reduce_add_sync(FULL, e2);
        if (walkers > 1) {
          if (lane < 3 && e2 != 0u) atomicAdd(&sh_e[d - 1][lane], lane == 0 ? e0 : lane == 1 ? e1 : e2);
        }
        if (lane == d - 1) { my_tok = tok; my_key = best; my_e0 = e0; my_e1 = e1; my_e2 = e2; }
        cur = tok; emitted = d;
      }
      if (tid == 0) sh_cur = cur;
    }
    if (d0 + nl <= D) {
      __syncthreads();
      cur = sh_cur;
      if (cur < 0) break;                               // (the same for everybody)
      for (int m = tid; m < M; m += blockDim.x) row_prev[m] = rows_t[(nl - 1) * stride + m];
      __syncthreads();
    }
  }
  if (walkers > 1) __syncthreads();                     // the edge sums are complete
  if (warp == 0) {
    if (lane < D) {
      if (walkers > 1) { my_e0 = sh_e[lane][0]; my_e1 = sh_e[lane][1]; my_e2 = sh_e[lane][2]; }
      const size_t at = (size_t)i * D + lane;
      const bool on = my_tok >= 0;
      draft_tok[at] = my_tok;
      if (draft_score)
        draft_score[at] = !on ? 0.0f : PACKED ? (float)eq5_weight(1.0, my_key >> tok_bits, 0u) : (float)__longlong_as_double((long long)my_key);
      if (draft_edge_w) draft_edge_w[at] = on ? (float)eq5_weight(PACKED ? 1.0 : s.alpha, ((u64)my_e1 << 16) + my_e0, my_e2) : 0.0f;
    }
    if (lane == 0) draft_len[i] = emitted;
  }
}

// ---- best path instead of the greedy walk (search mode 2) ------------------------------------------
// best(d, v) = w(d, v) + max over the successors v' of v of best(d + 1, v')  (0 for no successor), w the
// node's Eq. 5 in-weight; the draft follows, from the root, the successor with the largest best(), ties
// to the smaller token.  All D layers' node tables stay in shared memory at once; the layers are
// taken from the last to the first for best(), then every node's choice of successor is made for
// all layers together, and the walk is D look-ups.
constexpr int kPathWords = 9;     // per slot: best (2), largest successor best (2), key, sum lo16 / hi, count, chosen successor

struct PathTables {
  u64* best; u64* succ; int* key; unsigned* Slo; unsigned* Shi; unsigned* cnt; int* next;
};
__device__ __forceinline__ PathTables path_tables(int* pool, int cap, int l) {
  int* b = pool + (size_t)l * kPathWords * cap;
  PathTables t;
  t.best = reinterpret_cast<u64*>(b); t.succ = reinterpret_cast<u64*>(b + 2 * cap);
  t.key = b + 4 * cap; t.Slo = reinterpret_cast<unsigned*>(b + 5 * cap); t.Shi = reinterpret_cast<unsigned*>(b + 6 * cap);
  t.cnt = reinterpret_cast<unsigned*>(b + 7 * cap); t.next = b + 8 * cap;
  return t;
}
// Do the tables of all D layers fit beside the staged followers?
__device__ __forceinline__ bool best_path_fits(int M, int D, int* cap_out) {
  int cap = 64;
  while (cap <= M) cap *= 2;
  *cap_out = cap;
  return (long long)((2 * M * D + 1) & ~1) + (long long)D * kPathWords * cap <= kPoolWords;
}

__device__ void dag_best_path(const Dev& s, const Smem& sm, int i, int M, int cap, const int32_t* mlist,
                              const int32_t* plen, int poff, int32_t* draft_tok, int32_t* draft_len,
                              float* draft_score, float* draft_edge_w) {
  __shared__ int sh_draft[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_eSlo[SDMS_MAX_DRAFT], sh_eShi[SDMS_MAX_DRAFT], sh_ec[SDMS_MAX_DRAFT];
  __shared__ u64 sh_root_succ;
  __shared__ int sh_root_next, sh_emitted;
  const int tid = threadIdx.x, D = s.D;
  const int lcap = 31 - __clz(cap), shift = 32 - lcap;
  int* st_tok = sm.st_tok;                         // [m * D + d - 1], -1 past the end of the path
  int* st_pq = sm.st_tok + M * D;
  int* pool = sm.st_tok + ((2 * M * D + 1) & ~1);
  int lD = 0;
  while ((1 << lD) < D) ++lD;                      // items are numbered m << lD | d - 1

  for (int x = tid; x < (M << lD); x += blockDim.x) {
    const int m = x >> lD, dd = (x & ((1 << lD) - 1)) + 1;
    if (dd > D) continue;
    const int gpos = mlist[m];
    const int j = path_of(s, gpos);
    const bool on = gpos - j * s.L + dd <= plen[j - poff] - 1;
    st_tok[m * D + dd - 1] = on ? ldm(s.tok + gpos + dd) : -1;
    st_pq[m * D + dd - 1] = on ? ldm(s.pq + gpos + dd) : 0;
  }
  for (int x = tid; x < D * kPathWords * cap; x += blockDim.x) {
    const int w = (x >> lcap) % kPathWords;
    pool[x] = w == 4 ? -1 : (w == 8 ? INT_MAX : 0);
  }
  if (tid < D) { sh_eSlo[tid] = 0; sh_eShi[tid] = 0; sh_ec[tid] = 0; }
  if (tid == 0) { sh_root_succ = 0; sh_root_next = INT_MAX; sh_emitted = 0; }
  __syncthreads();
  // node sums of every layer
  for (int x = tid; x < (M << lD); x += blockDim.x) {
    const int m = x >> lD, l = x & ((1 << lD) - 1);
    if (l >= D) continue;
    const int v = st_tok[m * D + l];
    if (v < 0) continue;
    const PathTables t = path_tables(pool, cap, l);
    const int sl = table_slot<true>(t.key, cap, shift, v);
    add_split(&t.Slo[sl], &t.Shi[sl], &t.cnt[sl], (unsigned)st_pq[m * D + l]);
  }
  __syncthreads();
  // best(), last layer first: a candidate hands the best() of its next node to its node of this layer
  for (int d = D; d >= 1; --d) {
    const PathTables t = path_tables(pool, cap, d - 1);
    if (d < D) {
      const PathTables tn = path_tables(pool, cap, d);
      for (int m = tid; m < M; m += blockDim.x) {
        const int v = st_tok[m * D + d - 1], vn = st_tok[m * D + d];
        if (v < 0 || vn < 0) continue;
        atomicMax(&t.succ[table_slot<false>(t.key, cap, shift, v)], tn.best[table_slot<false>(tn.key, cap, shift, vn)]);
      }
      __syncthreads();
    }
    for (int x = tid; x < cap; x += blockDim.x)     // sums are only added to once per key: every slot on its own
      if (t.key[x] >= 0) {
        const double w = eq5_weight(s.alpha, ((u64)t.Shi[x] << 16) + t.Slo[x], t.cnt[x]);
        t.best[x] = (u64)__double_as_longlong(__dadd_rn(w, __longlong_as_double((long long)t.succ[x])));
      }
    __syncthreads();
  }
  // the root's best successor value (every first-layer node follows the root), then every node's
  // choice: the smallest successor token whose best() is the largest
  {
    const PathTables t = path_tables(pool, cap, 0);
    for (int x = tid; x < cap; x += blockDim.x)
      if (t.key[x] >= 0) atomicMax(&sh_root_succ, t.best[x]);
  }
  __syncthreads();
  for (int x = tid; x < (M << lD); x += blockDim.x) {
    const int m = x >> lD, l = x & ((1 << lD) - 1);
    if (l >= D) continue;
    const int v = st_tok[m * D + l];
    if (v < 0) continue;
    const PathTables t = path_tables(pool, cap, l);
    const u64 b = t.best[table_slot<false>(t.key, cap, shift, v)];
    if (l == 0) {
      if (b == sh_root_succ) atomicMin(&sh_root_next, v);
    } else {
      const PathTables tp = path_tables(pool, cap, l - 1);
      const int ps = table_slot<false>(tp.key, cap, shift, st_tok[m * D + l - 1]);
      if (b == tp.succ[ps]) atomicMin(&tp.next[ps], v);
    }
  }
  __syncthreads();
  if (tid == 0) {
    int next = sh_root_next, emitted = 0;
    for (int d = 1; d <= D && next != INT_MAX; ++d) {
      const PathTables t = path_tables(pool, cap, d - 1);
      const int sl = table_slot<false>(t.key, cap, shift, next);
      draft_tok[(size_t)i * D + d - 1] = next;
      if (draft_score)
        draft_score[(size_t)i * D + d - 1] = (float)eq5_weight(s.alpha, ((u64)t.Shi[sl] << 16) + t.Slo[sl], t.cnt[sl]);
      sh_draft[d - 1] = next;
      ++emitted;
      next = t.next[sl];
    }
    sh_emitted = emitted;
  }
  __syncthreads();
  // weight of the edges the draft took (Eq. 5 over the candidates that contain the edge)
  const int emitted = sh_emitted;
  for (int x = tid; x < (M << lD); x += blockDim.x) {
    const int m = x >> lD, d = (x & ((1 << lD) - 1)) + 1, at = m * D + d - 1;
    if (d > emitted || st_tok[at] != sh_draft[d - 1] || (d > 1 && st_tok[at - 1] != sh_draft[d - 2])) continue;
    add_split(&sh_eSlo[d - 1], &sh_eShi[d - 1], &sh_ec[d - 1], (unsigned)st_pq[at]);
  }
  __syncthreads();
  if (tid < emitted && draft_edge_w)
    draft_edge_w[(size_t)i * D + tid] =
        (float)eq5_weight(s.alpha, ((u64)sh_eShi[tid] << 16) + sh_eSlo[tid], sh_ec[tid]);
  if (tid == 0) draft_len[i] = emitted;
}

// Optional cap on the pool: of the matches of the query in one source path only the R with the largest end
// positions stay.  `list` holds the query's M matches (global memory, any order) and is compacted in
// place; the new count is returned (the same in every thread).  scratch: kStageWords * 2 shared words.
// Paths with at most R matches keep them all; for each of the others the R-th largest end position is
// found digit by digit, most significant first: one counting sweep over the list per digit fills a
// histogram of the digit for every such path (over the matches that agree with the digits found so
// far), and the path reads off which digit value its R-th largest position has.  No order among the
// matches is needed.
__device__ int cap_matches(const Dev& s, int g, int M, int32_t* list, int* scratch) {
  __shared__ int sh_warp_tot[kMaxWarps];
  __shared__ int sh_out;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int N = s.N, R = s.R, poff = g * N;
  // digits of `bits` bits: as wide as the histograms of N paths fit beside three words per path
  int bits = 5;
  while (bits > 1 && 3 * N + (N << bits) > 2 * kStageWords) --bits;
  int* cnt = scratch; int* lo = scratch + N; int* need = scratch + 2 * N; int* hist = scratch + 3 * N;   // hist[n << bits | digit]
  for (int n = tid; n < N; n += blockDim.x) { cnt[n] = 0; lo[n] = 0; need[n] = R; }
  __syncthreads();
  for (int m = tid; m < M; m += blockDim.x) atomicAdd(&cnt[path_of(s, list[m]) - poff], 1);
  __syncthreads();
  int over = 0;
  for (int n = tid; n < N; n += blockDim.x) over |= cnt[n] > R;
  if (!__syncthreads_or(over)) return M;
  int top = 0;
  while ((1 << top) < s.L) ++top;                     // positions have `top` bits
  // per path: the R-th largest position lies in [lo, lo + 2^shift) and is the need-th largest in there
  for (int shift = top; shift > 0;) {
    const int width = min(bits, shift);
    shift -= width;
    for (int x = tid; x < (N << bits); x += blockDim.x) hist[x] = 0;
    __syncthreads();
    for (int m = tid; m < M; m += blockDim.x) {
      const int gpos = list[m];
      const int j = path_of(s, gpos), n = j - poff;
      if (cnt[n] <= R) continue;
      const int rel = gpos - j * s.L - lo[n];
      if (rel >= 0 && (rel >> (shift + width)) == 0) atomicAdd(&hist[(n << bits) | (rel >> shift)], 1);
    }
    __syncthreads();
    for (int n = tid; n < N; n += blockDim.x)
      if (cnt[n] > R) {
        int left = need[n], digit = (1 << width) - 1;
        while (digit > 0 && hist[(n << bits) | digit] < left) { left -= hist[(n << bits) | digit]; --digit; }
        lo[n] += digit << shift; need[n] = left;
      }
    __syncthreads();
  }
  // keep what ends at or after the path's threshold; a chunk is read whole before any of it is written,
  // and what is written lands at or before the places already read
  if (tid == 0) sh_out = 0;
  __syncthreads();
  for (int base = 0; base < M; base += blockDim.x) {
    const int m = base + tid;
    int gpos = 0;
    bool keep = false;
    if (m < M) {
      gpos = list[m];
      const int j = path_of(s, gpos), n = j - poff;
      keep = cnt[n] <= R || gpos - j * s.L >= lo[n];
    }
    const unsigned b = __ballot_sync(FULL, keep);
    if (lane == 0) sh_warp_tot[warp] = __popc(b);
    __syncthreads();
    int before = sh_out;
    for (int w = 0; w < warp; ++w) before += sh_warp_tot[w];
    if (keep) list[before + __popc(b & ((1u << lane) - 1u))] = gpos;
    __syncthreads();
    if (tid == 0) { int t = sh_out; for (int w = 0; w < nwarps; ++w) t += sh_warp_tot[w]; sh_out = t; }
    __syncthreads();
  }
  return sh_out;
}

// Gather + DAG + search for query path i over its M (> 0) matches in mlist
// (shared or global memory).  Called by all threads of the CTA, after a barrier
// that follows write_defaults.
template <bool EXPORT>
__device__ __forceinline__ void dag_phase(const Dev& s, const Smem& sm, int i, int M, const int32_t* mlist,
                                          const int32_t* plen, int poff, int root, int32_t* draft_tok,
                                          int32_t* draft_len, float* draft_score, float* draft_edge_w) {
  // plen[j - poff] = length of path j (the prompt's lengths in shared memory, or the global array)
  if (!EXPORT && s.mode == 2) {
    int cap;
    if (best_path_fits(M, s.D, &cap)) {
      dag_best_path(s, sm, i, M, cap, mlist, plen, poff, draft_tok, draft_len, draft_score, draft_edge_w);
      return;
    }
    // too many matches for tables in shared memory: the path gets the greedy draft for now and is listed; the
    // launch that follows a best-path build (beams.cu) searches the listed paths, if need be over node tables in the
    // workspace's table area, and replaces their drafts.  Without a table area the greedy draft stays, and says so.
    if (s.beam_stride > 0) {
      if (threadIdx.x == 0) {
        const unsigned long long at = atomicAdd(&s.b_ctl[kBeamTodo], 1ull);
        if (at < (unsigned long long)s.P) s.bp_todo[at] = i;           // (a count left by a launch that failed)
      }
    } else if (threadIdx.x == 0) {
      atomicOr(s.status, SDMS_STATUS_SEARCH_FALLBACK);
    }
  }
  if (!EXPORT && s.pool == 0 && s.mode != 1) {
    if (M <= 32) {
      dag_walk_warp(s, i, M, mlist, plen, poff, draft_tok, draft_len, draft_score, draft_edge_w);
      return;
    }
    const WalkPlan w = walk_plan(s, M, sm.pool_words);
    if (w.layers > 0) {
      if (w.packed) dag_walk<true>(s, w, i, M, mlist, plen, poff, root, draft_tok, draft_len, draft_score, draft_edge_w);
      else dag_walk<false>(s, w, i, M, mlist, plen, poff, root, draft_tok, draft_len, draft_score, draft_edge_w);
      return;
    }
  }
  if (!EXPORT && s.pool == 2) list_pool(s, i, M, mlist, plen, poff, draft_tok, draft_len, draft_score, draft_edge_w);
  else if (M <= 32) dag_small<EXPORT>(s, sm, i, M, mlist, plen, poff, root, draft_tok, draft_len, draft_score, draft_edge_w);
  else if (!EXPORT && s.pool == 0 && s.mode == 1 && M * s.D <= kStageWords && layers_in_round_ok(M, s.D))
    dag_layers(s, sm, i, M, mlist, plen, poff, draft_tok, draft_len, draft_score, draft_edge_w);
  else dag_block<EXPORT>(s, sm, i, M, mlist, plen, poff, root, draft_tok, draft_len, draft_score, draft_edge_w);
}

// Matches above which a query of a large prompt goes to the wide pass (there 17-22 us in a launch that other queries need anyway;
// 1000 here 60 us).  64 here are 20 us, 32 are 10: the length of the launch where all its CTAs run at once (256 x 8192 tokens:
// 1487 us per session from 64, 1461 from 32; 96 x 3001 with tolerance 1: 585, 570), but out of the way of longer ones where they
// take turns (16 prompts of 128 x 4096: 3251, 3322).
__device__ __forceinline__ int wide_from(const Dev& s) { return (int)gridDim.x <= 2 * s.w_grid ? 32 : 64; }

template <bool EXPORT>
__global__ void __launch_bounds__(kDagThreads, EXPORT ? 1 : 2) dag_kernel(Dev s, int32_t* __restrict__ draft_tok,
                                                          int32_t* __restrict__ draft_len,
                                                          float* __restrict__ draft_score,
                                                          float* __restrict__ draft_edge_w, int round, int k,
                                                          int32_t* __restrict__ used_k) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Smem sm = carve<EXPORT>(smem_raw);
  __shared__ int32_t sh_len[SDMS_MAX_PATHS_PER_GROUP];
  const int i = blockIdx.x;
  // in a build the path lengths are older than the kernels this one follows (probe, scan: their CTAs let it start only
  // after their own wait): fetched while those drain.  The export follows any call, a step that still commits included
  if (EXPORT) grid_wait();
  for (int n = threadIdx.x; n < s.N; n += blockDim.x) sh_len[n] = ldm(s.len + (i / s.N) * s.N + n);
  const int32_t root = ldm(s.rec + (size_t)i * kRecWords + 1);
  if (!EXPORT) grid_wait();
  grid_release();
  // what probe and scan left for this path, in one round trip
  const int32_t q_mode = s.q_mode[i];
  const int q_found = min(s.q_cursor[i], s.q_reserved[i]), q_off = s.q_off[i];
  if (i == 0) {                                       // probe and scan are done with these: the next build finds them at zero
    for (int x = threadIdx.x; x < s.G; x += blockDim.x) s.g_nscan[x] = 0;
    // (the slices of a back-off build's earlier rounds stay where they are until its last round)
    if (threadIdx.x == 0 && (!(round & kRoundBackoff) || (round & kRoundLast))) *s.match_cursor = 0ull;
  }
  if ((round & kRoundNotFirst) && q_mode == Q_DONE) return;     // drafted in an earlier round, from a longer suffix
  write_defaults<EXPORT>(s, i, draft_tok, draft_score, draft_edge_w);
  const int M = q_mode == Q_NONE ? 0 : q_found;
  if (M == 0) {
    if (threadIdx.x == 0) { draft_len[i] = 0; if (used_k) used_k[i] = 0; }
    return;
  }
  const int g = i / s.N;
  __syncthreads();
  // (after the barrier: a warp that came to its own look at q_mode later would take the path for an earlier round's)
  if ((round & kRoundBackoff) && threadIdx.x == 0) { s.q_mode[i] = Q_DONE; if (used_k) used_k[i] = k; }
  int32_t* const mlist = s.matches + q_off;
  int Mk = M;
  if (s.R > 0) {                                    // (a second pass over the same build finds nothing left to cut)
    Mk = cap_matches(s, g, M, mlist, sm.st_tok);
    if (threadIdx.x == 0) s.q_cursor[i] = Mk;
    __syncthreads();
  }
  // many matches: all SMs share the work (the pass that follows this kernel)
  if (!EXPORT && s.pool == 0 && s.mode != 2 && Mk > wide_from(s) && wide_register(s, i, Mk)) return;
  dag_phase<EXPORT>(s, sm, i, Mk, mlist, sh_len, g * s.N, root, draft_tok, draft_len, draft_score, draft_edge_w);
}

// Whole draft construction of one query path in one CTA, for prompts whose
// histories are small enough that every CTA can afford to read them itself:
// probe the index; a k-gram with at most kInlineSlots occurrences is answered
// from its bucket, any other by streaming the other paths of the prompt with
// 128-bit loads (last token first, the rest of the window on a hit); then the
// gather / DAG / search phase runs on the matches just found.  The matches also
// go to the path's private slice of the match list for inspection.
// Do the first k - 2 tokens of the window that ends at `at` equal the query's?  (The last two have been
// compared by the caller.)
__device__ __forceinline__ bool window_head_equal(const int32_t* at, int k, const int32_t* q) {
  for (int t = 0; t < k - 2; ++t)
    if (ldm(at - (k - 1) + t) != q[t]) return false;
  return true;
}

// All positions of the other paths of prompt g that match the query q[0 .. k) of its path `own`: emit(position).  The
// prompt's rows lie one behind the other, so any row length is read in 16-byte chunks, eight of a thread's in flight.  A
// position is looked at more closely only if its own token and the one before it allow it (the neighbouring lane or the
// same chunk has that token).  FUZZY (one edit): the token at the end or the one before it is one of the query's last two.
template <bool FUZZY, class Emit>
__device__ __forceinline__ void scan_prompt(const Dev& s, int g, int own, int k, const int32_t* q, const int32_t* plen, Emit emit) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int row0 = g * s.N, lo = row0 * s.L, hi = lo + s.N * s.L, a0 = lo & ~3, total = (hi - a0 + 3) >> 2;
  const int4* const t4 = reinterpret_cast<const int4*>(s.tok) + (a0 >> 2);
  const int last = q[k - 1], before_last = k >= 2 ? q[k - 2] : -1;
  constexpr int kBatch = 8;
#pragma unroll 1
  for (int base = 0; base < total; base += kBatch * (int)blockDim.x) {       // same trip count for every thread
    int4 w[kBatch];
    int left0[kBatch];
#pragma unroll
    for (int r = 0; r < kBatch; ++r) {
      const int x = base + r * (int)blockDim.x + tid, at = a0 + 4 * x;
      w[r] = make_int4(-1, -1, -1, -1); left0[r] = -1;
      if (x >= total) continue;
      const int j = path_of(s, at), e = at - j * s.L, jn = j - row0;
      // nothing of the chunk's first row can match (its end, the query's own path), and no other row begins in it
      const bool dead = jn < 0 || jn == own || e > plen[jn] - 2;
      if (dead && e + 3 < s.L) continue;
      w[r] = ldm(t4 + x);
      if (lane == 0 && at > lo && k >= 2) left0[r] = ldm(s.tok + at - 1);
    }
    unsigned cand = 0;                                                       // bit 4 r + u: position u of chunk r is a candidate
#pragma unroll
    for (int r = 0; r < kBatch; ++r) {
      int left = __shfl_up_sync(FULL, w[r].w, 1);
      if (lane == 0) left = left0[r];
      const int v[5] = {left, w[r].x, w[r].y, w[r].z, w[r].w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool ok = FUZZY ? k < 2 || v[u + 1] == last || v[u + 1] == before_last || v[u] == last || v[u] == before_last
                              : v[u + 1] == last && (k < 2 || v[u] == before_last);
        cand |= (unsigned)ok << (4 * r + u);
      }
    }
    // one copy of the code that looks closer, run once per candidate
    while (cand) {
      const int bit = __ffs(cand) - 1;
      cand &= cand - 1;
      const int at = a0 + 4 * (base + (bit >> 2) * (int)blockDim.x + tid) + (bit & 3);
      const int j = path_of(s, at), e = at - j * s.L, jn = j - row0;
      if (jn < 0 || jn >= s.N || jn == own || e > plen[jn] - 2) continue;
      if (FUZZY) {
        if (k >= 2 && !one_edit_end(s.tok + at, e, q, k)) continue;
      } else {
        if (e < k - 1) continue;
        if (k >= 3 && !window_head_equal(s.tok + at, k, q)) continue;
      }
      emit(at);
    }
  }
}

// ---- a thread-block cluster shares the scan of its prompt ------------------------------------------
// In the single-launch build every query that its index bucket cannot answer streams the other paths
// of the prompt; with many such queries the same histories cross the chip once per query.  When the
// CTAs of a launch form clusters (paths [c * csize, (c + 1) * csize) of a prompt), each CTA instead
// scans 1 / csize of the prompt's tokens for ALL scan queries of its cluster and appends what it finds
// to the owning path's match slice (a cursor in global memory).  Queries are exchanged through
// distributed shared memory; two cluster barriers frame the scan.
constexpr int kShareMinTokens = 32768;   // below this a CTA reads its prompt faster than it talks to its cluster
constexpr int kPubWords = SDMS_MAX_K + 2;

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// word `w` of the array `local` (shared memory) as CTA `rank` of the cluster holds it
__device__ __forceinline__ int32_t ld_cluster(const int32_t* local, unsigned rank) {
  const uint32_t mine = (uint32_t)__cvta_generic_to_shared(local);
  uint32_t theirs;
  int32_t v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(theirs) : "r"(mine), "r"(rank));
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(theirs) : "memory");
  return v;
}

// This CTA's share of the prompt's tokens against the nq scan queries of the cluster.  cq[q] holds
// {path index of the query, unused, k tokens}.  16-byte chunks as in the single-CTA scan: a position
// passes on to the full comparison only if its own token and the one before it fit.
__device__ void shared_scan(const Dev& s, int g, int k, int nq, const int32_t (*cq)[kPubWords], const int32_t* sh_len,
                            unsigned crank, int csize) {
  const int tid = threadIdx.x;
  const int32_t* gtok = s.tok + (size_t)g * s.N * s.L;
  const int pos0 = g * s.N * s.L, slice = s.N * s.L;
  const int total = s.N * (s.L >> 2);
  const int4* g4 = reinterpret_cast<const int4*>(gtok);
  const int lo = (int)((long long)total * crank / csize), hi = (int)((long long)total * (crank + 1) / csize);
  constexpr int kBatch = 8;
  for (int base = lo; base < hi; base += kBatch * blockDim.x) {           // same trip count for every thread
    int4 w[kBatch];
    int e0[kBatch], e_hi[kBatch], jn[kBatch];
#pragma unroll
    for (int r = 0; r < kBatch; ++r) {
      const int x = base + r * blockDim.x + tid;
      jn[r] = x < hi ? path_of(s, 4 * x) : -1;
      e0[r] = jn[r] >= 0 ? 4 * x - jn[r] * s.L : 0;
      e_hi[r] = jn[r] >= 0 ? sh_len[jn[r]] - 2 : -1;
      w[r] = make_int4(-1, -1, -1, -1);
      if (e0[r] <= e_hi[r]) w[r] = ldm(g4 + x);
    }
    int left[kBatch];
#pragma unroll
    for (int r = 0; r < kBatch; ++r) left[r] = __shfl_up_sync(FULL, w[r].w, 1);   // last token of the chunk before this one
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
      const int i = cq[q][0], own = i - g * s.N;
      const int last = cq[q][2 + k - 1], before_last = k >= 2 ? cq[q][2 + k - 2] : -1;
      unsigned cand = 0;                                              // bit 4 r + u: position u of chunk r is a candidate
#pragma unroll
      for (int r = 0; r < kBatch; ++r) {
        const int v[5] = {left[r], w[r].x, w[r].y, w[r].z, w[r].w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool ok = v[u + 1] == last && jn[r] != own && e0[r] + u >= k - 1 && e0[r] + u <= e_hi[r] &&
                          (k < 2 || v[u] == before_last || (u == 0 && (tid & 31) == 0));
          cand |= (unsigned)ok << (4 * r + u);
        }
      }
      while (cand) {
        const int bit = __ffs(cand) - 1;
        cand &= cand - 1;
        const int at = 4 * (base + (bit >> 2) * (int)blockDim.x + tid) + (bit & 3);   // position within the prompt
        if (k >= 2 && (bit & 3) == 0 && (tid & 31) == 0 && ldm(gtok + at - 1) != before_last) continue;
        if (k >= 3 && !window_head_equal(gtok + at, k, &cq[q][2])) continue;
        const int n = atomicAdd(&s.q_cursor[i], 1);
        s.matches[(size_t)i * slice + n] = pos0 + at;
      }
    }
  }
}

// ---- hand-over of heavy queries to the wide pass (hand_over_from) ----------------------------------------
// Is the pass worth its while for this build (exact matches, k = 1)?  Without it the launch waits for the walk of the heaviest query, `most` matches;
// the pass has its fixed cost and takes `sum`, those of all queries handed over, by all SMs, which is more work than walks are.  The time gained (us), fitted
// to 156 builds with and without it (1 to 36 prompts of 16 to 256 paths, 20 to 97 % full, D = 6 to 16): of those this line takes 99, none slower with
// warm caches, nine up to 10 % slower with cold ones, and misses gains of up to 13 us.  All or none: with the heavier ones handed over and the others
// walked the launch waits for those first and then for the pass (32 x 16 x 4096, 97 % full: none 165, all 155, those above 1536 matches 208).
__device__ __forceinline__ bool hand_over_pays(const Dev& s, int most, int sum) {
  if ((unsigned long long)sum * s.D * 16 > s.w_slots * sizeof(WideSlot)) return false;
  const float x = 1e-3f * (float)s.D * (float)most, y = 1e-5f * (float)s.D * (float)sum;
  return 0.4f * x + 0.023f * x * x - 3.0f * y > 10.0f;
}
// Occurrences of the last tokens of paths p0 .. p1: the most, and the sum, of those that would be handed over; for the paths that this
// warp looks at.  Every thread of the CTA.
struct Heavy { int most[kFusedThreads / 32], sum[kFusedThreads / 32], said; };
__device__ __forceinline__ void occurrences(const Dev& s, int p0, int p1, Heavy& heavy) {
  const uint32_t epoch = epoch_of(ldm(s.rec + (size_t)p0 * kRecWords + kRecEpoch));
  unsigned most = 0u, sum = 0u;
  for (int p = p0 + (int)threadIdx.x; p < p1; p += kFusedThreads) {
    const int len = ldm(s.rec + (size_t)p * kRecWords), last = ldm(s.rec + (size_t)p * kRecWords + 1);
    if (len < 1 || len >= s.L) continue;
    uint4 lo, hi;
    if (!find_bucket(s, p / s.N, 1, gram_final(gram_step(gram_init(1), last)), epoch, &lo, &hi)) continue;
    const unsigned n = s.R > 0 ? min(lo.y, (unsigned)s.R * (unsigned)(s.N - 1)) : lo.y;
    if (n <= (unsigned)kHandOverFrom || n > (unsigned)wide_alone(s)) continue;
    most = max(most, n); sum += n;
  }
  most = __reduce_max_sync(FULL, most); sum = __reduce_add_sync(FULL, sum);
  if ((threadIdx.x & 31) == 0) { heavy.most[threadIdx.x >> 5] = (int)most; heavy.sum[threadIdx.x >> 5] = (int)sum; }
}
__device__ __forceinline__ bool hand_over_pays(const Dev& s, const Heavy& heavy) {
  int most = 0, sum = 0;
  for (int w = 0; w < kFusedThreads / 32; ++w) { most = max(most, heavy.most[w]); sum += heavy.sum[w]; }
  return hand_over_pays(s, most, sum);
}

// SHARE: the code of the cluster-shared scan is compiled in (kernels for prompts below kShareMinTokens leave it
// out: after a cold start the step fetches every instruction it may run past).  WEIGH: that of the exact hand-over.
template <bool EXPORT, bool SHARE, bool CHAINED, bool WEIGH>
__device__ void build_phase(const Dev& s, const Smem& sm, int k_hi, int k_lo, int32_t* draft_tok, int32_t* draft_len,
                            float* draft_score, float* draft_edge_w, int32_t* used_k,
                            const int32_t* own_rec, int csize, int hand) {
  __shared__ int sh_M;
  __shared__ int32_t sh_pub[kPubWords];                     // this CTA's query as its cluster sees it: path, mode, tokens
  __shared__ int32_t sh_cq[kMaxClusterPaths][kPubWords];    // the scan queries of the cluster
  __shared__ int sh_nq;
  __shared__ uint32_t sh_have[SDMS_MAX_K], sh_pos[SDMS_MAX_K][kInlineSlots];   // buckets of the path's last 1, 2, .. tokens: occurrences, positions
  __shared__ int32_t sh_rec[kRecWords];
  __shared__ Heavy sh_heavy;
  __shared__ int32_t sh_q[SDMS_MAX_K];
  __shared__ int32_t sh_len[SDMS_MAX_PATHS_PER_GROUP];
  const int i = blockIdx.x, tid = threadIdx.x;
  const int g = i / s.N;
  for (int n = tid; n < s.N; n += blockDim.x) sh_len[n] = ldm(s.len + g * s.N + n);
  const int slice = s.N * s.L;
  int32_t* my_matches = s.matches + (size_t)i * slice;

  write_defaults<EXPORT>(s, i, draft_tok, draft_score, draft_edge_w);
  // The path's record: length and last tokens (newest first) in one 128-byte line (or the copy the caller already holds in
  // shared memory).  Lane n - 1 looks up the path's last n tokens: the lengths that will be asked for, and, where the lengths are
  // chained, all shorter ones.
  if (tid >= (int)blockDim.x - 32) {                        // (the last warp: the first ones fetch lengths and write defaults)
    const int lane = tid & 31;
    const int32_t word = ldm((own_rec ? own_rec : s.rec + (size_t)i * kRecWords) + lane);
    sh_rec[lane] = word;
    __syncwarp();
    const int n = lane + 1, len_i = sh_rec[0];
    uint32_t have = 0u;
    if (s.eps == 0 && len_i < s.L && n <= min(min(k_hi, s.idx_n), len_i) && (CHAINED || n >= min(k_lo, s.idx_n))) {
      uint64_t h = gram_init(n);
      for (int t = n; t >= 1; --t) h = gram_step(h, sh_rec[t]);
      uint4 lo, hi;
      if (find_bucket(s, g, n, gram_final(h), epoch_of(sh_rec[kRecEpoch]), &lo, &hi)) {
        have = lo.y;
        uint32_t* const pos = sh_pos[n - 1];
        pos[0] = lo.z; pos[1] = lo.w; pos[2] = hi.x; pos[3] = hi.y; pos[4] = hi.z; pos[5] = hi.w;
      }
    }
    if (n <= SDMS_MAX_K) sh_have[n - 1] = have;
  }
  // Launches whose CTAs all run at once look at all queries here, beside their own; the others only when one of them has found a heavy query and
  // nobody has before (32 x 16 x 4096: 8 us for 2).  A step knows only its own prompt's paths as they will be.
  const bool at_once = (int)gridDim.x <= s.w_grid;
  const int w0 = own_rec ? g * s.N : 0, w1 = own_rec ? w0 + s.N : s.P;
  if (WEIGH && hand > 0 && at_once) occurrences(s, w0, w1, sh_heavy);
  // the cluster shares its scans (same decision in every CTA of the launch)
  const bool share = SHARE && csize > 1 && k_lo == k_hi && s.eps == 0 && (s.L & 3) == 0 && slice >= kShareMinTokens;
  if (tid == 0) sh_M = 0;
  __syncthreads();
  const int len_i = sh_rec[0];
  // With k_lo < k_hi the suffix length backs off: the longest k in [k_lo, k_hi] that has a match wins.
  int k = k_hi;
  for (;; --k) {
  // the index is asked for the query's last nx tokens: all k of them unless the context keeps fewer tables
  const int nx = min(k, s.idx_n);
  int mode = Q_NONE;
  if (len_i >= k && len_i < s.L) {
    if (s.eps > 0) mode = Q_SCAN;                           // fuzzy matches are found by scanning only
    else if (sh_have[CHAINED ? 0 : nx - 1] > 0u) mode = sh_have[nx - 1] <= (uint32_t)kInlineSlots ? Q_INLINE : Q_SCAN;
  }
  if (tid < k) sh_q[tid] = sh_rec[k - tid];
  if (tid == 0) {
    s.q_mode[i] = mode; s.q_reserved[i] = mode == Q_NONE ? 0 : slice; s.q_off[i] = i * slice;
    if (share) {
      sh_pub[0] = i; sh_pub[1] = mode;
      for (int t = 0; t < k; ++t) sh_pub[2 + t] = sh_rec[k - t];
      if (mode == Q_SCAN) s.q_cursor[i] = 0;              // the cluster's scanners count this query's matches here
    }
  }
  if (mode == Q_INLINE) {
    // all occurrences of the n-gram stand in its bucket, or in that and those of the shorter ones
    const int n0 = CHAINED ? 1 : nx;
    if (tid < (nx - n0 + 1) * kInlineSlots) {
      const int n = n0 + tid / kInlineSlots, slot = tid % kInlineSlots;
      if (slot < (int)min(sh_have[n - 1], (uint32_t)kInlineSlots)) {
        const uint32_t entry = sh_pos[n - 1][slot], lpos = CHAINED ? entry & s.pos_mask : entry;
        const int jn = (int)(lpos / (uint32_t)s.L);
        const int j = g * s.N + jn;
        const int e = (int)(lpos % (uint32_t)s.L);
        if (j != i && e >= k - 1 && e <= sh_len[jn] - 2 && (!CHAINED || n == k || entry_may_follow(s, entry, sh_rec[n + 1]))) {
          const int32_t* c = s.tok + (size_t)j * s.L + (e - k + 1);
          bool same = true;
          for (int t = 0; t < k; ++t) same = same && (ldm(c + t) == sh_rec[k - t]);
          if (same) {
            const int at = atomicAdd(&sh_M, 1);
            sm.list[at] = j * s.L + e;
            my_matches[at] = j * s.L + e;
          }
        }
      }
    }
  } else if (mode == Q_SCAN && !share) {
    __syncthreads();                                        // the query's tokens
  }
  if (share) {
    cluster_sync_all();                                     // every query of the cluster is published
    const unsigned crank = cluster_rank();
    for (int x = tid; x < csize * (k + 2); x += blockDim.x) {
      const int r = x / (k + 2), w = x - r * (k + 2);
      sh_cq[r][w] = ld_cluster(&sh_pub[w], (unsigned)r);
    }
    __syncthreads();
    if (tid == 0) {                                         // keep the scan queries, in rank order
      int nq = 0;
      for (int r = 0; r < csize; ++r)
        if (sh_cq[r][1] == Q_SCAN) {
          if (nq != r) for (int w = 0; w < k + 2; ++w) sh_cq[nq][w] = sh_cq[r][w];
          ++nq;
        }
      sh_nq = nq;
    }
    __syncthreads();
    if (sh_nq > 0) shared_scan(s, g, k, sh_nq, sh_cq, sh_len, crank, csize);
    cluster_sync_all();                                     // all shares scanned; nobody reads a neighbour's memory any more
    if (mode == Q_SCAN) {
      const int M = __ldcg(s.q_cursor + i);
      for (int x = tid; x < min(M, kListCap); x += blockDim.x) sm.list[x] = __ldcg(my_matches + x);
      if (tid == 0) sh_M = M;
    }
  } else if (mode == Q_SCAN) {
    auto emit = [&](int pos) {
      const int n = atomicAdd(&sh_M, 1);
      if (n < kListCap) sm.list[n] = pos;
      my_matches[n] = pos;
    };
    if (s.eps > 0) scan_prompt<true>(s, g, i - g * s.N, k, sh_q, sh_len, emit);
    else scan_prompt<false>(s, g, i - g * s.N, k, sh_q, sh_len, emit);
  }
  __syncthreads();
  if (sh_M > 0 || k <= k_lo) break;
  __syncthreads();                                   // everybody has read sh_M before the next length adds to it
  }
  int M = sh_M;
  if (s.R > 0 && M > s.R) {                          // (uniform) the cap can only bite with more than R matches
    const int M0 = M;
    M = cap_matches(s, g, M0, my_matches, sm.st_tok);
    if (M < M0 && M <= kListCap)
      for (int x = tid; x < M; x += blockDim.x) sm.list[x] = my_matches[x];
    __syncthreads();
  }
  if (tid == 0) { s.q_cursor[i] = M; if (used_k) used_k[i] = M > 0 ? k : 0; }
  if (M == 0) {
    if (tid == 0) draft_len[i] = 0;
    return;
  }
  if (hand > 0 && M > hand && M <= wide_alone(s)) {
    bool pays = true;
    if (WEIGH) {
      volatile unsigned long long* const known = &s.w_ctl[kWideHeavy];                   // 1: it pays, 2: it does not
      if (at_once) {
        pays = hand_over_pays(s, sh_heavy);
        if (own_rec) {                                       // what one prompt has reason enough for, the others' queries go along with
          if (pays && tid == 0) *known = 1ull;
          pays = __syncthreads_or(pays || (tid == 0 && *known == 1ull));
        }
      } else {
        if (tid == 0) sh_heavy.said = (int)*known;
        __syncthreads();
        pays = sh_heavy.said == 1;
        if (sh_heavy.said == 0) {
          occurrences(s, w0, w1, sh_heavy);
          __syncthreads();
          pays = hand_over_pays(s, sh_heavy);
          if (tid == 0) *known = pays ? 1ull : 2ull;
        }
      }
    }
    const bool last = (int)blockIdx.x + s.w_grid >= (int)gridDim.x;
    if (pays && M > (last ? hand : kHandOverEarly) && wide_register(s, i, M)) return;    // all SMs share the work (the launch that follows)
  }
  dag_phase<EXPORT>(s, sm, i, M, M <= kListCap ? sm.list : my_matches, sh_len, g * s.N, sh_q[k - 1], draft_tok,
                    draft_len, draft_score, draft_edge_w);
}

template <bool EXPORT, bool SHARE, bool CHAINED, bool WEIGH>
__global__ void __launch_bounds__(kFusedThreads, 1) build_fused_kernel(Dev s, int k_hi, int k_lo, int32_t* draft_tok,
                                                                  int32_t* draft_len, float* draft_score,
                                                                  float* draft_edge_w, int32_t* used_k, int csize, int hand) {
  grid_wait();
  grid_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Smem sm = carve<EXPORT>(smem_raw);
  build_phase<EXPORT, SHARE, CHAINED, WEIGH>(s, sm, k_hi, k_lo, draft_tok, draft_len, draft_score, draft_edge_w, used_k, nullptr, csize, hand);
}

// One launch per decode step.  The CTAs of a prompt form a thread-block cluster.  Each CTA first
// checks its path's previous draft against the sampled tokens and appends what was accepted (tokens,
// probabilities, index entries); after a cluster-wide barrier with release/acquire semantics every
// path of the prompt is up to date and each CTA builds its path's next draft.  draft_tok / draft_len
// hold the previous drafts on entry and the new ones on exit.
// k_lo < k: the suffix length backs off from k to k_lo (used_k, if given, receives each path's choice).
template <bool SHARE, bool CHAINED, bool WEIGH>
__global__ void __launch_bounds__(kFusedThreads, 1) step_kernel(Dev s, int k, int k_lo, const int32_t* sampled,
                                                           const float* sampled_lp, int32_t* accept_len,
                                                           int32_t* draft_tok, int32_t* draft_len,
                                                           float* draft_score, float* draft_edge_w,
                                                           int32_t* used_k, int hand) {
  grid_wait();
  grid_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Smem sm = carve<false>(smem_raw);
  __shared__ int32_t sh_own_rec[kRecWords];
  accept_commit_phase<CHAINED>(s, blockIdx.x, draft_tok, draft_len, sampled, sampled_lp, accept_len, sh_own_rec, k, k_lo);
  // every thread of every CTA of the cluster gets here exactly once (no early exit above)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  build_phase<false, SHARE, CHAINED, WEIGH>(s, sm, k, k_lo, draft_tok, draft_len, draft_score, draft_edge_w, used_k, sh_own_rec, s.N, hand);
}

}  // namespace

// Dynamic shared memory of the single-launch kernels.  A CTA has its SM to itself (registers), so prompts with room for
// thousands of matches take more for the walk over them (dag_walk; trees, lists and layer-wise search do not walk), small prompts
// keep the cache.  (Figures of builds that hand nothing over, see hand_over_from.)  An SM splits its 256 KB at 164, 196 and 228 KB: with 200 KB 28 KB of L1 are left, with 184 (and 10 KB
// of arrays) 60.  k = 1 builds of 64 x 2048 and 32 x 16 x 4096 tokens, queries of up to 4139 matches: 117 and 193 us with 200 KB, 98 and
// 172 with 184, 124 and 206 with 106; alpha = 0.5, whose tables are a third larger, 144 and 222 / 127 and 206 / 125 and 205;
// tree pools 126 and 197 with 200 KB, 101 and 175 with 106.  What loses: with alpha = 1, pools
// of 5089 to 6112 matches, whose walk_plan only fits the 200 (64 x 2048 tokens, V = 21 and 23, at most 6035 and 5497 matches: 198 and 185 us
// for 179 and 171).  On either side 184 is the faster: at most 6304 matches (V = 20) 212 for 239, at most 4228 (V = 30) 127 for 151.
constexpr size_t kBigPool = 184 * 1024;
constexpr long long kBigPoolFrom = 32768;             // tokens of a prompt
static size_t fused_smem_bytes(const Dev& s) {
  return (long long)s.N * s.L >= kBigPoolFrom && s.pool == 0 && s.mode != 1 ? kBigPool : dag_smem_bytes<false>();
}

namespace {
// Their instances: a context runs the one that has the code it needs (after a cold start a step fetches every instruction it may
// run past: 0.15 us of 9.7 with the chained index's code in the step of an index that is not; 0.2 of 15 with that of the exact hand-over in a step
// that has none; and 32 x 16 x 4096, k = 1, where every CTA scans for itself, 127 to 148 us, with the cluster-shared scan's code 142 to 170).
// All its launches run the same one, also those that hand nothing over: a session's k = 1 builds would fetch theirs each time (64 x 2048 tokens,
// 32 steps: 9 us of 735).
bool weighs(const Dev& s) { return s.w_grid > 0 && s.eps == 0; }
template <bool WEIGH>
auto build_variant_of(bool share, bool chained) {
  return share ? (chained ? build_fused_kernel<false, true, true, WEIGH> : build_fused_kernel<false, true, false, WEIGH>)
               : (chained ? build_fused_kernel<false, false, true, WEIGH> : build_fused_kernel<false, false, false, WEIGH>);
}
template <bool WEIGH>
auto step_variant_of(bool share, bool chained) {
  return share ? (chained ? step_kernel<true, true, WEIGH> : step_kernel<true, false, WEIGH>)
               : (chained ? step_kernel<false, true, WEIGH> : step_kernel<false, false, WEIGH>);
}
auto build_variant(bool share, bool chained, bool weigh) { return weigh ? build_variant_of<true>(share, chained) : build_variant_of<false>(share, chained); }
auto step_variant(bool share, bool chained, bool weigh) { return weigh ? step_variant_of<true>(share, chained) : step_variant_of<false>(share, chained); }
}  // namespace

cudaError_t dag_kernel_setup() {
  cudaError_t e = cudaFuncSetAttribute(dag_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)dag_smem_bytes<false>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(dag_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dag_smem_bytes<true>());
  for (int v = 0; v < 8 && e == cudaSuccess; ++v) {
    const auto build = build_variant(v & 1, v & 2, v & 4);
    const auto step = step_variant(v & 1, v & 2, v & 4);
    e = cudaFuncSetAttribute(build, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBigPool);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBigPool);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(step, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  return e;
}

// Matches from which the single-launch build of suffix lengths k_lo .. k hands a query over to the wide pass; 0: it hands none over, and
// is not followed by that pass.  A CTA walks a thousand matches in 15 to 60 us (D = 8 to 16), and the launch waits for the heaviest query; the pass
// costs 2 us where there is nothing to do and 17 to 25 and more where there is.  Only the shortest suffixes have such queries: k = 1, with
// tolerance 1 also k = 2.  The kernel decides whether they are worth it (hand_over_pays).  Builds without / with that rule, and handing over in any case (us):
//   k = 1, at most 4 rounds of CTAs, from 65536 tokens per prompt: 64 x 2048, 97 % full, 87 / 52 / 52, half full 68 / 53 / 53 and 45 / 48 / 40; 16 x 4096
//     119 / 56 / 55; 8 prompts of 16 x 4096 124 / 71 / 69; 4 of 128 x 1024 446 / 231 / 229; 36 of 16 x 8000 508 / 299 / 302; 32 of 16 x 4096, 97 % full, 165 / 152 / 150,
//     half full 94 / 97 / 111, a fifth full 66 / 66 / 82; 32 of 32 x 2048 (1024 paths) 80 / - / 101: there the SMs are busy either way
//     below: 16 of 32 x 1024 65 / - / 73, 16 of 16 x 2048 47 / - / 50, 16 x 1024 16 / - / 23
//   tolerance 1, at most 2 rounds, from 16384 tokens, k = 2: 16 x 1024 44 / 35 / 35, 32 x 2048 117 / 69 / 69, 8 of 32 x 1024 105 / 85 / 85, 18 of 16 x 1024 56 / 56 / 65;
//     32 of 16 x 1024 (512 paths) 72 / - / 94; 8 x 1024 17 / - / 19.  k = 3, with 284 matches at most, 46 / - / 52
// Queries split by classes of tokens (above wide_alone() matches) stay: with tolerance 1 and k = 1 every query is one (32 x 2048: 5.8 / 6.3 ms).
int hand_over_from(const Dev& s, int k, int k_lo, cudaStream_t stream) {
  if (!s.fused || s.w_grid == 0 || k_lo != k || k > (s.eps > 0 ? 2 : 1)) return 0;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(stream, &capture);             // (a graph is there for histories that have grown since)
  const int held = s.N * (capture == cudaStreamCaptureStatusNone ? s.held : s.L);
  if (s.eps == 0) return held * s.D >= kHandOverHeld ? kHandOverFrom : 0;
  return held >= (s.P <= s.w_grid ? kHandOverHeldFuzzy : kHandOverHeldFuzzyRounds) ? kHandOverFrom : 0;
}

namespace {
void step_launch_config(const Dev& s, cudaStream_t stream, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(s.P); cfg->blockDim = dim3(kFusedThreads);
  cfg->dynamicSmemBytes = fused_smem_bytes(s); cfg->stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = s.N; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = attr; cfg->numAttrs = 2;
}
}  // namespace

// Can the prompts of this context run as clusters (one CTA per path) on this device?
bool step_kernel_fits(const Dev& s) {
  if (!s.fused || s.N > kMaxClusterPaths) return false;
  cudaLaunchConfig_t cfg; cudaLaunchAttribute attr[2];
  step_launch_config(s, 0, &cfg, attr);
  cfg.numAttrs = 1;                                   // occupancy only looks at the cluster shape
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, step_variant(true, s.epochs, false), &cfg) != cudaSuccess) { cudaGetLastError(); return false; }
  // every prompt's cluster resident at once: large clusters leave SMs of a GPC idle, and a launch whose
  // clusters queue up for the device is slower than the separate accept and build launches
  return (long long)clusters * s.N >= s.P;
}

cudaError_t launch_step(const Dev& s, int k, int k_lo, const int32_t* sampled, const float* sampled_lp,
                        int32_t* accept_len, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                        float* draft_edge_w, int32_t* used_k, int hand, cudaStream_t stream) {
  cudaLaunchConfig_t cfg; cudaLaunchAttribute attr[2];
  step_launch_config(s, stream, &cfg, attr);
  const bool share = s.eps == 0 && (s.L & 3) == 0 && (long long)s.N * s.L >= kShareMinTokens;       // the prompt is worth sharing its scan
  return cudaLaunchKernelEx(&cfg, step_variant(share, s.epochs, weighs(s)), s, k, k_lo, sampled, sampled_lp, accept_len,
                            draft_tok, draft_len, draft_score, draft_edge_w, used_k, hand);
}

cudaError_t launch_dag(const Dev& s, bool with_export, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                       float* draft_edge_w, cudaStream_t stream, int round, int k, int32_t* used_k) {
  if (with_export)
    return launch_overlapped(dag_kernel<true>, dim3(s.P), dim3(kDagThreads), dag_smem_bytes<true>(), stream, s,
                             draft_tok, draft_len, draft_score, draft_edge_w, 0, 0, (int32_t*)nullptr);
  return launch_overlapped(dag_kernel<false>, dim3(s.P), dim3(kDagThreads), dag_smem_bytes<false>(), stream, s,
                           draft_tok, draft_len, draft_score, draft_edge_w, round, k, used_k);
}

// Cluster size (CTAs = consecutive paths of one prompt) of the single-launch build, 1 for none.  A cluster
// shares the scan of its prompt (shared_scan), which shortens the longest CTA of a launch but adds two
// barriers to every CTA: it pays when the whole launch is resident at once, i.e. when the launch's
// time is its slowest CTA's, and loses when CTAs queue for SMs anyway.  Sizes above 8 leave too many
// SMs of a GPC idle.
int build_cluster_size(const Dev& s) {
  if (!s.fused || (s.L & 3) != 0 || (long long)s.N * s.L < kShareMinTokens) return 1;
  for (int c = 8; c >= 2; --c) {
    if (s.N % c) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s.P); cfg.blockDim = dim3(kFusedThreads); cfg.dynamicSmemBytes = fused_smem_bytes(s);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, build_variant(true, s.epochs, false), &cfg) != cudaSuccess) { cudaGetLastError(); continue; }
    if ((long long)clusters * c >= s.P) return c;
  }
  return 1;
}

cudaError_t launch_build_fused(const Dev& s, int k_hi, int k_lo, int32_t* draft_tok, int32_t* draft_len,
                               float* draft_score, float* draft_edge_w, int32_t* used_k, int hand, cudaStream_t stream) {
  if (s.build_cluster <= 1 || k_lo != k_hi || s.eps > 0)
    return launch_overlapped(build_variant(false, s.epochs, weighs(s)), dim3(s.P), dim3(kFusedThreads), fused_smem_bytes(s), stream,
                             s, k_hi, k_lo, draft_tok, draft_len, draft_score, draft_edge_w, used_k, 0, hand);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(s.P); cfg.blockDim = dim3(kFusedThreads);
  cfg.dynamicSmemBytes = fused_smem_bytes(s); cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = s.build_cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, build_variant(true, s.epochs, weighs(s)), s, k_hi, k_lo, draft_tok, draft_len, draft_score, draft_edge_w,
                            used_k, (int)s.build_cluster, hand);
}

}  // namespace sdms
