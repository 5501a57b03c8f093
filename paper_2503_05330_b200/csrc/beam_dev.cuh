// The B best paths of a query's pool (several drafts per path), by one CTA over node tables in global
// memory.  Value of a path: the sum of its nodes' Eq. 5 in-weights, added from its end towards its
// start (the search-mode-2 value); only paths that run on to a leaf or to layer D count.
//
// Every node keeps its B best continuations, best first:
//   leaf (d, v):  [ w(d, v) ]
//   otherwise:    the B best of { w(d, v) + x : x a kept continuation of a successor v' },
// ordered by value (larger first), then v' (smaller first), then the rank of x in the list of v'.
// The layers are taken from the last to the first.  Rank r of a layer is found by two sweeps over the
// layer's (candidate, successor) items: every item offers the best of its successor's continuations
// that still comes strictly after the node's rank r - 1 entry (64-bit max on the value's bit pattern),
// then the items that hold exactly that value compete with (~v', rank) packed in 64 bits.  Equal
// offers from different items are the same entry, so duplicates do no harm.
#pragma once
#include "wide_dev.cuh"

namespace sdms {

constexpr u64 kBeamLeaf = 1ull;          // `next` of a continuation that ends at its node
struct BeamEnt { u64 value; u64 next; };  // value: bit pattern of the double; next: ~token << 32 | (7 - rank) << 24 | slot; 0 = no entry

__device__ __forceinline__ u64 beam_next(uint32_t tok, int rank, int slot) {
  return ((u64)(~tok) << 32) | ((u64)(7 - rank) << 24) | (u64)(unsigned)slot;
}
__device__ __forceinline__ bool beam_after(u64 v, u64 nx, const BeamEnt& prev) {   // (v, nx) comes strictly after prev
  return v < prev.value || (v == prev.value && nx < prev.next);
}

// One CTA (kWideThreads threads), query path i with M matches in `list`.  Needs D << lcap table slots
// starting at `base`, all zero (they are left zero).  Writes beam_tok [B][D], beam_len [B], beam_value [B]
// of the path.  `ent` = s.b_ent + base * stride.  With score0 / edge0 (each [D], either may be NULL; the
// caller asks with want0) the first beam also gets what a draft carries: the Eq. 5 in-weight of each of
// its nodes and the weight of each edge it takes.
__device__ __forceinline__ void beams_of_query(const Dev& s, int i, int M, const int32_t* list, unsigned base, int lcap, int B,
                               int32_t* beam_tok, int32_t* beam_len, float* beam_value, bool want0 = false,
                               float* score0 = nullptr, float* edge0 = nullptr) {
  __shared__ BeamEnt sh_root[SDMS_MAX_BEAMS];
  __shared__ int sh_bslot[SDMS_MAX_DRAFT];
  __shared__ u64 sh_bedge[SDMS_MAX_DRAFT];
  __shared__ int sh_blen;
  const int tid = threadIdx.x, D = s.D, stride = s.beam_stride;
  const unsigned cap = 1u << lcap;
  WideSlot* const tab = s.w_tab + base;
  BeamEnt* const ent = s.b_ent + (size_t)base * stride;
  const int* const item = s.w_item + base;           // [(d - 1) * M + m]
  for (int m0 = 0; m0 < M; m0 += kWideChunk) wide_insert_unit(s, list, base, lcap, M, m0);
  if (tid < SDMS_MAX_BEAMS) sh_root[tid] = BeamEnt{0ull, 0ull};
  __threadfence();
  __syncthreads();

  for (int d = D; d >= 0; --d) {
    // d >= 1: the lists of the nodes of layer d from those of layer d + 1; d = 0: the root's from layer 1
    if (d < D) {
      for (int r = 0; r < B; ++r) {
        for (int stage = 0; stage < 2; ++stage) {
          for (int m = tid; m < M; m += blockDim.x) {
            const int sv = __ldcg(item + (size_t)d * M + m);                 // the candidate's node at layer d + 1
            if (sv < 0) continue;
            BeamEnt* mine;                                                 // the list this item feeds
            double w_u = 0.0;
            if (d == 0) {
              mine = sh_root;
            } else {
              const int su = __ldcg(item + (size_t)(d - 1) * M + m);
              mine = ent + ((size_t)((d - 1) << lcap) + su) * stride;
              const u64 sum = __ldcg(&tab[((size_t)(d - 1) << lcap) + su].sum);
              w_u = eq5_weight(s.alpha, sum & ((1ull << kWideSumShift) - 1), (unsigned)(sum >> kWideSumShift));
            }
            BeamEnt prev{0ull, 0ull};
            if (r > 0) {
              prev = d == 0 ? sh_root[r - 1] : BeamEnt{__ldcg(&mine[r - 1].value), __ldcg(&mine[r - 1].next)};
              if (prev.next == 0ull) continue;                             // the node ran out of continuations before
            }
            const BeamEnt* theirs = ent + ((size_t)(d << lcap) + sv) * stride;
            const uint32_t tok = __ldcg(&tab[((size_t)d << lcap) + sv].tok1) - 1u;
            for (int j = 0; j < B; ++j) {                                  // best first: the first that qualifies is the offer
              const u64 nx = __ldcg(&theirs[j].next);
              if (nx == 0ull) break;
              const double x = __longlong_as_double((long long)__ldcg(&theirs[j].value));
              const u64 val = (u64)__double_as_longlong(d == 0 ? x : __dadd_rn(w_u, x));
              const u64 key = beam_next(tok, j, sv);
              if (r > 0 && !beam_after(val, key, prev)) continue;
              if (stage == 0) atomicMax(&mine[r].value, val);
              else if ((d == 0 ? mine[r].value : __ldcg(&mine[r].value)) == val) atomicMax(&mine[r].next, key);
              break;
            }
          }
          __threadfence();
          __syncthreads();
        }
      }
    }
    if (d >= 1) {
      // a node that nothing was offered to is a leaf: its only continuation is to stop
      for (unsigned x = tid; x < cap; x += blockDim.x) {
        const size_t sl = ((size_t)(d - 1) << lcap) + x;
        if (__ldcg(&s.w_key[base + sl]) == 0u) continue;
        BeamEnt* mine = ent + sl * stride;
        if (__ldcg(&mine[0].next) != 0ull) continue;
        const u64 sum = __ldcg(&tab[sl].sum);
        mine[0].value = (u64)__double_as_longlong(eq5_weight(s.alpha, sum & ((1ull << kWideSumShift) - 1), (unsigned)(sum >> kWideSumShift)));
        mine[0].next = kBeamLeaf;
      }
      __threadfence();
      __syncthreads();
    }
  }

  // the beams: follow the entries from the root
  if (tid < B) {
    BeamEnt e = sh_root[tid];
    int len = 0;
    if (e.next != 0ull) beam_value[tid] = (float)__longlong_as_double((long long)e.value);
    else beam_value[tid] = 0.0f;
    for (int d = 1; d <= D && e.next != 0ull && e.next != kBeamLeaf; ++d) {
      const uint32_t tok = ~(uint32_t)(e.next >> 32);
      const int rank = 7 - (int)((e.next >> 24) & 7u), slot = (int)(e.next & 0xffffffu);
      beam_tok[tid * D + len++] = (int32_t)tok;
      const BeamEnt* at = ent + ((size_t)((d - 1) << lcap) + slot) * stride + rank;
      e = BeamEnt{__ldcg(&at->value), __ldcg(&at->next)};
    }
    for (int d = len; d < D; ++d) beam_tok[tid * D + d] = -1;
    beam_len[tid] = len;
  }
  if (want0) {
    // the first beam once more, slot by slot; then the probabilities of the items on its edges
    if (tid < SDMS_MAX_DRAFT) sh_bedge[tid] = 0ull;
    if (tid == 0) {
      BeamEnt e = sh_root[0];
      int len = 0;
      for (int d = 1; d <= D && e.next != 0ull && e.next != kBeamLeaf; ++d) {
        const int rank = 7 - (int)((e.next >> 24) & 7u), slot = (int)(e.next & 0xffffffu);
        sh_bslot[len++] = slot;
        if (score0) {
          const u64 sum = __ldcg(&tab[((size_t)(d - 1) << lcap) + slot].sum);
          score0[d - 1] = (float)eq5_weight(s.alpha, sum & ((1ull << kWideSumShift) - 1), (unsigned)(sum >> kWideSumShift));
        }
        const BeamEnt* at = ent + ((size_t)((d - 1) << lcap) + slot) * stride + rank;
        e = BeamEnt{__ldcg(&at->value), __ldcg(&at->next)};
      }
      sh_blen = len;
    }
    __syncthreads();
    const int len = sh_blen;
    if (edge0) {
      for (int d = 1; d <= len; ++d) {
        for (int m0 = 0; m0 < M; m0 += blockDim.x) {             // whole warps: the lanes add up together
          const int m = m0 + tid;
          bool on = false;
          if (m < M) on = __ldcg(item + (size_t)(d - 1) * M + m) == sh_bslot[d - 1] &&
                          (d == 1 || __ldcg(item + (size_t)(d - 2) * M + m) == sh_bslot[d - 2]);
          const unsigned group = __ballot_sync(FULL, on);
          if (group == 0u) continue;
          const u64 sum = group_sum(group, group, on ? (unsigned)ldm(s.pq + list[m] + d) : 0u);
          if ((tid & 31) == __ffs(group) - 1) atomicAdd(&sh_bedge[d - 1], ((u64)__popc(group) << kWideSumShift) | sum);
        }
      }
      __syncthreads();
      if (tid < len) {
        const u64 sum = sh_bedge[tid];
        edge0[tid] = (float)eq5_weight(s.alpha, sum & ((1ull << kWideSumShift) - 1), (unsigned)(sum >> kWideSumShift));
      }
    }
  }
  __syncthreads();
  // leave the tables as they were found
  uint4* z = reinterpret_cast<uint4*>(tab);
  for (size_t x = tid; x < ((size_t)D << lcap) * 2; x += blockDim.x) z[x] = make_uint4(0u, 0u, 0u, 0u);
  uint4* zk = reinterpret_cast<uint4*>(s.w_key + base);
  for (size_t x = tid; x < ((size_t)D << lcap) / 4; x += blockDim.x) zk[x] = make_uint4(0u, 0u, 0u, 0u);
  uint4* ze = reinterpret_cast<uint4*>(ent);
  for (size_t x = tid; x < ((size_t)D << lcap) * stride; x += blockDim.x) ze[x] = make_uint4(0u, 0u, 0u, 0u);
}

// The same by one CTA with the node tables in shared memory (pools up to several hundred matches), the continuation lists
// there too if they fit, else in the table area.  Layers from the last to the first.  Most nodes carry one candidate, and
// such a node's list is its successor's with its own weight added: a thread each.  A node with several candidates is worked
// out by a warp: a lane per candidate holds the best continuation that its next node has left, and every rank is an arg-max
// over the lanes.  With more candidates than lanes the B best next nodes are found first, by the heads of their lists: no
// other one can contribute.  Bound by dependent accesses; with everything in the table area (two rounds of L2 atomics and a
// barrier per layer and rank) 139 us for 30 matches, 570 us for 760, D = 8, B = 4.
// ent0: the path's lists in the table area, ent_stride entries per slot (used if !SHARED_LISTS; left zero).  want0, score0,
// edge0: as for beams_of_query.
template <bool SHARED_LISTS>
__device__ __forceinline__ void beams_in_shared(const Dev& s, const BeamPlan w, int M, const int32_t* list, int B, BeamEnt* ent0,
                                                int ent_stride, int32_t* beam_tok, int32_t* beam_len, float* beam_value,
                                                bool want0 = false, float* score0 = nullptr, float* edge0 = nullptr) {
  extern __shared__ __align__(16) unsigned char beam_smem[];
  __shared__ BeamEnt sh_root[SDMS_MAX_BEAMS];
  __shared__ int sh_n, sh_members, sh_blen, sh_bslot[SDMS_MAX_DRAFT];
  __shared__ unsigned sh_be[SDMS_MAX_DRAFT][3];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5, D = s.D;
  const int cap = w.cap, mask = cap - 1, shift = __clz(cap) + 1, stride = w.stride, all = D * cap;
  const int es = SHARED_LISTS ? B : ent_stride;
  BeamEnt* const ent = SHARED_LISTS ? reinterpret_cast<BeamEnt*>(beam_smem) : ent0;          // [layer][slot][rank]
  int* const key = reinterpret_cast<int*>(beam_smem + (SHARED_LISTS ? (size_t)all * B * 16 : 0));   // [layer][slot] token, -1: free
  unsigned* const lo = reinterpret_cast<unsigned*>(key + all);         // sums of the lower 16 bits, of the rest
  unsigned* const hi = lo + all;
  unsigned* const cw = hi + all;                                       // a candidate of the node << 16 | count
  int* const start = reinterpret_cast<int*>(cw + all);                 // [slot] of the layer at hand: where its members are listed
  unsigned short* const todo = reinterpret_cast<unsigned short*>(start + cap);           // its nodes with several candidates
  unsigned short* const member = todo + cap;                           // [stride] candidates, node by node
  unsigned short* const slot = member + stride;                        // [layer][candidate], 0xffff: has ended
  constexpr int kEnded = 0xffff;

  for (int x = tid; x < all; x += blockDim.x) { key[x] = -1; lo[x] = 0u; hi[x] = 0u; cw[x] = 0u; }
  __syncthreads();
  // candidates' followers into the tables: a warp takes 32 candidates of one layer
  const int nchunk = stride >> 5;
  for (int t = warp, l = 0, c = warp; t < D * nchunk; t += nwarps, c += nwarps) {
    while (c >= nchunk) { c -= nchunk; ++l; }
    const int m = c * 32 + lane;
    int v = -1, sl = kEnded;
    unsigned p = 0u;
    if (m < M) {
      const int gpos = list[m], j = path_of(s, gpos);
      if (l + 1 <= ldm(s.len + j) - 1 - (gpos - j * s.L)) { v = ldm(s.tok + gpos + l + 1); p = (unsigned)ldm(s.pq + gpos + l + 1); }
    }
    if (v >= 0) {
      unsigned h = ((unsigned)v * 2654435761u) >> shift;
      int k;
#pragma unroll 1
      while (true) {                                                   // ends: more slots than candidates
        k = atomicCAS(&key[l * cap + h], -1, v);
        if (k == -1 || k == v) break;
        h = (h + 1) & mask;
      }
      sl = (int)h;
      atomicAdd(&lo[l * cap + h], p & 0xffffu);
      atomicAdd(&hi[l * cap + h], p >> 16);
      atomicAdd(&cw[l * cap + h], k == -1 ? (unsigned)m << 16 | 1u : 1u);
    }
    slot[l * stride + m] = (unsigned short)sl;
  }
  __syncthreads();
  auto weight = [&](int x) { return eq5_weight(s.alpha, ((u64)hi[x] << 16) + lo[x], cw[x] & 0xffffu); };
  struct Offer { u64 val, nx; };
  // what next node sn of layer l + 1 has to offer at rank j (nothing: nx = 0)
  auto offer_of = [&](int l, int sn, int j, bool add, double w_u) {
    Offer o{0ull, 0ull};
    if (sn == kEnded || j >= B) return o;
    const BeamEnt e = ent[((size_t)(l + 1) * cap + sn) * es + j];
    if (e.next == 0ull) return o;
    o.val = add ? (u64)__double_as_longlong(__dadd_rn(w_u, __longlong_as_double((long long)e.value))) : e.value;
    o.nx = beam_next((uint32_t)key[(l + 1) * cap + sn], j, sn);
    return o;
  };
  // The B best continuations of the n candidates cand(0 .. n - 1) at layer l (-1: the root), w_u added to each (add), written
  // to `to` by lane 0; false: none of them goes on.
  auto merge = [&](int l, int n, auto cand, bool add, double w_u, BeamEnt* to) -> bool {
    auto next_of = [&](int x) { return l + 1 < D ? (int)slot[(l + 1) * stride + cand(x)] : kEnded; };
    int sn = kEnded;                                                   // this lane's next node
    if (n <= 32) {
      if (lane < n) sn = next_of(lane);
    } else {
      Offer prev{~0ull, ~0ull};
      for (int r = 0; r < B; ++r) {
        Offer best{0ull, 0ull};
#pragma unroll 4
        for (int x = lane; x < n; x += 32) {
          const Offer o = offer_of(l, next_of(x), 0, add, w_u);
          const bool after = o.val < prev.val || (o.val == prev.val && o.nx < prev.nx);
          if (o.nx != 0ull && after && (o.val > best.val || (o.val == best.val && o.nx > best.nx))) best = o;
        }
        prev.val = warp_max64(best.val);
        prev.nx = warp_max64(best.val == prev.val ? best.nx : 0ull);
        if (prev.nx == 0ull) break;
        if (lane == r) sn = (int)(prev.nx & 0xffffffu);
      }
    }
    int j = 0;
    Offer mine = offer_of(l, sn, 0, add, w_u);
    for (int r = 0; r < B; ++r) {
      const u64 val = warp_max64(mine.val), nx = warp_max64(mine.val == val ? mine.nx : 0ull);
      if (nx == 0ull) {
        if (r == 0) return false;
        if (lane == 0) for (int x = r; x < B; ++x) to[x] = BeamEnt{0ull, 0ull};
        return true;
      }
      if (lane == 0) to[r] = BeamEnt{val, nx};
      if (mine.val == val && mine.nx == nx) mine = offer_of(l, sn, ++j, add, w_u);      // (every lane with this next node)
    }
    return true;
  };
#pragma unroll 1
  for (int l = D - 1; l >= 0; --l) {
    if (tid == 0) { sh_n = 0; sh_members = 0; }
    __syncthreads();
    for (int x = tid; x < cap; x += blockDim.x) {
      const int at = l * cap + x;
      if (key[at] < 0) continue;
      const unsigned c = cw[at];
      if ((c & 0xffffu) > 1u) {
        todo[atomicAdd(&sh_n, 1)] = (unsigned short)x;
        start[x] = atomicAdd(&sh_members, (int)(c & 0xffffu));
        continue;
      }
      const double w_u = weight(at);
      BeamEnt* const mine = ent + (size_t)at * es;
      const int sn = l + 1 < D ? (int)slot[(l + 1) * stride + (c >> 16)] : kEnded;
      if (sn == kEnded) mine[0] = BeamEnt{(u64)__double_as_longlong(w_u), kBeamLeaf};    // a leaf: its only continuation is to stop
      for (int r = sn == kEnded ? 1 : 0; r < B; ++r) {
        const Offer o = offer_of(l, sn, r, true, w_u);
        mine[r] = BeamEnt{o.val, o.nx};
      }
    }
    __syncthreads();
    const int n = sh_n;
    if (n > 0) {
      for (int m = tid; m < M; m += blockDim.x) {
        const int x = slot[l * stride + m];
        if (x != kEnded && (cw[l * cap + x] & 0xffffu) > 1u) member[atomicAdd(&start[x], 1)] = (unsigned short)m;
      }
      __syncthreads();
      for (int q = warp; q < n; q += nwarps) {
        const int x = todo[q], at = l * cap + x, cnt = (int)(cw[at] & 0xffffu);
        const unsigned short* const mem = member + start[x] - cnt;     // (start has moved to the end)
        const double w_u = weight(at);
        BeamEnt* const mine = ent + (size_t)at * es;
        if (!merge(l, cnt, [&](int y) { return (int)mem[y]; }, true, w_u, mine) && lane == 0)
          for (int r = 0; r < B; ++r) mine[r] = r == 0 ? BeamEnt{(u64)__double_as_longlong(w_u), kBeamLeaf} : BeamEnt{0ull, 0ull};
      }
      __syncthreads();
    }
  }
  if (warp == 0) {
    if (!merge(-1, M, [](int y) { return y; }, false, 0.0, sh_root) && lane == 0)
      for (int r = 0; r < B; ++r) sh_root[r] = BeamEnt{0ull, 0ull};
    __syncwarp();
    if (lane < B) {
      BeamEnt e = sh_root[lane];
      int len = 0;
      beam_value[lane] = e.next != 0ull ? (float)__longlong_as_double((long long)e.value) : 0.0f;
      for (int d = 0; d < D && e.next != 0ull && e.next != kBeamLeaf; ++d) {
        const int rank = 7 - (int)((e.next >> 24) & 7u), sl = (int)(e.next & 0xffffffu);
        if (lane == 0) sh_bslot[len] = sl;
        beam_tok[lane * D + len++] = (int32_t)~(uint32_t)(e.next >> 32);
        e = ent[((size_t)d * cap + sl) * es + rank];
      }
      if (lane == 0) sh_blen = len;
      for (int d = len; d < D; ++d) beam_tok[lane * D + d] = -1;
      beam_len[lane] = len;
    }
  }
  if (want0) {
    // node weights of the first beam, and of the edges it takes: a warp per layer
    if (tid < SDMS_MAX_DRAFT) { sh_be[tid][0] = 0u; sh_be[tid][1] = 0u; sh_be[tid][2] = 0u; }
    __syncthreads();
    const int len = sh_blen;
    if (score0 && tid < D) score0[tid] = tid < len ? (float)weight(tid * cap + sh_bslot[tid]) : 0.0f;
    if (edge0) {
      for (int l = warp; l < len; l += nwarps) {
        unsigned e0 = 0u, e1 = 0u, e2 = 0u;
        for (int m = lane; m < M; m += 32) {
          if (slot[l * stride + m] != sh_bslot[l] || (l > 0 && slot[(l - 1) * stride + m] != sh_bslot[l - 1])) continue;
          const unsigned p = (unsigned)ldm(s.pq + list[m] + l + 1);
          e0 += p & 0xffffu; e1 += p >> 16; ++e2;
        }
        e0 = __reduce_add_sync(FULL, e0); e1 = __reduce_add_sync(FULL, e1); e2 = __reduce_add_sync(FULL, e2);
        if (lane == 0) { sh_be[l][0] = e0; sh_be[l][1] = e1; sh_be[l][2] = e2; }
      }
      __syncthreads();
      if (tid < D) edge0[tid] = tid < len ? (float)eq5_weight(s.alpha, ((u64)sh_be[tid][1] << 16) + sh_be[tid][0], sh_be[tid][2]) : 0.0f;
    }
  }
  if (!SHARED_LISTS) {                                                  // leave the lists as they were found
    __syncthreads();
    for (int x = tid; x < all; x += blockDim.x)
      if (key[x] >= 0)
        for (int r = 0; r < B; ++r) ent[(size_t)x * es + r] = BeamEnt{0ull, 0ull};
  }
}

}  // namespace sdms
