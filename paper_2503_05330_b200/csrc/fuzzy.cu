// Fuzzy suffix matching (Eq. 4, tolerance 1) on prompts too large for the single-launch build.
//
// A position (j, e) matches query path i when some window of k - 1, k or k + 1 tokens that ends at e is
// within edit distance 1 of the query; each position counts once.  Index counts say nothing about how
// many such positions there are, so the match slices are sized by counting first:
//   fuzzy_prepare  every path with a query (k tokens, not full) is marked for scanning, counters zeroed
//   fuzzy_scan     (count) one CTA per 512-token tile of one path j: positions that can end a match of
//                  ANY query of the prompt are picked out by a bit table, then tested against every query;
//                  what matches is counted, and noted as (query, position) in the last two thirds of the match list
//   fuzzy_alloc    slices handed out from the match list by the counts
//   fuzzy_fill     the positions go from the notes to the slices; only if the notes did not have room for all
//                  matches, or slices would overlap them, does the same scan once more write the positions
// (96 x 2500 tokens, sessions of seven builds: 511 us with a second scan in every build, 397 with the notes)
// after which dag_kernel (and the wide pass) aggregate as for exact matching.
//
// The filter.  Let q be the query, |q| = k >= 2.  A window within one edit of q that ends at e either ends
// in q's last token, or differs from q only at its end: then the token at e or the one before it is
// q[k-1] or q[k-2] (substitution of the last token: tok[e-1] = q[k-2]; last token deleted: tok[e] =
// q[k-2]; a token appended: tok[e-1] = q[k-1]).  So a position passes when tok[e] or tok[e-1] hashes to
// a bit that some query set for q[k-1] or q[k-2].  With k = 1 every position is within one substitution
// of every query and nothing is filtered.
//
// The test: one_edit_end, for the pairs of candidate and query that the two tokens at the candidate's end do not rule
// out.  A scan of 96 x 3000 tokens took 84 us with every pair tested, 55 with the pairs sorted out first but tested where they
// turned up (one or two lanes of a warp at a time), 20.5 with the pairs queued per warp.
#include "sdms_internal.h"

namespace sdms {

namespace {

constexpr int kFzTile = 512;                       // 96 x 3000 tokens: 20.5 us a scan, with 256 21, with 1024 28.5 (too few CTAs)
constexpr int kFzThreads = 256;
constexpr int kFzHalo = SDMS_MAX_K + 1;            // tokens in front of a tile that a window may reach
constexpr int kFzBits = 65536;
constexpr int kFzQueries = 128;                    // queries whose tokens are staged at a time

// The notes of a build: pairs behind the first third of the match list.
__device__ __forceinline__ int64_t fz_notes_from(const Dev& s) { return (s.match_cap / 3 + 1) & ~1ll; }
__device__ __forceinline__ int64_t fz_notes_cap(const Dev& s) { return (s.match_cap - fz_notes_from(s)) / 2; }
__device__ __forceinline__ int2* fz_notes(const Dev& s) { return reinterpret_cast<int2*>(s.matches + fz_notes_from(s)); }

__device__ __forceinline__ uint32_t fz_bit(int32_t tok) { return ((uint32_t)tok * 2654435761u) >> 16; }

__global__ void __launch_bounds__(256) fuzzy_prepare_kernel(Dev s, int k, int skip_done) {
  grid_wait();
  grid_release();
  if (blockIdx.x == 0 && threadIdx.x == 0) *s.f_notes = 0ull;
  if (blockIdx.x == 0 && threadIdx.x < kWideCtlWords && s.w_grid) s.w_ctl[threadIdx.x] = 0ull;   // the wide pass of this build starts with an empty list
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= s.P) return;
  if (skip_done && s.q_mode[i] == Q_DONE) return;                // back-off: this path has its matches from a longer suffix
  const int len = s.len[i];
  s.q_fp[i] = 0u;
  s.q_mode[i] = len >= k && len < s.L ? Q_SCAN : Q_NONE;
  s.q_reserved[i] = 0; s.q_off[i] = 0; s.q_cursor[i] = 0;
}

__global__ void __launch_bounds__(256) fuzzy_alloc_kernel(Dev s) {
  grid_wait();
  grid_release();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= s.P || s.q_mode[i] != Q_SCAN) return;
  const long long count = s.q_reserved[i];
  const long long at = (long long)atomicAdd(s.match_cursor, (unsigned long long)count);
  if (at + count > s.match_cap) {
    s.q_mode[i] = Q_NONE; s.q_reserved[i] = 0;
    atomicOr(s.status, SDMS_STATUS_MATCH_OVERFLOW);
  } else {
    s.q_off[i] = (int32_t)at;
  }
}

// FILL: behind fuzzy_alloc; fills the slices from the notes if they are complete.
template <bool FILL>
__global__ void __launch_bounds__(kFzThreads) fuzzy_scan_kernel(Dev s, int k, int tiles) {
  __shared__ int32_t sh_tok[kFzHalo + kFzTile];            // sh_tok[kFzHalo + x] = token at t0 + x
  __shared__ uint32_t sh_bits[kFzBits / 32];
  __shared__ int32_t sh_q[kFzQueries][SDMS_MAX_K];
  __shared__ int32_t sh_qi[kFzQueries], sh_last[kFzQueries], sh_before[kFzQueries];   // its path, last token, the one before
  __shared__ int sh_count[kFzQueries];
  __shared__ int sh_pair[kFzThreads / 32][64];             // per warp: pairs that wait to be tested, position << 8 | query
  __shared__ int sh_cand[kFzTile];
  __shared__ int sh_ncand, sh_nq;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int j = blockIdx.x / tiles, t0 = (blockIdx.x - j * tiles) * kFzTile;
  const int g = j / s.N, len_j = s.len[j];
  const int e_hi = min(t0 + kFzTile - 1, len_j - 2);        // last position of the tile with a follower
  if (FILL) {
    grid_wait();
    grid_release();
    const int64_t notes = (int64_t)*s.f_notes;
    if (notes <= fz_notes_cap(s) && (int64_t)*s.match_cursor <= fz_notes_from(s)) {
      for (int64_t x = (int64_t)blockIdx.x * kFzThreads + tid; x < notes; x += (int64_t)gridDim.x * kFzThreads) {
        const int2 note = fz_notes(s)[x];
        const int n = atomicAdd(&s.q_cursor[note.x], 1);
        if (n < s.q_reserved[note.x]) s.matches[(size_t)s.q_off[note.x] + n] = note.y;
      }
      return;
    }
    if (t0 > e_hi) return;
  } else if (t0 > e_hi) {                                         // nothing to scan; but a launch none of whose CTAs waited would be over before
    grid_wait();                                           // the kernel in front of it, and the one behind would not wait for that
    return;
  }
  const int32_t* row = s.tok + (size_t)j * s.L;
  for (int x = tid; x < kFzHalo + kFzTile; x += blockDim.x) {
    const int at = t0 - kFzHalo + x;
    sh_tok[x] = at >= 0 && at < len_j ? row[at] : -1;
  }
  for (int x = tid; x < kFzBits / 32; x += blockDim.x) sh_bits[x] = 0u;
  if (tid == 0) sh_ncand = 0;
  // tokens and path lengths are older than the kernels this one follows (their CTAs let it start only after their own
  // wait): the tile was staged while those drained; the queries' state is read from here on
  if (!FILL) {
    grid_wait();
    grid_release();
  }
  // (earlier rounds of a back-off build have their slices at the front: they may reach into the notes)
  const int64_t room = !FILL && (int64_t)*s.match_cursor <= fz_notes_from(s) ? fz_notes_cap(s) : 0;
  __syncthreads();
  // the tokens that can sit at the end of a match: the last two of every query of the prompt
  if (k >= 2)
    for (int n = tid; n < s.N; n += blockDim.x) {
      const int i = g * s.N + n;
      if (i == j || s.q_mode[i] != Q_SCAN) continue;
      const int32_t* rec = s.rec + (size_t)i * kRecWords;   // rec[1 + t] = token t places from the end
      const uint32_t b0 = fz_bit(rec[1]), b1 = fz_bit(rec[2]);
      atomicOr(&sh_bits[b0 >> 5], 1u << (b0 & 31));
      atomicOr(&sh_bits[b1 >> 5], 1u << (b1 & 31));
    }
  __syncthreads();
  for (int x = tid; x <= e_hi - t0; x += blockDim.x) {
    bool pass = k < 2;
    if (!pass) {
      const uint32_t b0 = fz_bit(sh_tok[kFzHalo + x]);
      pass = sh_bits[b0 >> 5] >> (b0 & 31) & 1u;
      if (!pass && t0 + x >= 1) {
        const uint32_t b1 = fz_bit(sh_tok[kFzHalo + x - 1]);
        pass = sh_bits[b1 >> 5] >> (b1 & 31) & 1u;
      }
    }
    if (pass) sh_cand[atomicAdd(&sh_ncand, 1)] = x;
  }
  __syncthreads();
  const int ncand = sh_ncand;
  if (ncand == 0) return;
  // the candidates against every query of the prompt, kFzQueries queries at a time
  for (int n0 = 0; n0 < s.N; n0 += kFzQueries) {
    __syncthreads();
    if (tid == 0) sh_nq = 0;
    __syncthreads();
    for (int n = n0 + tid; n < min(s.N, n0 + kFzQueries); n += blockDim.x) {
      const int i = g * s.N + n;
      if (i == j || s.q_mode[i] != Q_SCAN) continue;
      const int at = atomicAdd(&sh_nq, 1);
      sh_qi[at] = i; sh_count[at] = 0;
      const int32_t* rec = s.rec + (size_t)i * kRecWords;
      for (int t = 0; t < k; ++t) sh_q[at][t] = rec[k - t];   // oldest token first
      sh_last[at] = rec[1]; sh_before[at] = k >= 2 ? rec[2] : rec[1];
    }
    __syncthreads();
    const int nq = sh_nq;
    // A warp per candidate, its lanes over the queries: the two tokens at the candidate's end decide almost always.  Pairs
    // that pass are queued and tested 32 at a time, so that no lane tests while the others wait.
    int waiting = 0;                                           // the same in every lane
    auto test = [&](int take) {
      __syncwarp();
      waiting -= take;
      int hit = -1, at = 0;
      if (lane < take) {
        const int pair = sh_pair[warp][waiting + lane], pos = pair >> 8, q = pair & 255;
        if (k < 2 || one_edit_end(sh_tok + kFzHalo + pos, t0 + pos, sh_q[q], k)) {
          hit = sh_qi[q];
          if (FILL) {
            const int n = atomicAdd(&s.q_cursor[hit], 1);
            if (n < s.q_reserved[hit]) s.matches[(size_t)s.q_off[hit] + n] = j * s.L + t0 + pos;
          } else {
            atomicAdd(&sh_count[q], 1);
            at = j * s.L + t0 + pos;
          }
        }
      }
      if (!FILL) {
        const unsigned hits = __ballot_sync(0xffffffffu, hit >= 0);
        if (hits) {                                            // the warp's matches side by side
          unsigned long long first = 0ull;
          if (lane == 0) first = atomicAdd(s.f_notes, (unsigned long long)__popc(hits));
          const int64_t note = (int64_t)__shfl_sync(0xffffffffu, first, 0) + __popc(hits & ((1u << lane) - 1u));
          if (hit >= 0 && note < room) fz_notes(s)[note] = make_int2(hit, at);
        }
      }
      __syncwarp();
    };
    for (int c = warp; c < ncand; c += kFzThreads / 32) {
      const int pos = sh_cand[c];                              // position t0 + pos; what lies before the path's start is -1
      const int32_t end = sh_tok[kFzHalo + pos], before_end = sh_tok[kFzHalo + pos - 1];
      for (int q0 = 0; q0 < nq; q0 += 32) {
        const int q = q0 + lane;
        bool pass = q < nq;
        if (pass && k >= 2) {
          const int32_t a = sh_last[q], b = sh_before[q];
          pass = end == a || end == b || before_end == a || before_end == b;
        }
        const unsigned who = __ballot_sync(0xffffffffu, pass);
        if (who == 0u) continue;
        if (pass) sh_pair[warp][waiting + __popc(who & ((1u << lane) - 1u))] = pos << 8 | q;
        waiting += __popc(who);
        if (waiting >= 32) test(32);
      }
    }
    if (waiting) test(waiting);
    if (!FILL) {
      __syncthreads();
      for (int q = tid; q < nq; q += blockDim.x)
        if (sh_count[q]) atomicAdd(&s.q_reserved[sh_qi[q]], sh_count[q]);
    }
  }
}

}  // namespace

// probe + scan of a build with tolerance 1 on a context that does not take the single-launch build
cudaError_t launch_fuzzy_match(const Dev& s, int k, int skip_done, cudaStream_t stream) {
  const int tiles = (s.L + kFzTile - 1) / kFzTile;
  const unsigned blocks = (unsigned)((s.P + 255) / 256);
  cudaError_t e = launch_overlapped(fuzzy_prepare_kernel, dim3(blocks), dim3(256), 0, stream, s, k, skip_done);
  if (e == cudaSuccess)
    e = launch_overlapped(fuzzy_scan_kernel<false>, dim3((unsigned)(s.P * tiles)), dim3(kFzThreads), 0, stream, s, k, tiles);
  if (e == cudaSuccess) e = launch_overlapped(fuzzy_alloc_kernel, dim3(blocks), dim3(256), 0, stream, s);
  if (e == cudaSuccess)
    e = launch_overlapped(fuzzy_scan_kernel<true>, dim3((unsigned)(s.P * tiles)), dim3(kFzThreads), 0, stream, s, k, tiles);
  return e;
}

}  // namespace sdms
