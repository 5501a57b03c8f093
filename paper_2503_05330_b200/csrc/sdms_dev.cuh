// Device-side view of a context and helpers shared by the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "sdms.h"

namespace sdms {

constexpr int kBucketWords = 8;        // one 32-byte sector: fingerprint, count, 6 positions
constexpr int kInlineSlots = kBucketWords - 2;
constexpr int kRecWords = 32;          // one 128-byte line per path: what a step needs first, in one load
constexpr int kRecEpoch = 31;          // its word that says which buckets of the index count (index_tag)
static_assert(kRecEpoch > SDMS_MAX_K, "length and tokens come first");
constexpr int kHalo = SDMS_MAX_K;      // tokens staged in front of a scan tile
constexpr int kScanTile = 1024;        // history tokens per scan CTA
constexpr int kScanThreads = 256;
constexpr int kDagThreads = 512;
constexpr int kMaxClusterPaths = 16;    // largest thread-block cluster (one CTA per path of a prompt)
constexpr int kFusedThreads = 512;     // the single-launch build: more loads in flight while it scans
constexpr int kDagCap = 1024;          // entries of the shared-memory node / edge tables
constexpr int kFusedMaxTokens = 131072; // largest N*L a CTA scans on its own
// The single-launch build's hand-over to the wide pass (hand_over_from, dag.cu): tokens N*L of a prompt from which, and paths up to which,
// there is one (exact, tolerance 1).
constexpr int kHandOverTokens = 65536, kHandOverPaths = 4 * 148;
constexpr int kHandOverTokensFuzzy = 16384, kHandOverPathsFuzzy = 2 * 148;
// Tokens held by a prompt (as far as the calls made tell) below which it is left out: the pass is 2 us (out of a cold cache 4 to 9) where there is nothing
// to do for it.  Exact, tokens times layers, which is what a walk costs: 64 x 409, D = 8, 33 / 36; 16 x 1230, D = 12, 47 / 33, 48 / 33, 54 / 43.  Tolerance 1 (where nothing is known of the queries before they are scanned), k = 2, without / with it: 16 x 614 29 and 34 / 33 and 31, 16 x 768
// 31 and 38 / 31 and 34; more CTAs than SMs: 8 x 32 x 614 75 and 76 / 81 and 73, x 768 86 and 86 / 86 and 84, x 1000 106 / 97; 9 x 32 x 900 108 and 92 / 103 and 94.
constexpr int kHandOverHeld = 229376, kHandOverHeldFuzzy = 11000, kHandOverHeldFuzzyRounds = 30000;
// Matches above which a query is handed over: 128 (256: 64 x 2048 47 to 58 us for 40 to 55, tolerance 1 36 to 46 for 34 to 41; 64: 46, but 113 for 108 with
// 4 x 128 x 512); for a CTA that others wait for an SM behind, whose time is not the launch's, 512 (k = 1, 32 x 16 x 4096: 125 us from 256, 122
// from 512, 126 from 1024, 144 from 2048; 4 x 64 x 2048: 65, 65, 73, 84).
constexpr int kHandOverFrom = 128, kHandOverEarly = 512;
constexpr int kMaxWide = 1024;          // queries one build can hand to the device-wide aggregation pass
constexpr int kWideSumShift = 47;       // packed node sums: count in the upper 17 bits, sum of probabilities below
constexpr int kWideMaxMatches = (1 << 17) - 1;   // so that both parts of a packed sum fit
// w_ctl: queries registered, slots handed out, tasks handed out, chunks handed out, chunks done, CTAs done, whether the pass
// is worth its while for this single-launch build.  Zero between builds
enum WideCtl : int { kWideListed = 0, kWideTaken = 1, kWideTask = 2, kWideChunkNext = 3, kWideChunksDone = 4, kWideLeft = 5, kWideHeavy = 6, kWideCtlWords = 7 };
// b_ctl: table slots handed out, a count that stays zero (sdms_debug_wait_timeout waits for it), paths in bp_todo, paths dealt out, CTAs done
enum BeamCtl : int { kBeamSlots = 0, kBeamNever = 1, kBeamTodo = 2, kBeamTicket = 3, kBeamDone = 4, kBeamCtlWords = 8 };

// Q_DONE: a back-off build on a large prompt has found this path's matches at a longer suffix length
enum QueryMode : int32_t { Q_NONE = 0, Q_INLINE = 1, Q_SCAN = 2, Q_DONE = 3 };
constexpr int kRoundBackoff = 1, kRoundNotFirst = 2, kRoundLast = 4;   // flags of one round of such a build

// One slot of a node table of one layer in the table area (32 bytes, one sector; beams).  All-zero = empty.  The keys
// (token + 1) that the probing looks at lie in an array of their own, eight to a sector.
struct WideSlot {
  uint32_t tok1;                 // token + 1, written by whoever claimed the slot
  uint32_t unused;
  unsigned long long sum;        // count << kWideSumShift | sum of fixed-point probabilities of the node
  unsigned long long pad[2];
};
struct BeamEnt;

// Everything a kernel needs, passed by value.
struct Dev {
  int32_t G, N, L, V, k_max, D, max_append, B, Ke, mode, P;
  int32_t idx_n;                       // n-gram lengths 1..idx_n have index tables (<= k_max; 0 with tolerance 1: nothing would look them up)
  int32_t pool;                        // 0 DAG, 1 tree, 2 list
  int32_t eps;                         // edit-distance tolerance of the suffix match (0 or 1)
  int32_t fused;                       // one kernel per build (small prompts) instead of probe + scan + dag
  int32_t build_cluster;               // CTAs per cluster of the single-launch build (they share their prompt's scan); 1 = none
  int32_t epochs;                      // a large index: a reset does not clear it but moves on to the next epoch, and its n-gram lengths are
                                       // chained (append_dev.cuh)
  int32_t held;                        // most tokens a path can hold, by the calls made so far
  int32_t R;                           // matches kept per (query path, source path): the R most recent; 0 = all
  double alpha;
  uint32_t table_cap;                  // buckets per (prompt, n) table, power of two
  uint32_t pos_mask;                   // bits of a bucket's entry that hold the position (entry_of)
  uint32_t L_magic; int32_t L_shift;   // x / L for 0 <= x < 2^31 as (x * L_magic) >> L_shift (path_of)
  int64_t match_cap;
  // path store
  int32_t* tok;                        // [P][L]
  int32_t* pq;                         // [P][L] fixed-point probabilities
  int32_t* len;                        // [P]
  int32_t* rec;                        // [P][kRecWords] per path: length, then its last k_max tokens, newest first; kRecEpoch
  uint32_t* status;
  uint32_t* index;                     // [G][k_max][table_cap][kBucketWords]
  // per-query scratch of the last build
  uint32_t* q_fp;                      // [P]
  int32_t* q_mode;                     // [P]
  int32_t* q_reserved;                 // [P] match slots reserved (index count)
  int32_t* q_off;                      // [P] start in `matches`
  int32_t* q_cursor;                   // [P] matches written
  unsigned long long* match_cursor;    // match slots handed to scan queries by the probe; zero between builds
  unsigned long long* f_notes;         // tolerance 1 on large prompts: matches noted by the counting scan
  int32_t* g_nscan;                    // [G] queries of the prompt that need the scan; zero between builds
  uint32_t* e_ctl;                     // [2] the word kRecEpoch of every record; CTAs of a reset that are done
  int2* a_plan;                        // [P] an append of wide rows: tokens the path held before, tokens it takes
  int32_t* g_trim;                     // [G] a path of the prompt was trimmed: its index is rebuilt
  int32_t* matches;                    // [match_cap] global positions j*L+e
  // device-wide aggregation of queries with many matches (dag_wide.cu); w_slots = 0: not in use
  unsigned long long* w_ctl;           // [kWideCtlWords]
  int4* w_desc;                        // [kMaxWide] query path, matches, first slot, -
  int* w_done;                         // [kMaxWide][2] tasks of the query that are done, of these sums; zero between builds
  WideSlot* w_tab;                     // [w_slots]
  uint32_t* w_key;                     // [w_slots] token + 1 of the node in the slot, 0 = free
  int32_t* w_item;                     // [w_slots] per (layer, match): slot of the item's token in the layer's table
  unsigned long long w_slots;
  BeamEnt* b_ent;                      // [w_slots][beam_stride] continuations kept per node (sdms_get_beams)
  unsigned long long* b_ctl;           // [kBeamCtlWords] counts of the beam kernels, all zero between calls
  int32_t beam_stride;                 // continuations kept per node: the context's max_beams, 1 for search mode 2 alone
  int32_t* bp_todo;                    // [P] search mode 2: paths whose best path is still to be searched, in no particular order
  int32_t w_grid;                      // CTAs of the wide pass
  // DAG export of the last build
  int32_t* x_node_tok; int64_t* x_node_S; int32_t* x_node_cnt; int32_t* x_node_count;
  int32_t* x_edge_dst; int64_t* x_edge_S; int32_t* x_edge_cnt; int32_t* x_out_degree;
};

// 64-bit hash of an n-gram, fed token by token (oldest first).
__device__ __forceinline__ uint64_t gram_init(int n) {
  return 0x9E3779B97F4A7C15ull * (uint64_t)(n + 1);
}
__device__ __forceinline__ uint64_t gram_step(uint64_t h, int32_t tok) {
  h = (h ^ (uint64_t)(uint32_t)tok) * 0xFF51AFD7ED558CCDull;
  return h ^ (h >> 29);
}
__device__ __forceinline__ uint64_t gram_final(uint64_t h) {
  h *= 0xC4CEB9FE1A85EC53ull;
  return h ^ (h >> 32);
}
// Non-zero 32-bit fingerprint and bucket number.
__device__ __forceinline__ uint32_t gram_fp(uint64_t h) { return (uint32_t)(h >> 32) | 1u; }
// First word of a bucket: 24 bits of fingerprint and the epoch (1 .. 255) in which the bucket was claimed.  A bucket of
// another epoch (0: never claimed) is empty, so that a reset of a large index has nothing to clear: clearing took
// 110 us for 0.84 GB, every time.  All paths hold the same epoch.  (Two n-grams with one fingerprint share a bucket: its
// count is an upper bound and its positions are verified token by token, as ever.)
__device__ __forceinline__ uint32_t epoch_of(int32_t rec_word) { return (uint32_t)rec_word + 1u; }
__device__ __forceinline__ uint32_t index_tag(uint64_t h, uint32_t epoch) { return ((uint32_t)(h >> 32) & ~0xffu) | epoch; }
__device__ __forceinline__ bool bucket_empty(uint32_t word, uint32_t epoch) { return (word & 0xffu) != epoch; }
__device__ __forceinline__ uint32_t gram_bucket(uint64_t h, uint32_t cap) { return (uint32_t)h & (cap - 1); }

__device__ __forceinline__ uint32_t* index_table(const Dev& s, int g, int n) {
  return s.index + ((size_t)(g * s.idx_n + (n - 1)) * s.table_cap) * kBucketWords;
}

// An entry of a bucket: the position (path within the prompt * L + position), and in a chained index, in the bits that leaves free, a hash of
// the token in front of the n-gram: a look-up for more tokens than the bucket's need not read the histories of those it cannot mean.
__device__ __forceinline__ uint32_t entry_of(const Dev& s, uint32_t lpos, int32_t before) {
  return lpos | ((uint32_t)before * 2654435761u & ~s.pos_mask);
}
__device__ __forceinline__ bool entry_may_follow(const Dev& s, uint32_t entry, int32_t before) {
  return ((entry ^ (uint32_t)before * 2654435761u) & ~s.pos_mask) == 0u;
}

// The bucket of the n-gram with hash h in the prompt's table, as two 16-byte words: false if there is none.  Ordinary loads: in the
// one-launch step other CTAs write the index earlier in the same launch.
__device__ __forceinline__ bool find_bucket(const Dev& s, int g, int n, uint64_t h, uint32_t epoch, uint4* lo, uint4* hi) {
  const uint4* const table = reinterpret_cast<const uint4*>(index_table(s, g, n));
  const uint32_t want = index_tag(h, epoch);
  uint32_t b = gram_bucket(h, s.table_cap);
#pragma unroll 1
  for (uint32_t probe = 0; probe < s.table_cap; ++probe) {
    *lo = table[2 * (size_t)b]; *hi = table[2 * (size_t)b + 1];        // both halves in flight together
    if (lo->x == want) return true;
    if (bucket_empty(lo->x, epoch)) return false;
    b = (b + 1) & (s.table_cap - 1);
  }
  return false;
}

// Path (row of the store) a global position x = j * L + e lies in, without a division: L_magic =
// ceil(2^(31 + l) / L) with l = ceil(log2 L) fits 32 bits and gives the exact quotient for every
// 0 <= x < 2^31 (round-up method of division by an invariant integer).
__device__ __forceinline__ int path_of(const Dev& s, int x) {
  return (int)(((uint64_t)(uint32_t)x * s.L_magic) >> s.L_shift);
}

// Eq. 5 on integer sums: alpha * S / 2^30 + (1 - alpha) * cnt, every operation
// rounded on its own (no fused multiply-add), so that any two evaluations of
// the same (S, cnt) agree bit for bit.
__device__ __forceinline__ double eq5_weight(double alpha, unsigned long long S, unsigned int cnt) {
  double t1 = __dmul_rn(alpha, (double)S);
  t1 = __dmul_rn(t1, 1.0 / 1073741824.0);
  double t2 = __dmul_rn(__dsub_rn(1.0, alpha), (double)cnt);
  return __dadd_rn(t1, t2);
}

// Is some window of k - 1, k or k + 1 tokens (at least one) that ends at `at` = row + e within one edit of q[0 .. k)?
// With a = common prefix and b = common suffix (each at most the shorter length) of q and the window: iff a + b >= the
// longer length - 1.  The window's tokens are compared with q at three offsets, one bit per token; all loads are independent.
__device__ __forceinline__ bool one_edit_end(const int32_t* at, int e, const int32_t* q, int k) {
  unsigned same = 0u, shorter = 0u, longer = 0u;       // bit t: the token t before the end equals q[k - 1 - t], q[k - 2 - t], q[k - t]
#pragma unroll 4
  for (int t = 0; t <= k; ++t) {
    const int x = t <= e ? at[-t] : -1;
    same |= (unsigned)(t < k && x == q[max(k - 1 - t, 0)]) << t;
    shorter |= (unsigned)(t + 1 < k && x == q[max(k - 2 - t, 0)]) << t;
    longer |= (unsigned)(t > 0 && x == q[k - t]) << t;
  }
  const int b = __ffs(~same) - 1;                      // common suffix of q and the path's end (the same for every window)
  auto ok = [&](int n, unsigned mask) {
    if (n < 1 || n > e + 1) return false;
    const int a = __clz(~(mask << (32 - n)));          // bits n - 1, n - 2, ...: the common prefix
    return min(a, min(k, n)) + min(b, min(k, n)) >= max(k, n) - 1;
  };
  return ok(k, same) || ok(k - 1, shorter) || ok(k + 1, longer);
}

// Programmatic dependent launch: a kernel launched with launch_overlapped() may be scheduled while
// the kernel before it on the stream is still draining.  grid_wait() returns once that kernel has
// completed and its writes are visible; everything that touches memory comes after it.
// grid_release() lets the next kernel on the stream start being scheduled.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Loads of path state (tokens, probabilities, lengths, records, index buckets).  In the one-launch step other CTAs write this
// state earlier in the same launch, and kernels that are launched over the step's end are resident while it still does: it is read
// with ordinary loads, which a cluster-scope acquire or grid_wait() keeps coherent, never through the read-only (non-coherent) path.
template <class T>
__device__ __forceinline__ T ldm(const T* p) { return *p; }

// Total order of the export and of the search: larger weight first, then smaller token.
__device__ __forceinline__ bool ranks_before(double wa, int ta, double wb, int tb) {
  return wa > wb || (wa == wb && ta < tb);
}

}  // namespace sdms
