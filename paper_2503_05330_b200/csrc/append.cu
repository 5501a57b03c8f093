// State update and acceptance kernels.
//
// append_kernel : one CTA per path; writes tokens and fixed-point probabilities
//                 into the path store and enters each new position into the prompt's
//                 hash tables: under every n-gram that ends at it, or once in a chained
//                 index (append_dev.cuh); with tolerance 1 there is no index.
// append_plan_kernel, append_bulk_kernel : the same for wide rows: how much each
//                 path takes, then many CTAs per path.
// accept_kernel : one CTA per path; longest accepted prefix of the draft
//                 ("Draft acceptance"), optionally followed by the same append.
// trim_*        : sliding window: shift the histories, empty and refill the tables.
#include "sdms_internal.h"
#include "append_dev.cuh"

namespace sdms {

namespace {

// (What a call is given may be what the call before it wrote, drafts or accept lengths, and this kernel is resident while that still
// does: no __restrict__ on inputs that are read behind grid_wait(), which would let them be read as read-only data.)
template <bool CHAINED>
__global__ void __launch_bounds__(128) append_kernel(Dev s, const int32_t* tokens, const float* logprobs, const int32_t* counts,
                                                     int row_width) {
  grid_wait();
  grid_release();
  const int p = blockIdx.x;
  __shared__ int sh_len0, sh_n, sh_bad;
  __shared__ uint32_t sh_st;
  __shared__ int32_t sh_rec[kRecWords];
  if (threadIdx.x < kRecWords) sh_rec[threadIdx.x] = s.rec[(size_t)p * kRecWords + threadIdx.x];
  if (threadIdx.x == 0) {
    uint32_t st = 0;
    int n = counts[p];
    if (n < 0) { st |= SDMS_STATUS_BAD_COUNT; n = 0; }
    if (n > row_width) { st |= SDMS_STATUS_BAD_COUNT; n = row_width; }
    const int len0 = sh_rec[0];
    if (n > s.L - len0) { st |= SDMS_STATUS_CAPACITY; n = s.L - len0; }
    sh_len0 = len0; sh_n = n; sh_bad = n; sh_st = st;
  }
  __syncthreads();
  const int32_t* in_tok = tokens + (size_t)p * row_width;
  const float* in_lp = logprobs + (size_t)p * row_width;
  for (int a = threadIdx.x; a < sh_n; a += blockDim.x) {
    const int32_t t = in_tok[a];
    if (t < 0 || t >= s.V) atomicMin(&sh_bad, a);
  }
  __syncthreads();
  uint32_t st = 0;
  const int n = sh_bad;
  if (threadIdx.x == 0 && n < sh_n) st |= SDMS_STATUS_BAD_TOKEN;
  append_tokens<CHAINED>(s, p, sh_len0, n, in_tok, in_lp, sh_rec, &st);
  if (st) atomicOr(&sh_st, st);
  __syncthreads();
  if (threadIdx.x == 0 && sh_st) atomicOr(s.status, sh_st);
}

// ---- wide rows ---------------------------------------------------------------------------------------
// Prefill: thousands of tokens per row.  What bounds it is the read-modify-write of the index at random, one or two 32-byte sectors
// per token (chained index), and how long each takes: 26 G positions/s with 1536 threads per SM and one bucket per thread at a time,
// DRAM at 19 % and L2 at 29 % of their rates.  So a row is cut into chunks with CTAs of their own (append of 32 x 16 x 3700 tokens, lengths
// up to 5: 118 us; 256 x 7800, up to 8: 140; with an entry per length 269 and 497, and the same in one CTA of 128 threads per path, append_kernel,
// 2270).  Also measured: four positions of a thread with their reads and claims on their way together, at 1024 threads per SM (32 x 16: 220 us,
// the lanes' ways through the lengths part), single tokens in a table of their own without hashing (256 x 7800: 155), prompts taken in turn (16 x 128 x 3900
// without a common token 351 for 302, with many 433 for 417).
// Small launches wait for the positions with the longest way along their chain, each length a look, a claim and a count.  Reset and append, with an entry
// per length / chained: 16 x 2200 tokens, lengths up to 8, 97 % full, little in common 18 / 15, a third 21 / 17, mostly the same phrases 19 / 26; a fifth full 11 / 13 and 10 / 21;
// 64 x 2048, up to 4, 97 % full 32 / 27 and 29 / 27, a fifth full 12 / 15 and 12 / 16.  (The builds behind it take 4 us less where a query has 7 to 12 occurrences.)  Also measured: all further
// lengths of a position at once, with places given out twice (16 x 2200 26 / 24, but 8 x 16 x 1024 20 / 28, 64 x 2048, up to 16, 42 / 67).
// Indexes that are cleared have an entry per length, and a CTA each for it: 16 x 1024 17 us.
constexpr int kPlanThreads = 256;
constexpr int kBulkThreads = 256;
constexpr int kBulkChunk = 512;          // most positions per CTA

// What every path takes of its row: tokens held so far, tokens to append.
__global__ void __launch_bounds__(kPlanThreads) append_plan_kernel(Dev s, const int32_t* tokens, const int32_t* counts, int row_width) {
  grid_wait();
  grid_release();
  __shared__ int sh_bad;
  const int p = blockIdx.x;
  uint32_t st = 0;
  int n = counts[p];
  if (n < 0) { st |= SDMS_STATUS_BAD_COUNT; n = 0; }
  if (n > row_width) { st |= SDMS_STATUS_BAD_COUNT; n = row_width; }
  const int len0 = s.len[p];
  if (n > s.L - len0) { st |= SDMS_STATUS_CAPACITY; n = s.L - len0; }
  if (threadIdx.x == 0) sh_bad = n;
  __syncthreads();
  const int32_t* in_tok = tokens + (size_t)p * row_width;
  int bad = n;
#pragma unroll 4
  for (int a = threadIdx.x; a < n; a += kPlanThreads) {
    const int32_t t = in_tok[a];
    if (t < 0 || t >= s.V) bad = min(bad, a);
  }
  if (bad < n) atomicMin(&sh_bad, bad);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sh_bad < n) st |= SDMS_STATUS_BAD_TOKEN;
    s.a_plan[p] = make_int2(len0, sh_bad);
    if (st) atomicOr(s.status, st);
  }
}

// Buckets that are known to be full, and what this CTA has to add to their counts.  The commonest token of a text is a few percent of
// it: counted one by one, its tens of thousands of occurrences queue up at one address (16 x 128 x 3900 tokens, a quarter of them
// Zipf(1.1): 568 us counted one by one, 417 with this; 2 x 256 x 3900, 60 % of them, 32000 different: 529 and 234).  Lengths 1 and 2 of a chained index; the whole hash is compared, and what
// hashes to the same is in the same bucket.
constexpr int kFullSlots = 128;
struct FullBuckets { unsigned long long key[2][kFullSlots]; uint32_t bucket[2][kFullSlots]; unsigned count[2][kFullSlots]; };
__device__ __forceinline__ void full_empty(FullBuckets& f) {
  for (int x = threadIdx.x; x < 2 * kFullSlots; x += kBulkThreads) { (&f.key[0][0])[x] = 0ull; (&f.count[0][0])[x] = 0u; }
}
__device__ __forceinline__ void full_count(const Dev& s, int g, const FullBuckets& f) {
  for (int x = threadIdx.x; x < 2 * kFullSlots; x += kBulkThreads) {
    const unsigned c = (&f.count[0][0])[x];
    if (c == 0u) continue;
    uint32_t* const bucket = index_table(s, g, x / kFullSlots + 1) + (size_t)(&f.bucket[0][0])[x] * kBucketWords;
    atomicAdd(reinterpret_cast<unsigned long long*>(bucket), (unsigned long long)c << 32);
  }
}

// The n-grams of length n that end at positions [x0, x1) of path p into the prompt's tables.  win[kHalo - 1 + t] = token at x0 + t
// (shared memory).
__device__ __forceinline__ uint64_t window_hash(const int32_t* win, int t, int n) {
  uint64_t h = gram_init(n);
  const int32_t* q = win + kHalo - n + t;
  for (int u = 0; u < n; ++u) h = gram_step(h, q[u]);
  return gram_final(h);
}
__device__ __forceinline__ void insert_positions(const Dev& s, int p, int n, int x0, int x1, const int32_t* win, uint32_t* st) {
  const int g = p / s.N;
  const uint32_t epoch = epoch_of(s.rec[(size_t)p * kRecWords + kRecEpoch]);
  const uint32_t lbase = (uint32_t)(p - g * s.N) * (uint32_t)s.L;
  for (int x = x0 + (int)threadIdx.x; x < x1; x += kBulkThreads)
    if (x + 1 >= n) index_insert<true, false>(s, g, n, window_hash(win, x - x0, n), lbase + (uint32_t)x, epoch, st);
}

// The same for a chained index, one length after the other.  FULL: with FullBuckets.  Every thread of the CTA, after a barrier.
template <bool FULL>
__device__ __forceinline__ void chain_positions(const Dev& s, int p, int x0, int x1, const int32_t* win, uint32_t* st) {
  __shared__ FullBuckets f;
  const int g = p / s.N;
  const uint32_t epoch = epoch_of(s.rec[(size_t)p * kRecWords + kRecEpoch]);
  const uint32_t lbase = (uint32_t)(p - g * s.N) * (uint32_t)s.L;
  if (FULL) {
    full_empty(f);
    __syncthreads();
  }
  for (int x = x0 + (int)threadIdx.x; x < x1; x += kBulkThreads) {
    const int last = min(s.idx_n, x + 1);
#pragma unroll 1
    for (int n = 1; n <= last; ++n) {
      const uint64_t h = window_hash(win, x - x0, n);
      const int at = (int)(h >> 40) & (kFullSlots - 1), l = n - 1;
      if (FULL && l < 2 && *(volatile unsigned long long*)&f.key[l][at] == h && h != 0ull) { atomicAdd(&f.count[l][at], 1u); continue; }
      auto full = [&](uint32_t b) {
        if (!FULL || l >= 2 || h == 0ull) return false;
        const unsigned long long k = atomicCAS(&f.key[l][at], 0ull, (unsigned long long)h);
        if (k != 0ull && k != h) return false;
        f.bucket[l][at] = b;
        atomicAdd(&f.count[l][at], 1u);
        return true;
      };
      const int32_t before = n < kHalo ? win[kHalo - 1 - n + x - x0] : 0;        // (no query is longer than kHalo)
      if (index_insert<true, true>(s, g, n, h, entry_of(s, lbase + (uint32_t)x, before), epoch, st, full)) break;
    }
  }
  if (FULL) {
    __syncthreads();
    full_count(s, g, f);
  }
}

// Grid: (path, chunk of its row) x n, n slowest; chained index, or none: x 1.
enum BulkForm { kPerLength, kChain, kChainFull };
constexpr int bulk_ctas(int form) { return form == kPerLength ? 8 : 6; }
template <int FORM>
__global__ void __launch_bounds__(kBulkThreads, bulk_ctas(FORM)) append_bulk_kernel(Dev s, const int32_t* __restrict__ tokens,
                                                                      const float* __restrict__ logprobs, int row_width,
                                                                      int chunk, int chunks) {
  __shared__ int32_t sh_win[kHalo - 1 + kBulkChunk];
  const int p = blockIdx.x / chunks, c0 = (blockIdx.x - p * chunks) * chunk, tid = threadIdx.x;
  const int32_t* in_tok = tokens + (size_t)p * row_width;
  // the row is older than the plan (whose CTAs let this kernel start only after their own wait)
  for (int t = tid; t < chunk; t += kBulkThreads) sh_win[kHalo - 1 + t] = c0 + t < row_width ? in_tok[c0 + t] : 0;
  grid_wait();
  grid_release();
  const int2 plan = s.a_plan[p];
  const int len0 = plan.x, n = plan.y;
  if (c0 >= n) return;
  int32_t* tok = s.tok + (size_t)p * s.L;
  if (tid < kHalo - 1) {                                              // the tokens before the chunk: of the row, or held before
    const int x = c0 - (kHalo - 1) + tid;
    sh_win[tid] = x >= 0 ? in_tok[x] : (len0 + x >= 0 ? tok[len0 + x] : 0);
  }
  __syncthreads();
  uint32_t st = 0;
  const int m = min(chunk, n - c0);
  if (blockIdx.y == 0) {
    if (c0 == 0) {                                                    // length and record as they are after the call
      const int x = len0 + n - 1 - tid;
      int32_t* rec = s.rec + (size_t)p * kRecWords;
      if (tid < s.k_max) rec[1 + tid] = x >= len0 ? in_tok[x - len0] : (x >= 0 ? tok[x] : 0);
      if (tid == s.k_max) { rec[0] = len0 + n; s.len[p] = len0 + n; }
    }
    const float* in_lp = logprobs + (size_t)p * row_width;
    for (int t = tid; t < m; t += kBulkThreads) {
      tok[len0 + c0 + t] = sh_win[kHalo - 1 + t];
      s.pq[(size_t)p * s.L + len0 + c0 + t] = prob_to_fixed(in_lp[c0 + t], &st);
    }
  }
  if (FORM != kPerLength) chain_positions<FORM == kChainFull>(s, p, len0 + c0, len0 + c0 + m, sh_win, &st);
  else if (s.idx_n > 0) insert_positions(s, p, (int)blockIdx.y + 1, len0 + c0, len0 + c0 + m, sh_win, &st);
  if (st) atomicOr(s.status, st);
}

template <bool CHAINED>
__global__ void __launch_bounds__(128) accept_kernel(Dev s, const int32_t* draft_tok, const int32_t* draft_len, const int32_t* sampled,
                                                     const float* sampled_lp, int32_t* accept_len) {
  grid_wait();
  grid_release();
  accept_commit_phase<CHAINED>(s, blockIdx.x, draft_tok, draft_len, sampled, sampled_lp, accept_len);
}

// sdms_reset of a large index: lengths, records and the small state between `a` / `b` and their ends become zero, the
// records get the next epoch.  Only when the epochs run out (every 255th time) the index is cleared.
__global__ void __launch_bounds__(256) reset_kernel(Dev s, uint4* a, size_t a_words, uint4* b, size_t b_words, size_t index_words) {
  grid_wait();
  grid_release();
  const uint32_t next = *(volatile uint32_t*)s.e_ctl + 1u < 255u ? *(volatile uint32_t*)s.e_ctl + 1u : 0u;
  const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
  const size_t rec0 = reinterpret_cast<uint4*>(s.rec) - a, rec1 = rec0 + (size_t)s.P * kRecWords / 4;
  for (size_t x = first; x < a_words; x += step) {
    const bool tail = x >= rec0 && x < rec1 && (x - rec0) % (kRecWords / 4) == kRecWords / 4 - 1;
    a[x] = make_uint4(0u, 0u, 0u, tail ? next : 0u);
  }
  for (size_t x = first; x < b_words; x += step) b[x] = make_uint4(0u, 0u, 0u, 0u);
  if (next == 0u)
    for (size_t x = first; x < index_words; x += step) reinterpret_cast<uint4*>(s.index)[x] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&s.e_ctl[1], 1u) == gridDim.x - 1) { s.e_ctl[1] = 0u; s.e_ctl[0] = next; }      // everybody has read it
  }
}

// sdms_trim, first launch: path p keeps its newest keep[p] tokens, moved to the front of its store.
__global__ void __launch_bounds__(128) trim_shift_kernel(Dev s, const int32_t* keep) {
  grid_wait();
  grid_release();
  const int p = blockIdx.x;
  const int len = s.len[p], want = keep[p];
  if (want < 0) {
    if (threadIdx.x == 0) atomicOr(s.status, SDMS_STATUS_BAD_COUNT);
    return;
  }
  if (want >= len) return;
  const int shift = len - want;
  int32_t* tok = s.tok + (size_t)p * s.L;
  int32_t* pq = s.pq + (size_t)p * s.L;
  // a block of the kept tokens is read whole before any of it is written: the source of a later
  // block lies behind everything written so far
  for (int base = 0; base < want; base += blockDim.x) {
    const int x = base + threadIdx.x;
    int32_t t = 0, q = 0;
    if (x < want) { t = tok[x + shift]; q = pq[x + shift]; }
    __syncthreads();
    if (x < want) { tok[x] = t; pq[x] = q; }
    __syncthreads();
  }
  int32_t* rec = s.rec + (size_t)p * kRecWords;
  if (threadIdx.x == 0) { s.len[p] = want; rec[0] = want; s.g_trim[p / s.N] = 1; }
  if (threadIdx.x >= 1 && threadIdx.x <= SDMS_MAX_K && (int)threadIdx.x > want) rec[threadIdx.x] = 0;   // tokens that are gone
}

// Second launch: the tables of the prompts that changed become empty.
__global__ void __launch_bounds__(256) trim_clear_kernel(Dev s) {
  grid_wait();
  grid_release();
  const size_t per_group = (size_t)s.idx_n * s.table_cap * kBucketWords / 4;      // 16-byte words of a prompt's tables
  uint4* index = reinterpret_cast<uint4*>(s.index);
  for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < per_group * s.G; x += (size_t)gridDim.x * blockDim.x)
    if (s.g_trim[x / per_group]) index[x] = make_uint4(0u, 0u, 0u, 0u);
}

// Third launch: every position of those prompts goes into the tables again.
template <int FORM>
__global__ void __launch_bounds__(kBulkThreads, bulk_ctas(FORM)) trim_reindex_kernel(Dev s, int chunk, int chunks) {
  __shared__ int32_t sh_win[kHalo - 1 + kBulkChunk];
  grid_wait();
  grid_release();
  const int p = blockIdx.x / chunks, x0 = (blockIdx.x - p * chunks) * chunk;
  if (!s.g_trim[p / s.N]) return;
  const int x1 = min(x0 + chunk, s.len[p]);
  if (x0 >= x1) return;
  const int32_t* tok = s.tok + (size_t)p * s.L;
  for (int t = threadIdx.x; t < kHalo - 1 + chunk; t += kBulkThreads) {
    const int x = x0 - (kHalo - 1) + t;
    sh_win[t] = x >= 0 && x < x1 ? tok[x] : 0;
  }
  __syncthreads();
  uint32_t st = 0;
  if (FORM != kPerLength) chain_positions<FORM == kChainFull>(s, p, x0, x1, sh_win, &st);
  else if (s.idx_n > 0) insert_positions(s, p, (int)blockIdx.y + 1, x0, x1, sh_win, &st);
  if (st) atomicOr(s.status, st);
}

}  // namespace

cudaError_t launch_reset(const Dev& s, void* a, size_t a_bytes, void* b, size_t b_bytes, size_t index_bytes, cudaStream_t stream) {
  const size_t words = (a_bytes + b_bytes) / 16;
  const unsigned ctas = (unsigned)(words < 148 * 256 ? (words + 255) / 256 : 148 * 4);
  return launch_overlapped(reset_kernel, dim3(ctas), dim3(256), 0, stream, s, static_cast<uint4*>(a), a_bytes / 16, static_cast<uint4*>(b),
                           b_bytes / 16, index_bytes / 16);
}

namespace {
// The kernels that index rows of `width` positions of every path.  Few, short CTAs where the device has room for all of them at once
// (16 x 700: 26 us, with 512 30 us).
struct BulkPlan { int chunk, chunks, lengths; BulkForm form; };
BulkPlan bulk_plan(const Dev& s, int width) {
  BulkPlan b;
  b.lengths = s.epochs || s.idx_n == 0 ? 1 : s.idx_n;
  const bool many = (long long)s.P * b.lengths * ((width + kBulkChunk - 1) / kBulkChunk) > 148LL * 8;
  b.chunk = many ? kBulkChunk : kBulkChunk / 2;
  b.chunks = (width + b.chunk - 1) / b.chunk;
  b.form = !s.epochs ? kPerLength : many ? kChainFull : kChain;
  return b;
}
}  // namespace

cudaError_t launch_trim(const Dev& s, int phase, const int32_t* keep, cudaStream_t stream) {
  if (phase == 0) return launch_overlapped(trim_shift_kernel, dim3(s.P), dim3(128), 0, stream, s, keep);
  if (phase == 1) return launch_overlapped(trim_clear_kernel, dim3(148 * 8), dim3(256), 0, stream, s);
  const BulkPlan b = bulk_plan(s, s.L);
  const auto kernel = b.form == kPerLength ? trim_reindex_kernel<kPerLength> : b.form == kChain ? trim_reindex_kernel<kChain> : trim_reindex_kernel<kChainFull>;
  return launch_overlapped(kernel, dim3((unsigned)(s.P * b.chunks), b.lengths), dim3(kBulkThreads), 0, stream, s, b.chunk, b.chunks);
}

cudaError_t launch_append(const Dev& s, const int32_t* tokens, const float* logprobs, const int32_t* counts,
                          int row_width, cudaStream_t stream) {
  if (row_width < kBulkAppendFrom)
    return launch_overlapped(s.epochs ? append_kernel<true> : append_kernel<false>, dim3(s.P), dim3(128), 0, stream, s, tokens, logprobs, counts, row_width);
  const cudaError_t e = launch_overlapped(append_plan_kernel, dim3(s.P), dim3(kPlanThreads), 0, stream, s, tokens, counts, row_width);
  if (e != cudaSuccess) return e;
  const int width = row_width < s.L ? row_width : s.L;                // no path takes more
  const BulkPlan b = bulk_plan(s, width);
  const auto kernel = b.form == kPerLength ? append_bulk_kernel<kPerLength> : b.form == kChain ? append_bulk_kernel<kChain> : append_bulk_kernel<kChainFull>;
  return launch_overlapped(kernel, dim3((unsigned)(s.P * b.chunks), b.lengths), dim3(kBulkThreads), 0, stream, s, tokens, logprobs,
                           row_width, b.chunk, b.chunks);
}

cudaError_t launch_accept(const Dev& s, const int32_t* draft_tok, const int32_t* draft_len,
                          const int32_t* sampled, const float* sampled_lp, int32_t* accept_len,
                          cudaStream_t stream) {
  return launch_overlapped(s.epochs ? accept_kernel<true> : accept_kernel<false>, dim3(s.P), dim3(128), 0, stream, s, draft_tok, draft_len, sampled, sampled_lp,
                           accept_len);
}

}  // namespace sdms
