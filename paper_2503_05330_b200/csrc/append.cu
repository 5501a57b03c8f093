// State update and acceptance kernels.
//
// append_kernel : one CTA per path; writes tokens and fixed-point probabilities
//                 into the path store and inserts the n-grams (n = 1..k_max) that
//                 end at each new position into the prompt's hash tables.
// append_plan_kernel, append_bulk_kernel : the same for wide rows: how much each
//                 path takes, then many CTAs per path.
// accept_kernel : one CTA per path; longest accepted prefix of the draft
//                 ("Draft acceptance"), optionally followed by the same append.
// trim_*        : sliding window: shift the histories, empty and refill the tables.
#include "sdms_internal.h"
#include "append_dev.cuh"

namespace sdms {

namespace {

__global__ void __launch_bounds__(128) append_kernel(Dev s, const int32_t* __restrict__ tokens,
                                                     const float* __restrict__ logprobs,
                                                     const int32_t* __restrict__ counts, int row_width) {
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
  append_tokens(s, p, sh_len0, n, in_tok, in_lp, sh_rec, &st);
  if (st) atomicOr(&sh_st, st);
  __syncthreads();
  if (threadIdx.x == 0 && sh_st) atomicOr(s.status, sh_st);
}

// ---- wide rows ---------------------------------------------------------------------------------------
// Prefill: thousands of tokens per row.  What bounds it is the random read-modify-write of the index, one 32-byte
// sector per token and n-gram length in tables far larger than L2 (a B200 does 24 G/s of them in a 1 GiB region,
// 110 G/s in 32 MiB).  So a row is cut into chunks with CTAs of their own, at 2048 threads per SM and one insert
// per thread at a time (four inserts per thread with their atomics in flight together, at half the threads, were no
// faster); and the n-gram lengths go one after the other over the grid, so that what is being written at a time is
// one table per prompt and not all k_max of them: 256 paths x 7800 tokens x 8 lengths 530 us, with all lengths in one
// CTA 750 us, with one CTA of 128 threads per path (append_kernel) 2270 us.
constexpr int kPlanThreads = 256;
constexpr int kBulkThreads = 256;
constexpr int kBulkChunk = 512;          // positions per CTA; half of it when that leaves SMs without a full load

// What every path takes of its row: tokens held so far, tokens to append.
__global__ void __launch_bounds__(kPlanThreads) append_plan_kernel(Dev s, const int32_t* __restrict__ tokens,
                                                                   const int32_t* __restrict__ counts, int row_width) {
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

// The n-grams of length n that end at positions [x0, x1) of path p into the prompt's table.  win[kHalo - 1 + t] = token
// at x0 + t (shared memory).
__device__ __forceinline__ void insert_positions(const Dev& s, int p, int n, int x0, int x1, const int32_t* win, uint32_t* st) {
  const int g = p / s.N;
  const uint32_t epoch = epoch_of(s.rec[(size_t)p * kRecWords + kRecEpoch]);
  const uint32_t lbase = (uint32_t)(p - g * s.N) * (uint32_t)s.L;
  for (int x = x0 + (int)threadIdx.x; x < x1; x += kBulkThreads) {
    if (x + 1 < n) continue;
    uint64_t h = gram_init(n);
    const int32_t* q = win + kHalo - n + (x - x0);
    for (int t = 0; t < n; ++t) h = gram_step(h, q[t]);
    index_insert<true>(s, g, n, gram_final(h), lbase + (uint32_t)x, epoch, st);
  }
}

// Grid: (path, chunk of its row) x n, n slowest.
__global__ void __launch_bounds__(kBulkThreads, 8) append_bulk_kernel(Dev s, const int32_t* __restrict__ tokens,
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
  insert_positions(s, p, (int)blockIdx.y + 1, len0 + c0, len0 + c0 + m, sh_win, &st);
  if (st) atomicOr(s.status, st);
}

__global__ void __launch_bounds__(128) accept_kernel(Dev s, const int32_t* __restrict__ draft_tok,
                                                     const int32_t* __restrict__ draft_len,
                                                     const int32_t* __restrict__ sampled,
                                                     const float* __restrict__ sampled_lp,
                                                     int32_t* __restrict__ accept_len) {
  grid_wait();
  grid_release();
  accept_commit_phase(s, blockIdx.x, draft_tok, draft_len, sampled, sampled_lp, accept_len);
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
__global__ void __launch_bounds__(128) trim_shift_kernel(Dev s, const int32_t* __restrict__ keep) {
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

// Third launch: every n-gram (n = 1..k_max) of every path of those prompts goes into the tables again.
__global__ void __launch_bounds__(kBulkThreads, 8) trim_reindex_kernel(Dev s, int chunk, int chunks) {
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
  insert_positions(s, p, (int)blockIdx.y + 1, x0, x1, sh_win, &st);
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
// Positions per CTA of the kernels that index rows of `width` positions of every path: few, short CTAs where the device
// has room for all of them at once (16 x 700: 26 us, with 512 30 us).
int bulk_chunk(const Dev& s, int width) {
  const long long ctas = (long long)s.P * s.idx_n * ((width + kBulkChunk - 1) / kBulkChunk);
  return ctas > 148LL * 8 ? kBulkChunk : kBulkChunk / 2;
}
}  // namespace

cudaError_t launch_trim(const Dev& s, int phase, const int32_t* keep, cudaStream_t stream) {
  if (phase == 0) return launch_overlapped(trim_shift_kernel, dim3(s.P), dim3(128), 0, stream, s, keep);
  if (phase == 1) return launch_overlapped(trim_clear_kernel, dim3(148 * 8), dim3(256), 0, stream, s);
  const int chunk = bulk_chunk(s, s.L), chunks = (s.L + chunk - 1) / chunk;
  return launch_overlapped(trim_reindex_kernel, dim3((unsigned)(s.P * chunks), s.idx_n), dim3(kBulkThreads), 0, stream, s, chunk, chunks);
}

cudaError_t launch_append(const Dev& s, const int32_t* tokens, const float* logprobs, const int32_t* counts,
                          int row_width, cudaStream_t stream) {
  if (row_width < kBulkAppendFrom)
    return launch_overlapped(append_kernel, dim3(s.P), dim3(128), 0, stream, s, tokens, logprobs, counts, row_width);
  const cudaError_t e = launch_overlapped(append_plan_kernel, dim3(s.P), dim3(kPlanThreads), 0, stream, s, tokens, counts, row_width);
  if (e != cudaSuccess) return e;
  const int width = row_width < s.L ? row_width : s.L;                // no path takes more
  const int chunk = bulk_chunk(s, width), chunks = (width + chunk - 1) / chunk;
  return launch_overlapped(append_bulk_kernel, dim3((unsigned)(s.P * chunks), s.idx_n), dim3(kBulkThreads), 0, stream, s, tokens,
                           logprobs, row_width, chunk, chunks);
}

cudaError_t launch_accept(const Dev& s, const int32_t* draft_tok, const int32_t* draft_len,
                          const int32_t* sampled, const float* sampled_lp, int32_t* accept_len,
                          cudaStream_t stream) {
  return launch_overlapped(accept_kernel, dim3(s.P), dim3(128), 0, stream, s, draft_tok, draft_len, sampled, sampled_lp,
                           accept_len);
}

}  // namespace sdms
