// sdms_get_beams: several drafts per path.  One CTA per query path works out the B best paths of the
// pool of the last build (beam_dev.cuh), in shared memory where its tables fit, else over node
// tables that it reserves in the workspace's table area and leaves empty again.
#include "sdms_internal.h"
#include "beam_dev.cuh"

namespace sdms {

namespace {

// First slot of the tables of a path with M matches in the table area, -1: no room.  By one thread.
__device__ __forceinline__ long long reserve_tables(const Dev& s, int M) {
  if (M <= 0 || M > kWideMaxMatches) return -1;
  const unsigned long long need = (unsigned long long)s.D << beam_lcap(M);
  const unsigned long long at = atomicAdd(&s.b_ctl[kBeamSlots], need);
  return at + need <= s.w_slots ? (long long)at : -1;
}

// The beams of path i, in `bytes` of shared memory if they fit.  (The room in the table area decides who is served, also then.)
__device__ __forceinline__ void beams_of_path(const Dev& s, unsigned bytes, int i, int M, long long first, int B, int32_t* tok, int32_t* len,
                                              float* value, bool want0 = false, float* score0 = nullptr, float* edge0 = nullptr) {
  const BeamPlan w = beam_plan(M, s.D, B, bytes);
  BeamEnt* const ent = s.b_ent + (size_t)(unsigned)first * s.beam_stride;
  const int32_t* const list = s.matches + s.q_off[i];
  if (!w.cap) beams_of_query(s, i, M, list, (unsigned)first, beam_lcap(M), B, tok, len, value, want0, score0, edge0);
  else if (w.lists) beams_in_shared<true>(s, w, M, list, B, ent, s.beam_stride, tok, len, value, want0, score0, edge0);
  else beams_in_shared<false>(s, w, M, list, B, ent, s.beam_stride, tok, len, value, want0, score0, edge0);
}

// The launch's last CTA leaves all counts at zero.  By one thread of each, once it has its last slots and tickets.
__device__ __forceinline__ void beam_counts_done(const Dev& s) {
  __threadfence();
  if (atomicAdd(&s.b_ctl[kBeamDone], 1ull) == gridDim.x - 1)
    s.b_ctl[kBeamSlots] = s.b_ctl[kBeamTodo] = s.b_ctl[kBeamTicket] = s.b_ctl[kBeamDone] = 0ull;
}

__global__ void __launch_bounds__(kWideThreads, 1) beam_kernel(Dev s, int B, unsigned bytes, int32_t* __restrict__ beam_tok,
                                                               int32_t* __restrict__ beam_len,
                                                               float* __restrict__ beam_value) {
  grid_wait();
  grid_release();
  __shared__ long long sh_first;
  const int i = blockIdx.x, tid = threadIdx.x, D = s.D;
  int32_t* const my_tok = beam_tok + (size_t)i * B * D;
  const int M = s.q_mode[i] == Q_NONE ? 0 : min(s.q_cursor[i], s.q_reserved[i]);
  if (tid == 0) {
    sh_first = reserve_tables(s, M);
    if (M > 0 && sh_first < 0) atomicOr(s.status, SDMS_STATUS_TABLES_FULL);
    beam_counts_done(s);
  }
  __syncthreads();
  if (sh_first < 0) {                                  // no match, or no room: no beam
    for (int x = tid; x < B * D; x += blockDim.x) my_tok[x] = -1;
    if (tid < B) { beam_len[(size_t)i * B + tid] = 0; beam_value[(size_t)i * B + tid] = 0.0f; }
    return;
  }
  beams_of_path(s, bytes, i, M, sh_first, B, my_tok, beam_len + (size_t)i * B, beam_value + (size_t)i * B);
}

// Search mode 2: the paths that the build could not search in shared memory (dag_phase lists them in
// bp_todo) get their best path: the first beam of their pool, with scores and edge weights, in place of
// the greedy draft.  The CTAs take the listed paths in turn (one for each path of the context: 2048 of them, mostly with
// nothing to do, took 20 us).
__global__ void __launch_bounds__(kWideThreads, 1) best_path_fix_kernel(Dev s, unsigned bytes, int32_t* __restrict__ draft_tok,
                                                                        int32_t* __restrict__ draft_len,
                                                                        float* __restrict__ draft_score,
                                                                        float* __restrict__ draft_edge_w) {
  grid_wait();
  grid_release();
  __shared__ long long sh_first;
  __shared__ int sh_next;
  __shared__ float sh_value;
  const int tid = threadIdx.x, D = s.D;
  const int todo = (int)min(__ldcg(&s.b_ctl[kBeamTodo]), (unsigned long long)s.P);
#pragma unroll 1
  for (int x = blockIdx.x; x < todo;) {
    const int i = s.bp_todo[x];
    const int M = min(s.q_cursor[i], s.q_reserved[i]);
    if (tid == 0) {
      sh_first = reserve_tables(s, M);
      if (sh_first < 0) atomicOr(s.status, SDMS_STATUS_SEARCH_FALLBACK);       // the greedy draft stays
      sh_next = (int)(gridDim.x + atomicAdd(&s.b_ctl[kBeamTicket], 1ull));
    }
    __syncthreads();
    const long long first = sh_first;
    x = sh_next;
    if (first >= 0)
      beams_of_path(s, bytes, i, M, first, 1, draft_tok + (size_t)i * D, draft_len + i, &sh_value, true,
                    draft_score ? draft_score + (size_t)i * D : nullptr, draft_edge_w ? draft_edge_w + (size_t)i * D : nullptr);
    __syncthreads();                                   // before the next path's tables
  }
  if (tid == 0) beam_counts_done(s);
}

}  // namespace

// Called when a context is created, with its device current.
cudaError_t beam_kernel_setup() {
  int bytes = 0;
  for (int d = 1; d <= SDMS_MAX_DRAFT; ++d)
    for (int b = 1; b <= SDMS_MAX_BEAMS; ++b) bytes = max(bytes, beam_bytes(d, b));
  const cudaError_t e = cudaFuncSetAttribute(beam_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(best_path_fix_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_best_path_fix(const Dev& s, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                                 float* draft_edge_w, cudaStream_t stream) {
  const int bytes = beam_bytes(s.D, 1);
  return launch_overlapped(best_path_fix_kernel, dim3((unsigned)(s.P < 148 ? s.P : 148)), dim3(kWideThreads), bytes, stream, s,
                           (unsigned)bytes, draft_tok, draft_len, draft_score, draft_edge_w);
}

cudaError_t launch_beams(const Dev& s, int B, int32_t* beam_tok, int32_t* beam_len, float* beam_value,
                         cudaStream_t stream) {
  const int bytes = beam_bytes(s.D, B);
  return launch_overlapped(beam_kernel, dim3(s.P), dim3(kWideThreads), bytes, stream, s, B, (unsigned)bytes, beam_tok, beam_len,
                           beam_value);
}

}  // namespace sdms
