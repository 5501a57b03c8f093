// sdms_get_beams: several drafts per path.  One CTA per query path works out the B best paths of the
// pool of the last build (beam_dev.cuh) over node tables that it reserves in the workspace's table
// area and leaves empty again.
#include "sdms_internal.h"
#include "beam_dev.cuh"

namespace sdms {

namespace {

constexpr int kBeamSmem = 200 * 1024;                 // shared memory of a CTA: one per SM

// Called by one thread of every CTA once its slots are reserved: the last one leaves the count of reserved slots at zero.
__device__ __forceinline__ void reserved(unsigned long long* slots, unsigned long long* done) {
  __threadfence();
  if (atomicAdd(done, 1ull) == gridDim.x - 1) { *slots = 0ull; *done = 0ull; }
}

__global__ void __launch_bounds__(kWideThreads, 1) beam_kernel(Dev s, int B, int32_t* __restrict__ beam_tok,
                                                               int32_t* __restrict__ beam_len,
                                                               float* __restrict__ beam_value) {
  grid_wait();
  grid_release();
  __shared__ long long sh_first;
  const int i = blockIdx.x, tid = threadIdx.x, D = s.D;
  int32_t* const my_tok = beam_tok + (size_t)i * B * D;
  const int M = s.q_mode[i] == Q_NONE ? 0 : min(s.q_cursor[i], s.q_reserved[i]);
  const int lcap = beam_lcap(M);
  if (tid == 0) {
    long long first = -1;
    if (M > 0 && M <= kWideMaxMatches) {
      const unsigned long long need = (unsigned long long)D << lcap;
      const unsigned long long at = atomicAdd(s.b_ctl, need);
      if (at + need <= s.w_slots) first = (long long)at;
      else atomicOr(s.status, SDMS_STATUS_TABLES_FULL);
    } else if (M > 0) {
      atomicOr(s.status, SDMS_STATUS_TABLES_FULL);
    }
    sh_first = first;
    reserved(s.b_ctl, s.b_ctl + 2);
  }
  __syncthreads();
  if (sh_first < 0) {                                  // no match, or no room: no beam
    for (int x = tid; x < B * D; x += blockDim.x) my_tok[x] = -1;
    if (tid < B) { beam_len[(size_t)i * B + tid] = 0; beam_value[(size_t)i * B + tid] = 0.0f; }
    return;
  }
  // (the room in the table area decides who is served, also where the work is done in shared memory)
  const BeamPlan w = beam_plan(M, D, B, kBeamSmem);
  if (w.cap) {
    BeamEnt* const ent = s.b_ent + (size_t)(unsigned)sh_first * s.beam_stride;
    if (w.lists) beams_in_shared<true>(s, w, M, s.matches + s.q_off[i], B, ent, s.beam_stride, my_tok, beam_len + (size_t)i * B, beam_value + (size_t)i * B);
    else beams_in_shared<false>(s, w, M, s.matches + s.q_off[i], B, ent, s.beam_stride, my_tok, beam_len + (size_t)i * B, beam_value + (size_t)i * B);
    return;
  }
  beams_of_query(s, i, M, s.matches + s.q_off[i], (unsigned)sh_first, lcap, B, my_tok, beam_len + (size_t)i * B,
                 beam_value + (size_t)i * B);
}

// After a build with search mode 2: the paths that the build marked (more matches than its shared-memory
// search takes) get their best path here, in place of the greedy draft the build left them.
__global__ void __launch_bounds__(kWideThreads, 1) best_path_fix_kernel(Dev s, int32_t* __restrict__ draft_tok,
                                                                        int32_t* __restrict__ draft_len,
                                                                        float* __restrict__ draft_score,
                                                                        float* __restrict__ draft_edge_w) {
  grid_wait();
  grid_release();
  __shared__ long long sh_first;
  __shared__ float sh_value;
  const int i = blockIdx.x, tid = threadIdx.x, D = s.D;
  const bool mine = s.bp_todo[i] != 0;
  __syncthreads();
  const int M = min(s.q_cursor[i], s.q_reserved[i]);
  const int lcap = beam_lcap(M);
  if (tid == 0) {
    long long first = -1;
    if (mine) {
      s.bp_todo[i] = 0;
      if (M > 0 && M <= kWideMaxMatches) {
        const unsigned long long need = (unsigned long long)D << lcap;
        const unsigned long long at = atomicAdd(s.b_ctl + 1, need);
        if (at + need <= s.w_slots) first = (long long)at;
      }
      if (first < 0) atomicOr(s.status, SDMS_STATUS_SEARCH_FALLBACK);     // the greedy draft stays
    }
    sh_first = first;
    reserved(s.b_ctl + 1, s.b_ctl + 3);
  }
  __syncthreads();
  if (sh_first < 0) return;
  const BeamPlan w = beam_plan(M, D, 1, kBeamSmem);
  if (w.cap) {
    BeamEnt* const ent = s.b_ent + (size_t)(unsigned)sh_first * s.beam_stride;
    float* const score = draft_score ? draft_score + (size_t)i * D : nullptr;
    float* const edge = draft_edge_w ? draft_edge_w + (size_t)i * D : nullptr;
    if (w.lists) beams_in_shared<true>(s, w, M, s.matches + s.q_off[i], 1, ent, s.beam_stride, draft_tok + (size_t)i * D, draft_len + i, &sh_value, true, score, edge);
    else beams_in_shared<false>(s, w, M, s.matches + s.q_off[i], 1, ent, s.beam_stride, draft_tok + (size_t)i * D, draft_len + i, &sh_value, true, score, edge);
    return;
  }
  beams_of_query(s, i, M, s.matches + s.q_off[i], (unsigned)sh_first, lcap, 1, draft_tok + (size_t)i * D, draft_len + i,
                 &sh_value, true, draft_score ? draft_score + (size_t)i * D : nullptr,
                 draft_edge_w ? draft_edge_w + (size_t)i * D : nullptr);
}

}  // namespace

// Called when a context is created, with its device current.
cudaError_t beam_kernel_setup() {
  const cudaError_t e = cudaFuncSetAttribute(beam_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBeamSmem);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(best_path_fix_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBeamSmem);
}

cudaError_t launch_best_path_fix(const Dev& s, int32_t* draft_tok, int32_t* draft_len, float* draft_score,
                                 float* draft_edge_w, cudaStream_t stream) {
  return launch_overlapped(best_path_fix_kernel, dim3(s.P), dim3(kWideThreads), kBeamSmem, stream, s, draft_tok, draft_len,
                           draft_score, draft_edge_w);
}

cudaError_t launch_beams(const Dev& s, int B, int32_t* beam_tok, int32_t* beam_len, float* beam_value,
                         cudaStream_t stream) {
  return launch_overlapped(beam_kernel, dim3(s.P), dim3(kWideThreads), kBeamSmem, stream, s, B, beam_tok, beam_len, beam_value);
}

}  // namespace sdms
