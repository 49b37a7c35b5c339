// Helper stream of a caller's stream: work that runs beside the caller's, forked from and joined
// back into it by events (also under stream capture, as a parallel branch).
#pragma once

#include <mutex>

#include "common.cuh"

namespace rlu {

// Created on first use, one per caller stream and device, so that concurrent calls on different
// streams keep separate helpers.
struct SideStream {
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  std::mutex mu;
};

int32_t side_stream(cudaStream_t main, SideStream** out);

// beside(helper stream) after everything enqueued on s so far, while body() enqueues on s; what
// follows on s waits for both.
template <typename Beside, typename Body>
int32_t run_beside(cudaStream_t s, Beside beside, Body body) {
  SideStream* ss = nullptr;
  RLU_TRY(side_stream(s, &ss));
  std::lock_guard<std::mutex> lock(ss->mu);
  RLU_CUDA_TRY(cudaEventRecord(ss->fork, s));
  RLU_CUDA_TRY(cudaStreamWaitEvent(ss->side, ss->fork, 0));
  const int32_t st = beside(ss->side);
  RLU_CUDA_TRY(cudaEventRecord(ss->join, ss->side));
  const int32_t bt = st == RLU_OK ? body() : st;
  RLU_CUDA_TRY(cudaStreamWaitEvent(s, ss->join, 0));  // also after an error: s stays ordered
  return bt;
}

}  // namespace rlu
