// side_stream.h -- the context's side stream: delay constants and tables of a
// likelihood call run on it beside the orbit (emri_api.cu, run_loglike).
#pragma once
#include <cuda_runtime.h>

namespace emri {

struct SideStream {
  cudaStream_t stream = nullptr;   // null: not available, everything stays on the caller's stream
  cudaEvent_t ev[2] = {nullptr, nullptr};   // fork, join

  // All of it or nothing.  Doing without is no error: a failure's code does not
  // stay behind for the next call's cudaGetLastError.
  void create() {
    if (cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) == cudaSuccess &&
        cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) == cudaSuccess)
      return;
    stream = nullptr;
    destroy();
    cudaGetLastError();
  }
  void destroy() {
    if (stream) cudaStreamDestroy(stream);
    stream = nullptr;
    for (cudaEvent_t& e : ev) {
      if (e) cudaEventDestroy(e);
      e = nullptr;
    }
  }
};

}  // namespace emri
