// The context's side stream over a fake runtime: the n-th creating call fails
// and leaves its error, as the CUDA runtime does, until somebody asks for it.
#include "side_stream.h"

static int g_calls, g_fail, g_live;
static cudaError_t g_last;

static cudaError_t make(void** out) {
  if (++g_calls == g_fail) return g_last = cudaErrorMemoryAllocation;
  ++g_live;
  *out = (void*)(size_t)g_calls;
  return cudaSuccess;
}

extern "C" {
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make((void**)e); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make((void**)s); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return --g_live, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return --g_live, cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}

// out: whether the stream exists, objects alive after create() and after
// destroy(), error left behind
void side_with_failure(int call, int* out) {
  g_calls = g_live = 0;
  g_fail = call;
  g_last = cudaSuccess;
  emri::SideStream s;
  s.create();
  out[0] = s.stream != nullptr;
  out[1] = g_live;
  out[3] = (int)cudaGetLastError();
  s.destroy();
  out[2] = g_live;
}
}
