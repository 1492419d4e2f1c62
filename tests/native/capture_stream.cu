// make_capture_stream with a creation that fails: no stream and no pending error.
#include <cstdio>

#include "pibm_internal.cuh"

namespace {
cudaError_t pending = cudaSuccess;
cudaError_t failing_create(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)8;  // what a failing call leaves there is not a stream
  return pending = cudaErrorMemoryAllocation;
}
cudaError_t good_create(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)16;
  return cudaSuccess;
}
cudaError_t take() {
  const cudaError_t e = pending;
  pending = cudaSuccess;
  return e;
}
}  // namespace

int main() {
  cudaStream_t s = nullptr;
  if (pibm::make_capture_stream(&s, failing_create, take) || s || pending != cudaSuccess) {
    printf("an error stays behind a stream that could not be made\n");
    return 1;
  }
  pending = cudaErrorInvalidValue;  // an error of someone else's is not taken
  if (!pibm::make_capture_stream(&s, good_create, take) || s != (cudaStream_t)16 ||
      pending != cudaErrorInvalidValue) {
    printf("a stream that could be made\n");
    return 1;
  }
  return 0;
}
