// The device-side end of a decode loop: the last kernel of a conditional graph node's body says whether the body runs again.
// (A translation unit of its own: cudaGraphSetConditional needs relocatable device code.)
#include "tw_internal.cuh"

namespace tw {

namespace {
__global__ void loop_cond_kernel(cudaGraphConditionalHandle handle, const int* rows, const int* err, int* iterations, int max_iterations) {
  const int n = *iterations + 1;
  *iterations = n;
  cudaGraphSetConditional(handle, *rows != 0 && *err == 0 && n < max_iterations ? 1u : 0u);
}
}  // namespace

void launch_loop_cond(cudaGraphConditionalHandle handle, const int* rows, const int* err, int* iterations, int max_iterations, cudaStream_t st) {
  loop_cond_kernel<<<1, 1, 0, st>>>(handle, rows, err, iterations, max_iterations);
}

}  // namespace tw
