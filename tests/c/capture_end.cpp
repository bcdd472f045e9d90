// end_capture (csrc/ba_capture.h) on fakes of the runtime's calls: argv[1] is
// the error of a launch during the capture, argv[2] that of the capture's end.
// Prints the result, whether the caller is left with a graph, and how many
// graphs were destroyed.
#include <cstdio>
#include <cstdlib>

#include "ba_capture.h"

static cudaError_t last_error, end_error;
static int destroyed;

extern "C" {
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  if (end_error == cudaSuccess) *g = reinterpret_cast<cudaGraph_t>(&destroyed);
  else last_error = end_error;
  return end_error;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) {
  ++destroyed;
  return cudaSuccess;
}
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  last_error = (cudaError_t)std::atoi(argv[1]);
  end_error = (cudaError_t)std::atoi(argv[2]);
  cudaGraph_t g = reinterpret_cast<cudaGraph_t>(&end_error);
  const cudaError_t e = ba::end_capture(nullptr, &g);
  std::printf("%d %d %d %d\n", (int)e, g != nullptr, destroyed, (int)last_error);
  return 0;
}
