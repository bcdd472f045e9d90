// The end of a stream capture whose launches report their errors through
// cudaGetLastError only (kernel launches, and cooperative launches whose result
// is not looked at one by one).
#pragma once

#include <cuda_runtime_api.h>

namespace ba {

// Ends the capture on s into *g.  A launch that was refused while capturing
// leaves no node: the rest would be a graph that skips it in every replay
// (without the PCG's launch: a step of 0).  So its error, the last one raised
// since the capture began (begin with the last error cleared), fails the
// capture; *g is then NULL.
inline cudaError_t end_capture(cudaStream_t s, cudaGraph_t* g) {
  *g = nullptr;
  const cudaError_t refused = cudaGetLastError();
  const cudaError_t e = cudaStreamEndCapture(s, g);
  if (e == cudaSuccess && refused == cudaSuccess) return cudaSuccess;
  if (*g) cudaGraphDestroy(*g);
  *g = nullptr;
  cudaGetLastError();
  return refused != cudaSuccess ? refused : e;
}

}  // namespace ba
