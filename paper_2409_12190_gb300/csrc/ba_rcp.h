// 1 / d in few FP64 instructions, for the PCG's scalars; also built by the host
// compiler for its test.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define BA_RCP_HD __host__ __device__ __forceinline__
#else
#define BA_RCP_HD inline
#endif

namespace ba {

BA_RCP_HD int rcp_hi(double d) {
#ifdef __CUDA_ARCH__
  return __double2hiint(d);
#else
  uint64_t b;
  memcpy(&b, &d, 8);
  return (int)(int32_t)(uint32_t)(b >> 32);
#endif
}
BA_RCP_HD int rcp_lo(double d) {
#ifdef __CUDA_ARCH__
  return __double2loint(d);
#else
  uint64_t b;
  memcpy(&b, &d, 8);
  return (int)(int32_t)(uint32_t)b;
#endif
}
BA_RCP_HD double rcp_make(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const uint64_t b = (uint64_t)(uint32_t)hi << 32 | (uint32_t)lo;
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// 1 / d: for a positive normal d well inside the range one step of the
// hyperpower (Schulz) iteration of order three, y (1 + r + r^2) with
// r = 1 - m y, on the FP32 reciprocal of d's significand (error 2^-23 -> below
// 2^-68, so the result is the rounding of it: within 0.51 ulp), scaled and
// checked on the integer side; else the division.  A warp issues an FP64
// instruction in some 70 cycles; the division's were on the PCG's critical path
// twice an iteration (with 1 / rz taken while the sums travel and no square root
// in the stopping test: sphere of 2,500 poses 2,514 -> 2,371 us, ring of 97
// cameras in FP32 757 -> 727 us).
BA_RCP_HD double gx_rcp(double d) {
  const int hi = rcp_hi(d), ex = hi >> 20;
  if (ex < 23 || ex > 2023) return 1.0 / d;
  const int up = (ex - 1023) * (1 << 20);
  const double m = rcp_make(hi - up, rcp_lo(d));
  const double y = (double)(1.0f / (float)m);
  const double r = fma(-m, y, 1.0);
  const double z = fma(y, fma(r, r, r), y);  // in (1/2, 1]
  return rcp_make(rcp_hi(z) - up, rcp_lo(z));
}

}  // namespace ba
