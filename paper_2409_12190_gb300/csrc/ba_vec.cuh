// The vector work of one PCG iteration on the implicit Schur product in one
// cooperative launch: q = U* p - (pass-B sums), alpha, x, r, z, beta, p, the
// work of k_pcg_q, k_pcg_update and k_pcg_direction with p.q, r.z and r.r
// crossing the grid inside (ba_gridx.cuh) and q and z in registers.  The same
// operations in the same order: the iterates have the same bits.
#pragma once

#include "ba_gridx.cuh"
#include "ba_kernels.cuh"

namespace ba {

template <typename T>
struct VecArgs {
  int C;
  const int32_t* cam_piece_ptr;
  const double* part;
  const double* U;
  const T* camtab;
  const double* lam_ptr;
  double dmin, dmax;
  const double* Minv;
  const uint8_t* fixed;
  double *x, *r, *p;
  T* pT;
  const double *dot_rz, *dot_bb;  // the blocks' r.z and b.b at the start
  double* scal;                   // r.z and b.b from one iteration to the next
  int k;                          // iteration
  double tol;
  GridX gx;
  DevState* st;
};

// Totals over the grid of the blocks' sums v (in every thread), added in
// block_sum_arrays' order; thread 32 i turns total i into v[i] = fin(i, total)
// (the divisions and roots of two totals side by side: one of them is 0.5 us
// of a single warp), the total itself in tot[i].  The slots' polls are spread
// over the block's threads.  Returns false if a wait ran out.
template <int NV, typename Finish>
__device__ __forceinline__ bool vec_totals(const GridX& gx, int set, unsigned int epoch, double (&v)[NV], Finish fin,
                                           double (&tot)[NV]) {
  __shared__ double red[VT / 32][NV];
  __shared__ double s_out[NV], s_tot[NV];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = gridDim.x;
  unsigned long long* base = gx.slots + (size_t)set * GX_COPIES * G * GX_WORDS;
  if (tid < GX_COPIES) {
#pragma unroll
    for (int i = 0; i < NV; ++i) gx_put(base + ((size_t)tid * G + blockIdx.x) * GX_WORDS + 2 * i, epoch, v[i]);
  }
  const unsigned long long* mine = base + (size_t)(blockIdx.x % GX_COPIES) * G * GX_WORDS;
  bool ok = true;
  if (32 * warp < G) {
    double t[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) t[i] = 0.0;
    for (int b = tid; b < G && ok; b += VT) {
      unsigned long long w[2 * NV];
      for (unsigned int spins = 0;; ++spins) {
        bool here = true;
#pragma unroll
        for (int i = 0; i < NV; ++i) gx_load2(mine + (size_t)b * GX_WORDS + 2 * i, w[2 * i], w[2 * i + 1]);
#pragma unroll
        for (int i = 0; i < NV; ++i) here = here && gx_has(w[2 * i], w[2 * i + 1], epoch);
        if (here) break;
        if (gx_give_up(gx, spins)) {
          ok = false;
          break;
        }
      }
#pragma unroll
      for (int i = 0; i < NV; ++i) t[i] += gx_value(w[2 * i], w[2 * i + 1]);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const double s = warp_sum(t[i]);
      if (lane == 0) red[warp][i] = s;
    }
  }
  if (!__syncthreads_and(ok)) return false;
  if (lane == 0 && warp < NV) {
    double t = 0.0;
    for (int w = 0; w < min(VT / 32, (G + 31) / 32); ++w) t += red[w][warp];
    s_tot[warp] = t;
    s_out[warp] = fin(warp, t);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    v[i] = s_out[i];
    tot[i] = s_tot[i];
  }
  return true;
}

// What bounds it: latency (two exchanges of about 2 us, the block sums, and
// the pass-B pieces' sums): 17.7 us for 4,000 cameras, against 27.7 us in the
// three launches (two trials of 30 iterations in FP32: 11.11 -> 10.71 ms).
template <typename T, bool MF>
static __global__ void __launch_bounds__(VT) k_pcg_vectors(VecArgs<T> a) {
  if (a.st->pcg_done) return;
  __shared__ double sp[CAM_THREADS][9], ss[CAM_THREADS][9];
  const int lc = threadIdx.x / 9, i = threadIdx.x % 9;
  const int c = blockIdx.x * CAM_THREADS + lc;
  const bool ok = c < a.C;
  const long long o = 9LL * c + i;
  const int k = a.k;
  const double lam = *a.lam_ptr;
  double rz_old, bb;
  if (k == 0) {
    const double* const srcs[2] = {a.dot_rz, a.dot_bb};
    double s[2];
    block_sum_arrays<2>(srcs, gridDim.x, s);
    rz_old = s[0];
    bb = s[1];
  } else {
    rz_old = a.scal[2 * ((k + 1) & 1)];
    bb = a.scal[2 * ((k + 1) & 1) + 1];
  }
  // everything the exchanges do not bring is loaded before the first of them
  double pv = 0.0, sum = 0.0, rv = 0.0, q = 0.0, xv = 0.0;
  double Urow[9], Mrow[9], Jl0 = 0.0, Jl1 = 0.0, Jl2 = 0.0, Jt0 = 0.0, Jt1 = 0.0, Jt2 = 0.0;
  bool frozen = false;
  if (ok) {
    pv = a.p[o];
    rv = a.r[o];
    xv = a.x[o];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      Urow[j] = a.U[45LL * c + sym9_rt(i, j)];
      Mrow[j] = a.Minv[45LL * c + sym9_rt(i, j)];
    }
    if (MF && i < 3) {
      const T* Jl = a.camtab + (long long)CT * c + CT_JL;
      Jt0 = (double)Jl[i];
      Jt1 = (double)Jl[3 + i];
      Jt2 = (double)Jl[6 + i];
      Jl0 = (double)Jl[3 * i];
      Jl1 = (double)Jl[3 * i + 1];
      Jl2 = (double)Jl[3 * i + 2];
    }
    frozen = a.fixed && a.fixed[o];
    const int p1 = a.cam_piece_ptr[c + 1];
    for (int j = a.cam_piece_ptr[c]; j < p1; ++j) sum += a.part[(long long)PART * j + i];
  }
  sp[lc][i] = pv;
  ss[lc][i] = sum;
  __syncthreads();
  double v1[1] = {0.0};
  if (ok) {
    if (MF && i < 3) sum = Jt0 * ss[lc][0] + Jt1 * ss[lc][1] + Jt2 * ss[lc][2];
    double Uii = Urow[0];
#pragma unroll
    for (int j = 1; j < 9; ++j) Uii = j == i ? Urow[j] : Uii;
    double y = damp(Uii, lam, a.dmin, a.dmax) * sp[lc][i];
#pragma unroll
    for (int j = 0; j < 9; ++j) y += Urow[j] * sp[lc][j];
    y -= sum;
    if (frozen) y = 0.0;
    q = y;
    v1[0] = pv * y;
  }
  block_sum_all<1>(v1);
  // alpha, or NaN: no positive curvature (b = 0 or breakdown) keeps x and stops
  double t1[1];
  bool lost = !vec_totals<1>(
      a.gx, 0, k + 1, v1, [&](int, double t) { return t > 0.0 && isfinite(t) ? rz_old / t : nan(""); }, t1);
  const bool first = blockIdx.x == 0 && threadIdx.x == 0;
  if (!lost) {
    const double alpha = v1[0];
    if (isnan(alpha)) {
      if (first) {
        a.st->pcg_done = 1;
        a.st->pcg_iters = k;
        if (k == 0) a.st->pcg_rel = 0.0;
      }
      return;
    }
    double zz = 0.0;
    if (ok) {
      xv += alpha * pv;
      a.x[o] = xv;
      rv = rv - alpha * q;
      a.r[o] = rv;
    }
    ss[lc][i] = rv;
    __syncthreads();
    if (ok) {
#pragma unroll
      for (int j = 0; j < 9; ++j) zz += Mrow[j] * ss[lc][j];
    }
    double v2[2] = {rv * zz, rv * rv};
    block_sum_all<2>(v2);
    // beta, and whether |r| <= tol |b|
    double t2[2];
    lost = !vec_totals<2>(
        a.gx, 1, k + 1, v2,
        [&](int n, double t) { return n == 0 ? t / rz_old : sqrt(t) <= a.tol * sqrt(bb) ? 1.0 : 0.0; }, t2);
    if (!lost && blockIdx.x == 0 && threadIdx.x == VT - 1) {
      a.scal[2 * (k & 1)] = t2[0];
      a.scal[2 * (k & 1) + 1] = bb;
      a.st->pcg_iters = k + 1;
      a.st->pcg_rel = bb > 0.0 ? sqrt(t2[1] / bb) : 0.0;
      if (v2[1] != 0.0) a.st->pcg_done = 1;
    }
    if (!lost) {
      if (v2[1] != 0.0) return;
      const double beta = v2[0];
      if (ok) {
        pv = zz + beta * pv;
        a.p[o] = pv;
      }
      sp[lc][i] = pv;
      __syncthreads();
      if (!ok) return;
      constexpr int XS = pass_vec_stride(MF);
      T* out = a.pT + (long long)XS * c;
      if (MF && i < 3) {
        out[i] = (T)(Jl0 * sp[lc][0] + Jl1 * sp[lc][1] + Jl2 * sp[lc][2]);
        out[9 + i] = T(0);
      } else {
        out[i] = (T)pv;
      }
      return;
    }
  }
  // a wait ran out: no more iterations (k_cam_trial makes it no step; other
  // blocks may have got through)
  if (threadIdx.x == 0) a.st->pcg_done = 1;
}

}  // namespace ba
