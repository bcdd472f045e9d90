// The reduced camera system S = U* - W V*^{-1} W^T formed block by block
// (only the camera pairs that share points), and the block-Jacobi PCG on it
// in one cooperative launch.
//
// The implicit product of the PCG passes works through every observation in
// every iteration; S has one 9 x 9 block per pair of cameras that see a common
// point, far fewer numbers.  Forming it costs a pass over the pairs of
// observations of each point, so it pays from a number of iterations on
// (SchurCost in ba_schur.cu).
//
//   pairs      (k, l), k and l observations of one point by cameras i <= l's
//              camera, sorted by (camera of k, camera of l): the entries of
//              block (i, l) are contiguous, in a fixed order
//   tasks      at most `seg` entries of one block, one warp each
//   panels     row i of S: 9 rows of 9 deg(i) columns, its neighbours'
//              columns in camera order; both triangles are stored, so that a
//              product writes nothing but its own rows
//
//   k_schur_form     per task: sum over its pairs of
//                    Jc_k^T (Jp_k V*^{-1} Jp_l^T) Jc_l, one pair a lane, 81
//                    sums a lane, lanes added in a fixed order
//   k_schur_combine  per block: its tasks in order, the sign, both triangles
//   k_schur_band     per block: into the band tiles of the direct solver
//   k_schur_pcg      the whole PCG
//
// Bound: the FP64 pipe for double (157 multiply-adds a pair in the lean form,
// 228 from the planes; a warp instruction takes 16 cycles of its SM), FP32
// arithmetic and the gathers of the points for float.
#pragma once

#include "ba_band.cuh"
#include "ba_gridx.cuh"
#include "ba_kernels.cuh"

namespace ba {

constexpr int SF_WARPS = 4;                  // warps of k_schur_form's blocks
constexpr int SX_THREADS = 512;              // k_schur_pcg
constexpr int SX_ROWS = SX_THREADS / 9;      // rows (cameras) of a block
constexpr int SX_PART = 81;                  // numbers of a task's partial block

// dynamic shared memory of k_schur_form: every lane's 81 sums
template <typename ACC>
constexpr int sf_smem() {
  return SF_WARPS * 32 * SX_PART * (int)sizeof(ACC);
}

// The lanes' 81 sums, four runs of eight lanes, to out (or added to it); nl
// lanes had an entry; red holds 32 x 81.  Float sums are added in float-float.
template <typename ACC, bool ADD>
__device__ __forceinline__ void sf_reduce(const ACC (&acc)[SX_PART], ACC* red, int nl, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < SX_PART; ++i) red[lane * SX_PART + i] = acc[i];
  __syncwarp();
  for (int i = lane; i < SX_PART; i += 32) {
    ACC s[4] = {ACC(0), ACC(0), ACC(0), ACC(0)};
    ACC l[4] = {ACC(0), ACC(0), ACC(0), ACC(0)};  // float: what the additions rounded off
    for (int q = 0; q < nl; q += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q + u < nl) {
          const ACC r = red[(q + u) * SX_PART + i];
          if constexpr (sizeof(ACC) == 4) {
            float e;
            two_sum(s[u], r, s[u], e);
            l[u] += e;
          } else {
            s[u] += r;
          }
        }
    double v;
    if constexpr (sizeof(ACC) == 4) {
      ff_add(s[0], l[0], s[1], l[1]);
      ff_add(s[2], l[2], s[3], l[3]);
      ff_add(s[0], l[0], s[2], l[2]);
      v = (double)s[0] + (double)l[0];
    } else {
      v = (s[0] + s[1]) + (s[2] + s[3]);
    }
    out[i] = ADD ? out[i] + v : v;
  }
}

// One observation's planes: all of them from the factored form (recompute
// mode), or read from memory six at a time, three columns of Jc or Jp, where
// they are used (stored mode: the 81 sums leave few registers).
template <typename T, bool MF>
struct SfObs {
  T pl[MF ? NPLANE : 1];
  const T* J;
  long long O, s;
  __device__ __forceinline__ void open(const T* __restrict__ Jcm, long long O_, int s_, const T* ct, T X0, T X1, T X2,
                                       const T* __restrict__ sw) {
    if constexpr (MF) {
      Fac<T> o;
      fac_obs(ct, X0, X1, X2, sw ? sw[s_] : T(1), o);
      fac_planes(o, ct, pl);
    } else {
      J = Jcm;
      O = O_;
      s = s_;
    }
  }
  // planes 6 grp .. 6 grp + 5: two rows of three (A, B, D, Jp)
  __device__ __forceinline__ void group(int grp, T (&v)[6]) const {
    if constexpr (MF) {
#pragma unroll
      for (int i = 0; i < 6; ++i) v[i] = pl[6 * grp + i];
    } else {
      using V2 = typename Vec2<T>::type;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const V2 w = reinterpret_cast<const V2*>(J)[(3LL * grp + q) * O + s];
        v[2 * q] = w.x;
        v[2 * q + 1] = w.y;
      }
    }
  }
};

template <typename T, bool MF, typename ACC>
static __global__ void __launch_bounds__(32 * SF_WARPS, 2)
k_schur_form(int ntask, const int4* __restrict__ task, const int2* __restrict__ blk_cam,
             const int32_t* __restrict__ pk, const int32_t* __restrict__ pl_, const int32_t* __restrict__ pj,
             const T* __restrict__ Jcm, int O, const T* __restrict__ camtab, const T* __restrict__ ptab,
             const T* __restrict__ cm_sw, const T* __restrict__ Vinv, double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char sf_raw[];
  __shared__ T sct[SF_WARPS][2][CT];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * SF_WARPS + warp;
  if (t >= ntask) return;
  const int4 tk = task[t];  // block, first entry, end, 0
  if (MF) {
    const int2 c = blk_cam[tk.x];
    sct[warp][0][lane] = camtab[(long long)CT * c.x + lane];
    sct[warp][1][lane] = camtab[(long long)CT * c.y + lane];
    __syncwarp();
  }
  ACC acc[SX_PART];
#pragma unroll
  for (int i = 0; i < SX_PART; ++i) acc[i] = ACC(0);
  for (int e = tk.y + lane; e < tk.z; e += 32) {
    const int k = pk[e], l = pl_[e], j = pj[e];
    T X0 = 0, X1 = 0, X2 = 0, pad;
    if (MF) load4(ptab + 8LL * j, X0, X1, X2, pad);
    const T* vi = Vinv + 6LL * j;
    const ACC v00 = (ACC)vi[0], v01 = (ACC)vi[1], v02 = (ACC)vi[2], v11 = (ACC)vi[3], v12 = (ACC)vi[4],
              v22 = (ACC)vi[5];
    SfObs<T, MF> a, b;
    a.open(Jcm, O, k, sct[warp][0], X0, X1, X2, cm_sw);
    b.open(Jcm, O, l, sct[warp][1], X0, X1, X2, cm_sw);
    // K = Jp_k V*^{-1} Jp_l^T; an observation paired with itself counts half
    // (its block is added with its transpose)
    ACC K[4];
    {
      T p[6], q[6];
      a.group(3, p);
      b.group(3, q);
      const ACC half = k == l ? ACC(0.5) : ACC(1);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const ACC p0 = (ACC)p[3 * r], p1 = (ACC)p[3 * r + 1], p2 = (ACC)p[3 * r + 2];
        const ACC t0 = p0 * v00 + p1 * v01 + p2 * v02;
        const ACC t1 = p0 * v01 + p1 * v11 + p2 * v12;
        const ACC t2 = p0 * v02 + p1 * v12 + p2 * v22;
#pragma unroll
        for (int c = 0; c < 2; ++c)
          K[2 * r + c] = half * (t0 * (ACC)q[3 * c] + t1 * (ACC)q[3 * c + 1] + t2 * (ACC)q[3 * c + 2]);
      }
    }
    // Jc = [B | A | D]: planes 1, 0, 2 are its columns 0-2, 3-5, 6-8
    ACC k0[9], k1[9];
#pragma unroll
    for (int grp = 0; grp < 3; ++grp) {
      T v[6];
      a.group(grp, v);
      const int c0 = grp == 0 ? 3 : grp == 1 ? 0 : 6;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        k0[c0 + c] = (ACC)v[c];
        k1[c0 + c] = (ACC)v[3 + c];
      }
    }
#pragma unroll
    for (int grp = 0; grp < 3; ++grp) {
      T v[6];
      b.group(grp, v);
      const int c0 = grp == 0 ? 3 : grp == 1 ? 0 : 6;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const ACC g0 = K[0] * (ACC)v[c] + K[1] * (ACC)v[3 + c];
        const ACC g1 = K[2] * (ACC)v[c] + K[3] * (ACC)v[3 + c];
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[9 * r + c0 + c] = fma(k1[r], g1, fma(k0[r], g0, acc[9 * r + c0 + c]));
      }
    }
  }
  sf_reduce<ACC, false>(acc, reinterpret_cast<ACC*>(sf_raw) + warp * 32 * SX_PART, min(32, tk.z - tk.y),
                        part + (long long)SX_PART * t);
}

// The same sums from the lean form (lean_obs), FP64: Jc' = [I | p] E with
// E = [-[RX]_x | I | e_3 q'^T], so a pair's block is E_k^T N E_l with the 3 x 3
// N = [I | p_k]^T K [I | p_l], K = (M^T Jp V*^{-1})_k (M^T Jp)_l^T: 157
// multiply-adds instead of 228 with the planes, 14 loads of 16 bytes instead
// of 27.  In the cameras' factored coordinates: J_l comes in with the block
// (sf_finish).  Pairs with a marked observation are left to k_schur_form_marked.
// FP64 pipe bound: 39M pairs of a 4,000-camera ring 17.9 -> 13.4 ms (lower bound
// at the measured FMA rate 11.6 ms), 2.9M pairs of 250 cameras 1.46 -> 1.1 ms.
static __global__ void __launch_bounds__(32 * SF_WARPS, 2)
k_schur_form_lean(int ntask, const int4* __restrict__ task, const int32_t* __restrict__ pk,
                  const int32_t* __restrict__ pl_, const double2* __restrict__ W, const double2* __restrict__ TV, int O,
                  double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char sf_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * SF_WARPS + warp;
  if (t >= ntask) return;
  const int4 tk = task[t];
  const long long o = O;
  double acc[SX_PART];
#pragma unroll
  for (int i = 0; i < SX_PART; ++i) acc[i] = 0.0;
  for (int e = tk.y + lane; e < tk.z; e += 32) {
    const int k = pk[e], l = pl_[e];
    const double2 k2 = W[2 * o + k], l2 = W[2 * o + l];  // (p1, q'0)
    if (isnan(k2.y) || isnan(l2.y)) continue;
    double N[9];
    {
      const double half = k == l ? 0.5 : 1.0;
      const double2 t0 = TV[k], t1 = TV[o + k], t2 = TV[2 * o + k];
      const double2 j0 = W[4 * o + l], j1 = W[5 * o + l], j2 = W[6 * o + l];
      const double a0 = half * t0.x, a1 = half * t0.y, a2 = half * t1.x;
      const double b0 = half * t1.y, b1 = half * t2.x, b2 = half * t2.y;
      N[0] = a0 * j0.x + a1 * j0.y + a2 * j1.x;
      N[1] = a0 * j1.y + a1 * j2.x + a2 * j2.y;
      N[3] = b0 * j0.x + b1 * j0.y + b2 * j1.x;
      N[4] = b0 * j1.y + b1 * j2.x + b2 * j2.y;
    }
    const double2 k0 = W[k], k1 = W[o + k], k3 = W[3 * o + k];  // (RX0, RX1) (RX2, p0) .. (q'1, q'2)
    const double2 l0 = W[l], l1 = W[o + l], l3 = W[3 * o + l];
    N[2] = N[0] * l1.y + N[1] * l2.x;
    N[5] = N[3] * l1.y + N[4] * l2.x;
#pragma unroll
    for (int c = 0; c < 3; ++c) N[6 + c] = k1.y * N[c] + k2.x * N[3 + c];
    const double R0 = k0.x, R1 = k0.y, R2 = k1.x;
    // one column of E_l at a time
#pragma unroll
    for (int c = 0; c < 9; ++c) {
      double F[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const double* n = N + 3 * r;
        F[r] = c == 0 ? n[2] * l0.y - n[1] * l1.x
             : c == 1 ? n[0] * l1.x - n[2] * l0.x
             : c == 2 ? n[1] * l0.x - n[0] * l0.y
             : c < 6 ? n[c - 3]
             : n[2] * (c == 6 ? l2.y : c == 7 ? l3.x : l3.y);
      }
      acc[c] = fma(R1, F[2], fma(-R2, F[1], acc[c]));
      acc[9 + c] = fma(R2, F[0], fma(-R0, F[2], acc[9 + c]));
      acc[18 + c] = fma(R0, F[1], fma(-R1, F[0], acc[18 + c]));
      acc[27 + c] += F[0];
      acc[36 + c] += F[1];
      acc[45 + c] += F[2];
      acc[54 + c] = fma(k2.y, F[2], acc[54 + c]);
      acc[63 + c] = fma(k3.x, F[2], acc[63 + c]);
      acc[72 + c] = fma(k3.y, F[2], acc[72 + c]);
    }
  }
  sf_reduce<double, false>(acc, reinterpret_cast<double*>(sf_raw) + warp * 32 * SX_PART, min(32, tk.z - tk.y),
                           part + (long long)SX_PART * t);
}

// The pairs that k_schur_form_lean left out, from the planes, in the same
// coordinates, added to its sums (a grid of two blocks an SM strides over the tasks: it
// returns at once when no observation is marked).
static __global__ void __launch_bounds__(32 * SF_WARPS)
k_schur_form_marked(int ntask, const int4* __restrict__ task, const int32_t* __restrict__ pk,
                    const int32_t* __restrict__ pl_, const int32_t* __restrict__ pj, const double2* __restrict__ W,
                    const double* __restrict__ Jcm, int O, const double* __restrict__ Vinv,
                    const int* __restrict__ marked, double* __restrict__ part) {
  if (!*marked) return;
  extern __shared__ __align__(16) unsigned char sf_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long o = O;
  auto rows = [&](int s, double(&j0)[9], double(&j1)[9], double(&jp)[6]) {
    double pl[NPLANE];
    load_planes(Jcm, o, s, pl);
    jc_rows(pl, j0, j1);
    const double2 r01 = W[s];
    const double R0 = r01.x, R1 = r01.y, R2 = W[o + s].x;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const double* A = pl + 3 * a;
      double* j = a == 0 ? j0 : j1;
      j[0] = R1 * A[2] - R2 * A[1];
      j[1] = R2 * A[0] - R0 * A[2];
      j[2] = R0 * A[1] - R1 * A[0];
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) jp[i] = pl[NPLANE_JC + i];
  };
  for (int t = blockIdx.x * SF_WARPS + warp; t < ntask; t += gridDim.x * SF_WARPS) {
    const int4 tk = task[t];
    double acc[SX_PART];
#pragma unroll
    for (int i = 0; i < SX_PART; ++i) acc[i] = 0.0;
    bool any = false;
    for (int e = tk.y + lane; e < tk.z; e += 32) {
      const int k = pk[e], l = pl_[e];
      if (!isnan(W[2 * o + k].y) && !isnan(W[2 * o + l].y)) continue;
      any = true;
      const double* vi = Vinv + 6LL * pj[e];
      double k0[9], k1[9], l0[9], l1[9], jk[6], jl[6], K[4];
      rows(k, k0, k1, jk);
      rows(l, l0, l1, jl);
      const double half = k == l ? 0.5 : 1.0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const double* p = jk + 3 * r;
        const double t0 = p[0] * vi[0] + p[1] * vi[1] + p[2] * vi[2];
        const double t1 = p[0] * vi[1] + p[1] * vi[3] + p[2] * vi[4];
        const double t2 = p[0] * vi[2] + p[1] * vi[4] + p[2] * vi[5];
#pragma unroll
        for (int c = 0; c < 2; ++c) K[2 * r + c] = half * (t0 * jl[3 * c] + t1 * jl[3 * c + 1] + t2 * jl[3 * c + 2]);
      }
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        const double g0 = K[0] * l0[c] + K[1] * l1[c], g1 = K[2] * l0[c] + K[3] * l1[c];
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[9 * r + c] += k0[r] * g0 + k1[r] * g1;
      }
    }
    if (__any_sync(0xffffffffu, any))
      sf_reduce<double, true>(acc, reinterpret_cast<double*>(sf_raw) + warp * 32 * SX_PART, min(32, tk.z - tk.y),
                              part + (long long)SX_PART * t);
    __syncwarp();
  }
}

// A block's 81 sums (in sv, row of its first camera, column of its second)
// from factored to plain coordinates: rows 0-2 by J_l^T of the first camera,
// columns 0-2 by J_l of the second.  96 threads, all of them.
__device__ __forceinline__ void sf_finish(double* sv, int e, const double* __restrict__ ct_i,
                                          const double* __restrict__ ct_l) {
  const int r = e / 9, q = e % 9;
  double v = 0.0;
  if (e < 27)
    for (int m = 0; m < 3; ++m) v += ct_i[CT_JL + 3 * m + r] * sv[9 * m + q];
  __syncthreads();
  if (e < 27) sv[e] = v;
  __syncthreads();
  const int r2 = e / 3, q2 = e % 3;
  v = 0.0;
  if (e < 27)
    for (int m = 0; m < 3; ++m) v += sv[9 * r2 + m] * ct_l[CT_JL + 3 * m + q2];
  __syncthreads();
  if (e < 27) sv[9 * r2 + q2] = v;
  __syncthreads();
}

// Block b of S from its tasks' partial sums, negated, into the row panels of
// both of its cameras.  blk_pos: its position in row i and in row l; a block
// of a camera with itself (a point observed twice by it) is added with its
// transpose.  camtab: the sums are in factored coordinates (the lean form).
template <typename VT>
static __global__ void __launch_bounds__(96)
k_schur_combine(const int2* __restrict__ blk_cam, const int2* __restrict__ blk_pos, const int* __restrict__ blk_task,
                const int32_t* __restrict__ rowblk, const double* __restrict__ part, VT* __restrict__ val,
                const double* __restrict__ camtab) {
  __shared__ double sv[SX_PART];
  const int b = blockIdx.x, e = threadIdx.x;
  const int2 c = blk_cam[b], pos = blk_pos[b];
  if (e < SX_PART) {
    double s = 0.0;
    for (int t = blk_task[b]; t < blk_task[b + 1]; ++t) s += part[(long long)SX_PART * t + e];
    sv[e] = s;
  }
  __syncthreads();
  if (camtab) sf_finish(sv, e, camtab + (long long)CT * c.x, camtab + (long long)CT * c.y);
  if (e >= SX_PART) return;
  const double v = sv[e];
  const int r = e / 9, q = e % 9;
  const long long bi = rowblk[c.x], bl = rowblk[c.y];
  const int wi = 9 * (rowblk[c.x + 1] - (int)bi), wl = 9 * (rowblk[c.y + 1] - (int)bl);
  if (c.x == c.y) {
    val[81 * bi + (long long)r * wi + 9 * pos.x + q] = (VT)(-(v + sv[9 * q + r]));
    return;
  }
  val[81 * bi + (long long)r * wi + 9 * pos.x + q] = (VT)(-v);
  val[81 * bl + (long long)r * wl + 9 * pos.y + q] = (VT)(-sv[9 * q + r]);  // transposed, coalesced
}

// The same block into the band tiles of the direct solver (lower triangle,
// tile (I, J) at (J (bwt + 1) + I - J) TB^2); the diagonal blocks (every
// camera has one, its observations paired with themselves) get U* added; rows
// and columns of frozen parameters become the identity's.
static __global__ void __launch_bounds__(96)
k_schur_band(const int2* __restrict__ blk_cam, const int* __restrict__ blk_task, const double* __restrict__ part,
             const double* __restrict__ U, const double* __restrict__ lam_ptr, double dmin, double dmax,
             const uint8_t* __restrict__ fixed, int bwt, double* __restrict__ T, const double* __restrict__ camtab) {
  __shared__ double sv[SX_PART];
  const int b = blockIdx.x, e = threadIdx.x;
  const int2 c = blk_cam[b];
  if (e < SX_PART) {
    double v = 0.0;
    for (int t = blk_task[b]; t < blk_task[b + 1]; ++t) v += part[(long long)SX_PART * t + e];
    sv[e] = v;
  }
  __syncthreads();
  if (camtab) sf_finish(sv, e, camtab + (long long)CT * c.x, camtab + (long long)CT * c.y);
  if (e >= SX_PART) return;
  const int r = e / 9, q = e % 9;  // row of camera c.y, column of camera c.x
  const int R = 9 * c.y + r, C = 9 * c.x + q;
  if (C > R) return;
  double v = -sv[9 * q + r];
  if (c.x == c.y) {
    double u = U[45LL * c.x + sym9_rt(r, q)];
    if (r == q) u += damp(u, *lam_ptr, dmin, dmax);
    v += u - sv[9 * r + q];
  }
  if (fixed && (fixed[R] || fixed[C])) v = R == C ? 1.0 : 0.0;
  const int I = R / BAND_TB, J = C / BAND_TB;
  T[((long long)J * (bwt + 1) + (I - J)) * (BAND_TB * BAND_TB) + (R % BAND_TB) * BAND_TB + C % BAND_TB] = v;
}

template <typename VT>
struct SchurPcg {
  int C, rpb;                // cameras, cameras a block
  const int32_t* rowblk;     // [C + 1] first neighbour of each row
  const VT* val;             // the panels: row i at 81 rowblk[i], 9 x 9 deg(i)
  const uint16_t* colloc;    // neighbour -> position in its block's camera list
  const int32_t* cams;       // the blocks' camera lists (their own cameras and their neighbours)
  const int32_t* cam_ptr;    // [blocks + 1]
  const int4* parts;         // (row in block, first column, end, 0): a warp's share of a product
  const int32_t* part_ptr;   // [blocks + 1]
  const int32_t* row_part;   // [C + 1] first part of each row
  const uint16_t* ownloc;    // [C] a camera's position in its own block's list
  int nc_max;                // longest camera list
  const double* Sii;         // [C][45]
  const double* Minv;        // [C][45]
  const double* b;           // [C][9] right-hand side
  const uint8_t* fixed;
  double* x;
  int maxiter;
  double tol;
  GridX gx;                  // slots, then 9C tagged doubles (z)
  DevState* st;
};

constexpr size_t sx_smem(int nc_max, int parts_max) {
  return (18ull * (size_t)nc_max + 9ull * (size_t)parts_max) * sizeof(double);
}
__host__ __device__ constexpr size_t sx_words(int blocks, int C) { return gx_bytes(blocks) / 8 + 18 * (size_t)C; }

// Warp totals of nine values: a reduce-scatter over 16 (the rest zero), lane
// 2 i or 2 i + 1 returns value i: 16 additions instead of 45.
template <int N, int OFF>
__device__ __forceinline__ void sx_rs_step(double (&h)[16], int lane) {
  const bool up = (lane & OFF) != 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double k = up ? h[N + i] : h[i];
    const double g = up ? h[i] : h[N + i];
    h[i] = k + __shfl_xor_sync(0xffffffffu, g, OFF);
  }
}
__device__ __forceinline__ double sx_warp_rs9(const double (&v)[9], int lane) {
  double h[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) h[i] = i < 9 ? v[i] : 0.0;
  sx_rs_step<8, 16>(h, lane);
  sx_rs_step<4, 8>(h, lane);
  sx_rs_step<2, 4>(h, lane);
  sx_rs_step<1, 2>(h, lane);
  return h[0] + __shfl_xor_sync(0xffffffffu, h[0], 1);
}
// the same of floats, with what the additions round off
__device__ __forceinline__ double sx_warp_rs9(const float (&v)[9], int lane) {
  float h[8], l[8];
  const bool up = (lane & 16) != 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float lo = v[i], hi = i == 0 ? v[8] : 0.f;
    two_sum(up ? hi : lo, __shfl_xor_sync(0xffffffffu, up ? lo : hi, 16), h[i], l[i]);
  }
  rs_pair_step<4, 8>(h, l, lane);
  rs_pair_step<2, 4>(h, l, lane);
  rs_pair_step<1, 2>(h, l, lane);
  const float gh = __shfl_xor_sync(0xffffffffu, h[0], 1), gl = __shfl_xor_sync(0xffffffffu, l[0], 1);
  float s, e;
  two_sum(h[0], gh, s, e);
  return (double)s + (double)((l[0] + gl) + e);
}

// Block-Jacobi PCG on S x = b from x = 0, the iteration of the per-launch
// kernels (k_pcg_q, k_pcg_update, k_pcg_direction): stop after the first
// iteration with |r| <= tol |b|, after maxiter, or before updating x when
// p^T S p is not positive and finite.  A block owns rpb consecutive cameras,
// thread (camera, component) its entries of x, r, z, p and its rows of the
// diagonal blocks and of M in registers; the directions of every camera the
// block's rows touch stay in shared memory (p = z + beta p is formed where it
// is needed), so only z and two sums an iteration cross the grid.
// S p: a warp takes a part of a row panel, a lane a column (nine rows), the
// panel streamed from L2 or HBM. Lanes add their columns in VT,
// what is added across lanes (and across the lanes of k_schur_form) keeps its
// rounding errors: with plain FP32 sums there the cameras of small problems (6-60
// cameras on an arc, 24 drawn) were 1.23 times the implicit product's distance
// from the 64-bit answer, now 0.90 times (rings of 24-1,200: 1.01 and 0.97).
// What bounds it: for small problems the two exchanges (about 2.3 us each);
// for large ones the FP64 pipe (double: 81 multiply-adds a block) or the
// panel's bytes (float).
template <typename VT>
static __global__ void __launch_bounds__(SX_THREADS, 1) k_schur_pcg(SchurPcg<VT> a) {
  extern __shared__ __align__(16) unsigned char sx_raw[];
  __shared__ double sr[SX_ROWS * 9];
  const int g = blockIdx.x;
  const int c0 = g * a.rpb, nr = min(a.rpb, a.C - c0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  const int lr = tid / 9, row = tid % 9;
  const bool live = lr < nr;
  const int cam = c0 + lr;
  const long long o = 9LL * cam + row;
  const int l0 = a.cam_ptr[g], nc = a.cam_ptr[g + 1] - l0;
  double* sp = reinterpret_cast<double*>(sx_raw);  // [nc][9] directions
  double* sz = sp + 9 * a.nc_max;                  // [nc][9] z of the same cameras
  double* spart = sz + 9 * a.nc_max;               // [parts][9]
  const int q0 = a.part_ptr[g], nq = a.part_ptr[g + 1] - q0;
  unsigned long long* zx = a.gx.slots + gx_bytes(gridDim.x) / 8;
  double Mrow[9], Srow[9];
  double ra = 0.0, xa = 0.0, za = 0.0, pa = 0.0;
  int own = 0, p0 = 0, p1 = 0;
  bool free_row = false;
  if (live) {
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      Mrow[j] = a.Minv[45LL * cam + sym9_rt(row, j)];
      Srow[j] = a.Sii[45LL * cam + sym9_rt(row, j)];
    }
    ra = a.b[o];
    sr[tid] = ra;
    own = 9 * a.ownloc[cam];
    p0 = a.row_part[cam] - q0;
    p1 = a.row_part[cam + 1] - q0;
    free_row = !(a.fixed && a.fixed[o]);
  }
  for (int e = tid; e < 9 * nc; e += blockDim.x) sp[e] = 0.0;
  __syncthreads();
  auto fetch_z = [&](unsigned int epoch) {
    return gx_gather<4>(a.gx, zx, epoch, 9 * nc, tid - 32, blockDim.x - 32,
                        [&](int e) { return 9 * __ldg(a.cams + l0 + e / 9) + e % 9; }, sz);
  };
  // row . 9 values, in three chains (a chain of nine FP64 multiply-adds is
  // some 400 cycles)
  auto dot9 = [](const double(&m)[9], const double* v) {
    double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 9; ++j) s[j % 3] += m[j] * v[j];
    return (s[0] + s[1]) + s[2];
  };
  const int nv = (9 * nr + 31) & ~31;  // threads that hold a component
  double v2[2] = {0.0, 0.0};
  if (live) {
    za = dot9(Mrow, sr + 9 * lr);
    gx_put(zx + 2 * o, 1, za);
    v2[0] = za * ra;
    v2[1] = ra * ra;
  }
  bool lost = !grid_exchange<2, SX_THREADS>(a.gx, 1, 1, v2, nv, [] {}, [](double(&)[2]) {}, [&] { return fetch_z(1); });
  // the polling warp keeps r . z and the last |r|^2; |b|^2 and the bound of |r|^2
  double rz = v2[0], rr = 0.0;
  const double bb = v2[1];
  const double stop = warp == 0 ? a.tol * a.tol * bb : 0.0;
  double inv_rz = 0.0;
  double beta = 0.0;
  int it = 0, done = 0;
  while (!lost && it < a.maxiter) {
    for (int e = tid; e < 9 * nc; e += blockDim.x) sp[e] = sz[e] + beta * sp[e];
    pa = za + beta * pa;
    __syncthreads();
    for (int q = warp; q < nq; q += nw) {
      const int4 pt = __ldg(a.parts + q0 + q);
      const int i = c0 + pt.x;
      const int rb = __ldg(a.rowblk + i), w = 9 * (__ldg(a.rowblk + i + 1) - rb);
      const VT* pv = a.val + 81LL * rb;
      VT acc[9];
#pragma unroll
      for (int r = 0; r < 9; ++r) acc[r] = VT(0);
#pragma unroll 2
      for (int c = pt.y + lane; c < pt.z; c += 32) {
        const int nb = c / 9;
        const VT p = (VT)sp[9 * __ldg(a.colloc + rb + nb) + (c - 9 * nb)];
#pragma unroll
        for (int r = 0; r < 9; ++r) acc[r] += __ldg(pv + (long long)r * w + c) * p;
      }
      const double s = sx_warp_rs9(acc, lane);
      if (!(lane & 1) && lane < 18) spart[9 * q + (lane >> 1)] = s;
    }
    __syncthreads();
    double qa = 0.0;
    if (live && free_row) {
      qa = dot9(Srow, sp + own);
      for (int q = p0; q < p1; ++q) qa += spart[9 * q + row];
    }
    double v1[1] = {live ? pa * qa : 0.0};
    // alpha = r . z / p . S p, or NaN to stop: no positive curvature (b = 0 or
    // breakdown) keeps x
    if (!grid_exchange<1, SX_THREADS>(
            a.gx, 0, it + 1, v1, nv, [&] { inv_rz = gx_rcp(rz); },
            [&](double(&t)[1]) { t[0] = t[0] > 0.0 && isfinite(t[0]) ? rz * gx_rcp(t[0]) : nan(""); },
            [] { return true; })) {
      lost = true;
      break;
    }
    const double alpha = v1[0];
    if (isnan(alpha)) {
      done = 1;
      break;
    }
    v2[0] = v2[1] = 0.0;
    if (live) {
      xa += alpha * pa;
      ra -= alpha * qa;
      sr[tid] = ra;
    }
    __syncthreads();
    if (live) {
      za = dot9(Mrow, sr + 9 * lr);
      gx_put(zx + 2 * o, it + 2, za);
      v2[0] = za * ra;
      v2[1] = ra * ra;
    }
    ++it;
    // beta and whether |r| <= tol |b|
    if (!grid_exchange<2, SX_THREADS>(
            a.gx, 1, it + 1, v2, nv, [] {},
            [&](double(&t)[2]) {
              rz = t[0];
              rr = t[1];
              t[0] = rz * inv_rz;
              t[1] = rr <= stop ? 1.0 : 0.0;
            },
            [&] { return fetch_z(it + 1); })) {
      lost = true;
      break;
    }
    beta = v2[0];
    if (v2[1] != 0.0) {
      done = 1;
      break;
    }
  }
  // after a wait that ran out k_cam_trial makes it no step (each block knows
  // only of its own waits, and some may have got through)
  if (live) a.x[o] = xa;
  if (g == 0 && tid == 0) {
    a.st->pcg_iters = it;
    a.st->pcg_rel = it > 0 ? (bb > 0.0 ? sqrt(rr / bb) : 0.0) : done ? 0.0 : 1.0;
    a.st->pcg_done = done;
  }
}

}  // namespace ba
