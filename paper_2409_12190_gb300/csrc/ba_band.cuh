// Banded Cholesky of an SPD system A x = b and its two triangular solves in
// one cooperative launch (the paper's sparse direct solver, Sec. IV-C,
// "Sparse Direct Solver (Cholesky Factorization)").  It solves the damped
// pose-graph system H + D (Sec. IV-D), whose band is narrow, and the
// bundle-adjustment reduced camera system S (Eq. 2), whose band is the
// whole lower triangle.
//
// Storage.  In the factored order (for the pose graphs, reverse
// Cuthill-McKee when narrower) the matrix has half-bandwidth bw unknowns, so
// its lower triangle lies in the TB x TB tiles of block rows at most
// bwt = ceil(bw / TB) apart.  Only those tiles are stored.  The block rows
// are eliminated in the order of BandShape (ba_band_sched.h): from the top,
// or from both ends towards the middle; I and J are positions in that order,
// tile (I, J) lies at T + (J (bwt + 1) + slot(I, J)) TB^2, row-major.  The
// matrix is padded to nb TB unknowns with identity rows.  Cholesky keeps the
// fill inside the band, so L takes the same tiles.
//
// Tasks (a dependency graph):
//   D_J     the diagonal chain: L_{J,J-1} = A_{J,J-1} L_{J-1,J-1}^{-T}, then
//           A_JJ -= L_{J,J-1} L_{J,J-1}^T and L_JJ = chol(A_JJ);
//   U       A_IJ -= L_IK L_JK^T for K in [Ka, Ka + cnt): the updates of a
//           tile, in ascending K (tile (J, J) leaves K = J - 1 to D_J);
//   T       L_IJ = A_IJ L_JJ^{-T} for I >= J + 2;
//   I_J     U_J = L_JJ^{-T} (the same solve with A = identity), so that the
//           triangular solves below are products, not serial substitutions;
//   F_J     y_J = U_J^T (b_J - sum_K L_JK y_K);
//   B_I     x_I = U_I (y_I - sum_K L_KI^T x_K).
// A chain D_0, D_1, ... is the critical path (33 us a step; from both ends
// two run at once, and the middle's follows them); one D_J is a triangular
// solve, a symmetric update and a factorisation of single tiles, while the U
// and T tasks of later columns run beside it.  The host orders the tasks by
// a list-scheduling simulation (a topological order) and splits them into two
// pools: the near-diagonal tasks that feed the chain, run by a few blocks of
// their own, and the bulk, run by the rest; each pool's blocks take its tasks
// in order from an atomic ticket.  A task waits only on tasks earlier in the
// simulated order.  The earliest unfinished task of that order has every
// predecessor done; if no block holds it, every block of its pool holds an
// earlier task of the same pool, which is impossible.  So the schedule cannot
// deadlock; every wait is bounded all the same (2^25 polls, about a second or
// more), and one that runs out sets BAND_LOST, after which every block stops.
//
// Each entry of L is a fixed-order sum (K ascending, then the tile's own
// columns), so the result does not depend on the schedule.
#pragma once

#include <cuda/atomic>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ba_band_sched.h"
#include "ba_dense.cuh"

namespace ba {

constexpr int BAND_TB = DB;        // tile size (32)
constexpr int BAND_THREADS = 256;  // threads per block
constexpr int BAND_TRI = BAND_TB * (BAND_TB + 1) / 2;  // entries of a tile's lower triangle

// The launch's arguments; the tasks are ba_band_sched.h's BandTask records,
// read as int4.
template <typename Shape>  // BandShape or BandTop
struct BandArgs {
  Shape sh;       // block rows (nb * TB >= n), half-bandwidth and elimination order
  int n;              // unknowns
  int ntask;          // tasks
  int ncrit;          // the near-diagonal pool's tasks (the first ncrit of the list)
  int ncta_crit;      // blocks 0 .. ncta_crit - 1 run that pool
  const int4* task;   // [ntask] in ticket order, per pool
  double* T;          // band tiles, L on return
  double* rsd;        // [nb TB] 1 / L_cc of every diagonal entry
  double* Ui;         // [nb TB TB] U_J = L_JJ^{-T}, row-major (upper triangular)
  const double* rhs;  // [n] b
  double* y;          // [nb TB] y, then x, in elimination order
  double* sol;        // [n] x
  int* tflag;         // [nb (bwt + 1)] tile final (L)
  int* tprog;         // [nb (bwt + 1)] updates applied to the tile
  int* ctr;           // BAND_CTRS counters
  int* iflag;         // [nb] U_J final
};

// The counters, before iflag.
enum {
  BAND_BULK = 0,   // the bulk pool's ticket
  BAND_FWD = 1,    // forward blocks done of each chain, in its order (3)
  BAND_BWD = 4,    // backward blocks done of each chain (3)
  BAND_LOST = 7,   // a wait ran out
  BAND_NEAR = 8,   // the near-diagonal pool's ticket
  BAND_FAIL = 9,   // a pivot not positive or not finite
  BAND_CTRS = 10
};

// The factorisation's flags: tflag, tprog, counters, iflag.
inline size_t band_flags(const BandShape& sh) {
  return 2 * (size_t)sh.nb * (sh.bwt + 1) + BAND_CTRS + sh.nb;
}

template <typename S>
__device__ __forceinline__ double* band_tile(const BandArgs<S>& a, int I, int J) {
  return a.T + a.sh.index(I, J) * (BAND_TB * BAND_TB);
}

template <typename S>
__device__ __forceinline__ int* band_flag(const BandArgs<S>& a, int I, int J) { return a.tflag + a.sh.index(I, J); }

template <typename S>
__device__ __forceinline__ int* band_prog(const BandArgs<S>& a, int I, int J) { return a.tprog + a.sh.index(I, J); }

// Thread-0 wait until *flag >= v (acquire).  False when the wait ran out or
// another one did (BAND_LOST).
static __device__ __noinline__ bool band_wait(int* flag, int v, int* err) {
  cuda::atomic_ref<int, cuda::thread_scope_device> f(*flag), e(*err);
  unsigned int spins = 0;
  while (f.load(cuda::memory_order_acquire) < v) {
    if (e.load(cuda::memory_order_relaxed) || ++spins > (1u << 25)) {
      e.store(1, cuda::memory_order_relaxed);
      return false;
    }
    if (spins > 64) __nanosleep(64);
  }
  return true;
}

__device__ __forceinline__ int band_load(int* p) {
  cuda::atomic_ref<int, cuda::thread_scope_device> f(*p);
  return f.load(cuda::memory_order_acquire);
}

// Publish v after the block's writes (called by every thread).
__device__ __forceinline__ void band_publish(int* flag, int v) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    cuda::atomic_ref<int, cuda::thread_scope_device> f(*flag);
    f.store(v, cuda::memory_order_release);
  }
}

typedef double BandTile[BAND_TB][BAND_TB + 1];

// Stage a tile (row-major, TB x TB) into shared memory, through L2.
__device__ __forceinline__ void band_stage(BandTile& s, const double* __restrict__ g) {
  for (int e = threadIdx.x; e < BAND_TB * BAND_TB; e += BAND_THREADS) s[e / BAND_TB][e % BAND_TB] = __ldcg(g + e);
}

__device__ __forceinline__ void band_store(double* __restrict__ g, const BandTile& t) {
  for (int e = threadIdx.x; e < BAND_TB * BAND_TB; e += BAND_THREADS) g[e] = t[e / BAND_TB][e % BAND_TB];
}

struct BandSmem {
  BandTile A, B, C;
  double rs[BAND_TB];
  double d[BAND_TB];
  double red[BAND_THREADS / 32][BAND_TB];
  uint16_t tri[BAND_TRI];  // (r << 8) | c of the row-major lower triangle
  int task;
  int bad;
  int ready;
};

// X L^T = A in place (s.A = A on entry, X on return), L = the staged tile
// s.B with 1 / L_cc in s.rs: column by column, x_rc = a_rc / L_cc, then
// a_rc' -= x_rc L_c'c for c' > c (L's column c prescaled by 1 / L_cc; the
// prescaling overwrites s.B).
static __device__ void band_trsm(BandSmem& s) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x, lane = tid % 32, wp = tid / 32;
  for (int e = tid; e < TB * TB; e += BAND_THREADS) {
    const int rr = e / TB, cc = e % TB;
    if (rr > cc) s.B[rr][cc] *= s.rs[cc];
  }
  __syncthreads();
  for (int c = 0; c < TB - 1; ++c) {
    const double x = s.A[lane][c];
    for (int cp = c + 1 + wp; cp < TB; cp += BAND_THREADS / 32) s.A[lane][cp] = fma(-x, s.B[cp][c], s.A[lane][cp]);
    __syncthreads();
  }
  for (int e = tid; e < TB * TB; e += BAND_THREADS) s.A[e / TB][e % TB] *= s.rs[e % TB];
  __syncthreads();
}

// Factor the diagonal tile in s.C (lower triangle) into L, in place, with
// 1 / L_cc in s.rs: right-looking, one barrier per column; the scaling of
// column c is deferred (a_rc' -= a_rc a_c'c / d_c).  Lane 0 of warp 0
// updates each next pivot and takes its reciprocal square root, the serial
// chain of the factorisation; the other entries of the trailing triangle go
// to warps 1-3 and 5-7, so that the chain's FP64 instructions do not queue
// behind theirs (warps w and w + 4 share a scheduler).  A pivot that is not
// positive or not finite is replaced by 1 and counted in s.bad.
static __device__ void band_potrf(BandSmem& s) {
  constexpr int TB = BAND_TB, NU = BAND_THREADS - 64;  // updating threads
  const int tid = threadIdx.x, wp = tid / 32;
  const bool pivot = tid == 0;
  const bool upd = wp % 4 != 0;
  const int u = (wp < 4 ? wp - 1 : wp - 2) * 32 + tid % 32;  // 0 .. NU - 1 for the updating warps
  if (pivot) {
    const double d0 = s.C[0][0];
    const bool ok = d0 > 0.0 && isfinite(d0);
    s.d[0] = ok ? d0 : 1.0;
    s.rs[0] = ok ? rsqrt(d0) : 1.0;
    s.bad = ok ? 0 : 1;
  }
  __syncthreads();
  for (int c = 0; c < TB - 1; ++c) {
    const int m = TB - 1 - c, ne = m * (m + 1) / 2;
    const double inv = s.rs[c] * s.rs[c];
    if (pivot) {  // (c + 1, c + 1): the next pivot
      const double a = s.C[c + 1][c];
      const double v = fma(-(a * inv), a, s.C[c + 1][c + 1]);
      s.C[c + 1][c + 1] = v;
      const bool ok = v > 0.0 && isfinite(v);
      s.d[c + 1] = ok ? v : 1.0;
      s.rs[c + 1] = ok ? rsqrt(v) : 1.0;
      if (!ok) s.bad = 1;
    } else if (upd) {
      for (int e = 1 + u; e < ne; e += NU) {
        const int rr = c + 1 + (s.tri[e] >> 8), cc = c + 1 + (s.tri[e] & 0xff);
        s.C[rr][cc] = fma(-(s.C[rr][c] * inv), s.C[cc][c], s.C[rr][cc]);
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < TB * TB; e += BAND_THREADS) {
    const int rr = e / TB, cc = e % TB;
    s.C[rr][cc] = rr > cc ? s.C[rr][cc] * s.rs[cc] : (rr == cc ? s.d[cc] * s.rs[cc] : 0.0);
  }
  __syncthreads();
}

// D_J: the subdiagonal tile's solve, the last update of the diagonal tile
// and its factorisation.
template <typename S>
static __device__ bool band_task_D(const BandArgs<S>& a, BandSmem& s, int J) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x;
  if (a.sh.chained(J)) {
    // tiles (J, J - 1) and (J, J) hold every update before K = J - 1
    // (the two tiles of row J usually finish first: stage them while
    // L_{J-1,J-1} is still being factored)
    int w = 1;
    if (tid == 0)
      w = band_wait(band_prog(a, J, J - 1), a.sh.updates(J, J - 1, J - 1), a.ctr + BAND_LOST) &&
          band_wait(band_prog(a, J, J), a.sh.updates(J, J, J - 1), a.ctr + BAND_LOST);
    if (!__syncthreads_and(w)) return false;
    band_stage(s.A, band_tile(a, J, J - 1));
    band_stage(s.C, band_tile(a, J, J));
    w = 1;
    if (tid == 0) w = band_wait(band_flag(a, J - 1, J - 1), 1, a.ctr + BAND_LOST);
    if (!__syncthreads_and(w)) return false;
    band_stage(s.B, band_tile(a, J - 1, J - 1));
    if (tid < TB) s.rs[tid] = __ldcg(a.rsd + (long long)(J - 1) * TB + tid);
    __syncthreads();
    band_trsm(s);  // s.A = L_{J,J-1}
    band_store(band_tile(a, J, J - 1), s.A);
    band_publish(band_flag(a, J, J - 1), 1);
    // A_JJ -= L_{J,J-1} L_{J,J-1}^T on the lower triangle
    for (int e = tid; e < BAND_TRI; e += BAND_THREADS) {
      const int r = s.tri[e] >> 8, c = s.tri[e] & 0xff;
      double v = s.C[r][c];
#pragma unroll 8
      for (int k = 0; k < TB; ++k) v = fma(-s.A[r][k], s.A[c][k], v);
      s.C[r][c] = v;
    }
    __syncthreads();
  } else {
    band_stage(s.C, band_tile(a, J, J));
    __syncthreads();
  }
  band_potrf(s);  // s.C = L_JJ
  band_store(band_tile(a, J, J), s.C);
  if (tid < TB) a.rsd[(long long)J * TB + tid] = s.rs[tid];
  if (tid == 0 && s.bad) atomicExch(a.ctr + BAND_FAIL, 1);
  band_publish(band_flag(a, J, J), 1);
  return true;
}

// U: A_IJ -= L_IK L_JK^T for K = Ka .. Ka + cnt - 1, after the tile's
// earlier updates.  A lane each looks at the flags of the first columns: those
// that are final already (most, in the bulk) are not waited for, and their
// tiles are fetched while the column before is multiplied (250 cameras, with
// segments of four columns: 8.31 -> 6.95 ms, 7.63 without the fetching ahead;
// the multiply-adds alone take 8.5 us a tile at the SM's FP64 rate, 3.6 ms).
template <typename S>
static __device__ bool band_task_U(const BandArgs<S>& a, BandSmem& s, int I, int J, int Ka, int cnt) {
  constexpr int TB = BAND_TB, E = TB * TB / BAND_THREADS, RS = BAND_THREADS / TB;
  const int tid = threadIdx.x, col = tid % TB, row0 = tid / TB;
  const int before = a.sh.updates(I, J, Ka);
  int w = 1;
  if (tid < 32) {
    const int j = tid >> 1;
    const bool there = j < cnt && band_load(band_flag(a, tid & 1 ? J : I, Ka + j)) != 0;
    const unsigned int got = __ballot_sync(0xffffffffu, there);
    if (tid == 0) {
      s.ready = got == 0xffffffffu ? 16 : (__ffs(~got) - 1) >> 1;  // leading columns with both tiles final
      w = band_wait(band_prog(a, I, J), before, a.ctr + BAND_LOST);
    }
  }
  if (!__syncthreads_and(w)) return false;
  const int ready = s.ready;
  double* Tij = band_tile(a, I, J);
  double acc[E], fa[E], fb[E];
#pragma unroll
  for (int m = 0; m < E; ++m) acc[m] = __ldcg(Tij + (row0 + m * RS) * TB + col);
  auto fetch = [&](int K) {
    const double *A = band_tile(a, I, K), *B = band_tile(a, J, K);
#pragma unroll
    for (int m = 0; m < E; ++m) fa[m] = __ldcg(A + tid + m * BAND_THREADS);
    if (I != J) {
#pragma unroll
      for (int m = 0; m < E; ++m) fb[m] = __ldcg(B + tid + m * BAND_THREADS);
    }
  };
  for (int k = 0; k < cnt; ++k) {
    if (k >= ready) {
      w = 1;
      if (tid == 0)
        w = band_wait(band_flag(a, I, Ka + k), 1, a.ctr + BAND_LOST) &&
            band_wait(band_flag(a, J, Ka + k), 1, a.ctr + BAND_LOST);
      if (!__syncthreads_and(w)) return false;
    }
    if (k == 0 || k >= ready) fetch(Ka + k);
#pragma unroll
    for (int m = 0; m < E; ++m) s.A[row0 + m * RS][col] = fa[m];
    if (I != J) {
#pragma unroll
      for (int m = 0; m < E; ++m) s.B[row0 + m * RS][col] = fb[m];
    }
    __syncthreads();
    if (k + 1 < min(cnt, ready)) fetch(Ka + k + 1);
    const BandTile& LJ = (I != J) ? s.B : s.A;
#pragma unroll 8
    for (int kk = 0; kk < TB; ++kk) {
      const double b = LJ[col][kk];
#pragma unroll
      for (int m = 0; m < E; ++m) acc[m] = fma(-s.A[row0 + m * RS][kk], b, acc[m]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < E; ++m) Tij[(row0 + m * RS) * TB + col] = acc[m];
  band_publish(band_prog(a, I, J), before + cnt);
  return true;
}

// T: L_IJ = A_IJ L_JJ^{-T} (I >= J + 2) after the tile's updates.
template <typename S>
static __device__ bool band_task_T(const BandArgs<S>& a, BandSmem& s, int I, int J) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x;
  int w = 1;
  if (tid == 0)
    w = band_wait(band_flag(a, J, J), 1, a.ctr + BAND_LOST) && band_wait(band_prog(a, I, J), a.sh.updates(I, J, J), a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  band_stage(s.A, band_tile(a, I, J));
  band_stage(s.B, band_tile(a, J, J));
  if (tid < TB) s.rs[tid] = __ldcg(a.rsd + (long long)J * TB + tid);
  __syncthreads();
  band_trsm(s);
  band_store(band_tile(a, I, J), s.A);
  band_publish(band_flag(a, I, J), 1);
  return true;
}

// I_J: U_J = L_JJ^{-T}, the solution of X L_JJ^T = identity.
template <typename S>
static __device__ bool band_task_I(const BandArgs<S>& a, BandSmem& s, int J) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x;
  int w = 1;
  if (tid == 0) w = band_wait(band_flag(a, J, J), 1, a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  band_stage(s.B, band_tile(a, J, J));
  if (tid < TB) s.rs[tid] = __ldcg(a.rsd + (long long)J * TB + tid);
  for (int e = tid; e < TB * TB; e += BAND_THREADS) s.A[e / TB][e % TB] = (e / TB == e % TB) ? 1.0 : 0.0;
  __syncthreads();
  band_trsm(s);
  band_store(a.Ui + (long long)J * TB * TB, s.A);
  band_publish(a.iflag + J, 1);
  return true;
}

// Thread 0: wait until the counter *p reaches v; *known caches the last value
// read, so a satisfied wait costs no load.
__device__ __forceinline__ bool band_wait_count(int* p, int v, int* known, int* err) {
  if (*known >= v) return true;
  *known = band_load(p);
  if (*known >= v) return true;
  if (!band_wait(p, v, err)) return false;
  *known = v;
  return true;
}

// Forward block F_J: y_J = L_JJ^{-1} (b_J - sum_{K < J} L_JK y_K).
template <typename S>
static __device__ bool band_forward_task(const BandArgs<S>& a, BandSmem& s, int J) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x, r = tid / 8, q = tid % 8;  // row r, columns 4q .. 4q + 3
  int known[3] = {0, 0, 0};                              // forward blocks known done (thread 0)
  double part = 0.0;
  const int cj = a.sh.chain(J);
  // the columns of row J: of the top, then the rest
  int K = cj == 1 ? a.sh.first_rest(J) : a.sh.first_top(J);
  while (K < J) {
    if (cj == 2 && K == a.sh.top) K = a.sh.first_rest(J);
    const int ck = a.sh.chain(K);
    int w = 1;
    if (tid == 0) {
      w = band_wait(band_flag(a, J, K), 1, a.ctr + BAND_LOST);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (w && c == ck)
          w = band_wait_count(a.ctr + BAND_FWD + c, K - a.sh.chain_begin(c) + 1, known + c, a.ctr + BAND_LOST);
    }
    if (!__syncthreads_and(w)) return false;
    const double* L = band_tile(a, J, K) + r * TB + 4 * q;
    const double* yk = a.y + (long long)K * TB + 4 * q;
#pragma unroll
    for (int c = 0; c < 4; ++c) part = fma(__ldcg(L + c), __ldcg(yk + c), part);
    ++K;
  }
  part += __shfl_xor_sync(0xffffffffu, part, 4);
  part += __shfl_xor_sync(0xffffffffu, part, 2);
  part += __shfl_xor_sync(0xffffffffu, part, 1);
  const long long row = (long long)a.sh.row_of(J) * TB + r;
  if (q == 0) s.d[r] = (row < a.n ? a.rhs[row] : 0.0) - part;
  int w = 1;
  if (tid == 0) w = band_wait(a.iflag + J, 1, a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  {
    // y = U_J^T v: lane r, rows c = wp, wp + 8, ... of U_J, summed over the
    // warps in order
    const int lane = tid % 32, wp = tid / 32;
    const double* U = a.Ui + (long long)J * TB * TB;
    double p = 0.0;
#pragma unroll
    for (int m = 0; m < TB / (BAND_THREADS / 32); ++m) {
      const int c = wp + m * (BAND_THREADS / 32);
      p = fma(__ldcg(U + c * TB + lane), s.d[c], p);
    }
    s.red[wp][lane] = p;
    __syncthreads();
    if (tid < 32) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < BAND_THREADS / 32; ++k) v += s.red[k][lane];
      a.y[(long long)J * TB + lane] = v;
    }
  }
  // a chain's blocks are published in order
  const int done = J - a.sh.chain_begin(cj);
  w = 1;
  if (tid == 0) w = band_wait(a.ctr + BAND_FWD + cj, done, a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  band_publish(a.ctr + BAND_FWD + cj, done + 1);
  return true;
}

// Backward block B_I: x_I = L_II^{-T} (y_I - sum_{K > I} L_KI^T x_K); x
// overwrites y.
template <typename S>
static __device__ bool band_backward_task(const BandArgs<S>& a, BandSmem& s, int I) {
  constexpr int TB = BAND_TB;
  const int tid = threadIdx.x, lane = tid % 32, wp = tid / 32;  // x row lane; L rows wp, wp + 8, ...
  int known[3] = {0, 0, 0};                                     // backward blocks known done (thread 0)
  const int ci = a.sh.chain(I), cl = a.sh.chain(a.sh.nb - 1);
  int w = 1;
  // every y final (the last chain's forward blocks come after the others'), so every tile
  if (tid == 0) w = band_wait(a.ctr + BAND_FWD + cl, a.sh.nb - a.sh.chain_begin(cl), a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  double part = 0.0;
  // the rows of column I: of the middle, then of its own chain, descending
  const int end = a.sh.chain_end(ci);
  for (int K = a.sh.nb - 1; K > I; --K) {
    if (K >= end && K < a.sh.joint) K = end - 1;                                    // the other end
    if (K < end && K - I > a.sh.bwt) K = I + a.sh.bwt;
    if (K <= I) break;
    if (a.sh.slot(K, I) > a.sh.bwt) continue;
    const int ck = a.sh.chain(K);
    w = 1;
    if (tid == 0) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (c == ck)
          w = band_wait_count(a.ctr + BAND_BWD + c, a.sh.chain_end(c) - K, known + c, a.ctr + BAND_LOST);
    }
    if (!__syncthreads_and(w)) return false;
    const double* L = band_tile(a, K, I);
    const double* xk = a.y + (long long)K * TB;
#pragma unroll
    for (int m = 0; m < TB / (BAND_THREADS / 32); ++m) {
      const int c = wp + m * (BAND_THREADS / 32);
      part = fma(__ldcg(L + c * TB + lane), __ldcg(xk + c), part);
    }
  }
  s.red[wp][lane] = part;
  __syncthreads();
  if (tid < 32) {
    double v = __ldcg(a.y + (long long)I * TB + lane);
#pragma unroll
    for (int k = 0; k < BAND_THREADS / 32; ++k) v -= s.red[k][lane];
    s.d[lane] = v;
  }
  __syncthreads();
  {
    // x = U_I v: row r of U_I, columns 4q .. 4q + 3, summed over the 8
    // threads of the row
    const int r = tid / 8, q = tid % 8;
    const double* U = a.Ui + (long long)I * TB * TB + r * TB + 4 * q;
    double p = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) p = fma(__ldcg(U + c), s.d[4 * q + c], p);
    p += __shfl_xor_sync(0xffffffffu, p, 4);
    p += __shfl_xor_sync(0xffffffffu, p, 2);
    p += __shfl_xor_sync(0xffffffffu, p, 1);
    const long long row = (long long)a.sh.row_of(I) * TB + r;
    if (q == 0) {
      a.y[(long long)I * TB + r] = p;
      if (row < a.n) a.sol[row] = p;
    }
  }
  w = 1;
  if (tid == 0) w = band_wait(a.ctr + BAND_BWD + ci, end - 1 - I, a.ctr + BAND_LOST);
  if (!__syncthreads_and(w)) return false;
  band_publish(a.ctr + BAND_BWD + ci, end - I);
  return true;
}

// The whole factorisation and both solves; launched cooperatively so that
// every block is resident.
template <typename S>
static __global__ void __launch_bounds__(BAND_THREADS, 1) k_band_chol(BandArgs<S> a) {
  __shared__ BandSmem s;
  for (int e = threadIdx.x; e < BAND_TRI; e += BAND_THREADS) {
    int r = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);  // FP32 guess, corrected below
    while ((r + 1) * (r + 2) / 2 <= e) ++r;
    while (r * (r + 1) / 2 > e) --r;
    s.tri[e] = (uint16_t)((r << 8) | (e - r * (r + 1) / 2));
  }
  const bool near = blockIdx.x < a.ncta_crit;
  const int lim = near ? a.ncrit : a.ntask;
  for (;;) {
    if (threadIdx.x == 0)
      s.task = band_load(a.ctr + BAND_LOST) ? lim
                                           : (near ? 0 : a.ncrit) + atomicAdd(a.ctr + (near ? BAND_NEAR : BAND_BULK), 1);
    __syncthreads();
    const int q = s.task;
    __syncthreads();
    if (q >= lim) break;
    const int4 t = a.task[q];
    bool ok = true;
    switch (t.x & 7) {
      case BAND_D: ok = band_task_D(a, s, t.z); break;
      case BAND_U: ok = band_task_U(a, s, t.y, t.z, t.w, t.x >> 3); break;
      case BAND_T: ok = band_task_T(a, s, t.y, t.z); break;
      case BAND_I: ok = band_task_I(a, s, t.z); break;
      case BAND_F: ok = band_forward_task(a, s, t.z); break;
      default: ok = band_backward_task(a, s, t.z); break;
    }
    if (!ok) break;
  }
}

// Identity rows of the padding (n .. nb TB - 1) on the zeroed tiles.
static __global__ void k_band_pad(int n, BandShape sh, double* __restrict__ T) {
  const int R = n + blockIdx.x * blockDim.x + threadIdx.x;
  if (R >= sh.nb * BAND_TB) return;
  const int J = sh.place_of(R / BAND_TB);
  T[sh.index(J, J) * (BAND_TB * BAND_TB) + (R % BAND_TB) * (BAND_TB + 1)] = 1.0;
}

// After k_band_chol: a failed factorisation (a pivot not positive or not
// finite) or a wait that ran out gives x = 0, counted; the solve's statistics.
static __global__ void k_band_finish(int n, const int* __restrict__ ctr, double* __restrict__ sol, DevState* st) {
  const bool bad = ctr[BAND_FAIL] != 0 || ctr[BAND_LOST] != 0;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (bad && i < n) sol[i] = 0.0;
  if (i == 0) {
    st->pcg_done = 1;
    st->pcg_iters = 0;
    st->pcg_rel = bad ? 1.0 : 0.0;
    if (bad) st->fallbacks += 1;
  }
}

// The factorisation and the solves (a cooperative launch of `blocks` blocks)
// on zeroed flags, then k_band_finish.
inline cudaError_t band_chol(const BandShape& sh, int n, int ntask, int ncrit, int ncta_crit, const int4* task, double* T,
                             double* rsd, double* Ui, const double* rhs, double* y, double* sol, int* flags, int blocks,
                             DevState* st, cudaStream_t s) {
  const size_t ntile = (size_t)sh.nb * (sh.bwt + 1);
  int* ctr = flags + 2 * ntile;
  BandArgs<BandShape> a{sh, n, ntask, ncrit, ncta_crit, task, T, rsd, Ui, rhs, y, sol, flags, flags + ntile, ctr,
                        ctr + BAND_CTRS};
  BandArgs<BandTop> t{{sh.nb, sh.bwt, sh.top, sh.joint}, n, ntask, ncrit, ncta_crit, task, T, rsd, Ui, rhs, y, sol,
                      flags, flags + ntile, ctr, ctr + BAND_CTRS};
  const bool ends = sh.top < sh.nb;
  void* args[] = {ends ? (void*)&a : (void*)&t};
  const void* k = ends ? (const void*)k_band_chol<BandShape> : (const void*)k_band_chol<BandTop>;
  const cudaError_t e = cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(BAND_THREADS), args, 0, s);
  if (e != cudaSuccess) return e;
  k_band_finish<<<(n + 255) / 256, 256, 0, s>>>(n, ctr, sol, st);
  return cudaGetLastError();
}

}  // namespace ba
