// Grid-wide exchange of per-block sums for cooperative launches: a barrier
// that carries its payload.
//
// Every block publishes its NV sums in a slot of its own, each double as two
// 64-bit words of (epoch << 32 | half), and every block polls every slot
// until it holds the epoch.  A value and its epoch are one word, so nothing
// has to be ordered: no fences, and vectors that go from block to block travel
// the same way (gx_put / gx_get).  It costs one hop, the store of a slot and
// the load that sees it; a counter barrier followed by a read of the blocks'
// sums takes three, and two fences of 1,000 cycles each (measured, clock64).
// Everything is added in a fixed order: every block gets the same bits.
#pragma once

#include <cuda/atomic>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ba_kernels.cuh"
#include "ba_rcp.h"

namespace ba {

constexpr int GX_WORDS = 4;     // 64-bit words of a slot: two doubles in halves
// Copies of the slots, so that the blocks' polls spread over the L2 slices:
// with one copy, 147 blocks polling 147 slots took longer than the counter
// barriers (21.4 us an iteration of k_pgo_pcg_res).
constexpr int GX_COPIES = 8;

// Bytes of the slots of `blocks` blocks: two sets, used in turn.  A block
// writes a set again only after it has seen every block's slot of the other
// set, so after every block has read the earlier epoch of this one.  The
// slots must be zero before the launch (epochs start at 1).
__host__ __device__ constexpr size_t gx_bytes(int blocks) {
  return 2ull * GX_COPIES * (size_t)blocks * GX_WORDS * sizeof(unsigned long long);
}

// Polls before a wait gives up by default (each at least an L2 round trip of
// about 0.7 us: a second or more in all).
constexpr unsigned int GX_SPINS = 1u << 21;

struct GridX {
  unsigned long long* slots;  // gx_bytes(gridDim.x)
  int* err;                   // set by a wait that ran out; every later wait returns
  unsigned int spins;         // polls before a wait gives up
};

// Two 64-bit words at a 16-byte boundary; each word carries its own epoch, so
// only the words have to be single copies.
__device__ __forceinline__ void gx_store2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void gx_load2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// One double of a vector that other blocks read: two tagged words, 16 bytes.
__device__ __forceinline__ void gx_put(unsigned long long* p, unsigned int epoch, double v) {
  const unsigned long long tag = (unsigned long long)epoch << 32;
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  gx_store2(p, tag | (b & 0xffffffffull), tag | (b >> 32));
}
__device__ __forceinline__ bool gx_has(unsigned long long a, unsigned long long b, unsigned int epoch) {
  return (unsigned int)(a >> 32) == epoch && (unsigned int)(b >> 32) == epoch;
}
__device__ __forceinline__ double gx_value(unsigned long long a, unsigned long long b) {
  return __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
}
// Whether a wait of `spins` polls gives up (the caller then stops for good).
__device__ __forceinline__ bool gx_give_up(const GridX& gx, unsigned int spins) {
  const bool out = spins >= gx.spins;
  if (!out && (spins & 63) != 63) return false;
  cuda::atomic_ref<int, cuda::thread_scope_device> err(*gx.err);
  if (!out && !err.load(cuda::memory_order_relaxed)) return false;
  err.store(1, cuda::memory_order_relaxed);
  return true;
}

// dst[e] = the element index(e) of the published vector, e < n, once it holds
// the epoch; threads t of nt call it.  U elements of a thread in flight.
// Returns false if a wait ran out.
template <int U, typename Index>
__device__ __forceinline__ bool gx_gather(const GridX& gx, const unsigned long long* __restrict__ vec,
                                          unsigned int epoch, int n, int t, int nt, Index index, double* dst) {
  for (int e0 = t; e0 < n; e0 += U * nt) {
    unsigned long long a[U], b[U];
    const unsigned long long* src[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * nt;
      src[u] = vec + 2 * (size_t)(e < n ? index(e) : index(e0));
    }
    for (unsigned int spins = 0;; ++spins) {
      bool here = true;
#pragma unroll
      for (int u = 0; u < U; ++u) gx_load2(src[u], a[u], b[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) here = here && gx_has(a[u], b[u], epoch);
      if (here) break;
      if (gx_give_up(gx, spins)) return false;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (e0 + u * nt < n) dst[e0 + u * nt] = gx_value(a[u], b[u]);
  }
  return true;
}

// warp_sum of NV values, the trees interleaved (the shuffles of one keep their
// program order: one tree after the other took twice the latency).
template <int NV>
__device__ __forceinline__ void gx_warp_sums(double (&t)[NV]) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    double s[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] = __shfl_xor_sync(0xffffffffu, t[i], off);
#pragma unroll
    for (int i = 0; i < NV; ++i) t[i] += s[i];
  }
}

// Sums v over the block, then over the grid; the warp that has the totals
// turns them into what the block goes on with, finish(totals), NV numbers that
// every thread of every block returns in v.  (A division or a square root in
// every warp of a block of 16 cost 5 us: 16 cycles for each of their FP64
// instructions and warp.)  It runs prepare() while its sums travel; meanwhile
// the other warps run overlap(), which returns false if it gave up.  Returns false in every thread of the block if
// a wait ran out.  set 0 or 1 alternates between calls, epoch is the call's
// number in its set (1, 2, ...).  blockDim.x is a multiple of 32, at least 64
// and at most NT; only the first nv threads (a multiple of 32) hold values.
// The call begins and ends with a block barrier.
//
// One warp does the adding: an FP64 warp instruction takes 16 cycles of its
// SM here, and a shuffle tree in every warp of every block was a quarter of a
// PCG iteration.
template <int NV, int NT, typename Prepare, typename Finish, typename Overlap>
__device__ __forceinline__ bool grid_exchange(const GridX& gx, int set, unsigned int epoch, double (&v)[NV], int nv,
                                              Prepare prepare, Finish finish, Overlap overlap) {
  static_assert(2 * NV <= GX_WORDS, "a slot holds two doubles");
  __shared__ double s_v[NV][NT];
  __shared__ double s_tot[NV];
  __shared__ int s_fail[2];  // of the polling warp, of the others
  if (threadIdx.x == 32) s_fail[1] = 0;  // (it was 0: a call that failed was the last)
#pragma unroll
  for (int i = 0; i < NV; ++i) s_v[i][threadIdx.x] = v[i];
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const int G = gridDim.x;
    unsigned long long* base = gx.slots + (size_t)set * GX_COPIES * G * GX_WORDS;
    double t[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) t[i] = s_v[i][lane];
    for (int k = 32; k < nv; k += 32)
#pragma unroll
      for (int i = 0; i < NV; ++i) t[i] += s_v[i][lane + k];
    gx_warp_sums(t);
    if (lane < GX_COPIES) {
#pragma unroll
      for (int i = 0; i < NV; ++i)
        gx_put(base + ((size_t)lane * G + blockIdx.x) * GX_WORDS + 2 * i, epoch, t[i]);
    }
    prepare();
    constexpr int U = 5;  // slots of a lane in flight: 160 blocks a round
    const unsigned long long* mine = base + (size_t)(blockIdx.x % GX_COPIES) * G * GX_WORDS;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < NV; ++i) t[i] = 0.0;
    for (int b0 = 0; b0 < G && ok; b0 += 32 * U) {
      unsigned long long w[U][2 * NV];
      for (unsigned int spins = 0;; ++spins) {
        bool here = true;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int b = min(b0 + 32 * u + lane, G - 1);
#pragma unroll
          for (int i = 0; i < NV; ++i) gx_load2(mine + (size_t)b * GX_WORDS + 2 * i, w[u][2 * i], w[u][2 * i + 1]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int i = 0; i < NV; ++i) here = here && gx_has(w[u][2 * i], w[u][2 * i + 1], epoch);
        if (__all_sync(0xffffffffu, here)) break;
        if (__any_sync(0xffffffffu, gx_give_up(gx, spins))) {
          ok = false;
          break;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (b0 + 32 * u + lane < G) t[i] += gx_value(w[u][2 * i], w[u][2 * i + 1]);
    }
    gx_warp_sums(t);
    finish(t);
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (lane == 0) s_tot[i] = t[i];
    if (lane == 0) s_fail[0] = ok ? 0 : 1;
  } else if (!overlap()) {
    s_fail[1] = 1;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = s_tot[i];
  return !(s_fail[0] | s_fail[1]);
}

}  // namespace ba
