// Host side of the explicitly formed reduced camera system (ba_schur.cuh):
// when it pays, its symbolic phase, and the launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "ba.h"
#include "ba_internal.h"
#include "ba_problem.h"
#include "ba_schur.cuh"

namespace ba {

namespace {

#define SCU(call)                                                                                       \
  do {                                                                                                  \
    cudaError_t e_ = (call);                                                                            \
    if (e_ != cudaSuccess)                                                                              \
      return set_error(e_ == cudaErrorMemoryAllocation ? BA_ERR_OOM : BA_ERR_CUDA, "%s failed: %s (%s:%d)", #call, \
                       cudaGetErrorString(e_), __FILE__, __LINE__);                                     \
  } while (0)

inline unsigned nb_(long long n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr long long MAX_PAIRS = 1ll << 27;  // 12 bytes each kept, 36 more while they are sorted

// FP32: formed only where the implicit iteration is mostly launches (20 us of
// which 12 are launches at this size).  Neither time nor accuracy sets this
// line: on 4,000 cameras and 8.0M observations two trials take 10.7 ms with the
// implicit product and 7.8 with S formed, both as far from the FP64 answer
// (cameras 1.2e-6, points 3.1e-5, four seeds), and below it rings of 250-4,000
// cameras with 4.5-8 views a point are as near on either route.  What moves is
// the answer itself: points that three neighbouring views see amplify FP32
// rounding, so that the two routes' are up to 3e-3 apart there, and larger
// problems keep the answers of the implicit product.
constexpr long long F32_MAX_OBS = 1ll << 19;

// The pairs of each point's observations (with the observation itself when
// self): thread per observation q, rank a among its point's, writes pairs
// (a, b), b > a (or >= a), the lower camera first.
__global__ void k_pair_emit(int O, int self, const int32_t* __restrict__ rowptr_pt, const int32_t* __restrict__ poff,
                            const int32_t* __restrict__ pm_pt, const int32_t* __restrict__ pm_cam,
                            const int32_t* __restrict__ pm2cm, int32_t* __restrict__ ki, int32_t* __restrict__ kl,
                            int32_t* __restrict__ sk, int32_t* __restrict__ sl) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= O) return;
  const int j = pm_pt[q], r0 = rowptr_pt[j], n = rowptr_pt[j + 1] - r0;
  const long long a = q - r0;
  // entries before rank a: sum of (n - 1 - a') (or n - a' with self)
  long long w = poff[j] + (self ? a * n - a * (a - 1) / 2 : a * (n - 1) - a * (a - 1) / 2);
  const int ca = pm_cam[q], s = pm2cm[q];
  for (long long p = q + (self ? 0 : 1); p < r0 + n; ++p, ++w) {
    const int cb = pm_cam[p], t = pm2cm[p];
    const bool up = ca <= cb;
    ki[w] = up ? ca : cb;
    kl[w] = up ? cb : ca;
    sk[w] = up ? s : t;
    sl[w] = up ? t : s;
  }
}

__global__ void k_pair_key(int n, const int32_t* __restrict__ perm, const int32_t* __restrict__ key,
                           int32_t* __restrict__ out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) out[e] = key[perm[e]];
}

// Entry e of the sorted order: its slots, point and cameras.
__global__ void k_pair_gather(int n, const int32_t* __restrict__ perm_l, const int32_t* __restrict__ perm_i,
                              const int32_t* __restrict__ ki, const int32_t* __restrict__ kl,
                              const int32_t* __restrict__ sk, const int32_t* __restrict__ sl,
                              const int32_t* __restrict__ cm_pt, int32_t* __restrict__ pk, int32_t* __restrict__ pl,
                              int32_t* __restrict__ pj, int2* __restrict__ cams) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int p = perm_l[perm_i[e]];
  const int s = sk[p];
  pk[e] = s;
  pl[e] = sl[p];
  pj[e] = cm_pt[s];
  cams[e] = make_int2(ki[p], kl[p]);
}

// 0 where a new camera pair begins, else 1 (a stable sort by it lists the heads).
__global__ void k_pair_heads(int n, const int2* __restrict__ cams, int32_t* __restrict__ out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  out[e] = e > 0 && cams[e].x == cams[e - 1].x && cams[e].y == cams[e - 1].y;
}

__global__ void k_pair_head_cams(int n, const int32_t* __restrict__ head, const int2* __restrict__ cams,
                                 int2* __restrict__ out) {
  const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (b < n) out[b] = cams[head[b]];
}

const void* form_kernel(bool direct, bool f32, bool mf) {
  if (direct && f32)
    return mf ? (const void*)k_schur_form<float, true, double> : (const void*)k_schur_form<float, false, double>;
  if (f32) return mf ? (const void*)k_schur_form<float, true, float> : (const void*)k_schur_form<float, false, float>;
  return mf ? (const void*)k_schur_form<double, true, double> : (const void*)k_schur_form_lean;
}

// Whether the PCG on the formed S takes less time than the implicit product
// (us, one GB300; each constant beside what it was measured on).  An LM trial
// at ordinary damping runs 30-80 iterations (rings of 64-4,000 cameras,
// lambda 1e-4 to 2e-3, tol 1e-4), or maxiter: 32 are assumed.  It weighs one
// trial against another.  Set-up is not in it: sorting the pairs takes 0.3 ms for
// 16 cameras, 0.7 for 97 (FP32, 108,000 observations), 0.7 for 250 (480,000),
// which a trial or two earn back (1.7, 0.4 and 4 ms a trial) but a problem made
// for one FP32 trial of a few iterations may not.
struct SchurCost {
  bool f32;
  int maxiter;
  double iters() const { return std::min(maxiter, 32); }
  // five launches and the passes over the observations (8.0M: 1,030 us FP64,
  // 120 us FP32); an iteration past convergence still launches
  double implicit_us(double O) const {
    return iters() * (12.0 + O * (f32 ? 1.5e-5 : 1.28e-4)) + (maxiter - iters()) * 6.0;
  }
  // forming: FP64 pipe (13 ns per 32 pairs), FP32 arithmetic and gathers.  In
  // FP64 both sides are understated, an implicit iteration by the latency of its
  // passes (24 us), forming by the lean form (2e-4 us an observation, in the
  // linearisation and the Schur blocks) and by short tasks (1e-4 a pair); what the
  // second exceeds the first by counts.  Formed over implicit without it, and
  // what it chooses: 2,500 cameras, 2.0M observations, 2.6 pairs each, 8 iterations
  // 1.06 (implicit), 10 0.97 (formed); 5.4 pairs each, 16 1.12 (implicit), 20
  // 1.01 and 30 0.83 (formed); 1,000 cameras, 0.9M, 10 1.05 (implicit), 12
  // 0.97 (formed); 4,000 cameras, 4.7M, 12 1.07 (implicit), 16 0.94 (formed).
  double form_us(double pairs, double O) const {
    const double more = f32 ? 0.0 : std::max(0.0, 2.0e-4 * O + 1.0e-4 * pairs - 24.0 * iters());
    return 25.0 + pairs * (f32 ? 5.0e-5 : 3.1e-4) + more;
  }
  // more pairs than this and forming alone takes longer
  long long most_pairs(double O) const { return (long long)(std::max(0.0, implicit_us(O) - 25.0) / (f32 ? 5.0e-5 : 3.1e-4)); }
  // two exchanges, then 81 multiply-adds or 324 bytes a block
  double iter_us(double blocks) const { return 8.0 + 162.0 * blocks * (f32 ? 0.8e-6 : 1.7e-6); }
};

}  // namespace

SchurPairs::~SchurPairs() { cudaFree(mem); }

void SchurPairs::keep(std::vector<void*>& allocs) {
  allocs.push_back(mem);
  mem = nullptr;
}

ba_status schur_pairs(ba_problem* h, const std::vector<int32_t>& rq, bool self, long long most, SchurPairs& out) {
  const int C = h->C, P = h->P, O = h->O;
  std::vector<int32_t> poff(P + 1);
  long long np = 0;
  for (int j = 0; j < P; ++j) {
    const long long n = rq[j + 1] - rq[j];
    poff[j] = (int32_t)std::min<long long>(np, INT32_MAX);
    np += n * (n - 1) / 2 + (self ? n : 0);
    if (np > std::min(most, MAX_PAIRS)) return BA_OK;
  }
  poff[P] = (int32_t)np;
  if (np == 0) return BA_OK;
  cudaStream_t s = h->s;
  const int n = (int)np;
  // two allocations, what is kept and what is not (each takes some 50 us)
  const size_t scratch_bytes = csr_scratch_bytes(n);
  auto al = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t need = al(4ull * (P + 1)) + 7 * al(4ull * n) + al(4ull * (std::max(C, 2) + 1)) + al(8ull * n) +
                      al(scratch_bytes);
  char* base = nullptr;
  cudaError_t e = cudaMalloc(&base, need);
  if (e == cudaSuccess) e = cudaMalloc(&out.mem, 3 * al(4ull * n));
  struct Free {
    char* p;
    ~Free() { cudaFree(p); }
  } free_base{base};
  if (e != cudaSuccess) {
    cudaGetLastError();  // no room: the implicit product (or the dense build) as before
    return BA_OK;
  }
  out.pk = out.mem;
  out.pl = out.pk + al(4ull * n) / 4;
  out.pj = out.pl + al(4ull * n) / 4;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base + off;
    off += al(bytes);
    return p;
  };
  int32_t* d_poff = (int32_t*)take(4ull * (P + 1));
  int32_t *ki = (int32_t*)take(4ull * n), *kl = (int32_t*)take(4ull * n), *sk = (int32_t*)take(4ull * n),
          *sl = (int32_t*)take(4ull * n), *perm_l = (int32_t*)take(4ull * n), *perm_i = (int32_t*)take(4ull * n),
          *key = (int32_t*)take(4ull * n), *rows = (int32_t*)take(4ull * (std::max(C, 2) + 1));
  int2* cams = (int2*)take(8ull * n);
  void* scratch = take(scratch_bytes);
  int* derr = &h->st->err;
  SCU(cudaMemcpyAsync(d_poff, poff.data(), 4ull * (P + 1), cudaMemcpyHostToDevice, s));
  k_pair_emit<<<nb_(O, 256), 256, 0, s>>>(O, self ? 1 : 0, h->rowptr_pt, d_poff, h->pm_pt, h->pm_cam, h->pm2cm, ki, kl,
                                          sk, sl);
  SCU(csr_build_async(kl, n, C, perm_l, rows, scratch, derr, s));
  k_pair_key<<<nb_(n, 256), 256, 0, s>>>(n, perm_l, ki, key);
  SCU(csr_build_async(key, n, C, perm_i, rows, scratch, derr, s));
  k_pair_gather<<<nb_(n, 256), 256, 0, s>>>(n, perm_l, perm_i, ki, kl, sk, sl, h->cm_pt, out.pk, out.pl, out.pj, cams);
  k_pair_heads<<<nb_(n, 256), 256, 0, s>>>(n, cams, key);
  SCU(csr_build_async(key, n, 2, perm_l, rows, scratch, derr, s));
  count_launch(4);
  int32_t hrow[3];
  SCU(cudaMemcpyAsync(hrow, rows, 12, cudaMemcpyDeviceToHost, s));
  SCU(cudaStreamSynchronize(s));
  const int nhead = hrow[1];
  // the heads' cameras over ki and kl, which are adjacent and done with
  int2* d_hcam = (int2*)ki;
  k_pair_head_cams<<<nb_(nhead, 256), 256, 0, s>>>(nhead, perm_l, cams, d_hcam);
  count_launch();
  out.head.resize(nhead);
  out.cam.resize(nhead);
  SCU(cudaMemcpyAsync(out.head.data(), perm_l, 4ull * nhead, cudaMemcpyDeviceToHost, s));
  SCU(cudaMemcpyAsync(out.cam.data(), d_hcam, 8ull * nhead, cudaMemcpyDeviceToHost, s));
  SCU(cudaStreamSynchronize(s));
  out.n = n;
  return BA_OK;
}

ba_status schur_build(ba_problem* h, const std::vector<int32_t>& rq) {
  const bool direct = h->opt.solver == BA_SOLVER_CHOLESKY;
  const bool f32 = h->prec == BA_PREC_F32;
  if (h->batched || !h->may_form) return BA_OK;
  const int C = h->C, O = h->O;
  const SchurCost cost{f32, h->opt.pcg_maxiter};
  int dev = 0, nsm = 0, coop = 0;
  SCU(cudaGetDevice(&dev));
  SCU(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  SCU(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  int rpb = 1;
  long long most = MAX_PAIRS;
  if (!direct) {
    // FP64 that recomputes its Jacobians in every pass keeps the implicit
    // product: a pair would recompute two observations in FP64
    if (!coop || (!f32 && h->mf) || h->opt.pcg_maxiter < 1) return BA_OK;
    if (f32 && O > F32_MAX_OBS) return BA_OK;
    rpb = (C + nsm - 1) / nsm;
    if (rpb > SX_ROWS) return BA_OK;
    most = cost.most_pairs(O);
  }
  SchurPairs pr;
  const ba_status ps = schur_pairs(h, rq, direct, most, pr);
  if (ps != BA_OK || pr.n == 0) return ps;
  const int n = pr.n, nhead = (int)pr.head.size();
  const long long np = n;
  const std::vector<int32_t>& head = pr.head;
  const std::vector<int2>& hcam = pr.cam;
  auto& x = h->sx;
  cudaStream_t s = h->s;
  cudaError_t e = cudaSuccess;
  const size_t vs = f32 ? 4 : 8;  // the panels' values
  if (!direct && (cost.form_us((double)np, O) + cost.iters() * cost.iter_us(nhead) >= cost.implicit_us(O) ||
                  2ull * nhead * SX_PART * vs > (16ull << 30)))
    return BA_OK;

  // tasks: about eight warps an SM a round and at least four rounds of lanes
  // where there are that many pairs (a task ends with 81 x 32 additions)
  const int seg = (int)std::min<long long>(512, std::max<long long>(32, (np / (8LL * nsm) + 31) / 32 * 32));
  std::vector<int4> task;
  std::vector<int2> bcam;
  std::vector<int> btask;
  auto block = [&](int2 c, int b0, int b1) {
    btask.push_back((int)task.size());
    for (int q = b0; q < b1; q += seg) task.push_back(make_int4((int)bcam.size(), q, std::min(b1, q + seg), 0));
    bcam.push_back(c);
  };
  int next = 0;  // direct: every camera has a diagonal block, observed or not
  for (int b = 0; b < nhead; ++b) {
    if (direct)
      for (; next <= hcam[b].x; ++next)
        if (next < hcam[b].x || hcam[b].y != hcam[b].x) block(make_int2(next, next), 0, 0);
    block(hcam[b], head[b], b + 1 < nhead ? head[b + 1] : n);
  }
  if (direct)
    for (; next < C; ++next) block(make_int2(next, next), 0, 0);
  btask.push_back((int)task.size());
  const int nblk = x.nblk = (int)bcam.size();
  x.ntask = (int)task.size();
  // the lists and buffers of the formed system: one allocation, one copy (a
  // call each was some 0.2 ms of a small problem's set-up of 4-8 ms)
  struct Item {
    void* p;  // the pointer's place
    const void* src;
    size_t bytes;
  };
  std::vector<Item> items;
  auto up = [&](auto** p, const auto& v) { items.push_back({p, v.data(), v.size() * sizeof(v[0])}); };
  auto room = [&](auto** p, size_t bytes) { items.push_back({p, nullptr, bytes}); };
  auto place = [&] {
    if (e != cudaSuccess) return;
    auto al = [](size_t n) { return (n + 255) / 256 * 256; };
    size_t copied = 0, all = 0;
    for (const Item& i : items) {
      copied += i.src ? al(i.bytes) : 0;
      all += al(i.bytes);
    }
    char* base = nullptr;
    e = cudaMalloc(&base, all);
    if (e != cudaSuccess) return;
    h->sx_allocs.push_back(base);
    std::vector<char> host(copied);
    size_t at = 0, free_at = copied;  // the copied ones first
    for (const Item& i : items) {
      size_t& o = i.src ? at : free_at;
      const char* v = base + o;
      std::memcpy(i.p, &v, sizeof v);
      if (i.src) std::copy((const char*)i.src, (const char*)i.src + i.bytes, host.begin() + o);
      o += al(i.bytes);
    }
    e = cudaMemcpy(base, host.data(), copied, cudaMemcpyHostToDevice);
  };
  auto keep = [&] {
    x.pk = pr.pk;
    x.pl = pr.pl;
    x.pj = pr.pj;
    pr.keep(h->sx_allocs);
  };
  auto kernel_attr = [&](const void* k, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  kernel_attr(form_kernel(direct, f32, h->mf), direct || !f32 ? sf_smem<double>() : sf_smem<float>());
  const bool lean = !f32 && !h->mf;
  if (lean) {
    kernel_attr((const void*)k_schur_form_marked, sf_smem<double>());
    x.marked_grid = 2 * nsm;
    room(&x.lean_w, 8ull * NLEAN * O);
    room(&x.lean_t, 8ull * 6 * O);
    room(&x.lean_marked, sizeof(int));
  }
  up(&x.task, task);
  up(&x.blk_cam, bcam);
  up(&x.blk_task, btask);
  room(&x.part, (size_t)x.ntask * SX_PART * 8);
  auto unmark = [&] {
    if (e == cudaSuccess && lean) e = cudaMemsetAsync(x.lean_marked, 0, sizeof(int), s);
  };
  if (direct) {
    place();
    unmark();
    if (e != cudaSuccess) {
      cudaGetLastError();
      schur_drop(h);
      return BA_OK;
    }
    keep();
    x.direct = true;
    x.lean = lean;
    return BA_OK;
  }

  // row panels: neighbours in camera order (blocks come sorted by their lower
  // camera, so every row meets its lower neighbours in order)
  std::vector<int32_t> rowblk(C + 1, 0), lower(C, 0), fill(C, 0);
  for (const int2& c : bcam) {
    ++rowblk[c.x + 1];
    if (c.x != c.y) {
      ++rowblk[c.y + 1];
      ++lower[c.y];
    }
  }
  for (int i = 0; i < C; ++i) rowblk[i + 1] += rowblk[i];
  std::vector<int32_t> col(rowblk[C]), upper(C, 0);
  std::vector<int2> pos(nblk);
  for (int b = 0; b < nblk; ++b) {
    const int i = bcam[b].x, l = bcam[b].y;
    pos[b].x = lower[i] + upper[i]++;
    col[rowblk[i] + pos[b].x] = l;
    pos[b].y = pos[b].x;
    if (i != l) {
      pos[b].y = fill[l]++;
      col[rowblk[l] + pos[b].y] = i;
    }
  }
  const int groups = (C + rpb - 1) / rpb;
  std::vector<int32_t> list, lptr{0}, mark(C, -1), rpart{0}, pptr{0};
  std::vector<uint16_t> colloc(col.size()), ownloc(C);
  std::vector<int4> parts;
  long long wmax = 1;
  for (int g = 0; g < groups; ++g)
    wmax = std::max<long long>(wmax, 9LL * (rowblk[std::min(C, (g + 1) * rpb)] - rowblk[g * rpb]));
  // a warp's share: FP64 adds the lanes of a share at 17 instructions of 16
  // cycles, so few shares, but enough loads in flight (three rows of 900
  // columns: 27.8k cycles a product with 3 shares, 17.9k with 12, of which
  // 14.4k are the multiply-adds); FP32 takes a share for every warp
  const int shares = f32 ? SX_THREADS / 32 : 8;
  const int pcol = (int)std::max<long long>(32, (wmax / shares + 31) / 32 * 32);
  bool fits = true;
  for (int g = 0; g < groups && fits; ++g) {
    const int i0 = g * rpb, i1 = std::min(C, i0 + rpb);
    const size_t l0 = list.size();
    auto local = [&](int c) {
      if (mark[c] < (int)l0 || mark[c] >= (int)list.size() || list[mark[c]] != c) {
        mark[c] = (int)list.size();
        list.push_back(c);
      }
      return mark[c] - (int)l0;
    };
    for (int i = i0; i < i1; ++i) ownloc[i] = (uint16_t)local(i);
    for (int i = i0; i < i1; ++i) {
      for (int q = rowblk[i]; q < rowblk[i + 1]; ++q) colloc[q] = (uint16_t)local(col[q]);
      const int w = 9 * (rowblk[i + 1] - rowblk[i]);
      for (int c = 0; c < w; c += pcol) parts.push_back(make_int4(i - i0, c, std::min(w, c + pcol), 0));
      rpart.push_back((int32_t)parts.size());
    }
    x.nc_max = std::max(x.nc_max, (int)(list.size() - l0));
    x.parts_max = std::max(x.parts_max, (int)parts.size() - pptr.back());
    lptr.push_back((int32_t)list.size());
    pptr.push_back((int32_t)parts.size());
    fits = x.nc_max < 65536 && sx_smem(x.nc_max, x.parts_max) <= 200u * 1024u;
  }
  if (!fits) {
    x = {};
    return BA_OK;
  }
  if (parts.empty()) parts.push_back(make_int4(0, 0, 0, 0));
  const size_t smem = sx_smem(x.nc_max, x.parts_max);
  const void* kern = f32 ? (const void*)k_schur_pcg<float> : (const void*)k_schur_pcg<double>;
  int occ = 0;
  SCU(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  SCU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, SX_THREADS, smem));
  if ((long long)occ * nsm < groups) {
    x = {};
    return BA_OK;
  }
  x.words = sx_words(groups, C) + 1;  // and the error flag
  up(&x.blk_pos, pos);
  up(&x.rowblk, rowblk);
  up(&x.cams, list);
  up(&x.cam_ptr, lptr);
  up(&x.part_ptr, pptr);
  up(&x.row_part, rpart);
  up(&x.colloc, colloc);
  up(&x.ownloc, ownloc);
  up(&x.parts, parts);
  room(&x.val, (size_t)rowblk[C] * SX_PART * vs);
  room(&x.gx, 8 * x.words);
  place();
  unmark();
  if (e == cudaSuccess && !h->Sii) e = h->alloc(&h->Sii, 45ull * C * 8);
  if (e != cudaSuccess) {
    cudaGetLastError();
    schur_drop(h);
    return BA_OK;
  }
  keep();
  x.groups = groups;
  x.rpb = rpb;
  x.pcg = true;
  x.lean = lean;
  return BA_OK;
}

namespace {

template <typename T, bool MF, typename ACC>
void form(ba_problem* h) {
  auto& x = h->sx;
  static_assert(sizeof(ACC) >= sizeof(T), "the sums hold what the Jacobians hold");
  k_schur_form<T, MF, ACC><<<nb_(x.ntask, SF_WARPS), 32 * SF_WARPS, sf_smem<ACC>(), h->s>>>(
      x.ntask, x.task, x.blk_cam, x.pk, x.pl, x.pj, (const T*)h->Jcm, h->O, (const T*)h->camtab, (const T*)h->ptab,
      (const T*)h->cm_sw, (const T*)h->Vinv, (double*)x.part);
  count_launch();
}

template <typename VT>
void pcg(ba_problem* h, int maxiter, double tol) {
  auto& x = h->sx;
  cudaStream_t s = h->s;
  k_schur_combine<VT><<<x.nblk, 96, 0, s>>>(x.blk_cam, x.blk_pos, x.blk_task, x.rowblk, (const double*)x.part,
                                            (VT*)x.val, x.lean ? (const double*)h->camtab : nullptr);
  cudaMemsetAsync(x.gx, 0, 8 * x.words, s);
  SchurPcg<VT> a;
  a.C = h->C;
  a.rpb = x.rpb;
  a.rowblk = x.rowblk;
  a.val = (const VT*)x.val;
  a.colloc = x.colloc;
  a.cams = x.cams;
  a.cam_ptr = x.cam_ptr;
  a.parts = x.parts;
  a.part_ptr = x.part_ptr;
  a.row_part = x.row_part;
  a.ownloc = x.ownloc;
  a.nc_max = x.nc_max;
  a.Sii = h->Sii;
  a.Minv = h->Minv;
  a.b = h->r;
  a.fixed = h->fixed;
  a.x = h->x;
  a.maxiter = maxiter;
  a.tol = tol;
  a.gx = GridX{x.gx, reinterpret_cast<int*>(x.gx + x.words - 1), h->wait_polls};
  a.st = h->st;
  void* args[] = {&a};
  cudaLaunchCooperativeKernel((const void*)k_schur_pcg<VT>, dim3(x.groups), dim3(SX_THREADS), args,
                              sx_smem(x.nc_max, x.parts_max), s);
  count_launch(2);
}

}  // namespace

void schur_drop(ba_problem* h) {
  for (void* v : h->sx_allocs) cudaFree(v);
  h->sx_allocs.clear();
  h->sx = {};
}

void schur_form(ba_problem* h) {
  const bool f32 = h->prec == BA_PREC_F32;
  if (h->sx.lean) {
    auto& x = h->sx;
    const unsigned g = nb_(x.ntask, SF_WARPS);
    k_schur_form_lean<<<g, 32 * SF_WARPS, sf_smem<double>(), h->s>>>(
        x.ntask, x.task, x.pk, x.pl, (const double2*)x.lean_w, (const double2*)x.lean_t, h->O, (double*)x.part);
    k_schur_form_marked<<<std::min(g, (unsigned)x.marked_grid), 32 * SF_WARPS, sf_smem<double>(), h->s>>>(
        x.ntask, x.task, x.pk, x.pl, x.pj, (const double2*)x.lean_w, (const double*)h->Jcm, h->O,
        (const double*)h->Vinv, x.lean_marked, (double*)x.part);
    count_launch(2);
    return;
  }
  if (h->sx.direct) {
    if (f32) h->mf ? form<float, true, double>(h) : form<float, false, double>(h);
    else form<double, true, double>(h);
  } else {
    h->mf ? form<float, true, float>(h) : form<float, false, float>(h);
  }
}

void schur_to_band(ba_problem* h, const double* lam_ptr) {
  auto& x = h->sx;
  k_schur_band<<<x.nblk, 96, 0, h->s>>>(x.blk_cam, x.blk_task, (const double*)x.part, h->U, lam_ptr, h->opt.diag_min,
                                        h->opt.diag_max, h->fixed, h->bwt, h->bT, h->sx.lean ? (const double*)h->camtab : nullptr);
  count_launch();
}

void schur_pcg(ba_problem* h, int maxiter, double tol) {
  if (h->prec == BA_PREC_F32) pcg<float>(h, maxiter, tol);
  else pcg<double>(h, maxiter, tol);
}

}  // namespace ba
