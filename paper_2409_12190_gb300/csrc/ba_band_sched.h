// Host side of the banded Cholesky (ba_band.cuh): the task list and its
// order.  Plain C++ (no CUDA), so that the schedule can be checked on a
// host: tests/c/band_schedule.cpp prints it, and the tests execute it.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <queue>
#include <utility>
#include <vector>

namespace ba {

// Task types (ba_band.cuh): D the diagonal chain, U an update, T a tile's
// solve, F / B the forward / backward block solves, I a diagonal tile's
// inverse transpose.
enum { BAND_D = 0, BAND_U = 1, BAND_T = 2, BAND_F = 3, BAND_B = 4, BAND_I = 5 };
constexpr int BAND_CRIT_BLOCKS = 4;             // blocks of the near-diagonal pool
constexpr long long BAND_SIM_MAX_TASKS = 2000000;  // longest list that is simulated

#ifdef __CUDACC__
#define BAND_HD __host__ __device__ inline
#else
#define BAND_HD inline
#endif

// The elimination order of the block rows and the tiles it fills.  A band of
// half-bandwidth bwt is eliminated from one end (top = joint = nb), or from
// both ends towards the middle: block rows 0 .. top - 1 are the matrix's
// first ones in order, rows top .. joint - 1 its last ones in reverse, and
// rows joint .. nb - 1 the bwt rows between them, which couple to both ends.
// Each end is a chain of its own (the two meet only in the middle rows), so
// the serial chain of nb diagonal tiles becomes one of about (nb + bwt) / 2;
// the factor has the same number of tiles and operations.  All indices below
// are positions in the elimination order; a column has the tiles of the rows
// at most bwt rows away in the matrix.
struct BandShape {
  int nb;     // block rows
  int bwt;    // half-bandwidth in tiles
  int top;    // block rows eliminated from the top
  int joint;  // first row of the middle

  // the matrix's block row at position J, and the position of block row I
  BAND_HD int row_of(int J) const { return J < top ? J : J < joint ? nb - 1 - (J - top) : top + (J - joint); }
  BAND_HD int place_of(int I) const {
    const int mid = nb - joint;
    return I < top ? I : I < top + mid ? joint + (I - top) : top + (nb - 1 - I);
  }
  // the distance of rows I >= J in the matrix: the tile's place in column J
  BAND_HD int slot(int I, int J) const {
    if (I < joint || J >= joint) return I - J;
    return J < top ? (I - joint) + (top - J) : (nb - 1 - I) + (joint - J);
  }
  BAND_HD long long index(int I, int J) const { return (long long)J * (bwt + 1) + slot(I, J); }
  // the first column of row I among those of the top, or of the rest
  BAND_HD int first_top(int I) const {
    const int k = I < top ? I - bwt : top - bwt + (I - joint);
    return k > 0 ? k : 0;
  }
  BAND_HD int first_rest(int I) const {
    const int k = I < joint ? I - bwt : joint + (nb - 1 - I) - bwt;
    return k > top ? k : top;
  }
  // Tile (I, J) is updated by the columns before J that both rows have:
  // [first(I, J), end of the run), and for J in the middle a second run.
  // (A row further from an end has fewer of its columns.)
  BAND_HD int first(int I, int J) const {
    return J < top || J >= joint ? first_top(I) : first_rest(I);
  }
  BAND_HD int second(int J) const { return first_rest(J); }  // J >= joint: its second run, up to J
  // how many of them come before column K (K one of them, or J)
  BAND_HD int updates(int I, int J, int K) const {
    if (J < joint || K < top) return K - first(I, J);
    return (top - first_top(I)) + (K - second(J));
  }
  // whether column J - 1 has a tile in row J (D_J then solves it)
  BAND_HD bool chained(int J) const { return J >= 1 && bwt >= 1 && J != top; }
  // the chain of position J: 0 top, 1 bottom, 2 middle; its first position, its end
  BAND_HD int chain(int J) const { return J < top ? 0 : J < joint ? 1 : 2; }
  BAND_HD int chain_begin(int c) const { return c == 0 ? 0 : c == 1 ? top : joint; }
  BAND_HD int chain_end(int c) const { return c == 0 ? top : c == 1 ? joint : nb; }
};

// The same for the elimination from the top: what the device code of that
// order is compiled for (the direct solve of 250 cameras took 0.6 % longer
// with the general indices).
struct BandTop {
  int nb, bwt, top, joint;
  BAND_HD int row_of(int J) const { return J; }
  BAND_HD int slot(int I, int J) const { return I - J; }
  BAND_HD long long index(int I, int J) const { return (long long)J * (bwt + 1) + (I - J); }
  BAND_HD int first_top(int I) const { return I > bwt ? I - bwt : 0; }
  BAND_HD int first_rest(int) const { return nb; }
  BAND_HD int updates(int I, int, int K) const { return K - first_top(I); }
  BAND_HD bool chained(int J) const { return J >= 1 && bwt >= 1; }
  BAND_HD int chain(int) const { return 0; }
  BAND_HD int chain_begin(int) const { return 0; }
  BAND_HD int chain_end(int) const { return nb; }
};

// From one end, or from both where that shortens the chain by a third or more
// (nb >= 3 bwt) and the band couples anything.  Two trials of a pose graph,
// one GB300: garage of 1,661 poses (312 block rows) 21.5 -> 11.8 ms, 280 poses
// (48 rows) 3.76 -> 2.34 ms, spheres of 2,500 (469) 32.2 -> 19.3 ms, 360 (68)
// 5.1 -> 3.2 ms, 96 (18) 1.69 -> 1.35 ms.
inline BandShape band_shape(int nb, int bwt) {
  if (bwt < 1 || nb < 3 * bwt || nb < bwt + 2) return BandShape{nb, bwt, nb, nb};
  return BandShape{nb, bwt, (nb - bwt + 1) / 2, nb - bwt};
}

// Columns per update segment: one where the chain of D tasks bounds (33 us a
// step), four where the bulk updates do (12 us a column over `workers`
// blocks): a segment reads and writes its tile and waits for its turn once.
// One trial with S formed, one GB300, segments of 1 / 2 / 4 / 8 columns: 100
// cameras (29 block rows) 2.22 / 2.23 / 2.29 / 2.52 ms, 160 (45 rows) 3.54 /
// 3.39 / 3.52 / 3.99, 250 (71 rows) 7.79 / 7.22 / 6.95 / 6.98, 400 (113 rows)
// 22.7 / 20.4 / 19.3 / 18.9; the line lies at 50 rows of a full triangle.  More
// where the list would pass 4M updates.
inline int band_segment(const BandShape& sh, int workers) {
  const long long updates = (long long)sh.nb * sh.bwt * (sh.bwt + 1) / 2;
  const long long chain = sh.top < sh.nb ? (sh.nb + sh.bwt) / 2 : sh.nb;
  const double tiles = sh.bwt + 1 < sh.nb ? (double)updates : updates / 3.0;  // a triangle's columns get shorter
  const int seg = 12.0 * tiles > 33.0 * (double)chain * workers ? 4 : 1;
  return (int)std::max<long long>(seg, (updates + (4LL << 20) - 1) / (4LL << 20));
}

// One task, as the device reads it (an int4): x = type + 8 count (count:
// U's columns), y = I, z = J, w = Ka (U's first column); for D, I, F:
// y = z = J; for B: y = z = I.
struct BandTask {
  int x, y, z, w;
};

// The banded Cholesky's tasks in ticket order.
//  1. A topological enumeration by step s = 0 .. nb - 1: D_s; I_s; the update
//     segments whose last column is s - 1; the solves T(I, s); F_s; then
//     B_{nb-1} .. B_0.  Each task's predecessors are listed; D_J's
//     subdiagonal tile L_{J,J-1} is published early (after its solve, before
//     the update and factorisation of L_JJ).
//  2. Each task's longest path to the end (its priority), from rough
//     durations in microseconds (D 20, of which 8 before the early output;
//     U 12 per column; T 7; I 8; F and B 4; 1 per dependency).
//  3. A list-scheduling simulation on `workers` blocks: a free block takes
//     the ready task of highest priority.  The tickets follow the simulated
//     start times.  A task starts after its predecessors' outputs, which
//     come after their starts, so the order is topological.
// s_upd: columns per update segment; workers blocks in all, crit_workers
// of them for the near-diagonal pool; *ncrit: that pool's tasks (the list's
// first ones).  A list of more than sim_max tasks is returned in the
// enumeration's order (topological), in one pool (*ncrit = 0).
inline std::vector<BandTask> band_tasks(const BandShape& sh, int s_upd, int workers, int crit_workers, int* ncrit,
                                        long long sim_max = BAND_SIM_MAX_TASKS) {
  const int nb = sh.nb, bwt = sh.bwt;
  const long long ntile = (long long)nb * (bwt + 1);
  // the rows below J in column J, ascending
  auto rows = [&](int J, std::vector<int>& out) {
    out.clear();
    const int end = sh.chain_end(sh.chain(J));
    for (int I = J + 1; I < std::min(end, J + bwt + 1); ++I) out.push_back(I);
    if (J < sh.joint)
      for (int I = sh.joint; I < nb; ++I)
        if (sh.slot(I, J) <= bwt) out.push_back(I);
  };
  // a tile's updates by U tasks, as segments of its one or two runs
  // ((J, J) leaves K = J - 1 to D_J)
  auto segs = [&](int n) { return (std::max(0, n) + s_upd - 1) / s_upd; };
  auto last = [&](int I, int J) { return I == J && sh.chained(J) ? J - 1 : J; };
  auto segs_top = [&](int I, int J) { return J >= sh.joint ? segs(sh.top - sh.first_top(I)) : 0; };
  auto seg_of = [&](int I, int J, int K) {  // the segment of column K
    if (J < sh.joint || K < sh.top) return (K - sh.first(I, J)) / s_upd;
    return segs_top(I, J) + (K - sh.second(J)) / s_upd;
  };
  std::vector<int> col;
  std::vector<long long> seg0(ntile + 1, 0);
  for (int J = 0; J < nb; ++J) {
    rows(J, col);
    col.push_back(J);
    for (int I : col) {
      const int from = J < sh.joint ? sh.first(I, J) : sh.second(J);
      seg0[sh.index(I, J) + 1] = segs_top(I, J) + segs(last(I, J) - from);
    }
  }
  for (long long t = 0; t < ntile; ++t) seg0[t + 1] += seg0[t];
  // a list too long to simulate keeps the enumeration's order, in one pool
  const bool simulate = seg0[ntile] + 6LL * nb <= sim_max;
  if (!simulate) crit_workers = 0;
  std::vector<int> segid(seg0[ntile], -1), idD(nb), idI(nb), idF(nb), idB(nb), idT(ntile, -1);
  std::vector<BandTask> task;
  std::vector<int> dur;
  std::vector<int> pbeg(1, 0), pred;  // predecessors: id * 2 + (1: D's early output)
  auto prod = [&](int I, int K) {
    return I == K ? 2 * idD[K] : (I == K + 1 ? 2 * idD[K + 1] + 1 : 2 * idT[sh.index(I, K)]);
  };
  auto last_seg = [&](int I, int J) {
    const long long t = sh.index(I, J);
    return seg0[t + 1] > seg0[t] ? segid[seg0[t + 1] - 1] : -1;
  };
  auto dep = [&](int p2) {
    if (p2 >= 0 && simulate) pred.push_back(p2);
  };
  auto add = [&](int type, int cnt, int I, int J, int Ka, int d) {
    task.push_back(BandTask{type + 8 * cnt, I, J, Ka});
    dur.push_back(d);
    pbeg.push_back((int)pred.size());
    return (int)task.size() - 1;
  };
  for (int st = 0; st < nb; ++st) {
    if (sh.chained(st)) {
      dep(2 * idD[st - 1]);
      const int a = last_seg(st, st - 1), b = last_seg(st, st);
      if (a >= 0) dep(2 * a);
      if (b >= 0) dep(2 * b);
    }
    idD[st] = add(BAND_D, 0, st, st, 0, 20);
    dep(2 * idD[st]);
    idI[st] = add(BAND_I, 0, st, st, 0, 8);
    if (st >= 1) {
      const int K = st - 1;  // the segments that end with column K
      rows(K, col);
      for (size_t j = 0; j < col.size(); ++j)
        for (size_t i = j; i < col.size(); ++i) {
          const int I = col[i], J = col[j], e = last(I, J);
          if (K >= e) continue;
          const int run = J < sh.joint || K < sh.top ? sh.first(I, J) : sh.second(J);
          const int run_end = J >= sh.joint && K < sh.top ? sh.top : e;
          if ((K - run + 1) % s_upd != 0 && K != run_end - 1) continue;
          const int m = seg_of(I, J, K), Ka = run + (K - run) / s_upd * s_upd;
          if (m >= 1) dep(2 * segid[seg0[sh.index(I, J)] + m - 1]);
          for (int k = Ka; k <= K; ++k) {
            dep(prod(I, k));
            dep(prod(J, k));
          }
          segid[seg0[sh.index(I, J)] + m] = add(BAND_U, st - Ka, I, J, Ka, 12 * (st - Ka));
        }
    }
    rows(st, col);
    for (int I : col) {
      if (I == st + 1) continue;  // D's
      dep(2 * idD[st]);
      const int a = last_seg(I, st);
      if (a >= 0) dep(2 * a);
      idT[sh.index(I, st)] = add(BAND_T, 0, I, st, 0, 7);
    }
    const int c = sh.chain(st);
    if (st > sh.chain_begin(c)) dep(2 * idF[st - 1]);
    else if (c == 2) {
      dep(2 * idF[sh.top - 1]);
      dep(2 * idF[sh.joint - 1]);
    }
    if (c != 1)
      for (int K = sh.first_top(st); K < std::min(st, sh.top); ++K) dep(prod(st, K));
    if (c != 0)
      for (int K = sh.first_rest(st); K < st; ++K) dep(prod(st, K));
    dep(prod(st, st));
    dep(2 * idI[st]);
    idF[st] = add(BAND_F, 0, st, st, 0, 4);
  }
  for (int I = nb - 1; I >= 0; --I) {
    dep(2 * idF[nb - 1]);
    if (I + 1 < sh.chain_end(sh.chain(I))) dep(2 * idB[I + 1]);
    else if (I + 1 < nb) dep(2 * idB[sh.joint]);
    idB[I] = add(BAND_B, 0, I, I, 0, 4);
  }
  const int nt = (int)task.size();
  if (!simulate) {
    *ncrit = 0;
    return task;
  }
  const int lat = 1, early = 8;
  // longest path to the end
  std::vector<int> bl(nt, 0);
  for (int t = nt - 1; t >= 0; --t) {
    bl[t] = std::max(bl[t], dur[t]);
    for (int k = pbeg[t]; k < pbeg[t + 1]; ++k) {
      const int p = pred[k] >> 1;
      bl[p] = std::max(bl[p], ((pred[k] & 1) ? early : dur[p]) + lat + bl[t]);
    }
  }
  // the near-diagonal tasks (the chain D_J and what feeds it: updates that
  // reach a tile at most two block rows below their column, the solves two
  // below the diagonal) form a pool of their own, run by `crit_workers`
  // blocks, so that they never queue behind the bulk updates
  std::vector<int> crit(nt, 0);
  for (int t = 0; t < nt && crit_workers > 0; ++t) {
    const BandTask q = task[t];
    const int type = q.x & 7;
    crit[t] = type == BAND_D || (type == BAND_U && sh.slot(q.y, q.w + (q.x >> 3) - 1) <= 2) ||
              (type == BAND_T && sh.slot(q.y, q.z) <= 2);
  }
  // list scheduling: at each moment the idle blocks of a pool take its ready
  // tasks, highest priority (longest path, then first enumerated) first.  Times
  // are whole numbers: the outputs that fall due are kept in a ring of one bucket
  // a time, as long as the longest task, and what they release is ready `lat`
  // later.
  std::vector<int> sbeg(nt + 1, 0), succ(pred.size()), npred(nt, 0);
  for (int p : pred) ++sbeg[(p >> 1) + 1];
  for (int t = 0; t < nt; ++t) {
    sbeg[t + 1] += sbeg[t];
    npred[t] = pbeg[t + 1] - pbeg[t];
  }
  std::vector<int> sfill(sbeg.begin(), sbeg.end() - 1);
  for (int t = 0; t < nt; ++t)
    for (int k = pbeg[t]; k < pbeg[t + 1]; ++k) succ[sfill[pred[k] >> 1]++] = t * 2 + (pred[k] & 1);
  std::vector<std::vector<int>> ring((size_t)std::max(early, *std::max_element(dur.begin(), dur.end())) + 1);
  std::priority_queue<uint64_t> avail[2];
  auto key = [&](int t) { return ((uint64_t)bl[t] << 32) | (uint32_t)~(uint32_t)t; };
  int idle[2] = {std::max(1, workers - crit_workers), crit_workers};
  std::vector<int> due, soon, first;  // ready now, ready after lat, started now
  for (int t = 0; t < nt; ++t)
    if (npred[t] == 0) due.push_back(t);
  std::vector<int> order[2];  // a pool's tasks by start, then by enumeration
  size_t at = 0;              // the clock's place in the ring
  while ((int)(order[0].size() + order[1].size()) < nt) {
    // outputs due now release their successors; ready tasks join their pool
    for (int code : ring[at]) {
      const int p = code >> 1, early_out = code & 1;
      if (!early_out) ++idle[crit[p]];
      for (int k = sbeg[p]; k < sbeg[p + 1]; ++k)
        if ((succ[k] & 1) == early_out && --npred[succ[k] >> 1] == 0) soon.push_back(succ[k] >> 1);
    }
    ring[at].clear();
    for (int t : due) avail[crit[t]].push(key(t));
    for (int pl = 0; pl < 2; ++pl) {
      first.clear();
      for (; idle[pl] > 0 && !avail[pl].empty(); --idle[pl]) {
        const int t = (int)~(uint32_t)avail[pl].top();
        avail[pl].pop();
        first.push_back(t);
        ring[(at + dur[t]) % ring.size()].push_back(2 * t);
        if ((task[t].x & 7) == BAND_D) ring[(at + early) % ring.size()].push_back(2 * t + 1);
      }
      std::sort(first.begin(), first.end());
      order[pl].insert(order[pl].end(), first.begin(), first.end());
    }
    due.clear();
    due.swap(soon);
    // to the next moment at which something is due
    size_t step = 1;
    while (due.empty() && step < ring.size() && ring[(at + step) % ring.size()].empty()) ++step;
    if (due.empty() && step == ring.size()) break;  // not reached: the enumeration is acyclic
    at = (at + step) % ring.size();
  }
  // tickets: the near-diagonal pool's tasks, then the bulk pool's
  *ncrit = (int)order[1].size();
  std::vector<BandTask> out;
  out.reserve(nt);
  for (int pl = 1; pl >= 0; --pl)
    for (int t : order[pl]) out.push_back(task[t]);
  return out;
}

// The elimination from one end.
inline std::vector<BandTask> band_tasks(int nb, int bwt, int s_upd, int workers, int crit_workers, int* ncrit,
                                        long long sim_max = BAND_SIM_MAX_TASKS) {
  return band_tasks(BandShape{nb, bwt, nb, nb}, s_upd, workers, crit_workers, ncrit, sim_max);
}

}  // namespace ba
