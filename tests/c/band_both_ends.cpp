// Prints a banded Cholesky's elimination order and task list
// (ba_band_sched.h) for the tests:
//   band_both_ends nb bwt s_upd workers crit_workers
// first line "nb bwt top joint ncrit", second the matrix's block row of each
// position, then one task per line: x y z w and, for U, the updates before it.
#include <cstdio>
#include <cstdlib>

#include "ba_band_sched.h"

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  int ncrit = 0;
  const ba::BandShape sh = ba::band_shape(std::atoi(argv[1]), std::atoi(argv[2]));
  const std::vector<ba::BandTask> t =
      ba::band_tasks(sh, std::atoi(argv[3]), std::atoi(argv[4]), std::atoi(argv[5]), &ncrit);
  std::printf("%d %d %d %d %d\n", sh.nb, sh.bwt, sh.top, sh.joint, ncrit);
  for (int J = 0; J < sh.nb; ++J) {
    if (sh.place_of(sh.row_of(J)) != J) return 3;
    std::printf("%d ", sh.row_of(J));
  }
  std::printf("\n");
  // every tile has a place of its own in its column
  for (int J = 0; J < sh.nb; ++J) {
    std::vector<int> seen(sh.bwt + 1, 0);
    for (int I = J; I < sh.nb; ++I)
      if (std::abs(sh.row_of(I) - sh.row_of(J)) <= sh.bwt) {
        const int k = sh.slot(I, J);
        if (k < 0 || k > sh.bwt || seen[k]++) return 4;
      }
  }
  for (const ba::BandTask& q : t)
    std::printf("%d %d %d %d %d\n", q.x, q.y, q.z, q.w, (q.x & 7) == ba::BAND_U ? sh.updates(q.y, q.z, q.w) : 0);
  return 0;
}
