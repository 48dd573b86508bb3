// Uniform faces and the lists of the other midpoints, for N = 2..3 species and
// D = 1..3 dimensions (see hrm_sweep.cuh). Built without FMA contraction.
#include "hrm_sweep.cuh"

namespace hrm {

namespace {
template <int N, int D>
void mark64(const double* W, const double* V, const DevGrid& g, const SweepLists& lists, int all, cudaStream_t s) {
  const unsigned gr = grid_for(g.nint, kCellThreads);
  k_equal<N, D><<<gr, kCellThreads, 0, s>>>(W, g, lists.eq, lists.cnt);
  k_mark<N, D><<<gr, kCellThreads, 0, s>>>(W, V, g, lists, all);
}
}  // namespace

void launch_mark64(int N, int D, const double* W, const double* V, const DevGrid& g, const SweepLists& lists, int all,
                   cudaStream_t s) {
  if (N == 2 && D == 1) mark64<2, 1>(W, V, g, lists, all, s);
  if (N == 2 && D == 2) mark64<2, 2>(W, V, g, lists, all, s);
  if (N == 2 && D == 3) mark64<2, 3>(W, V, g, lists, all, s);
  if (N == 3 && D == 1) mark64<3, 1>(W, V, g, lists, all, s);
  if (N == 3 && D == 2) mark64<3, 2>(W, V, g, lists, all, s);
  if (N == 3 && D == 3) mark64<3, 3>(W, V, g, lists, all, s);
}

}  // namespace hrm
