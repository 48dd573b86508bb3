// Uniform faces and the lists of the other midpoints, for N = 2..3 species and
// D = 1..3 dimensions (see hrm_sweep.cuh). Built without FMA contraction.
#include "hrm_sweep.cuh"

namespace hrm {

namespace {
template <int N, int D>
void mark(const double* W, const double* V, const float* P32, const DevGrid& g, const SweepLists& lists,
          cudaStream_t s) {
  const unsigned gr = grid_for(g.nint, kCellThreads);
  if (P32) {
    k_equal<N, D, float><<<gr, kCellThreads, 0, s>>>(P32, nullptr, g, lists.eq, lists.cnt);
    k_mark<N, D, true><<<gr, kCellThreads, 0, s>>>(W, V, P32, g, lists);
  } else {
    k_equal<N, D, double><<<gr, kCellThreads, 0, s>>>(W, V, g, lists.eq, lists.cnt);
    k_mark<N, D, false><<<gr, kCellThreads, 0, s>>>(W, V, P32, g, lists);
  }
}
}  // namespace

void launch_mark(int N, int D, const double* W, const double* V, const float* P32, const DevGrid& g,
                 const SweepLists& lists, cudaStream_t s) {
  if (N == 2 && D == 1) mark<2, 1>(W, V, P32, g, lists, s);
  if (N == 2 && D == 2) mark<2, 2>(W, V, P32, g, lists, s);
  if (N == 2 && D == 3) mark<2, 3>(W, V, P32, g, lists, s);
  if (N == 3 && D == 1) mark<3, 1>(W, V, P32, g, lists, s);
  if (N == 3 && D == 2) mark<3, 2>(W, V, P32, g, lists, s);
  if (N == 3 && D == 3) mark<3, 3>(W, V, P32, g, lists, s);
}

}  // namespace hrm
