// FP32-bulk per-midpoint kernels for D = 3, N = 2..3 species (the precision
// form: interpolation, Riemann fluxes and HCS in FP32; limiter theta in FP64).
#include "hrm_face32.cuh"
#include "hrm_face32_net.cuh"
#include "hrm_launch.h"

namespace hrm {
namespace {

constexpr int kD = 3;

// Blocks of the sweep with the network, of the screened one and of the full one.
template <int N, int DIR, bool LISTED>
void launch_as(unsigned net, unsigned fast, unsigned full, const double* W, const double* V, const double* AUX,
               const float* P32, double* out, const DevGrid& g, const DevFluid& f, const DevParams& p, const StepState* st,
               const GateArgs& gate, cudaStream_t s) {
  if (!gate.defer_list) {
    k_face32<N, kD, DIR, LISTED><<<full, kFaceThreads, 0, s>>>(W, V, AUX, P32, out, g, f, p, st, gate.fixed, gate.list,
                                                               gate.list_cnt);
    return;
  }
  if (gate.net)
    k_face32_net<N, kD, DIR, LISTED><<<net, kFaceThreads, 0, s>>>(
        W, P32, gate.R32, out, g, f, p, st, static_cast<const mlp::GateBlob*>(gate.net), gate.zthr, gate.out_gate,
        gate.list, gate.list_cnt, gate.defer_list);
  else
    k_face32_fast<N, kD, DIR, LISTED><<<fast, kFaceThreads, 0, s>>>(W, P32, out, g, f, p, st, gate.fixed, gate.list,
                                                                    gate.list_cnt, gate.defer_list);
  const cudaStream_t sf = fix_stream(gate, s);
  k_face32_fix<N, kD, DIR><<<kFixBlocks, kFixThreads, 0, sf>>>(W, P32, out, g, f, p, st, gate.fixed, gate.defer_list,
                                                                gate.list_cnt + 2);
  fix_done(gate);
}

template <int N, int DIR>
void launch(const double* W, const double* V, const double* AUX, const float* P32, double* out, const DevGrid& g,
            const DevFluid& f, const DevParams& p, const StepState* st, const GateArgs& gate, cudaStream_t s) {
  if constexpr (DIR < kD) {
    if (gate.list)
      launch_as<N, DIR, true>(list_grid(g, DIR, 5), list_grid(g, DIR, 6), list_grid(g, DIR, 3), W, V, AUX, P32, out, g, f, p, st,
                              gate, s);
    else
      launch_as<N, DIR, false>(all_grid(g, DIR), all_grid(g, DIR), all_grid(g, DIR), W, V, AUX, P32, out, g, f, p, st, gate, s);
  }
}

}  // namespace

void update32_d3(int N, const double* Wn, const double* Wsrc, double* Wout, const double* F0, const double* F1,
                 const double* F2, const DevGrid& g, const DevFluid& f, StepState* st, double a, double b, int relax,
                 int count, cudaStream_t s) {
  const unsigned gr = grid_for(g.nint, kCellThreads);
  if (N == 2)
    k_update<2, kD, 0, true><<<gr, kCellThreads, 0, s>>>(Wn, Wsrc, Wout, F0, F1, F2, g, f, st, a, b, relax, count);
  else if (N == 3)
    k_update<3, kD, 0, true><<<gr, kCellThreads, 0, s>>>(Wn, Wsrc, Wout, F0, F1, F2, g, f, st, a, b, relax, count);
}

void update32p_d3(int N, const Update32Args& A, const DevGrid& g, const DevFluid& f, int tau, const SweepLists& lists,
                  int phase, cudaStream_t s) {
  uint32_t* cnt = lists.cnt + 3 * kSweepCounts;
  if (phase == 0) {
    const unsigned gr = grid_for(g.nint, kCellThreads);
    if (N == 2)
      k_keep32<2, kD><<<gr, kCellThreads, 0, s>>>(A, g, f, tau, lists.cells, cnt);
    else if (N == 3)
      k_keep32<3, kD><<<gr, kCellThreads, 0, s>>>(A, g, f, tau, lists.cells, cnt);
    return;
  }
  if (!A.uni) {
    const unsigned th = cell_threads(g.nint), gr = grid_for(g.nint, th);
    if (N == 2)
      k_update32p_all<2, kD><<<gr, th, 0, s>>>(A, g, f, tau);
    else if (N == 3)
      k_update32p_all<3, kD><<<gr, th, 0, s>>>(A, g, f, tau);
    return;
  }
  const unsigned gr = resident_grid(g.nint, kCellThreads, 3);
  if (N == 2)
    k_update32p<2, kD><<<gr, kCellThreads, 0, s>>>(A, g, f, tau, lists.cells, cnt);
  else if (N == 3)
    k_update32p<3, kD><<<gr, kCellThreads, 0, s>>>(A, g, f, tau, lists.cells, cnt);
}

void face32_d3(int N, int dir, const double* W, const double* V, const double* AUX, const float* P32, double* out,
               const DevGrid& g, const DevFluid& f, const DevParams& p, const StepState* st, const GateArgs& gate,
               cudaStream_t s) {
  if (N == 2) {
    if (dir == 0) launch<2, 0>(W, V, AUX, P32, out, g, f, p, st, gate, s);
    if (dir == 1) launch<2, 1>(W, V, AUX, P32, out, g, f, p, st, gate, s);
    if (dir == 2) launch<2, 2>(W, V, AUX, P32, out, g, f, p, st, gate, s);
  } else if (N == 3) {
    if (dir == 0) launch<3, 0>(W, V, AUX, P32, out, g, f, p, st, gate, s);
    if (dir == 1) launch<3, 1>(W, V, AUX, P32, out, g, f, p, st, gate, s);
    if (dir == 2) launch<3, 2>(W, V, AUX, P32, out, g, f, p, st, gate, s);
  }
}

void prim32_d3(int N, const double* W, float* P32, float* R32, const DevGrid& g, const DevFluid& f, StepState* st,
               int tau, cudaStream_t s) {
  const unsigned gr = grid_for(g.ncells, kCellThreads);
  if (N == 2)
    k_prim32<2, kD><<<gr, kCellThreads, 0, s>>>(W, P32, R32, g, f, st, tau);
  else if (N == 3)
    k_prim32<3, kD><<<gr, kCellThreads, 0, s>>>(W, P32, R32, g, f, st, tau);
}

}  // namespace hrm
