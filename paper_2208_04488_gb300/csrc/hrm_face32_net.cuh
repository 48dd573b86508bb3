// Precision-form screened sweep with the learned smoothness detector evaluated
// inside it: the step path of the precision form with the learned gate.
//
// The sweep's list (k_mark) holds the midpoints whose stencil is not uniform; a
// uniform stencil takes the node's physical flux, which no interpolation choice
// affects, and needs no network. A warp forms the 30 features of each of its 32
// listed stencils (stencil_features, the gate kernel's function) and runs the
// network on them with warp-level MMA (mlp::warp_logit); a stencil whose logit
// exceeds the threshold then uses the linear weights. Compared with a gate kernel
// before the sweep, this removes one launch per direction and the second read of
// the stencil planes, and the network runs only where a stencil is not uniform.
//
// Gate bytes (one per midpoint, in `gate`): 1 linear weights, 0 full WENO-IS,
// 2 uniform stencil (exact node flux; written by k_mark). The deferred-midpoint
// kernel reads them. Five blocks per SM: 2.8 % of a pass over six at 1024x512. Not
// LISTED (small grids): a thread per midpoint, which tests its own stencil; a warp
// of uniform ones leaves the network out. Four blocks there: few warps, no spills.
#pragma once

#include "hrm_learned.cuh"

namespace hrm {

template <int N, int D, int DIR, bool LISTED>
__global__ void __launch_bounds__(kFaceThreads, LISTED ? 5 : 4)
    k_face32_net(const double* __restrict__ W, const float* __restrict__ P32, const float* __restrict__ R32,
                 double* __restrict__ out, DevGrid g, DevFluid f, DevParams pr, const StepState* __restrict__ st,
                 const mlp::GateBlob* __restrict__ blob, float zthr, uint8_t* __restrict__ gate,
                 const uint32_t* __restrict__ list, uint32_t* __restrict__ cnt, uint32_t* __restrict__ deferred) {
  __shared__ __align__(16) __nv_bfloat16 X[kFaceThreads / 32][32][mlp::kWarpRow];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the warp's 32 midpoints; `in`: this lane has one, and it is not uniform
  auto group = [&](int64_t t, const Nodes6& nd, bool in) {
    float x[mlp::kIn];
    if (in) {
      mlp::stencil_features<N, D, DIR>(nd, P32, R32, g.ncells, x);
    } else {
#pragma unroll
      for (int k = 0; k < mlp::kIn; ++k) x[k] = 0.f;
    }
    mlp::warp_store_row(X[warp], lane, x);
    __syncwarp();
    const float z = mlp::warp_logit(*blob, X[warp], lane);
    bool need = false;
    if (in) {
      const bool lin = z > zthr;
      gate[t] = lin ? 1 : 0;
      need = !face32_body<N, D, DIR, true>(t, nd, W, nullptr, nullptr, P32, out, g, f, pr, st->lam[DIR], lin);
    }
    defer_push(g, need, t, deferred, &cnt[2], face_count<DIR>(g));
  };
  if constexpr (!LISTED) {
    const int64_t t = (int64_t)blockIdx.x * kFaceThreads + threadIdx.x;
    Nodes6 nd;
    bool in = face_nodes<DIR>(g, t, nd);
    if (in && uniform_midpoint32<N, D, DIR>(t, nd, P32, out, g)) {
      gate[t] = 2;
      in = false;
    }
    if (__any_sync(0xffffffffu, in)) group(t, nd, in);
    return;
  }
  const uint32_t n = cnt[0];
  uint32_t i;
  while (next_entries(cnt, n, i)) {
    const int64_t t = i < n ? listed_midpoint<DIR>(g, list, i) : 0;
    Nodes6 nd;
    const bool in = i < n && face_nodes<DIR>(g, t, nd);
    group(t, nd, in);
  }
}

}  // namespace hrm
