// Which midpoints of a stage need the whole midpoint body. A midpoint whose six
// node states are identical takes the node's physical flux (see face_body), and
// over most of a flow that is what the midpoints do: quiescent gas, interiors,
// post-shock states. Instead of every sweep reading all planes at six nodes of
// every midpoint to find out, one pass compares each cell with its next
// neighbour in every direction (k_equal, one byte per cell), a second one
// combines five such bytes per midpoint, writes for each cell which of its faces
// are uniform and appends the other midpoints to a list per direction (k_mark).
// The sweeps then run the body over full warps of listed midpoints, and the
// update forms a uniform face's flux from the cell's own state, which the face's
// nodes equal, so such faces are neither written nor read. (Small grids and the
// first-order scheme go without: `listed` in hrm_api.cu.)
#pragma once

#include "hrm_face32.cuh"
#include "hrm_launch.h"

namespace hrm {

// Cell that follows cell i (index ijk) along direction d, or with LOW the one
// before it, through the boundary condition of that side.
template <int D, bool LOW>
__device__ __forceinline__ int64_t neighbour(const DevGrid& g, int d, const int64_t* ijk, int64_t c) {
  const int64_t stride = d == 0 ? 1 : (d == 1 ? g.n[0] : g.n[0] * g.n[1]);
  const int64_t n = g.n[d], j = ijk[d] + (LOW ? -1 : 1);
  if (j >= 0 && j < n) return c + (LOW ? -stride : stride);
  const int b = 2 * d + (LOW ? 0 : 1);
  if (g.bc[b] == 2) {
    const int64_t tr = d == 0 ? ijk[2] * g.n[1] + ijk[1] : (d == 1 ? ijk[2] * g.n[0] + ijk[0] : ijk[1] * g.n[0] + ijk[0]);
    return g.goff[b] + tr;
  }
  return c + (bc_map(g, d, j) - ijk[d]) * stride;
}

// eq[c], bit d: every plane the same in cell c and the cell after it along d; bit
// 3 + d, for the first cell of a line: in cell c and the ghost cell before it; bit
// 6 (kFluxOverflow): the cell's physical flux may not be finite. T double: the M
// planes of W, bit for bit (the FP64 form's uniform stencils; its velocities and
// pressure from V); T float: the precision form's FP32 planes, by value. Thread by
// thread the lists' counters are cleared.
// Bit 6 by exponents: every factor of a flux term, p included, lies below 2^(a+1)
// and every velocity below 2^(b+1) for their largest exponents a and b, so the
// terms and their sums (E + p and + p) lie below 2^(a + b + 4).
template <int N, int D, typename T>
__global__ void __launch_bounds__(kCellThreads)
    k_equal(const T* __restrict__ W, const double* __restrict__ V, DevGrid g, uint8_t* __restrict__ eq,
            uint32_t* __restrict__ cnt) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < kSweepCounters) cnt[c] = 0u;
  if (c >= g.nint) return;
  constexpr int M = sizeof(T) == 8 ? Lay<N, D>::M : P32Lay<N, D>::PLANES;
  auto same_value = [](T x, T y) {
    if constexpr (sizeof(T) == 8)
      return __double_as_longlong(x) == __double_as_longlong(y);
    else
      return x == y;
  };
  int64_t ijk[3];
  cell_index(g, c, ijk);
  constexpr int kBias = sizeof(T) == 8 ? 1023 : 127, kMant = sizeof(T) == 8 ? 20 : 23;
  // larger magnitude: bits ordered as |x|, exponent field on top (float: one
  // instruction, which passes NaN over -- a cell that holds one equals no other)
  auto larger = [](uint32_t h, T x) -> uint32_t {
    if constexpr (sizeof(T) == 8)
      return max(h, (uint32_t)__double2hiint(x) & 0x7fffffffu);
    else
      return __float_as_uint(fmaxf(__uint_as_float(h), fabsf(x)));
  };
  T w[M];
  uint32_t hw = 0, hu = 0;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    w[m] = W[m * g.ncells + c];
    // what a flux multiplies or adds (uniform_flux64, uniform_flux32)
    using L = Lay<N, D>;
    const bool factor = sizeof(T) == 8 ? m < L::AL : (m < N || m == L::EN || (m >= L::M + 3 && m <= L::M + 3 + D));
    if (factor) hw = larger(hw, w[m]);
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    constexpr int u = Lay<N, D>::MOM;
    if constexpr (sizeof(T) == 8)
      hu = larger(hu, V[(u + d) * g.ncells + c]);
    else
      hu = larger(hu, w[u + d]);
  }
  if constexpr (sizeof(T) == 8) hw = larger(hw, V[Lay<N, D>::EN * g.ncells + c]);
  const int ew = (int)(hw >> kMant), eu = (int)(hu >> kMant);  // 2 kBias + 1 for infinities and NaN
  unsigned bits = (ew > 2 * kBias - 4 || eu > 2 * kBias || ew + eu > 3 * kBias - 4) ? kFluxOverflow : 0u;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    auto same = [&](int64_t o) {
      o = HRM_IDX(g, o, g.ncells);
      bool s = true;
#pragma unroll
      for (int m = 0; m < M; ++m) s = s & same_value(W[m * g.ncells + o], w[m]);
      return s;
    };
    if (same(neighbour<D, false>(g, d, ijk, c))) bits |= 1u << d;
    if (ijk[d] == 0 && g.bc[2 * d] != 1 && same(neighbour<D, true>(g, d, ijk, c))) bits |= 8u << d;
  }
  eq[c] = (uint8_t)bits;
}

// uni[c], bits 2 d and 2 d + 1: the faces of cell c on the low and the high side
// of direction d are uniform; bit kFluxOverflow as in eq[c]. The
// other midpoints go to lists.list[d] in the order of their cells, one atomic per
// block and direction. With lists.F (every midpoint's flux wanted) the uniform
// faces' fluxes are written too, and with lists.gate their gate bytes. FP32: the
// precision form (P32), else the FP64 form (W, V).
template <int N, int D, bool FP32>
__global__ void __launch_bounds__(kCellThreads)
    k_mark(const double* __restrict__ W, const double* __restrict__ V, const float* __restrict__ P32, DevGrid g,
           SweepLists lists) {
  using L = Lay<N, D>;
  constexpr int kWarps = kCellThreads / 32;
  __shared__ uint32_t base[D][kWarps];
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool in = c < g.nint;
  int64_t ijk[3] = {0, 0, 0};
  if (in) cell_index(g, c, ijk);
  unsigned uni = 0;
  if (in) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int64_t stride = d == 0 ? 1 : (d == 1 ? g.n[0] : g.n[0] * g.n[1]);
      const int64_t n = g.n[d], i = ijk[d];
      bool pair[6];  // cells i + j - 3 and i + j - 2 equal
      if (i >= 3 && i + 2 < n) {
#pragma unroll
        for (int j = 0; j < 6; ++j) pair[j] = (lists.eq[HRM_IDX(g, c + (j - 3) * stride, g.nint)] >> d) & 1u;
      } else {
        const bool per = g.bc[2 * d] == 1;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          int64_t q = i + j - 3;
          if (per) q = q < 0 ? q + n : (q >= n ? q - n : q);
          const bool low = q == -1;
          pair[j] = true;
          if (q >= -1 && q < n) {
            const unsigned e = lists.eq[HRM_IDX(g, c + ((low ? 0 : q) - i) * stride, g.nint)];
            pair[j] = (e >> (low ? 3 + d : d)) & 1u;
          }
        }
      }
      const bool mid = pair[1] & pair[2] & pair[3] & pair[4];
      uni |= (unsigned)(pair[0] & mid) << (2 * d) | (unsigned)(mid & pair[5]) << (2 * d + 1);
    }
  }
  if (in) lists.uni[c] = (uint8_t)(uni | (lists.eq[c] & kFluxOverflow));
  uint32_t at[D];
  bool lo[D], hi[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    lo[d] = in && !(uni >> (2 * d) & 1u);
    hi[d] = in && ijk[d] == g.n[d] - 1 && !(uni >> (2 * d + 1) & 1u);
    const unsigned a = __ballot_sync(0xffffffffu, lo[d]), b = __ballot_sync(0xffffffffu, hi[d]);
    const unsigned below = (1u << lane) - 1u;
    at[d] = __popc(a & below) + __popc(b & below);
    if (lane == 0) base[d][warp] = __popc(a) + __popc(b);
  }
  __syncthreads();
  if (threadIdx.x < D) {
    uint32_t n = 0;
    for (int w = 0; w < kWarps; ++w) n += base[threadIdx.x][w];
    uint32_t b = n ? atomicAdd(&lists.cnt[kSweepCounts * threadIdx.x], n) : 0u;
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t k = base[threadIdx.x][w];
      base[threadIdx.x][w] = b;
      b += k;
    }
  }
  __syncthreads();
  if (!in) return;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int64_t f0 = g.n[0] + (d == 0), f1 = g.n[1] + (d == 1);
    const int64_t t = (ijk[2] * f1 + ijk[1]) * f0 + ijk[0];
    const int64_t up = t + (d == 0 ? 1 : (d == 1 ? f0 : f0 * f1));
    const uint32_t p = base[d][warp] + at[d];
    if (lo[d]) lists.list[d][HRM_IDX(g, p, f0 * f1 * (g.n[2] + (d == 2)))] = (uint32_t)t;
    if (hi[d]) lists.list[d][HRM_IDX(g, p + (lo[d] ? 1u : 0u), f0 * f1 * (g.n[2] + (d == 2)))] = (uint32_t)up;
    const bool last = ijk[d] == g.n[d] - 1 && !hi[d];
    if (lists.gate[d]) {
      const int64_t nf = f0 * f1 * (g.n[2] + (d == 2));
      if (!lo[d]) lists.gate[d][HRM_IDX(g, t, nf)] = 2;
      if (last) lists.gate[d][HRM_IDX(g, up, nf)] = 2;
    }
    if (lists.F[d] && (!lo[d] || last)) {
      const int64_t nf = f0 * f1 * (g.n[2] + (d == 2));
      double G[L::NC];
      if constexpr (FP32)
        uniform_flux32<N, D>(c, d, P32, g.ncells, G);
      else
        uniform_flux64<N, D>(c, d, W, V, g.ncells, G);
#pragma unroll
      for (int m = 0; m < L::M + N - 1; ++m) {
        const double v = m < L::NC ? G[m < L::NC ? m : 0] : 0.0;
        if (!lo[d]) lists.F[d][m * nf + HRM_IDX(g, t, nf)] = v;
        if (last) lists.F[d][m * nf + HRM_IDX(g, up, nf)] = v;
      }
    }
  }
}

}  // namespace hrm
