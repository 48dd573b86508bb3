// FP64 per-midpoint body: characteristic projection, WENO-IS, interpolation
// limiter, HLLC, HCS, sensor blend, quasi-conservative fluxes and flux limiter,
// each rounding as the oracle's expression order fixes it.
//
// What bounds it is the FP64 unit (19 cycles of the SM per warp instruction,
// hrm_soft64.cuh), so the two loops that most of the work is in (the interpolation
// of the fields, and the flux slots) give that unit the additions and form the
// products and quotients on the integer pipes beside it. Multiplications by powers
// of two that feed an addition are folded into it as an FMA (the product is exact,
// so the sum rounds once as before), and the sums' common powers of two are taken
// out. A non-uniform midpoint of three species in 2D issued about 2900 FP64
// instructions before and about 1200 now. Straight-line code runs once per
// midpoint, so there its size counts (unrolled with integer products everywhere,
// the body's warps waited for instructions more than for anything else): the two
// sides share one copy, with their values in a per-thread column of shared memory.
// Measured, a pass of one step: shock-bubble 1024x512 6.18 -> 3.97 ms, 72x60x50
// interface 7.10 -> 2.57 (with the lists of hrm_sweep.cuh), smooth advection
// 250x250 (no stencil uniform) 1.61 -> 1.13. Three blocks per SM at 168 registers
// against four at 128, us a pass: 301x151 jet 1191 against 1455, 72x60x50 box 2497
// against 2568, shock-bubble 3819 against 3784, 250x250 advection 1129 against 1049.
#pragma once

#include "hrm_kernels.cuh"

namespace hrm {

// 1, 2, 4 and 1/4 in registers, unknown to the compiler (read from memory once per
// thread).
struct FmaUnits {
  double one, two, four, quarter;
};
__device__ const double kFmaUnits[4] = {1.0, 2.0, 4.0, 0.25};
__device__ __forceinline__ FmaUnits load_units() {
  const volatile double* p = kFmaUnits;
  return {p[0], p[1], p[2], p[3]};
}

// WENO-IS (App. C) of weno_is, value by value the same, on the stencil (a, b, c,
// d, e) = u_{i-2} .. u_{i+2}; a3, c3, d3: three times a, c, d; b0 = (c - d)^2.
// For values that are zero or of a magnitude within [2^-200, 2^80) and eps
// within [2^-60, 2^170] every product here is zero or normal.
// With x_k the sub-stencil sums of S_k = x_k / 2, / 2, / 8, / 8 and p_k the
// products of eta_k = (15 p_0, 5 p_1, 10 p_2, 2 p_3) / 32, the powers of two move
// through the roundings: sum eta_k S_k / sum eta_k = V / ES / 4 below.
// Additions go through an FMA with a multiplier in registers (FmaUnits): the FP64
// unit takes a DFMA of three registers every 16 cycles, but a DADD, a DMUL or a
// DFMA with a constant operand only every 19 (measured).
__device__ __forceinline__ double weno_side(double a, double b, double c, double d, double e, double a3, double c3,
                                            double d3, double b0, double eps, const FmaUnits& u) {
  using soft::mul_in;
  auto sq = [](double x) { return mul_in<true, false>(x, x); };      // of any sign
  auto pos = [](double x, double y) { return mul_in<false, false>(x, y); };
  auto any = [](double x, double y) { return mul_in<true, true>(x, y); };
  auto add = [&](double x, double y) { return fma(x, u.one, y); };
  auto sub = [&](double x, double y) { return fma(x, u.one, -y); };
  constexpr double k = 13.0 / 12.0;
  // k t^2 + t'^2 / 4 as ((k t) t) + ((t' / 4) t'): the last product is exact in the FMA
  auto beta = [&](double t, double tt) { return fma(u.quarter, sq(tt), mul_in<true, false>(any(k, t), t)); };
  const double x0 = add(c, d);
  const double x1 = sub(c3, b);
  const double x2 = sub(fma(u.two, d3, c3), e);
  const double x3 = add(sub(a3, any(10.0, b)), any(15.0, c));
  const double b1 = sq(sub(b, c));
  const double b01 = beta(add(fma(u.two, -c, b), d), sub(b, d));
  const double b2 = beta(add(fma(u.two, -d, c), e), add(fma(u.four, -d, c3), e));
  const double b3 = beta(add(fma(u.two, -b, a), c), add(fma(u.four, -b, a), c3));
  const double tau = beta(add(fma(u.four, -b, fma(u.two, c3, fma(u.four, -d, e))), a),
                          sub(fma(u.two, b, fma(u.two, -d, e)), a));
  const double A = add(b0, eps), B = add(b1, eps), C = add(b01, eps), g2 = add(b2, eps), g3 = add(b3, eps);
  const double t2 = sq(tau);
  const double g23 = pos(g2, g3), ABC = pos(pos(A, B), C);
  const double E0 = pos(15.0, pos(add(pos(A, C), t2), pos(B, g23)));
  const double E1 = pos(5.0, pos(add(pos(B, C), t2), pos(A, g23)));
  const double E2 = pos(5.0, pos(add(g2, tau), pos(ABC, g3)));
  const double E3 = pos(add(g3, tau), pos(ABC, g2));
  const double ES = fma(u.two, E3, fma(u.two, E2, add(E0, E1)));
  const double V = add(fma(u.two, add(any(E0, x0), any(E1, x1)), any(E2, x2)), any(E3, x3));
  return (((uint32_t)__double2hiint(V) & 0x7ff00000u) == 0u) ? V : soft::div_in<-2>(V, ES);
}

// The same stencil with the linear weights d_k = (15, 5, 10, 2) / 32 (weno_lin).
__device__ __forceinline__ double linear_side(double a, double b, double c, double d, double e, double a3, double c3,
                                              double d3) {
  auto any = [](double x, double y) { return soft::mul_in<true, true>(x, y); };
  const double x2 = fma(2.0, d3, c3) - e;
  const double x3 = (a3 - any(10.0, b)) + any(15.0, c);
  return soft::scale<-7>(fma(2.0, any(15.0, c + d) + any(5.0, c3 - b), any(5.0, x2)) + x3);
}

// Both biased values at x_{i+1/2} of one characteristic field from its six node
// values; lin: the linear weights (gated midpoint).
__device__ __forceinline__ void weno_both(const double* v, double eps, bool lin, const FmaUnits& units, double& left,
                                          double& right) {
  bool in = (eps >= 0x1p-60) & (eps <= 0x1p170);
#pragma unroll
  for (int j = 0; j < 6; ++j) in = in & soft::within<-200, 80>(v[j]);
  if (!in) {
    left = weno_sel<double>(lin, v[0], v[1], v[2], v[3], v[4], eps);
    right = weno_sel<double>(lin, v[5], v[4], v[3], v[2], v[1], eps);
    return;
  }
  auto bits = [](double x) { return __double_as_longlong(x); };
  const long long m = bits(v[2]);
  const bool mid = (bits(v[1]) == m) & (bits(v[3]) == m) & (bits(v[4]) == m);
  // constant stencils (five bit-identical values) return their value
  const bool cl = mid & (bits(v[0]) == m), cr = mid & (bits(v[5]) == m);
  left = v[2];
  right = v[3];
  if (cl & cr) return;
  auto triple = [](double x) { return soft::mul_in<true, true>(3.0, x); };
  const double t2 = triple(v[2]), t3 = triple(v[3]);
  const double dd = v[2] - v[3];
  const double b0 = soft::mul_in<true, false>(dd, dd);
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const double a = s ? v[5] : v[0], b = s ? v[4] : v[1], c = s ? v[3] : v[2], d = s ? v[2] : v[3], e = s ? v[1] : v[4];
    const double c3 = s ? t3 : t2, d3 = s ? t2 : t3;
    const double x = lin ? linear_side(a, b, c, d, e, triple(a), c3, d3)
                         : weno_side(a, b, c, d, e, triple(a), c3, d3, b0, eps, units);
    if (s == 0)
      left = cl ? left : x;
    else
      right = cr ? right : x;
  }
}

// First-order HLLC flux and u_* of a midpoint from its two node states (Sec. 4.1.1).
template <int N, int D, int DIR>
__device__ __forceinline__ void first_order64(const Nodes6& nd, const double* __restrict__ V, int64_t nc, const DevFluid& f,
                                              FluxPack<N, D>& H) {
  using L = Lay<N, D>;
  PrimState<double, N, D> a, b;
#pragma unroll
  for (int m = 0; m < L::M; ++m) {
    a.V[m] = V[m * nc + nd.c[2]];
    b.V[m] = V[m * nc + nd.c[3]];
  }
  double GH[L::M];
  const double uH = hllc<double, N, D, DIR>(f, a, b, GH);
#pragma unroll
  for (int m = 0; m < L::NC; ++m) H.Gc[m] = GH[m];
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    H.gm[k] = GH[L::AL + k] - uH * a.V[L::AL + k];
    H.gp[k] = GH[L::AL + k] - uH * b.V[L::AL + k];
  }
}

template <int N, int D, int DIR>
__device__ __forceinline__ void store_flux64(int64_t t, const FluxPack<N, D>& G, double* __restrict__ out, int64_t nf) {
  using L = Lay<N, D>;
#pragma unroll
  for (int m = 0; m < L::NC; ++m) out[m * nf + t] = G.Gc[m];
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    out[(L::AL + k) * nf + t] = G.gm[k];
    out[(L::M + k) * nf + t] = G.gp[k];
  }
}

// Column of a thread in the shared memory of a block of kFaceThreads: the biased
// values of the two sides, then the midpoint states with their rho, E and c, then
// the midpoint flux; 2 sides x (M + 3) slots.
template <int N, int D>
constexpr int kFaceCol = 2 * (Lay<N, D>::M + 3) * kFaceThreads;

// Whether the interpolation limiter provably returns the midpoint state as it
// is: every checked quantity at or above its limiter and hard-switch thresholds
// (theta = 1 gives 0 lo + 1 hi, the value itself). rc2: its rho c^2.
template <int N, int D>
__device__ __forceinline__ bool interp_limit_noop(const double* Vt, double rc2, const DevParams& pr) {
  using L = Lay<N, D>;
  const double tar = pr.eps_ar > pr.hs_ar ? pr.eps_ar : pr.hs_ar;
  const double ta = pr.eps_a > pr.hs_a ? pr.eps_a : pr.hs_a;
  bool ok = rc2 >= pr.hs_rc2;
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) ok = ok & (Vt[k] >= tar);
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    ok = ok & (Vt[L::AL + k] >= ta);
    s += Vt[L::AL + k];
  }
  return ok & (1.0 - s >= ta);
}

// One midpoint t of direction DIR (t inside the face grid); lam = lambda_DIR.
// Outputs: M + N - 1 planes over the face grid of the direction -- the NC
// conservative flux slots, the N-1 alpha slots of G^-_{i+1/2} (planes AL..M-1)
// and the N-1 alpha slots of G^+_{i+1/2} (planes M..M+N-2).
// lin: the midpoint is gated smooth -- the WENO-IS weights are replaced by the
// linear weights d_k; everything else is unchanged. col: kFaceCol doubles of
// shared memory. The six node states are known to differ (a uniform stencil takes
// the node's flux, uniform_flux64).
// LANES > 1: that many consecutive lanes of a warp share the midpoint (and call
// with the same arguments): the fields, the sides, the sensor's halves and the
// flux slots are dealt out to them, the rest each does itself, and they exchange
// through the column. The same values in the same order of operations; for short
// lists, where a lone warp's chain of FP64 instructions is the time.
template <int N, int D, int DIR, int LANES = 1>
__device__ __forceinline__ void face_body(int64_t t, const Nodes6& nd, const double* __restrict__ W,
                                          const double* __restrict__ V, const double* __restrict__ AUX,
                                          double* __restrict__ out, const DevGrid& g, const DevFluid& f,
                                          const DevParams& pr, double lam, double* col, bool lin = false) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
  const int64_t nc = g.ncells;
  const int64_t nf = face_count<DIR>(g);
  const double* __restrict__ Cc = AUX;           // sound speed
  const double* __restrict__ Rr = AUX + nc;      // mixture density
  const double* __restrict__ RC2 = AUX + 2 * nc; // rho c^2
  constexpr int kGroups = kFaceThreads / LANES;
  const int sub = threadIdx.x % LANES;
  auto slot = [&](int side, int m) -> double& { return col[(side * (M + 3) + m) * kGroups + threadIdx.x / LANES]; };
  // (LANES > 1) half-cell state of side s, behind the slots
  auto half = [&](int s, int m) -> double& { return col[(2 * (M + 3) + s * M + m) * kGroups + threadIdx.x / LANES]; };
  auto group_sync = [&]() {
    if constexpr (LANES > 1) __syncwarp(((1u << LANES) - 1u) << ((threadIdx.x & 31) / LANES * LANES));
  };

  double p6[6], u6[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    p6[j] = V[L::EN * nc + nd.c[j]];
    u6[j] = V[(L::MOM + DIR) * nc + nd.c[j]];
  }
  // characteristic projection with the face-averaged state (App. D), and the
  // biased values of every field: field 0 is u - p / (rho c) (slot 0), 1..N the
  // species alpha_k rho_k - (alpha_k rho_k)~ p / (rho c^2) (slots 1..N), then the
  // tangential velocities and the volume fractions as they are (slots N+1..M-2)
  // and last u + p / (rho c) (slot M-1)
  const double rhob = halved(Rr[nd.c[2]] + Rr[nd.c[3]]);
  const double cb = halved(Cc[nd.c[2]] + Cc[nd.c[3]]);
  const double rc = prod(rhob, cb);
  {
    // (a lone warp's DADD takes the same 64 cycles: no loads there)
    const FmaUnits units = LANES == 1 ? load_units() : FmaUnits{1.0, 2.0, 4.0, 0.25};
    const double inv_rc = quot(1.0, rc);
    const double rc2b = prod(rc, cb);
#pragma unroll 1
    for (int fi = sub; fi < M; fi += LANES) {
      double w6[6];
      if (fi == 0 || fi == M - 1) {
        const double q = fi == 0 ? -inv_rc : inv_rc;
#pragma unroll
        for (int j = 0; j < 6; ++j) w6[j] = u6[j] + prod(q, p6[j]);
      } else {
        int plane = fi - 1;                                                      // species, then the volume fractions
        if (fi > N) plane = fi < N + D ? L::MOM + (fi - N - 1 < DIR ? fi - N - 1 : fi - N) : fi + 1;
        const double* __restrict__ P = V + (int64_t)plane * nc;
#pragma unroll
        for (int j = 0; j < 6; ++j) w6[j] = P[nd.c[j]];
        if (fi <= N) {
          const double q = quot(halved(w6[2] + w6[3]), rc2b);
#pragma unroll
          for (int j = 0; j < 6; ++j) w6[j] = w6[j] - prod(q, p6[j]);
        }
      }
      double left, right;
      weno_both(w6, pr.weno_eps, lin, units, left, right);
      slot(0, fi) = left;
      slot(1, fi) = right;
    }
  }
  group_sync();
  // back to primitive variables, V~ = R U~, limited for positivity (Sec. 4.3.2);
  // the code of the straight-line parts from here on exists once for both sides
  // (it runs once per midpoint, so its size is what it costs beside its FP64
  // instructions: products are the FP64 unit's here)
  {
    const double c2 = soft::scale<1>(cb), rc_2 = halved(rc);
    double h[N];
#pragma unroll
    for (int k = 0; k < N; ++k) h[k] = quot(halved(V[k * nc + nd.c[2]] + V[k * nc + nd.c[3]]), c2);
#pragma unroll 1
    for (int side = LANES > 1 ? sub & 1 : 0; side < 2; side += LANES > 1 ? 2 : 1) {
      PrimState<double, N, D> S;
      const double U0 = slot(side, 0), U1 = slot(side, M - 1);
#pragma unroll
      for (int k = 0; k < N; ++k) S.V[k] = (-h[k]) * U0 + slot(side, 1 + k) + h[k] * U1;
      S.V[L::MOM + DIR] = 0.5 * U0 + 0.5 * U1;
      int t_ = 0;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        if (d == DIR) continue;
        S.V[L::MOM + d] = slot(side, N + 1 + t_);
        ++t_;
      }
      S.V[L::EN] = (-rc_2) * U0 + rc_2 * U1;
#pragma unroll
      for (int k = 0; k < N - 1; ++k) S.V[L::AL + k] = slot(side, N + D + k);
      double rc2;
      prim_state<double, N, D>(f, S, &rc2);
      if (pr.limiters && !interp_limit_noop<N, D>(S.V, rc2, pr)) {
        const int64_t cn = side ? nd.c[3] : nd.c[2];
        double Vn[M];
#pragma unroll
        for (int m = 0; m < M; ++m) Vn[m] = V[m * nc + cn];
        interp_limit<double, N, D>(S.V, Vn, RC2[cn], f, pr);
        prim_state<double, N, D>(f, S);
      }
      group_sync();
      if (sub < 2) {
#pragma unroll
        for (int m = 0; m < M; ++m) slot(side, m) = S.V[m];
        slot(side, M) = S.rho;
        slot(side, M + 1) = S.E;
        slot(side, M + 2) = S.c;
      }
    }
  }
  group_sync();
  // high-order midpoint flux G~ and velocity u~ (HLLC, Sec. 4.1.1)
  double ut;
  {
    double Gt[M], sL, sR;
    ut = hllc_speeds<double>(slot(0, L::MOM + DIR), slot(1, L::MOM + DIR), slot(0, L::EN), slot(1, L::EN), slot(0, M),
                             slot(1, M), slot(0, M + 2), slot(1, M + 2), sL, sR);
    const bool one = (ut > 0.0) | (ut < 0.0);  // else both sides with weight 1/2
#pragma unroll
    for (int m = 0; m < M; ++m) Gt[m] = 0.0;
#pragma unroll 1
    for (int side = ut < 0.0 ? 1 : 0; side < (ut > 0.0 ? 1 : 2); ++side)
      hllc_side<double, N, D, DIR>([&](int m) { return slot(side, m); }, slot(side, M), slot(side, M + 1),
                                   side ? sR : sL, side ? dmax(0.0, sR) : dmin(0.0, sL), ut,
                                   [&](int m, double v) { Gt[m] = one ? plus_zero(v) : Gt[m] + 0.5 * v; });
    group_sync();
    if (sub == 0) {
#pragma unroll
      for (int m = 0; m < M; ++m) slot(0, m) = Gt[m];
    }
  }
  // shock sensor (Sec. 4.3.1) on rho and p
  double sig = 0.0;
  if (pr.blend) {
    // the halves about nodes i + 1 and i of rho, then of p (slots 0..3 of side 1,
    // free by now)
#pragma unroll 1
    for (int k = sub; k < 4; k += LANES) {
      double x[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) x[j] = k >= 2 ? p6[j] : Rr[nd.c[j]];
      const bool e = k & 1;
      const double a = e ? x[0] : x[1], b = e ? x[1] : x[2], c30 = 30.0 * (e ? x[2] : x[3]), d = e ? x[3] : x[4],
                   r = e ? x[4] : x[5];
      const double num = fabs(fma(16.0, d, fma(16.0, b, -a) - c30) - r);
      const double den = fabs(fma(16.0, d, fma(16.0, b, a) + c30) + r);
      slot(1, k) = den == 0.0 ? 0.0 : quot(num, den);
    }
    group_sync();
    const double pw1 = (0.5 * (slot(1, 0) + slot(1, 1))) * (0.5 * (slot(1, 2) + slot(1, 3)));
    double pw = pw1;
    for (int e = 1; e < pr.qexp; ++e) pw = pw * pw1;
    sig = tanh_r<LANES == 1>(pr.Cs * pw);
  }
  group_sync();
  const double one_m = 1.0 - sig;
  // explicit HCS reconstruction (Eqs. reconstructed_G, reconstructed_vel), blended
  constexpr double psi = 256.0 / 175.0;
  constexpr double a1 = 75.0 * psi / 128.0 - 37.0 / 60.0;
  constexpr double a2 = 25.0 * psi / 256.0 - 2.0 / 15.0;
  constexpr double a3 = 3.0 * psi / 256.0 - 1.0 / 60.0;
  // Slot by slot (first, m = -1, the velocity u^): the node fluxes G of the
  // flux-source form at the six nodes, the blended midpoint flux (kept in the
  // column; the alpha slots of G^- on side 1 and of G^+ on side 0), and the
  // half-cell states W_i^{+}, W_{i+1}^{-} that tell whether the flux limiter can
  // act: it provably leaves G unchanged where every quantity it checks
  // (alpha_k rho_k, all N alpha_k, rho e~) lies at or above both its limiter and
  // its hard-switch thresholds, whatever the first-order states (NaN fails the
  // test).
  const double tar = pr.eps_ar > pr.hs_ar ? pr.eps_ar : pr.hs_ar;
  const double ta = pr.eps_a > pr.hs_a ? pr.eps_a : pr.hs_a;
  const double tre = pr.eps_rhoe > pr.hs_rhoe ? pr.eps_rhoe : pr.hs_rhoe;
  const double l2 = 2.0 * lam;
  bool ok = true;
  double uhat = 0.0;
  double rho[2] = {0.0, 0.0}, rq[2] = {0.0, 0.0}, kin[2] = {0.0, 0.0}, en[2] = {0.0, 0.0}, as[2] = {0.0, 0.0};
  // quantities the limiter checks of one half-cell state, slot by slot in order
  auto account = [&](int m, int s, double h) {
    if (m < L::MOM) {
      ok = ok & (h >= tar);
      rho[s] += h;
      if (f.has_q) rq[s] += h * f.q[m];
    } else if (m < L::EN) {
      kin[s] += h * h;
    } else if (m == L::EN) {
      en[s] = h;
    } else {
      ok = ok & (h >= ta);
      as[s] += h;
    }
  };
  auto check = [&](int s) {
    ok = ok & (1.0 - as[s] >= ta);
    ok = ok & (en[s] - quot(halved(kin[s]), rho[s]) - rq[s] >= tre);
  };
#pragma unroll 1
  for (int m = -1; m < M; m = m < 0 ? sub : m + LANES) {
    double w6[6], n6[6], gt = ut;
    if (m < 0) {
#pragma unroll
      for (int j = 0; j < 6; ++j) n6[j] = u6[j];
    } else {
      const double* __restrict__ P = W + (int64_t)m * nc;
#pragma unroll
      for (int j = 0; j < 6; ++j) n6[j] = w6[j] = P[nd.c[j]];
      if (m == L::EN) {
#pragma unroll
        for (int j = 0; j < 6; ++j) n6[j] = n6[j] + p6[j];
      }
#pragma unroll
      for (int j = 0; j < 6; ++j) n6[j] = prod(n6[j], u6[j]);
      if (m == L::MOM + DIR) {
#pragma unroll
        for (int j = 0; j < 6; ++j) n6[j] = n6[j] + p6[j];
      } else if (m >= L::MOM && m < L::EN) {
#pragma unroll
        for (int j = 0; j < 6; ++j) n6[j] = plus_zero(n6[j]);
      }
      gt = slot(0, m);
    }
    const double hcs = prod(psi, gt) - prod(a1, n6[2] + n6[3]) + prod(a2, n6[1] + n6[4]) - prod(a3, n6[0] + n6[5]);
    const double gh = prod(sig, gt) + prod(one_m, hcs);
    if (m < 0) {
      uhat = gh;
      continue;
    }
    double x0 = gh, x1 = gh;
    if (m < L::NC) {
      slot(1, m) = gh;
      x0 = x0 - n6[2];
      x1 = x1 - n6[3];
    } else {
      // quasi-conservative alpha slots (Eq. G_pm, high-order form)
      x0 = x0 - prod(uhat, w6[2]);
      x1 = x1 - prod(uhat, w6[3]);
      slot(1, m) = x0;
      slot(0, m) = x1;
    }
    const double h[2] = {w6[2] - prod(l2, x0), w6[3] + prod(l2, x1)};
    if constexpr (LANES > 1) {
      half(0, m) = h[0];
      half(1, m) = h[1];
    } else {
      account(m, 0, h[0]);
      account(m, 1, h[1]);
    }
  }
  group_sync();
  if constexpr (LANES > 1) {
#pragma unroll 1
    for (int m = 0; m < M; ++m) account(m, 0, half(sub & 1, m));
    check(0);
    const bool other = __shfl_xor_sync(((1u << LANES) - 1u) << ((threadIdx.x & 31) / LANES * LANES), (int)ok, 1) != 0;
    ok = ok & other;
  } else {
    check(0);
    check(1);
  }
  if (pr.limiters && !ok) {
    FluxPack<N, D> G, H;
    first_order64<N, D, DIR>(nd, V, nc, f, H);
    double Wi[M], Wj[M], Fi[L::NC], Fj[L::NC];
    {
      double Vi[M], Vj[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        Vi[m] = V[m * nc + nd.c[2]];
        Vj[m] = V[m * nc + nd.c[3]];
        Wi[m] = W[m * nc + nd.c[2]];
        Wj[m] = W[m * nc + nd.c[3]];
      }
      node_flux<N, D, DIR>(Wi, Vi, Fi);
      node_flux<N, D, DIR>(Wj, Vj, Fj);
    }
#pragma unroll
    for (int m = 0; m < L::NC; ++m) G.Gc[m] = slot(1, m);
#pragma unroll
    for (int k = 0; k < N - 1; ++k) {
      G.gm[k] = slot(1, L::AL + k);
      G.gp[k] = slot(0, L::AL + k);
    }
    flux_limit<N, D>(Wi, Wj, Fi, Fj, lam, G, H, f, pr);
    if (sub == 0) store_flux64<N, D, DIR>(t, G, out, nf);
    group_sync();  // the column is the next midpoint's
    return;
  }
  if constexpr (LANES > 1) {
    for (int m = sub; m < M + N - 1; m += LANES) out[m * nf + t] = m < M ? slot(1, m) : slot(0, L::AL + m - M);
    group_sync();  // the column is the next midpoint's
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) out[m * nf + t] = slot(1, m);
#pragma unroll
    for (int k = 0; k < N - 1; ++k) out[(M + k) * nf + t] = slot(0, L::AL + k);
  }
}

// Without a list LANES lanes test the six nodes of their midpoint t themselves:
// whether they are bit-identical (every plane of W), and if so its flux written.
template <int N, int D, int DIR, int LANES>
__device__ __forceinline__ bool uniform_midpoint64(int64_t t, const Nodes6& nd, const double* __restrict__ W,
                                                   const double* __restrict__ V, double* __restrict__ out,
                                                   const DevGrid& g) {
  using L = Lay<N, D>;
  const int lane = threadIdx.x & 31, sub = lane % LANES;
  bool same = true;
#pragma unroll
  for (int m = 0; m < L::M; m += LANES) {
    const int64_t plane = (int64_t)(m + sub < L::M ? m + sub : 0) * g.ncells;
    const long long b = __double_as_longlong(W[plane + nd.c[2]]);
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (j != 2) same = same & (__double_as_longlong(W[plane + nd.c[j]]) == b);
  }
  if (!__all_sync(((1u << LANES) - 1u) << (lane / LANES * LANES), same)) return false;
  if (sub == 0) {
    const int64_t nf = face_count<DIR>(g);
    double G[L::NC];
    uniform_flux64<N, D>(nd.c[2], DIR, W, V, g.ncells, G);
#pragma unroll
    for (int m = 0; m < L::M + N - 1; ++m) out[m * nf + t] = m < L::NC ? G[m < L::NC ? m : 0] : 0.0;
  }
  return true;
}

// Sweep of direction DIR over its list (k_mark), a warp of 32 entries at a time
// taken from a counter: every lane then runs the whole body (the FP64 unit's time
// does not depend on the active lanes), and the warps end within one entry of one
// another. Three blocks per SM. Shorter lists leave each SM a warp or two that
// issue an FP64 instruction every 64 cycles; there several lanes share an entry,
// the groups dealt out to the first warp of every block, then to the second ones.
// Measured us per step (both sweeps of n listed midpoints each) with 8 | 4 | 2 | 1
// lanes, three species: n = 4704 443 | 429 | 537 | 661, 8256 606 | 439 | 507 | 701,
// 12880 815 | 582 | 606 | 758, 20100 1307 | 1028 | 710 | 835, 32896 2048 | 1500 |
// 1083 | 1043; two: 3080 228 | 228 | 260 | 411, 5256 341 | 351 | 369 | 445, 12210
// 559 | 420 | 435 | 478, 17030 757 | 633 | 462 | 484, 25760 965 | 701 | 497 | 481.
// No list (small grids, `listed` in hrm_api.cu): every midpoint, by the same rule.
constexpr uint32_t kSplit8 = 4608, kSplit4 = 13312, kSplit2 = 20480;

template <int N, int D, int DIR, int LANES>
__device__ __forceinline__ void sweep_split(const double* __restrict__ W, const double* __restrict__ V,
                                            const double* __restrict__ AUX, double* __restrict__ out, const DevGrid& g,
                                            const DevFluid& f, const DevParams& pr, const StepState* __restrict__ st,
                                            const uint8_t* __restrict__ gate, const uint32_t* __restrict__ list,
                                            uint32_t n, double* col) {
  const uint32_t warps = gridDim.x * (kFaceThreads / 32), per = 32 / LANES;
  for (uint32_t k = blockIdx.x + gridDim.x * (threadIdx.x >> 5); k * per < n; k += warps) {
    Nodes6 nd;
    const uint32_t i = k * per + (threadIdx.x & 31) / LANES;
    if (i >= n) continue;
    const int64_t t = list ? listed_midpoint<DIR>(g, list, i) : i;
    if (!face_nodes<DIR>(g, t, nd)) continue;
    if (!list && uniform_midpoint64<N, D, DIR, LANES>(t, nd, W, V, out, g)) continue;
    const bool lin = gate != nullptr && gate[t] != 0;
    face_body<N, D, DIR, LANES>(t, nd, W, V, AUX, out, g, f, pr, st->lam[DIR], col, lin);
  }
}

template <int N, int D, int DIR>
__global__ void __launch_bounds__(kFaceThreads, 3)
    k_face(const double* __restrict__ W, const double* __restrict__ V, const double* __restrict__ AUX,
           double* __restrict__ out, DevGrid g, DevFluid f, DevParams pr, const StepState* __restrict__ st,
           const uint8_t* __restrict__ gate, const uint32_t* __restrict__ list, uint32_t* __restrict__ cnt) {
  __shared__ double col[kFaceCol<N, D>];
  const uint32_t n = list ? cnt[0] : (uint32_t)face_count<DIR>(g);
  if (n <= kSplit8) return sweep_split<N, D, DIR, 8>(W, V, AUX, out, g, f, pr, st, gate, list, n, col);
  if (n <= kSplit4) return sweep_split<N, D, DIR, 4>(W, V, AUX, out, g, f, pr, st, gate, list, n, col);
  if (n <= kSplit2 || !list) return sweep_split<N, D, DIR, 2>(W, V, AUX, out, g, f, pr, st, gate, list, n, col);
  uint32_t i;
  while (next_entries(cnt, n, i)) {
    Nodes6 nd;
    if (i >= n) continue;
    const int64_t t = listed_midpoint<DIR>(g, list, i);
    if (!face_nodes<DIR>(g, t, nd)) continue;
    const bool lin = gate != nullptr && gate[t] != 0;
    face_body<N, D, DIR>(t, nd, W, V, AUX, out, g, f, pr, st->lam[DIR], col, lin);
  }
}

// The first-order scheme: every midpoint, a thread each.
template <int N, int D, int DIR>
__global__ void __launch_bounds__(kFaceThreads)
    k_face_first(const double* __restrict__ V, double* __restrict__ out, DevGrid g, DevFluid f) {
  const int64_t t = (int64_t)blockIdx.x * kFaceThreads + threadIdx.x;
  Nodes6 nd;
  if (!face_nodes<DIR>(g, t, nd)) return;
  FluxPack<N, D> H;
  first_order64<N, D, DIR>(nd, V, g.ncells, f, H);
  store_flux64<N, D, DIR>(t, H, out, face_count<DIR>(g));
}

}  // namespace hrm
