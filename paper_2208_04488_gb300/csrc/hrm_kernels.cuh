// Kernel templates of the PP-WCNS-IS fractional step (arXiv 2208.04488).
//
// One RK stage is: k_prim (per cell: primitive variables, sound speed, and at
// the first stage the CFL max-wave-speed reduction) -> k_face for each direction
// (per midpoint: characteristic projection, WENO-IS, interpolation limiter,
// two HLLC solves, HCS reconstruction, shock-sensor blending, quasi-conservative
// fluxes and the flux limiter) -> k_update (per cell: flux difference with the
// non-conservative alpha term, SSP-RK combination, thermal relaxation,
// admissibility counters).
#pragma once

#include "hrm_device.cuh"

namespace hrm {

constexpr int kFaceThreads = 128;
constexpr int kCellThreads = 256;

// Face grid of direction DIR: n with n[DIR] + 1 entries along DIR.
template <int DIR>
__device__ __forceinline__ int64_t face_count(const DevGrid& g) {
  return (g.n[0] + (DIR == 0)) * (g.n[1] + (DIR == 1)) * (g.n[2] + (DIR == 2));
}

// Entry i of a list of midpoints of direction DIR.
template <int DIR>
__device__ __forceinline__ int64_t listed_midpoint(const DevGrid& g, const uint32_t* __restrict__ list, int64_t i) {
  return HRM_IDX(g, list[HRM_IDX(g, i, face_count<DIR>(g))], face_count<DIR>(g));
}

// ---------------------------------------------------------------- interpolation limiter

// Positivity-preserving interpolation limiter (Sec. 4.3.2, Alg. interp_limit_densities,
// Alg. interp_limit_vol_frac, hard switch) applied to the midpoint primitive
// state Vt against the first-order (node) state Vn; velocity and pressure are
// held, partial densities and volume fractions are limited, theta in FP64.
template <typename R, int N, int D>
__device__ __forceinline__ void interp_limit(R* Vt, const double* Vn, double rc2n, const DevFluid& f,
                                             const DevParams& pr) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const double lo = Vn[k], hi = (double)Vt[k];
    const double tgt = dmin(pr.eps_ar, lo);
    double th = 1.0;
    if (hi < tgt) th = (tgt - lo) / (hi - lo);
    Vt[k] = R((1.0 - th) * lo + th * hi);
  }
  double alt[N], aln[N];
  {
    double st = 0.0, sn = 0.0;
#pragma unroll
    for (int k = 0; k < N - 1; ++k) {
      alt[k] = (double)Vt[L::AL + k];
      aln[k] = Vn[L::AL + k];
      st += alt[k];
      sn += aln[k];
    }
    alt[N - 1] = 1.0 - st;
    aln[N - 1] = 1.0 - sn;
  }
  double th = 1.0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const double tgt = dmin(pr.eps_a, aln[k]);
    double thk = 1.0;
    if (alt[k] < tgt) thk = (tgt - aln[k]) / (alt[k] - aln[k]);
    th = dmin(th, thk);
  }
#pragma unroll
  for (int k = 0; k < N - 1; ++k) Vt[L::AL + k] = R((1.0 - th) * aln[k] + th * alt[k]);
  // hard switch
  bool hs = false;
  {
    double st = 0.0;
#pragma unroll
    for (int k = 0; k < N - 1; ++k) {
      alt[k] = (double)Vt[L::AL + k];
      st += alt[k];
    }
    alt[N - 1] = 1.0 - st;
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {
    hs |= (double)Vt[k] < dmin(pr.hs_ar, Vn[k]);
    hs |= alt[k] < dmin(pr.hs_a, aln[k]);
  }
  double S, P;
  mix_SP<double, N>(f, alt, S, P);
  const double rc2 = rho_c2(S, P, (double)Vt[L::EN]);
  hs |= rc2 < dmin(pr.hs_rc2, rc2n);
  if (hs) {
#pragma unroll
    for (int m = 0; m < M; ++m) Vt[m] = R(Vn[m]);
  }
}

// ---------------------------------------------------------------- flux limiter helpers

// rho (e - qbar) of a conservative vector (Sec. 2).
template <int N, int D>
__device__ __forceinline__ double rhoe_tilde(const double* W, const DevFluid& f) {
  using L = Lay<N, D>;
  double rho = 0.0, kin = 0.0, rq = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    rho += W[k];
    rq += W[k] * f.q[k];
  }
#pragma unroll
  for (int d = 0; d < D; ++d) kin += W[L::MOM + d] * W[L::MOM + d];
  return W[L::EN] - quot(0.5 * kin, rho) - rq;
}

__device__ __forceinline__ double theta_of(double lo, double hi, double eps) {
  const double tgt = dmin(eps, lo);
  return (hi < tgt) ? (tgt - lo) / (hi - lo) : 1.0;
}

// A midpoint flux G^-_{i+1/2} / G^+_{i+1/2} (Eq. G_pm): the conservative slots Gc
// are shared, the alpha slots differ (gm uses alpha_i, gp uses alpha_{i+1}).
template <int N, int D>
struct FluxPack {
  double Gc[Lay<N, D>::NC];
  double gm[N - 1 > 0 ? N - 1 : 1];
  double gp[N - 1 > 0 ? N - 1 : 1];
};

// Half-cell state W_n + s (G - F_n): with minus = true the alpha slots of G^-
// (cell i side), otherwise those of G^+ (cell i+1 side); F has zero alpha slots.
template <int N, int D>
__device__ __forceinline__ void half_state(const double* Wn, const double* Fn, const FluxPack<N, D>& G,
                                           double s, bool minus, double* out) {
  using L = Lay<N, D>;
#pragma unroll
  for (int m = 0; m < L::NC; ++m) out[m] = Wn[m] + s * (G.Gc[m] - Fn[m]);
#pragma unroll
  for (int k = 0; k < N - 1; ++k) out[L::AL + k] = Wn[L::AL + k] + s * (minus ? G.gm[k] : G.gp[k]);
}

template <int N, int D>
__device__ __forceinline__ void mix_pack(const FluxPack<N, D>& H, const FluxPack<N, D>& G, double th,
                                         FluxPack<N, D>& out) {
  using L = Lay<N, D>;
#pragma unroll
  for (int m = 0; m < L::NC; ++m) out.Gc[m] = (1.0 - th) * H.Gc[m] + th * G.Gc[m];
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    out.gp[k] = (1.0 - th) * H.gp[k] + th * G.gp[k];
    out.gm[k] = (1.0 - th) * H.gm[k] + th * G.gm[k];
  }
}

template <int N, int D>
__device__ __forceinline__ void all_alpha_W(const double* W, double* al) {
  using L = Lay<N, D>;
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    al[k] = W[L::AL + k];
    s += al[k];
  }
  al[N - 1] = 1.0 - s;
}

// Quasi-positivity-preserving flux limiter (Sec. 4.3.2, Alg.
// flux_limit_densities_vol_frac, Alg. flux_limit_energy, hard switch), FP64.
// Wi/Wj: W_i, W_{i+1}; Fi/Fj: conservative fluxes F(W_i), F(W_{i+1});
// G: high-order midpoint flux, H: first-order HLLC flux; the result replaces G.
//
// The limiter's guarantee rests on the first-order half-cell states being
// admissible, which holds for the HLLC flux in exact arithmetic with no margin
// at CFL 1/2. REPAIR (the precision form, whose H is an FP32 evaluation):
// where a first-order half-cell state comes out inadmissible, H is evaluated
// again in FP64 from the node states Vi, Vj, as the FP64 form does.
template <int N, int D, int DIR = 0, bool REPAIR = false>
__device__ __forceinline__ void flux_limit(const double* Wi, const double* Wj, const double* Fi,
                                           const double* Fj, double lam, FluxPack<N, D>& G,
                                           const FluxPack<N, D>& H_in, const DevFluid& f,
                                           const DevParams& pr, const double* Vi = nullptr,
                                           const double* Vj = nullptr) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
  const double m2l = -2.0 * lam, p2l = 2.0 * lam;
  double Wp[M], Wm[M], WHp[M], WHm[M];
  FluxPack<N, D> H = H_in;
  half_state<N, D>(Wi, Fi, G, m2l, true, Wp);    // W_i^{+}
  half_state<N, D>(Wj, Fj, G, p2l, false, Wm);   // W_{i+1}^{-}
  half_state<N, D>(Wi, Fi, H, m2l, true, WHp);   // W_i^{HLLC,+}
  half_state<N, D>(Wj, Fj, H, p2l, false, WHm);  // W_{i+1}^{HLLC,-}
  // first-order states: volume fractions and rho e~ (also the limiter's lower ends)
  double aHp[N], aHm[N];
  all_alpha_W<N, D>(WHp, aHp);
  all_alpha_W<N, D>(WHm, aHm);
  double rHp = rhoe_tilde<N, D>(WHp, f), rHm = rhoe_tilde<N, D>(WHm, f);
  if constexpr (REPAIR) {
    bool bad = !(rHp > 0.0) || !(rHm > 0.0);
#pragma unroll
    for (int k = 0; k < N; ++k)
      bad |= !(WHp[k] >= 0.0) || !(WHm[k] >= 0.0) || !(aHp[k] >= 0.0) || !(aHm[k] >= 0.0);
    if (bad) {
      PrimState<double, N, D> a, b;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        a.V[m] = Vi[m];
        b.V[m] = Vj[m];
      }
      double GH[M];
      const double uH = hllc<double, N, D, DIR>(f, a, b, GH);
#pragma unroll
      for (int m = 0; m < L::NC; ++m) H.Gc[m] = GH[m];
#pragma unroll
      for (int k = 0; k < N - 1; ++k) {
        H.gm[k] = GH[L::AL + k] - uH * Vi[L::AL + k];
        H.gp[k] = GH[L::AL + k] - uH * Vj[L::AL + k];
      }
      half_state<N, D>(Wi, Fi, H, m2l, true, WHp);
      half_state<N, D>(Wj, Fj, H, p2l, false, WHm);
      all_alpha_W<N, D>(WHp, aHp);
      all_alpha_W<N, D>(WHm, aHm);
      rHp = rhoe_tilde<N, D>(WHp, f);
      rHm = rhoe_tilde<N, D>(WHm, f);
    }
  }
  double th = 1.0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    th = dmin(th, dmin(theta_of(WHp[k], Wp[k], pr.eps_ar), theta_of(WHm[k], Wm[k], pr.eps_ar)));
  }
  {
    double ap[N], am[N];
    all_alpha_W<N, D>(Wp, ap);
    all_alpha_W<N, D>(Wm, am);
#pragma unroll
    for (int k = 0; k < N; ++k)
      th = dmin(th, dmin(theta_of(aHp[k], ap[k], pr.eps_a), theta_of(aHm[k], am[k], pr.eps_a)));
  }
  // with theta = 1 the mixed flux is G itself, bit for bit ((1 - 1) H + 1 G), and
  // the half-cell states need no recomputation
  FluxPack<N, D> Gs;
  if (th < 1.0) {
    mix_pack<N, D>(H, G, th, Gs);
    half_state<N, D>(Wi, Fi, Gs, m2l, true, Wp);   // W_i^{*,+}
    half_state<N, D>(Wj, Fj, Gs, p2l, false, Wm);  // W_{i+1}^{*,-}
  } else {
    Gs = G;
  }
  // energy stage
  const double th2 = dmin(theta_of(rHp, rhoe_tilde<N, D>(Wp, f), pr.eps_rhoe),
                          theta_of(rHm, rhoe_tilde<N, D>(Wm, f), pr.eps_rhoe));
  FluxPack<N, D> Gss;
  if (th2 < 1.0) {
    mix_pack<N, D>(H, Gs, th2, Gss);
    half_state<N, D>(Wi, Fi, Gss, m2l, true, Wp);   // W_i^{**,+}
    half_state<N, D>(Wj, Fj, Gss, p2l, false, Wm);  // W_{i+1}^{**,-}
  } else {
    Gss = Gs;
  }
  // hard switch
  bool hs = false;
  {
    double ap[N], am[N];
    all_alpha_W<N, D>(Wp, ap);
    all_alpha_W<N, D>(Wm, am);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      hs |= Wp[k] < dmin(pr.hs_ar, WHp[k]);
      hs |= ap[k] < dmin(pr.hs_a, aHp[k]);
      hs |= Wm[k] < dmin(pr.hs_ar, WHm[k]);
      hs |= am[k] < dmin(pr.hs_a, aHm[k]);
    }
  }
  hs |= rhoe_tilde<N, D>(Wp, f) < dmin(pr.hs_rhoe, rHp);
  hs |= rhoe_tilde<N, D>(Wm, f) < dmin(pr.hs_rhoe, rHm);
  G = hs ? H : Gss;
}

// ---------------------------------------------------------------- per-midpoint kernel

// Loads of the six node cells i-2..i+3 of a midpoint.
struct Nodes6 {
  int64_t c[6];
};

template <int DIR>
__device__ __forceinline__ bool face_nodes(const DevGrid& g, int64_t t, Nodes6& nd) {
  const int64_t f0 = g.n[0] + (DIR == 0), f1 = g.n[1] + (DIR == 1), f2 = g.n[2] + (DIR == 2);
  if (t >= f0 * f1 * f2) return false;
  int64_t ijk[3];
  plane_index(t, f0, f1, ijk);
  const int64_t i0 = ijk[0], i1 = ijk[1], i2 = ijk[2];
  const int64_t fp = DIR == 0 ? i0 : (DIR == 1 ? i1 : i2);
  const bool dlo = g.bc[2 * DIR] == 2, dhi = g.bc[2 * DIR + 1] == 2;
  // cell of the Dirichlet slice that continues this line
  const int64_t tr = DIR == 0 ? i2 * g.n[1] + i1 : (DIR == 1 ? i2 * g.n[0] + i0 : i1 * g.n[0] + i0);
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const int64_t jj = fp - 3 + j;
    const int64_t q = bc_map(g, DIR, jj);
    nd.c[j] = DIR == 0 ? (i2 * g.n[1] + i1) * g.n[0] + q
                       : (DIR == 1 ? (i2 * g.n[1] + q) * g.n[0] + i0 : (q * g.n[1] + i1) * g.n[0] + i0);
    if (jj < 0 && dlo) nd.c[j] = g.goff[2 * DIR] + tr;
    if (jj >= g.n[DIR] && dhi) nd.c[j] = g.goff[2 * DIR + 1] + tr;
    nd.c[j] = HRM_IDX(g, nd.c[j], g.ncells);
  }
  return true;
}

// Conservative flux F^DIR of a node (Eq. F_x_F_y_def), NC slots.
template <int N, int D, int DIR>
__device__ __forceinline__ void node_flux(const double* W, const double* V, double* F) {
  using L = Lay<N, D>;
  const double un = V[L::MOM + DIR], p = V[L::EN];
#pragma unroll
  for (int k = 0; k < N; ++k) F[k] = W[k] * un;
#pragma unroll
  for (int d = 0; d < D; ++d) F[L::MOM + d] = W[L::MOM + d] * un + (d == DIR ? p : 0.0);
  F[L::EN] = (W[L::EN] + p) * un;
}

// Whether the six node states of a midpoint are bit-identical (every plane of W).
template <int N, int D>
__device__ __forceinline__ bool uniform_nodes(const double* __restrict__ W, int64_t nc, const Nodes6& nd) {
  bool same = true;
#pragma unroll
  for (int m = 0; m < Lay<N, D>::M; ++m) {
    const long long b = __double_as_longlong(W[m * nc + nd.c[2]]);
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (j != 2) same &= __double_as_longlong(W[m * nc + nd.c[j]]) == b;
  }
  return same;
}

// ---------------------------------------------------------------- thermal relaxation (Sec. 4.2)

// Precision-form relaxation (FP64 throughout): the same root p* and T* as
// relax_cell, with the quadratic A_p p^2 + B_p p + C_p = 0 multiplied by rho^2
// so that its coefficients need no division:
//   rho^2 A_p = rho C_v,  rho^2 B_p = -(R_e R_m - p_inf,1 rho (C_v + rho_1' R_1)),
//   rho^2 C_p = -R_e p_inf,1 (R_m - rho_1' R_1),
// with C_v = sum alpha_k rho_k c_v,k, R_m = sum alpha_k rho_k (c_p,k - c_v,k),
// rho_1' = alpha_1 rho_1 (species `liq`) and R_e = rho (rho e~) =
// rho (E - sum alpha_k rho_k q_k) - |rho u|^2 / 2. With
// Y = rho_1' (p* + gamma_1 p_inf,1) c_v,1 + (C_v - rho_1' c_v,1)(p* + p_inf,1),
// Eq. T_relax_e gives T* = R_e (p* + p_inf,1) / (rho Y), and the relaxed volume
// fractions alpha_k = alpha_k rho_k R_k T* / (p* + p_inf,k) share one division
// z = R_e / (rho Y p*). Two divisions and one square root per cell. Returns rho
// and R_e for a primitive evaluation that follows. SOFT: products on the integer
// pipes (where the registers allow three blocks of 256 per SM, 1-4 % of a pass; in
// the batched stage kernel's 80 registers they cost 2 %).
template <int N, int D, bool SOFT = false>
__device__ __forceinline__ void relax_fast(double* W, const DevFluid& f, double& rho_out, double& Re_out) {
  using L = Lay<N, D>;
  const int l = f.liq;
  double rho = 0.0, Cv = 0.0, Rm = 0.0, rq = 0.0, m2 = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    rho += W[k];
    Cv = fma(W[k], f.cv[k], Cv);
    Rm = fma(W[k], f.Rg[k], Rm);
  }
  if (f.has_q) {
#pragma unroll
    for (int k = 0; k < N; ++k) rq = fma(W[k], f.q[k], rq);
  }
#pragma unroll
  for (int d = 0; d < D; ++d) m2 = fma(W[L::MOM + d], W[L::MOM + d], m2);
  auto mul = [](double x, double y) { return SOFT ? prod(x, y) : x * y; };
  const double Re = fma(rho, W[L::EN] - rq, -halved(m2));
  const double pinf1 = f.pinf[l], Wl = W[l], WlR1 = mul(Wl, f.Rg[l]);
  const double A = mul(rho, Cv);
  const double B = fma(mul(pinf1, rho), Cv + WlR1, -mul(Re, Rm));
  const double C = -mul(mul(Re, pinf1), Rm - WlR1);
  const double sq = rsqrt_r(fma(B, B, mul(soft::scale<2>(-A), C)));
  const bool pos = B > 0.0;
  const double ps = quot(pos ? soft::scale<1>(-C) : sq - B, pos ? B + sq : soft::scale<1>(A));
  const double ppl = ps + pinf1;
  const double Y = fma(mul(Wl, fma(f.gamma[l], pinf1, ps)), f.cv[l], mul(fma(-Wl, f.cv[l], Cv), ppl));
  const double z = quot(Re, mul(mul(rho, Y), ps));
#pragma unroll
  for (int k = 0; k < N - 1; ++k)
    // alpha_k = rho_k' R_k T* / (p* + p_inf,k), one stiffened gas at most
    W[L::AL + k] = mul(mul(mul(W[k], f.Rg[k]), k == l ? ps : ppl), z);
  rho_out = rho;
  Re_out = Re;
}

// Relaxed pressure p* of one cell: the positive root of A_p p^2 + B_p p + C_p = 0
// (Eqs. Ap_Bp_Cp_1-3, p_relax) in the cancellation-free form; its rho, rho e~, c_v
// and Y of species `liq`, the stiffened gas. (Callers that need no more stop here:
// the compiler leaves no out-of-line quotient out.)
template <int N, int D>
__device__ __forceinline__ double relaxed_p(const double* W, const DevFluid& f, double& rho, double& re, double& cvb,
                                            double& Yl) {
  const int l = f.liq;
  rho = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) rho += W[k];
  double Y[N];
#pragma unroll
  for (int k = 0; k < N; ++k) Y[k] = quot(W[k], rho);
  re = rhoe_tilde<N, D>(W, f);
  cvb = 0.0;
  double cpb = 0.0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    cvb += prod(Y[k], f.cv[k]);
    cpb += prod(Y[k], f.cp[k]);
  }
  Yl = Y[l];
  const double pinf1 = f.pinf[l], R1 = f.Rg[l];
  const double Ap = cvb, Rb = cpb - cvb, YR = prod(Yl, R1);
  const double Bp = -(prod(re, Rb) - prod(pinf1, cvb) - prod(prod(pinf1, Yl), R1));
  const double Cp = -prod(prod(re, pinf1), Rb - YR);
  const double sq = rsqrt_r(prod(Bp, Bp) - prod(soft::scale<2>(Ap), Cp));
  const bool pos = Bp > 0.0;
  return quot(pos ? soft::scale<1>(-Cp) : sq - Bp, pos ? Bp + sq : soft::scale<1>(Ap));
}

// p* and T* (Eq. T_relax_e).
template <int N, int D>
__device__ __forceinline__ void relaxed_pT(const double* W, const DevFluid& f, double& ps, double& Ts) {
  const int l = f.liq;
  double rho, re, cvb, Yl;
  ps = relaxed_p<N, D>(W, f, rho, re, cvb, Yl);
  const double pinf1 = f.pinf[l], pl = ps + pinf1;
  const double den = quot(prod(prod(Yl, ps + prod(f.gamma[l], pinf1)), f.cv[l]), pl) + cvb - prod(Yl, f.cv[l]);
  Ts = quot(quot(re, rho), den);
}

// Infinite-rate thermal relaxation of one cell: keeps alpha_k rho_k, rho u, E and
// replaces the stored alpha_k by rho Y_k / rho_k(p*, T*). FAST (precision form):
// relax_fast.
template <int N, int D, bool FAST = false>
__device__ __forceinline__ void relax_cell(double* W, const DevFluid& f) {
  if constexpr (FAST) {
    double rho, Re;
    relax_fast<N, D>(W, f, rho, Re);
    return;
  }
  double ps, Ts;
  relaxed_pT<N, D>(W, f, ps, Ts);
#pragma unroll
  for (int k = 0; k < N - 1; ++k) {
    const double rhok = quot(ps + f.pinf[k], prod(f.Rg[k], Ts));
    W[Lay<N, D>::AL + k] = quot(W[k], rhok);
  }
}

// Admissibility of a conservative state: bit 0 negative partial density, bit 1 a
// volume fraction outside [0, 1], bit 2 rho c^2 <= 0, bit 3 rho e~ <= 0 (NaN counts).
template <int N, int D>
__device__ __forceinline__ int admissibility_bits(const double* W, const DevFluid& f) {
  using L = Lay<N, D>;
  int b = 0;
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (!(W[k] >= 0.0)) b |= 1;
  double al[N];
  all_alpha_W<N, D>(W, al);
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (!(al[k] >= 0.0 && al[k] <= 1.0)) b |= 2;
  const double re = rhoe_tilde<N, D>(W, f);
  double S, P;
  mix_SP<double, N>(f, &W[L::AL], S, P);
  const double p = quot(re - P, S);
  if (!(rho_c2(S, P, p) > 0.0)) b |= 4;
  if (!(re > 0.0)) b |= 8;
  return b;
}

__device__ __forceinline__ void count_bits(StepState* st, int b) {
  if (b) {
    for (int i = 0; i < 4; ++i)
      if (b & (1 << i)) atomicAdd(&st->counts[i], 1ull);
  }
}

// ---------------------------------------------------------------- per-cell update

// The precision form's FP64 arithmetic writes its multiply-adds as explicit
// fma(): its translation units are built without FMA contraction, so that every
// FP32 expression rounds as written whichever kernel it is inlined into.

// Flux of a midpoint in the precision form where every FP32 plane holds the same
// value at the six nodes (as uniform_flux64 below for the FP64 form), from the planes
// of one of the cells (the HCS node-flux expression). Formed directly instead of through rounded steps that
// would only cancel; every FP32 sweep takes it, so they stay bit-identical.
// Planes as in P32Lay: V, then c, rho, rho c^2, rho u_d, E.
template <int N, int D>
__device__ __forceinline__ void uniform_flux32(int64_t c, int d, const float* __restrict__ P32, int64_t nc, double* G) {
  using L = Lay<N, D>;
  const float un = P32[(L::MOM + d) * nc + c], pn = P32[L::EN * nc + c];
#pragma unroll
  for (int m = 0; m < L::NC; ++m) {
    float v;
    if (m < L::MOM)
      v = P32[m * nc + c] * un;
    else if (m < L::EN)
      v = P32[(L::M + 3 + (m - L::MOM)) * nc + c] * un + ((m - L::MOM) == d ? pn : 0.f);
    else
      v = (P32[(L::M + 3 + D) * nc + c] + pn) * un;
    G[m] = widen_f32(v);
  }
}

// Precision form: W_out = a W^n + b (W_src + dt RHS) of one interior cell c,
// with W_src + dt RHS accumulated directly and dt/dx_d folded into one
// coefficient per direction (one multiply-add per slot and direction). Ws: the
// cell's W_src, already loaded. The SSP-RK stages that combine with W^n have
// b = 1 - a, so their combination is formed as acc + a (W^n - acc): two
// operations as before, and exactly acc when W^n equals acc. ub: the cell's
// uniform faces (k_mark), whose flux comes from the cell's own planes P32; two
// of them leave acc as it is (acc + cd 0 with cd < 0), unless kFluxOverflow says
// that their flux or cd may not be finite.
template <int N, int D>
__device__ __forceinline__ void fast_combine(int64_t c, const double* Wn, const double* Ws,
                                             const double* __restrict__ F0, const double* __restrict__ F1,
                                             const double* __restrict__ F2, const DevGrid& g, double dt, double a,
                                             double b, double* Wo, unsigned ub = 0u,
                                             const float* __restrict__ P32 = nullptr) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
  const int64_t nc = g.ncells;
  int64_t ijk[3];
  cell_index(g, c, ijk);
  const int64_t i0 = ijk[0], i1 = ijk[1], i2 = ijk[2];
  double acc[M];
#pragma unroll
  for (int m = 0; m < M; ++m) acc[m] = Ws[m];
  const unsigned both = (ub & kFluxOverflow) ? 0u : ub & ub >> 1;  // bit 2 d: both faces, their difference zero
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const unsigned u = ub >> (2 * d) & 3u;
    if (both >> (2 * d) & 1u) continue;
    const double cd = -dt * g.inv_dx[d];
    const double* F = d == 0 ? F0 : (d == 1 ? F1 : F2);
    const int64_t f0 = g.n[0] + (d == 0), f1 = g.n[1] + (d == 1), f2 = g.n[2] + (d == 2);
    const int64_t nf = f0 * f1 * f2;
    const int64_t fl = HRM_IDX(g, (i2 * f1 + i1) * f0 + i0, nf);
    const int64_t fr = HRM_IDX(g, fl + (d == 0 ? 1 : (d == 1 ? f0 : f0 * f1)), nf);
    double own[L::NC];
    if (u) uniform_flux32<N, D>(c, d, P32, nc, own);
    // G^-_{i+1/2} - G^+_{i-1/2}: the alpha slots of the right face use alpha_i
    // (planes AL..), those of the left face alpha_i as its right neighbour (planes M..)
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const double fo = m < L::NC ? own[m < L::NC ? m : 0] : 0.0;
      const double vl = (u & 1u) ? fo : F[(m < L::NC ? m : M + m - L::AL) * nf + fl];
      const double vr = (u & 2u) ? fo : F[m * nf + fr];
      acc[m] = fma(cd, vr - vl, acc[m]);
    }
  }
  if (a == 0.0 && b == 1.0) {
#pragma unroll
    for (int m = 0; m < M; ++m) Wo[m] = acc[m];
  } else if (a == 0.0) {
#pragma unroll
    for (int m = 0; m < M; ++m) Wo[m] = b * acc[m];
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) Wo[m] = fma(a, Wn[m * nc + c] - acc[m], acc[m]);
  }
}

// Whether every flux difference G^-_{i+1/2} - G^+_{i-1/2} of cell c is exactly
// +0: the two faces' values bit-equal and finite in every slot and direction.
// Integer compares only.
template <int N, int D>
__device__ __forceinline__ bool faces_unchanged(int64_t c, const double* __restrict__ F0,
                                                const double* __restrict__ F1, const double* __restrict__ F2,
                                                const DevGrid& g) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
  int64_t ijk[3];
  cell_index(g, c, ijk);
  const int64_t i0 = ijk[0], i1 = ijk[1], i2 = ijk[2];
  auto bits = [](double x) { return (unsigned long long)__double_as_longlong(x); };
  auto same_finite = [&](double x, double y) {
    const unsigned long long bx = bits(x);
    return (bx == bits(y)) & (((bx >> 52) & 0x7ffull) != 0x7ffull);
  };
  bool same = true;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const double* F = d == 0 ? F0 : (d == 1 ? F1 : F2);
    const int64_t f0 = g.n[0] + (d == 0), f1 = g.n[1] + (d == 1), f2 = g.n[2] + (d == 2);
    const int64_t nf = f0 * f1 * f2;
    const int64_t fl = HRM_IDX(g, (i2 * f1 + i1) * f0 + i0, nf);
    const int64_t fr = HRM_IDX(g, fl + (d == 0 ? 1 : (d == 1 ? f0 : f0 * f1)), nf);
#pragma unroll
    for (int m = 0; m < L::NC; ++m) same = same & same_finite(F[m * nf + fr], F[m * nf + fl]);
#pragma unroll
    for (int k = 0; k < N - 1; ++k) same = same & same_finite(F[(L::AL + k) * nf + fr], F[(M + k) * nf + fl]);
  }
  return same;
}

// Whether the first `slots` components of W_src of cell c are W^n's bit for bit,
// with none -0.
template <int N, int D>
__device__ __forceinline__ bool same_state(int64_t c, const double* Wn, const double* Ws, int64_t nc,
                                           int slots = Lay<N, D>::M) {
  bool same = true;
#pragma unroll
  for (int m = 0; m < Lay<N, D>::M; ++m) {
    if (m >= slots) continue;
    const unsigned long long bs = (unsigned long long)__double_as_longlong(Ws[m]);
    same = same & (bs == (unsigned long long)__double_as_longlong(Wn[m * nc + c])) & (bs != 0x8000000000000000ull);
  }
  return same;
}

// Precision form: whether a stage returns cell c exactly as it is, so that its
// arithmetic can be left out. Every flux difference G^-_{i+1/2} - G^+_{i-1/2}
// is exactly zero when the two faces' values are bit-equal and finite; a stage
// that combines with W^n (with_wn) also needs W_src bit-equal to W^n. Then
// fast_combine returns W_src exactly (its weights sum to one), except that a
// component -0 would come back +0, so those are left to the arithmetic; and
// relax_fast, which recomputes the volume fractions from the conserved
// variables alone, returns the cell unchanged if it came out of relax_fast
// before -- the caller's condition. Only integer compares: no FP64 work.
template <int N, int D>
__device__ __forceinline__ bool stage_keeps_cell(int64_t c, const double* Wn, const double* Ws,
                                                 const double* __restrict__ F0, const double* __restrict__ F1,
                                                 const double* __restrict__ F2, const DevGrid& g, bool with_wn) {
  const int64_t nc = g.ncells;
  return faces_unchanged<N, D>(c, F0, F1, F2, g) && (!with_wn || same_state<N, D>(c, Wn, Ws, nc));
}

// Flux of a midpoint whose six node states are bit-identical, from the state of
// one of its cells: the node's physical flux F^d (NC conservative slots; the alpha
// slots are zero). In exact arithmetic every step of the midpoint body returns it:
// constants are reproduced by the interpolation (App. C), the HLLC flux of equal
// states is their flux (Sec. 4.1.1), the HCS weights sum to one, alpha u - u alpha
// = 0 (Eq. G_pm), and the node state is the limiters' own candidate (Sec. 4.3.2).
template <int N, int D>
__device__ __forceinline__ void uniform_flux64(int64_t c, int d, const double* __restrict__ W,
                                               const double* __restrict__ V, int64_t nc, double* G) {
  using L = Lay<N, D>;
  const double un = V[(L::MOM + d) * nc + c], p = V[L::EN * nc + c];
#pragma unroll
  for (int m = 0; m < L::EN; ++m) {
    G[m] = prod(W[m * nc + c], un);
    if (m == L::MOM + d) G[m] = G[m] + p;
  }
  G[L::EN] = prod(W[L::EN * nc + c] + p, un);
}

// RHS_i = -sum_d (G^{d,-}_{i+1/2} - G^{d,+}_{i-1/2}) / dx_d (Eq. semi_W_G_pm_eqn),
// then W_out = a W^n + b (W_src + dt RHS) (SSP-RK stage in Shu-Osher form),
// optionally followed by the thermal relaxation and the admissibility count.
// MODE 1 writes RHS instead of the combination. In-place (W_out == W_src or W^n)
// is allowed: each thread reads its own cell before writing it.
// FAST (precision form): reciprocal of dx and of rho instead of divisions.
// uni (nullable): the cell's uniform faces (k_mark), whose flux is formed here
// from W_src and its primitives V and not read.
// One interior cell c < nint (Dirichlet slices keep their state).
template <int N, int D, int MODE, bool FAST = false>
__device__ __forceinline__ void update_body(int64_t c, const double* Wn, const double* Wsrc, double* Wout,
                                            const double* __restrict__ F0, const double* __restrict__ F1,
                                            const double* __restrict__ F2, const DevGrid& g, const DevFluid& f,
                                            StepState* st, double dt, double a, double b, int relax, int count,
                                            uint8_t* __restrict__ same = nullptr,
                                            const uint8_t* __restrict__ uni = nullptr,
                                            const double* __restrict__ V = nullptr, int src_relaxed = 0) {
  using L = Lay<N, D>;
  constexpr int M = L::M;
  const int64_t nc = g.ncells;
  int64_t ijk[3];
  cell_index(g, c, ijk);
  const int64_t i0 = ijk[0], i1 = ijk[1], i2 = ijk[2];
  double Ws[M];
#pragma unroll
  for (int m = 0; m < M; ++m) Ws[m] = Wsrc[m * nc + c];
  if constexpr (FAST && MODE == 0) {
    const bool with_wn = a != 0.0;
    if ((!relax || st->wn_relaxed) && stage_keeps_cell<N, D>(c, Wn, Ws, F0, F1, F2, g, with_wn)) {
      // W_out = W_src exactly; already there in place, or (with_wn) in W^n
      if (Wout != Wsrc && !(with_wn && Wout == Wn)) {
#pragma unroll
        for (int m = 0; m < M; ++m) Wout[m * nc + c] = Ws[m];
      }
      if (count) count_bits(st, admissibility_bits<N, D>(Ws, f));
      return;
    }
    double Wo[M];
    fast_combine<N, D>(c, Wn, Ws, F0, F1, F2, g, dt, a, b, Wo);
    if (relax) relax_cell<N, D, FAST>(Wo, f);
    if (count) count_bits(st, admissibility_bits<N, D>(Wo, f));
#pragma unroll
    for (int m = 0; m < M; ++m) Wout[m * nc + c] = Wo[m];
    return;
  }
  double rhs[M];
#pragma unroll
  for (int m = 0; m < M; ++m) rhs[m] = 0.0;
  const unsigned ub = uni ? uni[c] : 0u, both = (ub & kFluxOverflow) ? 0u : ub & ub >> 1;
  // flat: every flux difference is exactly +0 (the two faces' values bit-equal and finite)
  bool flat = true;
  auto differ = [](double x, double y) {
    const long long bx = __double_as_longlong(x);
    return (bx != __double_as_longlong(y)) | (((uint32_t)(bx >> 32) & 0x7ff00000u) == 0x7ff00000u);
  };
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const unsigned u = ub >> (2 * d) & 3u;
    if (both >> (2 * d) & 1u) continue;  // the cell's own flux twice, and rhs - 0 / dx = rhs
    const double* F = d == 0 ? F0 : (d == 1 ? F1 : F2);
    const int64_t f0 = g.n[0] + (d == 0), f1 = g.n[1] + (d == 1), f2 = g.n[2] + (d == 2);
    const int64_t nf = f0 * f1 * f2;
    const int64_t fl = HRM_IDX(g, (i2 * f1 + i1) * f0 + i0, nf);
    const int64_t fr = HRM_IDX(g, fl + (d == 0 ? 1 : (d == 1 ? f0 : f0 * f1)), nf);
    const double dx = g.dx[d], idx = g.inv_dx[d];
    // where dx is a power of two (a significand field of zero), 1/dx is exact and
    // df / dx and df * (1/dx) are the same correctly rounded number: the product
    // then stands for the quotient at no change of any result
    const bool scale = FAST || (__double_as_longlong(dx) & 0xFFFFFFFFFFFFFll) == 0;
    double own[L::NC];
    if (u) uniform_flux64<N, D>(c, d, Wsrc, V, nc, own);
    // G^-_{i+1/2} - G^+_{i-1/2}: the alpha slots of the right face use alpha_i
    // (planes AL..), those of the left face alpha_i as its right neighbour (planes M..)
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const double fo = m < L::NC ? own[m < L::NC ? m : 0] : 0.0;
      const double vl = (u & 1u) ? fo : F[(m < L::NC ? m : M + m - L::AL) * nf + fl];
      const double vr = (u & 2u) ? fo : F[m * nf + fr];
      flat = flat & !differ(vl, vr);
      const double df = vr - vl;
      rhs[m] = rhs[m] - (scale ? df * idx : quot(df, dx));
    }
  }
  if (MODE == 1) {
#pragma unroll
    for (int m = 0; m < M; ++m) Wout[m * nc + c] = rhs[m];
    return;
  }
  double Wo[M];
  if (a == 0.0) {
#pragma unroll
    for (int m = 0; m < M; ++m) Wo[m] = b * (Ws[m] + dt * rhs[m]);
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m) Wo[m] = a * Wn[m * nc + c] + b * (Ws[m] + dt * rhs[m]);
  }
  // relax_cell recomputes the volume fractions from the conserved variables
  // alone: where those are bit-equal to a state's that came out of relax_cell --
  // W_src from the second relaxed stage of a step on (src_relaxed), W^n by the
  // host's flag -- it would return that state's volume fractions, taken directly.
  bool keep = false;
  if (relax && flat) {
    auto conserved_as = [&](auto value) {
      bool k = true;
#pragma unroll
      for (int m = 0; m < L::NC; ++m) k = k & (__double_as_longlong(Wo[m]) == __double_as_longlong(value(m)));
      return k;
    };
    if (src_relaxed && conserved_as([&](int m) { return Ws[m]; })) {
      keep = true;
#pragma unroll
      for (int k = 0; k < N - 1; ++k) Wo[L::AL + k] = Ws[L::AL + k];
    } else if (st->wn_relaxed && conserved_as([&](int m) { return Wn[m * nc + c]; })) {
      keep = true;
#pragma unroll
      for (int k = 0; k < N - 1; ++k) Wo[L::AL + k] = Wn[(L::AL + k) * nc + c];
    }
  }
  if (relax && !keep) relax_cell<N, D, FAST>(Wo, f);
  if (count) count_bits(st, admissibility_bits<N, D>(Wo, f));
  if (same) {
    // the next stage's primitive pass keeps this cell's V and AUX where W_out is W_src
    bool eq = true;
#pragma unroll
    for (int m = 0; m < M; ++m) eq = eq & (__double_as_longlong(Wo[m]) == __double_as_longlong(Ws[m]));
    same[c] = eq ? 1 : 0;
  }
#pragma unroll
  for (int m = 0; m < M; ++m) Wout[m * nc + c] = Wo[m];
}

template <int N, int D, int MODE, bool FAST = false>
__global__ void __launch_bounds__(kCellThreads)
    k_update(const double* Wn, const double* Wsrc, double* Wout, const double* __restrict__ F0,
             const double* __restrict__ F1, const double* __restrict__ F2, DevGrid g, DevFluid f,
             StepState* st, double a, double b, int relax, int count, uint8_t* __restrict__ same = nullptr,
             const uint8_t* __restrict__ uni = nullptr, const double* __restrict__ V = nullptr, int src_relaxed = 0) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= g.nint) return;
  update_body<N, D, MODE, FAST>(c, Wn, Wsrc, Wout, F0, F1, F2, g, f, st, MODE == 1 ? 0.0 : st->dt, a, b, relax,
                                count, same, uni, V, src_relaxed);
}

}  // namespace hrm
