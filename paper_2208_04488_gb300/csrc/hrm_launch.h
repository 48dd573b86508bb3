// Host-side launchers of the kernel templates, one table per (N, D), so that
// the C-ABI layer dispatches at run time and the heavy instantiations compile
// in separate translation units.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "hrm_device.cuh"

namespace hrm {

struct CellKernels {
  // P32 (nullable): FP32 planes for the precision form; R32 (nullable): FP32
  // rounding residues of rho, u_d, p for the learned gate
  // same (nullable; ignored with tau): per interior cell, nonzero where W is bit
  // for bit the state V, AUX, P32, R32 were computed from -- those cells are kept
  void (*prim)(const double* W, double* V, double* AUX, float* P32, float* R32, const DevGrid&, const DevFluid&,
               StepState*, int tau, const uint8_t* same, cudaStream_t);
  void (*ic)(const double* prim, double* W, const DevGrid&, const DevFluid&, int64_t c0, int64_t c1, cudaStream_t);
  void (*relax)(double* W, const DevGrid&, const DevFluid&, cudaStream_t);
  void (*fields)(const double* W, double* out, int field, const DevGrid&, const DevFluid&, cudaStream_t);
  void (*admiss)(const double* W, const DevGrid&, const DevFluid&, StepState*, cudaStream_t);
};

// Smoothness gate of a midpoint sweep: `fixed` (nullable) one byte per
// midpoint, nonzero = linear WENO weights there (a caller's fixed gate, or the
// bytes the learned detector's gate kernel wrote before the sweep).
struct GateArgs {
  const uint8_t* fixed = nullptr;
  // precision form with screens: the sweep defers midpoints whose screens fail
  // to a second kernel through this worklist (one entry per midpoint of the
  // direction; counted in list_cnt[2]); nullptr: one kernel with the fallbacks inline
  uint32_t* defer_list = nullptr;
  // optional: run the deferred midpoints on `side` (after ev_fast, recorded on
  // the sweep's stream) and record ev_fix there, so that they overlap the next
  // sweep; the caller joins ev_fix before the update
  cudaStream_t side = nullptr;
  cudaEvent_t ev_fast = nullptr, ev_fix = nullptr;
  cudaEvent_t prof_fix[2] = {nullptr, nullptr};  // profiling: recorded around it
  // precision form with the learned detector (with a worklist): the sweep
  // evaluates the network itself (k_face32_net) from the FP32 planes and their
  // residues R32, with the detector's inference blob (an mlp::GateBlob) and the
  // logit threshold, and writes its gate bytes to `out_gate` (which the
  // deferred-midpoint kernel then reads as `fixed`)
  const void* net = nullptr;
  const float* R32 = nullptr;
  float zthr = 0.f;
  uint8_t* out_gate = nullptr;
  // the midpoints to sweep (nullptr: all of the direction) and their counters
  // (SweepLists of the direction; without a list, list_cnt[2] must be 0)
  const uint32_t* list = nullptr;
  uint32_t* list_cnt = nullptr;
};

// Stream of the deferred-midpoint kernel: gate.side (forked from s after the
// sweep) or s itself.
inline cudaStream_t fix_stream(const GateArgs& gate, cudaStream_t s) {
  if (!gate.side) return s;
  cudaEventRecord(gate.ev_fast, s);
  cudaStreamWaitEvent(gate.side, gate.ev_fast, 0);
  if (gate.prof_fix[0]) cudaEventRecordWithFlags(gate.prof_fix[0], gate.side, cudaEventRecordExternal);
  return gate.side;
}
inline void fix_done(const GateArgs& gate) {
  if (!gate.side) return;
  if (gate.prof_fix[1]) cudaEventRecordWithFlags(gate.prof_fix[1], gate.side, cudaEventRecordExternal);
  cudaEventRecord(gate.ev_fix, gate.side);
}

// Launch shape of the deferred-midpoint kernel: one-warp blocks, 16 per SM.
constexpr int kFixBlocks = 2432;
constexpr int kFixThreads = 32;

struct FaceKernels {
  // precision: 0 FP64, 1 FP32 bulk
  void (*face[3])(int precision, const double* W, const double* V, const double* AUX, const float* P32,
                  double* out, const DevGrid&, const DevFluid&, const DevParams&, const StepState*,
                  const GateArgs& gate, cudaStream_t);
  // mode 0: RK combination, mode 1: write the RHS; fast: precision-form variant;
  // same (nullable; FP64 RK combination): per interior cell, set to 1 where
  // W_out equals W_src bit for bit, else 0; uni (nullable; FP64 RK combination):
  // the cells' uniform faces, whose fluxes are formed from W_src and V; src_relaxed:
  // every interior cell of W_src came out of the form's relaxation
  void (*update)(int mode, int fast, const double* Wn, const double* Wsrc, double* Wout, const double* F0,
                 const double* F1, const double* F2, const DevGrid&, const DevFluid&, StepState*, double a,
                 double b, int relax, int count, uint8_t* same, const uint8_t* uni, const double* V, int src_relaxed, cudaStream_t);
};

const CellKernels* cell_kernels(int N, int D);
const FaceKernels* face_kernels(int N, int D);
const FaceKernels* face_kernels_d1(int N);
const FaceKernels* face_kernels_d2(int N);
const FaceKernels* face_kernels_d3(int N);

// FP32-bulk midpoint kernels, compiled in their own units (with FMA contraction).
void update32_d1(int N, const double* Wn, const double* Wsrc, double* Wout, const double* F0, const double* F1,
                 const double* F2, const DevGrid&, const DevFluid&, StepState*, double a, double b, int relax,
                 int count, cudaStream_t);
void face32_d1(int N, int dir, const double* W, const double* V, const double* AUX, const float* P32, double* out,
               const DevGrid&, const DevFluid&, const DevParams&, const StepState*, const GateArgs& gate,
               cudaStream_t);
void update32_d2(int N, const double* Wn, const double* Wsrc, double* Wout, const double* F0, const double* F1,
                 const double* F2, const DevGrid&, const DevFluid&, StepState*, double a, double b, int relax,
                 int count, cudaStream_t);
void face32_d2(int N, int dir, const double* W, const double* V, const double* AUX, const float* P32, double* out,
               const DevGrid&, const DevFluid&, const DevParams&, const StepState*, const GateArgs& gate,
               cudaStream_t);
void update32_d3(int N, const double* Wn, const double* Wsrc, double* Wout, const double* F0, const double* F1,
                 const double* F2, const DevGrid&, const DevFluid&, StepState*, double a, double b, int relax,
                 int count, cudaStream_t);
void face32_d3(int N, int dir, const double* W, const double* V, const double* AUX, const float* P32, double* out,
               const DevGrid&, const DevFluid&, const DevParams&, const StepState*, const GateArgs& gate,
               cudaStream_t);

// Precision-form update fused with the next stage's FP32 planes (hrm_face32_dD.cu):
// phase 0 finishes the unchanged cells and lists the others (any time after the
// lists were built, beside the sweeps), phase 1 updates the listed ones. tau: also
// accumulate the CFL maxima of W_out into st->tau_bits (a step's last stage; grids
// without Dirichlet slices, five-equation sound speed).
struct Update32Args {
  const double* Wn;
  const double* Wsrc;
  double* Wout;
  const double* F0;
  const double* F1;
  const double* F2;
  StepState* st;
  double a, b;
  int relax, count;
  float* P32;
  float* R32;
  const uint8_t* uni;  // nullable: the cells' uniform faces (k_mark; their fluxes are not read)
  int src_relaxed;     // W_src came out of the form's relaxation (a step's second relaxed stage on)
};
void update32p_d1(int N, const Update32Args& A, const DevGrid&, const DevFluid&, int tau, const SweepLists&, int phase,
                  cudaStream_t);
void update32p_d2(int N, const Update32Args& A, const DevGrid&, const DevFluid&, int tau, const SweepLists&, int phase,
                  cudaStream_t);
void update32p_d3(int N, const Update32Args& A, const DevGrid&, const DevFluid&, int tau, const SweepLists&, int phase,
                  cudaStream_t);
inline void launch_update32p(int N, int D, const Update32Args& A, const DevGrid& g, const DevFluid& f, int tau,
                             const SweepLists& lists, int phase, cudaStream_t s) {
  if (D == 1) update32p_d1(N, A, g, f, tau, lists, phase, s);
  if (D == 2) update32p_d2(N, A, g, f, tau, lists, phase, s);
  if (D == 3) update32p_d3(N, A, g, f, tau, lists, phase, s);
}

// Primitive kernel of the precision form (FP32 planes only; hrm_face32_dD.cu).
void prim32_d1(int N, const double* W, float* P32, float* R32, const DevGrid&, const DevFluid&, StepState*, int tau,
               cudaStream_t);
void prim32_d2(int N, const double* W, float* P32, float* R32, const DevGrid&, const DevFluid&, StepState*, int tau,
               cudaStream_t);
void prim32_d3(int N, const double* W, float* P32, float* R32, const DevGrid&, const DevFluid&, StepState*, int tau,
               cudaStream_t);
inline void launch_prim32(int N, int D, const double* W, float* P32, float* R32, const DevGrid& g, const DevFluid& f,
                          StepState* st, int tau, cudaStream_t s) {
  if (D == 1) prim32_d1(N, W, P32, R32, g, f, st, tau, s);
  if (D == 2) prim32_d2(N, W, P32, R32, g, f, st, tau, s);
  if (D == 3) prim32_d3(N, W, P32, R32, g, f, st, tau, s);
}

void launch_finalize(StepState* st, const DevGrid& g, int D, double cfl, int mode, cudaStream_t s);
void launch_set_dt(StepState* st, double dt, cudaStream_t s);

inline unsigned grid_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Threads per block of a kernel with a thread per cell and FP64 work: 256, or 64
// where blocks of 256 would leave every other SM idle (a warp alone on its SM issues
// an FP64 instruction every 64 cycles, eight share the unit at 19 each). Measured us
// per step with 64 | 256: precision form 90x90 103 | 112, 128x64 175 | 179; 256x128
// 196 | 190.
inline unsigned cell_threads(long long n) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return n < 128ll * sms ? 64u : 256u;
}

// Uniform faces and the lists of the other midpoints of a stage's source state
// (hrm_sweep.cuh): two launches. P32 NULL: the FP64 form, from W and V; else the
// precision form, from its FP32 planes.
void launch_mark(int N, int D, const double* W, const double* V, const float* P32, const DevGrid& g,
                 const SweepLists& lists, cudaStream_t s);

// Blocks for up to n items of a list that its warps take from a counter: what is
// resident at per_sm blocks on each SM, or fewer where n needs no more.
inline unsigned resident_grid(long long n, int threads, int per_sm) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long all = (n + threads - 1) / threads, fit = (long long)(sms > 0 ? sms : 1) * per_sm;
  return (unsigned)(all < fit ? all : fit);
}

// Blocks of kFaceThreads with a thread per midpoint of a direction.
inline unsigned all_grid(const DevGrid& g, int dir) {
  return grid_for((g.n[0] + (dir == 0)) * (g.n[1] + (dir == 1)) * (g.n[2] + (dir == 2)), 128);
}

// Blocks of kFaceThreads of a list-driven sweep at `lanes` threads per midpoint.
inline unsigned list_grid(const DevGrid& g, int dir, int per_sm, int lanes = 1) {
  const long long f = (g.n[0] + (dir == 0)) * (g.n[1] + (dir == 1)) * (g.n[2] + (dir == 2));
  return resident_grid(f * lanes, 128, per_sm);
}

// Smallest float not below x (thresholds of the FP32 screens).
inline float float_up(double x) {
  float f = (float)x;
  if ((double)f < x) f = std::nextafter(f, INFINITY);
  return f;
}

// The screens certify "theta = 1 and no hard switch" from "every checked
// quantity >= its limiter threshold", which implies the hard-switch tests only
// when each hard-switch threshold is at most the limiter threshold.
inline void fill_screen(DevParams& d, int requested) {
  d.screen = requested && d.hs_ar <= d.eps_ar && d.hs_a <= d.eps_a && d.hs_rhoe <= d.eps_rhoe;
  d.eps_ar_f = float_up(d.eps_ar);
  d.eps_rhoe_f = float_up(d.eps_rhoe);
  d.hs_rc2_f = float_up(d.hs_rc2);
  d.eps_a_mf = float_up(d.eps_a + 1e-13);
  d.weno_eps_f = (float)d.weno_eps;
  d.Cs_f = (float)d.Cs;
  d.pad_ = 0;
}

}  // namespace hrm
