// Multi-shift CG on Mhat^dag Mhat (multishift.cu).
#pragma once
#include <cuda_runtime.h>

#include <string>

#include "jqcd.h"

namespace jqcd {

constexpr int kMsMaxShifts = 32;
constexpr int kMsBlock = 8;  // iterations between two updates of the shifted vectors

// Device-resident scalars of one multi-shift solve.
struct MsScalars {
  double rr, alpha, alpha_prev, beta, stop_rr, rhs2;
  double sigma[kMsMaxShifts], zeta_prev[kMsMaxShifts], zeta[kMsMaxShifts], zeta_next[kMsMaxShifts];
  double alpha_s[kMsMaxShifts], true_rr[kMsMaxShifts];
  int active[kMsMaxShifts], conv_iter[kMsMaxShifts];
  float2 alpha_dw;         // alpha as a (hi, lo) pair for the fused r update
  int nshift, iters, max_iters;
  int done;  // 1 every shift converged, 2 breakdown, 3 maxiter
  int halt;
};

// The shifted updates of the iterations since the last pass over the shifts:
// step j has x_i += alpha p_i (when xact) and p_i = zeta r_j + beta p_i (when
// pact), with the coefficients as (hi, lo) pairs.
struct MsSteps {
  float2 alpha[kMsBlock][kMsMaxShifts], zeta[kMsBlock][kMsMaxShifts], beta[kMsBlock][kMsMaxShifts];
  unsigned char xact[kMsBlock][kMsMaxShifts], pact[kMsBlock][kMsMaxShifts];
  int n;  // steps recorded
};

// The residual r_j of each recorded step.
struct MsResiduals {
  const float4 *r[kMsBlock];
};

// Per-shift solution and search direction (even parity, double-word).
struct MsVectors {
  float4 *x[kMsMaxShifts];
  float4 *p[kMsMaxShifts];
};

struct GaugeEntry;

cudaError_t launch_ms_start(const double *partials, int n, MsScalars *S, double tol2, int max_iters,
                            cudaStream_t s);
// alpha from the per-hop-block partials of ||Mhat p||^2; slot: this
// iteration's place among the steps (0 starts a new record).
cudaError_t launch_ms_alpha(const double *partials, int nhop, MsScalars *S, MsSteps *B, int slot, cudaStream_t s);
// beta from the per-hop-block partials of ||r||^2 and the record of the
// shifted updates (step slot), then p = r + beta p.
cudaError_t launch_ms_beta_p(const double *partials, int nhop, int nblas, MsScalars *S, MsSteps *B, int slot,
                             const float4 *r, float4 *pb, int64_t n, cudaStream_t s);
// The recorded updates of every shift, in one pass over x_i and p_i.
cudaError_t launch_ms_steps(const MsVectors &V, const MsResiduals &R, const MsScalars *S, const MsSteps *B, int nblas,
                            int64_t n, cudaStream_t s);
cudaError_t launch_ms_resid(const float4 *rhs, const float4 *Ax, const float4 *x, double sigma, int64_t n,
                            double *partials, int nblocks, cudaStream_t s);

// Solve (Mhat^dag Mhat + shifts[i]) x_i = rhs for the double-word even-parity
// rhs in G.vrhs (even half); x_even[i]: caller's even-parity buffers.
jqcd_status solve_multishift(GaugeEntry &G, const jqcd_solve_params &P, int nshift, const double *shifts,
                             float4 *const *x_even, cudaStream_t s, jqcd_solve_info *infos,
                             std::string *msg);

}  // namespace jqcd
