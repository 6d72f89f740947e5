// Multi-shift conjugate gradient: (A + sigma_i) x_i = rhs for all shifts at
// once, A = Mhat^dag Mhat on the even sites, in double-word arithmetic (the
// rational approximations of RHMC; the paper lists RHMC among its
// algorithms, section on the package's features).
//
// All shifted systems share the Krylov space of the unshifted CG: the shifted
// residuals are collinear, r_i = zeta_i r, so one operator application per
// iteration serves every shift.  With alpha, beta of the unshifted CG and
// zeta_i^{-1} = zeta_i^0 = 1, alpha^{-1} = 1, beta^{-1} = 0 (Jegerlehner's
// recurrences, written for A + sigma):
//   zeta_i^{k+1} = zeta_i^k zeta_i^{k-1} alpha^{k-1} /
//                  [alpha^k beta^{k-1} (zeta_i^{k-1} - zeta_i^k) + zeta_i^{k-1} alpha^{k-1} (1 + sigma_i alpha^k)]
//   alpha_i^k = alpha^k zeta_i^{k+1} / zeta_i^k,   x_i += alpha_i^k p_i
//   beta_i^k  = beta^k (zeta_i^{k+1} / zeta_i^k)^2, p_i = zeta_i^{k+1} r + beta_i^k p_i
// Shift i stops (x_i frozen) once |zeta_i| |r| <= tol |rhs|; the loop ends
// when every shift has.  Scalars live on the device; the host polls.
//
// The shifted recurrences never feed back into the base one, so their vectors
// are not touched in every iteration: up to kMsBlock residuals r_j are kept,
// the coefficients of each step are recorded, and one pass then applies all
// the recorded steps to x_i and p_i in registers (the same operations in the
// same order, so the same bits).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "dw.cuh"
#include "dw2.cuh"
#include "kernels.h"
#include "multishift.h"
#include "pdl.cuh"
#include "reduce.cuh"
#include "solver.h"

namespace jqcd {

namespace {

constexpr int kMsCheckEvery = 8;

__device__ __forceinline__ dw dw_from_double(double v) {
  const float h = __double2float_rn(v);
  return dw_make(h, __double2float_rn(v - (double)h));
}

__global__ void ms_start_kernel(const double *partials, int n, MsScalars *S, double tol2, int max_iters) {
  const double rhs2 = block_sum_partials(partials, n);
  if (threadIdx.x == 0) {
    S->rhs2 = rhs2;
    S->rr = rhs2;
    S->stop_rr = tol2 * rhs2;
    S->alpha = 0.0;
    S->alpha_prev = 1.0;
    S->beta = 0.0;
    S->iters = 0;
    S->max_iters = max_iters;
    S->done = 0;
    S->halt = 0;
    for (int i = 0; i < S->nshift; ++i) {
      S->zeta_prev[i] = S->zeta[i] = S->zeta_next[i] = 1.0;
      S->alpha_s[i] = 0.0;
      S->active[i] = rhs2 > 0.0;
      S->conv_iter[i] = 0;
    }
    if (!(rhs2 > 0.0)) {
      S->done = 1;
      S->halt = 1;
    }
  }
}

// Thread i takes the recurrences of shift i (a loop over the shifts in one
// thread put its chain of FP64 divisions on the iteration's critical path:
// 11.9 us per step for 8 shifts).
__global__ void ms_alpha_kernel(const double *partials, int n, MsScalars *S, MsSteps *B, int slot) {
  __shared__ double sh_pap;
  pdl_enter();
  if (slot == 0 && threadIdx.x == 0) B->n = 0;  // the last record has been applied
  const int i = threadIdx.x;
  const bool mine = i < S->nshift;
  // what the step reads, loaded beside the partials
  const int halt = S->halt, act = mine ? S->active[i] : 0;
  const double rr = S->rr, ap = S->alpha_prev, b = S->beta;
  const double z = mine ? S->zeta[i] : 1.0, zp = mine ? S->zeta_prev[i] : 1.0, sigma = mine ? S->sigma[i] : 0.0;
  const double v = block_sum_partials(partials, n);
  if (halt) return;
  if (threadIdx.x == 0) sh_pap = v;
  __syncthreads();
  if (i > 0 && !act) return;
  const double pAp = sh_pap;
  if (!(pAp > 0.0) || !isfinite(pAp)) {
    if (threadIdx.x == 0) { S->done = 2; S->halt = 1; }
    return;
  }
  const double a = rr / pAp;
  if (act) {
    const double zn = z * zp * ap / (a * b * (zp - z) + zp * ap * (1.0 + sigma * a));
    S->zeta_next[i] = zn;
    S->alpha_s[i] = a * zn / z;
  }
  if (i == 0) {
    S->alpha = a;
    const float ah = __double2float_rn(a);
    S->alpha_dw = make_float2(ah, __double2float_rn(a - (double)ah));
  }
}

__device__ __forceinline__ float2 split_pair(double v) {
  const float h = __double2float_rn(v);
  return make_float2(h, __double2float_rn(v - (double)h));
}

__global__ void ms_beta_kernel(const double *partials, int n, MsScalars *S, MsSteps *B, int slot) {
  __shared__ double sh_rr;
  pdl_enter();
  const int i = threadIdx.x;
  const bool mine = i < S->nshift;
  // what the step reads, loaded beside the partials
  const int halt = S->halt, iter = S->iters + 1;
  const bool last = iter >= S->max_iters, act = mine && S->active[i] != 0;
  const double rr = S->rr, stop_rr = S->stop_rr;
  const double z = mine ? S->zeta[i] : 1.0, zn = mine ? S->zeta_next[i] : 1.0, as = mine ? S->alpha_s[i] : 0.0;
  const double v = block_sum_partials(partials, n);
  if (halt) return;
  if (threadIdx.x == 0) sh_rr = v;
  __syncthreads();
  const double rr_new = sh_rr;
  const bool finite = isfinite(rr_new);
  const double b = mine || i == 0 ? rr_new / rr : 0.0;
  int running = 0;  // this thread's shift goes on
  if (finite && mine) {
    float2 al = make_float2(0.f, 0.f), ze = al, be = al;
    if (act) {
      al = split_pair(as);
      ze = split_pair(zn);
      be = split_pair(b * (zn / z) * (zn / z));
      S->zeta_prev[i] = z;
      S->zeta[i] = zn;
      if (zn * zn * rr_new <= stop_rr) {
        S->active[i] = 0;
        S->conv_iter[i] = iter;
      } else {
        running = 1;
      }
    }
    B->alpha[slot][i] = al;
    B->zeta[slot][i] = ze;
    B->beta[slot][i] = be;
    B->xact[slot][i] = act;
    B->pact[slot][i] = running && !last;
  }
  const int any = __syncthreads_or(running);  // every read of S->rr, S->iters is above
  if (threadIdx.x == 0) {
    S->iters = iter;
    if (!finite) { S->done = 2; S->halt = 1; return; }
    B->n = slot + 1;
    S->beta = b;
    S->alpha_prev = S->alpha;
    S->rr = rr_new;
    if (!any) { S->done = 1; S->halt = 1; }
    else if (last) { S->done = 3; S->halt = 1; }
  }
}

// p = r + beta p of the base system
__global__ void ms_p_kernel(float4 *__restrict__ pb, const float4 *__restrict__ r, int64_t n, const MsScalars *S) {
  pdl_enter();
  if (S->halt) return;  // uniform across the grid
  const dw beta = dw_from_double(S->beta);
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    dw rr, ri, pr, pi;
    dwc_unpack(r[q], rr, ri);
    dwc_unpack(pb[q], pr, pi);
    pb[q] = dwc_pack(dw_add(rr, dw_mul(beta, pr)), dw_add(ri, dw_mul(beta, pi)));
  }
}

__device__ __forceinline__ p2 ld_chunk(const float4 *p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
  return p2{v.x, v.y};
}
__device__ __forceinline__ mul2 bcast(float2 c) { return mul2{f2_make(c.x, c.x), f2_make(c.y, c.y)}; }
// c v for a real double-word scalar c, normalised (dw_mul on both lanes)
__device__ __forceinline__ p2 p2_scale(const mul2 &c, p2 v) { return p2_norm(acc2_get(acc2_first(c, v))); }

// The recorded steps of every shift: per element, the residuals of the block
// are loaded once, then x_i and p_i of each shift are read, taken through all
// the steps in registers and written back.  An update in every iteration
// moved 4 streams per running shift each time and was bound by HBM (285.6 us
// an iteration for 8 shifts at 24^3x48); a block of eight moves them once (610
// us, 76 us an iteration) and the solve went from 56.2 to 40.7 ms.
__global__ void __launch_bounds__(kBlasThreads)
    ms_steps_kernel(MsVectors V, MsResiduals R, int64_t n, const MsScalars *__restrict__ S,
                    const MsSteps *__restrict__ B) {
  __shared__ float4 cp[kMsMaxShifts][kMsBlock];  // (zeta, beta) of a step
  __shared__ float2 cx[kMsMaxShifts][kMsBlock];  // alpha
  __shared__ int nx[kMsMaxShifts], np[kMsMaxShifts];  // steps of x_i and of p_i (each shift's come first)
  pdl_enter();
  const int m = B->n;
  if (m == 0) return;  // uniform across the grid
  const int ns = S->nshift;
  for (int t = threadIdx.x; t < ns * m; t += blockDim.x) {
    const int i = t / m, j = t % m;
    const float2 z = B->zeta[j][i], b = B->beta[j][i];
    cp[i][j] = make_float4(z.x, z.y, b.x, b.y);
    cx[i][j] = B->alpha[j][i];
  }
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    int a = 0, c = 0;
    for (int j = 0; j < m; ++j) {
      a += B->xact[j][i];
      c += B->pact[j][i];
    }
    nx[i] = a;
    np[i] = c;
  }
  __syncthreads();
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    p2 r[kMsBlock];
#pragma unroll
    for (int j = 0; j < kMsBlock; ++j) r[j] = j < m ? ld_chunk(R.r[j] + q) : p2{0ull, 0ull};
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
      const int a = nx[i], c = np[i];
      if (a == 0) continue;
      float4 *xp = V.x[i] + q, *pp = V.p[i] + q;
      p2 x = ld_chunk(xp), p = ld_chunk(pp);
#pragma unroll
      for (int j = 0; j < kMsBlock; ++j) {
        if (j >= a) break;  // uniform over the block
        x = p2_norm(p2_add(x, p2_scale(bcast(cx[i][j]), p)));
        if (j < c) {
          const float4 w = cp[i][j];
          p = p2_norm(p2_add(p2_scale(bcast(make_float2(w.x, w.y)), r[j]),
                             p2_scale(bcast(make_float2(w.z, w.w)), p)));
        }
      }
      *reinterpret_cast<ulonglong2 *>(xp) = make_ulonglong2(x.h, x.l);
      if (c > 0) *reinterpret_cast<ulonglong2 *>(pp) = make_ulonglong2(p.h, p.l);
    }
  }
}

// r = rhs - Ax - sigma x, per-block partials of ||r||^2 (true residual).
__global__ void ms_resid_kernel(const float4 *__restrict__ rhs, const float4 *__restrict__ Ax,
                                const float4 *__restrict__ x, double sigma, int64_t n, double *partials) {
  const dw ms = dw_from_double(-sigma);
  dwacc A{0.f, 0.f};
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    dw br, bi, yr, yi, xr, xi;
    dwc_unpack(rhs[q], br, bi);
    dwc_unpack(Ax[q], yr, yi);
    dwc_unpack(x[q], xr, xi);
    const dw re = dw_add(dw_add(br, dw_neg(yr)), dw_mul(ms, xr));
    const dw im = dw_add(dw_add(bi, dw_neg(yi)), dw_mul(ms, xi));
    acc_sq(A, re);
    acc_sq(A, im);
  }
  const double s = block_sum_dw(A);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

}  // namespace

cudaError_t GaugeEntry::ensure_multishift(int nshift) {
  cudaError_t e = ensure_solver();
  const size_t half = spinor_parity_bytes(PREC_DW, g.vh);
  while (e == cudaSuccess && (int)ms_p.size() < nshift) {
    float4 *p = nullptr;
    e = alloc_t(&p, half);
    if (e == cudaSuccess) ms_p.push_back(p);
  }
  if (e == cudaSuccess && !ms_S) e = alloc_t(&ms_S, sizeof(MsScalars));
  if (e == cudaSuccess && !ms_B) e = alloc_t(&ms_B, sizeof(MsSteps));
  if (e == cudaSuccess && !ms_S_host) e = cudaMallocHost(&ms_S_host, sizeof(MsScalars));
  return e;
}

jqcd_status solve_multishift(GaugeEntry &G, const jqcd_solve_params &P, int nshift, const double *shifts,
                             float4 *const *x_even, cudaStream_t s, jqcd_solve_info *infos,
                             std::string *msg) {
#define CKM(call)                                                            \
  do {                                                                       \
    cudaError_t e_ = (call);                                                 \
    if (e_ != cudaSuccess) {                                                 \
      *msg = cudaGetErrorString(e_);                                         \
      return e_ == cudaErrorMemoryAllocation ? JQCD_ENOMEM : JQCD_ECUDA;     \
    }                                                                        \
  } while (0)
  if (nshift < 1 || nshift > kMsMaxShifts) {
    *msg = "nshift must lie in [1, 32]";
    return JQCD_EINVAL;
  }
  for (int i = 0; i < nshift; ++i)
    if (!(shifts[i] >= 0.0) || !std::isfinite(shifts[i])) {
      *msg = "shifts must be finite and >= 0 (A + sigma must stay positive definite)";
      return JQCD_EINVAL;
    }
  if (!(P.tol > 0.0) || P.maxiter < 1 || !(P.kappa >= 0.0) || !P.eo || P.mode != JQCD_CG_DW) {
    *msg = "multi-shift CG: eo = 1, mode JQCD_CG_DW, tol > 0, maxiter >= 1, kappa >= 0";
    return JQCD_EINVAL;
  }
  CKM(G.ensure_multishift(nshift));
  const int64_t vh = G.g.vh;
  const int64_t n = 12 * vh;  // complex double-word numbers of one parity
  const int nblas = (int)blas_blocks(n);
  const int nhop = (int)dw_hop_blocks(vh);  // partials of the double-word hops
  float4 *rhs = G.vec_even(G.vrhs), *pb = G.vec_even(G.vp), *Ap = G.vec_even(G.vAp);
  // step j of a block writes its residual to ring[j]: r, and the halves of the
  // solver's vectors that the iterations leave alone (Ap is formed after them)
  float4 *const ring[] = {G.vec_odd(G.vr), G.vec_odd(G.vp),   G.vec_even(G.vAp),  G.vec_odd(G.vAp),
                          G.vec_odd(G.vw), G.vec_even(G.vt), G.vec_odd(G.vrhs), G.vec_even(G.vr)};
  static_assert(sizeof ring / sizeof ring[0] == kMsBlock, "a place for each residual of a block");
  static_assert(kMsCheckEvery % kMsBlock == 0, "x_i is final when the solve has halted");
  MsResiduals R;
  for (int j = 0; j < kMsBlock; ++j) R.r[j] = ring[j];
  const float4 *r_last = ring[kMsBlock - 1];  // the newest residual
  MsSteps *B = G.ms_B;
  MsVectors V;
  memset(&V, 0, sizeof V);
  for (int i = 0; i < nshift; ++i) {
    V.x[i] = x_even[i];
    V.p[i] = G.ms_p[i];
  }
  MsScalars *S = G.ms_S;
  MsScalars *H = G.ms_S_host;
  memset(H, 0, sizeof(MsScalars));
  H->nshift = nshift;
  for (int i = 0; i < nshift; ++i) H->sigma[i] = shifts[i];
  CKM(cudaEventRecord(G.ev0, s));
  CKM(cudaMemcpyAsync(S, H, sizeof(MsScalars), cudaMemcpyHostToDevice, s));
  CKM(launch_dw_norm2(rhs, n, G.partials, s));
  CKM(launch_ms_start(G.partials, nblas, S, P.tol * P.tol, P.maxiter, s));
  CKM(cudaMemsetAsync(&B->n, 0, sizeof B->n, s));
  CKM(launch_dw_copy(ring[kMsBlock - 1], rhs, n, s));
  CKM(launch_dw_copy(pb, rhs, n, s));
  for (int i = 0; i < nshift; ++i) {
    CKM(launch_dw_copy(V.p[i], rhs, n, s));
    CKM(launch_dw_zero(V.x[i], n, s));
  }
  // One iteration: t = H_oe p; w = p - k^2 H_eo t with ||w||^2 = <p, Mhat^dag Mhat p>;
  // alpha; t = H^dag_oe w; the last hop forms Ap at its site and applies
  // r -= alpha Ap with ||r||^2 (Ap is not stored); beta; p = r + beta p.
  const double k2 = -P.kappa * P.kappa;
  float4 *t = G.vec_odd(G.vt), *w = G.vec_even(G.vw);
  auto iteration = [&](int slot) -> cudaError_t {
    float4 *r = ring[slot];
    HopParams H = G.hop_params(PREC_DW, 1, pb, nullptr, t, 0.0, 1.0, nullptr);
    H.guard = &S->halt;
    cudaError_t e = launch_hop(PREC_DW, H, false, false, false, s);
    if (e) return e;
    H = G.hop_params(PREC_DW, 0, t, pb, w, 1.0, k2, G.partials);
    H.guard = &S->halt;
    if ((e = launch_hop(PREC_DW, H, false, true, true, s))) return e;
    // the alpha step runs on the side stream beside t = H^dag_oe w, which
    // does not read it; the last hop waits for it
    if (G.side) {
      if ((e = cudaEventRecord(G.ev_fork, s))) return e;
      if ((e = cudaStreamWaitEvent(G.side, G.ev_fork, 0))) return e;
      if ((e = launch_ms_alpha(G.partials, nhop, S, B, slot, G.side))) return e;
      if ((e = cudaEventRecord(G.ev_join, G.side))) return e;
    } else if ((e = launch_ms_alpha(G.partials, nhop, S, B, slot, s))) {
      return e;
    }
    H = G.hop_params(PREC_DW, 1, w, nullptr, t, 0.0, 1.0, nullptr);
    H.guard = &S->halt;
    if ((e = launch_hop(PREC_DW, H, true, false, false, s))) return e;
    if (G.side && (e = cudaStreamWaitEvent(s, G.ev_join, 0))) return e;
    H = G.hop_params(PREC_DW, 0, t, w, nullptr, 1.0, k2, G.partials);
    H.guard = &S->halt;
    if ((e = launch_hop_dw_r(H, r_last, r, &S->alpha_dw, s))) return e;
    r_last = r;
    return launch_ms_beta_p(G.partials, nhop, nblas, S, B, slot, r, pb, n, s);
  };
  for (;;) {
    for (int k = 0; k < kMsCheckEvery; ++k) {
      const int slot = k % kMsBlock;
      CKM(iteration(slot));
      if (slot + 1 == kMsBlock) CKM(launch_ms_steps(V, R, S, B, nblas, n, s));
    }
    CKM(cudaMemcpyAsync(H, S, sizeof(MsScalars), cudaMemcpyDeviceToHost, s));
    CKM(cudaStreamSynchronize(s));
    if (P.verbose >= 3)
      fprintf(stderr, "jqcd multishift: iter %d  |r|/|rhs| = %.3e\n", H->iters,
              H->rhs2 > 0 ? std::sqrt(H->rr / H->rhs2) : 0.0);
    if (H->done) break;
  }
  CKM(cudaEventRecord(G.ev1, s));
  jqcd_status st = JQCD_OK;
  if (H->done == 2) {
    *msg = "multi-shift CG breakdown (<p,Ap> <= 0 or not finite)";
    st = JQCD_EBREAKDOWN;
  }
  // true residual of every shifted system
  std::vector<double> tr(nshift, 0.0);
  for (int i = 0; i < nshift && st == JQCD_OK; ++i) {
    CKM(apply_mdagm(G, PREC_DW, P.kappa, V.x[i], Ap, G.vec_odd(G.vt), G.vec_even(G.vw), nullptr, nullptr, s));
    CKM(launch_ms_resid(rhs, Ap, V.x[i], shifts[i], n, G.partials, nblas, s));
    CKM(launch_finalize_sum(G.partials, nblas, &S->true_rr[i], s));
  }
  CKM(cudaMemcpyAsync(H, S, sizeof(MsScalars), cudaMemcpyDeviceToHost, s));
  CKM(cudaStreamSynchronize(s));
  float ms = 0.f;
  CKM(cudaEventElapsedTime(&ms, G.ev0, G.ev1));
  const double hop_iter = (double)vh * (1536.0 * 4 + 192.0 * 2);  // 4 hops, 2 with axpy
  for (int i = 0; i < nshift; ++i) {
    jqcd_solve_info &f = infos[i];
    memset(&f, 0, sizeof f);
    f.iters = H->conv_iter[i] ? H->conv_iter[i] : H->iters;
    f.true_rel_resid = H->rhs2 > 0 ? std::sqrt(H->true_rr[i] / H->rhs2) : 0.0;
    f.gpu_seconds = ms * 1e-3;
    f.hop_count = 4.0 * H->iters;
    f.hop_bytes = hop_iter * H->iters;
    f.status = st;
    if (st == JQCD_OK && (H->conv_iter[i] == 0 && H->rhs2 > 0)) f.status = JQCD_ENOCONV;
    else if (st == JQCD_OK && f.true_rel_resid > P.tol * (1.0 + 1e-6)) f.status = JQCD_ENOCONV;
  }
  if (st == JQCD_OK)
    for (int i = 0; i < nshift; ++i)
      if (infos[i].status != JQCD_OK) {
        st = JQCD_ENOCONV;
        *msg = H->done == 3 ? "maximum iterations reached" : "a shifted system misses its tolerance";
      }
  return st;
#undef CKM
}

cudaError_t launch_ms_start(const double *partials, int n, MsScalars *S, double tol2, int max_iters,
                            cudaStream_t s) {
  note_launch();
  ms_start_kernel<<<1, reduce_threads(n), 0, s>>>(partials, n, S, tol2, max_iters);
  return cudaGetLastError();
}

cudaError_t launch_ms_alpha(const double *partials, int nhop, MsScalars *S, MsSteps *B, int slot, cudaStream_t s) {
  note_launch();
  return launch_pdl(ms_alpha_kernel, 1, reduce_threads(nhop), 0, s, partials, nhop, S, B, slot);
}

cudaError_t launch_ms_beta_p(const double *partials, int nhop, int nblas, MsScalars *S, MsSteps *B, int slot,
                             const float4 *r, float4 *pb, int64_t n, cudaStream_t s) {
  note_launch(2);
  const cudaError_t e = launch_pdl(ms_beta_kernel, 1, reduce_threads(nhop), 0, s, partials, nhop, S, B, slot);
  if (e != cudaSuccess) return e;
  return launch_pdl(ms_p_kernel, nblas, kBlasThreads, 0, s, pb, r, n, S);
}

cudaError_t launch_ms_steps(const MsVectors &V, const MsResiduals &R, const MsScalars *S, const MsSteps *B, int nblas,
                            int64_t n, cudaStream_t s) {
  note_launch();
  return launch_pdl(ms_steps_kernel, nblas, kBlasThreads, 0, s, V, R, n, S, B);
}

cudaError_t launch_ms_resid(const float4 *rhs, const float4 *Ax, const float4 *x, double sigma, int64_t n,
                            double *partials, int nblocks, cudaStream_t s) {
  note_launch();
  ms_resid_kernel<<<nblocks, kBlasThreads, 0, s>>>(rhs, Ax, x, sigma, n, partials);
  return cudaGetLastError();
}

}  // namespace jqcd
