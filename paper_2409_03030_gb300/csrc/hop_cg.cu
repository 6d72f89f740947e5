// Last hop of the double-word even-odd normal operator fused with the CG
// update (conjugate gradient on Mhat^dag Mhat, the paper's solve_DinvX! in
// section "Definition of Dirac operators"), for the double-word solver and
// for the FP32 / FP16-with-norm inner solver of the mixed-precision CG.
//
// In one CG iteration alpha = ||r||^2 / <p, Mhat^dag Mhat p> and
// <p, Mhat^dag Mhat p> = ||Mhat p||^2 are known once the second hop has
// formed w = Mhat p.  The fourth hop, Ap = w - k^2 H^dag_eo t, therefore
// applies x += alpha p and r -= alpha Ap at its own site and forms the
// block partial of ||r||^2: Ap never reaches memory and the separate update
// kernel (which read x, r, p, Ap and wrote x, r) is gone.
#include <cuda_runtime.h>

#include "fields.cuh"
#include "hop_dwp.cuh"
#include "hop_lp.cuh"
#include "kernels.h"
#include "pdl.cuh"
#include "cg_steps.cuh"
#include "reduce.cuh"
#include "solver.h"

namespace jqcd {

namespace {

// q = a*w + b*v is (Ap)(idx) for the NC components k0 .. k0 + NC - 1 of the
// site; x += alpha p in place (XUPD) and r = r_in - alpha q; returns its
// contribution to ||r||^2.  Every operand is a 16-byte double-word chunk.
template <bool XUPD, int NC>
__device__ __forceinline__ dwacc dwp_store_cg(const p2 (&v)[NC], int k0, const float4 *__restrict__ w_base,
                                              const float4 *__restrict__ p_base,
                                              float4 *__restrict__ x_base, const float4 *r_in, float4 *r_base,
                                              int64_t vh, int64_t idx, float2 a_split, float2 b_split,
                                              float2 alpha) {
  idx += (int64_t)k0 * vh;
  const mul2 Bm{f2_make(b_split.x, b_split.x), f2_make(b_split.y, b_split.y)};
  const mul2 Am{f2_make(a_split.x, a_split.x), f2_make(a_split.y, a_split.y)};
  const mul2 Al{f2_make(alpha.x, alpha.x), f2_make(alpha.y, alpha.y)};
  const mul2 Ml{f2_neg(Al.h), f2_neg(Al.l)};
  const ulonglong2 *__restrict__ wp = reinterpret_cast<const ulonglong2 *>(w_base) + idx;
  const ulonglong2 *__restrict__ pp = reinterpret_cast<const ulonglong2 *>(p_base) + idx;
  ulonglong2 *__restrict__ xp = reinterpret_cast<ulonglong2 *>(x_base) + idx;
  const ulonglong2 *ri = reinterpret_cast<const ulonglong2 *>(r_in) + idx;  // may be rp
  ulonglong2 *rp = reinterpret_cast<ulonglong2 *>(r_base) + idx;
  acc2 nq{0ull, 0ull};
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const ulonglong2 wv = __ldg(wp + k * vh), rv = ri[k * vh];
    acc2 R = acc2_first(Bm, p2_norm(v[k]));
    acc2_mad(R, Am, p2{wv.x, wv.y});
    const p2 q = p2_norm(acc2_get(R));
    if (XUPD) {
      const ulonglong2 pv = __ldg(pp + k * vh), xv = xp[k * vh];
      const p2 xn = p2_norm(p2_add(p2{xv.x, xv.y}, acc2_get(acc2_first(Al, p2{pv.x, pv.y}))));
      xp[k * vh] = make_ulonglong2(xn.h, xn.l);
    }
    const p2 rn = p2_norm(p2_add(p2{rv.x, rv.y}, acc2_get(acc2_first(Ml, q))));
    rp[k * vh] = make_ulonglong2(rn.h, rn.l);
    const mul2 Q{rn.h, rn.l};
    if (k == 0) nq = acc2_first(Q, rn);
    else acc2_mad(nq, Q, rn);
  }
  float s0, s1, c0, c1;
  f2_split(nq.s, s0, s1);
  f2_split(nq.c, c0, c1);
  float s, e;
  two_sum(s0, s1, s, e);
  return dwacc{s, __fadd_rn(__fadd_rn(c0, c1), e)};
}

template <bool XUPD>
__global__ void __launch_bounds__(kDwp1Threads, JQCD_DWP_MIN_BLOCKS)
    hop_dwp_cg_kernel(const HopParams P, const float4 *__restrict__ p, float4 *__restrict__ xs,
                      const float4 *r_in, float4 *r, const float2 *__restrict__ alpha) {
  extern __shared__ float4 dsm[];
  pdl_enter();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  dwacc nrm{0.f, 0.f};
  if (idx < P.g.vh) {
    p2 acc[4][3];
    dwp_hop_site<true, kDwp1Threads>(dsm, reinterpret_cast<const float4 *>(P.in),
                                     reinterpret_cast<const float4 *>(P.gauge), P.g, P.out_parity, idx, acc);
    p2 v[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = acc[k / 3][k % 3];
    nrm = dwp_store_cg<XUPD, 12>(v, 0, reinterpret_cast<const float4 *>(P.x), p, xs, r_in, r, P.g.vh, idx,
                                 P.a_split, P.b_split, *alpha);
  }
  const double s = block_sum_dw(nrm);
  if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
}

// The same with the sites of `whole` blocks at one thread each and eight
// threads for each of the others (dw_hop_whole).
template <bool XUPD>
__global__ void __launch_bounds__(kDwp1Threads, JQCD_DWP_MIN_BLOCKS)
    hop_dwx_cg_kernel(const HopParams P, unsigned whole, const float4 *__restrict__ p, float4 *__restrict__ xs,
                      const float4 *r_in, float4 *r, const float2 *__restrict__ alpha) {
  extern __shared__ float4 dsm[];
  pdl_wait();
  if (P.guard && *P.guard) return;  // uniform across the grid
  dwacc nrm{0.f, 0.f};
  const float4 *const in = reinterpret_cast<const float4 *>(P.in), *const x = reinterpret_cast<const float4 *>(P.x);
  const float4 *const gauge = reinterpret_cast<const float4 *>(P.gauge);
  if (blockIdx.x < whole) {  // every site of these blocks exists
    const int64_t idx = (int64_t)blockIdx.x * kDwp1Threads + threadIdx.x;
    p2 acc[4][3], v[12];
    dwp_hop_site<true, kDwp1Threads>(dsm, in, gauge, P.g, P.out_parity, idx, acc);
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = acc[k / 3][k % 3];
    nrm = dwp_store_cg<XUPD, 12>(v, 0, x, p, xs, r_in, r, P.g.vh, idx, P.a_split, P.b_split, *alpha);
    pdl_trigger();
  } else {
    ulonglong2(*sm)[kDwp8Threads] = reinterpret_cast<ulonglong2(*)[kDwp8Threads]>(dsm);
    const int64_t idx = (int64_t)whole * kDwp1Threads + (int64_t)(blockIdx.x - whole) * kDwp8Sites + (threadIdx.x & 15);
    if (idx < P.g.vh) dwp8_hop<true>(sm, in, gauge, P.g, P.out_parity, (unsigned)idx);
    pdl_trigger();
    __syncthreads();
    const int spin = threadIdx.x >> 4;
    if (spin < 4 && idx < P.g.vh) {
      p2 v[3];
      dwp8_sum<true>(sm, threadIdx.x & 15, spin, v);
      nrm = dwp_store_cg<XUPD, 3>(v, 3 * spin, x, p, xs, r_in, r, P.g.vh, idx, P.a_split, P.b_split, *alpha);
    }
  }
  const double s = block_sum_dw(nrm);
  if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
}

// The same with eight threads per output site (small lattices, dw_hop_split8).
template <bool XUPD>
__global__ void __launch_bounds__(kDwp8Threads, JQCD_DWP8_MIN_BLOCKS)
    hop_dwp8_cg_kernel(const HopParams P, const float4 *__restrict__ p, float4 *__restrict__ xs,
                       const float4 *r_in, float4 *r, const float2 *__restrict__ alpha) {
  __shared__ ulonglong2 sm[6][kDwp8Threads];
  pdl_wait();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t base = (int64_t)blockIdx.x * kDwp8Sites;
  const int64_t hop_idx = base + (threadIdx.x & 15);
  if (hop_idx < P.g.vh)
    dwp8_hop<true>(sm, reinterpret_cast<const float4 *>(P.in), reinterpret_cast<const float4 *>(P.gauge), P.g,
                   P.out_parity, (unsigned)hop_idx);
  pdl_trigger();
  __syncthreads();
  dwacc nrm{0.f, 0.f};
  const int j = threadIdx.x & 15, spin = threadIdx.x >> 4;
  if (spin < 4 && base + j < P.g.vh) {
    p2 v[3];
    dwp8_sum<true>(sm, j, spin, v);
    nrm = dwp_store_cg<XUPD, 3>(v, 3 * spin, reinterpret_cast<const float4 *>(P.x), p, xs, r_in, r, P.g.vh,
                                base + j, P.a_split, P.b_split, *alpha);
  }
  const double s = block_sum_dw(nrm);
  if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
}

// Low-precision form for the inner CG: Ap = a w + b H^dag t in FP32 registers
// (never rounded to the storage precision), then the FP32 update of the
// inner residual rs with alpha_f and ||rs||^2 per hop block.  Five blocks per SM:
// 96 registers, which the compiler also takes without the bound; cut for six
// the FP16 solve took 1.5% longer at 24^3x48.
template <int PREC>
__global__ void __launch_bounds__(kHopThreads, 5)
    hop_lp_cg_kernel(const HopParams P, float4 *__restrict__ rs, const SolverScalars *__restrict__ S) {
  typedef PT<PREC> T;
  extern __shared__ float4 lsm[];
  pdl_enter();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  float n2 = 0.f;
  if (idx < P.g.vh) {
    cf acc[4][3];
    lp_hop_site<PREC, true, false>(lsm, P.in, reinterpret_cast<const float4 *>(P.gauge), P.g,
                                   P.out_parity, idx, acc);
    const float a = (float)P.a, b = (float)P.b, al = S->alpha_f;
    cf w[4][3], rv[4][3];
    T::load_spinor(P.x, P.g.vh, idx, w);
    PT<PREC_F32>::load_spinor(rs, P.g.vh, idx, rv);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const cf q = T::axpby(a, w[k / 3][k % 3], b, acc[k / 3][k % 3]);
      cf &r = rv[k / 3][k % 3];
      r.re = fmaf(-al, q.re, r.re);
      r.im = fmaf(-al, q.im, r.im);
      n2 = fmaf(r.re, r.re, fmaf(r.im, r.im, n2));
    }
    PT<PREC_F32>::store_spinor(rs, P.g.vh, idx, rv);
  }
  const double s = block_sum_f(n2);
  if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
  if (P.fin) hop_finish_scalars(P);  // uniform over the grid
}

template <int PREC>
cudaError_t launch_lp_cg_t(const HopParams &P, float4 *rs, const SolverScalars *S, cudaStream_t s) {
  return launch_pdl(hop_lp_cg_kernel<PREC>, hop_blocks(P.g.vh), kHopThreads, lp_stage_smem<PREC>(), s, P, rs, S);
}

}  // namespace

cudaError_t launch_hop_lp_cg(int prec, const HopParams &P, float4 *rs, const SolverScalars *S, cudaStream_t s) {
  if (P.g.vh >= kMaxHopSites) return cudaErrorInvalidValue;  // 32-bit neighbour offsets
  if (P.fin && (!P.fin_S || hop_blocks(P.g.vh) > (unsigned)JQCD_FIN_MAX_BLOCKS)) return cudaErrorInvalidValue;
  note_launch();
  switch (prec) {
    case PREC_F32: return launch_lp_cg_t<PREC_F32>(P, rs, S, s);
    case PREC_F16N: return launch_lp_cg_t<PREC_F16N>(P, rs, S, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool XUPD>
static cudaError_t launch_dw_cg_t(const HopParams &P, const float4 *p, float4 *x, const float4 *r_in, float4 *r,
                                  const float2 *alpha, cudaStream_t s) {
  if (P.g.vh >= kMaxHopSites) return cudaErrorInvalidValue;  // 32-bit neighbour offsets
  note_launch();
  static OncePerDevice configured;  // per instantiation
  const DwHopForm F = dw_hop_form(P.g.vh);
  const cudaError_t e = configured(F.device, [] {
    const cudaError_t e1 = cudaFuncSetAttribute(hop_dwp_cg_kernel<XUPD>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwpSmallSmem);
    return e1 ? e1
              : cudaFuncSetAttribute(hop_dwx_cg_kernel<XUPD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kDwp1Smem);
  });
  if (e) return e;
  if (F.split8)
    return launch_pdl(hop_dwp8_cg_kernel<XUPD>, F.blocks, kDwp8Threads, 0, s, P, p, x, r_in, r, alpha);
  if (F.whole)
    return launch_pdl(hop_dwx_cg_kernel<XUPD>, F.blocks, kDwp1Threads, kDwp1Smem, s, P, F.whole, p, x, r_in, r,
                      alpha);
  return launch_pdl(hop_dwp_cg_kernel<XUPD>, F.blocks, kDwp1Threads, F.small ? kDwpSmallSmem : kDwp1Smem, s, P, p, x,
                    r_in, r, alpha);
}

cudaError_t launch_hop_dw_cg(const HopParams &P, const float4 *p, float4 *x, float4 *r,
                             const SolverScalars *S, cudaStream_t s) {
  return launch_dw_cg_t<true>(P, p, x, r, r, &S->alpha_dw, s);
}

cudaError_t launch_hop_dw_r(const HopParams &P, const float4 *r_in, float4 *r, const float2 *alpha_dw,
                            cudaStream_t s) {
  return launch_dw_cg_t<false>(P, nullptr, nullptr, r_in, r, alpha_dw, s);
}

}  // namespace jqcd
