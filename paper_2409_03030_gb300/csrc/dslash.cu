// Even-odd Wilson hop kernels: out_p = a * x_p + b * H_{p,1-p} in_{1-p}
// with an optional fused per-block partial of ||out_p||^2.
//
// One thread per output site.  Each of the 8 neighbours is loaded as a full
// spinor (16-byte chunks, read-only path), spin-projected to a half-spinor,
// multiplied by its link (streamed, each link is used once per hop) and
// spread back onto four spins in registers.  Neighbour reuse across threads
// is served by L1/L2: in the checkerboard order the x, y, z neighbours of a
// warp's sites are within a few kB and the t neighbours within one time slice.
#include <cuda_runtime.h>

#include "fields.cuh"
#include "hop.cuh"
#include "kernels.h"
#include "pdl.cuh"
#include "hop_dw.cuh"
#include "hop_dwp.cuh"
#include "hop_lp.cuh"
#include "cg_steps.cuh"
#include "reduce.cuh"

namespace jqcd {

template <int MU, int PREC, bool DAG>
__device__ __forceinline__ void hop_dir(const HopParams &P, const HopSite &site,
                                        typename PT<PREC>::C (&acc)[4][3]) {
  typedef PT<PREC> T;
  typedef typename T::C C;
  const Geom &g = P.g;
  const int p = P.out_parity;
  const char *gbase = reinterpret_cast<const char *>(P.gauge);
  const size_t link_bytes = (size_t)T::kLinkChunks * 16 * g.vh;  // one (parity, mu) block
  // forward neighbour x + mu: (1 - gamma_mu) U_mu(x) psi(x+mu)
  {
    const unsigned off = hop_offset(g, site, 2 * MU);
    C psi[4][3], h[2][3], r[2][3], u[3][3];
    T::load_spinor(P.in, g.vh, (off & ~1u) >> 4, psi);
    project<MU, DAG ? 1 : -1>(psi, h);
    T::negate_if(h, off & 1u);
    T::load_link(gbase + link_bytes * (size_t)(p * 4 + MU), g.vh, site.idx, u);
    matvec2<false>(u, h, r);
    reconstruct<MU, DAG ? 1 : -1>(r, acc);
  }
  // backward neighbour x - mu: (1 + gamma_mu) U_mu(x-mu)^dag psi(x-mu)
  {
    const unsigned off = hop_offset(g, site, 2 * MU + 1);
    C psi[4][3], h[2][3], r[2][3], u[3][3];
    T::load_spinor(P.in, g.vh, (off & ~1u) >> 4, psi);
    project<MU, DAG ? -1 : 1>(psi, h);
    T::negate_if(h, off & 1u);
    T::load_link(gbase + link_bytes * (size_t)((1 - p) * 4 + MU), g.vh, (off & ~1u) >> 4, u);
    matvec2<true>(u, h, r);
    reconstruct<MU, DAG ? -1 : 1>(r, acc);
  }
}

template <int PREC, bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kHopThreads) hop_kernel(const HopParams P) {
  typedef PT<PREC> T;
  typedef typename T::C C;
  pdl_enter();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool active = idx < P.g.vh;
  dwacc nrm{0.f, 0.f};
  double nrm64 = 0.0;  // FP64 hops accumulate their norm in FP64
  if (active) {
    const HopSite site = hop_site(P.g, (unsigned)idx, P.out_parity);
    C acc[4][3];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[a][c] = T::zero();
    hop_dir<0, PREC, DAG>(P, site, acc);
    hop_dir<1, PREC, DAG>(P, site, acc);
    hop_dir<2, PREC, DAG>(P, site, acc);
    hop_dir<3, PREC, DAG>(P, site, acc);
    const typename T::Scalar b = T::scalar(P.b, P.b_split);
    C o[4][3];
    if (AXPY) {
      const typename T::Scalar a = T::scalar(P.a, P.a_split);
      C xs[4][3];
      T::load_spinor(P.x, P.g.vh, idx, xs);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) o[s][c] = T::axpby(a, xs[s][c], b, acc[s][c]);
    } else {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) o[s][c] = T::scale(b, acc[s][c]);
    }
    T::store_spinor(P.out, P.g.vh, idx, o);
    if (NORM) {
      if constexpr (PREC == PREC_F64) nrm64 = site_norm2_d(o);
      else nrm = site_norm2<PREC>(o);
    }
  }
  if (NORM) {
    const double s = PREC == PREC_F64 ? block_sum_d(nrm64) : block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
    if (P.fin) hop_finish_scalars(P);  // uniform over the grid
  }
}

// Low-precision hop with the next hop's neighbour and link prefetched into
// shared memory (hop_lp.cuh); same epilogue as hop_kernel.  HBM-bound (78.6 us
// = 6.5 TB/s at 32^3x64); six blocks per SM (84 registers) measured best:
// 27.9 us at 24^3x48 against 28.2 us with the compiler's 72-80 registers, 28.8
// us cut for seven; mixed FP16 solve 14.11 -> 13.94 ms, at 32^3x64 40.0 ->
// 39.6 ms.  Plain loads (hop_kernel) ran 25.6 us at 24^3x48 but 83.2 us at
// 32^3x64 and 4.9 against 3.9 us at 16^4.
template <int PREC, bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kHopThreads, 6) hop_lp_kernel(const HopParams P) {
  typedef PT<PREC> T;
  extern __shared__ float4 lsm[];
  pdl_enter();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  dwacc nrm{0.f, 0.f};
  if (idx < P.g.vh) {
    cf acc[4][3];
    lp_hop_site<PREC, DAG, false>(lsm, P.in, reinterpret_cast<const float4 *>(P.gauge), P.g,
                                  P.out_parity, idx, acc);
    const float b = (float)P.b;
    cf o[4][3];
    if (AXPY) {
      const float a = (float)P.a;
      cf xs[4][3];
      T::load_spinor(P.x, P.g.vh, idx, xs);
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) o[s][c] = T::axpby(a, xs[s][c], b, acc[s][c]);
    } else {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) o[s][c] = T::scale(b, acc[s][c]);
    }
    T::store_spinor(P.out, P.g.vh, idx, o);
    if (NORM) nrm = site_norm2<PREC>(o);
  }
  if (NORM) {
    const double s = block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
    if (P.fin) hop_finish_scalars(P);  // uniform over the grid
  }
}

template <int PREC, bool DAG, bool AXPY, bool NORM>
static cudaError_t launch_hop_t(const HopParams &P, cudaStream_t s) {
  const unsigned blocks = hop_blocks(P.g.vh);
  note_launch();
  // FP16: staged (measured faster); FP32: plain loads (its six-chunk stages
  // cost more occupancy than the prefetch gains); FP64: plain.
  if (PREC == PREC_F16N)
    return launch_pdl(hop_lp_kernel<PREC_F16N, DAG, AXPY, NORM>, blocks, kHopThreads,
                      lp_stage_smem<PREC_F16N>(), s, P);
  else
    return launch_pdl(hop_kernel<PREC, DAG, AXPY, NORM>, blocks, kHopThreads, 0, s, P);
}

template <int PREC>
static cudaError_t launch_hop_p(const HopParams &P, bool dag, bool axpy, bool norm, cudaStream_t s) {
  const int key = (dag ? 4 : 0) | (axpy ? 2 : 0) | (norm ? 1 : 0);
  switch (key) {
    case 0: return launch_hop_t<PREC, false, false, false>(P, s);
    case 1: return launch_hop_t<PREC, false, false, true>(P, s);
    case 2: return launch_hop_t<PREC, false, true, false>(P, s);
    case 3: return launch_hop_t<PREC, false, true, true>(P, s);
    case 4: return launch_hop_t<PREC, true, false, false>(P, s);
    case 5: return launch_hop_t<PREC, true, false, true>(P, s);
    case 6: return launch_hop_t<PREC, true, true, false>(P, s);
    default: return launch_hop_t<PREC, true, true, true>(P, s);
  }
}

// ---------------------------------------------------------------------------
// Double-word hop in packed two-lane arithmetic (hop_dwp.cuh): one fma/add/
// mul.rn.f32x2 per complex operation halves the instruction issue of a
// scalar double-word hop, which was bound by issue rather than by the FP32
// datapath.
template <bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kDwp1Threads, JQCD_DWP_MIN_BLOCKS) hop_dwp_kernel(const HopParams P) {
  extern __shared__ float4 dsm[];
  pdl_enter();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  dwacc nrm{0.f, 0.f};
  if (idx < P.g.vh) {
    p2 acc[4][3];
    dwp_hop_site<DAG, kDwp1Threads>(dsm, reinterpret_cast<const float4 *>(P.in),
                                    reinterpret_cast<const float4 *>(P.gauge), P.g, P.out_parity, idx, acc);
    nrm = dwp_store<AXPY, NORM>(acc, reinterpret_cast<float4 *>(P.out),
                                reinterpret_cast<const float4 *>(P.x), P.g.vh, idx, P.a_split, P.b_split);
  }
  if (NORM) {
    const double s = block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
  }
}

// Small lattices: eight threads per output site (dwp8_hop).  A hop there is a
// latency chain, the loads' round trip and the arithmetic of as many hops as a
// thread runs, on too few warps to hide it: with one hop per thread, 8^4 (two
// threads: 5.3 us back to back) takes 2.7 us, 12^4 (8.3 us) 6.0 us.
template <bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kDwp8Threads, JQCD_DWP8_MIN_BLOCKS) hop_dwp8_kernel(const HopParams P) {
  __shared__ ulonglong2 sm[6][kDwp8Threads];
  pdl_wait();
  if (P.guard && *P.guard) return;  // uniform across the grid
  const int64_t base = (int64_t)blockIdx.x * kDwp8Sites;
  const int64_t hop_idx = base + (threadIdx.x & 15);
  if (hop_idx < P.g.vh)
    dwp8_hop<DAG>(sm, reinterpret_cast<const float4 *>(P.in), reinterpret_cast<const float4 *>(P.gauge), P.g,
                  P.out_parity, (unsigned)hop_idx);
  pdl_trigger();
  __syncthreads();
  dwacc nrm{0.f, 0.f};
  const int j = threadIdx.x & 15, spin = threadIdx.x >> 4;
  if (spin < 4 && base + j < P.g.vh) {
    p2 v[3];
    dwp8_sum<DAG>(sm, j, spin, v);
    nrm = dwp_store_chunks<AXPY, NORM, 3>(v, 3 * spin, reinterpret_cast<float4 *>(P.out),
                                          reinterpret_cast<const float4 *>(P.x), P.g.vh, base + j, P.a_split,
                                          P.b_split);
  }
  if (NORM) {
    const double s = block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
  }
}

// Eight threads per site up to SMs x JQCD_DWP8_BLOCKS blocks of 16 sites
// (29184 sites per parity).  Measured on GB300, Mhat^dag Mhat p with its norm
// and the solve, against the two threads per site that ran there before: 8^4
// 28.9 -> 22.5 us and 1.90 -> 1.58 ms, 12^4 40.9 -> 31.3 us and 2.95 -> 2.55
// ms, 16^3x12 58.7 -> 52.2 us and 4.18 -> 3.94 ms, 16^3x14 60.1 -> 58.2 us and
// 4.47 -> 4.41 ms.  One thread per site takes 55.2 us and 4.08 ms at 16^3x12,
// 55.6 us and 4.32 ms at 16^3x14 (but its sum of eight hops in a row has a 5%
// larger rounding error), and wins at 16^4 (56.6 against 67.6 us).
bool dw_hop_split8(int64_t vh) {
  static const int64_t max_vh = [] {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
      return (int64_t)0;
    return (int64_t)sms * JQCD_DWP8_BLOCKS * kDwp8Sites;
  }();
  return vh <= max_vh;
}

// A one-thread grid of at most SMs x JQCD_DWP_SMALL_BLOCKS blocks is launched
// with kDwpSmallSmem of shared memory, so that no SM takes a third block.
// Back to back, each grid's blocks are placed (programmatic launch) while the
// one before still runs; with room for three, some SMs get three and the grid
// waits for them.  Measured on GB300 at 16^4: 17.0 us with room for three,
// 12.8 us for two (13.4 us for the 184-register kernel that two blocks per SM
// were once cut for); Mhat^dag Mhat p with its norm 63.8 -> 57.2 us, the
// double-word solve 4.95 -> 4.71 ms.  All hops unrolled took 11.7 us when the
// same kernel ran back to back, but its code (four kernels of about 90 KB)
// misses the instruction cache in a real chain: 5.3 ms.
bool dw_hop_small(int64_t vh) {
  static const int64_t max_vh = [] {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
      return (int64_t)0;
    return (int64_t)sms * JQCD_DWP_SMALL_BLOCKS * kDwp1Threads;
  }();
  return !dw_hop_split8(vh) && vh <= max_vh && vh <= JQCD_DWP_SMALL_MAX_VH;
}

unsigned dw_hop_blocks(int64_t vh) {
  if (dw_hop_split8(vh)) return (unsigned)((vh + kDwp8Sites - 1) / kDwp8Sites);
  return (unsigned)((vh + kDwp1Threads - 1) / kDwp1Threads);
}

unsigned hop_norm_partials(int prec, int64_t vh) {
  return prec == PREC_DW ? dw_hop_blocks(vh) : hop_blocks(vh);
}

template <bool DAG, bool AXPY, bool NORM>
static cudaError_t launch_hop_dw_t(const HopParams &P, cudaStream_t s) {
  note_launch();
  static bool configured = false;  // one attribute call per instantiation
  auto kern = hop_dwp_kernel<DAG, AXPY, NORM>;
  if (!configured) {
    const cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwpSmallSmem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  if (dw_hop_split8(P.g.vh))
    return launch_pdl(hop_dwp8_kernel<DAG, AXPY, NORM>, dw_hop_blocks(P.g.vh), kDwp8Threads, 0, s, P);
  return launch_pdl(kern, dw_hop_blocks(P.g.vh), kDwp1Threads, dw_hop_small(P.g.vh) ? kDwpSmallSmem : kDwp1Smem, s,
                    P);
}

static cudaError_t launch_hop_dw(const HopParams &P, bool dag, bool axpy, bool norm, cudaStream_t s) {
  const int key = (dag ? 4 : 0) | (axpy ? 2 : 0) | (norm ? 1 : 0);
  switch (key) {
    case 0: return launch_hop_dw_t<false, false, false>(P, s);
    case 1: return launch_hop_dw_t<false, false, true>(P, s);
    case 2: return launch_hop_dw_t<false, true, false>(P, s);
    case 3: return launch_hop_dw_t<false, true, true>(P, s);
    case 4: return launch_hop_dw_t<true, false, false>(P, s);
    case 5: return launch_hop_dw_t<true, false, true>(P, s);
    case 6: return launch_hop_dw_t<true, true, false>(P, s);
    default: return launch_hop_dw_t<true, true, true>(P, s);
  }
}

cudaError_t launch_hop(int prec, const HopParams &P, bool dag, bool axpy, bool norm,
                       cudaStream_t s) {
  // the last-block scalar step (FP64, FP32 and FP16 hops) needs the partials
  // and at most JQCD_FIN_MAX_BLOCKS of them
  if (P.fin && (prec == PREC_DW || !norm || !P.fin_S ||
                hop_norm_partials(prec, P.g.vh) > (unsigned)JQCD_FIN_MAX_BLOCKS))
    return cudaErrorInvalidValue;
  if (P.g.vh >= kMaxHopSites) return cudaErrorInvalidValue;  // 32-bit neighbour offsets
  switch (prec) {
    case PREC_DW: return launch_hop_dw(P, dag, axpy, norm, s);
    case PREC_F64: return launch_hop_p<PREC_F64>(P, dag, axpy, norm, s);
    case PREC_F32: return launch_hop_p<PREC_F32>(P, dag, axpy, norm, s);
    case PREC_F16N: return launch_hop_p<PREC_F16N>(P, dag, axpy, norm, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace jqcd
