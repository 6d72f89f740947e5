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
    if (NORM) nrm = site_norm2<PREC>(o);
  }
  if (NORM) {
    const double s = block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
    if (P.fin) hop_finish_scalars(P);  // uniform over the grid
  }
}

// Low-precision hop with the next hop's neighbour and link prefetched into
// shared memory (hop_lp.cuh); same epilogue as hop_kernel.  HBM-bound (78.6 us
// = 6.5 TB/s at 32^3x64); six blocks per SM (80 registers) measured best:
// 27.9 us at 24^3x48 against 28.2 us with the compiler's own count (72, 80 with
// the axpy, 96 with the norm too), 28.8 us cut for seven; mixed FP16 solve 14.11 -> 13.94 ms, at 32^3x64 40.0 ->
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

// Native FP64 hop with eight threads per output site: a tile is 16 sites in 128
// threads, warp mu runs direction mu, lanes 0..15 its forward and 16..31 its
// backward hop.  The kernel is bound by the FP64 pipe (888 FP64 instructions
// per site), and a warp's FP64 instruction holds its sub-partition's unit for
// about 67 cycles: with one thread per site a site's 888 last 29 us however
// few warps there are, and an SM whose unit has one warp more than the others'
// ends that much later.  In pieces of 111 the work spreads evenly.  The
// products meet in shared memory; every thread then sums one or two of the
// 16 x 12 components over the hops, in the order of the one-thread form.
// Measured on GB300 against one thread per site: 8^4 32.7 -> 6.2 us, 16^4 94.9
// -> 54.8 us, 16^3x32 127 -> 104 us, 24^3x48 559 -> 517 us (the rate of
// the FP64 pipe); plain FP64 solve at 16^4 22.9 -> 15.1 ms.
constexpr int kF64x8Sites = 16;
constexpr int kF64x8Threads = 8 * kF64x8Sites;

// h = rows 0 and 1 of (1 + S gamma_mu) psi, S = +-1 at run time (riding on the fmas)
template <int MU>
__device__ __forceinline__ void project_rt_f64(const cd (&psi)[4][3], cd (&h)[2][3], double S) {
  typedef SpinTab<MU> T;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const cd q0 = phase<T::p0>(psi[T::j0][c]), q1 = phase<T::p1>(psi[T::j1][c]);
    h[0][c] = cd{fma(S, q0.re, psi[0][c].re), fma(S, q0.im, psi[0][c].im)};
    h[1][c] = cd{fma(S, q1.re, psi[1][c].re), fma(S, q1.im, psi[1][c].im)};
  }
}

__device__ __forceinline__ double flip_if(double v, bool neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}

template <bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kF64x8Threads, 4) hop_f64x8_kernel(const HopParams P, int tiles) {
  __shared__ double2 sm[6][kF64x8Threads];
  pdl_wait();
  if (P.guard && *P.guard) return;  // uniform across the grid
  typedef PT<PREC_F64> T;
  const Geom &g = P.g;
  const int p = P.out_parity;
  const unsigned j = threadIdx.x & 15;
  double nrm = 0.0;
  for (int tile = 0; tile < tiles; ++tile) {
    const unsigned idx = (blockIdx.x * tiles + tile) * kF64x8Sites + j;
    const bool active = idx < (unsigned)g.vh;
    if (tile) __syncthreads();  // the last tile's products have been summed
    if (active) {
      const int mu = threadIdx.x >> 5;
      const bool bwd = (threadIdx.x & 16) != 0;
      const HopSite site = hop_site(g, idx, p);
      unsigned off;
      switch (mu) {
        case 0: off = bwd ? hop_offset(g, site, 1) : hop_offset(g, site, 0); break;
        case 1: off = bwd ? hop_offset(g, site, 3) : hop_offset(g, site, 2); break;
        case 2: off = bwd ? hop_offset(g, site, 5) : hop_offset(g, site, 4); break;
        default: off = bwd ? hop_offset(g, site, 7) : hop_offset(g, site, 6);
      }
      const unsigned nb = (off & ~1u) >> 4;
      cd psi[4][3], h[2][3], u[3][3];
      T::load_spinor(P.in, g.vh, nb, psi);
      // W = U_mu(x), or the transpose of U_mu(x - mu), conjugated below
      const double2 *L = reinterpret_cast<const double2 *>(P.gauge) +
                         (int64_t)(((bwd ? 1 - p : p) * 4 + mu) * 9) * g.vh + (bwd ? nb : idx);
      const int sa = bwd ? 1 : 3, sb = bwd ? 3 : 1;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const double2 v = __ldg(L + (int64_t)((k / 3) * sa + (k % 3) * sb) * g.vh);
        u[k / 3][k % 3] = cd{v.x, flip_if(v.y, bwd)};
      }
      const double S = (bwd != DAG) ? 1.0 : -1.0;
      switch (mu) {
        case 0: project_rt_f64<0>(psi, h, S); break;
        case 1: project_rt_f64<1>(psi, h, S); break;
        case 2: project_rt_f64<2>(psi, h, S); break;
        default: project_rt_f64<3>(psi, h, S);
      }
      T::negate_if(h, off & 1u);
      cd r[2][3];
      matvec2<false>(u, h, r);
#pragma unroll
      for (int k = 0; k < 6; ++k) sm[k][threadIdx.x] = make_double2(r[k / 3][k % 3].re, r[k / 3][k % 3].im);
    }
    if (tile + 1 == tiles) pdl_trigger();
    __syncthreads();
    if (active) {
      const int grp = threadIdx.x >> 4;  // components grp and, for the first four groups, grp + 8
      const int nk = grp < 4 ? 2 : 1;
      for (int q = 0; q < nk; ++q) {
        const int k = grp + 8 * q, spin = k / 3, c = k - 3 * spin;
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
          const int mu = d >> 1;
          // spins 2 and 3 take the row the projector ties to them, times a phase
          // (SpinTab; S < 0 negates it)
          const int src = spin < 2 ? spin : (mu < 2 ? 3 - spin : spin - 2);
          int ph = 0;
          if (spin == 2) ph = (mu & 1) ? 0 : 3;
          if (spin == 3) ph = mu == 0 ? 3 : (mu == 1 ? 2 : (mu == 2 ? 1 : 0));
          if (spin >= 2 && (((d & 1) != 0) == DAG)) ph ^= 2;
          const double2 v = sm[3 * src + c][16 * d + j];
          const bool sw = ph & 1;
          re += flip_if(sw ? v.y : v.x, ph == 1 || ph == 2);
          im += flip_if(sw ? v.x : v.y, ph & 2);
        }
        cd o;
        if (AXPY) {
          const double2 xv = __ldg(reinterpret_cast<const double2 *>(P.x) + (int64_t)k * g.vh + idx);
          o = T::axpby(P.a, cd{xv.x, xv.y}, P.b, cd{re, im});
        } else {
          o = T::scale(P.b, cd{re, im});
        }
        reinterpret_cast<double2 *>(P.out)[(int64_t)k * g.vh + idx] = make_double2(o.re, o.im);
        if (NORM) {
          nrm = fma(o.re, o.re, nrm);
          nrm = fma(o.im, o.im, nrm);
        }
      }
    }
  }
  if (NORM) {
    const double s = block_sum_d(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
  }
}

// Tiles of 16 sites per block: one while the grid is small, then two, and no
// more than 16384 blocks (a norm's partial sums, one per block, have that much
// room in the allocation-free call up to JQCD_NOALLOC_MAX_SITES_PER_PARITY).
// 24^3x48: 512 us with one tile, 517 with two, 529 with four, 550 with eight;
// fewer partials keep the solve's sums short.
static int f64_tiles(int64_t vh) {
  if (vh <= 65536) return 1;
  int t = 2;
  while (vh > (int64_t)16384 * kF64x8Sites * t && t < 64) t *= 2;
  return t;
}
static unsigned f64_blocks(int64_t vh) {
  const int64_t sites = kF64x8Sites * f64_tiles(vh);
  return (unsigned)((vh + sites - 1) / sites);
}

template <int PREC, bool DAG, bool AXPY, bool NORM>
static cudaError_t launch_hop_t(const HopParams &P, cudaStream_t s) {
  note_launch();
  // FP64: eight threads per site.  FP16: staged (measured faster).  FP32: plain
  // loads (its six-chunk stages cost more occupancy than the prefetch gains).
  if constexpr (PREC == PREC_F64)
    return launch_pdl(hop_f64x8_kernel<DAG, AXPY, NORM>, f64_blocks(P.g.vh), kF64x8Threads, 0, s, P,
                      f64_tiles(P.g.vh));
  else if constexpr (PREC == PREC_F16N)
    return launch_pdl(hop_lp_kernel<PREC_F16N, DAG, AXPY, NORM>, hop_blocks(P.g.vh), kHopThreads,
                      lp_stage_smem<PREC_F16N>(), s, P);
  else
    return launch_pdl(hop_kernel<PREC, DAG, AXPY, NORM>, hop_blocks(P.g.vh), kHopThreads, 0, s, P);
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

// A grid a little over a whole number of one-thread blocks per SM (dw_hop_whole):
// the first `whole` blocks run 128 sites at one thread each, a multiple of the
// SM count; eight threads per site share the rest, 16 sites to a block.  The
// one-thread blocks of such a remainder would each last the whole chain of
// eight hops, about 7 us, on SMs that are otherwise idle; the tiles last 2.7
// us.  The trigger comes last (pdl.cuh): the tiles go to the SMs with room.
template <bool DAG, bool AXPY, bool NORM>
__global__ void __launch_bounds__(kDwp1Threads, JQCD_DWP_MIN_BLOCKS)
    hop_dwx_kernel(const HopParams P, unsigned whole) {
  extern __shared__ float4 dsm[];
  pdl_wait();
  if (P.guard && *P.guard) return;  // uniform across the grid
  dwacc nrm{0.f, 0.f};
  const float4 *const in = reinterpret_cast<const float4 *>(P.in), *const x = reinterpret_cast<const float4 *>(P.x);
  const float4 *const gauge = reinterpret_cast<const float4 *>(P.gauge);
  float4 *const out = reinterpret_cast<float4 *>(P.out);
  if (blockIdx.x < whole) {  // every site of these blocks exists
    const int64_t idx = (int64_t)blockIdx.x * kDwp1Threads + threadIdx.x;
    p2 acc[4][3];
    dwp_hop_site<DAG, kDwp1Threads>(dsm, in, gauge, P.g, P.out_parity, idx, acc);
    nrm = dwp_store<AXPY, NORM>(acc, out, x, P.g.vh, idx, P.a_split, P.b_split);
    pdl_trigger();
  } else {
    ulonglong2(*sm)[kDwp8Threads] = reinterpret_cast<ulonglong2(*)[kDwp8Threads]>(dsm);
    const int64_t idx = (int64_t)whole * kDwp1Threads + (int64_t)(blockIdx.x - whole) * kDwp8Sites + (threadIdx.x & 15);
    if (idx < P.g.vh) dwp8_hop<DAG>(sm, in, gauge, P.g, P.out_parity, (unsigned)idx);
    pdl_trigger();
    __syncthreads();
    const int spin = threadIdx.x >> 4;
    if (spin < 4 && idx < P.g.vh) {
      p2 v[3];
      dwp8_sum<DAG>(sm, threadIdx.x & 15, spin, v);
      nrm = dwp_store_chunks<AXPY, NORM, 3>(v, 3 * spin, out, x, P.g.vh, idx, P.a_split, P.b_split);
    }
  }
  if (NORM) {
    const double s = block_sum_dw(nrm);
    if (threadIdx.x == 0) P.partials[blockIdx.x] = s;
  }
}

// Small lattices: eight threads per output site (dwp8_hop).  A hop there is a
// latency chain, the loads' round trip and the arithmetic of as many hops as a
// thread runs, on too few warps to hide it: with one hop per thread, 8^4 (two
// threads: 5.3 us back to back) takes 2.7 us, 12^4 (8.3 us) 5.2 us.
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

// Eight threads per site up to SMs x JQCD_DWP8_BLOCKS blocks of 16 sites (29184
// sites per parity).  Measured on GB300 against the two threads per site that
// ran there before: one hop back to back 8^4 5.3 -> 2.7 us, 12^4 8.3 -> 5.2 us;
// the double-word solve 8^4 1.90 -> 1.46 ms, 12^4 2.95 -> 2.34 ms, 16^3x12 4.18
// -> 3.60 ms, 16^3x14 4.47 -> 3.95 ms.  Above, one thread per site solves in
// less: 16^4 4.44 against 4.53 ms, 16^3x18 4.62 against 5.14 ms, 16^3x24 5.88
// against 6.75 ms.  Four blocks per SM: with five (96 registers, 40 bytes
// spilled) 8^4 takes 2.9 us, with three 12^4 5.6 us.
static bool dw_hop_split8(int64_t vh, int64_t sms) { return vh <= sms * JQCD_DWP8_BLOCKS * kDwp8Sites; }

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
static bool dw_hop_small(int64_t vh, int64_t sms) {
  return !dw_hop_split8(vh, sms) && vh <= sms * JQCD_DWP_SMALL_BLOCKS * kDwp1Threads && vh <= JQCD_DWP_SMALL_MAX_VH;
}

// Whole blocks per SM at one thread per site and the rest at eight, where the
// rest is at most two fifths of a block per SM: one hop on GB300 against one
// thread for every site: 16^3x30 21.9 -> 18.1 us, 16^3x32 22.1 -> 19.8 us,
// 16^3x40 27.6 -> 25.1 us, 16^3x48 33.4 -> 29.9 us, 20^3x40 49.1 -> 47.5 us;
// the double-word solve at 20x18x14x26 8.25 -> 7.82 ms.  With a longer rest the
// tiles last longer than the blocks they replace (20^3x24, 0.93 of a block per
// SM: 29.5 -> 32.0 us), and past JQCD_DWX_MAX_VH a rest no longer shows (24^3x48
// 91.0 and 90.9 us; the solve at 24^3x32 21.9 and 22.1 ms).  Not below one
// wave of one-thread blocks, where only rests past the two fifths have been
// measured (16^3x24, 0.53 of a block: 16.9 -> 17.1 us; 16^3x28, 0.95: 17.1 ->
// 19.3 us).
static unsigned dw_hop_whole(int64_t vh, int64_t sms) {
  const int64_t wave = sms * JQCD_DWP_MIN_BLOCKS * kDwp1Threads;
  if (!sms || vh <= wave || vh > JQCD_DWX_MAX_VH) return 0;
  const int64_t blocks = (vh + kDwp1Threads - 1) / kDwp1Threads, whole = vh / kDwp1Threads / sms * sms;
  return 5 * (blocks - whole) <= 2 * sms ? (unsigned)whole : 0;
}

// SMs of a device, 0 when they cannot be asked for (and asked for again then)
static int device_sms(int device) {
  static std::atomic<int> known[64];
  const bool slot = device >= 0 && device < 64;
  int n = slot ? known[device].load(std::memory_order_relaxed) : 0;
  if (n > 0) return n;
  if (device < 0 || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n < 1)
    return 0;
  if (slot) known[device].store(n, std::memory_order_relaxed);
  return n;
}

DwHopForm dw_hop_form(int64_t vh) {
  const int device = current_device();
  const int64_t sms = device_sms(device);
  const int64_t whole = dw_hop_whole(vh, sms);
  const bool split8 = dw_hop_split8(vh, sms);
  const int64_t blocks = whole || split8 ? whole + (vh - whole * kDwp1Threads + kDwp8Sites - 1) / kDwp8Sites
                                         : (vh + kDwp1Threads - 1) / kDwp1Threads;
  return DwHopForm{device, split8, dw_hop_small(vh, sms), (unsigned)whole, (unsigned)blocks};
}

unsigned hop_norm_partials(int prec, int64_t vh) {
  if (prec == PREC_F64) return f64_blocks(vh);
  return prec == PREC_DW ? dw_hop_blocks(vh) : hop_blocks(vh);
}

template <bool DAG, bool AXPY, bool NORM>
static cudaError_t launch_hop_dw_t(const HopParams &P, cudaStream_t s) {
  note_launch();
  static OncePerDevice configured;  // per instantiation
  const DwHopForm F = dw_hop_form(P.g.vh);
  const cudaError_t e = configured(F.device, [] {
    const cudaError_t e1 = cudaFuncSetAttribute(
        hop_dwp_kernel<DAG, AXPY, NORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwpSmallSmem);
    return e1 ? e1
              : cudaFuncSetAttribute(hop_dwx_kernel<DAG, AXPY, NORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kDwp1Smem);
  });
  if (e) return e;
  if (F.split8) return launch_pdl(hop_dwp8_kernel<DAG, AXPY, NORM>, F.blocks, kDwp8Threads, 0, s, P);
  if (F.whole)
    return launch_pdl(hop_dwx_kernel<DAG, AXPY, NORM>, F.blocks, kDwp1Threads, kDwp1Smem, s, P, F.whole);
  return launch_pdl(hop_dwp_kernel<DAG, AXPY, NORM>, F.blocks, kDwp1Threads, F.small ? kDwpSmallSmem : kDwp1Smem, s,
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
  // the last-block scalar step (FP32 and FP16 hops) needs the partials and at
  // most JQCD_FIN_MAX_BLOCKS of them
  if (P.fin && ((prec != PREC_F32 && prec != PREC_F16N) || !norm || !P.fin_S ||
                hop_blocks(P.g.vh) > (unsigned)JQCD_FIN_MAX_BLOCKS))
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
