// Double-word hop in packed two-lane arithmetic, shared by the single-field
// kernel (dslash.cu) and the batched reliable-update stages (batch_kernels.cu).
//
// Every complex double-word operation runs its real and imaginary lanes in
// one fma/add/mul.rn.f32x2: projection and reconstruction by sign-carrying
// TwoSums, the SU(3) product W h = h.re W + i (h.im W) as sums of exact
// products on a fixed offset grid with broadcast half-spinor multipliers.  (Folding the link's signs into the
// multipliers instead saves FP32 multiplies but costs registers: the kernel
// then spills and runs slower on sm_103.)
//
// Neighbour spinors and links of the next hop are prefetched into shared
// memory with cp.async (chunk-major [k][thread], each thread touching only
// its own column).
#pragma once
#include "dw2.cuh"
#include "hop_dw.cuh"

namespace jqcd {

constexpr int kDwpStageChunks = 12;  // one double-word spinor per thread
constexpr int kDwpLinkChunks = 9;    // one double-word link per thread and stage
// one neighbour-spinor stage and two link stages, chunk-major [k][thread],
// and the eight neighbour offsets (4 bytes each), for blocks of nt threads
constexpr size_t dwp_smem(int nt = kHopThreads) {
  return (size_t)(kDwpStageChunks + 2 * kDwpLinkChunks + 2) * nt * 16;
}
constexpr size_t kDwpSmem = dwp_smem();

// Launch shapes of the single-field kernels: threads per block and the
// resident blocks per SM their register budget is cut for, one thread per
// output site (DWP) and eight (DWP8, small lattices: dwp8_hop).
#ifndef JQCD_DWP_THREADS
#define JQCD_DWP_THREADS 128
#endif
#ifndef JQCD_DWP_MIN_BLOCKS
#define JQCD_DWP_MIN_BLOCKS 3
#endif
// One-thread grids of at most SMs x JQCD_DWP_SMALL_BLOCKS blocks (16^4) ask
// for so much shared memory that an SM holds no more than that many: with
// room for three, the blocks of back-to-back launches crowd some SMs while
// others run one (dw_hop_small).
#ifndef JQCD_DWP_SMALL_BLOCKS
#define JQCD_DWP_SMALL_BLOCKS 2
#endif
#ifndef JQCD_DWP8_MIN_BLOCKS
#define JQCD_DWP8_MIN_BLOCKS 4
#endif
#ifndef JQCD_DWP8_BLOCKS
#define JQCD_DWP8_BLOCKS 12
#endif
constexpr int kDwp1Threads = JQCD_DWP_THREADS;
constexpr size_t kDwp1Smem = dwp_smem(kDwp1Threads);
// 227 KB of shared memory per SM, 1 KB of it reserved per block
constexpr size_t kDwpSmallSmem = (size_t)(227 / JQCD_DWP_SMALL_BLOCKS - 2) * 1024;
static_assert(kDwpSmallSmem >= kDwp1Smem, "the limit only pads the stages");

// Issue the copies of a spinor (byte offset off) into its stage column st
// (NT: threads per block, the stride of the chunk-major stage).  The chunk
// planes in + k vh are uniform over the grid, so the per-thread part of every
// address is the one 32-bit offset.
template <int NT>
__device__ __forceinline__ void stage_hop_p(float4 *st, const float4 *in, int64_t vh, unsigned off) {
#pragma unroll
  for (int k = 0; k < 12; ++k) cp_async16(st + k * NT, chunk_at(in + k * vh, off), false);
}

// Issue the copies of the link of hop d (mu = d/2, backward when d is odd)
// into a link stage column, element (a, b) at chunk 3a + b: U_mu(x) for a
// forward hop (own: byte offset of x), U_mu(x - mu) for a backward one (nb:
// byte offset of the neighbour); transposed and conjugated at use.
template <int NT = kHopThreads>
__device__ __forceinline__ void stage_link_p(float4 *st, const float4 *gauge, int64_t vh, int p, int d,
                                             unsigned own, unsigned nb) {
  const bool bwd = (d & 1) != 0;
  const float4 *L = gauge + (int64_t)(((bwd ? 1 - p : p) * 4 + (d >> 1)) * 9) * vh;
  const unsigned off = bwd ? nb : own;
#pragma unroll
  for (int k = 0; k < 9; ++k) cp_async16(st + k * NT, chunk_at(L + k * vh, off), false);
}

__device__ __forceinline__ p2 ld_p2(const float4 *p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
  return p2{v.x, v.y};
}

// (1 + S gamma_mu) psi, rows 0 and 1, DeGrand-Rossi basis.  With phi = i the
// swapped operand (im, re) carries the lane signs (-S, S).
template <int MU>
__device__ __forceinline__ void project_p(const p2 (&psi)[4][3], p2 (&h)[2][3], float S) {
  const f2 sS = f2_make(S, S), nS = f2_make(-S, -S), sI = f2_make(-S, S), sIm = f2_make(S, -S);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (MU == 0) { h[0][c] = p2_add_sgn(psi[0][c], p2_swap(psi[3][c]), sI); h[1][c] = p2_add_sgn(psi[1][c], p2_swap(psi[2][c]), sI); }
    if (MU == 1) { h[0][c] = p2_add_sgn(psi[0][c], psi[3][c], nS);          h[1][c] = p2_add_sgn(psi[1][c], psi[2][c], sS); }
    if (MU == 2) { h[0][c] = p2_add_sgn(psi[0][c], p2_swap(psi[2][c]), sI); h[1][c] = p2_add_sgn(psi[1][c], p2_swap(psi[3][c]), sIm); }
    if (MU == 3) { h[0][c] = p2_add_sgn(psi[0][c], psi[2][c], sS);          h[1][c] = p2_add_sgn(psi[1][c], psi[3][c], sS); }
  }
}

// r[a] = sum_b W_ab h[b] with TwoSum-compensated sums of exact products
// (twelve packed operations per product, error about 2^-48 |W||h|): the
// accumulation of the staggered hop, which is bound by HBM bandwidth.
__device__ __forceinline__ void matvec_half_ts(const p2 (&W)[3][3], const p2 (&h)[3], p2 (&r)[3]) {
  mul2 mr[3], mi[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    mr[b] = mul2{f2_lo(h[b].h), f2_lo(h[b].l)};
    mi[b] = mul2{f2_hi(h[b].h), f2_hi(h[b].l)};
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    acc2 A = acc2_first(mr[0], W[a][0]);
    acc2 B = acc2_first(mi[0], W[a][0]);
#pragma unroll
    for (int b = 1; b < 3; ++b) {
      acc2_mad(A, mr[b], W[a][b]);
      acc2_mad(B, mi[b], W[a][b]);
    }
    // i B = (-B.im, B.re): swap the lanes, flip the sign of lane 0
    constexpr f2 kLane0 = 0x0000000080000000ull;
    r[a] = p2_add(acc2_get(A), p2{f2_swap(B.s) ^ kLane0, f2_swap(B.c) ^ kLane0});
  }
}

// Largest |component| of the link's high words, the bound its products need.
__device__ __forceinline__ float link_max_hi(const p2 (&W)[3][3]) {
  float m = 0.f;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    float u, v;
    f2_split(W[k / 3][k % 3].h, u, v);
    m = fmaxf(m, fmaxf(fabsf(u), fabsf(v)));
  }
  return m;
}

// One exact-product step of an offset-grid sum: T = T0 + (partial sum) stays
// in the binade [sigma, 2 sigma), so the fma rounds the exact high product
// onto that binade's fixed grid, T - T_new is exact (Sterbenz lemma) and one
// more fma returns the part of the product below the grid to the low-order
// sum c, together with the two cross products of the low words.
__device__ __forceinline__ void grid_mad(f2 &T, f2 &c, const mul2 &A, p2 B, bool first) {
  const f2 Tn = f2_fma(A.h, B.h, T);
  const f2 d = f2_fma(A.h, B.h, f2_sub(T, Tn));  // product - (Tn - T), rounded
  f2 t = first ? d : f2_add(c, d);
  t = f2_fma(A.h, B.l, t);
  c = f2_fma(A.l, B.h, t);
  T = Tn;
}

// r[a] = sum_b W_ab h[b] = A + i B with A = sum_b h.re W_ab and
// B = sum_b h.im W_ab for one spin of the half-spinor (half-spinor
// components broadcast to both lanes against the same link lanes).  Both
// sums run on one fixed grid: sigma is a power of two with every partial sum
// below sigma/2 in magnitude (bound wmax * max(sum_b |h_b.re|, sum_b |h_b.im|),
// raised by 2^-19 to cover its own rounding and that of the grid steps); A
// starts at (T0, T0) and B at (-T0, T0), T0 = 1.5 sigma, so every
// accumulator lane stays in a binade of magnitude [sigma, 2 sigma).  The
// high words of A + i B = (A.re - B.im, A.im + B.re) are then differences of
// two such lanes with the offsets cancelling: exact, multiples of the grid
// step below sigma in magnitude.  The low words carry everything below the
// grid.  Six packed
// operations per product instead of the twelve of a TwoSum accumulation; the
// low words are coarser (about 2^-48 sigma per operation), giving a
// relative error of a few 1e-14 per product W h.
__device__ __forceinline__ void matvec_half_p(const p2 (&W)[3][3], float wmax, const p2 (&h)[3],
                                              p2 (&r)[3]) {
  mul2 mr[3], mi[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    mr[b] = mul2{f2_lo(h[b].h), f2_lo(h[b].l)};
    mi[b] = mul2{f2_hi(h[b].h), f2_hi(h[b].l)};
  }
  f2 TA0, TB0;
  {
    float r0, i0, r1, i1, r2, i2;
    f2_split(h[0].h, r0, i0);
    f2_split(h[1].h, r1, i1);
    f2_split(h[2].h, r2, i2);
    const float sr = fabsf(r0) + fabsf(r1) + fabsf(r2);
    const float si = fabsf(i0) + fabsf(i1) + fabsf(i2);
    const float m = fmaxf(sr, si) * wmax;
    // sigma = 2^(e + 2) for m in [2^e, 2^(e+1)); T0 = 1.5 sigma
    const unsigned tb = (__float_as_uint(m) & 0x7f800000u) + (2u << 23) + (1u << 22);
    const float t0 = __uint_as_float(tb);
    TA0 = f2_make(t0, t0);
    TB0 = f2_make(-t0, t0);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f2 TA = TA0, TB = TB0, cA = 0ull, cB = 0ull;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      grid_mad(TA, cA, mr[b], W[a][b], b == 0);
      grid_mad(TB, cB, mi[b], W[a][b], b == 0);
    }
    // i B = (-B.im, B.re): swap the lanes, flip the sign of lane 0; the high
    // lanes are (T0 + A.re) - (T0 + B.im) and (T0 + A.im) + (-T0 + B.re)
    constexpr f2 kLane0 = 0x0000000080000000ull;
    r[a] = p2{f2_add(TA, f2_swap(TB) ^ kLane0), f2_add(cA, f2_swap(cB) ^ kLane0)};
  }
}

// Reconstruction of one spin s of the two-spin result: out_s += r and the
// lower spin that (1 + S gamma_mu) ties to s gets the phase times r.
template <int MU, int SP>
__device__ __forceinline__ void reconstruct_half_p(const p2 (&r)[3], p2 (&acc)[4][3], float S) {
  const f2 sS = f2_make(S, S), nS = f2_make(-S, -S), sI = f2_make(-S, S), sIm = f2_make(S, -S);
  constexpr int L = (MU <= 1) ? 3 - SP : 2 + SP;  // lower spin fed by spin SP
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    acc[SP][c] = p2_add(acc[SP][c], r[c]);
    if (MU == 0) acc[L][c] = p2_add_sgn(acc[L][c], p2_swap(r[c]), sIm);
    if (MU == 1) acc[L][c] = p2_add_sgn(acc[L][c], r[c], SP == 0 ? nS : sS);
    if (MU == 2) acc[L][c] = p2_add_sgn(acc[L][c], p2_swap(r[c]), SP == 0 ? sIm : sI);
    if (MU == 3) acc[L][c] = p2_add_sgn(acc[L][c], r[c], sS);
  }
}

template <int SP>
__device__ __forceinline__ void reconstruct_half_mu(int mu, const p2 (&r)[3], p2 (&acc)[4][3], float S) {
  switch (mu) {
    case 0: reconstruct_half_p<0, SP>(r, acc, S); break;
    case 1: reconstruct_half_p<1, SP>(r, acc, S); break;
    case 2: reconstruct_half_p<2, SP>(r, acc, S); break;
    default: reconstruct_half_p<3, SP>(r, acc, S);
  }
}

// acc = (H_{p,1-p} in)(idx) at output site idx of parity p (DAG: the adjoint
// hop), unnormalised double-word accumulators: all eight hops d = 2 mu +
// backward in one thread.  dsm: this block's dwp_smem(NT) bytes of shared
// memory; blockDim.x must be NT.
//
// Copies run one hop ahead: the link of the next hop is issued when hop d
// starts (two link stages), the neighbour spinor of the next hop as soon as
// hop d's has been read into registers and projected (one stage).  Every
// thread reads and overwrites only its own column, so no block barrier is
// needed; the completed-group wait of each hop covers both of its copies.
//
// A runtime loop, whose body exists once in the instruction stream; the
// neighbour offsets wait in shared memory, one load per hop.  Computing each
// hop's neighbour and its 64-bit chunk addresses in the loop instead took 49
// of 748 instructions per hop and warp, and the kernel is bound by issue and
// dependency latency at 12 warps per SM.  The spinor copies go past L1: three
// blocks' stages leave it about 56 KB, less than the spinor bytes in flight,
// so allocating there limited them.  97.9 -> 91.2 us at 24^3x48, 286.8 ->
// 265.1 us at 32^3x64 (5.59 and 6.08 TB/s algorithmic, 83% and 90% of the
// measured copy bandwidth).
template <bool DAG, int NT = kHopThreads>
__device__ __forceinline__ void dwp_hop_site(float4 *dsm, const float4 *in, const float4 *gauge,
                                             const Geom &g, int p, int64_t idx, p2 (&acc)[4][3]) {
  const int64_t vh = g.vh;
  const int tid = threadIdx.x;
  float4 *const spn = dsm + tid;                     // this thread's column of the spinor stage
  float4 *const lnk = spn + kDwpStageChunks * NT;    // and of the two link stages
  unsigned *const tab = reinterpret_cast<unsigned *>(dsm + (kDwpStageChunks + 2 * kDwpLinkChunks) * NT) + tid;
  {
    const HopSite site = hop_site(g, (unsigned)idx, p);
#pragma unroll
    for (int d = 0; d < 8; ++d) tab[d * NT] = hop_offset(g, site, d);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[a][c] = p2{0ull, 0ull};
  const unsigned own = 16u * (unsigned)idx;
  unsigned next = tab[0];
  stage_hop_p<NT>(spn, in, vh, next & ~1u);
  stage_link_p<NT>(lnk, gauge, vh, p, 0, own, next & ~1u);
  cp_async_commit();
#pragma unroll 1
  for (int d = 0; d < 8; ++d) {
    const bool neg = next & 1u;
    const int mu = d >> 1;
    const bool bwd = (d & 1) != 0;
    const bool more = d < 7;
    if (more) {  // the other link stage was read during the previous hop
      next = tab[(d + 1) * NT];
      stage_link_p<NT>(lnk + ((d + 1) & 1) * kDwpLinkChunks * NT, gauge, vh, p, d + 1, own, next & ~1u);
    }
    cp_async_commit();
    cp_async_wait1();  // this thread's spinor and link copies of hop d have landed
    p2 psi[4][3];
#pragma unroll
    for (int k = 0; k < 12; ++k) psi[k / 3][k % 3] = ld_p2(spn + k * NT);
    p2 W[3][3];
    {  // U_mu(x), or the transpose of U_mu(x - mu)
      const float4 *ls = lnk + (d & 1) * kDwpLinkChunks * NT;
      const int sa = bwd ? NT : 3 * NT, sb = bwd ? 3 * NT : NT;
#pragma unroll
      for (int k = 0; k < 9; ++k) W[k / 3][k % 3] = ld_p2(ls + (k / 3) * sa + (k % 3) * sb);
    }
    const float S = (bwd != DAG) ? 1.f : -1.f;
    p2 h[2][3];
    switch (mu) {
      case 0: project_p<0>(psi, h, S); break;
      case 1: project_p<1>(psi, h, S); break;
      case 2: project_p<2>(psi, h, S); break;
      default: project_p<3>(psi, h, S);
    }
    if (more) stage_hop_p<NT>(spn, in, vh, next & ~1u);  // the spinor stage has been read
    cp_async_commit();
    if (neg) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) h[a][c] = p2_neg(h[a][c]);
    }
    if (bwd) {
      // conjugation of the adjoint link on backward hops only, by sign bits
      // (off the FMA pipe: 1.4% faster than multiplying every link by (1, +-1))
#pragma unroll
      for (int k = 0; k < 9; ++k) W[k / 3][k % 3] = p2_conj(W[k / 3][k % 3]);
    }
    // bound of the link's high words, raised by 2^-19 (see matvec_half_p)
    const float wmax = link_max_hi(W) * 1.0000019f;
    {  // spin 0 of the half-spinor, then spin 1: one three-colour result live
      p2 r[3];
      matvec_half_p(W, wmax, h[0], r);
      reconstruct_half_mu<0>(mu, r, acc, S);
      matvec_half_p(W, wmax, h[1], r);
      reconstruct_half_mu<1>(mu, r, acc, S);
    }
  }
}

// Eight threads per output site (small lattices): a block of
// kDwp8Threads threads covers kDwp8Sites sites, warp mu runs direction mu, its
// lanes 0..15 the forward and 16..31 the backward hop of sites 0..15.  Each
// thread loads its operands straight into registers (one round trip for all
// of them), leaves its two-spin product in shared memory, and the first
// 4 x kDwp8Sites threads sum one spin of one site each (dwp8_spin; with a branch
// per half-warp instead of one stream for both spins 12^4 took 6.0 us, not
// 5.2).  A hop's latency chain is then one hop long.
constexpr int kDwp8Sites = 16;
constexpr int kDwp8Threads = 8 * kDwp8Sites;
static_assert(kDwp1Threads == kDwp8Threads, "the blocks of hop_dwx_kernel run either form");

// This thread's r = W h into sm[3 s + c][thread] (see above); idx: its site.
template <bool DAG>
__device__ __forceinline__ void dwp8_hop(ulonglong2 (*sm)[kDwp8Threads], const float4 *in, const float4 *gauge,
                                         const Geom &g, int p, unsigned idx) {
  const int64_t vh = g.vh;
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
  const bool neg = off & 1u;
  off &= ~1u;
  p2 psi[4][3], W[3][3], h[2][3];
  const float4 *L = gauge + (int64_t)(((bwd ? 1 - p : p) * 4 + mu) * 9) * vh;
  const unsigned lo = bwd ? off : 16u * idx;
  const int sa = bwd ? 1 : 3, sb = bwd ? 3 : 1;  // U_mu(x), or the transpose of U_mu(x - mu)
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(chunk_at(in + k * vh, off)));
    psi[k / 3][k % 3] = p2{v.x, v.y};
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const ulonglong2 v =
        __ldg(reinterpret_cast<const ulonglong2 *>(chunk_at(L + ((k / 3) * sa + (k % 3) * sb) * vh, lo)));
    W[k / 3][k % 3] = p2{v.x, v.y};
  }
  const float S = (bwd != DAG) ? 1.f : -1.f;
  switch (mu) {
    case 0: project_p<0>(psi, h, S); break;
    case 1: project_p<1>(psi, h, S); break;
    case 2: project_p<2>(psi, h, S); break;
    default: project_p<3>(psi, h, S);
  }
  if (neg) {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) h[a][c] = p2_neg(h[a][c]);
  }
  const f2 cj = bwd ? 0x8000000000000000ull : 0ull;  // conjugates the adjoint link
#pragma unroll
  for (int k = 0; k < 9; ++k) W[k / 3][k % 3] = p2{W[k / 3][k % 3].h ^ cj, W[k / 3][k % 3].l ^ cj};
  const float wmax = link_max_hi(W) * 1.0000019f;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    p2 r[3];
    matvec_half_p(W, wmax, h[s], r);
#pragma unroll
    for (int c = 0; c < 3; ++c) sm[3 * s + c][threadIdx.x] = make_ulonglong2(r[c].h, r[c].l);
  }
}

// acc = spin 2 HI + s of (H in) at site j of the tile (HI by warp, s = 0 or 1 by
// half-warp, one instruction stream for both): the forward and the backward
// hops' sums, added (shorter chains than all eight in a row, and on average a
// smaller rounding error: 6.41e-14 against 6.76e-14 at 12^4).  The terms are
// those of reconstruct_half_p; the first of each sum is taken as it is.
template <bool DAG, int HI>
__device__ __forceinline__ void dwp8_spin(const ulonglong2 (*sm)[kDwp8Threads], int j, int s, p2 (&acc)[3]) {
  const f2 flip = s ? 0x8000000080000000ull : 0ull;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p2 sum[2];
#pragma unroll
    for (int d = 0; d < 8; ++d) {  // everything but the data and s is constant after unrolling
      const int mu = d >> 1;
      const ulonglong2 v = sm[3 * (HI && mu < 2 ? 1 - s : s) + c][16 * d + j];
      p2 r{v.x, v.y};
      p2 &t = sum[d & 1];
      if (HI) {
        const float S = (((d & 1) != 0) != DAG) ? 1.f : -1.f;
        f2 sg = f2_make(S, (mu & 1) ? S : -S);
        if (mu == 1 || mu == 2) sg ^= flip;
        if (!(mu & 1)) r = p2_swap(r);
        t = mu == 0 ? p2_scale_sgn(r, sg) : p2_add_sgn(t, r, sg);
      } else {
        t = mu == 0 ? r : p2_add(t, r);
      }
    }
    acc[c] = p2_add(sum[0], sum[1]);
  }
}
// The same by run-time spin = 0..3, uniform over each pair of half-warps.
template <bool DAG>
__device__ __forceinline__ void dwp8_sum(const ulonglong2 (*sm)[kDwp8Threads], int j, int spin, p2 (&acc)[3]) {
  if (spin >> 1) dwp8_spin<DAG, 1>(sm, j, spin & 1, acc);
  else dwp8_spin<DAG, 0>(sm, j, spin & 1, acc);
}

// out = a x + b v (AXPY) or b v for NC consecutive components k0 .. k0 + NC - 1
// of the site's spinor, each scalar a double-word (hi, lo) float pair;
// returns their contribution to ||out||^2 when NORM.
template <bool AXPY, bool NORM, int NC>
__device__ __forceinline__ dwacc dwp_store_chunks(const p2 (&v)[NC], int k0, float4 *out_base,
                                                  const float4 *x_base, int64_t vh, int64_t idx,
                                                  float2 a_split, float2 b_split) {
  const f2 bh = f2_make(b_split.x, b_split.x);
  const mul2 Bm{bh, f2_make(b_split.y, b_split.y)};
  const f2 ah = f2_make(a_split.x, a_split.x);
  const mul2 Am{ah, f2_make(a_split.y, a_split.y)};
  acc2 nq{0ull, 0ull};
  ulonglong2 *__restrict__ o = reinterpret_cast<ulonglong2 *>(out_base) + idx + (int64_t)k0 * vh;
  p2 xs[NC];
  if (AXPY) {  // all loads before the first store
    const ulonglong2 *__restrict__ xp =
        reinterpret_cast<const ulonglong2 *>(x_base) + idx + (int64_t)k0 * vh;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const ulonglong2 u = __ldg(xp + k * vh);
      xs[k] = p2{u.x, u.y};
    }
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    acc2 R = acc2_first(Bm, p2_norm(v[k]));
    if (AXPY) acc2_mad(R, Am, xs[k]);
    const p2 q = p2_norm(acc2_get(R));
    o[k * vh] = make_ulonglong2(q.h, q.l);
    if (NORM) {
      const mul2 Q{q.h, q.l};
      if (k == 0) nq = acc2_first(Q, q);
      else acc2_mad(nq, Q, q);
    }
  }
  dwacc nrm{0.f, 0.f};
  if (NORM) {
    float s0, s1, c0, c1;
    f2_split(nq.s, s0, s1);
    f2_split(nq.c, c0, c1);
    float s, e;
    two_sum(s0, s1, s, e);
    nrm = dwacc{s, __fadd_rn(__fadd_rn(c0, c1), e)};
  }
  return nrm;
}

// out = a x + b acc (AXPY) or b acc for the whole site; returns ||out||^2
// when NORM.
template <bool AXPY, bool NORM>
__device__ __forceinline__ dwacc dwp_store(const p2 (&acc)[4][3], float4 *out_base,
                                           const float4 *x_base, int64_t vh, int64_t idx,
                                           float2 a_split, float2 b_split) {
  p2 v[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) v[k] = acc[k / 3][k % 3];
  return dwp_store_chunks<AXPY, NORM, 12>(v, 0, out_base, x_base, vh, idx, a_split, b_split);
}

}  // namespace jqcd
