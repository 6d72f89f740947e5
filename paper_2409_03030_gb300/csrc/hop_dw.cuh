// Building blocks shared by the hop kernels of every precision: per-site
// norms of a hop's output, the cp.async helpers of the staged hops, and the
// neighbour lookup with its boundary sign.
#pragma once
#include "fields.cuh"
#include "hop.cuh"
#include "kernels.h"

namespace jqcd {

template <int PREC> __device__ __forceinline__ dwacc site_norm2(const typename PT<PREC>::C (&o)[4][3]);
template <> __device__ __forceinline__ dwacc site_norm2<PREC_DW>(const cw (&o)[4][3]) {
  dwacc A = acc_first(o[0][0].re, o[0][0].re);
  acc_sq(A, o[0][0].im);
#pragma unroll
  for (int k = 1; k < 12; ++k) {
    acc_sq(A, o[k / 3][k % 3].re);
    acc_sq(A, o[k / 3][k % 3].im);
  }
  return A;
}
template <int PREC> __device__ __forceinline__ dwacc site_norm2_f(const cf (&o)[4][3]) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < 12; ++k) s = fmaf(o[k / 3][k % 3].re, o[k / 3][k % 3].re, fmaf(o[k / 3][k % 3].im, o[k / 3][k % 3].im, s));
  return dwacc{s, 0.f};
}
template <> __device__ __forceinline__ dwacc site_norm2<PREC_F32>(const cf (&o)[4][3]) { return site_norm2_f<PREC_F32>(o); }
template <> __device__ __forceinline__ dwacc site_norm2<PREC_F16N>(const cf (&o)[4][3]) { return site_norm2_f<PREC_F16N>(o); }

// ---------------------------------------------------------------------------
// Staged hops copy the operands of the next hop into shared memory (cp.async,
// two stages), so each warp's memory latency overlaps its own arithmetic
// instead of depending on other resident warps.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, bool keep_l1) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  if (keep_l1)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Neighbour of hop d (mu = d/2, backward when d is odd) and its boundary sign.
__device__ __forceinline__ int64_t hop_neighbour(const Geom &g, int x, int y, int z, int t, int d,
                                                 bool &neg) {
  const int mu = d >> 1;
  const bool bwd = (d & 1) != 0;
  neg = false;
  if (!bwd) {
    switch (mu) {
      case 0: x = (x + 1 == g.nx) ? 0 : x + 1; break;
      case 1: y = (y + 1 == g.ny) ? 0 : y + 1; break;
      case 2: z = (z + 1 == g.nz) ? 0 : z + 1; break;
      default: if (t + 1 == g.nt) { t = 0; neg = g.tanti != 0; } else t = t + 1;
    }
  } else {
    switch (mu) {
      case 0: x = (x == 0) ? g.nx - 1 : x - 1; break;
      case 1: y = (y == 0) ? g.ny - 1 : y - 1; break;
      case 2: z = (z == 0) ? g.nz - 1 : z - 1; break;
      default: if (t == 0) { t = g.nt - 1; neg = g.tanti != 0; } else t = t - 1;
    }
  }
  return cb_index(g, x, y, z, t);
}

// A site of one parity and its neighbours in 32-bit arithmetic: a resident
// gauge field takes 2688 bytes per site of one parity, so vh < 2^27 on any
// device and 16 idx < 2^31.  The hops', fused hops' and force's launches refuse
// more; a batch admits a solve by launch_hop on its field.
constexpr int64_t kMaxHopSites = (int64_t)1 << 27;
struct HopSite {
  unsigned idx, xh, y, z, t;
  bool odd;  // x = 2 xh + odd
};
__device__ __forceinline__ HopSite hop_site(const Geom &g, unsigned idx, int p) {
  HopSite s;
  s.idx = idx;
  s.xh = idx % (unsigned)g.nxh;
  unsigned r = idx / (unsigned)g.nxh;
  s.y = r % (unsigned)g.ny;
  r /= (unsigned)g.ny;
  s.z = r % (unsigned)g.nz;
  s.t = r / (unsigned)g.nz;
  s.odd = (s.y + s.z + s.t + p) & 1;
  return s;
}

// Byte offset (16 x checkerboard index) of the neighbour of hop d = 2 mu +
// backward; bit 0 is set when the hop crosses an antiperiodic time boundary.
// d is a constant where the hops are unrolled.  One select of a constant step
// and one 32-bit offset beside grid-uniform chunk planes replace about 25
// instructions of 64-bit coordinates-to-index arithmetic per hop and two per
// chunk address.
__device__ __forceinline__ unsigned hop_offset(const Geom &g, const HopSite &s, int d) {
  const unsigned idx = s.idx, nxh = g.nxh, sz = nxh * (unsigned)g.ny, st = sz * (unsigned)g.nz;
  switch (d) {
    case 0: return 16u * (s.odd ? (s.xh + 1 == nxh ? idx + 1 - nxh : idx + 1) : idx);
    case 1: return 16u * (s.odd ? idx : (s.xh == 0 ? idx + nxh - 1 : idx - 1));
    case 2: return 16u * (s.y + 1 == (unsigned)g.ny ? idx + nxh - sz : idx + nxh);
    case 3: return 16u * (s.y == 0 ? idx + sz - nxh : idx - nxh);
    case 4: return 16u * (s.z + 1 == (unsigned)g.nz ? idx + sz - st : idx + sz);
    case 5: return 16u * (s.z == 0 ? idx + st - sz : idx - sz);
    case 6: {
      const bool e = s.t + 1 == (unsigned)g.nt;
      return 16u * (e ? idx + st - (unsigned)g.vh : idx + st) | (e && g.tanti ? 1u : 0u);
    }
    default: {
      const bool e = s.t == 0;
      return 16u * (e ? idx + (unsigned)g.vh - st : idx - st) | (e && g.tanti ? 1u : 0u);
    }
  }
}

// Address of the 16-byte chunk at byte offset off of a chunk plane.
template <typename T> __device__ __forceinline__ const T *chunk_at(const T *plane, unsigned off) {
  return reinterpret_cast<const T *>(reinterpret_cast<const char *>(plane) + off);
}

}  // namespace jqcd
