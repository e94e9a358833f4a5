// Device code that the verifiers share: results and pair geometry.
#pragma once

#include "mj_internal.cuh"

namespace mj {
namespace {

// The P planes' words of position word w (2-plane codes: 8 bytes, others 32).
template <int P>
__device__ __forceinline__ void load_plane_words(const uint32_t* __restrict__ planes, int64_t w, uint32_t (&x)[P]) {
  if constexpr (P == 2) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(planes) + w);
    x[0] = v.x;
    x[1] = v.y;
  } else {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(planes) + 2 * w);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
    if constexpr (P == 5) {
      x[4] = __ldg(planes + 8 * w + 4);
    } else {
      const uint4 u = __ldg(reinterpret_cast<const uint4*>(planes) + 2 * w + 1);
      x[4] = u.x;
      x[5] = u.y;
      x[6] = u.z;
      if constexpr (P == 8) x[7] = u.w;
    }
  }
}

// Result of pair t: ed[t] = v; a pair within the join's threshold (v <= K)
// is also listed in out_t (when given), so the join's output needs no pass
// over all candidates.
__device__ __forceinline__ void put_result(const VerifyArgs& a, uint64_t t, uint32_t v) {
  a.ed[t] = v;
  if (a.out_t && v <= a.K) a.out_t[atomicAdd(a.out_count, 1ull)] = (uint32_t)t;
}

// Geometry of the pair at order position q (index t): offsets of A (the
// longer string) and B, their lengths; false for an id out of range.
__device__ __forceinline__ bool pair_geometry(const VerifyArgs& a, uint64_t q, uint64_t t, int64_t& oA, int64_t& oB,
                                              int64_t& m, int64_t& n) {
  if (a.pair_geo) {   // written with the order: one load, no chain through the ids
    const uint4 g = a.pair_geo[q];
    if (g.w == kGeoBadIds) return false;
    oA = g.x;
    oB = g.y;
    m = g.z;
    n = g.w;
    return true;
  }
  const uint32_t x = a.pi[t], y = a.pj[t];
  if (x >= a.n_strings || y >= a.n_strings) return false;
  const int64_t ox = __ldg(a.offsets + x), lx = __ldg(a.offsets + x + 1) - ox;
  const int64_t oy = __ldg(a.offsets + y), ly = __ldg(a.offsets + y + 1) - oy;
  const bool xa = lx >= ly;
  oA = xa ? ox : oy;
  m = xa ? lx : ly;
  oB = xa ? oy : ox;
  n = xa ? ly : lx;
  return true;
}

}  // namespace
}  // namespace mj
