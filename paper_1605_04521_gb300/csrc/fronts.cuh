// Device side of the elimination-tree plan, shared by the factorisation kernels (fronts.cu, fronts_tc.cu).
#pragma once

#include "dev.cuh"

namespace oras {

// device copies of the plan (fronts.h)
struct FrDev {
  const FrontNode* nodes;
  const int32_t* border;
  const FrontSrc* own_src;
  const FrontSrc* border_src;
  uint8_t* weak;
};

// Node g needs some of its unknowns eliminated later.
__device__ __forceinline__ void mark_weak(const FrDev& f, int g, int32_t* status) {
  f.weak[g] = 1;
  status[ST_WEAK] = 1;
}
__device__ __forceinline__ bool grown(float re, float im) { return !(fmaxf(fabsf(re), fabsf(im)) <= FR_GROWTH); }

__device__ __forceinline__ FrontSrc front_src(const FrDev& f, const FrontNode& n, int i) {
  return i < n.n1 ? f.own_src[n.row0 + i] : f.border_src[n.bord + i - n.n1];
}

// The children's contributions to an entry of the front of node n whose rows have the sources s and t
// (lower entries of their blocks are stored).
template <typename R>
__device__ __forceinline__ CT<R> pull(const FrDev& f, const FrontNode& n, const CT<R>* __restrict__ C, FrontSrc s,
                                      FrontSrc t) {
  CT<R> r = {R(0), R(0)};
  if (s.a >= 0 && t.a >= 0) {
    const FrontNode& c = f.nodes[n.child[0]];
    const int64_t lo = min(s.a, t.a) - c.bord, hi = max(s.a, t.a) - c.bord;
    r = C[c.cblk + hi * c.ldc + lo];
  }
  if (s.b >= 0 && t.b >= 0) {
    const FrontNode& c = f.nodes[n.child[1]];
    const int64_t lo = min(s.b, t.b) - c.bord, hi = max(s.b, t.b) - c.bord;
    const CT<R> v = C[c.cblk + hi * c.ldc + lo];
    r.re += v.re;
    r.im += v.im;
  }
  return r;
}

}  // namespace oras
