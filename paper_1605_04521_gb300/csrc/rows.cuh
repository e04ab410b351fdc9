// Row assembly shared by the global matrix and the local matrices (assemble.cu, fronts.cu).
#pragma once

#include "dev.cuh"

namespace oras {

// ------------------------------------------------------------------ row assembly
// One warp per matrix row.  Contributions are summed in a fixed order (tets ascending, then
// impedance faces ascending) into FP64 accumulators indexed by the row's CSR pattern, so the
// result is deterministic.  GLOBAL: the row of A (outer faces only).  LOCAL: the row of A_s for
// subdomain s -- only tets of Omega_s^delta, outer faces of those tets, and faces with exactly
// one tet in Omega_s^delta (impedance transmission, omega~ of the inside tet) -- written to the
// dense tiled arena (column-major TB x TB tiles).
struct RowArgs {
  int nl, nfl;
  double k0;
  const int32_t* dofmap;
  const int64_t* tinc_ptr; const int32_t* tinc;
  const int64_t* finc_ptr; const int32_t* finc;
  const int32_t* if_tet0; const int32_t* if_tet1; const int32_t* if_dofs;
  const int64_t* rowptr; const int32_t* cols;
  const cplx* elem; const double* fmat;
  const cplx* eps; const cplx* mu;
  const double* if_beta;     // [nif] caller's beta of outer faces, or nullptr (derived)
  const uint8_t* fixed;      // [ndof] constrained by a metallic face (identity row and column), or nullptr
  const uint32_t* member; int64_t member_words;
  int dirichlet;             // local rows: 1 = rows of the global matrix (RAS), 0 = ORAS local problem
};

__device__ __forceinline__ int bsearch32(const int32_t* a, int n, int32_t key) {
  int lo = 0, hi = n - 1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    int32_t v = a[mid];
    if (v == key) return mid;
    if (v < key) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

__device__ __forceinline__ double omega_t(const RowArgs& A, int64_t t) {
  double mr = A.mu ? A.mu[t].re : 1.0;
  return A.k0 * sqrt(mr * A.eps[t].re);
}

__device__ __forceinline__ bool is_member(const RowArgs& A, int s, int64_t t) {
  return (A.member[(int64_t)s * A.member_words + (t >> 5)] >> (t & 31)) & 1u;
}

template <bool LOCAL>
__device__ __forceinline__ void accumulate_row(const RowArgs& A, int64_t g, int s, cplx* acc, int rn,
                               const int32_t* rc) {
  const int lane = threadIdx.x & 31;
  for (int p = lane; p < rn; p += 32) acc[p] = {0.0, 0.0};
  __syncwarp();
  for (int64_t q = A.tinc_ptr[g]; q < A.tinc_ptr[g + 1]; ++q) {
    int32_t e = A.tinc[q];
    int64_t t = e / A.nl;
    int a = e - (int)t * A.nl;
    if (LOCAL && !is_member(A, s, t)) continue;
    const cplx* er = A.elem + (t * A.nl + a) * A.nl;
    for (int b = lane; b < A.nl; b += 32) {
      int p = bsearch32(rc, rn, A.dofmap[t * A.nl + b]);
      if (p >= 0) acc[p] = cadd(acc[p], er[b]);
    }
    __syncwarp();
  }
  for (int64_t q = A.finc_ptr[g]; q < A.finc_ptr[g + 1]; ++q) {
    int32_t e = A.finc[q];
    int64_t slot = e / A.nfl;
    int af = e - (int)slot * A.nfl;
    int64_t t0 = A.if_tet0[slot], t1 = A.if_tet1[slot];
    int64_t tin;
    if (t1 < 0) {
      if (LOCAL && !is_member(A, s, t0)) continue;
      tin = t0;
    } else {
      if (!LOCAL) continue;
      bool m0 = is_member(A, s, t0), m1 = is_member(A, s, t1);
      if (m0 == m1) continue;
      tin = m0 ? t0 : t1;
    }
    // outer faces: the caller's beta when given; interfaces: omega~ of the inside tet
    double w = (t1 < 0 && A.if_beta) ? A.if_beta[slot] : omega_t(A, tin);
    const double* fr = A.fmat + (slot * A.nfl + af) * A.nfl;
    for (int bf = lane; bf < A.nfl; bf += 32) {
      int p = bsearch32(rc, rn, A.if_dofs[slot * A.nfl + bf]);
      if (p >= 0) acc[p].im += w * fr[bf];
    }
    __syncwarp();
  }
}

constexpr int ROW_WARPS = 8;

RowArgs row_args(const oras_handle* h, double k0);

}  // namespace oras
