// ORAS preconditioner apply with the sparse local factors (fronts.cu):
//   z = sum_s R_s^T D_s A_s^{-1} R_s v,   A_s = L D L^T by nodes with panels [S; L].
// Forward, from the leaves: a node's right-hand side is b on its own unknowns plus what its children
// hand up, y = b + sum of theirs; it hands up u = (the children's on its border) - L y.  Backward, from
// the roots: x = S y - L^T x(border), the panel [S; L] times [y; -x(border)] column by column (S is
// symmetric).  Every panel is read once a direction.  All nodes of a tree level run in one launch; a
// border row is formed by one block and children are added in a fixed order, so results do not depend on
// scheduling (OAS adds overlapping contributions into z with atomics).
//
// Bound: HBM, (S + 2 L) entries of 8 B (FP32): 3.5 GB a pass on the 16^3 degree-2 64-subdomain problem,
// where dense factors of the same matrices were 87 GB.
#include "fronts.h"

#include <algorithm>

#include "apply.cuh"

namespace oras {

struct FrApply {
  const FrontNode* nodes;
  const int32_t* child;
  const int32_t* border;
  const int32_t* map;
  const int32_t* row_dof;
  const uint8_t* row_pou;
  int weights;
  int64_t vs, off;   // v and z: right-hand side r of unknown g at g * vs + off + r
  int nr;            // live right-hand sides of the pass (<= KR)
};

constexpr int FR_THREADS = 256;
constexpr int FR_MAX_NB = 128;

// Handed up by the children at front index i (own unknowns, then border).
template <typename R, int KR>
__device__ __forceinline__ CT<R> pull_vec(const FrApply& a, const FrontNode& n, const CT<R>* __restrict__ u, int i,
                                          int r) {
  CT<R> t = {R(0), R(0)};
  for (int c = 0; c < n.nch; ++c) {
    const FrontNode& ch = a.nodes[a.child[n.child0 + c]];
    const int ci = n.map >= 0 ? a.map[n.map + (int64_t)c * (n.n1 + n.n2) + i] : i;
    if (ci < 0) continue;
    const CT<R> v = u[(ch.bord + ci) * KR + r];
    t.re += v.re;
    t.im += v.im;
  }
  return t;
}

// One block: 64 border rows of a node, 8 lanes a row.
template <typename R, int KR>
__global__ void __launch_bounds__(FR_THREADS) k_fr_fwd(FrApply a, const FrontItem* __restrict__ items,
                                                       const CT<R>* __restrict__ fac, const cplx* __restrict__ v,
                                                       CT<R>* __restrict__ y, CT<R>* __restrict__ u) {
  __shared__ __align__(16) CT<R> own[KR][FR_MAX_NB];
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, ld = n.ld;
  for (int e = threadIdx.x; e < ld * KR; e += FR_THREADS) {
    const int c = e / KR, r = e % KR;
    CT<R> t = {R(0), R(0)};
    if (c < n1) {
      if (r < a.nr) {
        const cplx b = v[(int64_t)a.row_dof[n.row0 + c] * a.vs + a.off + r];
        t = {R(b.re), R(b.im)};
      }
      const CT<R> up = pull_vec<R, KR>(a, n, u, c, r);
      t.re += up.re;
      t.im += up.im;
      if (it.t == 0) y[(int64_t)(n.row0 + c) * KR + r] = t;
    }
    own[r][c] = t;
  }
  __syncthreads();
  const int sub = threadIdx.x & 7;
#pragma unroll
  for (int rr = 0; rr < FR_FWD_ROWS; rr += FR_THREADS / 8) {
    const int i = it.t * FR_FWD_ROWS + rr + (threadIdx.x >> 3);
    CT<R> acc[KR];
#pragma unroll
    for (int r = 0; r < KR; ++r) acc[r] = {R(0), R(0)};
    if (i < n.n2) {
      const CT<R>* row = fac + n.panel + (int64_t)(n1 + i) * ld;
#pragma unroll 4
      for (int c = 2 * sub; c < ld; c += 16) {
        CT<R> m0, m1;
        ld_cpair(row + c, m0, m1);
#pragma unroll
        for (int r = 0; r < KR; ++r) {
          CT<R> y0, y1;
          ld_cpair(&own[r][c], y0, y1);
          CT<R>& t = acc[r];
          t.re = fma(m0.re, y0.re, t.re); t.re = fma(-m0.im, y0.im, t.re);
          t.re = fma(m1.re, y1.re, t.re); t.re = fma(-m1.im, y1.im, t.re);
          t.im = fma(m0.re, y0.im, t.im); t.im = fma(m0.im, y0.re, t.im);
          t.im = fma(m1.re, y1.im, t.im); t.im = fma(m1.im, y1.re, t.im);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < KR; ++r) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        acc[r].re += __shfl_xor_sync(0xffffffffu, acc[r].re, o);
        acc[r].im += __shfl_xor_sync(0xffffffffu, acc[r].im, o);
      }
      if (i < n.n2 && sub == r) {  // KR <= 8 lanes: one right-hand side each
        const CT<R> up = pull_vec<R, KR>(a, n, u, n1 + i, r);
        u[(n.bord + i) * KR + r] = {up.re - acc[r].re, up.im - acc[r].im};
      }
    }
  }
}

// One block: 32 own unknowns of a node, lane = unknown, the warps share the panel's rows.
template <typename R, typename ZT, int KR>
__global__ void __launch_bounds__(FR_THREADS) k_fr_bwd(FrApply a, const FrontItem* __restrict__ items,
                                                       const CT<R>* __restrict__ fac, const CT<R>* __restrict__ y,
                                                       CT<R>* __restrict__ x, ZT* __restrict__ z) {
  constexpr int ROWS = 256, NW = FR_THREADS / 32;
  __shared__ CT<R> w[ROWS][KR];
  __shared__ CT<R> red[NW][32][KR];
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, m = n.n1 + n.n2, ld = n.ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = it.t * FR_BWD_COLS + lane;
  const CT<R>* panel = fac + n.panel;
  CT<R> acc[KR];
#pragma unroll
  for (int r = 0; r < KR; ++r) acc[r] = {R(0), R(0)};
  for (int r0 = 0; r0 < m; r0 += ROWS) {
    const int rows = m - r0 < ROWS ? m - r0 : ROWS;
    __syncthreads();
    for (int e = threadIdx.x; e < rows * KR; e += FR_THREADS) {
      const int i = r0 + e / KR, r = e % KR;
      if (i < n1) {
        w[e / KR][r] = y[(int64_t)(n.row0 + i) * KR + r];
      } else {
        const CT<R> t = x[(int64_t)a.border[n.bord + i - n1] * KR + r];
        w[e / KR][r] = {-t.re, -t.im};
      }
    }
    __syncthreads();
    if (j < ld) {
#pragma unroll 8
      for (int i = warp; i < rows; i += NW) {
        const CT<R> mm = panel[(int64_t)(r0 + i) * ld + j];
#pragma unroll
        for (int r = 0; r < KR; ++r) {
          const CT<R> t = w[i][r];
          acc[r].re = fma(mm.re, t.re, acc[r].re); acc[r].re = fma(-mm.im, t.im, acc[r].re);
          acc[r].im = fma(mm.re, t.im, acc[r].im); acc[r].im = fma(mm.im, t.re, acc[r].im);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < KR; ++r) red[warp][lane][r] = acc[r];
  __syncthreads();
  for (int e = threadIdx.x; e < 32 * KR; e += FR_THREADS) {
    const int l = e / KR, r = e % KR, c = it.t * FR_BWD_COLS + l;
    if (c >= n1) continue;
    CT<R> t = red[0][l][r];
#pragma unroll
    for (int q = 1; q < NW; ++q) {
      t.re += red[q][l][r].re;
      t.im += red[q][l][r].im;
    }
    const int64_t row = n.row0 + c;
    x[row * KR + r] = t;
    if (r >= a.nr) continue;
    ZT* dst = z + (int64_t)a.row_dof[row] * a.vs + a.off + r;
    if (a.weights == ORAS_WEIGHTS_POU) {
      if (a.row_pou[row]) z_store(dst, (double)t.re, (double)t.im);
    } else {
      z_add(dst, (double)t.re, (double)t.im);
    }
  }
}

// ------------------------------------------------------------------ host side
// Right-hand sides of the next pass when `rem` are left.
static int fr_kr(const oras_handle* h, int rem) {
  if (h->opt.factor_bits == 64) return rem >= 2 ? 2 : 1;
  return rem >= 5 ? 8 : (rem >= 3 ? 4 : rem);
}

size_t fronts_ybytes(const oras_handle* h, int k) {
  const Fronts& f = h->fronts;
  const size_t el = h->opt.factor_bits == 64 ? sizeof(CT<double>) : sizeof(CT<float>);
  return (size_t)(2 * h->mesh.sub_ns_off[h->mesh.nsub] + f.border_elems) * el * fr_kr(h, k);
}

int fronts_passes(const oras_handle* h, int k) {
  int n = 0;
  for (int r0 = 0; r0 < k; ++n) r0 += fr_kr(h, k - r0);
  return n;
}

template <typename R, typename ZT, int KR>
static void fr_pass(const oras_handle* h, const cplx* v, ZT* z, int64_t vs, int64_t off, int nr) {
  const auto& d = h->dev;
  const Fronts& f = h->fronts;
  FrApply a;
  a.nodes = d.fr_nodes; a.child = d.fr_child; a.border = d.fr_border; a.map = d.fr_map;
  a.row_dof = d.fr_row_dof; a.row_pou = d.fr_row_pou;
  a.weights = h->opt.weights;
  a.vs = vs; a.off = off; a.nr = nr;
  const int64_t rows = h->mesh.sub_ns_off[h->mesh.nsub];
  CT<R>* y = (CT<R>*)d.ybuf;
  CT<R>* x = y + rows * KR;
  CT<R>* u = x + rows * KR;
  const CT<R>* fac = (const CT<R>*)d.arena;
  for (int l = 0; l < f.nlev(); ++l)
    k_fr_fwd<R, KR><<<(unsigned)(f.fwd.ptr[l + 1] - f.fwd.ptr[l]), FR_THREADS, 0, d.stream>>>(
        a, d.fr_fwd + f.fwd.ptr[l], fac, v, y, u);
  for (int l = f.nlev() - 1; l >= 0; --l)
    k_fr_bwd<R, ZT, KR><<<(unsigned)(f.bwd.ptr[l + 1] - f.bwd.ptr[l]), FR_THREADS, 0, d.stream>>>(
        a, d.fr_bwd + f.bwd.ptr[l], fac, y, x, z);
  count_launches(2 * f.nlev());
}

// z = M^{-1} v for k right-hand sides; right-hand side r of unknown g at g * vs + r * rs of v and z
// (rs = 1: adjacent, vs = k; else one at a time).
template <typename R, typename ZT>
static int fr_apply_t(const oras_handle* h, const cplx* v, ZT* z, int k, int64_t vs, int64_t rs) {
  const auto& d = h->dev;
  if (!d.ybuf || d.ybuf_bytes < fronts_ybytes(h, rs == 1 ? k : 1)) return -1;
  if (h->opt.weights != ORAS_WEIGHTS_POU &&
      cudaMemsetAsync(z, 0, sizeof(ZT) * (size_t)h->mesh.ndof * k, d.stream) != cudaSuccess)
    return -1;
  for (int r0 = 0; r0 < k;) {
    const int kr = rs == 1 ? fr_kr(h, k - r0) : 1, nr = std::min(kr, k - r0);
    const int64_t off = r0 * rs;
    if (kr == 1) fr_pass<R, ZT, 1>(h, v, z, vs, off, nr);
    else if (kr == 2) fr_pass<R, ZT, 2>(h, v, z, vs, off, nr);
    else if constexpr (sizeof(R) == 4) {
      if (kr == 4) fr_pass<R, ZT, 4>(h, v, z, vs, off, nr);
      else fr_pass<R, ZT, 8>(h, v, z, vs, off, nr);
    }
    r0 += nr;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int fronts_apply_f64out(const oras_handle* h, const cplx* v, cplx* z, int k, int64_t vs, int64_t rs) {
  return h->dev.factor_bits == 64 ? fr_apply_t<double, cplx>(h, v, z, k, vs, rs)
                                  : fr_apply_t<float, cplx>(h, v, z, k, vs, rs);
}
int fronts_apply_f32out(const oras_handle* h, const cplx* v, void* z, int k) {
  return fr_apply_t<float, CT<float>>(h, v, (CT<float>*)z, k, k, 1);
}

}  // namespace oras
