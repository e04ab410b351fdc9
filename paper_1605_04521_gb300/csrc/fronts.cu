// Batched sparse factorisation of the local matrices A_s (Sec. 4: the A_s^{-1} of ORAS).
//
// Every A_s is complex symmetric (the element, face and transmission terms all are, and constrained
// unknowns get identity rows and columns), so it is factored as block L D L^T over its elimination
// tree (fronts_plan.cpp) by the multifrontal method.  A node's front is its own n1 unknowns and its
// border of n2 later ones; with A11, A21 its assembled panel,
//   S = A11^{-1},   L = A21 S,   C = A22 - L A21^T,
// and the parent adds C's entries to its own front.  The solve needs only [S; L] (fronts_apply.cu).
// All nodes of a tree level, of all subdomains, go through each step in one launch:
//   k_fr_assemble  the children's C added to the panels (originals are scattered once, k_fr_rows);
//   k_fr_invert    S by Gauss-Jordan with row pivoting, the block held in registers;
//   k_fr_mul       L, then C with the children's C gathered into it (each C is read once).
// Pivots are chosen inside a pivot block (up to front_nb unknowns) and never outside it, so the tree
// stays as planned.
//
// Against dense factors of the same matrices (n_s^2 entries each) the largest subdomain of the
// 16^3 x 6, degree-2, 64-subdomain problem (17,896 unknowns) keeps 2% of the entries and needs 0.1%
// of the products.  FP32 factors are FP32 throughout (no TF32 operands): against FP64 solves their
// error is 5e-7 at degree 2 and 3e-6 at degree 3 or without losses, that of a dense FP32 LU with
// partial pivoting (1e-6 and 5e-6).
#include "rows.cuh"

namespace oras {

// device copies of the plan (fronts.h)
struct FrDev {
  const FrontNode* nodes;
  const int32_t* border;
  const FrontSrc* own_src;
  const FrontSrc* border_src;
};

static FrDev fr_dev(const oras_handle* h) {
  const auto& d = h->dev;
  return {d.fr_nodes, d.fr_border, d.fr_own_src, d.fr_border_src};
}

// ------------------------------------------------------------------ original entries
// Row i of A_s (one warp): its entries whose column is eliminated with or after it go to its node's
// panel, in the column of row i (A_s is symmetric).  The workspace is cleared before.
template <typename R>
__global__ void k_fr_rows(RowArgs A, FrDev f, int nsub, int64_t total_rows, const int64_t* __restrict__ ns_off,
                          const int32_t* __restrict__ sub_dofs, const int32_t* __restrict__ pos,
                          const int32_t* __restrict__ row_node, int maxnnz, CT<R>* __restrict__ work) {
  extern __shared__ cplx sacc[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * ROW_WARPS + w;
  if (row >= total_rows) return;
  int lo = 0, hi = nsub - 1;
  while (lo < hi) {  // last s with ns_off[s] <= row
    const int mid = (lo + hi + 1) >> 1;
    if (ns_off[mid] <= row) lo = mid; else hi = mid - 1;
  }
  const int s = lo;
  const int64_t base = ns_off[s];
  const int ns = (int)(ns_off[s + 1] - base);
  const int32_t* Ns = sub_dofs + base;
  const int32_t at = (int32_t)(base + pos[row]);  // elimination position
  const FrontNode n = f.nodes[row_node[at]];
  const int col = at - n.row0;
  const int64_t g = sub_dofs[row];
  if (A.fixed && A.fixed[g]) {  // constrained by a metallic face: identity row
    if (lane == 0) work[n.panel + (int64_t)col * n.ld + col] = {R(1), R(0)};
    return;
  }
  cplx* acc = sacc + w * maxnnz;
  const int64_t r0 = A.rowptr[g];
  const int rn = (int)(A.rowptr[g + 1] - r0);
  const int32_t* rc = A.cols + r0;
  if (A.dirichlet) accumulate_row<false>(A, g, s, acc, rn, rc);  // R_s A R_s^T: the global row
  else accumulate_row<true>(A, g, s, acc, rn, rc);
  for (int p = lane; p < rn; p += 32) {
    if (A.fixed && A.fixed[rc[p]]) continue;  // constrained column: zero
    const int lj = bsearch32(Ns, ns, rc[p]);
    if (lj < 0) continue;
    const int32_t c = (int32_t)(base + pos[base + lj]);
    int i = c - n.row0;
    if (i < 0) continue;  // eliminated before: in that node's panel
    if (i >= n.n1) {
      i = bsearch32(f.border + n.bord, n.n2, c);
      if (i < 0) continue;  // no coupling inside this subdomain (an exact zero of A_s)
      i += n.n1;
    }
    work[n.panel + (int64_t)i * n.ld + col] = {R(acc[p].re), R(acc[p].im)};
  }
}

// ------------------------------------------------------------------ children's contributions
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

// Panel rows of the nodes with children: 32 rows a block, lanes along the own columns.
template <typename R>
__global__ void __launch_bounds__(256) k_fr_assemble(FrDev f, const FrontItem* __restrict__ items,
                                                     CT<R>* __restrict__ work, const CT<R>* __restrict__ C) {
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = f.nodes[it.node];
  const int r0 = it.t * FR_ASM_ROWS;
  const int rows = n.n1 + n.n2 - r0 < FR_ASM_ROWS ? n.n1 + n.n2 - r0 : FR_ASM_ROWS;
  for (int e = threadIdx.x; e < rows * n.n1; e += 256) {
    const int i = r0 + e / n.n1, j = e % n.n1;
    const CT<R> t = pull<R>(f, n, C, front_src(f, n, i), f.own_src[n.row0 + j]);
    CT<R>& w = work[n.panel + (int64_t)i * n.ld + j];
    w.re += t.re;
    w.im += t.im;
  }
}

// ------------------------------------------------------------------ pivot blocks
// S = A11^{-1} by Gauss-Jordan elimination in place with row pivoting (max |Re| + |Im|, the lowest row
// on ties).  NW warps; warp w holds the rows w, w + NW, ..., lane l the columns l, l + 32, ...: NB x NB
// entries in registers.  Step c: the column's holders publish it, every warp finds the pivot row p,
// its warp publishes that row, and every entry is updated -- two barriers a step.  No row moves: after
// the last step entry (p(c), c') holds A^{-1}(c, p(c')), p(c) the pivot row of step c.
template <typename R, int NB> struct InvShared {
  alignas(16) CT<R> col[2][NB], row[2][NB];
  int prow[NB], rank[NB];   // pivot row of each step, and its inverse
  float amax;               // largest entry of the block
};

// *dst = v (shared memory) where `on`: one predicated store.  (A branch around plain stores of the row
// picked at run time makes the compiler index the register block, which puts it into local memory.)
__device__ __forceinline__ void store_if(bool on, CT<float>* dst, CT<float> v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p st.shared.v2.f32 [%1], {%2, %3};\n}"
               ::"r"((int)on), "r"(smem_u32(dst)), "f"(v.re), "f"(v.im) : "memory");
}
__device__ __forceinline__ void store_if(bool on, CT<double>* dst, CT<double> v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @p st.shared.v2.f64 [%1], {%2, %3};\n}"
               ::"r"((int)on), "r"(smem_u32(dst)), "d"(v.re), "d"(v.im) : "memory");
}

// The steps of the 32 columns held in register column b (a compile-time index: x stays in registers).
template <typename R, int NB, int NW, int b>
__device__ __forceinline__ void invert_columns(CT<R> (&x)[NB / NW][NB / 32], uint32_t (&used)[NB / 32],
                                               InvShared<R, NB>& sh, int n1, int n2, int sub, int32_t* status) {
  constexpr int RA = NB / NW, CB = NB / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 1
  for (int cl = 0; cl < 32; ++cl) {
    const int c = 32 * b + cl;
    if (c >= n1) return;
    const int buf = c & 1;
    if (lane == cl) {
#pragma unroll
      for (int a = 0; a < RA; ++a) sh.col[buf][warp + NW * a] = x[a][b];
    }
    __syncthreads();
    uint32_t key = 0u;
#pragma unroll
    for (int q = 0; q < CB; ++q) {
      const int i = lane + 32 * q;
      const CT<R> v = sh.col[buf][i];
      float mag = (float)(fabs(v.re) + fabs(v.im));
      if (mag != mag) mag = 0.0f;  // a non-finite entry still lets a row be chosen
      if (i < n1 && !((used[q] >> lane) & 1u))
        key = max(key, ((__float_as_uint(mag) << 1) & 0xFFFFFF00u) | 0x80u | (uint32_t)(127 - i));
    }
    key = __reduce_max_sync(0xffffffffu, key);
    const int p = 127 - (int)(key & 0x7Fu);
#pragma unroll
    for (int q = 0; q < CB; ++q)
      if ((p >> 5) == q) used[q] |= 1u << (p & 31);
    if (warp == p % NW) {
#pragma unroll
      for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int q = 0; q < CB; ++q) store_if(a == p / NW, &sh.row[buf][lane + 32 * q], x[a][q]);
    }
    if (threadIdx.x == 0) {
      sh.prow[c] = p;
      sh.rank[p] = c;
    }
    __syncthreads();
    const CT<R> pv = sh.row[buf][c];
    CT<R> inv = {R(0), R(0)};
    if (pv.re != R(0) || pv.im != R(0)) {
      const R den = pv.re * pv.re + pv.im * pv.im;
      inv = {pv.re / den, -pv.im / den};
    } else if (n2 > 0 && sh.amax > 0.0f) {
      // an exactly zero pivot column: the unknowns eliminated later can still make A_s regular, so the
      // pivot is taken as the rounding of the block's entries
      inv.re = R(1) / (R(sh.amax) * (sizeof(R) == 4 ? R(1.0 / (1 << 20)) : R(1.0 / (1ll << 45))));
    } else if (threadIdx.x == 0) {
      if (atomicCAS(&status[ST_ERR], DEV_OK, DEV_SINGULAR) == DEV_OK) status[ST_SUB] = sub;
    }
    CT<R> rj[CB];
#pragma unroll
    for (int q = 0; q < CB; ++q) {
      const CT<R> v = sh.row[buf][lane + 32 * q];
      rj[q] = {v.re * inv.re - v.im * inv.im, v.re * inv.im + v.im * inv.re};
    }
    if (lane == cl) rj[b] = inv;
#pragma unroll
    for (int a = 0; a < RA; ++a) {
      const int i = warp + NW * a;
      if (i == p) {
#pragma unroll
        for (int q = 0; q < CB; ++q) x[a][q] = rj[q];
      } else {
        const CT<R> l = sh.col[buf][i];
        if (lane == cl) x[a][b] = {R(0), R(0)};
#pragma unroll
        for (int q = 0; q < CB; ++q) {
          CT<R> t = x[a][q];
          t.re = fma(-l.re, rj[q].re, t.re);
          t.im = fma(-l.re, rj[q].im, t.im);
          t.re = fma(l.im, rj[q].im, t.re);
          t.im = fma(-l.im, rj[q].re, t.im);
          x[a][q] = t;
        }
      }
    }
  }
}

template <typename R, int NB, int NW>
__global__ void __launch_bounds__(NW * 32) k_fr_invert(FrDev f, int first, const CT<R>* __restrict__ work,
                                                       CT<R>* __restrict__ fac, int32_t* status) {
  constexpr int RA = NB / NW, CB = NB / 32;
  static_assert(NB <= 128 && NB % NW == 0 && NB % 32 == 0, "pivot keys hold 7 row bits");
  __shared__ InvShared<R, NB> sh;
  const FrontNode n = f.nodes[first + blockIdx.x];
  const int n1 = n.n1, ld = n.ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const CT<R>* src = work + n.panel;
  CT<R> x[RA][CB];
#pragma unroll
  for (int a = 0; a < RA; ++a)
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      const int i = warp + NW * a, j = lane + 32 * b;
      x[a][b] = (i < n1 && j < n1) ? src[(int64_t)i * ld + j] : CT<R>{R(i == j ? 1 : 0), R(0)};
    }
  {
    uint32_t big = 0u;  // magnitudes as ordered bits (NaN above infinity)
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
      for (int b = 0; b < CB; ++b)
        if (warp + NW * a < n1 && lane + 32 * b < n1)
          big = max(big, __float_as_uint((float)(fabs(x[a][b].re) + fabs(x[a][b].im))));
    big = __reduce_max_sync(0xffffffffu, big);
    if (threadIdx.x == 0) sh.amax = 0.0f;
    __syncthreads();
    if (lane == 0) atomicMax((unsigned int*)&sh.amax, big);  // visible after the first step's barrier
  }
  uint32_t used[CB];  // bit l of word q: row l + 32 q has been a pivot (CB words of 32 rows)
#pragma unroll
  for (int q = 0; q < CB; ++q) used[q] = 0u;
  invert_columns<R, NB, NW, 0>(x, used, sh, n1, n.n2, n.sub, status);
  if constexpr (CB > 1) invert_columns<R, NB, NW, 1>(x, used, sh, n1, n.n2, n.sub, status);
  if constexpr (CB > 2) invert_columns<R, NB, NW, 2>(x, used, sh, n1, n.n2, n.sub, status);
  if constexpr (CB > 3) invert_columns<R, NB, NW, 3>(x, used, sh, n1, n.n2, n.sub, status);
  static_assert(CB <= 4, "register columns");
  __syncthreads();
  CT<R>* dst = fac + n.panel;
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    const int i = warp + NW * a;
    if (i >= n1) continue;
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      const int j = lane + 32 * b;
      if (j < n1) dst[(int64_t)sh.rank[i] * ld + sh.prow[j]] = x[a][b];
    }
    if (lane < ld - n1) dst[(int64_t)i * ld + n1 + lane] = {R(0), R(0)};
  }
}

// ------------------------------------------------------------------ panel and contribution products
// out = A B^T over the panel's own unknowns (both operands row-major, contiguous along the sum), one
// 64 x 64 tile a block, 4 x 4 entries a thread.
//   SCHUR = false: L = A21 S       (B = S, symmetric)
//   SCHUR = true:  C = pulled children - L A21^T, tiles on and below the diagonal
template <typename R> struct FrK { static constexpr int KC = 16; };
template <> struct FrK<double> { static constexpr int KC = 8; };

template <typename R, bool SCHUR>
__global__ void __launch_bounds__(256) k_fr_mul(FrDev f, const FrontItem* __restrict__ items, CT<R>* __restrict__ work,
                                                CT<R>* __restrict__ fac, CT<R>* __restrict__ C) {
  constexpr int KC = FrK<R>::KC, LDS = FR_TILE + 2;
  __shared__ __align__(16) CT<R> As[KC][LDS], Bs[KC][LDS];
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = f.nodes[it.node];
  const int n1 = n.n1, n2 = n.n2, ld = n.ld;
  int ti, tj;
  if (SCHUR) {
    ti = (int)((sqrtf(8.0f * it.t + 1.0f) - 1.0f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= it.t) ++ti;
    while (ti * (ti + 1) / 2 > it.t) --ti;
    tj = it.t - ti * (ti + 1) / 2;
  } else {
    const int nj = (n1 + FR_TILE - 1) / FR_TILE;  // > 0: nodes that eliminate nothing have no such tiles
    ti = it.t / nj;
    tj = it.t % nj;
  }
  const int i0 = ti * FR_TILE, j0 = tj * FR_TILE;
  const int jn = SCHUR ? n2 : n1;
  const CT<R>* A = (SCHUR ? fac : work) + n.panel + (int64_t)n1 * ld;
  const CT<R>* B = SCHUR ? work + n.panel + (int64_t)n1 * ld : fac + n.panel;
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  CT<R> acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = {R(0), R(0)};
  for (int k0 = 0; k0 < ld; k0 += KC) {
    __syncthreads();
    for (int e = t; e < FR_TILE * KC; e += 256) {
      const int i = e / KC, k = e % KC;
      const bool in = k0 + k < ld;
      As[k][i] = (in && i0 + i < n2) ? A[(int64_t)(i0 + i) * ld + k0 + k] : CT<R>{R(0), R(0)};
      Bs[k][i] = (in && j0 + i < jn) ? B[(int64_t)(j0 + i) * ld + k0 + k] : CT<R>{R(0), R(0)};
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      CT<R> av[4], bv[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) av[p] = As[k][ty * 4 + p];
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = Bs[k][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc[p][q].re = fma(av[p].re, bv[q].re, acc[p][q].re);
          acc[p][q].im = fma(av[p].re, bv[q].im, acc[p][q].im);
          acc[p][q].re = fma(-av[p].im, bv[q].im, acc[p][q].re);
          acc[p][q].im = fma(av[p].im, bv[q].re, acc[p][q].im);
        }
    }
  }
  FrontSrc sj[4];
  if (SCHUR) {
#pragma unroll
    for (int q = 0; q < 4; ++q) sj[q] = j0 + tx + 16 * q < n2 ? f.border_src[n.bord + j0 + tx + 16 * q] : FrontSrc{-1, -1};
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = i0 + ty * 4 + p;
    if (i >= n2) continue;
    FrontSrc si = {-1, -1};
    if (SCHUR) si = f.border_src[n.bord + i];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = j0 + tx + 16 * q;
      if (SCHUR) {
        if (j >= n2) continue;
        const CT<R> v = pull<R>(f, n, C, si, sj[q]);
        C[n.cblk + (int64_t)i * n.ldc + j] = {v.re - acc[p][q].re, v.im - acc[p][q].im};
      } else if (j < ld) {  // columns n1 .. ld-1 are written as zeros
        fac[n.panel + (int64_t)(n1 + i) * ld + j] = acc[p][q];
      }
    }
  }
}

// ------------------------------------------------------------------ launchers
template <typename R>
static int launch_rows_t(const oras_handle* h, double k0) {
  const auto& m = h->mesh;
  const auto& d = h->dev;
  RowArgs A = row_args(h, k0);
  const int64_t total = m.sub_ns_off[m.nsub];
  const size_t smem = (size_t)ROW_WARPS * m.max_row_nnz * sizeof(cplx);
  if (smem > 48 * 1024) allow_max_smem((const void*)k_fr_rows<R>);
  if (cudaMemsetAsync(d.fr_work, 0, (size_t)h->fronts.panel_elems * sizeof(CT<R>), d.stream) != cudaSuccess) return -1;
  k_fr_rows<R><<<(unsigned)((total + ROW_WARPS - 1) / ROW_WARPS), ROW_WARPS * 32, smem, d.stream>>>(
      A, fr_dev(h), m.nsub, total, d.sub_ns_off, d.sub_dofs, d.fr_pos, d.fr_row_node, m.max_row_nnz, (CT<R>*)d.fr_work);
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_front_rows(const oras_handle* h, double k0) {
  return h->dev.factor_bits == 64 ? launch_rows_t<double>(h, k0) : launch_rows_t<float>(h, k0);
}

template <typename R>
static int factor_t(oras_handle* h) {
  const auto& d = h->dev;
  const Fronts& f = h->fronts;
  const FrDev fd = fr_dev(h);
  CT<R>* work = (CT<R>*)d.fr_work;
  CT<R>* fac = (CT<R>*)d.arena;
  CT<R>* C = (CT<R>*)d.fr_c;
  cudaStream_t st = d.stream;
  for (int l = 0; l < f.nlev(); ++l) {
    auto count = [&](const FrontLevels& v) { return (unsigned)(v.ptr[l + 1] - v.ptr[l]); };
    int pb = prof_begin(h);
    if (count(f.assemble)) {
      k_fr_assemble<R><<<count(f.assemble), 256, 0, st>>>(fd, d.fr_assemble + f.assemble.ptr[l], work, C);
      count_launches(1);
    }
    prof_end(h, KC_LU_SWAP, pb, 1);
    const int first = f.level_ptr[l], wide = f.level_wide[l], all = f.level_ptr[l + 1] - first;
    pb = prof_begin(h);
    if constexpr (sizeof(R) == 4) {
      if (wide) k_fr_invert<R, 128, 16><<<wide, 512, 0, st>>>(fd, first, work, fac, d.status);
      if (all > wide) k_fr_invert<R, 64, 8><<<all - wide, 256, 0, st>>>(fd, first + wide, work, fac, d.status);
    } else {
      if (wide) k_fr_invert<R, 64, 8><<<wide, 256, 0, st>>>(fd, first, work, fac, d.status);
      if (all > wide) k_fr_invert<R, 32, 4><<<all - wide, 128, 0, st>>>(fd, first + wide, work, fac, d.status);
    }
    count_launches((wide ? 1 : 0) + (all > wide ? 1 : 0));
    prof_end(h, KC_LU_TOURNAMENT, pb, 1);
    if (!count(f.schur)) continue;
    pb = prof_begin(h);
    if (count(f.lmul)) k_fr_mul<R, false><<<count(f.lmul), 256, 0, st>>>(fd, d.fr_lmul + f.lmul.ptr[l], work, fac, C);
    prof_end(h, KC_LU_TRSM, pb, 1);
    pb = prof_begin(h);
    k_fr_mul<R, true><<<count(f.schur), 256, 0, st>>>(fd, d.fr_schur + f.schur.ptr[l], work, fac, C);
    prof_end(h, KC_LU_UPDATE, pb, 1);
    count_launches(2);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_front_factor(oras_handle* h) { return h->dev.factor_bits == 64 ? factor_t<double>(h) : factor_t<float>(h); }

}  // namespace oras
