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
//   k_fr_invert    S by blocked Gauss-Jordan with row pivoting, the block held in registers;
//   k_fr_mul, k_fr_mul_tc (fronts_tc.cu)  L, then C with the children's C gathered into it (each C is read once).
// Pivots are chosen inside a pivot block (up to front_nb unknowns) and never outside it.  Where that is not enough (a
// zero pivot, or an entry of L above FR_GROWTH) the node is marked; the host then moves the unknowns in question to the
// node's parent, plans the trees anew and factors again (fronts_weak.cpp, oras_factor).  FP32, one subdomain of 6^3 x 6,
// degree 2, at the resonance of a leaf: without it the apply's error is 1e4 and nothing converges; with it 3e-6, one more
// factorisation.
//
// Against dense factors of the same matrices (n_s^2 entries each) the largest subdomain of the
// 16^3 x 6, degree-2, 64-subdomain problem (17,896 unknowns) keeps 2% of the entries and needs 0.1%
// of the products.  FP32 factors keep FP32's accuracy throughout (fronts_tc.cu).  Error of the apply against FP64, beside
// that of a dense FP32 LU with pivots over whole columns, on 8 subdomains of the head-like medium: degree 1 (6^3 x 6)
// 0.62e-6 and 0.45e-6, degree 2 (5^3, 8^3) 1.1e-6 and 1.0e-6, 2.3e-6 and 1.8e-6, degree 3 (5^3) 3.4e-6 and 3.8e-6; without
// losses, degree 2 (6^3) 1.3e-5 and 0.59e-5, degree 3 (5^3) 5.4e-5 and 1.9e-5.
#include "fronts.cuh"
#include "rows.cuh"

namespace oras {

void launch_front_mul_tc(const oras_handle* h, const FrDev& f, bool schur, const FrontItem* items, int64_t blocks);

static FrDev fr_dev(const oras_handle* h) {
  const auto& d = h->dev;
  return {d.fr_nodes, d.fr_border, d.fr_own_src, d.fr_border_src, d.fr_weak};
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

// ------------------------------------------------------------------ children's contributions (pull)
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
// S = A11^{-1} by Gauss-Jordan elimination in place with row pivoting (max |Re| + |Im|, the lowest row on
// ties), 8 columns at a time.  NW main warps hold the block in registers (warp w the rows w, w + NW, ...,
// lane l the columns l, l + 32, ...); NB / 32 panel warps, which hold none of it, eliminate the 8 columns of a
// panel, one row a lane: a column costs a warp-wide maximum, one barrier among them (each publishes its best
// candidate's row with its key) and 8 products a lane.  They leave W, the 8 columns of the inverse transformation
// (in place, as Gauss-Jordan does), and the 8 pivot rows p_c; every other entry then becomes
//   x(i, j) = [i not a pivot of the panel] x(i, j) + sum_c W(i, c) x(p_c, j).
// The main warps update the register column with the next panel first and hand that panel over, so its
// elimination runs beside the rest of the update.  No row moves: at the end entry (p(c), c') holds
// A^{-1}(c, p(c')), p(c) the pivot row of column c.
//
// Bound: FP32 arithmetic, 4 n1^3 fused multiply-adds a block, and on levels with few nodes the chain of n1 pivot
// searches.  One column at a time (two block barriers and a pivot search on the critical path each): 9.4 ms for all
// pivot blocks of the 16^3 x 6, degree-2, 64-subdomain problem; panels of 8 by one warp (4 rows a lane) 6.3 ms, by a
// warp for every 32 rows 4.7 ms.  4^3 x 6, 4 subdomains: 0.62, 0.45 and 0.36 ms.  In FP64 (8^3 x 6, degree 1) 1.97,
// 2.39 and 1.74 ms: the panel is then FP64 arithmetic, which one warp has a quarter of.
// One kernel for every 32 columns of width: a block of 97 in a 128-wide kernel costs 1.8 times its products.
// BLOCKS: 3 blocks of the 64-wide kernel an SM (48 bytes spilled) or 2 of the 96-wide one (288) measured the same.
template <typename R, int NB> struct InvShared {
  alignas(16) CT<R> pan[NB][10];     // the panel's 8 columns (rows padded against bank conflicts)
  alignas(16) CT<R> W[2][NB][10];
  alignas(16) CT<R> row[2][8][NB];   // the pivot rows before the panel
  alignas(16) CT<R> cand[2][NB / 32][8];   // each panel warp's best row of a column (by column parity)
  alignas(16) uint32_t ckey[2][4];         // and its key
  int piv[2][8];
  uint32_t pmask[2][NB / 32];        // the panel's pivot rows
  unsigned char prank[NB], pcol[NB]; // pivot row -> column, column -> pivot row
  float amax;                        // largest entry of the block
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
__device__ __forceinline__ void named_arrive(int id, int nthreads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// Named barriers: a panel's columns are in pan; its W, pivots are ready; its pivot rows are in row;
// and, among the panel warps, the candidates of a column.
enum { INV_BAR_PANEL = 1, INV_BAR_W = 2, INV_BAR_ROWS = 3, INV_BAR_CAND = 4 };

// Two adjacent complex entries of shared memory (16-byte aligned).
__device__ __forceinline__ void lds_pair(const CT<float>* p, CT<float>& a, CT<float>& b) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  a = {t.x, t.y}; b = {t.z, t.w};
}
__device__ __forceinline__ void lds_pair(const CT<double>* p, CT<double>& a, CT<double>& b) {
  const double2 t0 = reinterpret_cast<const double2*>(p)[0], t1 = reinterpret_cast<const double2*>(p)[1];
  a = {t0.x, t0.y}; b = {t1.x, t1.y};
}

// The leading bits of x >= 0, ordered as x is: all of FP64's exponents, which a conversion to FP32 would cut.  0 for NaN.
__device__ __forceinline__ uint32_t magnitude_bits(float x) {
  const uint32_t b = __float_as_uint(x);
  return b > 0x7F800000u ? 0u : b;
}
__device__ __forceinline__ uint32_t magnitude_bits(double x) {
  const uint32_t b = (uint32_t)__double2hiint(x);
  return b > 0x7FF00000u ? 0u : b;
}

// 1 / v of a pivot that is not zero.  v is first brought to about 1 by a power of two, so that the square of its
// magnitude neither overflows nor vanishes (entries of A_s scale with the mesh's unit and 1 / mu_r): the power comes from
// the pivot's key, whose top bits are the exponent of |re| + |im|, and is there before the pivot is.
template <typename R> __device__ __forceinline__ R pivot_scale(uint32_t key);
template <> __device__ __forceinline__ float pivot_scale<float>(uint32_t key) {
  const uint32_t e = key >> 24;
  return __uint_as_float((e < 253u ? 254u - e : 1u) << 23);
}
template <> __device__ __forceinline__ double pivot_scale<double>(uint32_t key) {
  const uint32_t e = key >> 21;
  return __hiloint2double((int)((e < 2045u ? 2046u - e : 1u) << 20), 0);
}
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
template <typename R> __device__ __forceinline__ CT<R> reciprocal(CT<R> v, R s) {
  const R re = v.re * s, im = v.im * s, r = recip(re * re + im * im);
  return {re * s * r, -(im * s) * r};
}

// Panel warp pw: columns c0 .. c0 + 7 of row 32 pw + lane (rows below `rows` take part).  taken: the row has been a
// pivot.
template <typename R, int NB>
__device__ __forceinline__ void invert_panel(InvShared<R, NB>& sh, int c0, int rows, int buf, bool& taken, int n2,
                                             int sub, const FrDev& f, int node, int32_t* status) {
  constexpr int PW = NB / 32;
  const int lane = threadIdx.x & 31, pw = (threadIdx.x >> 5) % PW, i = 32 * pw + lane;
  CT<R> x[8];
#pragma unroll
  for (int j = 0; j < 8; j += 2) lds_pair(&sh.pan[i][j], x[j], x[j + 1]);
  bool mine = false;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int par = c & 1;
    const R mag = fabs(x[c].re) + fabs(x[c].im);
    uint32_t key = 0u;  // a non-finite entry still lets a row be chosen
    if (i < rows && !taken) key = ((magnitude_bits(mag) << 1) & 0xFFFFFF00u) | 0x80u | (uint32_t)(127 - i);
    uint32_t best = __reduce_max_sync(0xffffffffu, key);
    if (best != 0u && key == best) {
#pragma unroll
      for (int j = 0; j < 8; ++j) sh.cand[par][pw][j] = x[j];
      sh.ckey[par][pw] = best;
    } else if (best == 0u && lane == 0) {
      sh.ckey[par][pw] = 0u;
    }
    if constexpr (PW > 1) {
      named_sync(INV_BAR_CAND, PW * 32);
#pragma unroll
      for (int q = 0; q < PW; ++q) best = max(best, sh.ckey[par][q]);
    } else {
      __syncwarp();
    }
    const int p = 127 - (int)(best & 0x7Fu);
    const bool own = i == p;
    const R scale = pivot_scale<R>(best);
    CT<R> r[8];
#pragma unroll
    for (int j = 0; j < 8; j += 2) lds_pair(&sh.cand[par][PW > 1 ? p >> 5 : 0][j], r[j], r[j + 1]);
    if (own) {
      taken = mine = true;
      sh.piv[buf][c] = p;
      sh.prank[p] = (unsigned char)(c0 + c);
      sh.pcol[c0 + c] = (unsigned char)p;
    }
    const CT<R> pv = r[c];
    CT<R> inv = {R(0), R(0)};
    if (pv.re != R(0) || pv.im != R(0)) {
      inv = reciprocal(pv, scale);
    } else if (n2 > 0) {
      // an exactly zero pivot column: the unknowns eliminated later can still make A_s regular.  The node is planned
      // anew; where that does not help, the pivot is taken as the rounding of the block's entries
      if (sh.amax > 0.0f) inv.re = R(1) / (R(sh.amax) * (sizeof(R) == 4 ? R(1.0 / (1 << 20)) : R(1.0 / (1ll << 45))));
      if (own) mark_weak(f, node, status);
    } else if (own) {
      if (atomicCAS(&status[ST_ERR], DEV_OK, DEV_SINGULAR) == DEV_OK) status[ST_SUB] = sub;
    }
    // x_j <- x_j - (x_c / pv) r_j; the pivot row itself becomes r_j / pv
    const CT<R> l = x[c];
    CT<R> m = inv;
    if (!own) {
      m.re = fma(l.im, inv.im, -l.re * inv.re);
      m.im = -fma(l.im, inv.re, l.re * inv.im);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      CT<R> t = own ? CT<R>{R(0), R(0)} : x[j];
      t.re = fma(m.re, r[j].re, t.re);
      t.im = fma(m.re, r[j].im, t.im);
      t.re = fma(-m.im, r[j].im, t.re);
      t.im = fma(m.im, r[j].re, t.im);
      x[j] = j == c ? m : t;
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) sh.W[buf][i][j] = x[j];
  const uint32_t m = __ballot_sync(0xffffffffu, mine);
  if (lane == 0) sh.pmask[buf][pw] = m;
}

// Register column b (columns 32 cb .. 32 cb + 31 of the block) of the main warps after a panel: the panel's own 8
// lanes (from lane 8 pl when `here`) take W, the others the rank-8 update.
template <typename R, int NB, int NW, int b>
__device__ __forceinline__ void invert_update(CT<R> (&x)[NB / NW][NB / 32], const InvShared<R, NB>& sh, int buf,
                                              int cb, bool here, int pl) {
  constexpr int RA = NB / NW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pc = lane - 8 * pl;
  const bool in_panel = here && pc >= 0 && pc < 8;
  CT<R> r[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) r[c] = sh.row[buf][c][lane + 32 * cb];
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    const int i = warp + NW * a;
    CT<R> t = ((sh.pmask[buf][i >> 5] >> (i & 31)) & 1u) ? CT<R>{R(0), R(0)} : x[a][b];
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
      CT<R> w0, w1;
      lds_pair(&sh.W[buf][i][c], w0, w1);
      t.re = fma(w0.re, r[c].re, t.re);
      t.im = fma(w0.re, r[c].im, t.im);
      t.re = fma(-w0.im, r[c].im, t.re);
      t.im = fma(w0.im, r[c].re, t.im);
      t.re = fma(w1.re, r[c + 1].re, t.re);
      t.im = fma(w1.re, r[c + 1].im, t.im);
      t.re = fma(-w1.im, r[c + 1].im, t.re);
      t.im = fma(w1.im, r[c + 1].re, t.im);
    }
    x[a][b] = in_panel ? sh.W[buf][i][pc & 7] : t;
    asm volatile("" ::: "memory");  // one row's W at a time: loaded ahead for all rows it spills
  }
}

// Columns 8 pl .. 8 pl + 7 of register column b into pan.
template <typename R, int NB, int NW, int b>
__device__ __forceinline__ void publish_panel(const CT<R> (&x)[NB / NW][NB / 32], InvShared<R, NB>& sh, int pl) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane - 8 * pl;
  if (c < 0 || c >= 8) return;
#pragma unroll
  for (int a = 0; a < NB / NW; ++a) sh.pan[warp + NW * a][c] = x[a][b];
}

// x's register columns shifted left by one, cyclically.
template <typename R, int RA, int CB>
__device__ __forceinline__ void rotate_columns(CT<R> (&x)[RA][CB]) {
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    const CT<R> t = x[a][0];
#pragma unroll
    for (int q = 0; q + 1 < CB; ++q) x[a][q] = x[a][q + 1];
    x[a][CB - 1] = t;
  }
}

// The main warps' steps, np panels.  Register column 0 is always the one worked on (register indices stay
// compile-time) and the columns rotate: slot s holds block column (s + returned rotation) % CB.  One instance of
// the update in a rolled loop: inlined for every column the compiler loads their operands ahead and spills.
template <typename R, int NB, int NW>
__device__ __forceinline__ int invert_main(CT<R> (&x)[NB / NW][NB / 32], InvShared<R, NB>& sh, int np) {
  constexpr int RA = NB / NW, CB = NB / 32, MAIN = NW * 32, ALL = MAIN + NB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int rot = 0;
  auto next = [&]() {
    rotate_columns<R, RA, CB>(x);
    rot = rot + 1 < CB ? rot + 1 : 0;
  };
#pragma unroll 1
  for (int p = 0; p < np; ++p) {
    const int pl = p & 3, buf = p & 1;
    named_sync(INV_BAR_W, ALL);
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {
      const int i = sh.piv[buf][c];
      if (i % NW == warp) {
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
          for (int q = 0; q < CB; ++q)
            store_if(a == i / NW, &sh.row[buf][c][lane + 32 * (q + rot < CB ? q + rot : q + rot - CB)], x[a][q]);
      }
    }
    named_sync(INV_BAR_ROWS, MAIN);
    // the column with the next panel first: this panel's own, or after its last panel the one that follows
    if (CB > 1 && pl == 3) next();
    const int own = CB > 1 && pl == 3 ? CB - 1 : 0;
#pragma unroll 1
    for (int s = 0; s < CB; ++s) {
      invert_update<R, NB, NW, 0>(x, sh, buf, rot, s == own, pl);
      if (s == 0 && p + 1 < np) {
        publish_panel<R, NB, NW, 0>(x, sh, (pl + 1) & 3);
        named_arrive(INV_BAR_PANEL, ALL);
      }
      if (CB > 1) next();
    }
  }
  return rot;
}

template <typename R, int NB, int NW, int BLOCKS>
__global__ void __launch_bounds__(NW * 32 + NB, BLOCKS)
    k_fr_invert(FrDev f, int first, const CT<R>* __restrict__ work, CT<R>* __restrict__ fac, int32_t* status) {
  constexpr int RA = NB / NW, CB = NB / 32, ALL = NW * 32 + NB;
  static_assert(NB <= 128 && NB % NW == 0 && NB % 32 == 0 && NW % (NB / 32) == 0, "pivot keys hold 7 row bits");
  __shared__ InvShared<R, NB> sh;
  const FrontNode n = f.nodes[first + blockIdx.x];
  const int n1 = n.n1, ld = n.ld, np = (n1 + 7) / 8;  // the last panel's columns past n1 are identity columns
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) sh.amax = 0.0f;
  __syncthreads();
  if (warp >= NW) {
    bool taken = false;
    __syncthreads();  // amax and the first panel
    for (int p = 0; p < np; ++p) {
      if (p > 0) named_sync(INV_BAR_PANEL, ALL);
      invert_panel<R, NB>(sh, 8 * p, 8 * np, p & 1, taken, n.n2, n.sub, f, first + blockIdx.x, status);
      named_arrive(INV_BAR_W, ALL);
    }
    __syncthreads();
    return;
  }
  const CT<R>* src = work + n.panel;
  CT<R> x[RA][CB];
  uint32_t big = 0u;  // magnitudes as ordered bits (NaN above infinity)
#pragma unroll
  for (int a = 0; a < RA; ++a)
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      const int i = warp + NW * a, j = lane + 32 * b;
      const bool in = i < n1 && j < n1;
      x[a][b] = {R(i == j ? 1 : 0), R(0)};
      if (in) {  // its halves by themselves, as where the block is stored: as one word the 128-wide kernel spills 376 bytes, not 136
        const R* e = &src[(int64_t)i * ld + j].re;
        x[a][b] = {e[0], e[1]};
      }
      if (in) big = max(big, __float_as_uint((float)(fabs(x[a][b].re) + fabs(x[a][b].im))));
    }
  big = __reduce_max_sync(0xffffffffu, big);
  if (lane == 0) atomicMax((unsigned int*)&sh.amax, big);
  publish_panel<R, NB, NW, 0>(x, sh, 0);
  __syncthreads();
  const int rot = invert_main<R, NB, NW>(x, sh, np);
  __syncthreads();
  CT<R>* dst = fac + n.panel;
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    const int i = warp + NW * a;
    if (i >= n1) continue;
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      const int j = lane + 32 * (b + rot < CB ? b + rot : b + rot - CB);
      if (j < n1) {
        R* out = &dst[(int64_t)sh.prank[i] * ld + sh.pcol[j]].re;
        out[0] = x[a][b].re;
        out[1] = x[a][b].im;
      }
    }
    if (lane < ld - n1) dst[(int64_t)i * ld + n1 + lane] = {R(0), R(0)};
  }
}

// ------------------------------------------------------------------ panel and contribution products (FP64; FP32: fronts_tc.cu)
// out = A B^T over the panel's own unknowns (both operands row-major, contiguous along the sum), one
// 64 x 64 tile a block, 4 x 4 entries a thread.
//   SCHUR = false: L = A21 S       (B = S, symmetric)
//   SCHUR = true:  C = pulled children - L A21^T, tiles on and below the diagonal
// A product with an explicit inverse leaves L A11 - A21 of the size of the rounding times k, the product of the
// largest entries of A21 and S, and the apply an error of about k^2, where a triangular solve leaves k.  k is the square
// of the wavelength over the mesh width at low frequencies.  Tiles with k above FR_REFINE (k is below 20 on the benchmark's
// medium at degrees 1 and 2) take one step of refinement, L += (A21 - L A11) S: 4^3 x 6, degree 2, apply error at
// k0 = 0.1 7.2e-12 -> 1.8e-12, at 0.01 5.8e-8 -> 4.5e-11 (dense LU 4.6e-13, 5.0e-11).  (FP32 does without: dense
// factors with TF32 products were worse off.)
constexpr double FR_REFINE = 128.0;

constexpr int FR_MUL_KC = 8, FR_MUL_LDS = FR_TILE + 2;
template <typename R> struct MulShared {
  alignas(16) CT<R> As[FR_MUL_KC][FR_MUL_LDS], Bs[FR_MUL_KC][FR_MUL_LDS];
};

// acc += A B^T of one tile: an x ld and bn x ld entries.  big: the largest entries of A and B that the thread has loaded.
template <typename R>
__device__ __forceinline__ void mul_tile(MulShared<R>& sh, CT<R> (&acc)[4][4], const CT<R>* A, int an, const CT<R>* B,
                                         int bn, int ld, uint32_t (&big)[2]) {
  constexpr int KC = FR_MUL_KC;
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  big[0] = big[1] = 0u;
  for (int k0 = 0; k0 < ld; k0 += KC) {
    __syncthreads();
    for (int e = t; e < FR_TILE * KC; e += 256) {
      const int i = e / KC, k = e % KC;
      const bool in = k0 + k < ld;
      const CT<R> a = (in && i < an) ? A[(int64_t)i * ld + k0 + k] : CT<R>{R(0), R(0)};
      const CT<R> b = (in && i < bn) ? B[(int64_t)i * ld + k0 + k] : CT<R>{R(0), R(0)};
      sh.As[k][i] = a;
      sh.Bs[k][i] = b;
      big[0] = max(big[0], max(magnitude_bits(fabs(a.re)), magnitude_bits(fabs(a.im))));
      big[1] = max(big[1], max(magnitude_bits(fabs(b.re)), magnitude_bits(fabs(b.im))));
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      CT<R> av[4], bv[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) av[p] = sh.As[k][ty * 4 + p];
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = sh.Bs[k][tx + 16 * q];
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
}

template <typename R, bool SCHUR>
__global__ void __launch_bounds__(256, 2) k_fr_mul(FrDev f, const FrontItem* __restrict__ items, CT<R>* __restrict__ work,
                                                CT<R>* __restrict__ fac, CT<R>* __restrict__ C, int32_t* status) {
  __shared__ MulShared<R> sh;
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
  uint32_t big[2];
  mul_tile<R>(sh, acc, A + (int64_t)i0 * ld, n2 - i0, B + (int64_t)j0 * ld, jn - j0, ld, big);
  if constexpr (!SCHUR) {
    static_assert(sizeof(R) == 8, "one tile has all own columns");
    __shared__ uint32_t part[2][8];
    for (int q = 0; q < 2; ++q) {
      const uint32_t m = __reduce_max_sync(0xffffffffu, big[q]);
      if ((t & 31) == 0) part[q][t >> 5] = m;
    }
    __syncthreads();
    uint32_t a = 0u, s = 0u;
    for (int q = 0; q < 8; ++q) { a = max(a, part[0][q]); s = max(s, part[1][q]); }
    if (__hiloint2double((int)a, 0) * __hiloint2double((int)s, 0) > FR_REFINE) {  // the same in every thread
      const CT<R>* A11 = work + n.panel;
      CT<R>* out = fac + n.panel + (int64_t)(n1 + i0) * ld;
      auto put = [&](const CT<R> (&v)[4][4]) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (i0 + ty * 4 + p < n2 && tx + 16 * q < ld) out[(int64_t)(ty * 4 + p) * ld + tx + 16 * q] = v[p][q];
        __syncthreads();
      };
      put(acc);
      CT<R> r[4][4] = {};
      mul_tile<R>(sh, r, out, n2 - i0, A11, n1, ld, big);
      __syncthreads();  // L has been read
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + ty * 4 + p, j = tx + 16 * q;
          const CT<R> a = i < n2 && j < ld ? A[(int64_t)i * ld + j] : CT<R>{R(0), R(0)};
          r[p][q] = {a.re - r[p][q].re, a.im - r[p][q].im};
        }
      put(r);
      mul_tile<R>(sh, acc, out, n2 - i0, B, n1, ld, big);
      __syncthreads();
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
        if (grown((float)acc[p][q].re, (float)acc[p][q].im)) mark_weak(f, it.node, status);
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
    pb = prof_begin(h);
    // pivot blocks by width; a level that fits on the chip at once goes in one launch
    const int32_t* cp = &f.level_class[(size_t)l * (FR_CLASSES + 1)];
    const bool one = cp[FR_CLASSES] - cp[0] <= d.num_sms;
    for (int c = 0; c < FR_CLASSES; ++c) {
      const int first = cp[c], nodes = (one ? cp[FR_CLASSES] : cp[c + 1]) - first;
      if (nodes == 0 || (c < FR_CLASSES - 1 && cp[c + 1] == cp[c])) continue;
      if constexpr (sizeof(R) == 4) {
        if (c == 0) k_fr_invert<R, 128, 16, 1><<<nodes, 640, 0, st>>>(fd, first, work, fac, d.status);
        else if (c == 1) k_fr_invert<R, 96, 12, 1><<<nodes, 480, 0, st>>>(fd, first, work, fac, d.status);
        else if (c == 2) k_fr_invert<R, 64, 8, 2><<<nodes, 320, 0, st>>>(fd, first, work, fac, d.status);
        else k_fr_invert<R, 32, 4, 4><<<nodes, 160, 0, st>>>(fd, first, work, fac, d.status);
      } else {
        if (c == 2) k_fr_invert<R, 64, 8, 1><<<nodes, 320, 0, st>>>(fd, first, work, fac, d.status);
        else k_fr_invert<R, 32, 4, 4><<<nodes, 160, 0, st>>>(fd, first, work, fac, d.status);
      }
      count_launches(1);
      if (one) break;
    }
    prof_end(h, KC_LU_TOURNAMENT, pb, 1);
    if (!count(f.schur)) continue;
    pb = prof_begin(h);
    if (count(f.lmul)) {
      if constexpr (sizeof(R) == 4) {
        launch_front_mul_tc(h, fd, false, d.fr_lmul + f.lmul.ptr[l], count(f.lmul));
      } else {
        k_fr_mul<R, false><<<count(f.lmul), 256, 0, st>>>(fd, d.fr_lmul + f.lmul.ptr[l], work, fac, C, d.status);
        count_launches(1);
      }
    }
    prof_end(h, KC_LU_TRSM, pb, 1);
    pb = prof_begin(h);
    if constexpr (sizeof(R) == 4) {
      launch_front_mul_tc(h, fd, true, d.fr_schur + f.schur.ptr[l], count(f.schur));
    } else {
      k_fr_mul<R, true><<<count(f.schur), 256, 0, st>>>(fd, d.fr_schur + f.schur.ptr[l], work, fac, C, d.status);
      count_launches(1);
    }
    prof_end(h, KC_LU_UPDATE, pb, 1);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_front_factor(oras_handle* h) { return h->dev.factor_bits == 64 ? factor_t<double>(h) : factor_t<float>(h); }

}  // namespace oras
