// ORAS preconditioner apply with the sparse local factors (fronts.cu):
//   z = sum_s R_s^T D_s A_s^{-1} R_s v,   A_s = L D L^T by nodes with panels [S; L].
// Forward, from the leaves: a node's right-hand side is b on its own unknowns plus what its children
// hand up, y = b + sum of theirs; it hands up u = (the children's on its border) - L y.  Backward, from
// the roots: x = S y - L^T x(border), the panel [S; L] times [y; -x(border)] column by column (S is
// symmetric).  Every panel is read once a direction.  All nodes of a tree level run in one launch; a
// row of a result is formed by one block and children are added in a fixed order, so results do not depend
// on scheduling (OAS adds overlapping contributions into z with atomics).
//
// Up to 4 right-hand sides a pass (k_fr_fwd, k_fr_bwd): bound by HBM, (S + 2 L) entries of 8 B (FP32):
// 3.2 GB a pass on the 16^3 degree-2 64-subdomain problem.  What costs beside it is the latency of a level
// (index, gather, panel, reduction, 30-odd levels a pass), so a block issues its panel loads and indices,
// which do not depend on the level before, first and only then waits for that level (programmatic dependent
// launch: the next level's blocks load while the last ones of this level finish), panels are read past L2
// (they are used once a direction, the vectors and indices stay), and the backward blocks get narrower
// where a level has few nodes.  ms an apply, before -> with these: 16^3 1.29 -> 0.81 (3.2 GB: 58% of the copy
// rate), 24^3 with 512 subdomains 0.54 -> 0.38, 8^3 0.24 -> 0.086.
// 5 and more right-hand sides (k_fr_fwd_multi, k_fr_bwd_multi): up to 32 a pass as small matrix products, bound
// by the FP32 pipes at 32 and by the latency of a block at 8: 32 columns of the 16^3 128-subdomain problem 5.2 -> 2.2 ms
// (four passes of 8 before).  With panels copied in the background, all of L before the wait and a ring of four stages
// backward, instead of one stage ahead through registers: 8 columns of the 9^3 x 6, degree-3 problem 1.11 -> 0.82 ms
// an apply (1.5 GB), of the 10^3 one with ports 0.37 -> 0.27 ms, 32 columns as before.
#include <algorithm>

#include "apply.cuh"

namespace oras {

struct FrApply {
  const FrontNode* nodes;
  const int32_t* border;
  const FrontSrc* own_src;
  const FrontSrc* border_src;
  const int32_t* row_dof;
  const uint8_t* row_pou;
  int weights;
  int64_t vs, off;   // v and z: right-hand side r of unknown g at g * vs + off + r
  int nr;            // live right-hand sides of the pass (<= KR)
};

constexpr int FR_THREADS = 256;
constexpr int FR_MAX_NB = 128;

// Programmatic dependent launch: lets the next kernel of the stream start its independent loads / waits until
// the kernels before this one have finished and their results are visible.
// The vectors that a kernel reads after the wait are plain pointers: through a restrict-qualified pointer to
// const the compiler may load them before it.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Two adjacent complex entries, read once: past L1, first out of L2.
__device__ __forceinline__ void ld_stream(const CT<float>* p, CT<float>& a, CT<float>& b) {
  const float4 t = __ldcs(reinterpret_cast<const float4*>(p));
  a = {t.x, t.y}; b = {t.z, t.w};
}
__device__ __forceinline__ void ld_stream(const CT<double>* p, CT<double>& a, CT<double>& b) {
  const double2 t0 = __ldcs(reinterpret_cast<const double2*>(p)), t1 = __ldcs(reinterpret_cast<const double2*>(p) + 1);
  a = {t0.x, t0.y}; b = {t1.x, t1.y};
}

template <typename R> __device__ __forceinline__ void cfma(CT<R>& t, CT<R> m, CT<R> y) {
  t.re = fma(m.re, y.re, t.re); t.re = fma(-m.im, y.im, t.re);
  t.im = fma(m.re, y.im, t.im); t.im = fma(m.im, y.re, t.im);
}

// Handed up by the children for a front row with sources s.
template <typename R, int KR>
__device__ __forceinline__ CT<R> pull_vec(const CT<R>* u, FrontSrc s, int r) {
  CT<R> t = {R(0), R(0)};
  if (s.a >= 0) t = u[(int64_t)s.a * KR + r];
  if (s.b >= 0) {
    const CT<R> v = u[(int64_t)s.b * KR + r];
    t.re += v.re;
    t.im += v.im;
  }
  return t;
}

// One block: 64 border rows of a node, 8 lanes a row, 32 rows at a time.
template <typename R, int KR>
__global__ void __launch_bounds__(FR_THREADS) k_fr_fwd(FrApply a, const FrontItem* __restrict__ items,
                                                       const CT<R>* __restrict__ fac, const cplx* v,
                                                       CT<R>* y, CT<R>* u) {
  constexpr int NB = sizeof(R) == 4 ? FR_MAX_NB : FR_MAX_NB / 2, NQ = NB / 16;
  constexpr int ROUND = FR_THREADS / 8;
  __shared__ __align__(16) CT<R> own[KR][NB];
  pdl_release();
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, ld = n.ld, sub = threadIdx.x & 7;
  const CT<R>* rows = fac + n.panel + (int64_t)n1 * ld;
  CT<R> m0[NQ], m1[NQ];
  auto load = [&](int i) {  // the lane's entries of border row i
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int c = 2 * sub + 16 * q;
      if (i < n.n2 && c < ld) ld_stream(rows + (int64_t)i * ld + c, m0[q], m1[q]);
    }
  };
  int i = it.t * FR_FWD_ROWS + (threadIdx.x >> 3);
  load(i);
  FrontSrc src = {-1, -1};
  if (i < n.n2) src = a.border_src[n.bord + i];
  // own unknown of this thread in the gather (one right-hand side after the other)
  const int c0 = threadIdx.x / KR, r0 = threadIdx.x % KR;
  FrontSrc osrc = {-1, -1};
  int32_t dof = 0;
  if (c0 < n1) {
    osrc = a.own_src[n.row0 + c0];
    dof = a.row_dof[n.row0 + c0];
  }
  pdl_wait();
  for (int c = c0; c < ld; c += FR_THREADS / KR) {
    CT<R> t = {R(0), R(0)};
    if (c < n1) {
      if (c != c0) {
        osrc = a.own_src[n.row0 + c];
        dof = a.row_dof[n.row0 + c];
      }
      if (r0 < a.nr) {
        const cplx b = v[(int64_t)dof * a.vs + a.off + r0];
        t = {R(b.re), R(b.im)};
      }
      const CT<R> up = pull_vec<R, KR>(u, osrc, r0);
      t.re += up.re;
      t.im += up.im;
      if (it.t == 0) y[(int64_t)(n.row0 + c) * KR + r0] = t;
    }
    own[r0][c] = t;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < FR_FWD_ROWS / ROUND; ++h) {
    if (h > 0) {
      i += ROUND;
      load(i);
      if (i < n.n2) src = a.border_src[n.bord + i];
    }
    CT<R> acc[KR];
#pragma unroll
    for (int r = 0; r < KR; ++r) acc[r] = {R(0), R(0)};
    if (i < n.n2) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int c = 2 * sub + 16 * q;
        if (c < ld) {
#pragma unroll
          for (int r = 0; r < KR; ++r) {
            CT<R> y0, y1;
            ld_cpair(&own[r][c], y0, y1);
            cfma(acc[r], m0[q], y0);
            cfma(acc[r], m1[q], y1);
          }
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
        const CT<R> up = pull_vec<R, KR>(u, src, r);
        u[(n.bord + i) * KR + r] = {up.re - acc[r].re, up.im - acc[r].im};
      }
    }
  }
}

// One block: CW own unknowns of a node, a lane two of them; the CW / 2-lane groups share the panel's rows.
template <typename R, typename ZT, int KR, int CW>
__global__ void __launch_bounds__(FR_THREADS) k_fr_bwd(FrApply a, const FrontItem* __restrict__ items,
                                                       const CT<R>* __restrict__ fac, const CT<R>* y,
                                                       CT<R>* x, ZT* z) {
  constexpr int LW = CW / 2, NG = FR_THREADS / LW;      // lanes a row, row groups
  constexpr int NQ = sizeof(R) == 4 ? 8 : 4;            // rows a group loads at once
  constexpr int ROWS = 512;                             // rows of [y; -x] staged at once
  constexpr int NW = FR_THREADS / 32;
  __shared__ CT<R> w[ROWS][KR];
  __shared__ CT<R> red[NW][CW][KR];
  pdl_release();
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, m = n.n1 + n.n2, ld = n.ld;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, grp = threadIdx.x / LW;
  const int j = it.t * CW + 2 * (threadIdx.x % LW);
  const CT<R>* panel = fac + n.panel + j;
  CT<R> m0[NQ], m1[NQ];
  auto load = [&](int i0) {  // this lane's columns of rows i0 + grp + NG q
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int i = i0 + grp + NG * q;
      if (i < m && j < ld) ld_stream(panel + (int64_t)i * ld, m0[q], m1[q]);
    }
  };
  load(0);
  int32_t row[ROWS / FR_THREADS];  // rows of [y; x] that this thread stages first
#pragma unroll
  for (int q = 0; q < ROWS / FR_THREADS; ++q) {
    const int i = threadIdx.x + FR_THREADS * q;
    row[q] = i < n1 ? n.row0 + i : (i < m ? a.border[n.bord + i - n1] : -1);
  }
  CT<R> acc0[KR], acc1[KR];
#pragma unroll
  for (int r = 0; r < KR; ++r) acc0[r] = acc1[r] = {R(0), R(0)};
  pdl_wait();
  for (int s0 = 0; s0 < m; s0 += ROWS) {
    if (s0 > 0) __syncthreads();
#pragma unroll
    for (int q = 0; q < ROWS / FR_THREADS; ++q) {
      const int i = s0 + threadIdx.x + FR_THREADS * q;
      if (s0 > 0) row[q] = i < n1 ? n.row0 + i : (i < m ? a.border[n.bord + i - n1] : -1);
      if (row[q] >= 0) {
#pragma unroll
        for (int r = 0; r < KR; ++r) {
          CT<R> t = (i < n1 ? y : x)[(int64_t)row[q] * KR + r];
          if (i >= n1) t = {-t.re, -t.im};
          w[i - s0][r] = t;
        }
      }
    }
    __syncthreads();
    const int end = m < s0 + ROWS ? m : s0 + ROWS;
    for (int i0 = s0; i0 < end; i0 += NG * NQ) {
      if (i0 > 0) load(i0);
      if (j < ld) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const int i = i0 + grp + NG * q;
          if (i < end) {
#pragma unroll
            for (int r = 0; r < KR; ++r) {
              const CT<R> t = w[i - s0][r];
              cfma(acc0[r], m0[q], t);
              cfma(acc1[r], m1[q], t);
            }
          }
        }
      }
    }
  }
  // over the row groups of the warp, then over the warps
#pragma unroll
  for (int r = 0; r < KR; ++r) {
#pragma unroll
    for (int o = LW; o < 32; o <<= 1) {
      acc0[r].re += __shfl_xor_sync(0xffffffffu, acc0[r].re, o);
      acc0[r].im += __shfl_xor_sync(0xffffffffu, acc0[r].im, o);
      acc1[r].re += __shfl_xor_sync(0xffffffffu, acc1[r].re, o);
      acc1[r].im += __shfl_xor_sync(0xffffffffu, acc1[r].im, o);
    }
    if (lane < LW) {
      red[warp][2 * lane][r] = acc0[r];
      red[warp][2 * lane + 1][r] = acc1[r];
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < CW * KR; e += FR_THREADS) {
    const int l = e / KR, r = e % KR, c = it.t * CW + l;
    if (c >= n1) continue;
    CT<R> t = red[0][l][r];
#pragma unroll
    for (int q = 1; q < NW; ++q) {
      t.re += red[q][l][r].re;
      t.im += red[q][l][r].im;
    }
    const int64_t g = n.row0 + c;
    x[g * KR + r] = t;
    if (r >= a.nr) continue;
    ZT* dst = z + (int64_t)a.row_dof[g] * a.vs + a.off + r;
    if (a.weights == ORAS_WEIGHTS_POU) {
      if (a.row_pou[g]) z_store(dst, (double)t.re, (double)t.im);
    } else {
      z_add(dst, (double)t.re, (double)t.im);
    }
  }
}

// ------------------------------------------------------------------ many right-hand sides (FP32)
// Products of a tile of JT rows with KR = 8, 16 or 32 right-hand sides: 4 x TC entries a thread; the threads left
// over split the sum (SG groups, added at the end in a fixed order).  On levels with few nodes, where the sums run up
// to a thousand long, the tiles are narrower (Fronts::multi_cols: below 200 tiles of 64; 16 wide they take 28 us where
// 64 wide ones take 48, but twice as long on levels that fill the chip).
template <int KR, int JT> struct FrTile {
  static constexpr int TR = 4, TC = KR == 16 ? 4 : 2;         // entries a thread
  static constexpr int CG = KR / TC, RG = JT / TR;            // column and row groups
  static constexpr int SG = FR_THREADS / (CG * RG);           // sum groups
  static constexpr int KS = SG > 1 ? 8 : 16, KC = KS * SG;     // sum indices a stage, of a group and of all
  static_assert(CG * RG * SG == FR_THREADS, "threads");
};

// acc += the products of sum group sg over one stage: As [KC][JT], Bs [KC][KR].
template <int KR, int JT>
__device__ __forceinline__ void tile_stage(CT<float> (&acc)[FrTile<KR, JT>::TR][FrTile<KR, JT>::TC], const CT<float>* As,
                                           const CT<float>* Bs, int sg, int rg, int cg) {
  using T = FrTile<KR, JT>;
#pragma unroll
  for (int k = 0; k < T::KS; ++k) {
    CT<float> av[T::TR], bv[T::TC];
    const CT<float>* pa = As + (sg * T::KS + k) * JT + rg * T::TR;
    const CT<float>* pb = Bs + (sg * T::KS + k) * KR + cg * T::TC;
#pragma unroll
    for (int p = 0; p < T::TR; p += 2) ld_cpair(pa + p, av[p], av[p + 1]);
#pragma unroll
    for (int q = 0; q < T::TC; q += 2) ld_cpair(pb + q, bv[q], bv[q + 1]);
#pragma unroll
    for (int p = 0; p < T::TR; ++p)
#pragma unroll
      for (int q = 0; q < T::TC; ++q) cfma(acc[p][q], av[p], bv[q]);
  }
}

// Adds the sum groups' accumulators into group 0's, through shared memory (buf: (SG - 1) x JT x KR entries).
template <int KR, int JT>
__device__ __forceinline__ void tile_reduce(CT<float> (&acc)[FrTile<KR, JT>::TR][FrTile<KR, JT>::TC], CT<float>* buf, int sg,
                                            int rg, int cg) {
  using T = FrTile<KR, JT>;
  if (T::SG == 1) return;
  __syncthreads();
  if (sg > 0) {
#pragma unroll
    for (int p = 0; p < T::TR; ++p)
#pragma unroll
      for (int q = 0; q < T::TC; ++q) buf[((sg - 1) * JT + rg * T::TR + p) * KR + cg * T::TC + q] = acc[p][q];
  }
  __syncthreads();
  if (sg > 0) return;
#pragma unroll
  for (int g = 0; g < T::SG - 1; ++g)
#pragma unroll
    for (int p = 0; p < T::TR; ++p)
#pragma unroll
      for (int q = 0; q < T::TC; ++q) {
        const CT<float> t = buf[(g * JT + rg * T::TR + p) * KR + cg * T::TC + q];
        acc[p][q].re += t.re;
        acc[p][q].im += t.im;
      }
}

// 16 bytes into shared memory in the background, first out of L2 with `pol`; on = false: zeros.
__device__ __forceinline__ uint64_t evict_first() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void cp16_stream(void* dst, const void* src, bool on, uint64_t pol) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(on ? 16 : 0), "l"(pol) : "memory");
}
__device__ __forceinline__ void cp16(void* dst, const void* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// u = (children's) - L y for 64 border rows.  The sum is 128 long at most, so the block's whole part of L is under way
// before the level before is waited for, with the indices.  Shared memory: L, rows 16 bytes past a multiple of 128 (8 rows of
// a warp on all banks), then y.
constexpr int FR_LDL = FR_MAX_NB + 2;
template <int KR> constexpr size_t fr_fwd_smem() { return sizeof(CT<float>) * ((size_t)64 * FR_LDL + (size_t)FR_MAX_NB * KR); }
template <int KR>
__global__ void __launch_bounds__(FR_THREADS) k_fr_fwd_multi(FrApply a, const FrontItem* __restrict__ items,
                                                             const CT<float>* __restrict__ fac,
                                                             const cplx* v, CT<float>* y,
                                                             CT<float>* u) {
  using T = FrTile<KR, 64>;
  using C = CT<float>;
  extern __shared__ __align__(16) unsigned char fr_smem[];
  __shared__ FrontSrc osrc[FR_MAX_NB];
  __shared__ int32_t odof[FR_MAX_NB];
  C* Ls = (C*)fr_smem;                                  // [64][FR_LDL]
  C* own = Ls + 64 * FR_LDL;                            // [FR_MAX_NB][KR]
  static_assert((T::SG - 1) * 64 * KR <= 64 * FR_LDL + FR_MAX_NB * KR && FR_THREADS % KR == 0, "the reduction fits, a thread has one column");
  pdl_release();
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, ld = n.ld, i0 = it.t * 64, tid = threadIdx.x;
  const C* rows = fac + n.panel + (int64_t)(n1 + i0) * ld;
  const uint64_t pol = evict_first();
  const int live = n.n2 - i0 < 64 ? n.n2 - i0 : 64;     // border rows of this block; the others' results are dropped
  for (int i = tid >> 4; i < live; i += FR_THREADS / 16)
    for (int c = 2 * (tid & 15); c < ld; c += 32) cp16_stream(Ls + i * FR_LDL + c, rows + (int64_t)i * ld + c, true, pol);
  cp_commit();
  if (tid < n1) {
    osrc[tid] = a.own_src[n.row0 + tid];
    odof[tid] = a.row_dof[n.row0 + tid];
  }
  const int cg = tid % T::CG, rg = tid / T::CG % T::RG, sg = tid / (T::CG * T::RG);
  FrontSrc bsrc[T::TR];                                 // of rows rg + RG p
#pragma unroll
  for (int p = 0; p < T::TR; ++p) {
    const int i = rg + T::RG * p;
    bsrc[p] = sg == 0 && i < live ? a.border_src[n.bord + i0 + i] : FrontSrc{-1, -1};
  }
  __syncthreads();
  pdl_wait();
  constexpr int BATCH = 4;                              // entries of y whose loads are in flight together
  for (int e0 = tid; e0 < ld * KR; e0 += BATCH * FR_THREADS) {
    C t[BATCH];
#pragma unroll
    for (int q = 0; q < BATCH; ++q) {
      const int c = (e0 + q * FR_THREADS) / KR, r = tid % KR;
      t[q] = {0.0f, 0.0f};
      if (c < n1) {
        if (r < a.nr) {
          const cplx b = v[(int64_t)odof[c] * a.vs + a.off + r];
          t[q] = {(float)b.re, (float)b.im};
        }
        const C up = pull_vec<float, KR>(u, osrc[c], r);
        t[q].re += up.re;
        t[q].im += up.im;
      }
    }
#pragma unroll
    for (int q = 0; q < BATCH; ++q) {
      const int e = e0 + q * FR_THREADS;
      if (e >= ld * KR) break;
      if (it.t == 0 && e < n1 * KR) y[(int64_t)n.row0 * KR + e] = t[q];
      own[e] = t[q];
    }
  }
  C acc[T::TR][T::TC];
#pragma unroll
  for (int p = 0; p < T::TR; ++p)
#pragma unroll
    for (int q = 0; q < T::TC; ++q) acc[p][q] = {0.0f, 0.0f};
  cp_wait<0>();
  __syncthreads();
  const int part = (ld + 2 * T::SG - 1) / (2 * T::SG) * 2;  // sum indices of a group, in pairs (ld is a multiple of 4)
  const int k1 = (sg + 1) * part < ld ? (sg + 1) * part : ld;
#pragma unroll 4
  for (int k = sg * part; k < k1; k += 2) {
    C a0[T::TR], a1[T::TR], b0[T::TC], b1[T::TC];
#pragma unroll
    for (int p = 0; p < T::TR; ++p) ld_cpair(Ls + (rg + T::RG * p) * FR_LDL + k, a0[p], a1[p]);
#pragma unroll
    for (int q = 0; q < T::TC; q += 2) {
      ld_cpair(own + k * KR + cg * T::TC + q, b0[q], b0[q + 1]);
      ld_cpair(own + (k + 1) * KR + cg * T::TC + q, b1[q], b1[q + 1]);
    }
#pragma unroll
    for (int p = 0; p < T::TR; ++p)
#pragma unroll
      for (int q = 0; q < T::TC; ++q) {
        cfma(acc[p][q], a0[p], b0[q]);
        cfma(acc[p][q], a1[p], b1[q]);
      }
  }
  tile_reduce<KR, 64>(acc, (C*)fr_smem, sg, rg, cg);
  if (sg > 0) return;
#pragma unroll
  for (int p = 0; p < T::TR; ++p) {
    const int i = rg + T::RG * p;
    if (i >= live) continue;
#pragma unroll
    for (int q = 0; q < T::TC; ++q) {
      const int r = cg * T::TC + q;
      const C up = pull_vec<float, KR>(u, bsrc[p], r);
      u[(n.bord + i0 + i) * KR + r] = {up.re - acc[p][q].re, up.im - acc[p][q].im};
    }
  }
}

// x = [S; L]^T [y; -x(border)] for JT own unknowns, FR_STAGES stages of panel rows and rows of [y; -x] in shared memory: a
// stage's loads have the products of the three before it to arrive in.  The x buffer holds -x, as the levels below use it.
constexpr int FR_STAGES = 4;
template <int KR, int JT> constexpr size_t fr_bwd_smem() {
  return sizeof(CT<float>) * (size_t)FR_STAGES * FrTile<KR, JT>::KC * (JT + KR);
}
template <typename ZT, int KR, int JT>
__global__ void __launch_bounds__(FR_THREADS) k_fr_bwd_multi(FrApply a, const FrontItem* __restrict__ items,
                                                             const CT<float>* __restrict__ fac,
                                                             const CT<float>* y, CT<float>* x,
                                                             ZT* z) {
  using T = FrTile<KR, JT>;
  using C = CT<float>;
  constexpr int KC = T::KC, STAGE = KC * (JT + KR);
  constexpr int GL = JT / 2, GQ = (KC * GL + FR_THREADS - 1) / FR_THREADS;   // 16-byte pieces of a panel row, per thread
  constexpr int WL = KR / 2, WQ = (KC * WL + FR_THREADS - 1) / FR_THREADS;   // of a row of [y; -x]
  static_assert((T::SG - 1) * JT * KR <= FR_STAGES * STAGE, "the reduction fits");
  extern __shared__ __align__(16) unsigned char fr_smem[];
  C* buf = (C*)fr_smem;                                       // [FR_STAGES] of [KC][JT], [KC][KR]
  pdl_release();
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = a.nodes[it.node];
  const int n1 = n.n1, m = n.n1 + n.n2, ld = n.ld, j0 = it.t * JT, tid = threadIdx.x;
  const C* panel = fac + n.panel;
  const uint64_t pol = evict_first();
  auto load_panel = [&](int s) {
    C* g = buf + s % FR_STAGES * STAGE;
#pragma unroll
    for (int q = 0; q < GQ; ++q) {
      const int e = tid + FR_THREADS * q, k = e / GL, c = e % GL * 2, i = s * KC + k;
      if (k >= KC) break;
      const bool on = i < m && j0 + c < ld;
      cp16_stream(g + k * JT + c, on ? panel + (int64_t)i * ld + j0 + c : panel, on, pol);
    }
  };
  int32_t row[WQ];                                            // rows of [y; -x] of the stage load_w takes next
  auto load_rows = [&](int s) {
#pragma unroll
    for (int q = 0; q < WQ; ++q) {
      const int k = (tid + FR_THREADS * q) / WL, i = s * KC + k;
      row[q] = k >= KC || i >= m ? -1 : (i < n1 ? n.row0 + i : a.border[n.bord + i - n1]);
    }
  };
  auto load_w = [&](int s) {
    C* w = buf + s % FR_STAGES * STAGE + KC * JT;
#pragma unroll
    for (int q = 0; q < WQ; ++q) {
      const int e = tid + FR_THREADS * q, k = e / WL, r = e % WL * 2;
      if (k >= KC) break;
      const C* src = s * KC + k < n1 ? y : x;
      cp16(w + k * KR + r, row[q] >= 0 ? src + (int64_t)row[q] * KR + r : y, row[q] >= 0);
    }
    load_rows(s + 1);
  };
  const int stages = (m + KC - 1) / KC;
  load_rows(0);
  for (int s = 0; s < FR_STAGES - 1 && s < stages; ++s) load_panel(s);
  pdl_wait();
#pragma unroll
  for (int s = 0; s < FR_STAGES - 1; ++s) {
    if (s < stages) load_w(s);
    cp_commit();
  }
  const int cg = tid % T::CG, rg = tid / T::CG % T::RG, sg = tid / (T::CG * T::RG);
  C acc[T::TR][T::TC];
#pragma unroll
  for (int p = 0; p < T::TR; ++p)
#pragma unroll
    for (int q = 0; q < T::TC; ++q) acc[p][q] = {0.0f, 0.0f};
  for (int s = 0; s < stages; ++s) {
    cp_wait<FR_STAGES - 2>();
    __syncthreads();  // stage s has arrived, stage s - 1 has been used
    if (s + FR_STAGES - 1 < stages) {
      load_panel(s + FR_STAGES - 1);
      load_w(s + FR_STAGES - 1);
    }
    cp_commit();
    const C* g = buf + s % FR_STAGES * STAGE;
    if (s * KC + sg * T::KS < m) tile_stage<KR, JT>(acc, g, g + KC * JT, sg, rg, cg);  // rows past the panel are zeros
  }
  cp_wait<0>();
  tile_reduce<KR, JT>(acc, buf, sg, rg, cg);
  if (sg > 0) return;
#pragma unroll
  for (int p = 0; p < T::TR; ++p) {
    const int c = j0 + rg * T::TR + p;
    if (c >= n1) continue;
    const int64_t row = n.row0 + c;
    const int64_t dof = a.row_dof[row];
    const bool pou = a.row_pou[row] != 0;
#pragma unroll
    for (int q = 0; q < T::TC; ++q) {
      const int r = cg * T::TC + q;
      const C t = acc[p][q];
      x[row * KR + r] = {-t.re, -t.im};
      if (r >= a.nr) continue;
      ZT* dst = z + dof * a.vs + a.off + r;
      if (a.weights == ORAS_WEIGHTS_POU) {
        if (pou) z_store(dst, (double)t.re, (double)t.im);
      } else {
        z_add(dst, (double)t.re, (double)t.im);
      }
    }
  }
}

// ------------------------------------------------------------------ host side
// Right-hand sides of the next pass when `rem` are left: the smallest pass that takes them all, up to 32
// (FP32) or 2 (FP64).
static int fr_kr(const oras_handle* h, int rem) {
  if (h->opt.factor_bits == 64) return rem >= 2 ? 2 : 1;
  return rem > 16 ? 32 : (rem > 8 ? 16 : (rem > 4 ? 8 : (rem > 2 ? 4 : rem)));
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

// A launch that may start before the kernel before it in the stream has finished (pdl_wait in the kernel).
template <typename... P, typename... A>
static void launch_pdl(void (*fn)(P...), int64_t blocks, size_t smem, cudaStream_t st, A... args) {
  if (blocks <= 0) return;
  if (smem > 48 * 1024) allow_max_smem((const void*)fn);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(FR_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
  count_launches(1);
}

template <typename R, typename ZT, int KR>
static void fr_pass(const oras_handle* h, void* buf, const cplx* v, ZT* z, int64_t vs, int64_t off, int nr) {
  const auto& d = h->dev;
  const Fronts& f = h->fronts;
  FrApply a;
  a.nodes = d.fr_nodes; a.border = d.fr_border; a.own_src = d.fr_own_src; a.border_src = d.fr_border_src;
  a.row_dof = d.fr_row_dof; a.row_pou = d.fr_row_pou;
  a.weights = h->opt.weights;
  a.vs = vs; a.off = off; a.nr = nr;
  const int64_t rows = h->mesh.sub_ns_off[h->mesh.nsub];
  CT<R>* y = (CT<R>*)buf;
  CT<R>* x = y + rows * KR;
  CT<R>* u = x + rows * KR;
  const CT<R>* fac = (const CT<R>*)d.arena;
  cudaStream_t st = d.stream;
  for (int l = 0; l < f.nlev(); ++l) {
    const FrontItem* items = d.fr_fwd + f.fwd.ptr[l];
    const int64_t nb = f.fwd.ptr[l + 1] - f.fwd.ptr[l];
    if constexpr (KR >= 8) launch_pdl(k_fr_fwd_multi<KR>, nb, fr_fwd_smem<KR>(), st, a, items, fac, v, y, u);
    else launch_pdl(k_fr_fwd<R, KR>, nb, 0, st, a, items, fac, v, y, u);
  }
  for (int l = f.nlev() - 1; l >= 0; --l) {
    if constexpr (KR >= 8) {
      const FrontItem* items = d.fr_bwd_multi + f.bwd_multi.ptr[l];
      const int64_t nb = f.bwd_multi.ptr[l + 1] - f.bwd_multi.ptr[l];
      if (f.multi_cols[l] == 64) launch_pdl(k_fr_bwd_multi<ZT, KR, 64>, nb, fr_bwd_smem<KR, 64>(), st, a, items, fac, y, x, z);
      else launch_pdl(k_fr_bwd_multi<ZT, KR, 16>, nb, fr_bwd_smem<KR, 16>(), st, a, items, fac, y, x, z);
    } else {
      const FrontItem* items = d.fr_bwd + f.bwd.ptr[l];
      const int64_t nb = f.bwd.ptr[l + 1] - f.bwd.ptr[l];
      if (f.bwd_cols[l] == 32) launch_pdl(k_fr_bwd<R, ZT, KR, 32>, nb, 0, st, a, items, fac, y, x, z);
      else if (f.bwd_cols[l] == 16) launch_pdl(k_fr_bwd<R, ZT, KR, 16>, nb, 0, st, a, items, fac, y, x, z);
      else launch_pdl(k_fr_bwd<R, ZT, KR, 8>, nb, 0, st, a, items, fac, y, x, z);
    }
  }
}

// z = M^{-1} v for k right-hand sides, right-hand side r of unknown g at g * vs + r * rs of v and z: adjacent ones
// (rs = 1, vs = k) in groups, with their local vectors in ybuf; or columns (vs = 1) one at a time, in y1.
template <typename R, typename ZT>
static int fr_apply_t(const oras_handle* h, const cplx* v, ZT* z, int k, int64_t vs, int64_t rs) {
  const auto& d = h->dev;
  void* buf = rs == 1 ? d.ybuf : d.y1;
  if (!buf || (rs == 1 && d.ybuf_bytes < fronts_ybytes(h, k))) return -1;
  if (h->opt.weights != ORAS_WEIGHTS_POU &&
      cudaMemsetAsync(z, 0, sizeof(ZT) * (size_t)h->mesh.ndof * k, d.stream) != cudaSuccess)
    return -1;
  for (int r0 = 0; r0 < k;) {
    const int kr = rs == 1 ? fr_kr(h, k - r0) : 1, nr = std::min(kr, k - r0);
    const int64_t off = r0 * rs;
    if (kr == 1) fr_pass<R, ZT, 1>(h, buf, v, z, vs, off, nr);
    else if (kr == 2) fr_pass<R, ZT, 2>(h, buf, v, z, vs, off, nr);
    else if constexpr (sizeof(R) == 4) {
      if (kr == 4) fr_pass<R, ZT, 4>(h, buf, v, z, vs, off, nr);
      else if (kr == 8) fr_pass<R, ZT, 8>(h, buf, v, z, vs, off, nr);
      else if (kr == 16) fr_pass<R, ZT, 16>(h, buf, v, z, vs, off, nr);
      else fr_pass<R, ZT, 32>(h, buf, v, z, vs, off, nr);
    }
    r0 += nr;
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int fronts_apply_f64out(const oras_handle* h, const cplx* v, cplx* z, int k) {
  return h->dev.factor_bits == 64 ? fr_apply_t<double, cplx>(h, v, z, k, k, 1) : fr_apply_t<float, cplx>(h, v, z, k, k, 1);
}
int fronts_apply_noalloc(const oras_handle* h, const cplx* v, cplx* z, int k) {
  const int64_t n = h->mesh.ndof;
  return h->dev.factor_bits == 64 ? fr_apply_t<double, cplx>(h, v, z, k, 1, n) : fr_apply_t<float, cplx>(h, v, z, k, 1, n);
}
int fronts_apply_f32out(const oras_handle* h, const cplx* v, void* z, int k) {
  return fr_apply_t<float, CT<float>>(h, v, (CT<float>*)z, k, k, 1);
}

}  // namespace oras
