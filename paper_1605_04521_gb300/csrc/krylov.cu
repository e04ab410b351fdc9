// FP64 Krylov kernels of the right-preconditioned FGMRES(m) (Sec. 5): complex CSR SpMV, Gram-Schmidt Arnoldi in blocks
// of 8 basis vectors (classical inside a block, modified from block to block) with fused (update + next dots) passes,
// complex Givens rotations on the device, the small triangular solve and the solution update.  Multi-vectors are
// stored [N][k] (the k right-hand sides of a pseudo-block solve adjacent in memory).
// Every reduction is a fixed two-stage sum (block partials, then a fixed-order sum), so the
// results do not depend on scheduling.
#include <algorithm>

#include "dev.cuh"

namespace oras {

constexpr int RED_BLOCKS = 304;   // 2 x 152 SMs
constexpr int RED_THREADS = 256;

template <typename XT> __device__ __forceinline__ cplx ld_c(const XT* p, int64_t i);
template <> __device__ __forceinline__ cplx ld_c<cplx>(const cplx* p, int64_t i) { return ld16(p + i); }
template <> __device__ __forceinline__ cplx ld_c<CT<float>>(const CT<float>* p, int64_t i) {
  CT<float> v = p[i];
  return {(double)v.re, (double)v.im};
}

// Both products with A give a row SPMV_LPR lanes: KL of them take one right-hand side each (x and y rows are
// adjacent in memory over the right-hand sides, a value of A is broadcast), the EL = SPMV_LPR / KL groups
// share the row's entries.  Each lane issues the (value, column) loads of UNR entries at once, then their x
// gathers, then the arithmetic.  The kernels are bound by issue slots (the FP32-pipe product has 44 arithmetic
// instructions an entry), so the rest is kept short: entries are indexed from the row's first in 32 bits, past
// the row's end its last entry is loaded again and not used, and an x address is one multiply-add.  With more
// than KL right-hand sides the blocks of the same rows are neighbours in the grid, so the rows of A come from L2
// after the first.
constexpr int SPMV_LPR = 8;

template <int KL> struct SpmvLane {
  static constexpr int EL = SPMV_LPR / KL;
  static constexpr int UNR = EL == 8 ? 6 : 4;   // a degree-2 row (42 entries) in one go of 8 lanes
  int64_t row;
  int r, el;
  bool on;
  __device__ SpmvLane(int64_t n, int k, int chunks) {
    const int sl = threadIdx.x % SPMV_LPR;
    row = ((int64_t)(blockIdx.x / chunks) * blockDim.x + threadIdx.x) / SPMV_LPR;
    r = (int)(blockIdx.x % chunks) * KL + sl % KL;
    el = sl / KL;
    on = row < n && r < k;
  }
};

// y = A x  (x: [N][k] in XT, y: [N][k] FP64), four fused multiply-adds an entry: bound by the FP64 pipe
// (2 lanes a clock an SM), so no lane idles for a whole row and the sums over lanes are few.  8 fields of the
// 20^3 degree-2 problem: a warp a row, unfused, 2.99 ms; now 0.84 ms.
template <typename XT, int KL>
__global__ void __launch_bounds__(256) k_spmv(int64_t n, const int64_t* __restrict__ rowptr,
                                              const int32_t* __restrict__ cols, const cplx* __restrict__ vals,
                                              const XT* __restrict__ x, cplx* __restrict__ y, int k, int chunks) {
  const SpmvLane<KL> L(n, k, chunks);
  constexpr int EL = SpmvLane<KL>::EL;
  constexpr int UNR = SpmvLane<KL>::UNR;
  cplx acc = {0.0, 0.0};
  if (L.on) {
    const int64_t p0 = rowptr[L.row];
    const int len = (int)(rowptr[L.row + 1] - p0);
    const cplx* av = vals + p0;
    const int32_t* cv = cols + p0;
    const char* xb = reinterpret_cast<const char*>(x + L.r);
    const uint32_t stride = (uint32_t)(k * sizeof(XT));
    for (int i = L.el; i < len; i += EL * UNR) {
      cplx a[UNR], v[UNR];
      uint32_t c[UNR];
#pragma unroll
      for (int u = 0; u < UNR; ++u) {
        const int q = min(i + u * EL, len - 1);
        a[u] = ld16(av + q);
        c[u] = (uint32_t)cv[q];
      }
#pragma unroll
      for (int u = 0; u < UNR; ++u) v[u] = ld_c<XT>(reinterpret_cast<const XT*>(xb + (uint64_t)c[u] * stride), 0);
#pragma unroll
      for (int u = 0; u < UNR; ++u)
        if (i + u * EL < len) {
          acc.re = fma(a[u].re, v[u].re, acc.re);
          acc.im = fma(a[u].re, v[u].im, acc.im);
          acc.re = fma(-a[u].im, v[u].im, acc.re);
          acc.im = fma(a[u].im, v[u].re, acc.im);
        }
    }
  }
#pragma unroll
  for (int o = SPMV_LPR / 2; o >= KL; o >>= 1) {
    acc.re += __shfl_down_sync(0xffffffffu, acc.re, o, SPMV_LPR);
    acc.im += __shfl_down_sync(0xffffffffu, acc.im, o, SPMV_LPR);
  }
  if (L.on && L.el == 0) st16(y + L.row * k + L.r, acc);
}

// ------------------------------------------------------------------ FP32-pipe SpMV, FP64 accuracy
// GB300 executes FP64 on a narrow pipe (about 1/64 of the FP32 rate), which caps the FP64 CSR
// SpMV far below the HBM bound.  The Arnoldi SpMV multiplies the FP64 matrix by preconditioned
// vectors that are exactly FP32 (z = M^-1 v with FP32 factors), so it is done on the FP32 pipes
// with error-free transformations: A = A_hi + A_lo with A_hi = fl32(A) and A_lo = fl32(A - A_hi)
// (the same 16 bytes per entry as FP64 complex), each product A_hi x split exactly into
// p + e by one FMA (two-product), each running sum kept as an unevaluated pair hi + lo with the
// rounding error of every addition recovered exactly (two-sum, Knuth).  The result carries
// about 2^-48 relative error per entry, the accuracy class of FP64, and is stored in FP64.

// hi + lo += a * x with a = a_hi + a_lo
__device__ __forceinline__ void df_mac(float& hi, float& lo, float a_hi, float a_lo, float x) {
  const float p = a_hi * x;
  const float ep = fmaf(a_hi, x, -p);           // a_hi * x - p, exactly
  const float t = hi + p;
  const float bp = t - hi;
  const float es = (hi - (t - bp)) + (p - bp);   // hi + p - t, exactly
  hi = t;
  lo += (ep + es) + a_lo * x;
}
// (h1 + l1) += (h2 + l2)
__device__ __forceinline__ void df_add(float& h1, float& l1, float h2, float l2) {
  const float t = h1 + h2;
  const float bp = t - h1;
  const float es = (h1 - (t - bp)) + (h2 - bp);
  h1 = t;
  l1 += es + l2;
}

// Exact float -> double by bit construction on the integer pipes (the conversion instruction runs
// on the FP64 pipe, which GB300 keeps narrow).  Subnormal floats become zero.
__device__ __forceinline__ double f2d_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t ex = (u >> 23) & 0xFFu;
  const uint64_t sign = (uint64_t)(u & 0x80000000u) << 32;
  if (ex == 0) return __longlong_as_double((long long)sign);
  const uint64_t e64 = ex == 0xFFu ? 0x7FFull : (uint64_t)ex + 896u;  // rebias 127 -> 1023
  return __longlong_as_double((long long)(sign | (e64 << 52) | ((uint64_t)(u & 0x7FFFFFu) << 29)));
}

// vals_df[p] = {re_hi, im_hi, re_lo, im_lo}
__global__ void k_split_vals(int64_t nnz, const cplx* __restrict__ vals, float4* __restrict__ out) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nnz) return;
  const cplx v = ld16(vals + p);
  const float rh = (float)v.re, ih = (float)v.im;
  out[p] = make_float4(rh, ih, (float)(v.re - (double)rh), (float)(v.im - (double)ih));
}

// y = A x with x complex FP32 ([N][k]), y FP64 ([N][k]).  Predicated 64-bit indexing against this: one field of the
// 12^3 x 6, degree-3 problem 98 -> 92 us (the public call), three of the 10^3 one 82 -> 70 ms for a whole solve's products.
template <int KL>
__global__ void __launch_bounds__(256) k_spmv_df(int64_t n, const int64_t* __restrict__ rowptr,
                                                 const int32_t* __restrict__ cols, const float4* __restrict__ vals,
                                                 const CT<float>* __restrict__ x, cplx* __restrict__ y, int k,
                                                 int chunks) {
  const SpmvLane<KL> L(n, k, chunks);
  constexpr int EL = SpmvLane<KL>::EL;
  constexpr int UNR = SpmvLane<KL>::UNR;
  float rh = 0.0f, rl = 0.0f, ih = 0.0f, il = 0.0f;
  if (L.on) {
    const int64_t p0 = rowptr[L.row];
    const int len = (int)(rowptr[L.row + 1] - p0);
    const float4* av = vals + p0;
    const int32_t* cv = cols + p0;
    const char* xb = reinterpret_cast<const char*>(x + L.r);
    const uint32_t stride = (uint32_t)(k * sizeof(CT<float>));
    for (int i = L.el; i < len; i += EL * UNR) {
      float4 a[UNR];
      uint32_t c[UNR];
#pragma unroll
      for (int u = 0; u < UNR; ++u) {
        const int q = min(i + u * EL, len - 1);
        a[u] = av[q];
        c[u] = (uint32_t)cv[q];
      }
      float2 xv[UNR];
#pragma unroll
      for (int u = 0; u < UNR; ++u) xv[u] = *reinterpret_cast<const float2*>(xb + (uint64_t)c[u] * stride);
#pragma unroll
      for (int u = 0; u < UNR; ++u)
        if (i + u * EL < len) {
          df_mac(rh, rl, a[u].x, a[u].z, xv[u].x);    // + a_re x_re
          df_mac(rh, rl, -a[u].y, -a[u].w, xv[u].y);  // - a_im x_im
          df_mac(ih, il, a[u].x, a[u].z, xv[u].y);    // + a_re x_im
          df_mac(ih, il, a[u].y, a[u].w, xv[u].x);    // + a_im x_re
        }
    }
  }
#pragma unroll
  for (int o = SPMV_LPR / 2; o >= KL; o >>= 1) {
    const float h2 = __shfl_down_sync(0xffffffffu, rh, o, SPMV_LPR), l2 = __shfl_down_sync(0xffffffffu, rl, o, SPMV_LPR);
    const float h3 = __shfl_down_sync(0xffffffffu, ih, o, SPMV_LPR), l3 = __shfl_down_sync(0xffffffffu, il, o, SPMV_LPR);
    df_add(rh, rl, h2, l2);
    df_add(ih, il, h3, l3);
  }
  if (L.on && L.el == 0) st16(y + L.row * k + L.r, {f2d_bits(rh) + f2d_bits(rl), f2d_bits(ih) + f2d_bits(il)});
}

// Reductions over [N][k] multi-vectors (element e belongs to right-hand side e % k).  The grid's
// threads are cut to a multiple of k, teff = floor(T / k) k, and thread t < teff visits the
// elements t, t + teff, t + 2 teff, ...: all of one right-hand side r = t % k, so each thread
// keeps one accumulator per reduced value.  Block partial sums per value and right-hand side, then a
// sum over the blocks by one warp each (k_sum_partials), all in a fixed order that depends on the
// sizes only: the results do not depend on scheduling.
__device__ __forceinline__ int64_t red_teff(int k) {
  const int64_t T = (int64_t)gridDim.x * blockDim.x;
  return T / k * k;
}

__device__ __forceinline__ cplx shfl_down_c(cplx v, int d) {
  return {__shfl_down_sync(0xffffffffu, v.re, d), __shfl_down_sync(0xffffffffu, v.im, d)};
}

// partials[(q k + r) gridDim.x + blockIdx.x] = sum of v[q] over the block's threads of right-hand side r,
// q < nv.  Through shared memory, one warp a value: lane r + k p adds the threads of r numbered p, p + P, ...
// (P = 32 / k lanes a right-hand side), then a tree over p.  FP64 adds cost 64 cycles a warp on a
// quarter of an SM, so every sum is formed once (a butterfly of all values over all lanes took 5x as many).
template <int NV>
__device__ void block_reduce_store(const cplx (&v)[NV], int nv, int k, cplx* __restrict__ partials) {
  __shared__ cplx sh[NV][RED_THREADS];
#pragma unroll
  for (int q = 0; q < NV; ++q)
    if (q < nv) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = (int)((int64_t)blockIdx.x * blockDim.x % k);  // right-hand side of thread 0
  const int P = k < 32 ? 32 / k : 1;
  for (int q = warp; q < nv; q += RED_THREADS / 32)
    for (int r0 = 0; r0 < k; r0 += 32) {
      const int r = r0 + lane % (k < 32 ? k : 32), p = k < 32 ? lane / k : 0;
      const bool on = r < k && p < P;
      cplx t = {0.0, 0.0};
      if (on) {
        const int first = r >= base ? r - base : r - base + k;  // first thread of right-hand side r
        for (int i = first + k * p; i < RED_THREADS; i += k * P) t = cadd(t, sh[q][i]);
      }
      for (int left = P; left > 1;) {
        const int half = (left + 1) / 2;
        const cplx o = shfl_down_c(t, half * k & 31);
        if (on && p + half < left) t = cadd(t, o);
        left = half;
      }
      if (on && p == 0) partials[((int64_t)q * k + r) * gridDim.x + blockIdx.x] = t;
    }
}

// Fixed-order sum of nb block partials by one warp: lane l adds those of blocks l, l + 32, ... (their loads
// overlap), a fixed xor-shuffle tree combines the lanes.  Every lane returns the total.
__device__ __forceinline__ cplx sum_partials_warp(const cplx* __restrict__ partials, int nb, int lane) {
  constexpr int PER = (RED_BLOCKS + 31) / 32;
  cplx v[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int b = lane + 32 * q;
    v[q] = b < nb ? partials[b] : cplx{0.0, 0.0};
  }
  cplx t = v[0];
#pragma unroll
  for (int q = 1; q < PER; ++q)
    if (32 * q < nb) t = cadd(t, v[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    t.re += __shfl_xor_sync(0xffffffffu, t.re, o);
    t.im += __shfl_xor_sync(0xffffffffu, t.im, o);
  }
  return t;
}

// hs[q k + r] = sum of the block partials; with H, also stored as H[r][i0 + q][j].  One warp a sum.
__global__ void __launch_bounds__(256) k_sum_partials(int n, int k, int nb, const cplx* __restrict__ partials,
                                                      cplx* __restrict__ hs, int m, int i0, int j,
                                                      cplx* __restrict__ H) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w >= n * k) return;
  const cplx t = sum_partials_warp(partials + (int64_t)w * nb, nb, lane);
  if (lane != 0) return;
  hs[w] = t;
  if (H) H[((int64_t)(w % k) * (m + 1) + i0 + w / k) * m + j] = t;
}

// One pass of the blocked Gram-Schmidt: w -= sum_q h_q V_q over the nv basis vectors from V (h
// from hs), then the block partials of <Vn_q, w> over the nn vectors from Vn (nn = 0: of |w|^2 instead).
// Vectors are nk apart.  A block's coefficients are taken together, blocks one after the other: against modified
// Gram-Schmidt over single vectors the basis loses a third more of its orthogonality (5^3 x 6, degree 2, 8 subdomains
// without overlap, after 40, 60 and 100 steps 1.2e-12, 3.2e-11 and 3.0e-8 against 0.9e-12, 2.5e-11 and 2.3e-8), the
// residuals agree to 2 digits and the steps to 1e-8, 1e-11 and 1e-13 are the same.  Bound: the FP64 pipe, 8 fused multiply-adds an entry
// and basis vector; a pass over 8 vectors of 352,170 entries
// takes 51 us with that pipe 70% busy.  One vector a pass (a launch, a reduction and w through memory each) took 21 us
// a vector of 542,736 entries.
constexpr int MGS_BLOCK = 8;
__global__ void __launch_bounds__(RED_THREADS) k_mgs_block(int64_t nk, int k, int nv, const cplx* __restrict__ V,
                                                           int nn, const cplx* __restrict__ Vn,
                                                           cplx* __restrict__ w, const cplx* __restrict__ hs,
                                                           cplx* __restrict__ partials) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, teff = red_teff(k);
  cplx acc[MGS_BLOCK];
#pragma unroll
  for (int q = 0; q < MGS_BLOCK; ++q) acc[q] = {0.0, 0.0};
  if (t < teff) {
    cplx h[MGS_BLOCK];
#pragma unroll
    for (int q = 0; q < MGS_BLOCK; ++q) h[q] = q < nv ? hs[q * k + t % k] : cplx{0.0, 0.0};
    for (int64_t e = t; e < nk; e += teff) {
      cplx x = ld16(w + e);
      cplx u[MGS_BLOCK];
      if (nv > 0) {
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nv) u[q] = ld16(V + q * nk + e);
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nv) {
            x.re = fma(-h[q].re, u[q].re, x.re);
            x.im = fma(-h[q].re, u[q].im, x.im);
            x.re = fma(h[q].im, u[q].im, x.re);
            x.im = fma(-h[q].im, u[q].re, x.im);
          }
        st16(w + e, x);
      }
      if (nn > 0) {
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nn) u[q] = ld16(Vn + q * nk + e);
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nn) {
            acc[q].re = fma(u[q].re, x.re, acc[q].re);
            acc[q].im = fma(u[q].re, x.im, acc[q].im);
            acc[q].re = fma(u[q].im, x.im, acc[q].re);
            acc[q].im = fma(-u[q].im, x.re, acc[q].im);
          }
      } else {
        acc[0].re = fma(x.re, x.re, acc[0].re);
        acc[0].re = fma(x.im, x.im, acc[0].re);
      }
    }
  }
  block_reduce_store<MGS_BLOCK>(acc, nn > 0 ? nn : 1, k, partials);
}

// Rotation j of right-hand side r from column j's running entry a and h_{j+1,j} = bb; updates g, res = |g_{j+1}|.
__device__ __forceinline__ void givens_finish(int r, int m, int j, cplx a, double bb, cplx* __restrict__ H,
                                              double* __restrict__ cs, cplx* __restrict__ sn, cplx* __restrict__ g,
                                              double* __restrict__ host_res) {
  cplx* Hr = H + (int64_t)r * (m + 1) * m;
  cplx* gr = g + (int64_t)r * (m + 1);
  const double aa = hypot(a.re, a.im);
  double cj;
  cplx sj;
  if (bb == 0.0) { cj = 1.0; sj = {0.0, 0.0}; }
  else if (aa == 0.0) { cj = 0.0; sj = {1.0, 0.0}; }
  else {
    const double den = hypot(aa, bb);
    cj = aa / den;
    sj = {a.re / aa * bb / den, a.im / aa * bb / den};
  }
  cs[(int64_t)r * m + j] = cj;
  sn[(int64_t)r * m + j] = sj;
  Hr[(int64_t)j * m + j] = cadd(cscale(a, cj), cscale(sj, bb));
  Hr[(int64_t)(j + 1) * m + j] = {0.0, 0.0};
  const cplx gj = gr[j];
  gr[j + 1] = cscale(cmul(cconj(sj), gj), -1.0);
  gr[j] = cscale(gj, cj);
  host_res[r] = hypot(gr[j + 1].re, gr[j + 1].im);
}

// ------------------------------------------------------------------ one launch an Arnoldi step
// The same blocked Gram-Schmidt, the norm, V_{j+1} and the Givens update in one cooperative launch, one block an SM
// with its share of w in shared memory; after a pass the blocks exchange their partial sums through a grid barrier
// and each adds all of them.  The passes of k_mgs_block cost 7-11 us each beside their arithmetic (two
// launches, w through memory, a reduction of 512 threads an SM), and their 512 entries a block left most SMs idle
// on short vectors.  Entries are dealt out evenly: every SM has the same share of the last, partial round.
// Bound: the FP64 pipe, as there.  Orthogonalisation of a whole solve, launches above -> this: three columns of the 10^3 x 6, degree-3
// problem (352,170 entries a vector, restart 100) 317 -> 239 ms (169 ms of FP64 instructions), one of the 24^3 one 176 -> 141,
// eight at degree 3 6.2 -> 5.0, one of the 16^3 one 2.31 -> 1.61, of the 4^3 one 0.52 -> 0.28.  A block adds the sums of all others, MGS_BLOCK k ones of gridDim.x
// partials, which is why k ends at ORTH_MAX_K; w ends at ORTH_MAX_ROUNDS rounds of the block's shared memory
// (1.4e6 entries).  Others take the launches above.
// Waits are bounded: a block that gives up reports DEV_TIMEOUT and leaves, and so do then the others.
constexpr int ORTH_THREADS = 512, ORTH_MAX_K = 8, ORTH_MAX_ROUNDS = 18;

struct OrthArgs {
  int64_t nk, chunk;                 // entries, entries a block (a multiple of k)
  int k, m, j;
  const cplx* V;                     // V_0
  const cplx* w;
  cplx* Vn;                          // V_{j+1}
  cplx* partials;                    // [2][MGS_BLOCK][gridDim.x][k], by pass parity
  cplx* H;
  double* cs;
  cplx* sn;
  cplx* g;
  double* host_res;
  int32_t* status;
  int32_t* host_status;
  uint64_t wait_ns;
};

// Sums over the p of the values of lanes r + k p, P of them, into lanes r.
__device__ __forceinline__ cplx sum_lanes(cplx t, int k, int P, int p) {
  for (int left = P; left > 1;) {
    const int half = (left + 1) / 2;
    const cplx o = shfl_down_c(t, half * k & 31);
    if (p + half < left) t = cadd(t, o);
    left = half;
  }
  return t;
}

__global__ void __launch_bounds__(ORTH_THREADS, 1) k_orth(OrthArgs a) {
  extern __shared__ __align__(16) unsigned char orth_smem[];
  cplx* red = (cplx*)orth_smem;                        // [MGS_BLOCK][ORTH_THREADS]
  cplx* sw = red + MGS_BLOCK * ORTH_THREADS;           // [rounds][ORTH_THREADS] this block's w
  __shared__ __align__(16) cplx half_sum[2][MGS_BLOCK * ORTH_MAX_K];
  __shared__ __align__(16) cplx hs[MGS_BLOCK * ORTH_MAX_K];
  __shared__ double hinv[ORTH_MAX_K];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = a.k, G = gridDim.x;
  const int64_t first = (int64_t)blockIdx.x * a.chunk, nk = a.nk;
  const int len = (int)(nk - first < a.chunk ? nk - first : a.chunk);
  const int stride = ORTH_THREADS / k * k;             // a thread's entries are of one right-hand side
  const int begin = tid < stride ? tid : len, rhs = tid % k;
  const int live = len < stride ? len : stride;        // threads with entries
  const int P = 32 / k, lp = lane / k;                 // lanes r + k p < k P share the sums of right-hand side r
  const cplx* V = a.V + first;
  const cplx* w = a.w + first;
  cplx u[MGS_BLOCK], rot = {0.0, 0.0};
  int passes = 0;
  bool ok = true;
  for (int i0 = -MGS_BLOCK; i0 <= a.j; i0 += MGS_BLOCK) {
    const int i1 = i0 + MGS_BLOCK;
    const int nv = i0 < 0 ? 0 : min(a.j + 1 - i0, MGS_BLOCK);
    const int nn = i1 > a.j ? 0 : min(a.j + 1 - i1, MGS_BLOCK);
    cplx acc[MGS_BLOCK];
#pragma unroll
    for (int q = 0; q < MGS_BLOCK; ++q) acc[q] = {0.0, 0.0};
    // the new entries of column j of H through the earlier rotations, beside the pass: rot is the running entry
    if (nv > 0 && blockIdx.x == 0 && warp == ORTH_THREADS / 32 - 1 && lane < k) {
      const double* c = a.cs + (int64_t)lane * a.m;
      const cplx* s = a.sn + (int64_t)lane * a.m;
      double cq[MGS_BLOCK];
      cplx sq[MGS_BLOCK];
#pragma unroll
      for (int q = 0; q < MGS_BLOCK; ++q)
        if (q < nv && i0 + q > 0) {
          cq[q] = c[i0 + q - 1];
          sq[q] = s[i0 + q - 1];
        }
#pragma unroll
      for (int q = 0; q < MGS_BLOCK; ++q)
        if (q < nv) {
          const cplx b = ld16(hs + q * k + lane);
          if (i0 + q == 0) {
            rot = b;
          } else {
            a.H[((int64_t)lane * (a.m + 1) + i0 + q - 1) * a.m + a.j] = cadd(cscale(rot, cq[q]), cmul(sq[q], b));
            rot = csub(cscale(b, cq[q]), cmul(cconj(sq[q]), rot));
          }
        }
    }
    cplx* wp = sw + tid;
    for (int e = begin; e < len; e += stride, wp += ORTH_THREADS) {
      cplx x = ld16(nv > 0 ? wp : w + e);
      if (nv > 0) {
        if (e != begin) {
#pragma unroll
          for (int q = 0; q < MGS_BLOCK; ++q)
            if (q < nv) u[q] = ld16(V + (i0 + q) * nk + e);
        }
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nv) {
            const cplx h = ld16(hs + q * k + rhs);
            x.re = fma(-h.re, u[q].re, x.re);
            x.im = fma(-h.re, u[q].im, x.im);
            x.re = fma(h.im, u[q].im, x.re);
            x.im = fma(-h.im, u[q].re, x.im);
          }
      }
      st16(wp, x);
      if (nn > 0) {
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nn) u[q] = ld16(V + (i1 + q) * nk + e);
#pragma unroll
        for (int q = 0; q < MGS_BLOCK; ++q)
          if (q < nn) {
            acc[q].re = fma(u[q].re, x.re, acc[q].re);
            acc[q].im = fma(u[q].re, x.im, acc[q].im);
            acc[q].re = fma(u[q].im, x.im, acc[q].re);
            acc[q].im = fma(-u[q].im, x.re, acc[q].im);
          }
      } else {
        acc[0].re = fma(x.re, x.re, acc[0].re);
        acc[0].re = fma(x.im, x.im, acc[0].re);
      }
    }
    // the block's sums, one warp a value
    const int nq = nn > 0 ? nn : 1;
#pragma unroll
    for (int q = 0; q < MGS_BLOCK; ++q)
      if (q < nq) st16(red + q * ORTH_THREADS + tid, acc[q]);
    __syncthreads();
    cplx* part = a.partials + (int64_t)(passes & 1) * MGS_BLOCK * G * k;
    if (warp < nq) {
      cplx t = {0.0, 0.0};
      if (lane < k * P)
        for (int i = lane; i < live; i += k * P) t = cadd(t, ld16(red + warp * ORTH_THREADS + i));
      t = sum_lanes(t, k, P, lp);
      if (lane < k) st16(part + ((int64_t)warp * G + blockIdx.x) * k + lane, t);
    }
    if (begin < len) {  // the next pass's first vectors do not depend on the sums
#pragma unroll
      for (int q = 0; q < MGS_BLOCK; ++q)
        if (q < nn) u[q] = ld16(V + (i1 + q) * nk + begin);
    }
    grid_arrive(a.status);
    ++passes;
    ok = grid_wait(a.status, passes * G, a.wait_ns);
    if (!ok) break;
    // all blocks' sums, half of the blocks a warp
    const int q = warp & (MGS_BLOCK - 1), hf = warp >> 3;
    if (q < nq) {
      const cplx* src = part + (int64_t)q * G * k;
      const int end = (hf ? G : G / 2) * k;
      cplx t = {0.0, 0.0};
      if (lane < k * P)
        for (int i = (hf ? G / 2 * k : 0) + lane; i < end; i += 4 * k * P) {
          double2 v[4];
#pragma unroll
          for (int n = 0; n < 4; ++n)
            v[n] = i + n * k * P < end ? __ldcg(reinterpret_cast<const double2*>(src + i + n * k * P)) : make_double2(0.0, 0.0);
#pragma unroll
          for (int n = 0; n < 4; ++n)
            if (i + n * k * P < end) t = cadd(t, {v[n].x, v[n].y});
        }
      t = sum_lanes(t, k, P, lp);
      if (lane < k) half_sum[hf][q * k + lane] = t;
    }
    __syncthreads();
    if (tid < nq * k) {
      const cplx t = cadd(half_sum[0][tid], half_sum[1][tid]);
      hs[tid] = t;
      if (nn == 0) {
        const double h = sqrt(t.re);
        hinv[tid] = h > 0.0 ? 1.0 / h : -1.0;
      }
    }
    __syncthreads();
  }
  if (ok) {  // V_{j+1} = w / |w| (0 where |w| is 0 or not a number)
    const double inv = hinv[rhs];
    const cplx* wp = sw + tid;
    for (int e = begin; e < len; e += stride, wp += ORTH_THREADS) {
      const cplx x = ld16(wp);
      st16(a.Vn + first + e, inv >= 0.0 ? cplx{x.re * inv, x.im * inv} : cplx{0.0, 0.0});
    }
  } else if (tid == 0) {
    atomicExch(&a.status[ST_ERR], DEV_TIMEOUT);
    __threadfence();
  }
  if (blockIdx.x == 0) {
    if (ok && warp == ORTH_THREADS / 32 - 1 && lane < k)
      givens_finish(lane, a.m, a.j, rot, sqrt(hs[lane].re), a.H, a.cs, a.sn, a.g, a.host_res);
    __syncthreads();
    if (tid < 8) a.host_status[tid] = *(volatile int32_t*)&a.status[tid];
  }
  // the last block to leave clears the counters: no block waits any more
  if (tid == 0 && atomicAdd(&a.status[ST_ORTH_LEFT], 1) == G - 1) {
    a.status[ST_ORTH_ARRIVED] = 0;
    a.status[ST_ORTH_LEFT] = 0;
  }
}

// h_{j+1,j} = ||w|| (hs[r] = |w|^2); V_{j+1} = w / h (0 if h == 0).  The last block instead runs the
// Givens update of every RHS beside them: apply rotations 0..j-1 to column j of H, build rotation j, update
// g, res = |g_{j+1}|; res and the device status go straight to the host's pinned words.
__global__ void __launch_bounds__(RED_THREADS) k_mgs_finish(int64_t nk, int k, int m, int j,
                                                            const cplx* __restrict__ w, cplx* __restrict__ Vn,
                                                            const cplx* __restrict__ hs, cplx* __restrict__ H,
                                                            double* __restrict__ cs, cplx* __restrict__ sn,
                                                            cplx* __restrict__ g, double* __restrict__ host_res,
                                                            const int32_t* __restrict__ status,
                                                            int32_t* __restrict__ host_status) {
  if (blockIdx.x + 1 < gridDim.x) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t T = (int64_t)(gridDim.x - 1) * blockDim.x, teff = T / k * k;
    if (t >= teff) return;
    const double h = sqrt(hs[t % k].re), inv = h > 0.0 ? 1.0 / h : 0.0;
    for (int64_t e = t; e < nk; e += teff) {
      const cplx x = ld16(w + e);
      st16(Vn + e, h > 0.0 ? cplx{x.re * inv, x.im * inv} : cplx{0.0, 0.0});
    }
    return;
  }
  if (threadIdx.x < 8) host_status[threadIdx.x] = status[threadIdx.x];
  for (int r = threadIdx.x; r < k; r += blockDim.x) {
    cplx* Hr = H + (int64_t)r * (m + 1) * m;
    double* c = cs + (int64_t)r * m;
    cplx* s = sn + (int64_t)r * m;
    const double bb = sqrt(hs[r].re);
    cplx a = Hr[j];                       // the running entry of column j
    for (int q = 0; q < j; ++q) {
      const cplx b = Hr[(int64_t)(q + 1) * m + j];
      const double cq = c[q];
      const cplx sq = s[q];
      Hr[(int64_t)q * m + j] = cadd(cscale(a, cq), cmul(sq, b));
      a = csub(cscale(b, cq), cmul(cconj(sq), a));
    }
    givens_finish(r, m, j, a, bb, H, cs, sn, g, host_res);
  }
}

// y = H(0:kk,0:kk)^{-1} g(0:kk) per RHS (back substitution), y = 0 for inactive RHS.
__global__ void k_hsolve(int k, int m, int kk, const cplx* __restrict__ H, const cplx* __restrict__ g,
                         const int32_t* __restrict__ active, cplx* __restrict__ y) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= k) return;
  const cplx* Hr = H + (int64_t)r * (m + 1) * m;
  cplx* yr = y + (int64_t)r * m;
  if (!active[r]) {
    for (int q = 0; q < kk; ++q) yr[q] = {0.0, 0.0};
    return;
  }
  for (int q = kk - 1; q >= 0; --q) {
    cplx t = g[(int64_t)r * (m + 1) + q];
    for (int l = q + 1; l < kk; ++l) t = csub(t, cmul(Hr[(int64_t)q * m + l], yr[l]));
    cplx d = Hr[(int64_t)q * m + q];
    double dd = d.re * d.re + d.im * d.im;
    yr[q] = dd > 0.0 ? cplx{(t.re * d.re + t.im * d.im) / dd, (t.im * d.re - t.re * d.im) / dd} : cplx{0.0, 0.0};
  }
}

// x += sum_q y_q Z_q   (Z: [m][N][k])
template <typename ZT>
__global__ void k_xupdate(int64_t nk, int k, int m, int kk, const ZT* __restrict__ Z, const cplx* __restrict__ y,
                          cplx* __restrict__ x) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nk) return;
  int r = (int)(e % k);
  cplx acc = ld16(x + e);
  for (int q = 0; q < kk; ++q) {
    const cplx c = y[(int64_t)r * m + q], v = ld_c<ZT>(Z, (int64_t)q * nk + e);
    acc.re = fma(c.re, v.re, acc.re);
    acc.im = fma(c.re, v.im, acc.im);
    acc.re = fma(-c.im, v.im, acc.re);
    acc.im = fma(c.im, v.re, acc.im);
  }
  st16(x + e, acc);
}

// r = b - A x (SpMV output in r already holds A x): r = b - r; partial |r|^2
__global__ void __launch_bounds__(RED_THREADS) k_residual(int64_t nk, int k, const cplx* __restrict__ b,
                                                          cplx* __restrict__ r, cplx* __restrict__ partials) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, teff = red_teff(k);
  cplx acc[1] = {{0.0, 0.0}};
  if (t < teff)
    for (int64_t e = t; e < nk; e += teff) {
      const cplx v = csub(ld16(b + e), ld16(r + e));
      st16(r + e, v);
      acc[0].re = fma(v.re, v.re, acc[0].re);
      acc[0].re = fma(v.im, v.im, acc[0].re);
    }
  block_reduce_store<1>(acc, 1, k, partials);
}

// norms[r] = sqrt(sum of the nb block partials) (single block)
__global__ void k_norms(int k, int nb, const cplx* __restrict__ partials, double* __restrict__ out) {
  for (int r = threadIdx.x >> 5; r < k; r += blockDim.x >> 5) {  // one warp per right-hand side
    const cplx t = sum_partials_warp(partials + (int64_t)r * nb, nb, threadIdx.x & 31);
    if ((threadIdx.x & 31) == 0) out[r] = sqrt(t.re);
  }
}

// V0 = r / beta for active RHS (0 otherwise); g = (beta, 0, ...)
__global__ void k_restart(int64_t nk, int k, int m, const cplx* __restrict__ rv, const double* __restrict__ beta,
                          const int32_t* __restrict__ active, cplx* __restrict__ V0, cplx* __restrict__ g) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < nk) {
    int q = (int)(e % k);
    double b = beta[q];
    const double inv = 1.0 / b;
    V0[e] = (active[q] && b > 0.0) ? cplx{rv[e].re * inv, rv[e].im * inv} : cplx{0.0, 0.0};
  }
  if (e < k) {
    for (int l = 0; l <= m; ++l) g[(int64_t)e * (m + 1) + l] = {0.0, 0.0};
    g[(int64_t)e * (m + 1)] = {active[e] ? beta[e] : 0.0, 0.0};
  }
}

// column-major host layout [k][N] <-> internal [N][k]
__global__ void k_to_internal(int64_t n, int k, const cplx* __restrict__ src, cplx* __restrict__ dst) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * k) return;
  int64_t g = e / k;
  int r = (int)(e % k);
  st16(dst + e, ld16(src + (int64_t)r * n + g));
}
__global__ void k_to_internal_c64(int64_t n, int k, const CT<float>* __restrict__ src, CT<float>* __restrict__ dst) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * k) return;
  dst[e] = src[(int64_t)(e % k) * n + e / k];
}
__global__ void k_to_external(int64_t n, int k, const cplx* __restrict__ src, cplx* __restrict__ dst) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * k) return;
  int64_t g = e / k;
  int r = (int)(e % k);
  st16(dst + (int64_t)r * n + g, ld16(src + e));
}

// ------------------------------------------------------------------ launchers
// Lanes on right-hand sides for k columns, and the launch of f(KL, blocks, chunks).
template <typename F>
static void spmv_launch(const oras_handle* h, int k, F&& f) {
  const int kl = k >= 5 ? 8 : (k >= 3 ? 4 : k), chunks = (k + kl - 1) / kl;
  const int64_t blocks = (h->mesh.ndof * SPMV_LPR + 255) / 256 * chunks;
  f(kl, (unsigned)blocks, chunks);
  count_launches(1);
}
void launch_spmv_f64(const oras_handle* h, const cplx* x, cplx* y, int k) {
  const auto& d = h->dev;
  spmv_launch(h, k, [&](int kl, unsigned blocks, int chunks) {
    auto* fn = kl == 8 ? k_spmv<cplx, 8> : kl == 4 ? k_spmv<cplx, 4> : kl == 2 ? k_spmv<cplx, 2> : k_spmv<cplx, 1>;
    fn<<<blocks, 256, 0, d.stream>>>(h->mesh.ndof, d.rowptr, d.cols, d.vals, x, y, k, chunks);
  });
}
// complex FP32 x: FP32-pipe kernel with FP64-class accuracy (k_spmv_df)
void launch_spmv_f32(const oras_handle* h, const void* x, cplx* y, int k) {
  const auto& d = h->dev;
  spmv_launch(h, k, [&](int kl, unsigned blocks, int chunks) {
    auto* fn = kl == 8 ? k_spmv_df<8> : kl == 4 ? k_spmv_df<4> : kl == 2 ? k_spmv_df<2> : k_spmv_df<1>;
    fn<<<blocks, 256, 0, d.stream>>>(h->mesh.ndof, d.rowptr, d.cols, d.vals_df, (const CT<float>*)x, y, k, chunks);
  });
}
void launch_split_vals(const oras_handle* h) {
  const int64_t nnz = (int64_t)h->mesh.cols.size();
  k_split_vals<<<(unsigned)((nnz + 255) / 256), 256, 0, h->dev.stream>>>(nnz, h->dev.vals, h->dev.vals_df);
  count_launches(1);
}

// Blocks of the reductions over nk entries: two per SM, fewer for short vectors (at least 512 entries each).
static int red_grid(int64_t nk) {
  const int64_t b = (nk + 2 * RED_THREADS - 1) / (2 * RED_THREADS);
  return (int)(b < 1 ? 1 : (b < RED_BLOCKS ? b : RED_BLOCKS));
}
// Orthogonalisation of w against V_0..V_j ([j + 1][N][k]): column j of H, |w|^2 in hs; partials and hs:
// red_elems(k) entries from `red`.
static void launch_mgs(const oras_handle* h, int k, int m, int j, const cplx* V, cplx* w, cplx* red, cplx* H) {
  const int64_t nk = h->mesh.ndof * k;
  const int grid = red_grid(nk);
  cplx* hs = red;
  cplx* partials = red + (int64_t)MGS_BLOCK * k;
  cudaStream_t st = h->dev.stream;
  for (int i0 = -MGS_BLOCK; i0 <= j; i0 += MGS_BLOCK) {  // the first pass has nothing to subtract
    const int i1 = i0 + MGS_BLOCK;
    const int nv = i0 < 0 ? 0 : (j + 1 - i0 < MGS_BLOCK ? j + 1 - i0 : MGS_BLOCK);
    const int nn = i1 > j ? 0 : (j + 1 - i1 < MGS_BLOCK ? j + 1 - i1 : MGS_BLOCK);
    k_mgs_block<<<grid, RED_THREADS, 0, st>>>(nk, k, nv, V + (i0 < 0 ? 0 : i0) * nk, nn, V + i1 * nk, w, hs, partials);
    const int sums = (nn > 0 ? nn : 1) * k;
    k_sum_partials<<<(sums + 7) / 8, 256, 0, st>>>(nn > 0 ? nn : 1, k, grid, partials, hs, m, i1, j,
                                                   nn > 0 ? H : nullptr);
    count_launches(2);
  }
}
size_t red_elems(int k) { return (size_t)(RED_BLOCKS + 1) * MGS_BLOCK * k; }
static void launch_mgs_finish(const oras_handle* h, int k, int m, int j, const cplx* w, cplx* Vn, const cplx* red,
                       cplx* H, double* cs, cplx* sn, cplx* g, double* host_res, int32_t* host_status) {
  const int64_t nk = h->mesh.ndof * k;
  int64_t blocks = (nk + RED_THREADS - 1) / RED_THREADS;
  if (blocks > 4 * RED_BLOCKS) blocks = 4 * RED_BLOCKS;
  k_mgs_finish<<<(unsigned)blocks + 1, RED_THREADS, 0, h->dev.stream>>>(nk, k, m, j, w, Vn, red, H, cs, sn, g, host_res,
                                                                       h->dev.status, host_status);
  count_launches(1);
}
static bool launch_orth_once(const oras_handle* h, int k, int m, int j, const cplx* V, const cplx* w, cplx* Vn, cplx* red,
                             cplx* H, double* cs, cplx* sn, cplx* g, double* host_res, int32_t* host_status) {
  if (k > ORTH_MAX_K) return false;
  OrthArgs a;
  a.nk = h->mesh.ndof * k;
  const int64_t most = std::max<int64_t>(1, std::min<int64_t>({h->dev.num_sms, RED_BLOCKS / 2, (a.nk + 31) / 32}));
  const int64_t unit = k % 2 ? 2 * k : k;  // whole right-hand side groups, 32-byte sectors
  a.chunk = ((a.nk + most - 1) / most + unit - 1) / unit * unit;
  const int64_t grid = (a.nk + a.chunk - 1) / a.chunk;
  const int64_t stride = ORTH_THREADS / k * k, rounds = (a.chunk + stride - 1) / stride;
  if (rounds > ORTH_MAX_ROUNDS) return false;
  a.k = k; a.m = m; a.j = j;
  a.V = V; a.w = w; a.Vn = Vn; a.partials = red; a.H = H; a.cs = cs; a.sn = sn; a.g = g;
  a.host_res = host_res; a.status = h->dev.status; a.host_status = host_status;
  a.wait_ns = wait_limit_ns(h);
  allow_max_smem((const void*)k_orth);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(ORTH_THREADS);
  cfg.dynamicSmemBytes = (size_t)(MGS_BLOCK + rounds) * ORTH_THREADS * sizeof(cplx);
  cfg.stream = h->dev.stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_orth, a) != cudaSuccess) {  // a device that cannot hold a block an SM at once
    cudaGetLastError();
    return false;
  }
  count_launches(1);
  return true;
}
// The end of Arnoldi step j: w orthogonalised against V_0..V_j, V_{j+1}, column j of H, the rotation and the residual
// estimates in host_res.  `red`: red_elems(k) entries; the status words behind the flags are zero.  Returns its launches.
int launch_orth(const oras_handle* h, int k, int m, int j, const cplx* V, cplx* w, cplx* Vn, cplx* red, cplx* H,
                double* cs, cplx* sn, cplx* g, double* host_res, int32_t* host_status) {
  if (launch_orth_once(h, k, m, j, V, w, Vn, red, H, cs, sn, g, host_res, host_status)) return 1;
  launch_mgs(h, k, m, j, V, w, red, H);
  launch_mgs_finish(h, k, m, j, w, Vn, red, H, cs, sn, g, host_res, host_status);
  return 2 * (j / MGS_BLOCK + 2) + 1;
}
void launch_hsolve(const oras_handle* h, int k, int m, int kk, const cplx* H, const cplx* g, const int32_t* active,
                   cplx* y) {
  k_hsolve<<<1, 64, 0, h->dev.stream>>>(k, m, kk, H, g, active, y);
  count_launches(1);
}
void launch_xupdate_f64(const oras_handle* h, int k, int m, int kk, const cplx* Z, const cplx* y, cplx* x) {
  int64_t nk = h->mesh.ndof * k;
  k_xupdate<cplx><<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(nk, k, m, kk, Z, y, x);
  count_launches(1);
}
void launch_xupdate_f32(const oras_handle* h, int k, int m, int kk, const void* Z, const cplx* y, cplx* x) {
  int64_t nk = h->mesh.ndof * k;
  k_xupdate<CT<float>><<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(nk, k, m, kk, (const CT<float>*)Z, y, x);
  count_launches(1);
}
void launch_residual(const oras_handle* h, int k, const cplx* b, cplx* r, cplx* partials) {
  k_residual<<<red_grid(h->mesh.ndof * k), RED_THREADS, 0, h->dev.stream>>>(h->mesh.ndof * k, k, b, r, partials);
  count_launches(1);
}
void launch_norms(const oras_handle* h, int k, const cplx* partials, double* out) {
  k_norms<<<1, 256, 0, h->dev.stream>>>(k, red_grid(h->mesh.ndof * k), partials, out);
  count_launches(1);
}
void launch_restart(const oras_handle* h, int k, int m, const cplx* rv, const double* beta, const int32_t* active,
                    cplx* V0, cplx* g) {
  int64_t nk = h->mesh.ndof * k;
  k_restart<<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(nk, k, m, rv, beta, active, V0, g);
  count_launches(1);
}
void launch_to_internal_c64(const oras_handle* h, int k, const void* src, void* dst) {
  const int64_t nk = h->mesh.ndof * k;
  k_to_internal_c64<<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(h->mesh.ndof, k, (const CT<float>*)src,
                                                                            (CT<float>*)dst);
  count_launches(1);
}
void launch_to_internal(const oras_handle* h, int k, const cplx* src, cplx* dst) {
  int64_t nk = h->mesh.ndof * k;
  k_to_internal<<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(h->mesh.ndof, k, src, dst);
  count_launches(1);
}
void launch_to_external(const oras_handle* h, int k, const cplx* src, cplx* dst) {
  int64_t nk = h->mesh.ndof * k;
  k_to_external<<<(unsigned)((nk + 255) / 256), 256, 0, h->dev.stream>>>(h->mesh.ndof, k, src, dst);
  count_launches(1);
}

}  // namespace oras
