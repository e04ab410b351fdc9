// Panel and contribution products of the sparse local factorisation (fronts.cu) on the tcgen05 tensor cores,
// FP32 factors:
//   L = A21 S                       (S symmetric, so both products are A B^T over the own unknowns)
//   C = pulled children - L A21^T   (tiles that reach the diagonal or lie below it)
// The complex sum runs over interleaved (re, im) pairs: row i of A as it is stored, against two real rows
// for every row j of B, (re, -im) for the real part of the result and (im, re) for the imaginary part.
//
// Precision: each FP32 operand is split into two TF32 values (2^-23 of it is left out) and hi hi, hi lo and lo hi are
// summed in FP32 in tensor memory, the two small products in an accumulator of their own.  The apply's error against
// FP64 is then that of FP32 fused multiply-adds in their place: 0.92e-6 to 1.0e-6 against 0.86e-6 to 0.98e-6 on a problem
// of degree 2, 1.72e-6 to 1.84e-6 against 1.82e-6 to 1.87e-6 on one of degree 3 (one accumulator for all three: 1.03e-6
// and 1.95e-6; lo lo as well: no change).  fronts.cu has the errors on more problems.
//
// A block owns 128 x 64 entries (256 accumulator columns) and walks the sum in chunks of 16 unknowns: all
// threads load, split and store a chunk in the 128-byte-swizzled K-major layout of the operands, one thread
// issues its 12 MMAs.  The sums are short (128 unknowns at most) and the operands are split anew in every tile, so
// the bound is the issue of those loads, splits and stores (half of the issue slots) and their latency, not the tensor
// cores; one chunk buffer of 64 KB lets two blocks share an SM, one's loads and stores beside the other's MMAs.
// The result goes through shared memory, so C is written and the children's blocks are read along rows, the reads of 4
// rows in flight together.
//
// 16^3 x 6, degree 2, 64 subdomains, all levels: L 4.5 -> 1.7 ms, C 8.5 -> 4.1 ms against 64 x 64 tiles of FP32 fused
// multiply-adds; 9^3 x 6, degree 3: 2.1 -> 0.82 and 3.9 -> 2.0 ms.
#include "fronts.cuh"

namespace oras {

constexpr int FT_THREADS = 256;
constexpr int FT_ROWS = 128, FT_COLS = 64;               // tile (also in fronts_plan.cpp: FR_TC_ROWS)
constexpr uint32_t FT_OPERAND = 128 * 128;               // 128 rows of 32 floats
constexpr int FT_LDD = FT_COLS + 1;                      // row stride of the result tile
constexpr size_t FT_SMEM = (size_t)FT_ROWS * FT_LDD * sizeof(CT<float>) + 1024;
static_assert(4 * FT_OPERAND + 1024 <= FT_SMEM, "the operands fit in the result tile");
static_assert(FT_ROWS == FR_TC_ROWS && FT_COLS == FR_TILE, "tiles of the plan");
constexpr uint32_t FT_TMEM = 256;   // re and im of the 64 columns: leading products, then the corrections

// K-major operand, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t ft_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// kind::tf32, D = F32, A = B = TF32, both K-major, M = 128, N = 128
constexpr uint32_t FT_IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void ft_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
      ::"r"(d), "l"(a), "l"(b), "r"(FT_IDESC), "r"(acc));
}

// 32 accumulator columns of this thread's lane.
__device__ __forceinline__ void ft_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

// x = hi + lo + (2^-23 of x), hi the nearest TF32 value (10 mantissa bits, ties away from zero), lo the remainder cut
// to TF32.  A NaN may round away in hi: it stays in lo.
__device__ __forceinline__ void tf32_split(float x, float& hi, float& lo) {
  hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
  lo = __uint_as_float(__float_as_uint(x - hi) & 0xFFFFE000u);
}

template <bool SCHUR>
__global__ void __launch_bounds__(FT_THREADS, 2) k_fr_mul_tc(FrDev f, const FrontItem* __restrict__ items,
                                                             const CT<float>* __restrict__ work, CT<float>* fac,
                                                             CT<float>* C, int32_t* status, uint64_t wait_ns) {
  extern __shared__ __align__(1024) unsigned char ft_raw[];
  __shared__ uint64_t bar;
  __shared__ uint32_t tmem_base;
  unsigned char* sm = (unsigned char*)(((uintptr_t)ft_raw + 1023) & ~(uintptr_t)1023);
  const FrontItem it = items[blockIdx.x];
  const FrontNode n = f.nodes[it.node];
  const int n1 = n.n1, n2 = n.n2, ld = n.ld;
  const int i0 = (it.t >> 16) * FT_ROWS, j0 = (it.t & 0xFFFF) * FT_COLS;
  const int jn = SCHUR ? n2 : n1;
  const CT<float>* A = (SCHUR ? fac : work) + n.panel + (int64_t)n1 * ld;
  const CT<float>* B = SCHUR ? work + n.panel + (int64_t)n1 * ld : fac + n.panel;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int chunks = (ld + 15) / 16;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(FT_TMEM));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = tmem_base;
  // a chunk: 16-byte granule g (two unknowns) of row r; this thread rows tid / 8 + 32 q, granule tid % 8
  const int g = tid & 7, r0 = tid >> 3;
  float4 av[4], bv[2];
  auto load = [&](int c) {
    const int k = c * 16 + 2 * g;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + r0 + 32 * q;
      av[q] = (i < n2 && k < ld) ? *reinterpret_cast<const float4*>(A + (int64_t)i * ld + k) : make_float4(0, 0, 0, 0);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = j0 + r0 + 32 * q;
      bv[q] = (j < jn && k < ld) ? *reinterpret_cast<const float4*>(B + (int64_t)j * ld + k) : make_float4(0, 0, 0, 0);
    }
  };
  auto put = [&](uint32_t operand, int r, float4 v) {
    *reinterpret_cast<float4*>(sm + operand * FT_OPERAND + (r >> 3) * 1024 + (r & 7) * 128 + ((g ^ (r & 7)) << 4)) = v;
  };
  bool bad = false;
  int issued = -1;  // thread 0: the last chunk whose MMAs are under way
  if (chunks > 0) load(0);
  for (int c = 0; c < chunks; ++c) {
    // the MMAs of the chunk before have read the buffer
    const bool ok = c == 0 || mbar_wait(&bar, (uint32_t)((c - 1) & 1), false, wait_ns);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4 h, l;
      tf32_split(av[q].x, h.x, l.x);
      tf32_split(av[q].y, h.y, l.y);
      tf32_split(av[q].z, h.z, l.z);
      tf32_split(av[q].w, h.w, l.w);
      put(0, r0 + 32 * q, h);
      put(1, r0 + 32 * q, l);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float4 h, l;
      tf32_split(bv[q].x, h.x, l.x);
      tf32_split(bv[q].y, h.y, l.y);
      tf32_split(bv[q].z, h.z, l.z);
      tf32_split(bv[q].w, h.w, l.w);
      put(2, r0 + 32 * q, make_float4(h.x, -h.y, h.z, -h.w));
      put(3, r0 + 32 * q, make_float4(l.x, -l.y, l.z, -l.w));
      put(2, 64 + r0 + 32 * q, make_float4(h.y, h.x, h.w, h.z));
      put(3, 64 + r0 + 32 * q, make_float4(l.y, l.x, l.w, l.z));
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (c + 1 < chunks) load(c + 1);
    bad = __syncthreads_or(!ok) != 0;
    if (bad) break;
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sb = smem_u32(sm);
      const uint64_t ah = ft_desc(sb), al = ft_desc(sb + FT_OPERAND);
      const uint64_t bh = ft_desc(sb + 2 * FT_OPERAND), bl = ft_desc(sb + 3 * FT_OPERAND);
#pragma unroll
      for (int k8 = 0; k8 < 4; ++k8) {  // K = 8 floats = 32 B per instruction
        const uint64_t dk = (uint64_t)(k8 * 32) >> 4;
        const uint32_t acc = (c == 0 && k8 == 0) ? 0u : 1u;
        ft_mma(tbase + 128, al + dk, bh + dk, acc);
        ft_mma(tbase + 128, ah + dk, bl + dk, 1u);
        ft_mma(tbase, ah + dk, bh + dk, acc);
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&bar))
                   : "memory");
      issued = c;
    }
  }
  if (!bad && chunks > 0) bad = __syncthreads_or(!mbar_wait(&bar, (uint32_t)((chunks - 1) & 1), false, wait_ns)) != 0;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (bad) {  // no MMA is issued after a wait that gave up; those in flight get more time to finish
    if (tid == 0) {
      atomicExch(&status[ST_ERR], DEV_TIMEOUT);
      if (issued >= 0) mbar_wait(&bar, (uint32_t)(issued & 1), false, drain_limit(wait_ns));
    }
  } else {
    // lanes 32 (warp % 4) .. + 31 are the tile's rows; warps 0-3 take columns 0-31, warps 4-7 columns 32-63
    CT<float>* D = reinterpret_cast<CT<float>*>(sm);
    const int half = warp >> 2, row = (warp & 3) * 32 + lane;
    if (chunks > 0) {
      const uint32_t t = tbase + ((uint32_t)((warp & 3) * 32) << 16) + half * 32;
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        float v[32], low[32];
        ft_ld32(t + 64 * part, v);
        ft_ld32(t + 64 * part + 128, low);
        float* out = &D[row * FT_LDD + half * 32].re + part;
#pragma unroll
        for (int q = 0; q < 32; ++q) out[2 * q] = v[q] + low[q];
      }
    } else {
      for (int q = 0; q < 32; ++q) D[row * FT_LDD + half * 32 + q] = {0.0f, 0.0f};
    }
    __syncthreads();
    if (SCHUR) {
      // this warp's rows warp + 8 t, their sources in lane t; columns lane and lane + 32
      constexpr int NW = FT_THREADS / 32, RW = FT_ROWS / NW, BATCH = 4;
      const int my = i0 + warp + NW * lane;
      const FrontSrc sr = lane < RW && my < n2 ? f.border_src[n.bord + my] : FrontSrc{-1, -1};
      const CT<float>* cp[2] = {C, C};
      int64_t ldc[2] = {0, 0}, bord[2] = {0, 0};
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (n.child[q] >= 0) {
          const FrontNode& c = f.nodes[n.child[q]];
          cp[q] += c.cblk;
          ldc[q] = c.ldc;
          bord[q] = c.bord;
        }
      FrontSrc sj[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int j = j0 + lane + 32 * q;
        sj[q] = j < n2 ? f.border_src[n.bord + j] : FrontSrc{-1, -1};
      }
#pragma unroll 1
      for (int t0 = 0; t0 < RW; t0 += BATCH) {  // a batch's loads are in flight together
        CT<float> va[BATCH][2], vb[BATCH][2];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
          const int i = i0 + warp + NW * (t0 + u);
          const int sa = __shfl_sync(0xffffffffu, sr.a, t0 + u), sb = __shfl_sync(0xffffffffu, sr.b, t0 + u);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const bool on = i < n2 && j0 + lane + 32 * q <= i;
            va[u][q] = vb[u][q] = {0.0f, 0.0f};
            // both borders ascend, so sa >= sj[q].a: a lower entry of the child's block
            if (on && sa >= 0 && sj[q].a >= 0) va[u][q] = cp[0][(sa - bord[0]) * ldc[0] + sj[q].a - bord[0]];
            if (on && sb >= 0 && sj[q].b >= 0) vb[u][q] = cp[1][(sb - bord[1]) * ldc[1] + sj[q].b - bord[1]];
          }
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
          const int r = warp + NW * (t0 + u), i = i0 + r;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int j = j0 + lane + 32 * q;
            if (i >= n2 || j > i) continue;  // above the diagonal: not kept
            const CT<float> d = D[r * FT_LDD + lane + 32 * q];
            C[n.cblk + (int64_t)i * n.ldc + j] = {va[u][q].re + vb[u][q].re - d.re, va[u][q].im + vb[u][q].im - d.im};
          }
        }
      }
    } else {
      bool weak = false;
      for (int r = warp; r < FT_ROWS; r += FT_THREADS / 32) {
        const int i = i0 + r;
        if (i >= n2) break;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int j = j0 + lane + 32 * q;
          const CT<float> v = D[r * FT_LDD + lane + 32 * q];
          if (j >= ld) continue;
          fac[n.panel + (int64_t)(n1 + i) * ld + j] = v;  // zeros past n1
          weak |= grown(v.re, v.im);
        }
      }
      if (weak) mark_weak(f, it.node, status);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(FT_TMEM));
}

void launch_front_mul_tc(const oras_handle* h, const FrDev& f, bool schur, const FrontItem* items, int64_t blocks) {
  const auto& d = h->dev;
  allow_max_smem((const void*)k_fr_mul_tc<true>);
  allow_max_smem((const void*)k_fr_mul_tc<false>);
  auto* fn = schur ? k_fr_mul_tc<true> : k_fr_mul_tc<false>;
  fn<<<(unsigned)blocks, FT_THREADS, FT_SMEM, d.stream>>>(f, items, (const CT<float>*)d.fr_work, (CT<float>*)d.arena,
                                                          (CT<float>*)d.fr_c, d.status, wait_limit_ns(h));
  count_launches(1);
}

}  // namespace oras
