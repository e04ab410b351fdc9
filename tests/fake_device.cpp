// A stand-in for the CUDA runtime and for the kernel launchers, so that the host code of the library (api.cpp and
// what it needs) runs on a machine without a GPU: "device" memory is host memory, allocations can be refused, and
// a launcher stands for its kernels by writing all of every buffer that they use.  A buffer that is missing ends the
// program with a message; one that is too small is found by its guard bytes.
//
// usage: fake_device <scenario>; prints one line a finding, exits 0 when there is none.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "internal.h"

using namespace oras;

// ------------------------------------------------------------------ memory
static std::map<void*, size_t> g_live;       // allocation -> bytes (guard bytes follow)
static int64_t g_count = 0, g_refuse_from = -1;
constexpr size_t GUARD = 64;

static int g_bad = 0;
static void bad(const std::string& what) {
  std::printf("%s\n", what.c_str());
  ++g_bad;
}
// Every byte of p, which has to be an allocation of exactly or at least `bytes`.
static void touch(const char* name, const void* p, size_t bytes) {
  auto it = g_live.find(const_cast<void*>(p));
  if (it == g_live.end()) {
    std::printf("a launch uses %s, which is not allocated\n", name);
    std::exit(3);
  }
  if (it->second < bytes) {
    std::printf("a launch uses %zu bytes of %s, which has %zu\n", bytes, name, it->second);
    std::exit(3);
  }
  std::memset(const_cast<void*>(p), 0, bytes);
}

extern "C" {
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  if (g_refuse_from >= 0 && g_count >= g_refuse_from) return cudaErrorMemoryAllocation;
  ++g_count;
  *p = std::malloc(n + GUARD);
  std::memset((char*)*p + n, 0x5A, GUARD);
  g_live[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  auto it = g_live.find(p);
  if (it == g_live.end()) { bad("a pointer is freed that is not allocated"); return cudaErrorInvalidValue; }
  for (size_t q = 0; q < GUARD; ++q)
    if (((unsigned char*)p)[it->second + q] != 0x5A) { bad("written past an allocation"); break; }
  std::free(p);
  g_live.erase(it);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { return cudaFreeAsync(p, nullptr); }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (!d) return cudaErrorInvalidValue;
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { *p = nullptr; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0.0f; return cudaSuccess; }
}

// ------------------------------------------------------------------ launchers
namespace oras { size_t apply_yglob_bytes_for(const oras_handle* h, int k); }
static size_t entry(const oras_handle* h) { return h->opt.factor_bits == 64 ? 16 : 8; }
static void touch_apply(const oras_handle* h, int k) {
  const auto& f = h->fronts;
  touch("the factors", h->dev.arena, (size_t)f.panel_elems * entry(h));
  touch("the apply's vectors", h->dev.ybuf, (size_t)(2 * h->mesh.sub_ns_off[h->mesh.nsub] + f.border_elems) * entry(h) * k);
}

namespace oras {
int launch_element(const oras_handle* h, double) {
  touch("the element matrices", h->dev.elem, (size_t)h->mesh.nt * h->mesh.nl * h->mesh.nl * 16);
  return 0;
}
int launch_faces(const oras_handle* h) {
  touch("the face matrices", h->dev.fmat, (size_t)h->mesh.nif * h->mesh.nfl * h->mesh.nfl * 8);
  return 0;
}
int launch_global_rows(const oras_handle* h, double) {
  touch("A", h->dev.vals, h->mesh.cols.size() * 16);
  return 0;
}
void launch_split_vals(const oras_handle* h) { touch("A in FP32 pairs", h->dev.vals_df, h->mesh.cols.size() * 16); }
int launch_front_rows(const oras_handle* h, double) {
  touch("the assembly workspace", h->dev.fr_work, (size_t)h->fronts.panel_elems * entry(h));
  return 0;
}
int launch_front_factor(oras_handle* h) {
  touch("the assembly workspace", h->dev.fr_work, (size_t)h->fronts.panel_elems * entry(h));
  touch("the factors", h->dev.arena, (size_t)h->fronts.panel_elems * entry(h));
  touch("the contribution blocks", h->dev.fr_c, (size_t)h->fronts.c_elems * entry(h));
  touch("the vectors of the allocation-free apply", h->dev.y1, apply_yglob_bytes_for(h, 1));
  return 0;
}
int launch_local_rows(const oras_handle* h, double) {
  touch("the dense factors", h->dev.arena, (size_t)h->mesh.arena_tiles * TB * TB * entry(h));
  return 0;
}
int lu_max_chunks(int64_t, int) { return 4; }
int launch_lu(oras_handle* h) {
  const auto& d = h->dev;
  const size_t nsub = h->mesh.nsub, slots = 2 * d.lu_max_chunks + 16;
  touch("the dense factors", d.arena, (size_t)h->mesh.arena_tiles * TB * TB * entry(h));
  touch("the tournament's candidates", d.lu_cand, nsub * slots * TB * 4);
  touch("the tournament's counters", d.lu_cnt, nsub * slots * 4);
  touch("the interchanges", d.lu_ipiv, nsub * (2 * TB * 2 + 1) * 4);
  touch("the diagonal tiles", d.lu_diag, nsub * TB * TB * entry(h));
  size_t blocks = 0;
  for (size_t s = 0; s < nsub; ++s) blocks += h->mesh.sub_np[s] / TB;
  touch("the inverted diagonal blocks", d.dinv, blocks * 2 * TB * TB * entry(h));
  if (!d.sub_inv_off) bad("no offsets of the inverted diagonal blocks");
  return 0;
}
int plan_apply_groups(const oras_handle*, int, std::vector<int32_t>&) { return 0; }
int apply_passes(const oras_handle*, int) { return 1; }
static int kr(const oras_handle* h, int k) { return h->opt.factor_bits == 64 ? (k > 1 ? 2 : 1) : (k > 2 ? 4 : k); }
size_t apply_yglob_bytes_for(const oras_handle* h, int k) {
  return (size_t)(2 * h->mesh.sub_ns_off[h->mesh.nsub] + h->fronts.border_elems) * entry(h) * kr(h, k);
}
int launch_apply_f64out(const oras_handle* h, const cplx*, cplx*, int k) { touch_apply(h, kr(h, k)); return 0; }
int launch_apply_f32out(const oras_handle* h, const cplx*, void*, int k) { touch_apply(h, kr(h, k)); return 0; }
size_t red_elems(int k) { return (size_t)305 * 8 * k; }
void launch_mask_fixed(const oras_handle*, cplx*, int) {}
void launch_to_internal(const oras_handle* h, int k, const cplx*, cplx* dst) {
  touch("the right-hand sides", dst, (size_t)h->mesh.ndof * k * 16);
}
void launch_to_external(const oras_handle*, int, const cplx*, cplx*) {}
// The start of a solve: all of the Krylov workspace of k columns.
void launch_residual(const oras_handle* h, int k, const cplx*, cplx*, cplx*) {
  const auto& d = h->dev;
  const size_t nk = (size_t)h->mesh.ndof * k, m = h->opt.restart;
  touch("V", d.V, nk * (m + 1) * 16);
  if (h->opt.factor_bits == 64) touch("Z", d.Zd, nk * m * 16);
  else touch("Z", d.Zf, nk * m * 8);
  for (const cplx* v : {d.w, d.xk, d.bk, d.tmp}) touch("a Krylov vector", v, nk * 16);
  touch("H", d.H, k * (m + 1) * m * 16);
  touch("the rotations", d.gcs, k * m * 8);
  touch("the rotations", d.gsn, k * m * 16);
  touch("g", d.g, k * (m + 1) * 16);
  touch("the partial sums", d.red, red_elems(k) * 16);
  touch("the scalars", d.scal, (k * 8 + k * m * 2 + 64) * 8);
  touch_apply(h, kr(h, k));
}
void launch_norms(const oras_handle*, int k, const cplx*, double* out) {  // |b| = 0: the solve ends there
  for (int r = 0; r < k; ++r) out[r] = 0.0;
}
}  // namespace oras

// ------------------------------------------------------------------ the unit cube in n^3 x 6 tetrahedra
struct Cube {
  std::vector<double> xyz;
  std::vector<int32_t> tets;
  std::vector<oras_complex> eps;
  oras_problem p{};
  Cube(int n, int r, int nsub) {
    const int m = n + 1, perm[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    for (int k = 0; k < m; ++k)
      for (int j = 0; j < m; ++j)
        for (int i = 0; i < m; ++i)
          for (double c : {double(i), double(j), double(k)}) xyz.push_back(c / n);
    const int step[3] = {1, m, m * m};
    for (int k = 0; k < n; ++k)
      for (int j = 0; j < n; ++j)
        for (int i = 0; i < n; ++i)
          for (auto& q : perm) {
            int v = i + m * (j + m * k);
            tets.push_back(v);
            for (int a : q) tets.push_back(v += step[a]);
          }
    eps.assign(tets.size() / 4, {44.0, -20.0});
    p.nv = m * m * m; p.xyz = xyz.data();
    p.nt = (int64_t)eps.size(); p.tets = tets.data();
    p.eps_r = eps.data(); p.k0 = 1.85;
    p.r = r; p.nsub = nsub; p.overlap = 1;
  }
};

static std::string at(const char* what, int64_t n, int rc) {
  return std::string(what) + " (allocation " + std::to_string(n) + " refused, code " + std::to_string(rc) + ")";
}

// oras_factor with every allocation from the n-th on refused, then again with memory, for every n.
static void factor_again(int bits, int engine) {
  Cube c(3, 2, 4);
  oras_options o{};
  o.factor_bits = bits;
  o.lu_engine = engine;
  for (int64_t n = 0;; ++n) {
    oras_handle* h = nullptr;
    if (oras_create(&c.p, &o, &h) != ORAS_OK) { bad("oras_create failed"); return; }
    g_count = 0;
    g_refuse_from = n;
    int rc = oras_factor(h, c.eps.data(), nullptr, c.p.k0, ORAS_MEM_HOST);
    g_refuse_from = -1;
    const bool refused = rc != ORAS_OK;
    if (refused && rc != ORAS_ERR_OUT_OF_MEMORY) bad(at("not reported as out of memory", n, rc));
    if (refused && (rc = oras_factor(h, c.eps.data(), nullptr, c.p.k0, ORAS_MEM_HOST)) != ORAS_OK)
      bad(at("oras_factor fails with memory again", n, rc));
    oras_destroy(h);
    if (!g_live.empty()) bad(at("memory left after oras_destroy", n, rc));
    if (!refused) return;
  }
}

// oras_setup with every allocation from the n-th on refused, for every n: nothing is left behind.
static void setup_fails(int engine) {
  Cube c(2, 1, 2);
  oras_options o{};
  o.lu_engine = engine;
  for (int64_t n = 0;; ++n) {
    oras_handle* h = nullptr;
    g_count = 0;
    g_refuse_from = n;
    const int rc = oras_setup(&c.p, &o, &h);
    g_refuse_from = -1;
    if (rc == ORAS_OK) { oras_destroy(h); break; }
    if (rc != ORAS_ERR_OUT_OF_MEMORY) bad(at("not reported as out of memory", n, rc));
    if (!g_live.empty()) bad(at("memory left after a set-up that failed", n, rc));
    while (!g_live.empty()) cudaFreeAsync(g_live.begin()->first, nullptr);
  }
}

// A solve of more columns with every allocation from the n-th on refused, then one of as many as before.
static void solve_again(int bits) {
  Cube c(3, 2, 4);
  oras_options o{};
  o.factor_bits = bits;
  o.restart = 5;
  for (int64_t n = 0;; ++n) {
    oras_handle* h = nullptr;
    if (oras_create(&c.p, &o, &h) != ORAS_OK || oras_factor(h, c.eps.data(), nullptr, c.p.k0, ORAS_MEM_HOST) != ORAS_OK) {
      bad("set-up failed");
      return;
    }
    std::vector<oras_complex> b((size_t)oras_ndof(h) * 3), x(b.size());
    int rc = oras_solve(h, b.data(), 2, 1e-8, x.data(), nullptr, ORAS_MEM_HOST);
    if (rc != ORAS_OK) bad(at("the first solve fails", n, rc));
    g_count = 0;
    g_refuse_from = n;
    rc = oras_solve(h, b.data(), 3, 1e-8, x.data(), nullptr, ORAS_MEM_HOST);
    g_refuse_from = -1;
    const bool refused = rc != ORAS_OK;
    if (refused && rc != ORAS_ERR_OUT_OF_MEMORY) bad(at("not reported as out of memory", n, rc));
    for (int k : {2, 3})
      if ((rc = oras_solve(h, b.data(), k, 1e-8, x.data(), nullptr, ORAS_MEM_HOST)) != ORAS_OK)
        bad(at("oras_solve fails with memory again", n, rc));
    oras_destroy(h);
    if (!g_live.empty()) bad(at("memory left after oras_destroy", n, rc));
    if (!refused) return;
  }
}

int main(int argc, char** argv) {
  const std::string s = argc > 1 ? argv[1] : "";
  if (s == "factor32") factor_again(32, ORAS_LU_AUTO);
  else if (s == "factor64") factor_again(64, ORAS_LU_AUTO);
  else if (s == "factor_dense") factor_again(32, ORAS_LU_CUDA_CORES);
  else if (s == "setup") setup_fails(ORAS_LU_AUTO);
  else if (s == "setup_dense") setup_fails(ORAS_LU_CUDA_CORES);
  else if (s == "solve32") solve_again(32);
  else if (s == "solve64") solve_again(64);
  else bad("unknown scenario");
  return g_bad ? 1 : 0;
}
