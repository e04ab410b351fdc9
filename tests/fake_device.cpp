// A stand-in for the CUDA runtime and for the kernel launchers, so that the host code of the library (api.cpp and
// what it needs) runs on a machine without a GPU: "device" memory is host memory, allocations can be refused, and
// a launcher stands for its kernels by writing all of every buffer that they use.  A buffer that is missing ends the
// program with a message; one that is too small is found by its guard bytes.
//
// usage: fake_device <scenario>; prints one line a finding, exits 0 when there is none.
#include <algorithm>
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
// What the factorisations find: nodes that should not eliminate their first unknown, in the first g_weak of them.
static int g_weak = 0;
static void plan_is_there(const oras_handle* h) {
  const auto& f = h->fronts;
  const auto& d = h->dev;
  auto same = [](const char* what, const void* dev, const auto& host) {
    auto it = g_live.find(const_cast<void*>(dev));
    const size_t bytes = host.size() * sizeof(host[0]);
    if (it == g_live.end() || it->second < bytes || (bytes && std::memcmp(dev, host.data(), bytes))) {
      std::printf("a launch uses %s, which is not the plan's\n", what);
      std::exit(3);
    }
  };
  same("nodes", d.fr_nodes, f.nodes);
  same("borders", d.fr_border, f.border);
  same("sources", d.fr_own_src, f.own_src);
  same("sources", d.fr_border_src, f.border_src);
  same("positions", d.fr_pos, f.pos);
  same("row nodes", d.fr_row_node, f.row_node);
  same("row unknowns", d.fr_row_dof, f.row_dof);
  same("row weights", d.fr_row_pou, f.row_pou);
  same("blocks", d.fr_bwd_multi, f.bwd_multi.items);
}
int launch_front_rows(const oras_handle* h, double) {
  plan_is_there(h);
  touch("the assembly workspace", h->dev.fr_work, (size_t)h->fronts.panel_elems * entry(h));
  return 0;
}
int launch_front_factor(oras_handle* h) {
  touch("the assembly workspace", h->dev.fr_work, (size_t)h->fronts.panel_elems * entry(h));
  touch("the factors", h->dev.arena, (size_t)h->fronts.panel_elems * entry(h));
  touch("the contribution blocks", h->dev.fr_c, (size_t)h->fronts.c_elems * entry(h));
  touch("the vectors of the allocation-free apply", h->dev.y1, apply_yglob_bytes_for(h, 1));
  for (size_t g = 0; g < h->fronts.nodes.size(); ++g)
    if (h->dev.fr_weak[g]) { bad("a factorisation starts with marks"); break; }
  if (g_weak > 0) {
    --g_weak;
    for (size_t g = 0; g < h->fronts.nodes.size(); g += 3) {
      const FrontNode& n = h->fronts.nodes[g];
      if (n.n1 == 0 || n.n2 == 0) continue;
      auto put = [&](int i, int j, float v) {  // identity, but for a small pivot that couples to the border
        if (h->opt.factor_bits == 64) ((cplx*)h->dev.fr_work)[n.panel + (int64_t)i * n.ld + j] = {v, 0.0};
        else ((float*)h->dev.fr_work)[2 * (n.panel + (int64_t)i * n.ld + j)] = v;
      };
      for (int i = 0; i < n.n1; ++i) put(i, i, i == 0 ? 1e-6f : 1.0f);
      put(n.n1, 0, 1.0f);
      h->dev.fr_weak[g] = 1;
      h->dev.status[ST_WEAK] = 1;
    }
  }
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

// The trees of a handle: every local unknown in one node, what a node hands up is in its parent's front, and
// unknowns that share a tetrahedron are in the front of the one that is eliminated first.  Non-zero: a finding.
static int check_trees(const oras_handle* h) {
  const auto& m = h->mesh;
  const auto& f = h->fronts;
  const int before = g_bad;
  std::vector<int> seen(m.sub_ns_off[m.nsub], 0);
  std::vector<int32_t> level(f.nodes.size());
  for (int l = 0; l < f.nlev(); ++l)
    for (int32_t g = f.level_ptr[l]; g < f.level_ptr[l + 1]; ++g) level[g] = l;
  auto front = [&](int32_t g) {
    const FrontNode& n = f.nodes[g];
    std::vector<int32_t> v;
    for (int i = 0; i < n.n1; ++i) v.push_back(n.row0 + i);
    v.insert(v.end(), f.border.begin() + n.bord, f.border.begin() + n.bord + n.n2);
    return v;
  };
  for (size_t g = 0; g < f.nodes.size(); ++g) {
    const FrontNode& n = f.nodes[g];
    if (n.n1 > front_nb(h->opt.factor_bits)) bad("a pivot block is too wide");
    for (int i = 0; i < n.n1; ++i) {
      ++seen[n.row0 + i];
      if (f.row_node[n.row0 + i] != (int32_t)g) bad("a row's node is wrong");
    }
    const auto mine = front((int32_t)g);
    if (!std::is_sorted(mine.begin(), mine.end())) bad("a front does not ascend");
    for (int q = 0; q < 2; ++q) {
      if (n.child[q] < 0) continue;
      if (level[n.child[q]] >= level[g]) bad("a child is not below its parent");
      const FrontNode& c = f.nodes[n.child[q]];
      std::vector<int> used(c.n2, 0);
      for (int i = 0; i < n.n1 + n.n2; ++i) {
        const FrontSrc s = i < n.n1 ? f.own_src[n.row0 + i] : f.border_src[n.bord + i - n.n1];
        const int32_t at = q == 0 ? s.a : s.b;
        if (at < 0) continue;
        if (at < c.bord || at >= c.bord + c.n2 || f.border[at] != mine[i]) bad("a source is wrong");
        else ++used[at - c.bord];
      }
      for (int u : used)
        if (u != 1) bad("a border entry is not handed up once");
    }
  }
  for (int v : seen)
    if (v != 1) { bad("an unknown is not eliminated once"); break; }
  for (int s = 0; s < m.nsub; ++s) {
    const int64_t off = m.sub_ns_off[s];
    const int32_t* Ns = m.sub_dofs.data() + off;
    for (int64_t q = m.sub_nt_off[s]; q < m.sub_nt_off[s + 1]; ++q) {
      std::vector<int32_t> p;
      for (int a = 0; a < m.nl; ++a)
        p.push_back((int32_t)(off + f.pos[off + (std::lower_bound(Ns, Ns + m.sub_ns[s], m.dofmap[(int64_t)m.sub_tets[q] * m.nl + a]) - Ns)]));
      for (int32_t u : p) {
        const auto v = front(f.row_node[u]);
        for (int32_t w : p)
          if (w > u && !std::binary_search(v.begin(), v.end(), w)) { bad("a coupling has no place"); return 1; }
      }
    }
  }
  return g_bad != before;
}

// Unknowns of random nodes moved up, again and again: the trees stay trees, full nodes pass them on, roots grow.
static void delay(int n, int r, int nsub, int bits) {
  Cube c(n, r, nsub);
  oras_options o{};
  o.factor_bits = bits;
  oras_handle* h = nullptr;
  if (oras_create(&c.p, &o, &h) != ORAS_OK) { bad("oras_create failed"); return; }
  check_trees(h);
  uint32_t seed = 12345;
  auto rnd = [&]() { return (seed = seed * 1664525u + 1013904223u) >> 8; };
  const int levels = h->fronts.nlev();
  for (int round = 0; round < 6 && !g_bad; ++round) {
    std::vector<std::vector<int32_t>> moves(h->fronts.nodes.size());
    for (size_t g = 0; g < moves.size(); ++g) {
      const FrontNode& x = h->fronts.nodes[g];
      if (x.n2 == 0 || x.n1 == 0 || rnd() % 3) continue;
      const int first = rnd() % x.n1, count = round == 5 ? x.n1 : 1 + rnd() % 3;  // at last whole nodes
      for (int i = 0; i < count && i < x.n1; ++i) moves[g].push_back((first + i) % x.n1);
    }
    delay_unknowns(h->mesh, bits, moves, h->fronts);
    check_trees(h);
  }
  if (h->fronts.nlev() <= levels) bad("no root grew: the scenario is too small");
  oras_destroy(h);
}

// oras_factor with every allocation from the n-th on refused, then again with memory, for every n.
static void factor_again(int bits, int engine, int weak = 0) {
  Cube c(3, 2, 4);
  oras_options o{};
  o.factor_bits = bits;
  o.lu_engine = engine;
  for (int64_t n = 0;; ++n) {
    oras::g_weak = weak;
    oras_handle* h = nullptr;
    if (oras_create(&c.p, &o, &h) != ORAS_OK) { bad("oras_create failed"); return; }
    g_count = 0;
    g_refuse_from = n;
    int rc = oras_factor(h, c.eps.data(), nullptr, c.p.k0, ORAS_MEM_HOST);
    g_refuse_from = -1;
    const bool refused = rc != ORAS_OK;
    if (refused && rc != ORAS_ERR_OUT_OF_MEMORY) bad(at("not reported as out of memory", n, rc));
    if (refused && h->factored) bad(at("factors that are not there count as there", n, rc));
    if (weak && !refused && (oras::g_weak || check_trees(h))) bad("the trees were not planned anew as they should");
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

// Factorisations that never stop finding such nodes: each ends after 8 new plans, all of them after 64, and the handle
// counts as factored.
static void always_weak() {
  Cube c(3, 2, 4);
  oras_options o{};
  oras_handle* h = nullptr;
  if (oras_create(&c.p, &o, &h) != ORAS_OK) { bad("oras_create failed"); return; }
  oras::g_weak = 1000;
  for (int call = 1; call <= 10; ++call) {
    if (oras_factor(h, c.eps.data(), nullptr, c.p.k0, ORAS_MEM_HOST) != ORAS_OK || !h->factored) bad("oras_factor failed");
    if (h->fronts.replans != std::min(8 * call, 64)) bad("new plans: " + std::to_string(h->fronts.replans));
  }
  oras::g_weak = 3;
  if (oras_autotune(h, nullptr, nullptr, 0) != ORAS_OK || !h->factored) bad("oras_autotune lost the factors");
  check_trees(h);
  oras_destroy(h);
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
  else if (s == "factor_weak32") factor_again(32, ORAS_LU_AUTO, 2);
  else if (s == "factor_weak64") factor_again(64, ORAS_LU_AUTO, 2);
  else if (s == "always_weak") always_weak();
  else if (s == "delay1") delay(4, 1, 5, 64);
  else if (s == "delay2") delay(5, 2, 2, 32);
  else if (s == "delay3") delay(3, 3, 3, 32);
  else if (s == "factor_dense") factor_again(32, ORAS_LU_CUDA_CORES);
  else if (s == "setup") setup_fails(ORAS_LU_AUTO);
  else if (s == "setup_dense") setup_fails(ORAS_LU_CUDA_CORES);
  else if (s == "solve32") solve_again(32);
  else if (s == "solve64") solve_again(64);
  else bad("unknown scenario");
  return g_bad ? 1 : 0;
}
