// Elimination trees of the local matrices (host, integers only; once per mesh).
//
// A_s couples two unknowns only when they share a tetrahedron of Omega_s^delta (16-80 couplings a
// row), so the set-up dissects each subdomain's tetrahedra: a set is cut in two along a coordinate
// axis, the unknowns carried by both halves form the separator, eliminated after either half, and
// the halves are cut again until few unknowns are left (nested dissection by substructuring; the
// separator of a cut is the unknowns of the cut's faces, the thinnest there is for edge elements).
// The cut is the one with the smallest separator among the middle 30% of the tetrahedra along the
// longer axes.  A tree node (a separator, or the interior of an uncut set) couples only to the
// separators above it that its tetrahedra touch, its border.  Wide nodes are split into a chain of
// at most front_nb unknowns.
#include "fronts.h"

#include <cmath>
#include <memory>
#include <stdexcept>

#include "internal.h"
#include "par.h"

namespace oras {

namespace {

struct LocalNode {
  std::vector<int32_t> own;       // local unknowns (indices into N_s), ascending
  std::vector<int32_t> border;    // local unknowns, then positions
  int32_t child[2] = {-1, -1};    // local node ids
  std::vector<FrontSrc> src;      // [n1 + n2] position in the children's borders, -1
  int32_t p0 = 0, level = 0;
};

// The tree of one subdomain.  An entity (edge, face or volume) carries consecutive unknowns with the
// same tetrahedra, so the dissection works on entities, named by their first unknown.
struct Builder {
  const HostMesh& m;
  int nb;
  int ne;                          // entities of a tetrahedron
  int wt[11];                      // unknowns of each
  int first[11];                   // tet-local index of its first unknown
  std::vector<int32_t> list;       // tetrahedra
  std::vector<int32_t> ent;        // [tets][ne] first unknown (index into N_s), -1: not in N_s
  std::vector<double> cen;         // [tets][3]
  std::vector<int32_t> tets;       // permutation of the subdomain's tetrahedra
  std::vector<uint8_t> width;      // [ns] unknowns of the entity starting here
  std::vector<uint8_t> taken;      // [ns] eliminated by a separator above
  std::vector<int32_t> stamp, lo, hi;
  int32_t now = 0;
  std::vector<LocalNode> nodes;

  Builder(const HostMesh& mesh, int nb_) : m(mesh), nb(nb_) {
    const int r = m.r;
    ne = 6 + (r >= 2 ? 4 : 0) + (r == 3 ? 1 : 0);
    int at = 0;
    for (int q = 0; q < ne; ++q) {
      wt[q] = q < 6 ? r : (q < 10 ? r * (r - 1) : r * (r - 1) * (r - 2) / 2);
      first[q] = at;
      at += wt[q];
    }
  }

  // loc: index in N_s of the global unknowns of N_s (others: any value).  dirichlet: A_s = R_s A R_s^T,
  // which also couples unknowns of N_s that share only a tetrahedron outside Omega_s^delta.
  void run(int s, const std::vector<int32_t>& loc, bool dirichlet) {
    const int64_t off = m.sub_ns_off[s], ns = m.sub_ns[s];
    auto local = [&](int32_t g) {
      const int32_t i = loc[g];
      return i < ns && m.sub_dofs[off + i] == g ? i : -1;
    };
    list.assign(m.sub_tets.begin() + m.sub_nt_off[s], m.sub_tets.begin() + m.sub_nt_off[s + 1]);
    if (dirichlet) {
      const size_t inside = list.size();
      for (int64_t i = 0; i < ns; ++i) {
        const int32_t g = m.sub_dofs[off + i];
        for (int64_t q = m.tinc_ptr[g]; q < m.tinc_ptr[g + 1]; ++q) list.push_back(m.tinc[q] / m.nl);
      }
      std::sort(list.begin() + inside, list.end());
      list.erase(std::unique(list.begin() + inside, list.end()), list.end());
      list.erase(std::remove_if(list.begin() + inside, list.end(),
                                [&](int32_t t) {
                                  return (m.member[(size_t)s * m.member_words + (t >> 5)] >> (t & 31)) & 1u;
                                }),
                 list.end());
    }
    const int64_t nt = (int64_t)list.size();
    ent.resize(nt * ne);
    cen.resize(nt * 3);
    tets.resize(nt);
    width.assign(ns, 0);
    taken.assign(ns, 0);
    stamp.assign(ns, 0);
    lo.resize(ns);
    hi.resize(ns);
    now = 0;
    nodes.clear();
    for (int64_t i = 0; i < nt; ++i) {
      const int64_t t = list[i];
      tets[i] = (int32_t)i;
      for (int q = 0; q < ne; ++q) {
        const int32_t e = local(m.dofmap[t * m.nl + first[q]]);
        ent[i * ne + q] = e;
        if (e >= 0) width[e] = (uint8_t)wt[q];
      }
      for (int d = 0; d < 3; ++d) {
        double c = 0.0;
        for (int q = 0; q < 4; ++q) c += m.xyz[(int64_t)m.st[t * 4 + q] * 3 + d];
        cen[i * 3 + d] = 0.25 * c;
      }
    }
    std::vector<int32_t> border, roots;
    dissect(0, (int32_t)nt, border, roots);
  }

  void link(LocalNode& x, const std::vector<int32_t>& children) {
    for (size_t q = 0; q < children.size(); ++q) {
      x.child[q] = children[q];
      x.level = std::max(x.level, nodes[children[q]].level + 1);
    }
  }

  // Nodes for `own` entities over `border` entities: a chain of at most nb unknowns each.
  // `roots`: in, the children; out, the chain's top.
  void add(std::vector<int32_t>& own, const std::vector<int32_t>& border, std::vector<int32_t>& roots) {
    std::sort(own.begin(), own.end());
    std::vector<int32_t> u, b;
    for (int32_t e : own)
      for (int w = 0; w < width[e]; ++w) u.push_back(e + w);
    for (int32_t e : border)
      for (int w = 0; w < width[e]; ++w) b.push_back(e + w);
    // at most two children a node: pairs of others are joined by nodes that eliminate nothing
    while (roots.size() > 2) {
      LocalNode x;
      std::vector<int32_t> c(roots.end() - 2, roots.end());
      roots.resize(roots.size() - 2);
      for (int q = 0; q < 2; ++q) x.border.insert(x.border.end(), nodes[c[q]].border.begin(), nodes[c[q]].border.end());
      std::sort(x.border.begin(), x.border.end());
      x.border.erase(std::unique(x.border.begin(), x.border.end()), x.border.end());
      link(x, c);
      roots.insert(roots.begin(), (int32_t)nodes.size());
      nodes.push_back(std::move(x));
    }
    const int n = (int)u.size(), parts = (n + nb - 1) / nb;
    for (int p = 0; p < parts; ++p) {
      LocalNode x;
      const int q0 = (int)((int64_t)n * p / parts), q1 = (int)((int64_t)n * (p + 1) / parts);
      x.own.assign(u.begin() + q0, u.begin() + q1);
      x.border.assign(u.begin() + q1, u.end());
      x.border.insert(x.border.end(), b.begin(), b.end());
      link(x, roots);
      roots.assign(1, (int32_t)nodes.size());
      nodes.push_back(std::move(x));
    }
  }

  // Tree over tets[b, e): its border entities (eliminated above) and the roots of its nodes.
  void dissect(int32_t b, int32_t e, std::vector<int32_t>& border, std::vector<int32_t>& roots) {
    const int32_t n = e - b;
    std::vector<int32_t> own;
    int weight = 0;
    ++now;
    for (int32_t i = b; i < e; ++i)
      for (int q = 0; q < ne; ++q) {
        const int32_t x = ent[(int64_t)tets[i] * ne + q];
        if (x < 0 || stamp[x] == now) continue;
        stamp[x] = now;
        if (taken[x]) border.push_back(x);
        else { own.push_back(x); weight += wt[q]; }
      }
    if (own.empty()) return;
    double best = INFINITY;
    int best_axis = -1;
    int32_t best_cut = 0;
    double ext[3];
    if (weight > nb && n > 1) {
      for (int d = 0; d < 3; ++d) {
        double c0 = INFINITY, c1 = -INFINITY;
        for (int32_t i = b; i < e; ++i) {
          c0 = std::min(c0, cen[(int64_t)tets[i] * 3 + d]);
          c1 = std::max(c1, cen[(int64_t)tets[i] * 3 + d]);
        }
        ext[d] = c1 - c0;
      }
      const double longest = std::max(ext[0], std::max(ext[1], ext[2]));
      std::vector<int32_t> cut(n + 1);
      for (int d = 0; d < 3; ++d) {
        if (ext[d] < 0.5 * longest) continue;
        sort_axis(b, e, d);
        // separator weight of every cut position: an entity whose tetrahedra have ranks lo..hi is
        // carried by both sides of the cuts lo < p <= hi
        std::fill(cut.begin(), cut.end(), 0);
        for (int32_t x : own) { lo[x] = n; hi[x] = -1; }
        for (int32_t i = b; i < e; ++i)
          for (int q = 0; q < ne; ++q) {
            const int32_t x = ent[(int64_t)tets[i] * ne + q];
            if (x < 0 || taken[x]) continue;
            lo[x] = std::min(lo[x], i - b);
            hi[x] = i - b;
          }
        for (int32_t x : own)
          if (hi[x] > lo[x]) { cut[lo[x] + 1] += width[x]; cut[hi[x] + 1 <= n ? hi[x] + 1 : n] -= width[x]; }
        for (int32_t p = 1; p <= n; ++p) cut[p] += cut[p - 1];
        const int32_t p0 = std::max<int32_t>(1, (int32_t)(n * 0.35)), p1 = std::min<int32_t>(n - 1, n - p0);
        for (int32_t p = std::min(p0, n / 2); p <= std::max(p1, n / 2); ++p) {
          if (p < 1 || p >= n) continue;
          const double off = std::fabs(p - 0.5 * n) / (0.5 * n);
          const double score = (cut[p] + 1) * (1.0 + 0.5 * off);
          if (score < best) { best = score; best_axis = d; best_cut = p; }
        }
      }
    }
    if (best_axis < 0) {
      add(own, border, roots);
      return;
    }
    sort_axis(b, e, best_axis);
    const int32_t mid = b + best_cut;
    std::vector<int32_t> sep;
    ++now;
    for (int32_t i = b; i < mid; ++i)
      for (int q = 0; q < ne; ++q) {
        const int32_t x = ent[(int64_t)tets[i] * ne + q];
        if (x >= 0) stamp[x] = now;
      }
    const int32_t left = now;
    ++now;
    for (int32_t i = mid; i < e; ++i)
      for (int q = 0; q < ne; ++q) {
        const int32_t x = ent[(int64_t)tets[i] * ne + q];
        if (x >= 0 && stamp[x] == left && !taken[x]) { stamp[x] = now; sep.push_back(x); }
      }
    if (sep.size() == own.size()) {  // nothing inside either half
      add(own, border, roots);
      return;
    }
    for (int32_t x : sep) taken[x] = 1;
    std::vector<int32_t> sub;
    dissect(b, mid, sub, roots);
    sub.clear();
    std::vector<int32_t> r2;
    dissect(mid, e, sub, r2);
    roots.insert(roots.end(), r2.begin(), r2.end());
    if (!sep.empty()) add(sep, border, roots);
  }

  void sort_axis(int32_t b, int32_t e, int d) {
    std::sort(tets.begin() + b, tets.begin() + e, [&](int32_t x, int32_t y) {
      const double cx = cen[(int64_t)x * 3 + d], cy = cen[(int64_t)y * 3 + d];
      return cx < cy || (cx == cy && x < y);
    });
  }
};

// Elimination positions (nodes in order: children first), borders as ascending positions, and where each front is
// in the children's borders.  pos: [ns] position of every local unknown.
void number(std::vector<LocalNode>& nodes, int64_t ns, std::vector<int32_t>& pos) {
  pos.assign(ns, -1);
  int32_t p = 0;
  for (auto& x : nodes) {
    x.p0 = p;
    for (int32_t u : x.own) pos[u] = p++;
  }
  for (auto& x : nodes) {
    for (int32_t& u : x.border) u = pos[u];
    std::sort(x.border.begin(), x.border.end());
  }
  for (auto& x : nodes) {
    const int n1 = (int)x.own.size(), n2 = (int)x.border.size();
    auto front = [&](int i) { return i < n1 ? x.p0 + i : x.border[i - n1]; };
    x.src.assign(n1 + n2, {-1, -1});
    for (int c = 0; c < 2; ++c) {
      if (x.child[c] < 0) continue;
      const auto& cb = nodes[x.child[c]].border;
      size_t k = 0;
      for (int i = 0; i < n1 + n2 && k < cb.size(); ++i)
        if (cb[k] == front(i)) (c == 0 ? x.src[i].a : x.src[i].b) = (int32_t)k++;
    }
  }
}

// The plan of all subdomains' numbered trees: node order, offsets, the rows' and borders' arrays, the blocks of every
// level.  f.pos is there.
void lay_out(const HostMesh& m, int factor_bits, const std::vector<std::vector<LocalNode>>& trees, Fronts& f) {
  const int64_t rows = m.sub_ns_off[m.nsub];
  // global node order: by level, wide pivot blocks first, then the larger fronts
  struct Key { int32_t level, wide, cost, sub, id; };
  std::vector<Key> keys;
  std::vector<std::vector<int32_t>> gid(m.nsub);
  int nlev = 0;
  for (int s = 0; s < m.nsub; ++s) {
    gid[s].resize(trees[s].size());
    for (size_t q = 0; q < trees[s].size(); ++q) {
      const LocalNode& x = trees[s][q];
      keys.push_back({x.level, front_class((int)x.own.size()), -(int32_t)x.border.size(), s, (int32_t)q});
      nlev = std::max(nlev, x.level + 1);
    }
  }
  std::sort(keys.begin(), keys.end(), [](const Key& a, const Key& b) {
    if (a.level != b.level) return a.level < b.level;
    if (a.wide != b.wide) return a.wide < b.wide;
    if (a.cost != b.cost) return a.cost < b.cost;
    return a.sub != b.sub ? a.sub < b.sub : a.id < b.id;
  });
  const int64_t nn = (int64_t)keys.size();
  f.nodes.resize(nn);
  f.level_ptr.assign(nlev + 1, 0);
  f.level_class.assign((size_t)nlev * (FR_CLASSES + 1), 0);
  f.row_node.resize(rows);
  f.row_dof.resize(rows);
  f.row_pou.resize(rows);
  int64_t panel = 0, cblk = 0, bord = 0;
  for (int64_t g = 0; g < nn; ++g) {
    const Key& k = keys[g];
    gid[k.sub][k.id] = (int32_t)g;
    const LocalNode& x = trees[k.sub][k.id];
    FrontNode& n = f.nodes[g];
    n.sub = k.sub;
    n.n1 = (int32_t)x.own.size();
    n.n2 = (int32_t)x.border.size();
    n.ld = (n.n1 + 3) / 4 * 4;
    n.ldc = (n.n2 + 3) / 4 * 4;
    n.row0 = (int32_t)(m.sub_ns_off[k.sub] + x.p0);
    n.panel = panel;
    n.cblk = cblk;
    n.bord = bord;
    for (int q = 0; q < 2; ++q) n.child[q] = x.child[q] < 0 ? -1 : gid[k.sub][x.child[q]];
    panel += (int64_t)(n.n1 + n.n2) * n.ld;
    cblk += (int64_t)n.n2 * n.ldc;
    bord += n.n2;
    f.level_ptr[k.level + 1]++;
    f.level_class[(size_t)k.level * (FR_CLASSES + 1) + k.wide + 1]++;
  }
  for (int l = 0; l < nlev; ++l) {
    f.level_ptr[l + 1] += f.level_ptr[l];
    int32_t* c = &f.level_class[(size_t)l * (FR_CLASSES + 1)];
    c[0] = f.level_ptr[l];
    for (int q = 0; q < FR_CLASSES; ++q) c[q + 1] += c[q];
  }
  f.panel_elems = panel;
  f.c_elems = cblk;
  f.border_elems = bord;
  if (bord >= (int64_t(1) << 31)) throw std::length_error("the borders of the elimination trees exceed 2^31 entries");
  f.border.resize(bord);
  f.border_src.resize(bord);
  f.own_src.resize(rows);
  parallel_for(nn, 64, [&](int64_t g, int) {
    const FrontNode& n = f.nodes[g];
    const LocalNode& x = trees[n.sub][keys[g].id];
    const int32_t base = (int32_t)m.sub_ns_off[n.sub];
    const int32_t b0 = n.child[0] < 0 ? 0 : (int32_t)f.nodes[n.child[0]].bord;
    const int32_t b1 = n.child[1] < 0 ? 0 : (int32_t)f.nodes[n.child[1]].bord;
    auto src = [&](int i) {
      const FrontSrc v = x.src[i];
      return FrontSrc{v.a < 0 ? -1 : b0 + v.a, v.b < 0 ? -1 : b1 + v.b};
    };
    for (int q = 0; q < n.n2; ++q) {
      f.border[n.bord + q] = base + x.border[q];
      f.border_src[n.bord + q] = src(n.n1 + q);
    }
    for (int q = 0; q < n.n1; ++q) {
      f.own_src[n.row0 + q] = src(q);
      f.row_node[n.row0 + q] = (int32_t)g;
      f.row_dof[n.row0 + q] = m.sub_dofs[base + x.own[q]];
      f.row_pou[n.row0 + q] = m.sub_pou[base + x.own[q]];
    }
  });
  // block lists of every level
  FrontLevels* all[] = {&f.assemble, &f.lmul, &f.schur, &f.fwd, &f.bwd, &f.bwd_multi};
  for (auto* v : all) { v->items.clear(); v->ptr.assign(1, 0); }
  f.bwd_cols.clear();
  f.multi_cols.clear();
  for (int l = 0; l < nlev; ++l) {
    // backward pass: narrower column blocks where a level has few nodes
    int cols = FR_BWD_COLS;
    auto blocks = [&](int c) {
      int64_t n = 0;
      for (int32_t g = f.level_ptr[l]; g < f.level_ptr[l + 1]; ++g) n += (f.nodes[g].n1 + c - 1) / c;
      return n;
    };
    while (cols > 8 && blocks(cols) < FR_BWD_BLOCKS) cols /= 2;
    f.bwd_cols.push_back(cols);
    const int multi = blocks(64) < 200 ? 16 : 64;
    f.multi_cols.push_back(multi);
    for (int32_t g = f.level_ptr[l]; g < f.level_ptr[l + 1]; ++g) {
      const FrontNode& n = f.nodes[g];
      if (n.child[0] >= 0 && n.n1 > 0)
        for (int t = 0; t * FR_ASM_ROWS < n.n1 + n.n2; ++t) f.assemble.items.push_back({g, t});
      const int ti = (n.n2 + FR_TILE - 1) / FR_TILE, tj = (n.n1 + FR_TILE - 1) / FR_TILE;
      if (factor_bits == 32) {
        for (int i = 0; i * FR_TC_ROWS < n.n2; ++i) {
          for (int j = 0; j < tj; ++j) f.lmul.items.push_back({g, i << 16 | j});
          for (int j = 0; j < ti && j * FR_TILE < (i + 1) * FR_TC_ROWS; ++j) f.schur.items.push_back({g, i << 16 | j});
        }
      } else {
        for (int t = 0; t < ti * tj; ++t) f.lmul.items.push_back({g, t});
        for (int t = 0; t < ti * (ti + 1) / 2; ++t) f.schur.items.push_back({g, t});
      }
      for (int t = 0; t == 0 || t * FR_FWD_ROWS < n.n2; ++t) f.fwd.items.push_back({g, t});
      for (int t = 0; t * cols < n.n1; ++t) f.bwd.items.push_back({g, t});
      for (int t = 0; t * multi < n.n1; ++t) f.bwd_multi.items.push_back({g, t});
    }
    for (auto* v : all) v->ptr.push_back((int64_t)v->items.size());
  }
}

}  // namespace

void build_fronts(const HostMesh& m, int factor_bits, bool dirichlet, Fronts& f) {
  const int nb = front_nb(factor_bits);
  const int64_t rows = m.sub_ns_off[m.nsub];
  f.pos.resize(rows);
  std::vector<std::vector<LocalNode>> trees(m.nsub);
  const int nw = workers_for(m.nsub, 1);
  std::vector<std::vector<int32_t>> loc(nw), pos(nw);
  std::vector<std::unique_ptr<Builder>> builders(nw);
  parallel_for(m.nsub, 1, [&](int64_t s64, int w) {
    const int s = (int)s64;
    if (!builders[w]) {
      builders[w] = std::make_unique<Builder>(m, nb);
      loc[w].assign(m.ndof, 0);
    }
    const int64_t off = m.sub_ns_off[s], ns = m.sub_ns[s];
    for (int64_t i = 0; i < ns; ++i) loc[w][m.sub_dofs[off + i]] = (int32_t)i;
    Builder& b = *builders[w];
    b.run(s, loc[w], dirichlet);
    number(b.nodes, ns, pos[w]);
    std::copy(pos[w].begin(), pos[w].end(), f.pos.begin() + off);
    trees[s] = std::move(b.nodes);
  });
  lay_out(m, factor_bits, trees, f);
}

// The trees behind a plan, named by local unknowns again.
static std::vector<std::vector<LocalNode>> trees_of(const HostMesh& m, const Fronts& f, std::vector<int32_t>& local) {
  std::vector<std::vector<LocalNode>> trees(m.nsub);
  local.resize(f.nodes.size());
  std::vector<int32_t> unknown(m.sub_ns_off[m.nsub]);  // at each position, index into N_s
  for (int s = 0; s < m.nsub; ++s)
    for (int64_t i = 0; i < m.sub_ns[s]; ++i) unknown[m.sub_ns_off[s] + f.pos[m.sub_ns_off[s] + i]] = (int32_t)i;
  for (int l = 0; l < f.nlev(); ++l)
    for (int32_t g = f.level_ptr[l]; g < f.level_ptr[l + 1]; ++g) {
      const FrontNode& n = f.nodes[g];
      LocalNode x;
      x.own.assign(unknown.begin() + n.row0, unknown.begin() + n.row0 + n.n1);
      for (int q = 0; q < n.n2; ++q) x.border.push_back(unknown[f.border[n.bord + q]]);
      for (int q = 0; q < 2; ++q) x.child[q] = n.child[q] < 0 ? -1 : local[n.child[q]];
      x.level = l;
      local[g] = (int32_t)trees[n.sub].size();
      trees[n.sub].push_back(std::move(x));
    }
  return trees;
}

void delay_unknowns(const HostMesh& m, int factor_bits, const std::vector<std::vector<int32_t>>& moves, Fronts& f) {
  const size_t nb = front_nb(factor_bits);
  std::vector<int32_t> local;
  auto trees = trees_of(m, f, local);
  std::vector<std::vector<int32_t>> parent(m.nsub);
  for (int s = 0; s < m.nsub; ++s) {
    parent[s].assign(trees[s].size(), -1);
    for (size_t q = 0; q < trees[s].size(); ++q)
      for (int32_t c : trees[s][q].child)
        if (c >= 0) parent[s][c] = (int32_t)q;
  }
  for (size_t g = 0; g < f.nodes.size(); ++g) {
    auto& tree = trees[f.nodes[g].sub];
    auto& up = parent[f.nodes[g].sub];
    std::vector<int32_t> x;  // unknowns that leave the node
    for (int32_t i : moves[g]) x.push_back(tree[local[g]].own[i]);
    for (int32_t u : x) {
      int32_t q = local[g];
      tree[q].own.erase(std::find(tree[q].own.begin(), tree[q].own.end(), u));
      // every node on the way has it in its border, and so in its front
      for (;;) {
        tree[q].border.push_back(u);
        if (up[q] < 0) {  // above the root: a node of its own
          LocalNode r;
          r.child[0] = q;
          r.level = tree[q].level + 1;
          up[q] = (int32_t)tree.size();
          up.push_back(-1);
          tree.push_back(std::move(r));
        }
        q = up[q];
        if (tree[q].own.size() < nb) break;
      }
      tree[q].own.push_back(u);
    }
  }
  Fronts next;  // f stays as it is when memory runs out
  next.use = f.use;
  next.replans = f.replans + 1;
  next.pos.resize(f.pos.size());
  parallel_for(m.nsub, 1, [&](int64_t s, int) {
    std::vector<int32_t> pos;
    number(trees[s], m.sub_ns[s], pos);
    std::copy(pos.begin(), pos.end(), next.pos.begin() + m.sub_ns_off[s]);
  });
  lay_out(m, factor_bits, trees, next);
  f = std::move(next);
}

}  // namespace oras
