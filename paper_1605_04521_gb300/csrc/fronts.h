// Sparse local factorisations (block L D L^T over a nested-dissection tree): the plan shared by
// the host set-up (fronts_plan.cpp), the numeric kernels (fronts.cu) and the apply (fronts_apply.cu).
#pragma once

#include <complex>
#include <cstdint>
#include <vector>

namespace oras {

// One node of a subdomain's elimination tree: n1 unknowns eliminated together (its own rows) and the
// n2 later-eliminated unknowns they couple to (its border, ascending).  The factor panel holds
// S = A11^{-1} (n1 rows) over L = A21 S (n2 rows), row-major with ld entries a row.
struct FrontNode {
  int64_t panel;    // first entry of the panel in the factor arena (and in the assembly workspace)
  int64_t cblk;     // first entry of the contribution block C = A22 - L A21^T (n2 x ldc, lower tiles)
  int64_t bord;     // first entry in the border list, and in the apply's border vectors
  int32_t row0;     // first own row (elimination positions of all subdomains, one after the other)
  int32_t sub;
  int32_t n1, n2, ld, ldc;
  int32_t child[2]; // nodes, -1: none
};
// Where a row of a front is in the borders of its node's two children: entries of the border list, -1: not
// there.  Own rows: own_src[row0 + i]; border rows: border_src[bord + i].
struct alignas(8) FrontSrc { int32_t a, b; };

// A block's share of a level's work: tile `t` of node `node`.
struct FrontItem { int32_t node, t; };

constexpr int FR_TILE = 64;     // tile of the panel and contribution products
constexpr int FR_TC_ROWS = 128; // and its rows on the tensor cores (FP32): item t = row tile << 16 | column tile
constexpr int FR_ASM_ROWS = 32; // panel rows per assembly block
constexpr int FR_FWD_ROWS = 64; // border rows per block of the forward pass
constexpr int FR_BWD_COLS = 32; // own columns per block of the backward pass at the widest
constexpr int FR_BWD_BLOCKS = 1216;  // levels with fewer blocks than this (8 an SM) take narrower ones

// Largest number of unknowns eliminated together: the pivot block is inverted by one thread block
// in registers.
inline int front_nb(int factor_bits) { return factor_bits == 64 ? 64 : 128; }

// Width class of a pivot block: kernels for up to 128, 96, 64 and 32 unknowns.
constexpr int FR_CLASSES = 4;
inline int front_class(int n1) { return n1 > 96 ? 0 : (n1 > 64 ? 1 : (n1 > 32 ? 2 : 3)); }

struct FrontLevels {  // per level: [ptr[l], ptr[l + 1]) of the item list
  std::vector<FrontItem> items;
  std::vector<int64_t> ptr;
};

struct Fronts {
  bool use = false;
  int replans = 0;                    // times delay_unknowns changed the plan
  std::vector<FrontNode> nodes;       // by level, wide pivot blocks first within a level
  std::vector<int32_t> level_ptr;     // [nlev + 1] first node of each level
  std::vector<int32_t> level_class;   // [nlev][FR_CLASSES + 1] first node of each width class (front_class)
  std::vector<int32_t> border;        // positions
  std::vector<FrontSrc> own_src, border_src;
  std::vector<int32_t> pos;           // [sum ns] position (within its subdomain) of the local unknown i
  std::vector<int32_t> row_node;      // [sum ns] node that eliminates the unknown at a position
  std::vector<int32_t> row_dof;       // [sum ns] global unknown at a position
  std::vector<uint8_t> row_pou;       // [sum ns] its partition-of-unity weight
  FrontLevels assemble, lmul, schur, fwd, bwd, bwd_multi;
  std::vector<int32_t> bwd_cols;      // [nlev] own columns per block of bwd: 8, 16 or 32
  std::vector<int32_t> multi_cols;    // [nlev] and of bwd_multi: 16 or 64
  int64_t panel_elems = 0, c_elems = 0, border_elems = 0;
  int nlev() const { return (int)multi_cols.size(); }
};

// Largest entry of L = A21 A11^{-1} that the factorisation takes as it is.  Ordinary trees stay below 7 (degrees 1 to 3,
// with and without losses, k0 from 0.01 to 9; 28 in one without losses near a resonance); the apply's error is the unit roundoff times its square: at 64 1e-4 in
// FP32 and 1e-12 in FP64.
constexpr float FR_GROWTH = 64.0f;
// Times a factorisation plans the trees anew before it takes what it has, and all factorisations of a handle together
// (at frequencies so low that FP32 holds no digit of A_s, every factorisation would).
constexpr int FR_REPLANS = 8, FR_REPLANS_HANDLE = 64;

struct HostMesh;
// Elimination trees of every subdomain of m for factors of the given precision (dirichlet: of the
// matrices R_s A R_s^T).
void build_fronts(const HostMesh& m, int factor_bits, bool dirichlet, Fronts& f);

// The own unknowns of a node that its parent should eliminate, so that no entry of L exceeds FR_GROWTH (fronts_weak.cpp).
// panel: [n1 + n2][n1] the assembled A11 over A21.  false: an own unknown has no coupling left, A_s is singular.
bool weak_unknowns(int n1, int n2, const std::vector<std::complex<double>>& panel, std::vector<int32_t>& out);

// The plan with own unknowns moves[g] (indices into node g's own) of every node eliminated by the next ancestor that has
// room, or by a new root.
void delay_unknowns(const HostMesh& m, int factor_bits, const std::vector<std::vector<int32_t>>& moves, Fronts& f);

}  // namespace oras
