// Unknowns of a tree node that have to be eliminated later than planned (host, FP64, up to 128 unknowns a node).
//
// A node's pivot block A11 can be nearly singular where A_s is not: the field inside the node's tetrahedra can
// resonate at the working frequency, or an unknown can couple only to its border.  L = A21 A11^{-1} is then large, and
// with it the rounding of the contribution block: the apply's error grows with the square of L's largest entry.
// Moving the unknown in which the resonating field is largest to the parent node makes both blocks regular again
// (delayed pivots, with the tree planned anew instead of a front that changes size).
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "fronts.h"

namespace oras {

using zc = std::complex<double>;

static double mag(zc v) { return std::max(std::fabs(v.real()), std::fabs(v.imag())); }

// S = A^{-1} by Gauss-Jordan elimination with row pivoting; a pivot below `least` is taken as `least`.
static void invert(int n, std::vector<zc>& A, double least, std::vector<zc>& S) {
  S.assign((size_t)n * n, zc(0.0));
  for (int i = 0; i < n; ++i) S[(size_t)i * n + i] = 1.0;
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int i = c + 1; i < n; ++i)
      if (mag(A[(size_t)i * n + c]) > mag(A[(size_t)p * n + c])) p = i;
    if (p != c)
      for (int j = 0; j < n; ++j) {
        std::swap(A[(size_t)p * n + j], A[(size_t)c * n + j]);
        std::swap(S[(size_t)p * n + j], S[(size_t)c * n + j]);
      }
    if (mag(A[(size_t)c * n + c]) < least) A[(size_t)c * n + c] = least;
    const zc inv = 1.0 / A[(size_t)c * n + c];
    for (int j = 0; j < n; ++j) { A[(size_t)c * n + j] *= inv; S[(size_t)c * n + j] *= inv; }
    for (int i = 0; i < n; ++i) {
      const zc f = A[(size_t)i * n + c];
      if (i == c || f == zc(0.0)) continue;
      for (int j = c; j < n; ++j) A[(size_t)i * n + j] -= f * A[(size_t)c * n + j];
      for (int j = 0; j < n; ++j) S[(size_t)i * n + j] -= f * S[(size_t)c * n + j];
    }
  }
}

bool weak_unknowns(int n1, int n2, const std::vector<std::complex<double>>& panel, std::vector<int32_t>& out) {
  out.clear();
  double amax = 0.0;
  for (const zc& v : panel) {
    if (!std::isfinite(v.real()) || !std::isfinite(v.imag())) return true;  // nothing to be gained
    amax = std::max(amax, mag(v));
  }
  for (int j = 0; j < n1; ++j) {  // an unknown without any coupling left: A_s is singular
    bool zero = true;
    for (int i = 0; i < n1 + n2 && zero; ++i) zero = panel[(size_t)i * n1 + j] == zc(0.0);
    if (zero) return false;
  }
  std::vector<zc> A(panel.begin(), panel.begin() + (size_t)n1 * n1), S;
  invert(n1, A, amax * 1e-16, S);
  std::vector<zc> L((size_t)n2 * n1, zc(0.0));
  for (int i = 0; i < n2; ++i)
    for (int k = 0; k < n1; ++k) {
      const zc a = panel[(size_t)(n1 + i) * n1 + k];
      if (a != zc(0.0))
        for (int j = 0; j < n1; ++j) L[(size_t)i * n1 + j] += a * S[(size_t)k * n1 + j];
    }
  // The inverse without unknown x is S - S(:, x) S(x, :) / S(x, x); x joins the border with the row -S(x, :) / S(x, x).
  std::vector<uint8_t> left(n1, 0);
  int rows = n2;
  while ((int)out.size() < n1) {
    double best = 0.0;
    int x = -1;
    for (int j = 0; j < n1; ++j)
      if (!left[j])
        for (int i = 0; i < rows; ++i)
          if (mag(L[(size_t)i * n1 + j]) > best) { best = mag(L[(size_t)i * n1 + j]); x = j; }
    if (!(best > 0.5 * FR_GROWTH)) break;
    left[x] = 1;
    out.push_back(x);
    const zc d = S[(size_t)x * n1 + x];
    if (d == zc(0.0)) continue;  // its partner follows
    std::vector<zc> r(S.begin() + (size_t)x * n1, S.begin() + (size_t)(x + 1) * n1);
    for (zc& v : r) v /= d;
    for (int i = 0; i < rows; ++i) {
      const zc l = L[(size_t)i * n1 + x];
      for (int j = 0; j < n1; ++j) L[(size_t)i * n1 + j] -= l * r[j];
    }
    for (int i = 0; i < n1; ++i) {
      const zc s = S[(size_t)i * n1 + x];
      if (i != x)
        for (int j = 0; j < n1; ++j) S[(size_t)i * n1 + j] -= s * r[j];
    }
    L.resize((size_t)(rows + 1) * n1);
    for (int j = 0; j < n1; ++j) L[(size_t)rows * n1 + j] = -r[j];
    ++rows;
  }
  return true;
}

}  // namespace oras
