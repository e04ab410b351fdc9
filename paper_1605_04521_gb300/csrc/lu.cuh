// Update regions of the dense LU (lu.cu).
#pragma once

#include <climits>

#include "dev.cuh"

namespace oras {

// Rectangular set of output tiles [i0, i1) x [j0, j1); an end of INT_MAX means the subdomain's
// tile count.
struct Region { int i0, i1, j0, j1; };
struct UpdArgs {
  int kk0, kk1;             // contraction over tile columns [kk0, kk1)
  int nreg;
  Region reg[2];
};

}  // namespace oras
