// Launch helpers of the binary64 passes (iops.cuh).
#pragma once

#include <math.h>

#include "iops.cuh"

namespace atkm {

inline double ifftflops(double n) { return 5.0 * n * log2(n); }

#define ATKM_IRUN(NAME, BYTES, FLOPS, OP, FLEN, PG)             \
  do {                                                         \
    prof_begin(p, NAME, BYTES, FLOPS, st);                     \
    cudaError_t e_ = irun(OP, FLEN, PG, st);                   \
    prof_end(p, st);                                           \
    count_launches(1);                                         \
    if (e_ != cudaSuccess) return e_;                          \
  } while (0)

// Exponent table of a line-major pass (one entry a tile of lines) ...
inline ExpTab exp_lines(int* e, const IPassGrid& pg) { return ExpTab{e, pg.tsh, 16, 1}; }
// ... and of a column pass (one entry an outer index and column tile).
inline ExpTab exp_cols(int* e, const IPassGrid& pg) { return ExpTab{e, 0, pg.tsh, (int)pg.grid.x}; }

// The plan's binary64 tables of axis a (see AxT in atkm_internal.cuh).
inline AxT iaxt(const atkm_plan* p, int a) {
  const int Ns[3] = {p->g.Nx, p->g.Ny, p->g.Nz};
  size_t off = 0;
  for (int b = 0; b < a; ++b) off += 4 * (size_t)Ns[b];
  const double* t = p->axtab + off;
  const size_t n = (size_t)Ns[a];
  AxT r;
  r.nuN = t; r.kinN = t + n; r.hnu2 = t + 2 * n; r.hxc2 = t + 3 * n;
  return r;
}

}  // namespace atkm
