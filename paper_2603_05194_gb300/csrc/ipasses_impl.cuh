// Launch helpers of the binary64 passes (iops.cuh).
#pragma once

#include <math.h>

#include "iops.cuh"

namespace atkm {

inline double ifftflops(double n) { return 5.0 * n * log2(n); }

#define ATKM_IRUN(NAME, BYTES, FLOPS, OP, FLEN, PG)             \
  do {                                                         \
    prof_begin(p, NAME, BYTES, FLOPS, st);                     \
    cudaError_t e_ = irun<true>(OP, FLEN, PG, st);             \
    prof_end(p, st);                                           \
    count_launches(1);                                         \
    if (e_ != cudaSuccess) return e_;                          \
  } while (0)

// The same for a pass that is rarely run: k_imix is not instantiated for it
// (its grid is made with mix = false).
#define ATKM_IRUN_GEN(NAME, BYTES, FLOPS, OP, FLEN, PG)         \
  do {                                                         \
    prof_begin(p, NAME, BYTES, FLOPS, st);                     \
    cudaError_t e_ = irun<false>(OP, FLEN, PG, st);            \
    prof_end(p, st);                                           \
    count_launches(1);                                         \
    if (e_ != cudaSuccess) return e_;                          \
  } while (0)

// Exponent table of a line-major pass (one entry a tile of lines) ...
inline ExpTab exp_lines(int* e, const IPassGrid& pg) { return ExpTab{e, pg.tsh, 16, 1}; }
// ... and of a column pass (one entry an outer index and column tile).
inline ExpTab exp_cols(int* e, const IPassGrid& pg) { return ExpTab{e, 0, pg.tsh, (int)pg.grid.x}; }
// The same with one entry a line (kLineExp): of an x line, of column x of X.
inline ExpTab exp_each_line(int* e) { return ExpTab{e, 0, 16, 1}; }
inline ExpTab exp_each_col(int* e, int X) { return ExpTab{e, 0, 0, X}; }

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

// The passes, each in its own translation unit (ipasses_*.cu).
cudaError_t iatkm_xf(atkm_plan* p, bool dw, int mode, const double* a, const double* b, const IPassGrid& gx,
                     cudaStream_t st);
cudaError_t iatkm_yf(atkm_plan* p, bool dw, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st);
cudaError_t iatkm_z(atkm_plan* p, bool dw, const IPassGrid& gy, const IPassGrid& gz, cudaStream_t st);
cudaError_t iatkm_yi(atkm_plan* p, bool dw, const IPassGrid& gz, const IPassGrid& gy, cudaStream_t st);
cudaError_t iatkm_xi(atkm_plan* p, bool dw, double* phi, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st);

struct HArgs {
  const Phys* ph;
  const double* f;
  const double* phi;
  const double* Phi;
  double* Hf;
  IPassGrid gx, gy, gz;
};
cudaError_t ih_x(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st);
cudaError_t ih_y(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st);
cudaError_t ih_z(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st);

cudaError_t ip_xf(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                  const double* Phi, const IPassGrid& gx, cudaStream_t st);
template <int S, bool LINES>
cudaError_t ip_y(atkm_plan* p, const char* name, c64* buf, const ExpTab& in, int ex, const IPassGrid& gy, cudaStream_t st);
cudaError_t ip_z(atkm_plan* p, const double* alpha_dev, const IPassGrid& gy, const IPassGrid& gz, cudaStream_t st);
cudaError_t ip_xi(atkm_plan* p, double* Pr, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st);

}  // namespace atkm
