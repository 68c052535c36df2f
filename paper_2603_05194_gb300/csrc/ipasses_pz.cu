// The z pass of the binary64 preconditioner (see ipasses_p.cu).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t ip_z(atkm_plan* p, const double* alpha_dev, const IPassGrid& gy, const IPassGrid& gz, cudaStream_t st) {
  const Geo& g = p->g;
  IPZ op;
  op.Wk = p->T1; op.in = exp_cols(p->ex[1], gy); op.ex = exp_cols(p->ex[2], gz); op.alpha = alpha_dev;
  op.nx2 = iaxt(p, 0).hnu2; op.ny2 = iaxt(p, 1).hnu2; op.nz2 = iaxt(p, 2).hnu2;
  op.Nt = (double)g.Nx * (double)g.Ny * (double)g.Nz; op.Nx = g.Nx; op.Ny = g.Ny;
  ATKM_IRUN("P_z_f64", 32.0 * g.Nx * g.Ny * g.Nz, 2.0 * g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
  return cudaSuccess;
}

}  // namespace atkm
