// The binary64 dipolar potential: five integer passes (iops.cuh).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t launch_atkm64(atkm_plan* p, bool dw, int mode, const double* a, const double* b, double* phi,
                          cudaStream_t st) {
  const Geo& g = p->g;
  const IPassGrid gx = ipass_grid(p, g.Nx, true, (long)g.Nz * g.Ny, 0, 0);
  const IPassGrid gy = ipass_grid(p, g.My, false, 0, g.Xh, g.Nz);
  const IPassGrid gz = ipass_grid(p, g.Mz, false, 0, g.Xh, g.My);
  cudaError_t e = iatkm_xf(p, dw, mode, a, b, gx, st);
  if (e == cudaSuccess) e = iatkm_yf(p, dw, gx, gy, st);
  if (e == cudaSuccess) e = iatkm_z(p, dw, gy, gz, st);
  if (e == cudaSuccess) e = iatkm_yi(p, dw, gz, gy, st);
  if (e == cudaSuccess) e = iatkm_xi(p, dw, phi, gx, gy, st);
  return e;
}

}  // namespace atkm
