// The binary64 preconditioner and the 3D transform of the spectral
// interpolation: integer passes (iops.cuh).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t launch_precond64(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                             const double* Phi, double* Pr, cudaStream_t st) {
  const Geo& g = p->g;
  const IPassGrid gx = ipass_grid(p, g.Nx, true, (long)g.Nz * g.Ny, 0, 0);
  const IPassGrid gy = ipass_grid(p, g.Ny, false, 0, g.Nx, g.Nz);
  const IPassGrid gz = ipass_grid(p, g.Nz, false, 0, g.Nx, g.Ny);
  cudaError_t e = ip_xf(p, ph, alpha_dev, r, phi, Phi, gx, st);
  if (e == cudaSuccess) e = ip_y<-1, true>(p, "P_y_f64", p->T1, exp_lines(p->ex[0], gx), 1, gy, st);
  if (e == cudaSuccess) e = ip_z(p, alpha_dev, gy, gz, st);
  if (e == cudaSuccess) e = ip_y<1, false>(p, "P_y_f64", p->T1, exp_cols(p->ex[2], gz), 0, gy, st);
  if (e == cudaSuccess) e = ip_xi(p, Pr, gx, gy, st);
  return e;
}

namespace {
template <int S> cudaError_t run_cfft3(atkm_plan* p, double2* buf, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const IPassGrid gx = ipass_grid(p, g.Nx, true, nl, 0, 0, false);
  const IPassGrid gy = ipass_grid(p, g.Ny, false, 0, g.Nx, g.Nz);
  const IPassGrid gz = ipass_grid(p, g.Nz, false, 0, g.Nx, g.Ny, false);
  {
    ICX<S> op;
    op.buf = buf; op.ex = exp_lines(p->ex[0], gx); op.Nx = g.Nx; op.nl = nl;
    ATKM_IRUN_GEN("fft3_x", 32 * N, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  }
  const cudaError_t e = ip_y<S, true>(p, "fft3_y", reinterpret_cast<c64*>(buf), exp_lines(p->ex[0], gx), 1, gy, st);
  if (e != cudaSuccess) return e;
  {
    ICZ<S> op;
    op.buf = buf; op.in = exp_cols(p->ex[1], gy); op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN_GEN("fft3_z", 32 * N, (double)g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_cfft3(atkm_plan* p, double2* buf, int sign, cudaStream_t st) {
  return sign < 0 ? run_cfft3<-1>(p, buf, st) : run_cfft3<1>(p, buf, st);
}

}  // namespace atkm
