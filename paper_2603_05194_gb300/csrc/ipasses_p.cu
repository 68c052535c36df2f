// The binary64 preconditioner and the 3D transform of the spectral
// interpolation: integer passes (iops.cuh).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t launch_precond64(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                             const double* Phi, double* Pr, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const double fx = (double)nl * ifftflops(g.Nx), fy = (double)g.Nz * g.Nx * ifftflops(g.Ny);
  const IPassGrid gx = ipass_grid(p, 0, g.Nx, true, nl, 0, 0);
  const IPassGrid gy = ipass_grid(p, 0, g.Ny, false, 0, g.Nx, g.Nz);
  const IPassGrid gz = ipass_grid(p, 0, g.Nz, false, 0, g.Nx, g.Ny);
  const AxT ax = iaxt(p, 0), ay = iaxt(p, 1), az = iaxt(p, 2);
  c64* Wk = p->T1;
  {
    IPXF op;
    op.r = reinterpret_cast<const double2*>(r); op.phi = reinterpret_cast<const double2*>(phi); op.Phi = Phi;
    op.Wk = Wk; op.Pw = p->Pw; op.ex = exp_lines(p->ex[0], gx);
    op.hx2 = ax.hxc2; op.hy2 = ay.hxc2; op.hz2 = az.hxc2;
    op.gx2 = ph.gx2; op.gy2 = ph.gy2; op.gz2 = ph.gz2; op.beta = ph.beta; op.alam = fabs(ph.lambda);
    op.alpha = alpha_dev; op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
    ATKM_IRUN("P_x_fwd_f64", 64 * N, fx, op, p->iN[0], gx);
  }
  {
    IPY<-1, true> op;
    op.Wk = Wk; op.in = exp_lines(p->ex[0], gx); op.ex = exp_cols(p->ex[1], gy);
    op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN("P_y_f64", 32 * N, fy, op, p->iN[1], gy);
  }
  {
    IPZ op;
    op.Wk = Wk; op.in = exp_cols(p->ex[1], gy); op.ex = exp_cols(p->ex[2], gz); op.alpha = alpha_dev;
    op.nx2 = ax.hnu2; op.ny2 = ay.hnu2; op.nz2 = az.hnu2;
    op.invN = 1.0 / ((double)g.Nx * (double)g.Ny * (double)g.Nz); op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN("P_z_f64", 32 * N, 2.0 * g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
  }
  {
    IPY<1, false> op;
    op.Wk = Wk; op.in = exp_cols(p->ex[2], gz); op.ex = exp_cols(p->ex[0], gy);
    op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN("P_y_f64", 32 * N, fy, op, p->iN[1], gy);
  }
  {
    IPXI op;
    op.Wk = Wk; op.Pw = p->Pw; op.Pr = reinterpret_cast<double2*>(Pr); op.in = exp_cols(p->ex[0], gy);
    op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
    ATKM_IRUN("P_x_inv_f64", 40 * N, fx, op, p->iN[0], gx);
  }
  return cudaSuccess;
}

namespace {
template <int S> cudaError_t run_cfft3(atkm_plan* p, double2* buf, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const IPassGrid gx = ipass_grid(p, 0, g.Nx, true, nl, 0, 0);
  const IPassGrid gy = ipass_grid(p, 0, g.Ny, false, 0, g.Nx, g.Nz);
  const IPassGrid gz = ipass_grid(p, 0, g.Nz, false, 0, g.Nx, g.Ny);
  {
    ICX<S> op;
    op.buf = buf; op.ex = exp_lines(p->ex[0], gx); op.Nx = g.Nx; op.nl = nl;
    ATKM_IRUN("fft3_x", 32 * N, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  }
  {
    IPY<S, true> op;
    op.Wk = reinterpret_cast<c64*>(buf); op.in = exp_lines(p->ex[0], gx); op.ex = exp_cols(p->ex[1], gy);
    op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN("fft3_y", 32 * N, (double)g.Nz * g.Nx * ifftflops(g.Ny), op, p->iN[1], gy);
  }
  {
    ICZ<S> op;
    op.buf = buf; op.in = exp_cols(p->ex[1], gy); op.Nx = g.Nx; op.Ny = g.Ny;
    ATKM_IRUN("fft3_z", 32 * N, (double)g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_cfft3(atkm_plan* p, double2* buf, int sign, cudaStream_t st) {
  return sign < 0 ? run_cfft3<-1>(p, buf, st) : run_cfft3<1>(p, buf, st);
}

}  // namespace atkm
