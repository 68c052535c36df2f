// The binary64 dipolar potential: five integer passes (iops.cuh).
#include "ipasses_impl.cuh"

namespace atkm {

namespace {
template <int MODE>
cudaError_t run_xf(atkm_plan* p, const char* name, double inb, const double* a, const double* b, const IPassGrid& gx,
                   cudaStream_t st) {
  const Geo& g = p->g;
  const double N = (double)g.Nx * g.Ny * g.Nz, H1 = (double)g.Nz * g.Ny * g.Xh;
  IAtkmXF<MODE> op;
  op.a = a; op.b = b; op.W1 = p->W1; op.wM = p->tw_x; op.ex = exp_lines(p->ex[0], gx);
  op.Nx = g.Nx; op.nl = g.Nz * g.Ny; op.XS = g.XS;
  ATKM_IRUN(name, inb * N + 16 * H1, (double)g.Nz * g.Ny * ifftflops(g.Nx), op, p->iN[0], gx);
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_atkm64(atkm_plan* p, bool dw, int mode, const double* a, const double* b, double* phi,
                          cudaStream_t st) {
  const Geo& g = p->g;
  const int r = dw ? 2 : 0;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz, H1 = (double)nl * g.Xh;
  const double fy = (double)g.Nz * g.Xh * ifftflops(g.My);
  const IPassGrid gx = ipass_grid(p, r, g.Nx, true, nl, 0, 0);
  const IPassGrid gy = ipass_grid(p, r, g.My, false, 0, g.Xh, g.Nz);
  const IPassGrid gz = ipass_grid(p, r, g.Mz, false, 0, g.Xh, g.My);
  cudaError_t e;
  const char* nx = dw ? "atkm_x_fwd_df" : "atkm_x_fwd_f64";
  if (mode == SRC_RHO) e = run_xf<SRC_RHO>(p, nx, 8.0, a, b, gx, st);
  else if (mode == SRC_PSI) e = run_xf<SRC_PSI>(p, nx, 16.0, a, b, gx, st);
  else e = run_xf<SRC_PAIR>(p, nx, 32.0, a, b, gx, st);
  if (e != cudaSuccess) return e;
  {
    IAtkmYF op;
    op.W1 = p->W1; op.W2 = p->W2; op.in = exp_lines(p->ex[0], gx); op.ex = exp_cols(p->ex[1], gy);
    op.Nx = g.Nx; op.Ny = g.Ny; op.My = g.My; op.XS = g.XS;
    ATKM_IRUN(dw ? "atkm_y_fwd_df" : "atkm_y_fwd_f64", 48 * H1, fy, op, p->iM[1], gy);
  }
  {
    IAtkmZ op;
    op.W2 = p->W2; op.K = p->Kz; op.in = exp_cols(p->ex[1], gy); op.ex = exp_cols(p->ex[2], gz);
    op.Nx = g.Nx; op.Nz = g.Nz; op.My = g.My; op.XS = g.XS; op.mb = p->k_midbits; op.ms = p->k_midshift;
    ATKM_IRUN(dw ? "atkm_z_df" : "atkm_z_f64", 64 * H1 + 8.0 * g.Mz * g.My * g.Xh, 2.0 * g.My * g.Xh * ifftflops(g.Mz),
              op, p->iM[2], gz);
  }
  {
    IAtkmYI op;
    op.W2 = p->W2; op.W1 = p->W1; op.in = exp_cols(p->ex[2], gz); op.ex = exp_cols(p->ex[0], gy);
    op.Nx = g.Nx; op.Ny = g.Ny; op.My = g.My; op.XS = g.XS;
    ATKM_IRUN(dw ? "atkm_y_inv_df" : "atkm_y_inv_f64", 48 * H1, fy, op, p->iM[1], gy);
  }
  {
    IAtkmXI op;
    op.W1 = p->W1; op.phi = phi; op.wM = p->tw_x; op.in = exp_cols(p->ex[0], gy);
    op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl; op.XS = g.XS;
    ATKM_IRUN(dw ? "atkm_x_inv_df" : "atkm_x_inv_f64", 16 * H1 + 8 * N, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  }
  return cudaSuccess;
}

}  // namespace atkm
