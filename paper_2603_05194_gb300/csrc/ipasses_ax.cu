// The x passes of the binary64 dipolar potential (see ipasses_a.cu), in a unit
// of their own so that the kernels compile in parallel.
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

cudaError_t iatkm_xf(atkm_plan* p, bool dw, int mode, const double* a, const double* b, const IPassGrid& gx,
                     cudaStream_t st) {
  const char* nx = dw ? "atkm_x_fwd_df" : "atkm_x_fwd_f64";
  if (mode == SRC_RHO) return run_xf<SRC_RHO>(p, nx, 8.0, a, b, gx, st);
  if (mode == SRC_PSI) return run_xf<SRC_PSI>(p, nx, 16.0, a, b, gx, st);
  return run_xf<SRC_PAIR>(p, nx, 32.0, a, b, gx, st);
}

cudaError_t iatkm_xi(atkm_plan* p, bool dw, double* phi, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz, H1 = (double)nl * g.Xh;
  IAtkmXI op;
  op.W1 = p->W1; op.phi = phi; op.wM = p->tw_x; op.in = exp_cols(p->ex[0], gy);
  op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl; op.XS = g.XS;
  ATKM_IRUN(dw ? "atkm_x_inv_df" : "atkm_x_inv_f64", 16 * H1 + 8 * N, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  return cudaSuccess;
}

}  // namespace atkm
