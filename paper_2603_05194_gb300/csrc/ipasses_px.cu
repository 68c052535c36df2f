// The x passes of the binary64 preconditioner (see ipasses_p.cu), in a unit of
// their own so that the kernels compile in parallel.
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t ip_xf(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                  const double* Phi, const IPassGrid& gx, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  const AxT ax = iaxt(p, 0), ay = iaxt(p, 1), az = iaxt(p, 2);
  IPXF op;
  op.r = reinterpret_cast<const double2*>(r); op.phi = reinterpret_cast<const double2*>(phi); op.Phi = Phi;
  op.Wk = p->T1; op.Pw = p->Pw; op.ex = exp_lines(p->ex[0], gx);
  op.hx2 = ax.hxc2; op.hy2 = ay.hxc2; op.hz2 = az.hxc2;
  op.gx2 = ph.gx2; op.gy2 = ph.gy2; op.gz2 = ph.gz2; op.beta = ph.beta; op.alam = fabs(ph.lambda);
  op.alpha = alpha_dev; op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
  ATKM_IRUN("P_x_fwd_f64", 64.0 * nl * g.Nx, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  return cudaSuccess;
}

cudaError_t ip_xi(atkm_plan* p, double* Pr, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st) {
  const Geo& g = p->g;
  const int nl = g.Nz * g.Ny;
  IPXI op;
  op.Wk = p->T1; op.Pw = p->Pw; op.Pr = reinterpret_cast<double2*>(Pr); op.in = exp_cols(p->ex[0], gy);
  op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
  ATKM_IRUN("P_x_inv_f64", 40.0 * nl * g.Nx, (double)nl * ifftflops(g.Nx), op, p->iN[0], gx);
  return cudaSuccess;
}

}  // namespace atkm
