// The y passes of the binary64 dipolar potential (see ipasses_a.cu).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t iatkm_yf(atkm_plan* p, bool dw, const IPassGrid& gx, const IPassGrid& gy, cudaStream_t st) {
  const Geo& g = p->g;
  IAtkmYF op;
  op.W1 = p->W1; op.W2 = p->W2; op.in = exp_lines(p->ex[0], gx); op.ex = exp_cols(p->ex[1], gy);
  op.Nx = g.Nx; op.Ny = g.Ny; op.My = g.My; op.XS = g.XS;
  ATKM_IRUN(dw ? "atkm_y_fwd_df" : "atkm_y_fwd_f64", 48.0 * g.Nz * g.Ny * g.Xh, (double)g.Nz * g.Xh * ifftflops(g.My), op,
            p->iM[1], gy);
  return cudaSuccess;
}

cudaError_t iatkm_yi(atkm_plan* p, bool dw, const IPassGrid& gz, const IPassGrid& gy, cudaStream_t st) {
  const Geo& g = p->g;
  IAtkmYI op;
  op.W2 = p->W2; op.W1 = p->W1; op.in = exp_cols(p->ex[2], gz); op.ex = exp_cols(p->ex[0], gy);
  op.Nx = g.Nx; op.Ny = g.Ny; op.My = g.My; op.XS = g.XS;
  ATKM_IRUN(dw ? "atkm_y_inv_df" : "atkm_y_inv_f64", 48.0 * g.Nz * g.Ny * g.Xh, (double)g.Nz * g.Xh * ifftflops(g.My), op,
            p->iM[1], gy);
  return cudaSuccess;
}

}  // namespace atkm
