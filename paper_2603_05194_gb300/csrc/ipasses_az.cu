// The z pass of the binary64 dipolar potential (see ipasses_a.cu).
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t iatkm_z(atkm_plan* p, bool dw, const IPassGrid& gy, const IPassGrid& gz, cudaStream_t st) {
  const Geo& g = p->g;
  IAtkmZ op;
  op.W2 = p->W2; op.K = p->Kz; op.in = exp_cols(p->ex[1], gy); op.ex = exp_cols(p->ex[2], gz);
  op.Nx = g.Nx; op.Nz = g.Nz; op.My = g.My; op.XS = g.XS; op.mb = p->k_midbits; op.ms = p->k_midshift;
  ATKM_IRUN(dw ? "atkm_z_df" : "atkm_z_f64", 64.0 * g.Nz * g.Ny * g.Xh + 8.0 * g.Mz * g.My * g.Xh,
            2.0 * g.My * g.Xh * ifftflops(g.Mz), op, p->iM[2], gz);
  return cudaSuccess;
}

}  // namespace atkm
