// The y transforms of the binary64 preconditioner and of the 3D transform (see
// ipasses_p.cu).
#include "ipasses_impl.cuh"

namespace atkm {

template <int S, bool LINES>
cudaError_t ip_y(atkm_plan* p, const char* name, c64* buf, const ExpTab& in, int ex, const IPassGrid& gy, cudaStream_t st) {
  const Geo& g = p->g;
  IPY<S, LINES> op;
  op.Wk = buf; op.in = in; op.ex = exp_cols(p->ex[ex], gy); op.Nx = g.Nx; op.Ny = g.Ny;
  ATKM_IRUN(name, 32.0 * g.Nx * g.Ny * g.Nz, (double)g.Nz * g.Nx * ifftflops(g.Ny), op, p->iN[1], gy);
  return cudaSuccess;
}
template cudaError_t ip_y<-1, true>(atkm_plan*, const char*, c64*, const ExpTab&, int, const IPassGrid&, cudaStream_t);
template cudaError_t ip_y<1, false>(atkm_plan*, const char*, c64*, const ExpTab&, int, const IPassGrid&, cudaStream_t);
template cudaError_t ip_y<1, true>(atkm_plan*, const char*, c64*, const ExpTab&, int, const IPassGrid&, cudaStream_t);

}  // namespace atkm
