// The y pass of the binary64 H_phi f (see ipasses_h.cu), in a unit of its own
// so that the kernels compile in parallel.
#include "ipasses_impl.cuh"

namespace atkm {

namespace {
template <bool RED>
cudaError_t run(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  const Phys& ph = *h.ph;
  const IPassGrid &gy = h.gy;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const double pi = 3.14159265358979323846264338327950288, ky = pi / g.Ly;
  const double2* fin = reinterpret_cast<const double2*>(h.f);
  IHY<RED> op;
  op.f = fin; op.A = p->T2; op.ex = exp_each_col(p->ex[4], g.Nx); op.Nx = g.Nx; op.Ny = g.Ny;
  op.ck = 0.5 * ky * ky / g.Ny; op.cr = -ph.Omega * ky / g.Ny;
  op.kin = iaxt(p, 1).kinN; op.nu = iaxt(p, 1).nuN; op.Om = ph.Omega; op.Lx = g.Lx; op.hx = g.hx;
  op.part = p->partials; op.pstride = gy.grid.x * gy.grid.y; op.sums_out = p->scal + red_slot + 2; op.cnt = p->cnt;
  ATKM_IRUN(dw ? "H_y_df" : "H_y_f64", 32 * N, 2.0 * g.Nz * g.Nx * ifftflops(g.Ny), op, p->iN[1], gy);
  return cudaSuccess;
}
}  // namespace

cudaError_t ih_y(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  return red_slot >= 0 ? run<true>(p, dw, h, red_slot, st) : run<false>(p, dw, h, red_slot, st);
}

}  // namespace atkm
