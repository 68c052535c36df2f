// The x pass of the binary64 H_phi f (see ipasses_h.cu), in a unit of its own
// so that the kernels compile in parallel.
#include "ipasses_impl.cuh"

namespace atkm {

namespace {
template <bool RED>
cudaError_t run(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  const Phys& ph = *h.ph;
  const IPassGrid &gx = h.gx;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const double pi = 3.14159265358979323846264338327950288, kx = pi / g.Lx;
  const double2* fin = reinterpret_cast<const double2*>(h.f);
  IHX<RED> op;
  op.f = fin; op.A = p->T1; op.ex = exp_each_line(p->ex[3]); op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
  op.ck = 0.5 * kx * kx / g.Nx; op.cr = ph.Omega * kx / g.Nx;
  op.kin = iaxt(p, 0).kinN; op.nu = iaxt(p, 0).nuN; op.Om = ph.Omega; op.Ly = g.Ly; op.hy = g.hy;
  op.part = p->partials; op.pstride = gx.grid.x; op.sums_out = p->scal + red_slot; op.cnt = p->cnt;
  ATKM_IRUN(dw ? "H_x_df" : "H_x_f64", 32 * N, 2.0 * nl * ifftflops(g.Nx), op, p->iN[0], gx);
  return cudaSuccess;
}
}  // namespace

cudaError_t ih_x(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  return red_slot >= 0 ? run<true>(p, dw, h, red_slot, st) : run<false>(p, dw, h, red_slot, st);
}

}  // namespace atkm
