// The z pass of the binary64 H_phi f (see ipasses_h.cu), in a unit of its own
// so that the kernels compile in parallel.
#include "ipasses_impl.cuh"

namespace atkm {

namespace {
template <bool RED>
cudaError_t run(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  if (RED && h.f != h.phi) return cudaErrorInvalidValue;  // the sums are those of phi
  const Phys& ph = *h.ph;
  const IPassGrid &gx = h.gx, &gy = h.gy, &gz = h.gz;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const double pi = 3.14159265358979323846264338327950288, kz = pi / g.Lz;
  const double2* fin = reinterpret_cast<const double2*>(h.f);
  IHZ<RED> op;
  op.f = fin; op.phi = reinterpret_cast<const double2*>(h.phi); op.Phi = h.Phi; op.AX = p->T1; op.AY = p->T2;
  op.ix = exp_each_line(p->ex[3]); op.iy = exp_each_col(p->ex[4], g.Nx);
  op.Hf = reinterpret_cast<double2*>(h.Hf); op.kin = iaxt(p, 2).kinN; op.Nx = g.Nx; op.Ny = g.Ny; op.Nz = g.Nz;
  op.hx2 = iaxt(p, 0).hxc2; op.hy2 = iaxt(p, 1).hxc2; op.hz2 = iaxt(p, 2).hxc2;
  op.gx2 = ph.gx2; op.gy2 = ph.gy2; op.gz2 = ph.gz2; op.beta = ph.beta; op.lambda = ph.lambda;
  op.ck = 0.5 * kz * kz / g.Nz; op.same = h.f == h.phi;
  op.part = p->partials; op.pstride = gz.grid.x * gz.grid.y; op.sums_out = p->scal + red_slot + 4; op.cnt = p->cnt;
  ATKM_IRUN(dw ? "H_z_df" : "H_z_f64", (op.same ? 72 : 88) * N, 2.0 * g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
  return cudaSuccess;
}
}  // namespace

cudaError_t ih_z(atkm_plan* p, bool dw, const HArgs& h, int red_slot, cudaStream_t st) {
  return red_slot >= 0 ? run<true>(p, dw, h, red_slot, st) : run<false>(p, dw, h, red_slot, st);
}

}  // namespace atkm
