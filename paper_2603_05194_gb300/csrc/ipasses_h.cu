// The binary64 H_phi f: three integer passes (iops.cuh).
#include "ipasses_impl.cuh"

namespace atkm {

namespace {
template <bool RED>
cudaError_t run_H(atkm_plan* p, bool dw, const Phys& ph, const double* f, const double* phi, const double* Phi, double* Hf,
                  int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  const int r = dw ? 2 : 0;
  const int nl = g.Nz * g.Ny;
  const double N = (double)g.Nx * g.Ny * g.Nz;
  const double pi = 3.14159265358979323846264338327950288;
  const double kx = pi / g.Lx, ky = pi / g.Ly, kz = pi / g.Lz;
  const IPassGrid gx = ipass_grid(p, r, g.Nx, true, nl, 0, 0);
  const IPassGrid gy = ipass_grid(p, r, g.Ny, false, 0, g.Nx, g.Nz);
  const IPassGrid gz = ipass_grid(p, r, g.Nz, false, 0, g.Nx, g.Ny);
  c64* AX = p->T1;
  c64* AY = p->W2;  // free outside the ATKM passes, and at least as large as the grid
  const double2* fin = reinterpret_cast<const double2*>(f);
  cudaError_t e;
  {
    IHX<RED> op;
    op.f = fin; op.A = AX; op.ex = exp_lines(p->ex[0], gx); op.Nx = g.Nx; op.Ny = g.Ny; op.nl = nl;
    op.ck = 0.5 * kx * kx / g.Nx; op.cr = ph.Omega * kx / g.Nx;
    op.kin = iaxt(p, 0).kinN; op.nu = iaxt(p, 0).nuN; op.Om = ph.Omega; op.Ly = g.Ly; op.hy = g.hy;
    op.part = p->partials; op.pstride = gx.grid.x;
    ATKM_IRUN(dw ? "H_x_df" : "H_x_f64", 32 * N, 2.0 * nl * ifftflops(g.Nx), op, p->iN[0], gx);
    if (RED && (e = launch_finalize(p, 2, op.pstride, red_slot, st)) != cudaSuccess) return e;
  }
  {
    IHY<RED> op;
    op.f = fin; op.A = AY; op.ex = exp_cols(p->ex[1], gy); op.Nx = g.Nx; op.Ny = g.Ny;
    op.ck = 0.5 * ky * ky / g.Ny; op.cr = -ph.Omega * ky / g.Ny;
    op.kin = iaxt(p, 1).kinN; op.nu = iaxt(p, 1).nuN; op.Om = ph.Omega; op.Lx = g.Lx; op.hx = g.hx;
    op.part = p->partials; op.pstride = gy.grid.x * gy.grid.y;
    ATKM_IRUN(dw ? "H_y_df" : "H_y_f64", 32 * N, 2.0 * g.Nz * g.Nx * ifftflops(g.Ny), op, p->iN[1], gy);
    if (RED && (e = launch_finalize(p, 2, op.pstride, red_slot + 2, st)) != cudaSuccess) return e;
  }
  {
    IHZ<RED> op;
    op.f = fin; op.phi = reinterpret_cast<const double2*>(phi); op.Phi = Phi; op.AX = AX; op.AY = AY;
    op.ix = exp_lines(p->ex[0], gx); op.iy = exp_cols(p->ex[1], gy);
    op.Hf = reinterpret_cast<double2*>(Hf); op.kin = iaxt(p, 2).kinN; op.Nx = g.Nx; op.Ny = g.Ny; op.Nz = g.Nz;
    op.hx2 = iaxt(p, 0).hxc2; op.hy2 = iaxt(p, 1).hxc2; op.hz2 = iaxt(p, 2).hxc2;
    op.gx2 = ph.gx2; op.gy2 = ph.gy2; op.gz2 = ph.gz2; op.beta = ph.beta; op.lambda = ph.lambda;
    op.ck = 0.5 * kz * kz / g.Nz; op.same = f == phi;
    op.part = p->partials; op.pstride = gz.grid.x * gz.grid.y;
    ATKM_IRUN(dw ? "H_z_df" : "H_z_f64", (op.same ? 72 : 88) * N, 2.0 * g.Ny * g.Nx * ifftflops(g.Nz), op, p->iN[2], gz);
    if (RED && (e = launch_finalize(p, 6, op.pstride, red_slot + 4, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_H64(atkm_plan* p, bool dw, const Phys& ph, const double* f, const double* phi, const double* Phi,
                       double* Hf, int red_slot, cudaStream_t st) {
  return red_slot >= 0 ? run_H<true>(p, dw, ph, f, phi, Phi, Hf, red_slot, st)
                       : run_H<false>(p, dw, ph, f, phi, Phi, Hf, red_slot, st);
}

}  // namespace atkm
