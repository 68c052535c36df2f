// The binary64 H_phi f: three integer passes (iops.cuh).  The x and y passes
// leave their parts in T1 and T2, the z pass adds them up.  Nothing here is
// shared with the ATKM passes, so that the two may run side by side.
#include "ipasses_impl.cuh"

namespace atkm {

cudaError_t launch_H64(atkm_plan* p, bool dw, const Phys& ph, const double* f, const double* phi, const double* Phi,
                       double* Hf, int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  HArgs h{&ph, f, phi, Phi, Hf, ipass_grid(p, g.Nx, true, (long)g.Nz * g.Ny, 0, 0),
          ipass_grid(p, g.Ny, false, 0, g.Nx, g.Nz), ipass_grid(p, g.Nz, false, 0, g.Nx, g.Ny)};
  cudaError_t e = ih_x(p, dw, h, red_slot, st);
  if (e == cudaSuccess) e = ih_y(p, dw, h, red_slot, st);
  if (e == cudaSuccess) e = ih_z(p, dw, h, red_slot, st);
  return e;
}

}  // namespace atkm
