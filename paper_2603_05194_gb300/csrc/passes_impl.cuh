// Launchers of the three spectral operators in FP32 (instantiated in
// passes_f32*.cu).
#pragma once

#include <math.h>

#include "ops.cuh"

namespace atkm {

inline double fftflops(double n) { return 5.0 * n * log2(n); }

#define ATKM_RUN(NAME, BYTES, FLOPS, OP, FLEN, PG)              \
  do {                                                         \
    prof_begin(p, NAME, BYTES, FLOPS, st);                     \
    cudaError_t e_ = run_pass<R>(OP, FLEN, PG, st);            \
    prof_end(p, st);                                           \
    count_launches(1);                                         \
    if (e_ != cudaSuccess) return e_;                          \
  } while (0)

// What every ATKM pass needs of the plan: workspaces, constants, the byte and
// flop counts of the profiler.
template <typename R> struct AtkmCtx {
  const Geo* g;
  cx<R>* W1;
  cx<R>* W2;
  const R* K;
  Cst<R> c;
  const cx<R>* twM;
  double N, s, H1, fx, fy, fz, kb;
  long nl;
};
template <typename R> inline AtkmCtx<R> atkm_ctx(atkm_plan* p) {
  AtkmCtx<R> x;
  const Geo& g = p->g;
  x.g = &g;
  x.W1 = p->W1f;
  x.W2 = p->W2f;
  x.K = p->U0f;
  x.c = make_cst<R>(g);
  x.twM = tw_table_host<R>(p->fM[0]);
  x.N = (double)g.Nx * g.Ny * g.Nz;
  x.s = (double)sizeof(cx<R>);
  x.H1 = (double)g.Nz * g.Ny * g.Xh;  // half-spectrum elements of W1
  x.fx = (double)g.Nz * g.Ny * fftflops(g.Nx);
  x.fy = (double)g.Nz * g.Xh * fftflops(g.My);
  x.fz = 2.0 * g.My * g.Xh * fftflops(g.Mz);
  // multiplier: the U0 octant
  x.kb = (double)sizeof(R) * (g.Nx + 1) * (g.Ny + 1) * (g.Nz + 1);
  x.nl = (long)g.Nz * g.Ny;
  return x;
}

// The five passes of one ATKM evaluation, each a function of its own (same
// signature) so that heavy instantiations can compile in separate
// translation units.
// x forward (real data: complex FFT of length Nx + post-twist)
template <typename R>
cudaError_t atkm_pass_xf(atkm_plan* p, int mode, const double* a, const double* b, double*, cudaStream_t st) {
  const AtkmCtx<R> x = atkm_ctx<R>(p);
  const Geo& g = *x.g;
  if (!x.W1) return cudaErrorInvalidValue;
  const double inb = mode == SRC_RHO ? 8.0 : (mode == SRC_PSI ? 16.0 : 32.0);
  const PassGrid gx = pass_grid<R>(p, g.Nx, true, x.nl, 0, 0);
  const char* nx = "atkm_x_fwd_f32";
  if (mode == SRC_RHO) {
    OpAtkmXF<R, SRC_RHO> op; op.a = a; op.b = b; op.W1 = x.W1; op.twM = x.twM; op.c = x.c; op.XS = g.XS;
    ATKM_RUN(nx, inb * x.N + x.H1 * x.s, x.fx, op, p->fN[0], gx);
  } else if (mode == SRC_PSI) {
    OpAtkmXF<R, SRC_PSI> op; op.a = a; op.b = b; op.W1 = x.W1; op.twM = x.twM; op.c = x.c; op.XS = g.XS;
    ATKM_RUN(nx, inb * x.N + x.H1 * x.s, x.fx, op, p->fN[0], gx);
  } else {
    OpAtkmXF<R, SRC_PAIR> op; op.a = a; op.b = b; op.W1 = x.W1; op.twM = x.twM; op.c = x.c; op.XS = g.XS;
    ATKM_RUN(nx, inb * x.N + x.H1 * x.s, x.fx, op, p->fN[0], gx);
  }
  return cudaSuccess;
}

// y forward on the Nx + 1 half-spectrum columns
template <typename R>
cudaError_t atkm_pass_yf(atkm_plan* p, int, const double*, const double*, double*, cudaStream_t st) {
  const AtkmCtx<R> x = atkm_ctx<R>(p);
  const Geo& g = *x.g;
  if (!x.W1 || !x.W2) return cudaErrorInvalidValue;
  const PassGrid gy = pass_grid<R>(p, g.My, false, 0, g.Xh, g.Nz);
  OpAtkmYF<R> op; op.W1 = x.W1; op.W2 = x.W2; op.c = x.c; op.XS = g.XS;
  ATKM_RUN("atkm_y_fwd_f32", 3 * x.H1 * x.s, x.fy, op, p->fM[1], gy);
  return cudaSuccess;
}

// z forward * K_sym * inverse
template <typename R>
cudaError_t atkm_pass_z(atkm_plan* p, int, const double*, const double*, double*, cudaStream_t st) {
  const AtkmCtx<R> x = atkm_ctx<R>(p);
  const Geo& g = *x.g;
  if (!x.W2 || !x.K) return cudaErrorInvalidValue;
  OpAtkmZ<R> op; op.W2 = x.W2; op.U0 = x.K; op.c = x.c; op.XS = g.XS;
  op.n0 = (R)p->n[0]; op.n1 = (R)p->n[1]; op.n2 = (R)p->n[2];
  op.invM = (R)(0.5 / ((double)g.Mx * g.My * g.Mz));  // with the x forward pass's 1/2 (OpAtkmXF)
  const PassGrid pg = pass_grid<R>(p, g.Mz, false, 0, g.Xh, g.My);
  ATKM_RUN("atkm_z_f32", 4 * x.H1 * x.s + x.kb, x.fz, op, p->fM[2], pg);
  return cudaSuccess;
}

// y inverse
template <typename R>
cudaError_t atkm_pass_yi(atkm_plan* p, int, const double*, const double*, double*, cudaStream_t st) {
  const AtkmCtx<R> x = atkm_ctx<R>(p);
  const Geo& g = *x.g;
  if (!x.W1 || !x.W2) return cudaErrorInvalidValue;
  const PassGrid gy = pass_grid<R>(p, g.My, false, 0, g.Xh, g.Nz);
  OpAtkmYI<R> op; op.W2 = x.W2; op.W1 = x.W1; op.c = x.c; op.XS = g.XS;
  ATKM_RUN("atkm_y_inv_f32", 3 * x.H1 * x.s, x.fy, op, p->fM[1], gy);
  return cudaSuccess;
}

// x inverse (C2R) + crop
template <typename R>
cudaError_t atkm_pass_xi(atkm_plan* p, int, const double*, const double*, double* phi, cudaStream_t st) {
  const AtkmCtx<R> x = atkm_ctx<R>(p);
  const Geo& g = *x.g;
  if (!x.W1) return cudaErrorInvalidValue;
  const PassGrid gx = pass_grid<R>(p, g.Nx, true, x.nl, 0, 0);
  OpAtkmXI<R> op; op.W1 = x.W1; op.phi = phi; op.twM = x.twM; op.c = x.c; op.XS = g.XS;
  ATKM_RUN("atkm_x_inv_f32", x.H1 * x.s + 8 * x.N, x.fx, op, p->fN[0],
           gx);
  return cudaSuccess;
}

template <typename R>
cudaError_t launch_atkm(atkm_plan* p, int mode, const double* a, const double* b, double* phi, cudaStream_t st) {
  if (!p->W1f || !p->W2f || !p->U0f) return cudaErrorInvalidValue;
  cudaError_t e = atkm_pass_xf<R>(p, mode, a, b, phi, st);
  if (e == cudaSuccess) e = atkm_pass_yf<R>(p, mode, a, b, phi, st);
  if (e == cudaSuccess) e = atkm_pass_z<R>(p, mode, a, b, phi, st);
  if (e == cudaSuccess) e = atkm_pass_yi<R>(p, mode, a, b, phi, st);
  if (e == cudaSuccess) e = atkm_pass_xi<R>(p, mode, a, b, phi, st);
  return e;
}

// One axis pass of H_phi f (a function of its own so that heavy
// instantiations can be compiled in separate translation units).
template <typename R>
cudaError_t h_pass_x(atkm_plan* p, const Phys& ph, const double* f, const double*, const double*, double*, int red_slot,
                    cudaStream_t st) {
  const Geo& g = p->g;
  cx<R>* acc = p->T1f;
  if (!acc) return cudaErrorInvalidValue;
  const bool red = red_slot >= 0;
  const Cst<R> c = make_cst<R>(g);
  const PhysR<R> pr = make_physr<R>(ph);
  const double2* fin = reinterpret_cast<const double2*>(f);
  const double N = (double)g.Nx * g.Ny * g.Nz, s = (double)sizeof(cx<R>);
  const long nl = (long)g.Nz * g.Ny;
  // x
  {
    const PassGrid pg = pass_grid<R>(p, g.Nx, true, nl, 0, 0);
    const double fl = 2.0 * nl * fftflops(g.Nx);
    const char* n = "H_x_f32";
    if (red) {
      OpHX<R, true> op; op.f = fin; op.acc = acc; op.c = c; op.Omega = pr.Omega;
      op.part = p->partials; op.pstride = pg.grid.x * pg.grid.y;
      op.sums = p->scal + red_slot + 0; op.cnt = p->cnt;
      ATKM_RUN(n, 16 * N + N * s, fl, op, p->fN[0], pg);
    } else {
      OpHX<R, false> op; op.f = fin; op.acc = acc; op.c = c; op.Omega = pr.Omega;
      ATKM_RUN(n, 16 * N + N * s, fl, op, p->fN[0], pg);
    }
  }
  return cudaSuccess;
}

template <typename R>
cudaError_t h_pass_y(atkm_plan* p, const Phys& ph, const double* f, const double*, const double*, double*, int red_slot,
                    cudaStream_t st) {
  const Geo& g = p->g;
  cx<R>* acc = p->T1f;
  if (!acc) return cudaErrorInvalidValue;
  const bool red = red_slot >= 0;
  const Cst<R> c = make_cst<R>(g);
  const PhysR<R> pr = make_physr<R>(ph);
  const double2* fin = reinterpret_cast<const double2*>(f);
  const double N = (double)g.Nx * g.Ny * g.Nz, s = (double)sizeof(cx<R>);
  // y
  {
    const PassGrid pg = pass_grid<R>(p, g.Ny, false, 0, g.Nx, g.Nz);
    const double fl = 2.0 * g.Nz * g.Nx * fftflops(g.Ny);
    const char* n = "H_y_f32";
    if (red) {
      OpHY<R, true> op; op.f = fin; op.acc = acc; op.c = c; op.Omega = pr.Omega;
      op.part = p->partials; op.pstride = pg.grid.x * pg.grid.y;
      op.sums = p->scal + red_slot + 2; op.cnt = p->cnt;
      ATKM_RUN(n, 16 * N + 2 * N * s, fl, op, p->fN[1], pg);
    } else {
      OpHY<R, false> op; op.f = fin; op.acc = acc; op.c = c; op.Omega = pr.Omega;
      ATKM_RUN(n, 16 * N + 2 * N * s, fl, op, p->fN[1], pg);
    }
  }
  return cudaSuccess;
}

template <typename R>
cudaError_t h_pass_z(atkm_plan* p, const Phys& ph, const double* f, const double* phi, const double* Phi, double* Hf,
                    int red_slot, cudaStream_t st) {
  const Geo& g = p->g;
  cx<R>* acc = p->T1f;
  if (!acc) return cudaErrorInvalidValue;
  const bool red = red_slot >= 0;
  const Cst<R> c = make_cst<R>(g);
  const PhysR<R> pr = make_physr<R>(ph);
  const double2* fin = reinterpret_cast<const double2*>(f);
  const double2* pin = reinterpret_cast<const double2*>(phi);
  double2* out = reinterpret_cast<double2*>(Hf);
  const double N = (double)g.Nx * g.Ny * g.Nz, s = (double)sizeof(cx<R>);
  // z + pointwise
  {
    const PassGrid pg = pass_grid<R>(p, g.Nz, false, 0, g.Nx, g.Ny);
    const double fl = 2.0 * g.Ny * g.Nx * fftflops(g.Nz);
    const char* n = "H_z_f32";
    if (red) {
      OpHZ<R, true> op; op.f = fin; op.phi = pin; op.Phi = Phi; op.acc = acc; op.Hf = out; op.c = c; op.ph = pr;
      op.same = fin == pin;
      op.part = p->partials; op.pstride = pg.grid.x * pg.grid.y;
      op.sums = p->scal + red_slot + 4; op.cnt = p->cnt;
      ATKM_RUN(n, (op.same ? 40 : 56) * N + N * s, fl, op, p->fN[2], pg);
    } else {
      OpHZ<R, false> op; op.f = fin; op.phi = pin; op.Phi = Phi; op.acc = acc; op.Hf = out; op.c = c; op.ph = pr;
      op.same = fin == pin;
      ATKM_RUN(n, (op.same ? 40 : 56) * N + N * s, fl, op, p->fN[2], pg);
    }
  }
  return cudaSuccess;
}

template <typename R>
cudaError_t launch_H(atkm_plan* p, const Phys& ph, const double* f, const double* phi, const double* Phi, double* Hf,
                     int red_slot, cudaStream_t st) {
  cudaError_t e = h_pass_x<R>(p, ph, f, phi, Phi, Hf, red_slot, st);
  if (e == cudaSuccess) e = h_pass_y<R>(p, ph, f, phi, Phi, Hf, red_slot, st);
  if (e == cudaSuccess) e = h_pass_z<R>(p, ph, f, phi, Phi, Hf, red_slot, st);
  return e;
}

template <typename R>
cudaError_t launch_precond(atkm_plan* p, const Phys& ph, const double* alpha_dev, const double* r, const double* phi,
                           const double* Phi, double* Pr, cudaStream_t st) {
  const Geo& g = p->g;
  cx<R>* Wk = p->T1f;
  if (!Wk) return cudaErrorInvalidValue;
  const Cst<R> c = make_cst<R>(g);
  const PhysR<R> pr = make_physr<R>(ph);
  const double N = (double)g.Nx * g.Ny * g.Nz, s = (double)sizeof(cx<R>);
  const long nl = (long)g.Nz * g.Ny;
  const double fx = (double)nl * fftflops(g.Nx), fy = (double)g.Nz * g.Nx * fftflops(g.Ny);
  const PassGrid gx = pass_grid<R>(p, g.Nx, true, nl, 0, 0);
  const PassGrid gy = pass_grid<R>(p, g.Ny, false, 0, g.Nx, g.Nz);
  const PassGrid gz = pass_grid<R>(p, g.Nz, false, 0, g.Nx, g.Ny);
  {
    OpPXF<R> op; op.r = reinterpret_cast<const double2*>(r); op.phi = reinterpret_cast<const double2*>(phi);
    op.Phi = Phi; op.Wk = Wk; op.c = c; op.ph = pr; op.alpha = alpha_dev;
    const double by = 40.0 * N + N * s;
    ATKM_RUN("P_x_fwd_f32", by, fx, op, p->fN[0], gx);
  }
  {
    OpPY<R, -1> op; op.Wk = Wk; op.c = c;
    ATKM_RUN("P_y_f32", 2 * N * s, fy, op, p->fN[1], gy);
  }
  {
    OpPZ<R> op; op.Wk = Wk; op.c = c; op.alpha = alpha_dev;
    ATKM_RUN("P_z_f32", 2 * N * s, 2.0 * g.Ny * g.Nx * fftflops(g.Nz), op, p->fN[2], gz);
  }
  {
    OpPY<R, 1> op; op.Wk = Wk; op.c = c;
    ATKM_RUN("P_y_f32", 2 * N * s, fy, op, p->fN[1], gy);
  }
  {
    OpPXI<R> op; op.Wk = Wk; op.phi = reinterpret_cast<const double2*>(phi); op.Phi = Phi;
    op.Pr = reinterpret_cast<double2*>(Pr); op.c = c; op.ph = pr; op.alpha = alpha_dev;
    const double by = 40.0 * N + N * s;
    ATKM_RUN("P_x_inv_f32", by, fx, op, p->fN[0], gx);
  }
  return cudaSuccess;
}

#undef ATKM_RUN

}  // namespace atkm
