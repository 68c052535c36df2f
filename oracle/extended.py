"""Algorithm 1 of atkm_oracle with every array and scalar in extended precision
(numpy's long double: 80 bits on x86, 113 on Arm): TEST INFRASTRUCTURE ONLY.

The binary64 oracle's trajectory is itself good to about 1e-12 of E for the
first 40 iterations of the 128x128x32 workload and to 1e-10 ... 3e-10 at the
50th, where an instability of the iterates amplifies the rounding of its
transforms (with those alone in 80 bits the same code ends 5e-12 from here).
This one moves by 2e-13 when psi_0 is perturbed by one ulp.  The multiplier K and
psi_0 are the binary64 ones.

`python -m oracle.extended FILE` writes that workload's trajectory (an 80-bit
host, about ten minutes): one line an iteration with n, E, the residual, the
number of halvings, whether Step 4 (i) reset the direction, whether the step was
accepted."""
from __future__ import annotations

import importlib.util
import os
import sys

import numpy as np

LD, CLD = np.longdouble, np.clongdouble


def _module():
    """A copy of atkm_oracle of its own whose scalars are long doubles."""
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "atkm_oracle.py")
    spec = importlib.util.spec_from_file_location("oracle._atkm_oracle_extended", path)
    m = importlib.util.module_from_spec(spec)
    sys.modules[spec.name] = m  # the dataclasses look their module up
    spec.loader.exec_module(m)
    return m


def pcg_ground_state(N, L, n, gamma, beta, lam, Omega, psi0, max_iter):
    """atkm_oracle.pcg_ground_state(...) of these arguments, from psi0."""
    m = _module()
    plan = m.Plan(N, L, n)
    plan.K = plan.K.astype(LD)
    g = plan.grid
    for a in ("x", "y", "z", "nu_x", "nu_y", "nu_z"):
        setattr(g, a, getattr(g, a).astype(LD))
    g.nu2 = g.nu_x ** 2 + g.nu_y ** 2 + g.nu_z ** 2
    g.hvol = LD(g.h[0]) * LD(g.h[1]) * LD(g.h[2])

    def convolution(rho, mult):
        nz, ny, nx = rho.shape
        pad = np.zeros((2 * nz, 2 * ny, 2 * nx), dtype=CLD)
        pad[:nz, :ny, :nx] = rho
        return np.real(np.fft.ifftn(mult * np.fft.fftn(pad))[:nz, :ny, :nx]).copy()

    class Math:
        sqrt, cos, sin = (staticmethod(lambda v, f=f: f(LD(v))) for f in (np.sqrt, np.cos, np.sin))

    m.truncated_convolution, m.math, m.float = convolution, Math, LD
    prm = m.Params(tuple(LD(v) for v in gamma), LD(beta), LD(lam), LD(Omega))
    return m.pcg_ground_state(plan, prm, psi0.astype(CLD), m.PcgOptions(max_iter=max_iter))


def main(path):
    import atkm_workloads as W
    w, k = W.CONFIGS["cfg2_128x128x32"], 50
    log = pcg_ground_state(w.N, w.L, w.n, w.gamma, w.beta, w.lam, w.Omega, W.initial_guess(w), k).log[:k]
    with open(path, "w") as fh:
        for e in log:
            fh.write(f"{e['n']} {float(e['E'])!r} {float(e['residual'])!r} {e['halvings']} {int(e['reset'])} "
                     f"{int(e['accepted'])}\n")


if __name__ == "__main__":
    main(sys.argv[1])
