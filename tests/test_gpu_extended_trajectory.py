"""The 128x128x32 pancake of test_gpu_trajectories.py (gamma_z = 50, Omega =
0.8, eight seeded phase windings): 50 iterations against Algorithm 1 in 80 bits
(oracle/extended.py), kept in golden/trajectory_128x128x32.txt.  The binary64
oracle's own rounding is 1e-10 ... 3e-10 of E at the 50th iterate, so that it
cannot judge the last iterates to 1e-10; that trajectory moves by 2e-13 when
psi_0 is perturbed by one ulp.  Bars: E to 1e-10 (the parity bar of the solver),
to 1e-11 up to n = 40, before the iterates' instability sets in (every binary64
form agrees to 1e-12 there); the residual to 1e-6; the decisions equal."""
import os

import pytest
import torch

import atkm_workloads as W

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "trajectory_128x128x32.txt")


def test_fp64_trajectory_matches_extended_precision(lib):
    w, k = W.CONFIGS["cfg2_128x128x32"], 50
    plan, prm = lib.Plan(w.N, w.L, w.n), lib.make_params(w.gamma, w.beta, w.lam, w.Omega)
    psi = torch.from_numpy(W.initial_guess(w)).cuda()
    log = plan.pcg_ground_state(prm, psi, tol_residual=1e-8, max_iter=k, log_capacity=k + 2)["log"]
    rows = [line.split() for line in open(GOLDEN)]
    assert len(rows) == k
    for a, (n, E, res, halvings, reset, accepted) in zip(log, rows):
        assert a["n"] == int(n)
        assert abs(a["E"] - float(E)) <= (1e-11 if int(n) <= 40 else 1e-10) * abs(float(E)), (n, a["E"], E)
        assert abs(a["residual"] - float(res)) <= 1e-6 * float(res) + 1e-13, (n, a["residual"], res)
        assert (a["halvings"], bool(a["reset_to_sd"]), bool(a["accepted"])) == (
            int(halvings), reset == "1", accepted == "1"), n
