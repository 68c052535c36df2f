"""The extended-precision oracle against the binary64 one it is built from, and
its committed trajectory against the binary64 oracle's first iterates."""
import os

import atkm_workloads as W
import oracle as O
from oracle import extended as X


def test_extended_oracle_follows_the_binary64_one():
    """32x32x16, eight iterations: E to 1e-13 (the binary64 rounding of a few
    iterations), the same decisions."""
    w, k = W.CONFIGS["cfg1_32x32x16"], 8
    psi0 = W.initial_guess(w)
    a = O.pcg_ground_state(O.Plan(w.N, w.L, w.n), O.Params(w.gamma, w.beta, w.lam, w.Omega), psi0,
                           O.PcgOptions(max_iter=k))
    b = X.pcg_ground_state(w.N, w.L, w.n, w.gamma, w.beta, w.lam, w.Omega, psi0, k)
    assert b.phi.dtype == X.CLD
    for x, y in zip(a.log[:k], b.log[:k]):
        assert abs(x["E"] - float(y["E"])) <= 1e-13 * abs(x["E"]), x["n"]
        assert abs(x["residual"] - float(y["residual"])) <= 1e-10 * x["residual"], x["n"]
        assert (x["halvings"], x["reset"], x["accepted"]) == (y["halvings"], y["reset"], y["accepted"])


def test_committed_trajectory():
    """The first two iterates of golden/trajectory_128x128x32.txt."""
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "trajectory_128x128x32.txt")
    rows = [line.split() for line in open(path)]
    w = W.CONFIGS["cfg2_128x128x32"]
    ref = O.pcg_ground_state(O.Plan(w.N, w.L, w.n), O.Params(w.gamma, w.beta, w.lam, w.Omega), W.initial_guess(w),
                             O.PcgOptions(max_iter=1))
    for e, row in zip(ref.log, rows):
        assert abs(e["E"] - float(row[1])) <= 1e-13 * e["E"] and abs(e["residual"] - float(row[2])) <= 1e-10 * e["residual"]
