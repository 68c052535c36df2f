"""The FP32 form's iterates bit for bit: ten iterations of pcg_ground_state with
precision 1, all in the FP32 phase, from start states formed by IEEE additions,
multiplications and divisions alone (the same on every host), against the values
in golden/f32_form_256x256x64.txt.  Those were taken with the reductions' former
two-kernel form on a GB300 (152 SMs; the order of a grid sum follows from the
number of SMs).  A sum that is added up in another order moves the last bit of a
norm, and an iterate then by about 1e-7 at the points where the rounding to
binary32 falls the other way."""
import hashlib
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "f32_form_256x256x64.txt")
N, L, AXIS = (256, 256, 64), (16.0, 16.0, 1.5), (0.6, 0.0, 0.8)
STATES, ITERS = 10, 10


def start_state(i):
    """A cloud 1 / (1 + q)^2, q a quadratic form, with three vortices."""
    ax = [-L[a] + (2.0 * L[a] / N[a]) * np.arange(N[a]) for a in range(3)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    q = (x * x + 1.25 * y * y) / (10.0 + i) + (8.0 + 0.5 * i) * z * z
    env = 1.0 / ((1.0 + q) * (1.0 + q))
    re, im = env, 0.0 * env
    for v in range(3):
        dx, dy = x - (1.5 * v - 1.0 - 0.125 * i), y + (0.75 * v - 0.5 + 0.25 * i)
        re, im = re * dx - im * dy, re * dy + im * dx
    s = 1.0 + x * x + y * y
    psi = np.empty((N[2], N[1], N[0]), dtype=np.complex128)
    psi.real, psi.imag = re / s, im / s
    return psi


def run_states(lib):
    """One line a state: its number, E, mu and the residual as hexadecimal
    floats, the SHA-256 of psi."""
    plan = lib.Plan(N, L, AXIS, f32=True)
    prm = lib.make_params((1.0, 1.2, 30.0), 500.0, 200.0, 0.8)
    out = []
    for i in range(STATES):
        psi = torch.from_numpy(start_state(i)).cuda()
        res = plan.pcg_ground_state(prm, psi, max_iter=ITERS, precision=lib.PRECISION_F32_F64)
        assert res["iters"] == ITERS and res["f32_iters"] == ITERS
        h = hashlib.sha256(psi.cpu().numpy().tobytes()).hexdigest()
        out.append(f"{i} {res['E'].hex()} {res['mu'].hex()} {res['residual'].hex()} {h}")
    return out


def test_f32_form_bits(lib):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip(f"{sms} SMs: the sums are added up in another order")
    assert run_states(lib) == open(GOLDEN).read().split("\n")[:STATES]
