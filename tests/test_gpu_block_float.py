"""The binary64 operators' integer (block-floating-point) passes where that
arithmetic can go wrong: the smallest and the composite line lengths, inputs
whose scale lies far from one or varies over hundreds of orders of magnitude,
zeros, and NaNs.  Bars: relative 2-norm 1e-13 against the oracle (its own
rounding is below 1e-15 here; the integer passes carry 58 bits), bitwise where
the arithmetic is exact under a power of two."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import atkm_workloads as W
import oracle as O

pytestmark = pytest.mark.gpu
GAMMA, BETA, LAM, OM = (1.0, 1.3, 3.0), 30.0, 12.0, 0.4


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


def rel2(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def convolution(plan, rho):
    """The padded convolution with the plan's own multiplier (its quadrature is
    compared with the oracle's elsewhere), by numpy's transforms."""
    nz, ny, nx = rho.shape
    pad = np.zeros((2 * nz, 2 * ny, 2 * nx))
    pad[:nz, :ny, :nx] = rho
    return np.fft.ifftn(np.fft.fftn(pad) * host(plan.multiplier())).real[:nz, :ny, :nx]


# smallest lengths, every radix of the generic engine, lengths beside the
# register engine's (16 ... 1024), 2048 as a padded length
GRIDS = [(2, 2, 2), (4, 6, 10), (12, 2, 30), (18, 50, 8), (16, 18, 54), (90, 16, 20), (36, 150, 6), (8, 10, 1024),
         (1024, 4, 2), (250, 12, 16), (2, 720, 6)]


@pytest.mark.parametrize("N", GRIDS)
def test_operators_on_edge_lengths(lib, N):
    L, n = (3.0, 2.5, 2.0), (0.6, 0.0, 0.8)
    plan, oplan = lib.Plan(N, L, n), O.Plan(N, L, n)
    prm, oprm = lib.make_params(GAMMA, BETA, LAM, OM), O.Params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    f, phi = W.random_field(shape, 11), W.random_field(shape, 12)
    Phi = W.random_field(shape, 13, complex_valued=False)
    assert rel2(host(plan.dipolar_potential_from_psi(dev(f))), convolution(plan, np.abs(f) ** 2)) <= 1e-12
    assert rel2(host(plan.apply_H(prm, dev(f), dev(phi), dev(Phi))), O.apply_H(oplan, oprm, f, phi, Phi)) <= 1e-13
    got = host(plan.apply_preconditioner(prm, 7.0, dev(f), dev(phi), dev(Phi)))
    assert rel2(got, O.apply_precond(oplan, oprm, f, phi, Phi, 7.0)) <= 1e-13


def precond_at_rest(N, L, gamma, alpha, f, fused):
    """P f for phi = Phi = 0 by numpy's transforms.  The middle of the grid has
    V = 0 up to the rounding of its coordinates -L + i h, which differs with a
    fused multiply-add (the library's tables are formed on the host, which may
    have one): both forms."""
    def coord(a):
        h = 2.0 * L[a] / N[a]
        if fused:
            return np.array([float(Fraction(i) * Fraction(h) - Fraction(L[a])) for i in range(N[a])])
        return -L[a] + np.arange(N[a]) * h
    view = [(None, None, slice(None)), (None, slice(None), None), (slice(None), None, None)]
    den = alpha + sum(
        (gamma[a] * gamma[a] * (0.5 * coord(a) * coord(a)))[view[a]] for a in (2, 1, 0))
    k2 = sum((0.5 * (np.pi / L[a] * N[a] * np.fft.fftfreq(N[a])) ** 2)[view[a]] for a in range(3))
    w = 1.0 / np.sqrt(den)
    return w * np.fft.ifftn(np.fft.fftn(w * f) / (alpha + k2))


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18)])
@pytest.mark.parametrize("alpha", [1e-40, 2.0 ** -20, 2.0 ** 40, 1e40])
def test_preconditioner_weights_at_range_edges(lib, N, alpha):
    """The integer square roots and reciprocals of the weights: arguments next
    to powers of two, and beyond the binary32 range on either side (the bar of
    this file; phi = Phi = 0, so that the weights range from 1 / sqrt(alpha))."""
    L, n = (3.0, 2.5, 2.0), (0.6, 0.0, 0.8)
    plan, prm = lib.Plan(N, L, n), lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    f, z, zr = W.random_field(shape, 14), np.zeros(shape, complex), np.zeros(shape)
    got = host(plan.apply_preconditioner(prm, alpha, dev(f), dev(z), dev(zr)))
    assert min(rel2(got, precond_at_rest(N, L, GAMMA, alpha, f, fused)) for fused in (False, True)) <= 1e-13


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18)])
def test_scaling_by_powers_of_two_is_exact(lib, N):
    """H and P are linear in f and r, and a tile's exponent takes up a power
    of two: the results scale bit for bit (over the range where no binary64
    value of the result is subnormal)."""
    plan = lib.Plan(N, (4.0, 3.0, 2.0), (0.0, 0.0, 1.0))
    prm = lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    f, phi = W.random_field(shape, 21), W.random_field(shape, 22)
    Phi = dev(W.random_field(shape, 23, complex_valued=False))
    H, P = (host(plan.apply_H(prm, dev(f), dev(phi), Phi)),
            host(plan.apply_preconditioner(prm, 5.0, dev(f), dev(phi), Phi)))
    for k in (-900, -301, 1, 640, 980):
        g = dev(np.ldexp(f.real, k) + 1j * np.ldexp(f.imag, k))
        a, b = host(plan.apply_H(prm, g, dev(phi), Phi)), host(plan.apply_preconditioner(prm, 5.0, g, dev(phi), Phi))
        for x, y in ((a, H), (b, P)):
            assert np.array_equal(x.real, np.ldexp(y.real, k)) and np.array_equal(x.imag, np.ldexp(y.imag, k)), k


def test_wide_dynamic_range_and_zeros(lib):
    """Planes whose sizes differ by 150 orders of magnitude; a zero input gives
    zeros."""
    N, L = (32, 16, 16), (4.0, 3.0, 2.0)
    plan, oplan = lib.Plan(N, L, (0.0, 0.0, 1.0)), O.Plan(N, L, (0.0, 0.0, 1.0))
    prm, oprm = lib.make_params(GAMMA, BETA, LAM, OM), O.Params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    zero, phi = np.zeros(shape, np.complex128), W.random_field(shape, 32)
    Phi = W.random_field(shape, 33, complex_valued=False)
    for out in (plan.dipolar_potential_from_psi(dev(zero)), plan.apply_H(prm, dev(zero), dev(phi), dev(Phi)),
                plan.apply_preconditioner(prm, 5.0, dev(zero), dev(phi), dev(Phi))):
        assert not host(out).any()
    f = W.random_field(shape, 31) * (10.0 ** np.linspace(-150, 0, N[2]))[:, None, None]
    assert rel2(host(plan.apply_H(prm, dev(f), dev(phi), dev(Phi))), O.apply_H(oplan, oprm, f, phi, Phi)) <= 1e-13
    assert rel2(host(plan.dipolar_potential_from_psi(dev(f))), convolution(plan, np.abs(f) ** 2)) <= 1e-12


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_stays_on_its_lines(lib, N, bad):
    """A NaN or an infinity in f spoils the three lines of H f through it and
    no other point; in P r and Phi it reaches every point."""
    plan = lib.Plan(N, (4.0, 3.0, 2.0), (0.0, 0.0, 1.0))
    prm = lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    f, phi = W.random_field(shape, 41), W.random_field(shape, 42)
    Phi = dev(W.random_field(shape, 43, complex_valued=False))
    clean = host(plan.apply_H(prm, dev(f), dev(phi), Phi))
    z, y, x = 3, 5, 7
    f[z, y, x] = bad
    got = host(plan.apply_H(prm, dev(f), dev(phi), Phi))
    lines = np.zeros(shape, bool)
    lines[z, y, :] = lines[z, :, x] = lines[:, y, x] = True
    assert not np.isfinite(got[lines]).any()
    assert rel2(got[~lines], clean[~lines]) <= 1e-14
    assert not np.isfinite(host(plan.apply_preconditioner(prm, 5.0, dev(f), dev(phi), Phi))).any()
    assert not np.isfinite(host(plan.dipolar_potential_from_psi(dev(f)))).any()
    # the same plan afterwards
    f[z, y, x] = 1.0
    assert np.isfinite(host(plan.dipolar_potential_from_psi(dev(f)))).all()
