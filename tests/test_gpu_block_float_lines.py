"""The binary64 operators' integer passes, line by line: H f of a quiet line
beside loud ones, every line length that the composite-length engine is built
for, and values next to the ends of the binary64 range."""
import numpy as np
import pytest
import torch

import atkm_workloads as W

pytestmark = pytest.mark.gpu
GAMMA, BETA, LAM, OM = (1.0, 1.3, 3.0), 30.0, 12.0, 0.4


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    return t.detach().cpu().numpy()


def rel2(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def mesh(N, L):
    ax = [-L[a] + (2.0 * L[a] / N[a]) * np.arange(N[a]) for a in range(3)]
    k = [np.fft.fftfreq(N[a], 1.0 / N[a]).round() * np.pi / L[a] for a in range(3)]
    view = [(None, None, slice(None)), (None, slice(None), None), (slice(None), None, None)]
    return [ax[a][view[a]] for a in range(3)], [k[a][view[a]] for a in range(3)]


def ref_H(N, L, f, phi, Phi):
    """H_phi f by numpy's transforms of each axis's lines."""
    (x, y, z), (kx, ky, kz) = mesh(N, L)
    line = lambda a, m: np.fft.ifft(m * np.fft.fft(f, axis=a), axis=a)  # noqa: E731
    V = 0.5 * ((GAMMA[0] * x) ** 2 + (GAMMA[1] * y) ** 2 + (GAMMA[2] * z) ** 2)
    return (line(2, 0.5 * kx ** 2 + OM * y * kx) + line(1, 0.5 * ky ** 2 - OM * x * ky) + line(0, 0.5 * kz ** 2)
            + (V + BETA * np.abs(phi) ** 2 + LAM * Phi) * f)


# each engine in each role: k_ifast (256; 512), k_imix (144, 36; 32, 16 on a small grid), k_igen (54, 50, 12)
@pytest.mark.parametrize("N", [(256, 16, 64), (16, 512, 32), (144, 36, 20), (32, 16, 16), (54, 50, 12)])
@pytest.mark.parametrize("quiet", [1e-9, 1e-30, 1e-200])
def test_quiet_lines_beside_loud_ones(lib, N, quiet):
    """f is of size `quiet` where all indices are even, and of size one where two
    are odd and z or y even: the three lines through an all-even point hold quiet
    values only, and their neighbours in the x, y and z pass (indexed y, x, x)
    loud ones.  H f at those points is as good as their own lines allow: 4e-15
    of its 2-norm (a binary64 transform pair is good to a few 1e-16)."""
    L = (6.0, 5.0, 4.0)
    plan, prm = lib.Plan(N, L, (0.0, 0.0, 1.0)), lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    g, phi = W.random_field(shape, 51), W.random_field(shape, 52)
    Phi = W.random_field(shape, 53, complex_valued=False)
    f = np.zeros(shape, complex)
    f[::2, 1::2, 1::2] = g[::2, 1::2, 1::2]
    f[1::2, ::2, 1::2] = g[1::2, ::2, 1::2]
    f[::2, ::2, ::2] = quiet * g[::2, ::2, ::2]
    got, ref = host(plan.apply_H(prm, dev(f), dev(phi), dev(Phi))), ref_H(N, L, f, phi, Phi)
    assert rel2(got[::2, ::2, ::2] / quiet, ref[::2, ::2, ::2] / quiet) <= 4e-15
    assert rel2(got, ref) <= 4e-15


def test_H_rounds_to_nearest(lib):
    """The integers of H's passes are rounded, not cut off: its error on a smooth
    cloud with long z lines is below 1e-15 of the 2-norm, about a quarter of what
    binary64 transforms have there (3.7e-15; integers cut off, 1.6e-15).
    Reference: the same lines in long double."""
    N, L = (16, 8, 256), (16.0, 16.0, 1.5)
    plan, prm = lib.Plan(N, L, (0.0, 0.0, 1.0)), lib.make_params((1.0, 1.2, 30.0), 1000.0, 400.0, 0.9)
    (x, y, z), _ = mesh(N, L)
    f = np.exp(0.3j * x) / (1.0 + x * x + y * y + z * z)
    Phi = 0.02 * np.exp(-0.03 * (x * x + y * y)) * np.cos(0.5 * x + 0.3 * y) + 0.0 * z
    got = host(plan.apply_H(prm, dev(f), dev(f), dev(Phi)))
    LD = np.longdouble
    pi = LD("3.14159265358979323846264338327950288")
    ax = [-LD(L[a]) + 2 * LD(L[a]) / N[a] * np.arange(N[a]).astype(LD) for a in range(3)]
    k = [np.fft.fftfreq(N[a], 1.0 / N[a]).round().astype(LD) * pi / LD(L[a]) for a in range(3)]
    view = [(None, None, slice(None)), (None, slice(None), None), (slice(None), None, None)]
    (x, y, z), (kx, ky, kz) = [ax[a][view[a]] for a in range(3)], [k[a][view[a]] for a in range(3)]
    F = f.astype(np.clongdouble)
    line = lambda a, m: np.fft.ifft(m * np.fft.fft(F, axis=a), axis=a)  # noqa: E731
    om = LD(0.9)
    V = (x * x + LD(1.2) * LD(1.2) * y * y + 900 * z * z) / 2
    ref = (line(2, kx ** 2 / 2 + om * y * kx) + line(1, ky ** 2 / 2 - om * x * ky) + line(0, kz ** 2 / 2)
           + (V + 1000 * (F.real ** 2 + F.imag ** 2) + 400 * Phi.astype(LD)) * F)
    err = np.abs(got.astype(np.clongdouble) - ref)
    assert float(np.sqrt((err ** 2).sum() / (np.abs(ref) ** 2).sum())) <= 1e-15


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18), (54, 50, 12)])
def test_inputs_next_to_the_smallest_normal(lib, N):
    """H, P and the dipolar potential are linear: inputs scaled by 2^-980 give
    results scaled by it bit for bit (no value of theirs is subnormal), inputs
    scaled by 2^-1015 to 1e-13 of the 2-norm (their smallest are)."""
    plan = lib.Plan(N, (4.0, 3.0, 2.0), (0.0, 0.0, 1.0))
    prm = lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    f, phi = W.random_field(shape, 71), dev(W.random_field(shape, 72))
    Phi, rho = dev(W.random_field(shape, 73, complex_valued=False)), np.abs(f) + 0.125
    ops = [lambda g: plan.apply_H(prm, dev(g), phi, Phi), lambda g: plan.apply_preconditioner(prm, 5.0, dev(g), phi, Phi)]
    scaled = lambda a, k: np.ldexp(a.real, k) + 1j * np.ldexp(a.imag, k)  # noqa: E731
    for op in ops:
        one, a, b = host(op(f)), host(op(scaled(f, -980))), host(op(scaled(f, -1015)))
        assert np.array_equal(a, scaled(one, -980))
        assert rel2(scaled(b, 1000), scaled(one, -15)) <= 1e-13
    one = host(plan.dipolar_potential(dev(rho)))
    assert np.array_equal(host(plan.dipolar_potential(dev(np.ldexp(rho, -980)))), np.ldexp(one, -980))
    assert rel2(np.ldexp(host(plan.dipolar_potential(dev(np.ldexp(rho, -1015)))), 1000), np.ldexp(one, -15)) <= 1e-13


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18), (54, 50, 12)])
@pytest.mark.parametrize("k", [-500, -300, 300])
def test_energies_of_scaled_states(lib, N, k):
    """E_kin and E_rot are quadratic in phi: they scale by 2^(2 k), to 1e-13 (sums
    of positive and of mixed terms), as long as they are normal values."""
    plan = lib.Plan(N, (4.0, 3.0, 2.0), (0.0, 0.0, 1.0))
    prm = lib.make_params(GAMMA, 0.0, 0.0, OM)
    shape = (N[2], N[1], N[0])
    f, Phi = W.random_field(shape, 81), dev(np.zeros(shape))
    one = plan.energy_parts(prm, dev(f), Phi)
    got = plan.energy_parts(prm, dev(np.ldexp(f.real, k) + 1j * np.ldexp(f.imag, k)), Phi)
    for key in ("E_kin", "E_rot"):
        assert abs(np.ldexp(got[key], -2 * k) - one[key]) <= 1e-13 * one["E_kin"], (key, got[key], one[key])


@pytest.mark.parametrize("N", [(32, 64, 16), (36, 20, 18), (54, 50, 12)])
def test_largest_finite_multipliers(lib, N):
    """alpha = 1e-304, phi = Phi = 0: the zero frequency's multiplier is 1e304, so
    that P r is w / alpha times the mean of w r (the rest is 1e-304 of it), w =
    V^{-1/2} away from the centre (where r = 0, and w is as large as V's rounding
    there allows).  Finite, and to 1e-13 of that mean's part; 1 / 1e-313 is infinite."""
    L = (4.0, 3.0, 2.0)
    plan, prm = lib.Plan(N, L, (0.0, 0.0, 1.0)), lib.make_params(GAMMA, BETA, LAM, OM)
    shape = (N[2], N[1], N[0])
    c = (N[2] // 2, N[1] // 2, N[0] // 2)
    r, zero = W.random_field(shape, 91) + 2.0, np.zeros(shape)
    r[c] = 0.0
    (x, y, z), _ = mesh(N, L)
    V = 0.5 * ((GAMMA[0] * x) ** 2 + (GAMMA[1] * y) ** 2 + (GAMMA[2] * z) ** 2)
    V[c] = 1.0
    w = 1.0 / np.sqrt(V)
    got = host(plan.apply_preconditioner(prm, 1e-304, dev(r), dev(zero.astype(complex)), dev(zero)))
    away = np.ones(shape, bool)
    away[c] = False
    ref = w * np.mean(w * r)
    assert np.isfinite(got[away]).all() and rel2(got[away] * 1e-304, ref[away]) <= 1e-13
    assert not np.isfinite(host(plan.apply_preconditioner(prm, 1e-313, dev(r), dev(zero.astype(complex)), dev(zero)))).any()


# every length that k_imix is built for (i64.cuh, int_radices), as the x line, as
# an unpadded and as a padded column
IMIX = [16, 32, 64, 128, 256, 18, 20, 24, 30, 36, 40, 48, 60, 72, 80, 90, 96, 100, 108, 120, 144, 150, 160, 180, 192, 200, 216,
        240, 288, 320, 384]


@pytest.mark.parametrize("n", IMIX)
def test_every_composite_length(lib, n):
    """Every length of k_imix in each of its forms, on grids of few lines (where
    the powers of two run on it too): n as Nx, as Ny and Nz (H, P), and n = 2 Ny,
    2 Nz where n / 2 is a length (the potential).  Against transforms of numpy's
    (1e-14 of the 2-norm: a few 1e-16 on either side, and H's nu^2 / 2 that raises
    the reference's error at the low frequencies by less than ten) and the same
    operators by the generic engine."""
    grids = [(n, 4, 6), (6, n, 4), (4, 6, n)] + ([(4, n // 2, 6), (6, 4, n // 2)] if n % 4 == 0 else [])
    L = (4.0, 3.0, 2.0)
    for N in grids:
        fixed, gen = lib.Plan(N, L, (0.6, 0.0, 0.8)), lib.Plan(N, L, (0.6, 0.0, 0.8), generic_fft=True)
        prm = lib.make_params(GAMMA, BETA, LAM, OM)
        shape = (N[2], N[1], N[0])
        f, phi = W.random_field(shape, n), W.random_field(shape, n + 1)
        Phi = W.random_field(shape, n + 2, complex_valued=False)
        nz, ny, nx = shape
        pad = np.zeros((2 * nz, 2 * ny, 2 * nx))
        pad[:nz, :ny, :nx] = np.abs(f) ** 2
        A = np.fft.ifftn(np.fft.fftn(pad) * host(fixed.multiplier())).real[:nz, :ny, :nx]
        (x, y, z), (kx, ky, kz) = mesh(N, L)
        V = 0.5 * ((GAMMA[0] * x) ** 2 + (GAMMA[1] * y) ** 2 + (GAMMA[2] * z) ** 2)
        w = 1.0 / np.sqrt(7.0 + V + BETA * np.abs(phi) ** 2 + LAM * np.maximum(Phi, 0.0))
        P = w * np.fft.ifftn(np.fft.fftn(w * f) / (7.0 + 0.5 * (kx ** 2 + ky ** 2 + kz ** 2)))
        for plan in (fixed, gen):
            got = (host(plan.dipolar_potential_from_psi(dev(f))), host(plan.apply_H(prm, dev(f), dev(phi), dev(Phi))),
                   host(plan.apply_preconditioner(prm, 7.0, dev(f), dev(phi), dev(Phi))))
            for a, b in zip(got, (A, ref_H(N, L, f, phi, Phi), P)):
                assert rel2(a, b) <= 1e-14, (N, plan is gen)
            # the forms with fused sums: E_kin and E_rot are sums over the lines' spectra
            e = plan.energy_parts(prm, dev(f), dev(Phi))
            h3 = np.prod([2.0 * L[i] / N[i] for i in range(3)])
            s = [(np.abs(np.fft.fft(f, axis=a)) ** 2) / shape[a] for a in range(3)]
            kin = h3 * sum(np.sum(0.5 * k ** 2 * s[2 - i]) for i, k in enumerate((kx, ky, kz)))
            rot = h3 * np.sum(OM * y * kx * s[2] - OM * x * ky * s[1])
            assert abs(e["E_kin"] - kin) <= 1e-13 * kin and abs(e["E_rot"] - rot) <= 1e-13 * kin, (N, plan is gen)
        fixed.close()
        gen.close()
