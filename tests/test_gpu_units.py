"""complex128 in any units.  The equation is unchanged when lengths go with l, dt
with l^2, the trap frequencies with l^-2, g with l and psi with l^(-3/2) (2D: g
stays, psi with l^-1): a cloud of micrometres in metres has |psi| near 10^9.  With l a
power of two the FP64 method is exactly as accurate in every unit.

Tolerance: 1e-12 of the norm against the oracle in the same units (a few
hundred roundings of 2^-53), as for the unscaled problems."""
import numpy as np
import pytest

import oracle
from paper_1206_1361_gb300 import gp
from tests.gpu_util import oracle_params, rel_l2, require_gpu

TOL = 1e-12


def state(shape, seed=17):
    """Random amplitudes under a broad envelope, zero on the Dirichlet nodes."""
    rng = np.random.default_rng(seed)
    a = (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1])) * 0.3
    a[:, :, 0] = a[:, 0, :] = 0
    if shape[2] > 1:
        a[0] = 0
    return a


def scaled(shape, kappa, l, mode):
    """(h, dt, w, g, psi) of the problem in units l."""
    dt, nd = 1e-3, 3 if shape[2] > 1 else 2
    h = (dt / (4.0 * kappa)) ** 0.5
    h = (h, 1.1 * h, 1.25 * h if nd == 3 else 1.0)
    w = (1.0, 1.5, 2.0 if nd == 3 else 0.0)
    psi = state(shape)
    if mode == gp.GP_IMAG:
        psi /= np.sqrt(np.prod(h) * (np.abs(psi) ** 2).sum())
    g = 1e-3 / (dt * (np.abs(psi) ** 2).max())          # phases up to 1e-3 a step
    # (h[2] of a 2D grid is not used)
    return (tuple(x * l for x in h[:nd]) + (1.0,) * (3 - nd), dt * l ** 2, tuple(x / l ** 2 for x in w),
            g * (l if nd == 3 else 1.0), psi * float(l) ** (-1.5 if nd == 3 else -1.0))


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(40, 33, 20), (66, 130, 1)])
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("strang", [False, True])
@pytest.mark.parametrize("l", [2.0 ** -36, 2.0 ** -20, 2.0 ** -14, 1.0, 2.0 ** 20, 2.0 ** 36])
def test_the_nonlinear_step_is_as_accurate_in_every_unit(shape, mode, strang, l):
    require_gpu()
    h, dt, w, g, psi = scaled(shape, 0.0125, l, mode)
    with gp.Solver(shape, h, dt, *w, g, mode, gp.GP_C128) as s:
        s.set_splitting(gp.GP_SPLIT_STRANG if strang else gp.GP_SPLIT_LIE)
        got = s.load(psi).step(3).psi()
    want = oracle.step_ext(oracle_params(shape, h, dt, w, g, mode), psi.copy(), 3, 0, strang)
    assert rel_l2(got, want) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("l", [2.0 ** -36, 2.0 ** -20, 1.0, 2.0 ** 20, 2.0 ** 36])
def test_the_axial_nonlinear_step_is_as_accurate_in_every_unit(mode, l):
    require_gpu()
    nr, nz = 49, 70
    h, dt, w, g, psi = scaled((nr, nz, 1), 0.0125, 1.0, mode)
    psi = psi[0]
    psi[1:, 0] = psi[1:, -1]                       # (rho = h / 2 is a live row)
    hr, hz, dt, g, psi = h[0] * l, h[1] * l, dt * l ** 2, g * l, psi * l ** -1.5
    with gp.Solver.axial(nr, nz, hr, hz, dt, 1.0 / l ** 2, 2.0 / l ** 2, g, mode) as s:
        got = s.load(psi).step(3).psi()
    par = oracle.AxialParams.make(nr, nz, hr, hz, dt, 1.0 / l ** 2, 2.0 / l ** 2, g, mode)
    assert rel_l2(got, oracle.axial_step(par, psi.copy(), 3)) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("c", [2.0 ** -40, 2.0 ** 20, 2.0 ** 60, 2.0 ** 85])
@pytest.mark.parametrize("table", [0, 1])
def test_real_time_with_any_amplitude_and_g(c, table):
    """psi with c, g with c^-2."""
    require_gpu()
    shape = (40, 33, 20)
    h, dt, w, g, psi = scaled(shape, 0.0125, 1.0, gp.GP_REAL)
    psi, g = psi * c, g / c ** 2
    with gp.Solver(shape, h, dt, *w, g, gp.GP_REAL, gp.GP_C128) as s:
        gp.gp_set_option(s.ctx, gp.GP_OPT_POTENTIAL_TABLE, table)
        got = s.load(psi).step(3).psi()
    want = psi.copy()
    oracle.step(oracle_params(shape, h, dt, w, g, gp.GP_REAL), want, 3)
    assert rel_l2(got, want) <= TOL
