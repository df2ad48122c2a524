"""complex128 steps of states that are small (or large) everywhere, or over
part of the grid.  Linear steps scale exactly by powers of two, so every scale
has the same relative accuracy: 1e-12 of the norm against the oracle (a few
hundred roundings of 2^-53) -- whatever lift the increment sweeps choose for a block."""
import numpy as np
import pytest

import oracle
from paper_1206_1361_gb300 import gp
from tests.gpu_util import oracle_params, rel_l2, require_gpu

TOL = 1e-12
# the lift's own range, either side of its ends (2^-135, 2^33), of the chosen
# lifts' lower end (2^-940), and near FP64's own
SCALES = [2.0 ** e for e in (-1000, -942, -936, -860, -300, -137, -133, -73, 0, 31, 35, 95, 400)]


def state(shape, seed=23):
    rng = np.random.default_rng(seed)
    a = (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1])) * 0.3
    a[:, :, 0] = a[:, 0, :] = 0
    if shape[2] > 1:
        a[0] = 0
    return a


def grid(shape, kappa=0.0125, dt=1e-3):
    h = (dt / (4.0 * kappa)) ** 0.5
    return (h, 1.1 * h, 1.25 * h if shape[2] > 1 else 1.0), dt


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(34, 18, 17), (49, 35, 66), (128, 20, 9), (66, 130, 1), (4, 1100, 1)])
@pytest.mark.parametrize("scale", SCALES)
def test_real_time_steps_scale(shape, scale):
    require_gpu()
    h, dt = grid(shape)
    w = (1.0, 1.5, 2.0) if shape[2] > 1 else (1.0, 1.5, 0.0)
    psi = state(shape)
    with gp.Solver(shape, h, dt, *w, 0.0, gp.GP_REAL, gp.GP_C128) as s:
        got = s.load(psi * scale).step(3).psi() / scale
    want = psi.copy()
    oracle.step(oracle_params(shape, h, dt, w, 0.0, gp.GP_REAL), want, 3)
    assert rel_l2(got, want) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(34, 18, 17), (66, 130, 1)])
@pytest.mark.parametrize("scale", [2.0 ** -400, 2.0 ** -140, 2.0 ** 100])
def test_imaginary_time_steps_scale(shape, scale):
    """The first step normalises: the same result from every scale."""
    require_gpu()
    h, dt = grid(shape)
    w = (1.0, 1.5, 2.0) if shape[2] > 1 else (1.0, 1.5, 0.0)
    psi = state(shape)
    with gp.Solver(shape, h, dt, *w, 0.0, gp.GP_IMAG, gp.GP_C128) as s:
        got = s.load(psi * scale).step(3).psi()
    want = psi.copy()
    oracle.step(oracle_params(shape, h, dt, w, 0.0, gp.GP_IMAG), want, 3)
    assert rel_l2(got, want) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("nr,nz", [(49, 18), (100, 70), (1500, 35)])
@pytest.mark.parametrize("scale", SCALES)
def test_axial_steps_scale(nr, nz, scale):
    require_gpu()
    (hr, hz, _), dt = grid((nr, nz, 1), 0.02)
    psi = state((nr, nz, 1))[0]
    psi[1:, 0] = psi[1:, -1]                       # (rho = h / 2 is a live row)
    with gp.Solver.axial(nr, nz, hr, hz, dt, 1.0, 2.0, 0.0, gp.GP_REAL) as s:
        got = s.load(psi * scale).step(3).psi() / scale
    par = oracle.AxialParams.make(nr, nz, hr, hz, dt, 1.0, 2.0, 0.0, gp.GP_REAL)
    assert rel_l2(got, oracle.axial_step(par, psi.copy(), 3)) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
def test_a_state_that_falls_off_along_an_axis(axis, mode):
    """From 1 to 2^-1020 along one axis: ordinary, small and FP64 blocks, and blocks
    with values of every size, in one sweep."""
    require_gpu()
    shape = (65, 70, 66)
    h, dt = grid(shape)
    n = shape[axis]
    fall = 2.0 ** (-np.arange(n) * (1020.0 / n)).round()
    psi = state(shape) * fall.reshape([-1 if d == 2 - axis else 1 for d in range(3)])
    with gp.Solver(shape, h, dt, 1.0, 1.5, 2.0, 0.0, mode, gp.GP_C128) as s:
        got = s.load(psi).step(1).psi()
    want = psi.copy()
    oracle.step(oracle_params(shape, h, dt, (1.0, 1.5, 2.0), 0.0, mode), want, 1)
    assert rel_l2(got, want) <= TOL
