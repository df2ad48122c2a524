"""A path that the caller asks for is the path that runs: GP_PATH_EXACT sweeps
complex128 in FP64 arithmetic where GP_PATH_AUTO adds float-float increments.
The two round differently, so their bits differ; each agrees with the oracle to
1e-12 of the norm (a few hundred roundings of 2^-53)."""
import numpy as np
import pytest

import oracle
from paper_1206_1361_gb300 import gp
from tests.gpu_util import oracle_params, rel_l2, require_gpu


def rand(shape, seed=3):
    rng = np.random.default_rng(seed)
    a = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * 0.3
    for axis, n in enumerate(shape):
        if n > 1:
            a[(slice(None),) * axis + (0,)] = 0
    return a


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(64, 48, 40), (300, 129, 1), (128, 128, 32)])
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
def test_the_exact_path_is_not_the_increment_form(shape, mode):
    require_gpu()
    dt, w, g = 1e-3, (1.0, 1.5, 2.0 if shape[2] > 1 else 0.0), 4.0
    h = ((dt / (4.0 * 0.0125)) ** 0.5,) * 3
    psi = rand(shape[::-1])
    got = {}
    for path in (gp.GP_PATH_AUTO, gp.GP_PATH_EXACT):
        with gp.Solver(shape, h, dt, *w, g, mode, gp.GP_C128) as s:
            s.set_path(path)
            got[path] = s.load(psi).step(4).psi()
            assert gp.gp_sweep_paths(s.ctx)[0] == gp.GP_PATH_EXACT
    want = psi.copy()
    oracle.step(oracle_params(shape, h, dt, w, g, mode), want, 4)
    assert not np.array_equal(got[gp.GP_PATH_AUTO], got[gp.GP_PATH_EXACT])
    assert all(rel_l2(a, want) <= 1e-12 for a in got.values())


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
def test_axial_windows_run_on_request(mode):
    """Three launches a step (calcnu, two windowed sweeps) and a norm's finish, where
    the increment form needs one less."""
    require_gpu()
    nr, nz, dt, g = 256, 300, 1e-3, 4.0
    h = (dt / (4.0 * 0.0125)) ** 0.5
    psi = rand((nz, nr))
    psi[1:, 0] = psi[1:, -1]                       # (rho = h / 2 is a live row)
    got, launches = [], []
    for path in (gp.GP_PATH_AUTO, gp.GP_PATH_WINDOW, gp.GP_PATH_EXACT):
        with gp.Solver.axial(nr, nz, h, h, dt, 1.0, 2.0, g, mode) as s:
            s.set_path(path)
            got.append(s.load(psi).step(4).psi())
            launches.append(gp.gp_launches_per_step(s.ctx)[0])
    par = oracle.AxialParams.make(nr, nz, h, h, dt, 1.0, 2.0, g, mode)
    want = oracle.axial_step(par, psi.copy(), 4)
    assert launches[1] == launches[0] + 1
    assert not np.array_equal(got[0], got[1]) and not np.array_equal(got[0], got[2])
    assert all(rel_l2(a, want) <= 1e-12 for a in got)
