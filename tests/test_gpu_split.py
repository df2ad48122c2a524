"""Sub-line sweeps (sscn_split.cu, sscn_inc.cu): grids whose lines are cut into pieces that
many lanes solve.  Shapes put every remainder of that cut on some axis (one
row, one row more or less than full pieces, a single piece), uneven tiles of
neighbouring lines, and lines longer than a block of 8 rows a lane holds.

Tolerances.  FP64 against the oracle: 1e-12 of the norm (a few hundred
roundings of 2^-53).  complex64 sweeps alone (no trap, g = 0) against the
oracle: 4 roundings of 2^-23 per sweep set.  complex64 against the TMA sweeps
it stands in for, whose arithmetic it keeps: one rounding, 2^-24."""
import numpy as np
import pytest

import oracle
from paper_1206_1361_gb300 import gp
from tests.gpu_util import oracle_params, rel_l2, require_gpu

W3 = (1.0, 1.5, 2.0)
# n - 1 = 16 k, 16 k + 1, 32 k + 1, one piece, 2 and 3 rows
SHAPES = [(17, 33, 18), (34, 16, 3), (49, 35, 66), (200, 7, 140), (131, 3, 4), (500, 129, 1),
          (3, 1100, 1), (4100, 5, 1), (33, 2051, 1)]


def rand_state(shape, seed):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((nz, ny, nx)) + 1j * rng.standard_normal((nz, ny, nx))
    a[:, :, 0] = a[:, 0, :] = 0
    if nz > 1:
        a[0] = 0
    return a * 0.3


def spacing(shape, kappa, dt):
    h = (dt / (4.0 * kappa)) ** 0.5
    return (h, 1.1 * h, 1.25 * h if shape[2] > 1 else 1.0)


def trap_of(shape):
    return W3 if shape[2] > 1 else (1.0, 1.5, 0.0)


def run(shape, h, dt, w, g, mode, prec, steps, psi0, path=gp.GP_PATH_AUTO):
    with gp.Solver(shape, h, dt, *w, g, mode, prec) as s:
        s.set_path(path)
        s.load(psi0.astype(s.dtype)).step(steps)
        return s.psi().astype(np.complex128)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("kappa", [0.0125, 0.05, 0.4])
def test_fp64_matches_the_oracle(shape, mode, kappa):
    require_gpu()
    dt, g, steps, w = 1e-3, 4.0, 3, trap_of(shape)
    h = spacing(shape, kappa, dt)
    psi0 = rand_state(shape, 7)
    got = run(shape, h, dt, w, g, mode, gp.GP_C128, steps, psi0)
    want = psi0.copy()
    oracle.step(oracle_params(shape, h, dt, w, g, mode), want, steps)
    assert rel_l2(got, want) <= 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("kappa", [0.0125, 0.05, 0.4])
@pytest.mark.parametrize("path", [gp.GP_PATH_AUTO, gp.GP_PATH_EXACT])
def test_complex64_sweeps_match_the_oracle(shape, mode, kappa, path):
    require_gpu()
    dt, steps = 1e-3, 3
    h = spacing(shape, kappa, dt)
    psi0 = rand_state(shape, 8).astype(np.complex64)
    got = run(shape, h, dt, (0.0, 0.0, 0.0), 0.0, mode, gp.GP_C64, steps, psi0, path)
    want = psi0.astype(np.complex128)
    oracle.step(oracle_params(shape, h, dt, (0.0, 0.0, 0.0), 0.0, mode), want, steps)
    assert rel_l2(got, want) <= steps * 4 * 2.0 ** -23


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(18, 33, 17), (200, 7, 140), (500, 129, 1), (66, 1025, 1), (4, 3, 35)])
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("strang", [False, True])
def test_complex64_keeps_the_tma_sweeps_arithmetic(shape, mode, strang):
    require_gpu()
    dt, w = 1e-3, trap_of(shape)
    h = spacing(shape, 0.02, dt)
    psi0 = rand_state(shape, 5)
    got = []
    for path in (gp.GP_PATH_AUTO, gp.GP_PATH_TMA):
        with gp.Solver(shape, h, dt, *w, 4.0, mode, gp.GP_C64) as s:
            s.set_path(path).set_splitting(gp.GP_SPLIT_STRANG if strang else gp.GP_SPLIT_LIE)
            s.load(psi0.astype(np.complex64)).step(4)
            got.append(s.psi().astype(np.complex128))
    assert rel_l2(got[0], got[1]) <= 2.0 ** -24


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("prec", [gp.GP_C128, gp.GP_C64])
@pytest.mark.parametrize("table", [0, 1])
@pytest.mark.parametrize("shape", [(49, 35, 18), (130, 67, 1)])
def test_symmetric_splitting_and_modulated_g(mode, prec, table, shape):
    require_gpu()
    dt, g, g1, omega, steps = 2e-3, 6.0, 4.0, 25.0, 12
    h = spacing(shape, 0.03, dt)
    psi0 = rand_state(shape, 9)
    w = trap_of(shape)
    with gp.Solver(shape, h, dt, *w, g, mode, prec) as s:
        gp.gp_set_option(s.ctx, gp.GP_OPT_POTENTIAL_TABLE, table)
        s.set_splitting(gp.GP_SPLIT_STRANG).set_modulation(g1, omega)
        s.load(psi0.astype(s.dtype)).step(steps)
        got = s.psi().astype(np.complex128)
    want = oracle.step_ext(oracle_params(shape, h, dt, w, g, mode), psi0.copy(), steps, 0, True, g1, omega)
    assert rel_l2(got, want) <= (1e-12 if prec == gp.GP_C128 else steps * 4 * 2.0 ** -23)


def special_state(shape, seed):
    """Values whose significands sit where the FP64 <-> float-float conversions
    carry or borrow: powers of two and their neighbours, ties at the 24th bit,
    all-ones significands, zeros."""
    rng = np.random.default_rng(seed)
    m = np.array([0.0, 1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -24, 1.0 + 2.0 ** -24 + 2.0 ** -52, 1.0 + 2.0 ** -23,
                  1.0 + 2.0 ** -52, 2.0 - 2.0 ** -24, 2.0 - 2.0 ** -25, 1.5 + 2.0 ** -24 - 2.0 ** -52])

    def part():
        v = rng.choice(m, shape[::-1]) * 2.0 ** rng.integers(-3, 3, shape[::-1])
        return v * rng.choice([-1.0, 1.0], shape[::-1])

    a = part() + 1j * part()
    a[:, :, 0] = a[:, 0, :] = 0
    if shape[2] > 1:
        a[0] = 0
    return a


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("shape", [(34, 18, 17), (66, 130, 1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 100, 2.0 ** 92, 2.0 ** -60])
def test_fp64_conversions_at_their_corners(mode, shape, scale):
    """Sweeps of special values, also where a block leaves the float-float
    range (2^93) for FP64 and at the lower end of its full precision."""
    require_gpu()
    dt, steps = 1e-3, 2
    h = spacing(shape, 0.02, dt)
    psi0 = special_state(shape, 3) * scale
    got = run(shape, h, dt, (0.0, 0.0, 0.0), 0.0, mode, gp.GP_C128, steps, psi0)
    want = psi0.copy()
    oracle.step(oracle_params(shape, h, dt, (0.0, 0.0, 0.0), 0.0, mode), want, steps)
    assert rel_l2(got, want) <= 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("g", [4.0, 4000.0, -50.0])
def test_fp64_nonlinear_factor_on_both_sides_of_its_series(mode, g):
    """dt g |psi|^2 below 2^-8 everywhere, on both sides of it, negative g."""
    require_gpu()
    shape, dt, steps = (40, 33, 20), 1e-3, 3
    h = spacing(shape, 0.0125, dt)
    psi0 = rand_state(shape, 21)
    got = run(shape, h, dt, W3, g, mode, gp.GP_C128, steps, psi0)
    want = psi0.copy()
    oracle.step(oracle_params(shape, h, dt, W3, g, mode), want, steps)
    assert rel_l2(got, want) <= 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(3, 3, 3), (33, 5, 4), (257, 3, 1), (64, 65, 9), (500, 129, 1), (40, 70, 300)])
@pytest.mark.parametrize("prec", [gp.GP_C128, gp.GP_CFF])
def test_fp64_observables_of_every_walk(shape, prec):
    """Walks of 4 to 64 lines, ragged x segments and line chunks, one and two
    finish launches: N, mu, E and the rms sizes of a random state against the
    oracle within 1e-12 (FP64: a few hundred roundings; pairs: 2^-46 a term)."""
    require_gpu()
    h, dt, g, w = (0.2, 0.25, 0.3), 1e-3, 5.0, trap_of(shape)
    psi0 = rand_state(shape, 13)
    with gp.Solver(shape, h, dt, *w, g, gp.GP_REAL, prec) as s:
        got = s.load(psi0).observables()
    want = oracle.observables(oracle_params(shape, h, dt, w, g, gp.GP_REAL), psi0)
    for k in ("norm", "mu", "energy", "rms_x", "rms_y", "rms_z", "rms_r"):
        assert abs(got[k] - want[k]) <= 1e-12 * abs(want[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [gp.GP_C64, gp.GP_C128])
def test_batch_launch_forms_agree_bit_for_bit(prec):
    """A launch per sweep and the persistent launch (selected by a wait
    budget): the same tiles and arithmetic, the same bits; states stored to a
    device buffer and to the host are the same."""
    require_gpu()
    import torch
    dtype = torch.complex64 if prec == gp.GP_C64 else torch.complex128
    shapes = [(33, 20, 17, 0), (96, 40, 1, 1), (130, 97, 12, 0), (48, 112, 33, 1)]
    got = []
    for queue in (False, True):
        with gp.Batch(prec, cap_bytes=1 << 31) as b:
            if queue:
                b.set_wait_ns(2 * 10 ** 9)
            slots = [b.add((nx, ny, nz), (0.2, 0.22, 0.25), 0.004, 1.0, 1.2, 1.5 if nz > 1 else 0.0, 8.0, mode,
                           psi=rand_state((nx, ny, nz), 31).astype(np.complex64 if prec == gp.GP_C64 else np.complex128))
                     for nx, ny, nz, mode in shapes]
            b.step(5)
            obs = b.observables()
            out = []
            for s, (nx, ny, nz, _) in zip(slots, shapes):
                dev = torch.empty(nx * ny * nz, dtype=dtype, device="cuda")
                gp.gp_batch_store(b.b, s, dev)
                host = b.psi(s)
                assert np.array_equal(dev.cpu().numpy().reshape(host.shape), host)
                out.append(host)
            got.append((out, obs))
    for a, c in zip(got[0][0], got[1][0]):
        assert np.array_equal(a, c)
    assert got[0][1] == got[1][1]


def axial_run(nr, nz, kappa, g, mode, psi0, steps, path=gp.GP_PATH_AUTO, strang=False):
    dt = 1e-3
    h = (dt / (4.0 * kappa)) ** 0.5
    with gp.Solver.axial(nr, nz, h, 1.1 * h, dt, 1.0, 2.0, g, mode) as s:
        s.set_path(path)
        if strang:
            s.set_splitting(gp.GP_SPLIT_STRANG).set_modulation(3.0, 40.0)
        return s.load(psi0).step(steps).psi()


@pytest.mark.gpu
@pytest.mark.parametrize("nr,nz", [(3, 3), (16, 40), (17, 33), (49, 18), (256, 130), (1023, 301), (1500, 35), (21, 2048),
                                   (3700, 4), (5000, 4), (24, 2300)])
@pytest.mark.parametrize("mode,kappa", [(gp.GP_IMAG, 0.004), (gp.GP_IMAG, 0.024), (gp.GP_REAL, 0.0125), (gp.GP_REAL, 0.059)])
@pytest.mark.parametrize("strang", [False, True])
def test_axial_increment_sweeps_match_the_oracle(nr, nz, mode, kappa, strang):
    """The radial increment sweep (and the axial one) at every remainder of the
    cut, at the longest lines it takes and past them."""
    require_gpu()
    dt, g, steps = 1e-3, 5.0, 5
    h = (dt / (4.0 * kappa)) ** 0.5
    psi0 = rand_state((nr, nz, 1), 5)[0]
    psi0[1:, 0] = psi0[1:, -1]                        # (the axis rho = h / 2 is a live row)
    got = axial_run(nr, nz, kappa, g, mode, psi0, steps, strang=strang)
    par = oracle.AxialParams.make(nr, nz, h, 1.1 * h, dt, 1.0, 2.0, g, mode)
    want = oracle.axial_step(par, psi0.copy(), steps, 0, True, 3.0, 40.0) if strang else oracle.axial_step(par, psi0.copy(), steps)
    assert rel_l2(got, want) <= 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [2.0 ** -300, 2.0 ** 77, 2.0 ** 79, 2.0 ** 92, 2.0 ** 400])
def test_axial_values_beyond_the_lifted_floats(scale):
    """Linear real-time steps scale exactly by powers of two: large values take
    the FP64 branch, tiny ones lose only what is far below the largest."""
    require_gpu()
    nr, nz = 100, 70
    psi0 = rand_state((nr, nz, 1), 6)[0]
    want = axial_run(nr, nz, 0.02, 0.0, gp.GP_REAL, psi0, 3, path=gp.GP_PATH_EXACT)
    got = axial_run(nr, nz, 0.02, 0.0, gp.GP_REAL, psi0 * scale, 3) / scale
    # below the lifted range the increment is dropped: up to 8 kappa per sweep
    assert rel_l2(got, want) <= (1e-12 if scale > 1e-30 else 3 * 2 * 8 * 0.02)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", [gp.GP_IMAG, gp.GP_REAL])
@pytest.mark.parametrize("kappa", [0.006, 0.018])
def test_float_float_matches_the_oracle(shape, mode, kappa):
    """The float-float form on the sub-line sweeps: about 10 roundings of 2^-47 a
    step, 3 steps: 2e-13 of the norm."""
    require_gpu()
    dt, g, steps, w = 1e-3, 4.0, 3, trap_of(shape)
    h = spacing(shape, kappa, dt)
    psi0 = rand_state(shape, 7)
    got = run(shape, h, dt, w, g, mode, gp.GP_CFF, steps, psi0)
    want = psi0.copy()
    oracle.step(oracle_params(shape, h, dt, w, g, mode), want, steps)
    assert rel_l2(got, want) <= 2e-13
