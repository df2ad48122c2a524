"""FP64 sub-line sweeps: no row is rounded to one side.  The coefficients' own
roundings repeat at every step; where they differ from row to row they leave
a pattern in the state that grows.  One sweep of smooth random lines
against the same sweep in numpy's longest real: the mean relative error of
each row over many lines may differ from the typical row's by 2^-54 -- the
rows' random roundings (about 2^-53 each) average to 2^-58 over 1024 lines,
3.5 of that over all rows, and the coefficients off the diagonal leave 4 kappa
2^-53 < 2^-55 between a cut's rows and the others.  Rows near the ends, whose
coefficients differ anyway, are left out."""
import numpy as np
import pytest

from paper_1206_1361_gb300 import gp
from tests.gpu_util import require_gpu

CL = np.clongdouble


def exact_sweep(p, kappa):
    """(I - kappa L)^-1 (I + kappa L) along the first axis."""
    one = CL(1)
    r, e, mult = CL(0), np.zeros_like(p), []
    for j in range(len(p)):
        e[j] = p[j] + (r * e[j - 1] if j else 0)
        mult.append(one / (one + 2 * kappa - kappa * r))
        r = kappa * mult[-1]
    v = np.zeros_like(p)
    for j in range(len(p) - 1, -1, -1):
        v[j] = mult[j] * (e[j] + (kappa * v[j + 1] if j + 1 < len(p) else 0))
    return 2 * v - p


@pytest.mark.gpu
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("mode,kappa", [(gp.GP_IMAG, 0.031), (gp.GP_IMAG, 0.037), (gp.GP_IMAG, 0.047),
                                        (gp.GP_IMAG, 0.05), (gp.GP_REAL, 0.07), (gp.GP_REAL, 0.1)])
def test_no_row_is_rounded_to_one_side(axis, mode, kappa):
    require_gpu()
    import torch
    n, lines, h = 384, 1024, 0.1
    rng = np.random.default_rng(5)
    x = np.linspace(-1.0, 1.0, n)[:, None]
    p = 1.0 + 0.3 * np.cos(rng.uniform(1, 3, lines) * x + rng.uniform(0, 6, lines)) * rng.uniform(0.2, 1, lines)
    p = p * np.exp(1j * rng.uniform(0, 6, lines)) * rng.uniform(0.5, 2.0, lines)
    p[0] = 0
    dt = kappa * 4.0 * h * h
    shape = (n, lines, 1) if axis == 0 else (lines, n, 1)
    psi = torch.from_numpy(np.ascontiguousarray(p.T if axis == 0 else p)).cuda()
    gp.gp_sweep_noalloc(psi, shape, axis, h, dt, mode, gp.GP_C128)
    torch.cuda.synchronize()
    got = psi.cpu().numpy()
    got = (got.T if axis == 0 else got)[1:]
    k = CL(dt / (4.0 * h * h))
    want = exact_sweep(p[1:].astype(CL), k * (CL(1j) if mode == gp.GP_REAL else 1))
    rows = ((got - want) / want).mean(axis=1)[40:-40].astype(complex)
    typical = np.median(rows.real) + 1j * np.median(rows.imag)
    assert np.abs(rows - typical).max() <= 2.0 ** -54
