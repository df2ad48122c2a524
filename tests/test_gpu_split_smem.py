"""Sub-line sweeps whose dynamic shared memory lies just below 48 KB: with a
kernel's static shared memory on top the block needs more than a kernel may
have that did not ask for it.  Edges are walked upwards in a process of its
own, so no larger launch has asked before."""
import subprocess
import sys

import pytest

from tests.gpu_util import require_gpu

RUN = """
import numpy as np
import oracle
from paper_1206_1361_gb300 import gp
from tests.gpu_util import oracle_params, rel_l2
prec, kappa, shape, axis, edges, tol = %r
dt, w, g = 1e-3, (0.0, 0.0, 0.0), 0.0
h = (dt / (4.0 * kappa)) ** 0.5
h = (h, 1.1 * h, 1.25 * h if shape[2] > 1 else 1.0)
for n in range(*edges):
    s = list(shape)
    s[axis] = n
    rng = np.random.default_rng(n)
    psi = (rng.standard_normal(s[::-1]) + 1j * rng.standard_normal(s[::-1])) * 0.3
    psi[:, :, 0] = psi[:, 0, :] = 0
    if s[2] > 1:
        psi[0] = 0
    with gp.Solver(s, h, dt, *w, g, gp.GP_IMAG, prec) as c:
        got = c.load(psi.astype(c.dtype)).step(1).psi().astype(np.complex128)
    want = psi.copy()
    oracle.step(oracle_params(s, h, dt, w, g, gp.GP_IMAG), want, 1)
    assert rel_l2(got, want) <= tol, (n, rel_l2(got, want))
"""


# One step of the sweeps (no trap, g = 0) against the oracle: 1e-12 (FP64, a few
# hundred roundings), 2e-13 (float-float, 10 roundings of 2^-47), 4 roundings of
# 2^-23 (complex64).
@pytest.mark.gpu
@pytest.mark.parametrize("case", [
    ("GP_C128", 0.02, (8, 0, 1), 1, (1330, 1346), 1e-12), ("GP_C128", 0.05, (8, 0, 1), 1, (1340, 1358), 1e-12),
    ("GP_C128", 0.05, (40, 40, 0), 2, (332, 340), 1e-12), ("GP_CFF", 0.015, (8, 0, 1), 1, (1330, 1346), 2e-13),
    ("GP_C64", 0.02, (8, 0, 1), 1, (1340, 1364), 4 * 2.0 ** -23)])
def test_blocks_just_below_48_kilobytes(case):
    require_gpu()
    from paper_1206_1361_gb300 import gp
    p = subprocess.run([sys.executable, "-c", RUN % ((getattr(gp, case[0]),) + case[1:],)], capture_output=True,
                       text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
