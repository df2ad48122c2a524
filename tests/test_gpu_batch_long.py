"""Long gp_batch_step calls: the same bits as many short ones, also when the
batch changes between them, and the call returns while the GPU still works."""
import time

import numpy as np
import pytest

from paper_1206_1361_gb300 import gp
from tests.gpu_util import require_gpu


def state(shape, prec, seed=6):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1])).astype(
        "complex64" if prec == gp.GP_C64 else "complex128")


def add(b, shape, mode, prec):
    return b.add(shape, (0.2, 0.22, 0.25), 0.002, 1.0, 1.2, 1.5 if shape[2] > 1 else 0.0, 8.0, mode,
                 psi=state(shape, prec))


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [gp.GP_C64, gp.GP_C128])
@pytest.mark.parametrize("n", [127, 128, 160, 161, 300])
def test_long_calls_are_short_ones(prec, n):
    require_gpu()
    got = []
    for pieces in ([n, n], [1] * n + [37] * (n // 37) + [n % 37]):
        with gp.Batch(prec, cap_bytes=1 << 28) as b:
            a = add(b, (33, 20, 17), gp.GP_IMAG, prec)
            half = sum(pieces) // 2
            done = 0
            for k in pieces:
                if done == half:                # another instance joins
                    c = add(b, (24, 40, 1), gp.GP_REAL, prec)
                b.step(k)
                done += k
            got.append((b.psi(a), b.psi(c), b.observables()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert got[0][2] == got[1][2]


@pytest.mark.gpu
def test_a_long_call_returns_before_its_steps_are_done():
    """4000 steps of about 20 us against 125 graph launches of a few us each: the
    call takes under half of the whole (launched one by one it waits for all but
    the last thousand launches)."""
    require_gpu()
    with gp.Batch(gp.GP_C64, cap_bytes=1 << 28) as b:
        add(b, (96, 96, 32), gp.GP_IMAG, gp.GP_C64)
        b.step(200)
        gp.gp_batch_sync(b.b)
        t0 = time.perf_counter()
        b.step(4000)
        t1 = time.perf_counter()
        gp.gp_batch_sync(b.b)
        t2 = time.perf_counter()
    assert t1 - t0 < 0.5 * (t2 - t0)
