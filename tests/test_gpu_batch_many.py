"""Several batches in one process: one with large tiles keeps stepping when
another with small ones was prepared after it, in both launch forms and from
several threads."""
import threading

import numpy as np
import pytest

from paper_1206_1361_gb300 import gp
from tests.gpu_util import require_gpu


def batch(prec, shape, queue):
    rng = np.random.default_rng(4)
    psi = (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1]))
    b = gp.Batch(prec, cap_bytes=1 << 28)
    if queue:
        b.set_wait_ns(2 * 10 ** 9)
    slot = b.add(shape, (0.2, 0.2, 0.2), 0.002, 1.0, 1.0, 1.0, 5.0, gp.GP_REAL,
                 psi=psi.astype("complex64" if prec == gp.GP_C64 else "complex128"))
    return b, slot


@pytest.mark.gpu
@pytest.mark.parametrize("prec,edge", [(gp.GP_C64, 512), (gp.GP_C128, 384)])
@pytest.mark.parametrize("queue", [False, True])
def test_a_small_batch_does_not_shrink_another_ones_tiles(prec, edge, queue):
    require_gpu()
    big, at = batch(prec, (edge, 12, 9), queue)
    alone, at1 = batch(prec, (edge, 12, 9), queue)
    alone.step(4)
    want = alone.psi(at1)
    big.step(2)
    small, _ = batch(prec, (8, 6, 5), queue)
    small.step(1)
    big.step(2)
    assert np.array_equal(big.psi(at), want)
    for b in (big, alone, small):
        b.close()


@pytest.mark.gpu
def test_batches_step_from_several_threads():
    require_gpu()
    failed = []

    def work(shape):
        try:
            b, slot = batch(gp.GP_C64, shape, False)
            for _ in range(200):
                b.step(2)
            assert np.isfinite(b.psi(slot)).all()
            b.close()
        except Exception as e:               # (an exception of a thread would be lost)
            failed.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in ((512, 8, 6), (8, 6, 5), (96, 20, 6), (16, 12, 9))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
