"""gp_batch_store to buffers that are not memory of the batch's own GPU: with a
scale pending or without, the same copy serves them, with the same outcome."""
import ctypes

import numpy as np
import pytest

from paper_1206_1361_gb300 import gp
from tests.gpu_util import require_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("prec,dtype", [(gp.GP_C64, "complex64"), (gp.GP_C128, "complex128")])
@pytest.mark.parametrize("buffer", ["device", "pinned", "offset"])
def test_a_pending_scale_does_not_change_what_a_store_accepts(prec, dtype, buffer):
    require_gpu()
    import torch
    shape = (20, 18, 16)
    n = shape[0] * shape[1] * shape[2]
    rng = np.random.default_rng(3)
    psi = (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1])).astype(dtype)
    # one real in, an address that is a multiple of 4 or 8 bytes only
    real = torch.float32 if prec == gp.GP_C64 else torch.float64
    flat = (torch.zeros(2 * n + 1, dtype=real).pin_memory() if buffer == "pinned"
            else torch.zeros(2 * n + 1, dtype=real, device="cuda"))
    part = flat[1:] if buffer == "offset" else flat[:-1]
    lib, got, codes = gp.load_library(), [], []
    with gp.Batch(prec, cap_bytes=1 << 28) as b:
        slot = b.add(shape, (0.2, 0.2, 0.2), 0.002, 1.0, 1.0, 1.0, 5.0, gp.GP_IMAG, psi=psi)
        b.step(3)
        for _ in range(2):                   # the scale pending, then applied
            flat.zero_()
            torch.cuda.synchronize()
            codes.append(lib.gp_batch_store(b.b, slot, ctypes.c_void_p(part.data_ptr()), n, 1))
            got.append(part.cpu().numpy().copy())
        host = b.psi(slot)
    assert codes[0] == codes[1] and (codes[0] == gp.GP_OK or buffer == "pinned")
    assert np.array_equal(got[0], got[1])
    if codes[0] == gp.GP_OK:
        assert np.array_equal(got[0].view(dtype).reshape(shape[::-1]), host)
