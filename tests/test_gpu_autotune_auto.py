"""gp_autotune reaches the kernels that only GP_PATH_AUTO chooses, and the cache
keeps that choice: a float-float grid of few lines runs ten times faster on the cut
lines than on any tile shape of the TMA pipeline."""
import numpy as np
import pytest

from paper_1206_1361_gb300 import autotune, gp
from tests.gpu_util import require_gpu


@pytest.mark.gpu
def test_autotune_keeps_the_automatic_choice_where_it_is_fastest(tmp_path):
    require_gpu()
    shape, dt, cache = (500, 384, 1), 1e-3, str(tmp_path / "tune.json")
    h = (dt / (4.0 * 0.0125)) ** 0.5
    h = (h, h, 1.0)
    rng = np.random.default_rng(2)
    psi = (rng.standard_normal(shape[::-1]) + 1j * rng.standard_normal(shape[::-1])) * 0.3
    ms = []
    for again in (False, True):
        with gp.Solver(shape, h, dt, 1.0, 1.5, 0.0, 4.0, gp.GP_REAL, gp.GP_CFF) as s:
            s.load(psi)
            pick = autotune.tune(s, h, dt, gp.GP_REAL, steps=3, path=cache)
            assert pick["cached"] == again
            assert pick["option"] == gp.gp_get_option(s.ctx, gp.GP_OPT_SWEEP_PATH) == gp.GP_PATH_AUTO
            assert pick["path"] == gp.GP_PATH_TMA and gp.gp_get_option(s.ctx, gp.GP_OPT_TILE_SHAPE) == 0
            ms.append(pick["ms"])
    assert ms[0] == ms[1]


def test_choices_cached_before_a_change_of_the_kernels_are_not_applied():
    assert autotune.problem_key((64, 64, 64), (0.2,) * 3, 0.002, 1, 0).endswith("/t%d" % autotune.SHAPE_TABLE)
    assert autotune.SHAPE_TABLE > 2
