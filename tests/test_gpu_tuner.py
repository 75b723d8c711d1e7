"""The tuner against the tiles that nobody set: never clearly slower (the margin is the spread of short runs), and the state as
it was."""
import time

import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_tiles import grid, pf, state  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


def attempt(g):
    best = 1e9
    g.run_fixed(16, 1e-4)
    for _ in range(6):
        t = time.perf_counter()
        g.run_fixed(16, 1e-4)
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("model,prec,shape", [
    (I.MODEL_MICRO, I.PREC_FP64, (32, 32, 32)), (I.MODEL_TEMP, I.PREC_FP64, (16, 16, 16)), (I.MODEL_TEMP, I.PREC_FP64, (24, 24, 24)),
    (I.MODEL_MICRO, I.PREC_FP64, (64, 64, 64)), (I.MODEL_FULL, I.PREC_FP64, (32, 32, 32)), (I.MODEL_FULL, I.PREC_FP64, (50, 50, 100)),
    (I.MODEL_FULL, I.PREC_FP32, (64, 64, 64)), (I.MODEL_FULL, I.PREC_FP32, (128, 128, 128))])
def test_tuned_is_not_slower_than_untuned(pf, model, prec, shape):  # noqa: F811
    free, tuned = grid(pf, shape, model, prec), grid(pf, shape, model, prec)
    before = state(tuned)
    by, zc, ms = tuned.autotune()
    assert tuned.get_tiles() == (by, zc) and ms > 0 and np.array_equal(state(tuned), before)
    assert attempt(tuned) <= 1.12 * attempt(free), (free.get_tiles(), (by, zc))
    assert np.array_equal(state(tuned), state(free))
    free.close()
    tuned.close()


def test_long_grids_are_tuned(pf):  # noqa: F811
    """Candidates that a launch cannot cover are left out (70000 chunks of two planes, 75000 rows of tiles)."""
    for shape in ((1, 1, 140000), (32, 300000, 1)):
        g = pf.Grid(shape, 1e-7, I.MODEL_MICRO, I.REACT_SIGMAP1P, I.PREC_FP64,
                    I.default_params(xi=1e-7, xi_G=4e-8, zeta=2.0, theta_micro=-0.5, alpha=I.TABLE1["alpha"]))
        g.set_glass(np.zeros(g.N))
        g.set_state(None, np.random.default_rng(3).random(g.N), 0.0, 1e-7)
        by, zc, ms = g.autotune()
        assert ms > 0 and g.run_fixed(2, 1e-7)["n_accepted"] == 2
        g.close()
