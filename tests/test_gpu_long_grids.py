"""Grids longer than 65535 tiles along y or chunks along z (what one launch takes), on tiles nobody set: the same numbers as
with tiles that cover them."""
import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_tiles import pf, state  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 270000, 1), (2, 520000, 2), (1, 2, 1700000), (1, 1, 2090000)])
def test_grids_longer_than_a_launch(pf, shape):  # noqa: F811
    got = []
    for tiles in (None, (8, 32)):
        g = pf.Grid(shape, 1e-7, I.MODEL_MICRO, I.REACT_SIGMAP1P, I.PREC_FP64,
                    I.default_params(xi=1e-7, xi_G=4e-8, zeta=2.0, theta_micro=-0.5, alpha=I.TABLE1["alpha"]))
        g.set_glass(np.zeros(g.N))
        g.set_state(None, np.random.default_rng(3).random(g.N), 0.0, 1e-7)
        if tiles:
            g.set_tiles(*tiles)
        assert g.run_fixed(2, 1e-7)["n_accepted"] == 2
        got.append(state(g))
        g.close()
    assert np.all(np.isfinite(got[0])) and np.array_equal(*got)
