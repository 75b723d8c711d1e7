"""Grids on the NULL stream, which the C ABI accepts: the stage kernels are dependent launches there too, and give the numbers of a
stream of the grid's own."""
import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_tiles import pf, state  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [I.PREC_FP64, I.PREC_FP32])
@pytest.mark.parametrize("model", [I.MODEL_FULL, I.MODEL_TEMP, I.MODEL_MICRO])
def test_null_stream(pf, model, prec):  # noqa: F811
    torch = pytest.importorskip("torch")
    got = []
    for stream in (None, torch.cuda.default_stream()):
        assert stream is None or stream.cuda_stream == 0
        th, ph, G = I.random_fields((40, 18, 9), 5)
        p = I.default_params(xi=3e-4, xi_G=1.2e-4, zeta=2.0, alpha=I.ALPHA_MACRO["large"], dirichlet_faces=I.FACE_ZP,
                             theta_freeze=-5.0, theta_thaw=2.0, theta_micro=-0.5)
        g = pf.Grid((40, 18, 9), 3e-4, model, I.REACT_SIGMAP1P, prec, p, stream=stream)
        g.set_glass(G)
        g.set_state(None if model == I.MODEL_MICRO else th, None if model == I.MODEL_TEMP else ph, 0.0, 1e-3)
        g.run_fixed(37, 1e-3)
        r = g.run_to(1e30, 1e-6, 21)
        got.append((state(g), r["t"], r["n_accepted"]))
        g.close()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1:] == got[1][1:]
