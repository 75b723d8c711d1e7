"""Tiles nobody set against the 8 x 32 of a fixed choice: never clearly slower, whatever the model, the grid's shape and where
the temperatures lie (the margin is the spread of short runs; the shapes are chosen within 2 to 3 % of it)."""
import time

import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_tiles import grid, pf  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


def attempt(g):
    best = 1e9
    g.run_fixed(16, 1e-4)
    for _ in range(5):
        t = time.perf_counter()
        g.run_fixed(16, 1e-4)
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("model,prec,shape", [
    (I.MODEL_TEMP, I.PREC_FP64, (128, 128, 128)), (I.MODEL_TEMP, I.PREC_FP64, (160, 160, 160)),
    (I.MODEL_TEMP, I.PREC_FP64, (128, 128, 64)), (I.MODEL_TEMP, I.PREC_FP64, (300, 300, 4)), (I.MODEL_TEMP, I.PREC_FP64, (17, 2000, 5)),
    (I.MODEL_TEMP, I.PREC_FP64, (50, 50, 100)), (I.MODEL_TEMP, I.PREC_FP32, (100, 100, 100)),
    (I.MODEL_MICRO, I.PREC_FP64, (300, 300, 2)), (I.MODEL_MICRO, I.PREC_FP32, (1000, 1000, 1)),
    (I.MODEL_FULL, I.PREC_FP64, (700, 700, 2)), (I.MODEL_MICRO, I.PREC_FP64, (64, 64, 64))])
def test_default_tiles_are_not_slower(pf, model, prec, shape):  # noqa: F811
    free, fixed = grid(pf, shape, model, prec), grid(pf, shape, model, prec)
    fixed.set_tiles(8, 32)
    assert attempt(free) <= 1.15 * attempt(fixed), free.get_tiles()
    free.close()
    fixed.close()
