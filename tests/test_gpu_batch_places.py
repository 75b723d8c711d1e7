"""Batches of a few more tiles than the chip has places for blocks: the tiles left over do not make an attempt twice as long as
that of the same tiles one plane higher, and the numbers are the same (the margin is the spread of short runs)."""
import time

import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_batch_tuner import batch
from test_gpu_tiles import pf, state  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,prec,tiles,other", [
    (I.MODEL_FULL, I.PREC_FP64, (4, 9), (4, 11)), (I.MODEL_TEMP, I.PREC_FP64, (4, 9), (4, 11)),
    (I.MODEL_MICRO, I.PREC_FP64, (4, 9), (4, 11)), (I.MODEL_TEMP, I.PREC_FP64, (8, 8), (8, 11)),
    (I.MODEL_FULL, I.PREC_FP32, (8, 8), (8, 11))])
def test_a_few_tiles_more_than_places(pf, model, prec, tiles, other):  # noqa: F811
    torch = pytest.importorskip("torch")
    ms, ends = [], []
    for t in (tiles, other):  # 1.12 tiles a place (binary64), and 0.84
        b, grids, init = batch(pf, [(64, 64, 64)] * 4, model, prec, torch.cuda.Stream(), t)
        best = 1e9
        for _ in range(5):
            for g, f in zip(grids, init):
                g.set_state(*f, 0.0, 1e-5)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            b.run_to([1e30] * len(grids), 1e-6, 16)
            best = min(best, time.perf_counter() - t0)
        ms.append(best)
        ends.append([state(g) for g in grids])
        b.close()
    assert all(np.array_equal(u, v) for u, v in zip(*ends))
    assert ms[0] <= 1.25 * ms[1], ms
