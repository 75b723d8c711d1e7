"""The batch tuner against the tiles that nobody set: never clearly slower (the margin is the spread of short runs), the state as
it was, the same numbers after, and each instance's own tiles in the file for the single-grid tuner."""
import time

import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I
from test_gpu_tiles import pf, state  # noqa: F401  (pf is a fixture)

pytestmark = pytest.mark.gpu


def batch(pf, shapes, model, prec, stream, tiles=None):  # noqa: F811
    grids, init = [], []
    for q, shape in enumerate(shapes):
        th, ph, G = I.random_fields(shape, q)
        p = I.default_params(xi=3e-4, xi_G=1.2e-4, zeta=2.0, alpha=I.ALPHA_MACRO["large"], dirichlet_faces=I.FACE_ZP,
                             theta_freeze=-5.0, theta_thaw=2.0, theta_micro=-0.5)
        g = pf.Grid(shape, 3e-4, model, I.REACT_SIGMAP1P, prec, p, stream=stream)
        g.set_glass(G)
        if tiles:
            g.set_tiles(*tiles)
        init.append((None if model == I.MODEL_MICRO else th, None if model == I.MODEL_TEMP else ph))
        g.set_state(*init[-1], 0.0, 1e-5)
        grids.append(g)
    return pf.Batch(grids), grids, init


@pytest.mark.parametrize("model,prec,shapes", [
    (I.MODEL_FULL, I.PREC_FP32, [(64, 64, 64)] * 8), (I.MODEL_TEMP, I.PREC_FP32, [(64, 64, 64)] * 8),
    (I.MODEL_TEMP, I.PREC_FP64, [(24, 24, 24), (96, 96, 96), (50, 50, 100)]),
    (I.MODEL_MICRO, I.PREC_FP32, [(24, 24, 24), (96, 96, 96), (50, 50, 100)]), (I.MODEL_MICRO, I.PREC_FP64, [(33, 20, 9)] * 63)])
def test_tuned_batch_is_not_slower(pf, tmp_path, model, prec, shapes):  # noqa: F811
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    ms, ends = [], []
    for tune in (False, True):
        b, grids, init = batch(pf, shapes, model, prec, stream)
        if tune:
            before = [state(g) for g in grids]
            tiles = b.autotune()
            assert len({by for by, _ in tiles}) == 1
            assert all(np.array_equal(state(g), s) for g, s in zip(grids, before))
        best = 1e9
        for _ in range(5):
            for g, f in zip(grids, init):
                g.set_state(*f, 0.0, 1e-5)
            torch.cuda.synchronize()
            t = time.perf_counter()
            b.run_to([1e30] * len(grids), 1e-6, 24)
            best = min(best, time.perf_counter() - t)
        ms.append(best)
        ends.append([state(g) for g in grids])
        b.close()
    assert all(np.array_equal(u, v) for u, v in zip(*ends))
    assert ms[1] <= 1.1 * ms[0], (ms, tiles)


def test_instances_own_tiles_are_cached(pf, tmp_path):  # noqa: F811
    torch = pytest.importorskip("torch")
    cache = str(tmp_path / "tiles.txt")
    b, grids, _ = batch(pf, [(24, 20, 18), (40, 33, 21)], I.MODEL_MICRO, I.PREC_FP32, torch.cuda.Stream())
    b.autotune(cache)
    lines = [line.split() for line in open(cache)]
    assert [line[0].split("/")[0] for line in lines] == ["24x20x18", "40x33x21"]
    b.close()
    alone, grids, _ = batch(pf, [(40, 33, 21)], I.MODEL_MICRO, I.PREC_FP32, torch.cuda.Stream())
    assert grids[0].autotune(cache)[:2] == tuple(int(v) for v in lines[1][1:3])
    alone.close()
