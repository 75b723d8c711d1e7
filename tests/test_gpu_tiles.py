"""Lateral tile shapes (rows of 32 cells and narrower, taller ones), the attempts of a run in groups and one by one, and
batches with more instances than the kernel parameters hold: each against another way to the same numbers, bit for bit."""
import numpy as np
import pytest

from paper_2401_01672_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_01672_gb300 import pf
    return pf


def grid(pf, shape, model, prec, seed=5):
    h = 3e-4
    th, ph, G = I.random_fields(shape, seed)
    p = I.default_params(xi=h, xi_G=0.4 * h, zeta=2.0, alpha=I.ALPHA_MACRO["large"], dirichlet_faces=I.FACE_ZP,
                         theta_freeze=-5.0, theta_thaw=2.0, theta_micro=-0.5)
    g = pf.Grid(shape, h, model, I.REACT_SIGMAP1P, prec, p)
    g.set_glass(G)
    g.set_state(None if model == I.MODEL_MICRO else th, None if model == I.MODEL_TEMP else ph, 0.0, 1e-3)
    return g


def state(g):
    th, ph, t, dt = g.get_state()
    return np.concatenate([np.asarray(th).ravel(), np.asarray(ph).ravel(), [t]])


@pytest.mark.parametrize("prec", [I.PREC_FP64, I.PREC_FP32])
@pytest.mark.parametrize("model", [I.MODEL_FULL, I.MODEL_TEMP, I.MODEL_MICRO])
@pytest.mark.parametrize("n1,n2,n3", [(21, 13, 7), (25, 5, 9), (33, 6, 6), (40, 18, 5), (50, 50, 8), (64, 9, 4), (63, 4, 11)])
def test_every_tile_gives_the_same_numbers(pf, n1, n2, n3, model, prec):
    """n1 = 21, 40, 63 take tiles of 21 x 6, 25 and 50 of 25 x 5, 64 of 32 x 4 with blocks of 128 threads; the blocks of 256
    and 512 take other shapes."""
    want = None
    for tiles in (None, (4, 1), (4, 3), (8, 2), (8, 32), (16, 4)):
        g = grid(pf, (n1, n2, n3), model, prec)
        if tiles:
            g.set_tiles(*tiles)
        g.run_fixed(3, 1e-3)
        s = state(g)
        g.close()
        assert np.all(np.isfinite(s))
        want = s if want is None else want
        assert np.array_equal(s, want), tiles


@pytest.mark.parametrize("n", [1, 15, 16, 21, 37, 300])
def test_runs_of_any_length(pf, n):
    one, many = (grid(pf, (20, 12, 10), I.MODEL_FULL, I.PREC_FP64) for _ in range(2))
    for _ in range(n):
        one.run_fixed(1, 1e-3)
    s = many.run_fixed(n, 1e-3)
    assert s["n_accepted"] == n and s["launches"] == 6 * n
    assert np.array_equal(state(one), state(many))
    a, b = one.run_to(1e30, 1e-6, n), many.run_to(1e30, 1e-6, n)
    assert a["n_accepted"] + a["n_rejected"] == n and (a["t"], a["n_accepted"]) == (b["t"], b["n_accepted"])
    assert np.array_equal(state(one), state(many))
    end = a["t"] + 2.5 * a["dt"]  # ends within the first launches
    a = one.run_to(end, 1e-6, 1000)
    assert a["t"] == end
    one.close()
    many.close()


@pytest.mark.parametrize("prec", [I.PREC_FP64, I.PREC_FP32])
def test_batch_beyond_the_kernel_parameters(pf, prec):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    h, grids, alone = 1e-7, [], []
    for q in range(63):
        shape = (8 + q % 5, 9, 7 + q % 3)
        _, ph, G = I.random_fields(shape, q)
        p = I.default_params(xi=h, xi_G=0.4 * h, zeta=2.0, theta_micro=-0.5, alpha=I.TABLE1["alpha"])
        for out, kw in ((grids, {"stream": stream}), (alone, {})):
            g = pf.Grid(shape, h, I.MODEL_MICRO, I.REACT_SIGMAP1P, prec, p, **kw)
            g.set_glass(G)
            g.set_state(None, ph, 0.0, 1e-6)
            out.append(g)
    b = pf.Batch(grids)
    res = b.run_to([1e30] * 63, 1e-6, 9)
    for g, a, r in zip(grids, alone, res):
        s = a.run_to(1e30, 1e-6, 9)
        assert (r["n_accepted"], r["n_rejected"], r["t"]) == (s["n_accepted"], s["n_rejected"], s["t"])
        assert np.array_equal(state(g), state(a))
