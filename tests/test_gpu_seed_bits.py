"""The seed constraint on grids whose rows end inside a word, span several tiles, or take the byte form, against
scipy's morphology on the CPU (the outputs are selections of the inputs, so they are equal bit for bit)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def expected(prob, seed, G, zeta, halo, erode):
    nd = pytest.importorskip("scipy.ndimage")
    face = nd.generate_binary_structure(3, 1)
    water = 1.0 - zeta * G > 0.0
    ice = (prob > 0.5) & water
    cut = nd.binary_erosion(ice, face, erode, border_value=1) if erode else ice
    start = seed > 0.5
    grown = start | nd.binary_propagation(start | (nd.binary_dilation(start, face) & cut), face, mask=cut | start)
    for _ in range(erode):
        grown = grown | (nd.binary_dilation(grown, face) & ice)
    if halo:
        grown = nd.binary_dilation(grown, face, halo)
    p = np.clip(prob, 0.0, 1.0).astype(np.float64)
    return np.where(water & grown, np.maximum(p, seed), seed)


def labyrinth(shape):
    """Ice everywhere but in walls normal to y, open at one end in turn: the fill crosses every row of tiles."""
    prob = np.full(shape, 0.9, np.float32)
    for q, j in enumerate(range(2, shape[1] - 1, 3)):
        prob[:, j, :] = 0.1
        prob[:, j, -1 if q % 2 == 0 else 0] = 0.9
    return prob


@pytest.mark.parametrize("n1,n2,n3,halo,erode,walls", [
    (17, 21, 19, 3, 0, False), (5, 40, 33, 2, 1, False), (31, 16, 16, 0, 0, False), (32, 17, 33, 3, 1, False),
    (33, 19, 18, 3, 2, False), (64, 16, 15, 1, 0, False), (65, 33, 17, 3, 1, False), (130, 35, 40, 3, 0, False),
    (130, 70, 20, 0, 0, True), (200, 96, 4, 2, 0, True), (16, 30, 9, 3, 0, True), (1, 64, 64, 1, 0, False)])
def test_seed_constraint_against_morphology(n1, n2, n3, halo, erode, walls):
    import torch
    from paper_2401_01672_gb300 import nn as NN
    g = np.random.default_rng(n1 * 1000 + n2 + n3)
    shape = (n3, n2, n1)
    prob = labyrinth(shape) if walls else (g.random(shape) < (0.9 if erode else 0.55)).astype(np.float32) * 0.8
    prob = (prob + 0.1 * g.random(shape)).astype(np.float32)
    seed = np.zeros(shape)
    seed[0, 0, :3] = 1.0
    if not walls:
        seed[:, n2 // 2, n1 // 2] = 0.75
    G = np.where(g.random(shape) < 0.02, 0.6, 0.0) if not walls else np.zeros(shape)
    out, sweeps = NN.seed_connect(torch.from_numpy(prob.ravel()).cuda(), torch.from_numpy(seed.ravel()).cuda(),
                                  torch.from_numpy(G.ravel()).cuda(), (n1, n2, n3), 2.0, halo=halo, erode=erode)
    assert sweeps % 16 == 0 and sweeps > 0
    assert np.array_equal(out.cpu().numpy().reshape(shape), expected(prob, seed, G, 2.0, halo, erode))
