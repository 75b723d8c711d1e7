"""The flood fill over more sweeps than a tile's one-byte note counts (251): a serpentine of ice through many rows of tiles, against
scipy's morphology."""
import numpy as np
import pytest

from test_gpu_seed_bits import expected, labyrinth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2,n3,sweeps", [(700, 96, 1, 251), (1500, 200, 2, 3 * 251)])
def test_more_sweeps_than_a_note_counts(n1, n2, n3, sweeps):
    import torch
    from paper_2401_01672_gb300 import nn as NN
    shape = (n3, n2, n1)
    prob, seed, G = labyrinth(shape), np.zeros(shape), np.zeros(shape)
    seed[0, 0, :3] = 1.0
    out, done = NN.seed_connect(torch.from_numpy(prob.ravel()).cuda(), torch.from_numpy(seed.ravel()).cuda(),
                                torch.from_numpy(G.ravel()).cuda(), (n1, n2, n3), 2.0, halo=0, erode=0)
    assert done > sweeps
    assert np.array_equal(out.cpu().numpy().reshape(shape), expected(prob, seed, G, 2.0, 0, 0))
