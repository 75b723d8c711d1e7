"""Layers of 16 and 32 channels on both sides: forward, the kernel with resident weights adds a cell's products in the order of the
kernel with a box per tap (bit for bit); backward data takes a flipped copy of the weights there, so its taps come in the
other order (each within 2e-5 of the largest of the exact sums)."""
import math

import pytest

from test_gpu_nn import env, no_failed_waits  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flip", [0, 1])
@pytest.mark.parametrize("cin,cout", [(16, 16), (16, 32), (32, 16), (32, 32)])
def test_narrow_layers_against_thin_grids(env, cin, cout, flip):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    h, w = 33, 20
    x = torch.randn((4, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    x[3] = 0  # changes no sum of the first three planes
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y4, y3 = torch.zeros((4, h, w, cout), device="cuda"), torch.zeros((3, h, w, cout), device="cuda")
    for y, d in ((y4, 4), (y3, 3)):
        assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, flip, None, nn._p(y), cout, 0, 0, 1, d, h, w,
                             None) == 0
    torch.cuda.synchronize()
    if not flip:
        assert torch.equal(y4[:3], y3)
    assert float((y4[:3] - y3).abs().max()) <= 4e-5 * float(y3.abs().max())
    assert no_failed_waits(nn)
