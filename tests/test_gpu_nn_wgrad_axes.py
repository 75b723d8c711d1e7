"""The weight gradient on grids a few cells wide, whose axes change places in its tiles: every order of the three axes (with
several samples only the first two), against the FP64 oracle (2e-5 of the largest, as for the other tests of this kernel), and
no slower than a cube of the same voxels times the share of the tiles that such a grid fills at best."""
import numpy as np
import pytest

from test_gpu_nn import bf, env, no_failed_waits, relerr  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(16, 16), (32, 64), (128, 32)])
@pytest.mark.parametrize("n,d,h,w", [(1, 40, 2, 3), (1, 2, 40, 3), (1, 2, 3, 40), (1, 40, 17, 2), (1, 17, 40, 2), (1, 2, 17, 40),
                                     (1, 33, 2, 18), (2, 3, 3, 40), (3, 5, 40, 3), (2, 40, 3, 5)])
def test_axes_against_oracle(env, cin, cout, n, d, h, w):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(cin + cout + d + 2 * h)
    xt, x = bf(torch, g.standard_normal((n, d, h, w, cin + 16)))
    dyt, dy = bf(torch, g.standard_normal((n, d, h, w, cout)))
    dw = torch.zeros((27, cout, cin), dtype=torch.float32, device="cuda")
    nb = L.pfnn_conv3d_wgrad_work_bytes(cout, cin, n, d, h, w)
    buf = torch.empty(nb, dtype=torch.uint8, device="cuda")
    assert L.pfnn_conv3d_wgrad(nn._p(dyt), cout, 0, cout, nn._p(xt), cin + 16, 8, cin, nn._p(dw), n, d, h, w, nn._p(buf), nb,
                               None) == 0
    torch.cuda.synchronize()
    assert relerr(dw.cpu().numpy(), O.conv3d_bwd_weight(dy, x[..., 8:8 + cin])) <= 2e-5
    assert no_failed_waits(nn)


@pytest.mark.parametrize("d,h,w", [(2000, 2, 2), (2, 2, 2000)])
def test_thin_grids(env, d, h, w):  # noqa: F811
    """8 x 16 tiles along the long axis are a quarter full: four times a cube of as many voxels, and half again."""
    torch, nn, O = env
    L = nn._lib()
    cin = cout = 128
    t = []
    for shape in ((d, h, w), (20, 20, 20)):
        x, dy = (torch.randn(shape + (c,), device="cuda").to(torch.bfloat16) for c in (cin, cout))
        dw = torch.zeros((27, cout, cin), device="cuda")
        nb = L.pfnn_conv3d_wgrad_work_bytes(cout, cin, 1, *shape)
        buf = torch.empty(nb, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        best = 1e9
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(torch.cuda.default_stream())
            for _ in range(10):
                assert L.pfnn_conv3d_wgrad(nn._p(dy), cout, 0, cout, nn._p(x), cin, 0, cin, nn._p(dw), 1, *shape, nn._p(buf), nb,
                                           None) == 0
            e1.record(torch.cuda.default_stream())
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        t.append(best)
    assert t[0] <= 6 * t[1], t
    assert no_failed_waits(nn)
