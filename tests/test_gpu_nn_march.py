"""The convolution kernel that keeps all taps' weights in shared memory and marches through bricks of 8 x 16 columns, against
the FP64 oracle: every pair of channel counts it takes, bricks cut off on every side, more bricks than blocks, and its
failure path.  fp32 outputs of sums of at most 27 x 64 bf16 products accumulated in fp32: 2e-5 of the largest, as for the
other tensor-core kernels."""
import math

import numpy as np
import pytest

from test_gpu_nn import bf, env, no_failed_waits, relerr  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(16, 16), (16, 32), (16, 64), (32, 16), (32, 32), (32, 64), (64, 16), (64, 32)])
@pytest.mark.parametrize("n,d,h,w", [(1, 4, 16, 8), (2, 9, 17, 21)])
def test_march_against_oracle(env, cin, cout, n, d, h, w):
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(cin + cout + d)
    wide, x = bf(torch, g.standard_normal((n, d, h, w, cin + 16)))
    wt, wv = bf(torch, g.standard_normal((27, cout, cin)) / math.sqrt(27 * cin))
    b = g.standard_normal(cout).astype(np.float32)
    y = torch.full((n * d * h * w, cout + 8), 5.0, dtype=torch.float32, device="cuda")
    assert L.pfnn_conv3d(nn._p(wide), cin + 16, 8, nn._p(wt), cin, cout, nn._p(torch.from_numpy(b).cuda()), 1, 0, None,
                         nn._p(y), cout + 8, 8, 0, n, d, h, w, None) == 0
    torch.cuda.synchronize()
    o = y.cpu().numpy()
    ref = O.conv3d(x[..., 8:8 + cin], wv, b.astype(np.float64), relu=True).reshape(-1, cout)
    assert relerr(o[:, 8:], ref) <= 2e-5 and np.all(o[:, :8] == 5.0)
    # backward data, added to what is there
    dyt, dy = bf(torch, g.standard_normal((n, d, h, w, cin)))
    wtr, wv = bf(torch, g.standard_normal((27, cout, cin)) / math.sqrt(27 * cin))
    base = g.standard_normal((n * d * h * w, cout)).astype(np.float32)
    dx = torch.from_numpy(base.copy()).cuda()
    assert L.pfnn_conv3d(nn._p(dyt), cin, 0, nn._p(wtr), cin, cout, None, 0, 1, None, nn._p(dx), cout, 0, 1, n, d, h, w,
                         None) == 0
    torch.cuda.synchronize()
    ref = O.conv3d(dy, wv[::-1]).reshape(-1, cout)
    assert relerr(dx.cpu().numpy() - base, ref) <= 2e-5
    assert no_failed_waits(nn)


@pytest.mark.parametrize("cin,cout", [(16, 16), (64, 32)])
def test_march_more_bricks_than_blocks(env, cin, cout):
    """Blocks that walk several bricks (both accumulator sets, slots reused across bricks of different heights): every
    sample equals the same sample run by itself."""
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(cin)
    n, d, h, w = 24, 11, 48, 40
    x = torch.randn((n, d, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y = torch.zeros((n, d, h, w, cout), device="cuda")
    one = torch.zeros((d, h, w, cout), device="cuda")
    assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, 0, None, nn._p(y), cout, 0, 0, n, d, h, w, None) == 0
    for q in (0, 7, n - 1):
        assert L.pfnn_conv3d(nn._p(x[q]), cin, 0, nn._p(wt), cin, cout, None, 0, 0, None, nn._p(one), cout, 0, 0, 1, d, h, w,
                             None) == 0
        torch.cuda.synchronize()
        assert torch.equal(y[q], one)
    assert no_failed_waits(nn)


@pytest.mark.parametrize("flip", [0, 1])
@pytest.mark.parametrize("cin,cout", [(16, 64), (32, 64), (64, 16), (64, 32)])
def test_march_equals_thin_grids(env, cin, cout, flip):
    """Grids of three planes take the kernel with one box per tap; a fourth plane of zeros changes no sum, and both add a
    cell's products in the same order."""
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(cin)
    h, w = 33, 20
    x = torch.randn((4, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    x[3] = 0
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y4, y3 = torch.zeros((4, h, w, cout), device="cuda"), torch.zeros((3, h, w, cout), device="cuda")
    for y, d in ((y4, 4), (y3, 3)):
        assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, flip, None, nn._p(y), cout, 0, 0, 1, d, h, w,
                             None) == 0
    torch.cuda.synchronize()
    assert torch.equal(y4[:3], y3)
    assert no_failed_waits(nn)


@pytest.mark.parametrize("plane", [1, 3])
def test_march_gives_up_a_withheld_plane_and_recovers(env, plane):
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(13)
    n, d, h, w, cin, cout = 1, 8, 16, 16, 32, 32
    xt, x = bf(torch, g.standard_normal((n, d, h, w, cin)))
    wt, wv = bf(torch, g.standard_normal((27, cout, cin)) / math.sqrt(27 * cin))
    y = torch.full((n * d * h * w, cout), 3.0, dtype=torch.float32, device="cuda")
    assert no_failed_waits(nn)
    assert L.pfnn_test_withhold_stage(plane, 1 << 10) == 0
    call = (nn._p(xt), cin, 0, nn._p(wt), cin, cout, None, 0, 0, None, nn._p(y), cout, 0, 0, n, d, h, w, None)
    assert L.pfnn_conv3d(*call) == 0
    torch.cuda.synchronize()
    assert not no_failed_waits(nn)
    assert bool(torch.all(y == 3.0))
    assert no_failed_waits(nn)
    assert L.pfnn_conv3d(*call) == 0
    torch.cuda.synchronize()
    assert relerr(y.cpu().numpy(), O.conv3d(x, wv).reshape(-1, cout)) <= 2e-5
    assert no_failed_waits(nn)
