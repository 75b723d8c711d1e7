"""The convolution kernel that streams its weights past pairs of bricks: against the FP64 oracle (fp32 outputs of at most
27 x 192 bf16 products accumulated in fp32: 2e-5 of the largest, as for the other tensor-core kernels), and bit for bit
against the kernel that small calls take, which adds the products of a cell in the same order."""
import math

import numpy as np
import pytest

from test_gpu_nn import bf, env, no_failed_waits, relerr  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,h,w,cin,cout", [(39, 13, 16, 16, 128, 64), (5, 20, 33, 28, 64, 64), (2, 16, 40, 41, 128, 128),
                                              (1, 5, 150, 180, 96, 32), (16, 9, 30, 26, 192, 16), (1, 1, 270, 480, 64, 64)])
def test_wide_against_oracle(env, n, d, h, w, cin, cout):
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(cin + cout + d)
    xt, x = bf(torch, g.standard_normal((n, d, h, w, cin)))
    wt, wv = bf(torch, g.standard_normal((27, cout, cin)) / math.sqrt(27 * cin))
    b = g.standard_normal(cout).astype(np.float32)
    base = g.standard_normal((n * d * h * w, cout)).astype(np.float32)
    y = torch.full((n * d * h * w, cout + 8), 5.0, dtype=torch.float32, device="cuda")
    dx = torch.from_numpy(base.copy()).cuda()
    assert L.pfnn_conv3d(nn._p(xt), cin, 0, nn._p(wt), cin, cout, nn._p(torch.from_numpy(b).cuda()), 1, 0, None,
                         nn._p(y), cout + 8, 8, 0, n, d, h, w, None) == 0
    assert L.pfnn_conv3d(nn._p(xt), cin, 0, nn._p(wt), cin, cout, None, 0, 1, None, nn._p(dx), cout, 0, 1, n, d, h, w,
                         None) == 0
    torch.cuda.synchronize()
    o = y.cpu().numpy()
    assert relerr(o[:, 8:], O.conv3d(x, wv, b.astype(np.float64), relu=True).reshape(-1, cout)) <= 2e-5
    assert np.all(o[:, :8] == 5.0)
    assert relerr(dx.cpu().numpy() - base, O.conv3d(x, wv[::-1]).reshape(-1, cout)) <= 2e-5
    assert no_failed_waits(nn)


@pytest.mark.parametrize("flip", [0, 1])
@pytest.mark.parametrize("n,d,h,w,cin,cout", [(20, 26, 16, 16, 128, 64), (13, 40, 16, 16, 64, 64), (9, 5, 32, 40, 128, 128)])
def test_wide_equals_small_calls(env, n, d, h, w, cin, cout, flip):
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(cin + d)
    x = torch.randn((n, d, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y = torch.zeros((n, d, h, w, cout), device="cuda")
    one = torch.zeros((d, h, w, cout), device="cuda")
    assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, flip, None, nn._p(y), cout, 0, 0, n, d, h, w,
                         None) == 0
    for q in (0, n - 1):
        assert L.pfnn_conv3d(nn._p(x[q]), cin, 0, nn._p(wt), cin, cout, None, 0, flip, None, nn._p(one), cout, 0, 0, 1, d, h, w,
                             None) == 0
        torch.cuda.synchronize()
        assert torch.equal(y[q], one)
    assert no_failed_waits(nn)


@pytest.mark.parametrize("stage", [0, 7])
def test_wide_gives_up_a_withheld_stage_and_recovers(env, stage):
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(14)
    n, d, h, w, cin, cout = 1, 32, 64, 64, 64, 64
    xt, x = bf(torch, g.standard_normal((n, d, h, w, cin)))
    wt, wv = bf(torch, g.standard_normal((27, cout, cin)) / math.sqrt(27 * cin))
    y = torch.full((n * d * h * w, cout), 3.0, dtype=torch.float32, device="cuda")
    assert no_failed_waits(nn)
    assert L.pfnn_test_withhold_stage(stage, 1 << 10) == 0
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
