"""The weight gradient's division over blocks: input channels in blocks of 32 of which the last may be half filled, 128 at once with
few output channels, grids of one and two planes (taps that meet no plane) and long thin ones (many chunks along z), against the
FP64 oracle (sums of n d h w bf16 products accumulated in fp32: 2e-5 of the largest, as for the other tests of this kernel),
and its time against that of a layer with more channels."""
import numpy as np
import pytest

from test_gpu_nn import bf, env, no_failed_waits, relerr  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


def work(torch, L, cout, cin, n, d, h, w):
    nb = L.pfnn_conv3d_wgrad_work_bytes(cout, cin, n, d, h, w)
    return torch.empty(nb, dtype=torch.uint8, device="cuda"), nb


@pytest.mark.parametrize("cin,cout", [(16, 64), (32, 16), (48, 32), (48, 128), (64, 64), (80, 16), (128, 16), (128, 32), (128, 64),
                                      (192, 128), (256, 32)])
@pytest.mark.parametrize("n,d,h,w", [(1, 1, 17, 9), (2, 2, 5, 8), (1, 200, 2, 3), (2, 7, 18, 17)])
def test_wgrad_against_oracle(env, cin, cout, n, d, h, w):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = np.random.default_rng(cin + cout + d)
    xt, x = bf(torch, g.standard_normal((n, d, h, w, cin)))
    dyt, dy = bf(torch, g.standard_normal((n, d, h, w, cout)))
    dw = torch.zeros((27, cout, cin), dtype=torch.float32, device="cuda")
    buf, nb = work(torch, L, cout, cin, n, d, h, w)
    assert L.pfnn_conv3d_wgrad(nn._p(dyt), cout, 0, cout, nn._p(xt), cin, 0, cin, nn._p(dw), n, d, h, w, nn._p(buf), nb, None) == 0
    torch.cuda.synchronize()
    assert relerr(dw.cpu().numpy(), O.conv3d_bwd_weight(dy, x)) <= 2e-5
    assert no_failed_waits(nn)


@pytest.mark.parametrize("n,d,h,w", [(2, 33, 33, 33), (1, 1, 300, 300)])
def test_channels_cost_no_more_than_their_share(env, n, d, h, w):  # noqa: F811
    """192 input channels take no longer than three times 64 (the margin is the spread of short runs), nor 64 than twice 32."""
    torch, nn, O = env
    L = nn._lib()
    cout, t = 128, {}
    dy = torch.randn((n, d, h, w, cout), device="cuda").to(torch.bfloat16)
    for cin in (32, 64, 192):
        x = torch.randn((n, d, h, w, cin), device="cuda").to(torch.bfloat16)
        dw = torch.zeros((27, cout, cin), device="cuda")
        buf, nb = work(torch, L, cout, cin, n, d, h, w)
        torch.cuda.synchronize()
        t[cin] = 1e9
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(torch.cuda.default_stream())
            for _ in range(10):
                assert L.pfnn_conv3d_wgrad(nn._p(dy), cout, 0, cout, nn._p(x), cin, 0, cin, nn._p(dw), n, d, h, w, nn._p(buf), nb,
                                           None) == 0
            e1.record(torch.cuda.default_stream())
            e1.synchronize()
            t[cin] = min(t[cin], e0.elapsed_time(e1))
    assert t[64] <= 1.15 * 2 * t[32] and t[192] <= 1.15 * 3 * t[64], t
    assert no_failed_waits(nn)
