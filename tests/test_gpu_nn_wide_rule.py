"""Which layers take the kernel that streams its weights: a call takes no longer than four calls on a quarter of its rows, which
are too few for that kernel (the margin is the spread of short runs)."""
import math

import pytest

from test_gpu_nn import env, no_failed_waits  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(64, 64), (128, 64), (192, 32), (128, 16), (64, 128), (128, 128), (32, 128), (64, 80), (64, 48),
                                      (48, 80), (96, 96), (16, 256)])
def test_a_call_is_not_slower_than_four_on_a_quarter(env, cin, cout):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(cin)
    n, d, h, w = 4, 16, 60, 64
    x = torch.randn((n, d, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y = torch.empty((n, d, h, w, cout), dtype=torch.bfloat16, device="cuda")

    def time(rows, calls):
        best = 1e9
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(calls):
                assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, 0, nn._p(y), None, cout, 0, 0, n, d,
                                     rows, w, None) == 0
            e1.record(stream)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    stream = torch.cuda.default_stream()
    whole, parts = time(h, 10), time(h // 4, 40)
    assert whole <= 1.15 * parts, (whole, parts)
    assert no_failed_waits(nn)
