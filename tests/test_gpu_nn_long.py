"""A wide layer on a grid of many planes: choosing the planes of a work item takes time that grows with the planes, not with
their square, and the first planes equal those of a short grid bit for bit (the products of a
cell are added in the same order by every kernel)."""
import math
import time

import pytest

from test_gpu_nn import env, no_failed_waits  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu


def test_wide_layer_on_many_planes(env):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(1)
    d, h, w, cin, cout, short = 12000, 16, 9, 64, 64, 40
    x = torch.randn((d, h, w, cin), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((27, cout, cin), generator=g, device="cuda") / math.sqrt(27 * cin)).to(torch.bfloat16)
    y, part = (torch.empty((q, h, w, cout), dtype=torch.bfloat16, device="cuda") for q in (d, short))
    host = []
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, 0, nn._p(y), None, cout, 0, 0, 1, d, h, w,
                             None) == 0
        host.append(time.perf_counter() - t)
    assert min(host) < 0.01
    assert L.pfnn_conv3d(nn._p(x), cin, 0, nn._p(wt), cin, cout, None, 0, 0, nn._p(part), None, cout, 0, 0, 1, short, h, w,
                         None) == 0
    torch.cuda.synchronize()
    assert torch.equal(y[:short - 1], part[:short - 1])
    assert no_failed_waits(nn)
