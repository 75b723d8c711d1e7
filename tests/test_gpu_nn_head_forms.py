"""The head with and without a target (two instances of one kernel): the same probabilities bit for bit, every channel count."""
import numpy as np
import pytest

from test_gpu_nn import env  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [1, 3, 8, 12, 16, 20, 24, 31, 32])
@pytest.mark.parametrize("nvox", [1, 1000])
def test_probabilities_with_and_without_a_target(env, c, nvox):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    g = torch.Generator(device="cuda").manual_seed(c)
    x = torch.randn((nvox, c), generator=g, device="cuda").to(torch.bfloat16)
    w, b = torch.randn(c, generator=g, device="cuda"), torch.randn(1, generator=g, device="cuda")
    target = torch.rand(nvox, generator=g, device="cuda")
    a, p, dl = (torch.empty(nvox, device="cuda") for _ in range(3))
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert L.pfnn_head_forward(nn._p(x), c, nn._p(w), nn._p(b), None, nvox, nn._p(a), None, None, None) == 0
    assert L.pfnn_head_forward(nn._p(x), c, nn._p(w), nn._p(b), nn._p(target), nvox, nn._p(p), nn._p(dl), nn._p(loss), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(a, p)
    z = (x.double() @ w.double() + b.double()).cpu().numpy()
    assert np.allclose(a.cpu().numpy(), 1.0 / (1.0 + np.exp(-z)), rtol=0, atol=1e-5)
    t = target.double().cpu().numpy()
    lp, lq = (np.clip(q, np.log(1e-7), np.log1p(-1e-7)) for q in (-np.logaddexp(0, -z), -np.logaddexp(0, z)))
    assert abs(loss.item() - np.mean(-(t * lp + (1 - t) * lq))) <= 1e-5
