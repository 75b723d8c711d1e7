"""Bias sums of any channel count: against binary64 (sums of 32^3 fp32 values: 1e-5 of the sum of their absolute values, which
covers any order), and vectors no slower than the single channels of an unaligned array."""
import numpy as np
import pytest

from test_gpu_nn import env  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c", [4, 8, 12, 16, 32, 64, 128, 256, 1024])
@pytest.mark.parametrize("nvox", [1, 37, 32768])
def test_bias_sums(env, c, nvox):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    x = np.random.default_rng(c + nvox).standard_normal((nvox, c)).astype(np.float32)
    t = torch.from_numpy(x).cuda()
    db = torch.ones(c, device="cuda")
    assert L.pfnn_bias_grad(nn._p(t), c, 0, c, nvox, nn._p(db), None) == 0
    torch.cuda.synchronize()
    err = np.abs(db.cpu().numpy() - 1.0 - x.astype(np.float64).sum(0))
    assert np.all(err <= 1e-5 * (1.0 + np.abs(x).astype(np.float64).sum(0)))


@pytest.mark.parametrize("c", [64, 128, 256])
def test_vectors_are_not_slower_than_single_channels(env, c):  # noqa: F811
    torch, nn, O = env
    L = nn._lib()
    nvox = 32768
    buf = torch.randn(nvox * (c + 4) + 4, device="cuda")
    db = torch.zeros(c, device="cuda")

    def time(at):
        best = 1e9
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(torch.cuda.default_stream())
            for _ in range(20):
                assert L.pfnn_bias_grad(buf.data_ptr() + 4 * at, c, 0, c, nvox, nn._p(db), None) == 0
            e1.record(torch.cuda.default_stream())
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    assert time(0) <= 1.5 * time(1)  # (one float off 16 bytes: the kernel for any alignment)
