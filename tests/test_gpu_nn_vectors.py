"""Vector and single-channel forms of the network's data-movement, head and bias kernels: channel counts, leading
dimensions and offsets that take 16-byte vectors and ones that do not, against plain numpy in binary64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_01672_gb300 import nn
    return torch, nn, nn._lib()


def children(a):
    """(n, d, h, w, c) -> (n, d/2, h/2, w/2, 8, c)"""
    n, d, h, w, c = a.shape
    return a.reshape(n, d // 2, 2, h // 2, 2, w // 2, 2, c).transpose(0, 1, 3, 5, 2, 4, 6, 7).reshape(
        n, d // 2, h // 2, w // 2, 8, c)


def spread(a):
    return a.repeat(2, 1).repeat(2, 2).repeat(2, 3)


# (channels, channels per voxel of the wide buffer, offset): vectors of 8, of 4 only, single channels
@pytest.mark.parametrize("c,ld,off", [(16, 16, 0), (8, 24, 8), (32, 48, 16), (4, 12, 4), (5, 9, 3), (16, 20, 2)])
@pytest.mark.parametrize("shape", [(1, 2, 2, 2), (2, 4, 6, 10)])
def test_pool_and_upsample(env, c, ld, off, shape):
    torch, nn, L = env
    g = np.random.default_rng(c + 7 * ld)
    n, d, h, w = shape
    big = torch.from_numpy(g.standard_normal((n, d, h, w, ld)).astype(np.float32)).cuda().to(torch.bfloat16)
    x = big[..., off:off + c].double().cpu().numpy()
    y = torch.zeros((n, d // 2, h // 2, w // 2, ld), dtype=torch.bfloat16, device="cuda")
    assert L.pfnn_avgpool(nn._p(big), ld, off, nn._p(y), ld, off, c, n, d, h, w, None) == 0
    ref = np.zeros((n, d // 2, h // 2, w // 2, c), np.float32)  # the children in order, in binary32
    for o in range(8):
        ref += children(x)[..., o, :].astype(np.float32)
    torch.cuda.synchronize()
    assert torch.equal(y[..., off:off + c].cpu(), torch.from_numpy(ref * np.float32(0.125)).to(torch.bfloat16))
    small = y[..., off:off + c].contiguous()
    up = torch.zeros((n, d, h, w, ld), dtype=torch.bfloat16, device="cuda")
    assert L.pfnn_upsample(nn._p(small), c, nn._p(up), ld, off, n, d, h, w, None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(up[..., off:off + c].float().cpu().numpy(), spread(small.float().cpu().numpy()))
    rest = torch.ones(ld, dtype=torch.bool)
    rest[off:off + c] = False
    assert not bool(up[..., rest.cuda()].any()) and not bool(y[..., rest.cuda()].any())
    # adjoints, accumulating
    gf = torch.from_numpy(g.standard_normal((n, d, h, w, ld)).astype(np.float32)).cuda()
    gc = torch.from_numpy(g.standard_normal((n, d // 2, h // 2, w // 2, c)).astype(np.float32)).cuda()
    want_f = gf.double().cpu().numpy()
    want_f[..., off:off + c] += spread(gc.double().cpu().numpy()) / 8
    want_c = gc.double().cpu().numpy() + children(gf[..., off:off + c].double().cpu().numpy()).sum(axis=4)
    acc = gc.clone()
    assert L.pfnn_upsample_bwd(nn._p(gf), ld, off, c, nn._p(acc), n, d // 2, h // 2, w // 2, None) == 0
    assert L.pfnn_avgpool_bwd(nn._p(gc), c, nn._p(gf), ld, off, n, d, h, w, None) == 0
    torch.cuda.synchronize()
    assert np.abs(acc.double().cpu().numpy() - want_c).max() <= 9 * 2 ** -24 * 20
    assert np.abs(gf.double().cpu().numpy() - want_f).max() <= 2 ** -23 * 8


@pytest.mark.parametrize("c,ld,off", [(16, 16, 0), (128, 128, 0), (8, 24, 8), (48, 48, 0), (5, 9, 3), (200, 200, 0)])
@pytest.mark.parametrize("nvox", [1, 700])
def test_relu_backward_and_bias(env, c, ld, off, nvox):
    torch, nn, L = env
    g = np.random.default_rng(c + nvox)
    dy = torch.from_numpy(g.standard_normal((nvox, ld)).astype(np.float32)).cuda()
    y = torch.from_numpy(g.standard_normal((nvox, ld)).astype(np.float32)).cuda().to(torch.bfloat16)
    want = dy[:, off:off + c].double().cpu().numpy() * (y[:, off:off + c].double().cpu().numpy() > 0)
    dzf = torch.empty((nvox, c), dtype=torch.float32, device="cuda")
    dzb = torch.empty((nvox, c), dtype=torch.bfloat16, device="cuda")
    assert L.pfnn_relu_bwd_cast(nn._p(dy), ld, off, nn._p(y), ld, off, c, nvox, nn._p(dzf), nn._p(dzb), None) == 0
    db = torch.full((c,), 0.5, dtype=torch.float32, device="cuda")
    assert L.pfnn_bias_grad(nn._p(dzf), c, 0, c, nvox, nn._p(db), None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(dzf.double().cpu().numpy(), want)
    assert torch.equal(dzb, dzf.to(torch.bfloat16))
    ref = 0.5 + want.sum(axis=0)
    bound = nvox * 2 ** -24 * (0.5 + np.abs(want).sum(axis=0)) + 1e-7
    assert np.all(np.abs(db.double().cpu().numpy() - ref) <= bound)


@pytest.mark.parametrize("c", [1, 8, 13, 16, 24, 32])
@pytest.mark.parametrize("nvox", [1, 3000])
def test_head(env, c, nvox):
    torch, nn, L = env
    g = np.random.default_rng(c + nvox)
    x = torch.from_numpy(g.standard_normal((nvox, c)).astype(np.float32) * 2).cuda().to(torch.bfloat16)
    w = torch.from_numpy((g.standard_normal(c) * 3).astype(np.float32)).cuda()  # some probabilities reach the clamp
    b = torch.tensor([0.3], dtype=torch.float32, device="cuda")
    t = torch.from_numpy(g.uniform(0, 1, nvox).astype(np.float32)).cuda()
    prob, dl = torch.empty(nvox, device="cuda"), torch.empty(nvox, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert L.pfnn_head_forward(nn._p(x), c, nn._p(w), nn._p(b), nn._p(t), nvox, nn._p(prob), nn._p(dl), nn._p(loss), None) == 0
    dx = torch.empty((nvox, c), device="cuda")
    dw, db = torch.zeros(c, device="cuda"), torch.zeros(1, device="cuda")
    assert L.pfnn_head_backward(nn._p(x), c, nn._p(w), nn._p(dl), nvox, nn._p(dx), nn._p(dw), nn._p(db), None) == 0
    torch.cuda.synchronize()
    xd, wd, td = (v.double().cpu().numpy() for v in (x, w, t))
    s = xd @ wd + float(b)
    size = np.abs(xd) @ np.abs(wd) + 1.0  # the fp32 logit is within (c + 1) 2^-24 of this
    ds = (c + 1) * 2 ** -24 * size
    p = 1 / (1 + np.exp(-s))
    assert np.all(np.abs(prob.double().cpu().numpy() - p) <= 0.25 * ds + 2 ** -21)
    pc, qc = np.clip(p, 1e-7, 1 - 1e-7), np.clip(1 / (1 + np.exp(s)), 1e-7, 1 - 1e-7)
    ref = -(td * np.log(pc) + (1 - td) * np.log(qc)).mean()
    assert abs(float(loss) - ref) <= ds.mean() + 1e-12
    d = dl.double().cpu().numpy()
    assert np.all(np.abs(d - (p - td) / nvox) <= (0.25 * ds + 2 ** -20) / nvox)
    assert np.all(np.abs(dx.double().cpu().numpy() - d[:, None] * wd) <= 2 ** -23 * np.abs(d[:, None] * wd) + 1e-30)
    tol = (nvox + 10) * 2 ** -24
    assert np.all(np.abs(dw.double().cpu().numpy() - d @ xd) <= tol * (np.abs(d) @ np.abs(xd)) + 1e-30)
    assert abs(float(db) - d.sum()) <= tol * np.abs(d).sum() + 1e-30


# every division of the taps over blocks (all dz in one block, one dz, one (dz, dy); dy stacked along M or not),
# channel blocks of 16, 32, 64 and 128, several z chunks, ragged columns, slices that are not on 16 bytes
@pytest.mark.parametrize("cin,cout,shape,skew", [
    (16, 16, (1, 37, 17, 9), 0), (16, 32, (2, 5, 16, 8), 1), (16, 64, (1, 4, 33, 7), 0), (32, 32, (1, 21, 5, 17), 0),
    (32, 128, (1, 3, 18, 10), 0), (64, 16, (1, 7, 20, 12), 3), (64, 32, (3, 2, 3, 8), 0), (64, 64, (1, 6, 15, 9), 0),
    (128, 128, (1, 3, 9, 9), 0), (96, 16, (1, 2, 17, 8), 0), (256, 32, (1, 2, 3, 5), 0), (16, 16, (1, 1, 1, 1), 0)])
def test_weight_gradient_plans(env, cin, cout, shape, skew):
    torch, nn, L = env
    from oracle import nn_oracle as O
    g = np.random.default_rng(cin + 3 * cout)
    n, d, h, w = shape
    big = [torch.from_numpy(g.standard_normal((n, d, h, w, c + skew)).astype(np.float32)).cuda().to(torch.bfloat16)
           for c in (cin, cout)]
    x, dy = (b[..., skew:].double().cpu().numpy() for b in big)
    dw = torch.zeros((27, cout, cin), device="cuda")
    wb = L.pfnn_conv3d_wgrad_work_bytes(cout, cin, n, d, h, w)
    work = torch.full((wb,), 255, dtype=torch.uint8, device="cuda")
    assert L.pfnn_conv3d_wgrad(nn._p(big[1]), cout + skew, skew, cout, nn._p(big[0]), cin + skew, skew, cin, nn._p(dw),
                               n, d, h, w, nn._p(work), wb, None) == 0
    torch.cuda.synchronize()
    ref = O.conv3d_bwd_weight(dy, x)
    # binary32 sums of n d h w products in any order
    assert np.abs(dw.double().cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
    flag = nn.C.c_int(-1)
    assert L.pfnn_status(nn.C.byref(flag)) == 0 and flag.value == 0
