"""The training kernels at the edges of their tiles: FP32 convolutions around chunks of 16 input
channels and groups of four pixels, weight gradients around the channel counts that choose a
kernel and with several tiles per block, ReLU masks and losses around vector and grid sizes.

An FP32 sum of n products in any order differs from the exact one by at most about
n 2^-24 of the sum of the terms' magnitudes; the products of BF16 with FP32 values add half an
ulp each, which fmaf does not take.  The tolerances are that bound with n + 2.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import cnn_ref  # noqa: E402

EPS = 2.0 ** -24


@pytest.fixture(scope="module")
def m():
    from paper_2001_09678_gb300 import build, mpv
    build.build()
    mpv.load()
    return mpv


def _bf(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda().to(torch.bfloat16)


@pytest.mark.parametrize("n,cin,h,w,bias,relu", [
    (1, 1, 1, 1, True, False), (2, 15, 16, 16, False, True), (1, 16, 17, 20, True, True),
    (1, 17, 15, 33, False, False), (3, 32, 33, 18, True, False), (1, 33, 5, 64, False, False)])
def test_conv_fp32_input(m, n, cin, h, w, bias, relu):
    rng = np.random.default_rng(cin * 3 + w)
    x = rng.normal(size=(n, cin, h, w)).astype(np.float32)
    wt = rng.normal(size=(32, cin, 3, 3)).astype(np.float32)
    b = rng.normal(size=32).astype(np.float32) if bias else None
    out = torch.full((n, 32, h, w), float("nan"), dtype=torch.float32, device="cuda")
    outb = torch.empty((n, 32, h, w), dtype=torch.bfloat16, device="cuda")
    m.mpv_cnn_conv3x3(torch.from_numpy(x).cuda(), _bf(wt),
                      None if b is None else torch.from_numpy(b).cuda(), 32, relu,
                      out_bf16=outb, out_f32=out)
    wq = cnn_ref.bf16(wt)
    want = cnn_ref.conv3x3(x.astype(np.float64), wq, b)
    scale = cnn_ref.conv3x3(np.abs(x).astype(np.float64), np.abs(wq), None if b is None else np.abs(b))
    if relu:
        want = np.maximum(want, 0)
    got = out.cpu().numpy()
    assert np.all(np.abs(got - want) <= (9 * cin + 3) * EPS * scale)
    assert torch.equal(outb, out.to(torch.bfloat16))


# Cin around the kernel's limit (40) and a warp's 4 channels; Cout 32, 1 and neither; tiles of
# 16 x 16 with remainders; the last two have more tiles than resident blocks
@pytest.mark.parametrize("n,cin,cout,h,w,bias", [
    (1, 1, 32, 1, 1, True), (1, 1, 1, 3, 5, True), (2, 32, 32, 17, 31, False),
    (1, 33, 32, 16, 16, True), (1, 40, 32, 15, 33, True), (1, 40, 1, 15, 33, True),
    (1, 41, 32, 18, 17, True), (1, 41, 1, 18, 17, False), (1, 5, 7, 20, 20, True),
    (3, 3, 32, 190, 170, True), (3, 6, 1, 190, 170, True)])
def test_weight_gradient(m, n, cin, cout, h, w, bias):
    rng = np.random.default_rng(cin * 5 + cout + h)
    x = rng.normal(size=(n, cin, h, w)).astype(np.float32)
    g = rng.normal(size=(n, cout, h, w)).astype(np.float32)
    dw0 = rng.normal(size=(cout, cin, 3, 3)).astype(np.float32)
    db0 = rng.normal(size=cout).astype(np.float32)
    dw, db = torch.from_numpy(dw0).cuda(), torch.from_numpy(db0).cuda()
    m.mpv_cnn_conv3x3_wgrad(_bf(x), torch.from_numpy(g).cuda(), dw, db if bias else None)
    xq, zero = cnn_ref.bf16(x), np.zeros((cout, cin, 3, 3))
    _, want_w, want_b = cnn_ref.conv3x3_backward(xq, zero, g.astype(np.float64))
    _, scale_w, scale_b = cnn_ref.conv3x3_backward(np.abs(xq), zero, np.abs(g).astype(np.float64))
    tol = (n * h * w + 2) * EPS
    assert np.all(np.abs(dw.cpu().numpy() - dw0 - want_w) <= tol * (scale_w + np.abs(dw0)))
    if bias:
        assert np.all(np.abs(db.cpu().numpy() - db0 - want_b) <= tol * (scale_b + np.abs(db0)))
    else:
        assert np.array_equal(db.cpu().numpy(), db0)


@pytest.mark.parametrize("count,offset", [(1, 0), (3, 0), (4, 0), (1024, 0), (1028, 0), (1027, 0),
                                          (1024, 1), (1024, 2), (4096, 4)])
def test_relu_backward(m, count, offset):
    rng = np.random.default_rng(count)
    g = torch.from_numpy(rng.normal(size=count + 8).astype(np.float32)).cuda()
    a = _bf(rng.normal(size=count + 8))
    a[::7] = 0
    a[3::11] = -0.0
    a[5::13] = float("nan")
    a[6::17] = float("inf")
    out = torch.full((count + 8,), 9.0, device="cuda")
    m.mpv_cnn_relu_backward(g[offset:offset + count], a[offset:offset + count],
                            out[offset:offset + count])
    want = torch.full_like(out, 9.0)
    want[offset:offset + count] = torch.where(a > 0, g, torch.zeros_like(g))[offset:offset + count]
    assert torch.equal(out, want)


@pytest.mark.parametrize("count", [1, 255, 257, 152 * 256, 152 * 256 + 1, 300001])
def test_huber(m, count):
    rng = np.random.default_rng(count)
    p = rng.normal(size=count).astype(np.float32)
    t = rng.normal(size=count).astype(np.float32)
    pd, td = torch.from_numpy(p).cuda(), torch.from_numpy(t).cuda()
    grad, again = torch.empty(count, device="cuda"), torch.empty(count, device="cuda")
    loss = torch.full((1,), 0.5, device="cuda")
    m.mpv_cnn_huber(pd, td, 0.75, grad, loss)
    m.mpv_cnn_huber(pd, td, 0.75, again, None)
    want, gref = cnn_ref.huber(p.astype(np.float64), t.astype(np.float64), 0.75)
    # one rounding of each term (the difference, the square, the quotient: 8 at most) and one
    # per block's addition
    assert abs(loss.item() - 0.5 - want) <= (8 + 152) * EPS * (want + 0.5)
    assert np.all(np.abs(grad.cpu().numpy() - gref) <= 4 * EPS * (np.abs(gref) + 2.0 / count))
    assert torch.equal(grad, again)
