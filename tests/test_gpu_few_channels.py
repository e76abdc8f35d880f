"""Training kernels at the few input channels where another kernel takes over: whole numbers small
enough that every FP32 sum is exact, compared by equality."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    from paper_2001_09678_gb300 import build, mpv
    build.build()
    mpv.load()
    return mpv


def _whole(rng, *shape):
    return torch.from_numpy(rng.integers(-3, 4, shape).astype(np.float32)).cuda()


# the limit of the thread-per-pixel kernel (2 channels) and the next two
@pytest.mark.parametrize("cin", [1, 2, 3, 4])
@pytest.mark.parametrize("n,h,w,bias,relu", [(1, 1, 1, True, False), (2, 17, 33, False, False),
                                             (3, 16, 20, True, True)])
def test_convolution_of_few_fp32_channels(m, cin, n, h, w, bias, relu):
    rng = np.random.default_rng(cin * 7 + w)
    x, wt, b = _whole(rng, n, cin, h, w), _whole(rng, 32, cin, 3, 3), _whole(rng, 32)
    out = torch.full((n, 32, h, w), float("nan"), device="cuda")
    outb = torch.empty((n, 32, h, w), dtype=torch.bfloat16, device="cuda")
    m.mpv_cnn_conv3x3(x, wt.to(torch.bfloat16), b if bias else None, 32, relu, out_bf16=outb,
                      out_f32=out)
    want = torch.nn.functional.conv2d(x.double(), wt.double(), b.double() if bias else None,
                                      padding=1)
    if relu:
        want = want.clamp(min=0)
    assert torch.equal(out.double(), want)
    assert torch.equal(outb, out.to(torch.bfloat16))


# both sides of each line of wgrad_tiled's rule on a GPU of 152 SMs: tiles of 16 x 16 around 60, 91
# and 456, and channel counts of less than one warp
@pytest.mark.parametrize("cin,cout,tiles", [
    (1, 32, 60), (1, 32, 61), (2, 32, 91), (2, 32, 92), (2, 32, 456), (2, 32, 457), (3, 32, 92),
    (1, 1, 456), (1, 1, 457), (2, 1, 457), (3, 1, 5), (4, 1, 500)])
def test_weight_gradient_of_few_channels(m, cin, cout, tiles):
    rng = np.random.default_rng(cin * 3 + cout + tiles)
    n, h, w = 1, 9, 16 * tiles - 5
    x, g = _whole(rng, n, cin, h, w), _whole(rng, n, cout, h, w)
    dw0, db0 = _whole(rng, cout, cin, 3, 3), _whole(rng, cout)
    dw, db = dw0.clone(), db0.clone()
    m.mpv_cnn_conv3x3_wgrad(x.to(torch.bfloat16), g, dw, db)
    pad = torch.nn.functional.pad(x.double(), (1, 1, 1, 1))
    for ky in range(3):
        for kx in range(3):
            tap = torch.einsum("nohw,nihw->oi", g.double(), pad[:, :, ky:ky + h, kx:kx + w])
            assert torch.equal(dw[:, :, ky, kx].double(), dw0[:, :, ky, kx].double() + tap), (ky, kx)
    assert torch.equal(db.double(), db0.double() + g.double().sum((0, 2, 3)))
