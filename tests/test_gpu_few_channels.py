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
