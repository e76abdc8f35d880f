"""Weight gradients in whole numbers, compared by equality: every product is counted once.

Inputs and gradients are whole numbers of at most 3 and every sum of products stays below 2^24, so
that FP32 sums in any order are exact: a tile that is left out, taken twice or misplaced shows,
also where a block walks over many tiles (304 resident blocks for 32 channels, 456 for one).
"""
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


# (n, cin, cout, h, w), tiles of 16 x 16: 1, 6, 9 (edges of maps and warps); 396 and 714 (a second
# and a third tile per block) with the fewest and the most input channels; 528 and 2,160 for one
# channel; the general kernel
@pytest.mark.parametrize("n,cin,cout,h,w", [
    (1, 1, 32, 3, 3), (3, 33, 32, 17, 16), (1, 40, 32, 33, 47), (3, 3, 32, 190, 170),
    (2, 40, 32, 270, 330), (2, 34, 32, 270, 330), (1, 1, 1, 3, 3), (1, 40, 1, 33, 47),
    (4, 6, 1, 190, 170), (9, 32, 1, 180, 320), (2, 41, 32, 40, 33), (2, 5, 7, 40, 33)])
def test_weight_gradient_counts_every_product_once(m, n, cin, cout, h, w):
    rng = np.random.default_rng(cin * 11 + cout + w)
    x = torch.from_numpy(rng.integers(-3, 4, (n, cin, h, w)).astype(np.float32)).cuda()
    g = torch.from_numpy(rng.integers(-3, 4, (n, cout, h, w)).astype(np.float32)).cuda()
    dw0 = torch.from_numpy(rng.integers(-9, 10, (cout, cin, 3, 3)).astype(np.float32)).cuda()
    db0 = torch.from_numpy(rng.integers(-9, 10, cout).astype(np.float32)).cuda()
    assert 9 * n * h * w + 9 < 2 ** 24
    dw, db = dw0.clone(), db0.clone()
    m.mpv_cnn_conv3x3_wgrad(x.to(torch.bfloat16), g, dw, db)
    pad = torch.nn.functional.pad(x.double(), (1, 1, 1, 1))
    for ky in range(3):
        for kx in range(3):
            tap = torch.einsum("nohw,nihw->oi", g.double(), pad[:, :, ky:ky + h, kx:kx + w])
            assert torch.equal(dw[:, :, ky, kx].double(), dw0[:, :, ky, kx].double() + tap), (ky, kx)
    assert torch.equal(db.double(), db0.double() + g.double().sum((0, 2, 3)))
