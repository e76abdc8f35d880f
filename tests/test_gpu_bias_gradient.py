"""Bias gradients: one FP32 sum per 16 x 16 tile, in row order, and every tile added by itself.

The sums of a gradient clipped to +-1/n round alike wherever they are cut, so the cut is part of
the result.  Both tests compare by equality: their tile sums and totals are whole numbers (or
whole multiples of 2^-13) that every order of adding the tiles keeps exact.
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


def _bias(m, g, cin, db0):
    x = torch.zeros((g.shape[0], cin) + tuple(g.shape[2:]), dtype=torch.bfloat16, device="cuda")
    dw = torch.zeros((g.shape[1], cin, 3, 3), device="cuda")
    db = torch.from_numpy(db0).cuda()
    m.mpv_cnn_conv3x3_wgrad(x, torch.from_numpy(g).cuda(), dw, db)
    return db.cpu().numpy()


# (n, cin, cout, h, w): the kernels for 32 channels and for one, with fewer tiles than resident
# blocks and with several tiles per block, from one warp of threads to the most; the general kernel
SHAPES = [(1, 1, 1, 1, 1), (2, 1, 32, 17, 31), (2, 34, 32, 16, 33), (2, 32, 1, 15, 17),
          (1, 40, 32, 33, 48), (8, 32, 1, 180, 320), (2, 34, 32, 270, 330), (1, 41, 32, 18, 17),
          (1, 5, 7, 20, 20)]


@pytest.mark.parametrize("n,cin,cout,h,w", SHAPES)
def test_bias_gradient_counts_every_pixel_once(m, n, cin, cout, h, w):
    rng = np.random.default_rng(n * 7 + cin + w)
    g = rng.integers(-3, 4, (n, cout, h, w)).astype(np.float32)
    db0 = rng.integers(-9, 10, cout).astype(np.float32)
    assert np.array_equal(_bias(m, g, cin, db0), db0 + g.sum((0, 2, 3), dtype=np.float64))


@pytest.mark.parametrize("n,cin,cout,h,w", SHAPES)
def test_bias_gradient_rounds_a_tile_at_a_time(m, n, cin, cout, h, w):
    # a tile's first pixel is 1, and the 2^-25 of the others are below half an ulp of any sum that
    # holds it: its sum is 1 (or what its pixels make, where one further pixel is 2^-13)
    g = np.full((n, cout, h, w), 2.0 ** -25, np.float32)
    g[:, :, ::16, ::16] = 1.0
    odd = (np.arange(cout) % 3 == 1)
    g[:, odd, 1::16, 2::16] = 2.0 ** -13
    want = np.full(cout, n * g[0, 0, ::16, ::16].size, np.float64)
    want[odd] += n * g[0, 0, 1::16, 2::16].size * 2.0 ** -13
    assert np.array_equal(_bias(m, g, cin, np.zeros(cout, np.float32)), want)
