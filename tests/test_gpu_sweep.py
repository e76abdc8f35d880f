"""The gradient-weighted passes' byte sums, against the oracle (integers: equality of energies and
maps): paths around chunks of 8 steps and groups of 8, label strides of 16 and 32, whole and
padded, windows that move by more than their width, slopes of 0, steep tables, the largest
truncation whose sums fit a byte and the next one (16-bit sums)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ref  # noqa: E402
from paper_2001_09678_gb300 import synth  # noqa: E402


@pytest.fixture(scope="module")
def mpv():
    from paper_2001_09678_gb300 import build, mpv as m
    build.build()
    m.load()
    return m


def _table(p1, sigma):
    g = np.arange(256, dtype=np.float64)
    return np.floor(p1 * np.exp(-g / sigma) + 0.5).astype(np.int32)


# (width, height, D, scales, window, paths, p1, T, sigma, lr); sigma 0: slopes alternate between
# 0 and p1
CASES = [(7, 9, 4, 1, 0, 8, 10, 30, 16, 1), (24, 8, 16, 1, 0, 8, 10, 30, 16, 1),
         (17, 7, 16, 1, 0, 4, 10, 30, 4, 1), (40, 33, 32, 1, 0, 8, 10, 30, 16, 1),
         (33, 15, 27, 1, 0, 8, 10, 30, 0, 0), (31, 40, 20, 1, 0, 8, 31, 31, 8, 1),
         (66, 35, 64, 2, 16, 8, 10, 30, 16, 1), (71, 37, 64, 2, 11, 4, 10, 30, 16, 1),
         (65, 34, 64, 2, 32, 8, 10, 30, 4, 1), (67, 49, 64, 2, 25, 8, 10, 30, 0, 1),
         (130, 70, 128, 3, 32, 8, 10, 30, 16, 1), (131, 41, 128, 2, 16, 8, 1, 30, 30, 1),
         (131, 41, 128, 2, 16, 8, 3, 31, 3, 1), (140, 40, 128, 2, 32, 8, 10, 32, 16, 1),
         (140, 40, 128, 2, 30, 4, 20, 63, 12, 1), (140, 40, 128, 2, 32, 4, 20, 64, 12, 1),
         (101, 33, 48, 1, 0, 8, 10, 30, 16, 1)]


@pytest.mark.parametrize("W,H,D,scales,window,paths,p1,T,sigma,lr", CASES)
def test_gradient_passes_bit_exact(mpv, W, H, D, scales, window, paths, p1, T, sigma, lr):
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=9)
    R = R.copy()
    R[:, : W // 5] = 255 - L[:, : W // 5]          # windows that jump
    lut = _table(p1, sigma) if sigma else (np.arange(256) % 2 * p1).astype(np.int32)
    kw = dict(max_disparity=D, num_scales=scales, num_paths=paths, p1=p1, trunc=T, lr_check=lr,
              window=window)
    p = ref.params(ssim_window=5, block=(0, 0, 0, 0), lr_tol=1, grad_lut=lut, **kw)
    want = ref.match(L, R, p)
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(**kw))
        mpv.mpv_set_gradient_penalty(ctx, lut)
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        d = torch.full(L.shape, -2, dtype=torch.int16, device="cuda")
        mpv.mpv_match(ctx, l, r, d)
        mpv.mpv_sync(ctx)
        assert np.array_equal(d.cpu().numpy().view(np.uint16), want)
        for level in range(scales):
            _, Cv, S, _ = ref.view_stage(L, R, p, level)
            gc = torch.zeros(Cv.shape, dtype=torch.int16, device="cuda")
            gs = torch.zeros(Cv.shape, dtype=torch.int32, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, 0, level, None, gc, gs, None)
            assert np.array_equal(gc.cpu().numpy().view(np.uint16).astype(np.int64), Cv)
            assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
