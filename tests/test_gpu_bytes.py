"""Byte sums of the packed passes: every label stride, with and without windows, at the limits
of their rule, against the oracle (integers: equality of windows, energies and maps)."""
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


# (width, height, D, scales, window, paths, p1, T, lr): strides 16, 32, 48 and 64, whole and
# padded; paths fewer than a warp's and not a multiple of them; the largest truncation whose
# sums fit a byte (255 / paths) and the next one, which keeps 16-bit sums; radius 2 and 3
CASES = [(9, 7, 4, 1, 0, 8, 10, 30, 1), (33, 34, 16, 1, 0, 8, 10, 30, 1),
         (70, 41, 64, 2, 16, 8, 10, 30, 1), (71, 37, 64, 2, 11, 4, 10, 30, 1),
         (66, 35, 32, 1, 0, 8, 10, 30, 0), (140, 67, 128, 2, 32, 8, 10, 30, 1),
         (137, 45, 128, 2, 17, 8, 10, 30, 1), (138, 30, 128, 2, 25, 8, 11, 31, 1),
         (138, 30, 128, 2, 32, 8, 11, 32, 1), (138, 30, 128, 2, 32, 4, 21, 63, 1),
         (138, 30, 128, 2, 32, 4, 22, 64, 1), (138, 30, 128, 2, 32, 8, 7, 22, 1),
         (101, 33, 48, 1, 0, 8, 10, 30, 1), (203, 41, 96, 2, 48, 8, 10, 30, 1),
         (202, 40, 96, 2, 39, 8, 10, 30, 1), (99, 31, 64, 1, 0, 8, 10, 30, 1),
         (160, 33, 150, 2, 64, 8, 10, 30, 1), (161, 33, 150, 2, 57, 8, 3, 9, 1),
         (640, 360, 128, 3, 0, 8, 10, 30, 1), (700, 400, 150, 2, 30, 8, 10, 30, 0)]


@pytest.mark.parametrize("W,H,D,scales,window,paths,p1,T,lr", CASES)
def test_byte_sums_bit_exact(mpv, W, H, D, scales, window, paths, p1, T, lr):
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=15)
    R = R.copy()
    R[:, : W // 5] = 255 - L[:, : W // 5]
    kw = dict(max_disparity=D, num_scales=scales, num_paths=paths, p1=p1, trunc=T, lr_check=lr,
              window=window)
    p = ref.params(ssim_window=5, block=(0, 0, 0, 0), lr_tol=1, **kw)
    want = ref.match(L, R, p)
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(**kw))
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        d = torch.full(L.shape, -2, dtype=torch.int16, device="cuda")
        mpv.mpv_match(ctx, l, r, d)
        mpv.mpv_sync(ctx)
        assert np.array_equal(d.cpu().numpy().view(np.uint16), want)
        if W * H > 20000:
            return
        for level in range(scales):
            _, Cv, S, _ = ref.view_stage(L, R, p, level)
            gc = torch.zeros(Cv.shape, dtype=torch.int16, device="cuda")
            gs = torch.zeros(Cv.shape, dtype=torch.int32, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, 0, level, None, gc, gs, None)
            assert np.array_equal(gc.cpu().numpy().view(np.uint16).astype(np.int64), Cv)
            assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
