"""The layered merge's passes at the edges of their staging, against the oracle (integers:
equality of energies and maps): paths around chunks of 8 steps and groups of 4, label strides of
16 and 32, whole and padded, with and without windows, 2 and 4 layers, truncations up to the
packed bound."""
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


# (width, height, D, scales, window, paths, p1, T, lr)
CASES = [(7, 9, 4, 1, 0, 8, 10, 30, 1), (24, 8, 16, 1, 0, 8, 10, 30, 1),
         (17, 7, 16, 1, 0, 4, 10, 30, 1), (40, 33, 32, 1, 0, 8, 10, 30, 1),
         (33, 15, 27, 1, 0, 8, 10, 30, 0), (31, 40, 20, 1, 0, 8, 10, 20, 1),
         (66, 35, 64, 2, 16, 8, 10, 30, 1),
         (71, 37, 64, 2, 11, 4, 10, 30, 1), (65, 34, 64, 2, 32, 8, 10, 30, 1),
         (67, 49, 64, 2, 25, 8, 10, 30, 1), (130, 70, 128, 3, 32, 8, 10, 30, 1),
         (64, 32, 32, 2, 16, 8, 800, 1612, 1), (64, 33, 60, 2, 32, 8, 700, 1612, 1)]


@pytest.mark.parametrize("W,H,D,scales,window,paths,p1,T,lr", CASES)
def test_layers_bit_exact(mpv, W, H, D, scales, window, paths, p1, T, lr):
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=9)
    R = R.copy()
    R[:, : W // 5] = 255 - L[:, : W // 5]          # windows that move
    kw = dict(max_disparity=D, num_scales=scales, num_paths=paths, p1=p1, trunc=T, lr_check=lr,
              window=window, merge_mode=1)
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
        for level in range(scales):
            _, Cv, S, _ = ref.view_stage(L, R, p, level)
            gs = torch.zeros(Cv.shape, dtype=torch.int32, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, 0, level, None, None, gs, None)
            assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
