"""Byte sums where a direction's paths don't fill its last warp: the lanes that are left over repeat
another path and add nothing.  Widths of every remainder of 8 (and fewer than 8 columns), rows long
enough for the straight-line steps (at least 20 of them), every label stride, with and without
windows, 8 and 4 paths; costs, summed energies and maps equal the oracle's.
"""
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


# (width, height, D, scales, window, paths, lr): strides 16 and 32; 48 and 64 (8 lanes, 4 paths)
CASES = [(5, 60, 5, 1, 0, 8, 1)] + \
        [(w, 47, w, 1, 0, 8 if w % 2 else 4, w % 3 > 0) for w in range(17, 25)] + \
        [(w, 44, 30, 2, 14, 8, 1) for w in range(41, 49, 2)] + \
        [(w, 41, 60, 2, 27, 8, 0) for w in range(74, 81, 2)] + \
        [(49, 45, 40, 1, 0, 8, 1), (94, 42, 90, 2, 45, 4, 1), (77, 44, 64, 1, 0, 8, 1),
         (130, 43, 128, 2, 60, 8, 0),
         # narrow, tall levels with windows of 16 labels, and the first ones outside that rule
         (20, 90, 14, 2, 7, 8, 1), (29, 58, 20, 2, 16, 4, 1), (29, 57, 20, 2, 16, 8, 0),
         (256, 512, 14, 2, 7, 8, 1), (257, 514, 14, 2, 7, 8, 1)]


@pytest.mark.parametrize("W,H,D,scales,window,paths,lr", CASES)
def test_spare_lanes_add_nothing(mpv, W, H, D, scales, window, paths, lr):
    L, R, _ = synth.slanted_pair(W, H, seed=W + H, d_max=max(1.0, 0.9 * (D - 1)), n_planes=9)
    kw = dict(max_disparity=D, num_scales=scales, num_paths=paths, p1=10, trunc=30,
              lr_check=int(lr), window=window)
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
            gs = torch.zeros(S.shape, dtype=torch.int32, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, 0, level, None, None, gs, None)
            assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
