"""The wide full-range passes (byte sums) against the oracle and at the edges of their rule.

Energies are integers: costs, summed energies and maps are compared by equality.  Cases just
outside the rule (label count, truncation, radius) run the general passes on the same pair, and
each must equal the oracle too.
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


# (width, height, D, scales, paths, p1, T, lr_check): 8 lanes with 3 to 8 cost words, whole and
# padded; images narrower and shorter than a warp's paths; the largest penalty whose sums fit a
# byte (255 / paths) and the next one; radius 2 and 3; no penalty; labels 64 and 257 (other
# passes); a frame of enough warps for 4 lanes
CASES = [(65, 5, 65, 1, 8, 10, 30, 1), (70, 33, 66, 1, 8, 10, 30, 1), (99, 6, 96, 1, 8, 10, 30, 0),
         (131, 9, 97, 1, 4, 10, 30, 1), (130, 40, 128, 1, 8, 10, 30, 1),
         (171, 35, 160, 1, 8, 11, 31, 1), (171, 11, 161, 1, 8, 11, 32, 1),
         (230, 7, 200, 1, 4, 21, 63, 1), (230, 7, 200, 1, 4, 22, 64, 1),
         (260, 10, 225, 1, 8, 3, 9, 1), (260, 10, 256, 1, 8, 7, 21, 1),
         (260, 10, 256, 1, 8, 7, 22, 1), (260, 9, 257, 1, 4, 10, 30, 1),
         (131, 17, 128, 1, 8, 0, 30, 1), (131, 17, 128, 1, 8, 40, 30, 1),
         (131, 17, 64, 1, 8, 10, 30, 1), (300, 40, 280, 2, 8, 10, 30, 1),
         (1501, 300, 100, 1, 8, 10, 30, 1)]


@pytest.mark.parametrize("W,H,D,scales,paths,p1,T,lr", CASES)
def test_wide_levels_bit_exact(mpv, W, H, D, scales, paths, p1, T, lr):
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=8)
    R = R.copy()
    R[:, : W // 5] = 255 - L[:, : W // 5]          # costs near 255: path minima above 255 - T
    kw = dict(max_disparity=D, num_scales=scales, num_paths=paths, p1=p1, trunc=T, lr_check=lr)
    p = ref.params(ssim_window=5, window=0, block=(0, 0, 0, 0), lr_tol=1, **kw)
    want = ref.match(L, R, p)
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(**kw))
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        d = torch.full(L.shape, -2, dtype=torch.int16, device="cuda")
        mpv.mpv_match(ctx, l, r, d)
        mpv.mpv_sync(ctx)
        assert np.array_equal(d.cpu().numpy().view(np.uint16), want)
        if W * H * D > 2_000_000:
            return
        lo, Cv, S, _ = ref.view_stage(L, R, p, 0)
        gc = torch.zeros(Cv.shape, dtype=torch.int16, device="cuda")
        gs = torch.zeros(Cv.shape, dtype=torch.int32, device="cuda")
        mpv.mpv_debug_stage(ctx, l, r, 0, 0, None, gc, gs, None)
        assert np.array_equal(gc.cpu().numpy().view(np.uint16).astype(np.int64), Cv)
        assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
