"""The wide full-range passes on 4 lanes per path, against the oracle: every number of cost words,
whole and with padding labels, 8 and 4 paths, two views and one.  4 lanes are chosen where a level
has enough warps: long images of few rows keep the oracle quick.  Costs, summed energies and maps
are whole numbers and compared by equality; the lanes that the rule chose are part of each case.
"""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import wide_rules  # noqa: E402
from oracle import ref  # noqa: E402
from paper_2001_09678_gb300 import synth  # noqa: E402


@pytest.fixture(scope="module")
def mpv():
    from paper_2001_09678_gb300 import build, mpv as m
    build.build()
    m.load()
    return m


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    return wide_rules.compile_rules(tmp_path_factory.mktemp("wide"))


# (width, height, D, paths, lr_check, words per lane)
CASES = [(1300, 9, 65, 8, 1, 5), (1300, 9, 80, 8, 1, 5), (1301, 7, 81, 8, 1, 6),
         (1300, 8, 96, 8, 1, 6), (1303, 9, 97, 8, 1, 7), (1300, 9, 112, 8, 1, 7),
         (1300, 17, 113, 8, 1, 8), (1299, 9, 128, 8, 1, 8), (2600, 6, 77, 8, 0, 5),
         (2601, 5, 128, 8, 0, 8), (3700, 5, 90, 4, 1, 6), (3701, 6, 127, 4, 1, 8),
         (7400, 5, 105, 4, 0, 7)]


@pytest.mark.parametrize("W,H,D,paths,lr,words", CASES)
def test_four_lanes_bit_exact(mpv, rules, W, H, D, paths, lr, words):
    p1, T = (10, 30) if paths == 8 else (21, 63)
    assert wide_rules.ask(rules, [f"shape {W} {H} {D} {1 + lr} {paths} {T} 2"]) == [(4, words)]
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=8)
    R = R.copy()
    R[:, : W // 5] = 255 - L[:, : W // 5]          # costs near 255: path minima above 255 - T
    kw = dict(max_disparity=D, num_scales=1, num_paths=paths, p1=p1, trunc=T, lr_check=lr)
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
        lo, Cv, S, _ = ref.view_stage(L, R, p, 0)
        gc = torch.zeros(Cv.shape, dtype=torch.int16, device="cuda")
        gs = torch.zeros(Cv.shape, dtype=torch.int32, device="cuda")
        mpv.mpv_debug_stage(ctx, l, r, 0, 0, None, gc, gs, None)
        assert np.array_equal(gc.cpu().numpy().view(np.uint16).astype(np.int64), Cv)
        assert np.array_equal(gs.cpu().numpy().astype(np.int64), S)
    finally:
        mpv.mpv_destroy(ctx)
