"""Window starts from 2 x 2 coarse blocks and from single coarse pixels at every remainder of the
image's sides modulo 4 (whole and partial blocks, vector and single stores), against the oracle
(integers: equality)."""
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


@pytest.mark.parametrize("block", [(0, 0, 0, 0), (2, 2, 0, 0), (1, 1, 0, 0), (3, 1, 0, 0)])
@pytest.mark.parametrize("W,H", [(64, 32), (65, 33), (66, 34), (67, 35), (68, 29), (36, 9), (520, 20)])
def test_window_starts_bit_exact(mpv, W, H, block):
    kw = dict(max_disparity=32, num_scales=3, num_paths=8, window=8)
    L, R, _ = synth.slanted_pair(W, H, seed=W, d_max=28, n_planes=12)
    p = ref.params(ssim_window=3, block=block, lr_check=1, lr_tol=1, **kw)
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(ssim_window=3, block=block, **kw))
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        for level in (1, 2):
            want = ref.view_stage(L, R, p, level)[0]
            lo = torch.full(want.shape, -1, dtype=torch.int16, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, 0, level, lo, None, None, None)
            assert np.array_equal(lo.cpu().numpy().view(np.uint16).astype(np.int64), want)
    finally:
        mpv.mpv_destroy(ctx)
