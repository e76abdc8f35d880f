"""The cost volume of every label stride, patch side and row-segment shape against the oracle.

Costs are integers: every comparison is equality.  The images mix textured parts with ones
whose quotient sits on an integer (equal, inverted and flat patches), so that the fp32
estimate is not enough, and their windows move along the rows.
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


def _images(W, H, d):
    L, R, _ = synth.slanted_pair(W, H, seed=W + d, d_max=0.9 * (d - 1), n_planes=12)
    L, R = L.copy(), R.copy()
    t = W // 4
    R[:, :t] = L[:, :t]                        # equal patches at u = 0: cost 0
    R[: H // 2, t:2 * t] = 255 - L[: H // 2, t:2 * t]   # inverted
    L[:, 3 * t:] = 0                           # flat, saturated against flat and textured
    R[H // 2:, 3 * t:] = 255
    return L, R


# (width, height, D, scales, window, N): label strides 16, 32, 48 and 80 at the finest level,
# rows of one, two and five segments with whole and ragged ends, rows shorter than a chunk
CASES = [(5, 5, 4, 1, 0, 5), (3, 4, 2, 1, 0, 3), (17, 9, 12, 1, 0, 5), (319, 6, 20, 1, 0, 5),
         (321, 6, 33, 1, 0, 5), (326, 12, 64, 2, 16, 5), (323, 12, 64, 2, 11, 3),
         (641, 12, 128, 2, 32, 5), (645, 14, 128, 2, 25, 3), (330, 12, 96, 2, 48, 5),
         (329, 12, 96, 2, 41, 5), (340, 12, 160, 2, 77, 5), (1284, 12, 64, 2, 17, 5)]


@pytest.mark.parametrize("W,H,D,scales,window,N", CASES)
@pytest.mark.parametrize("view", [0, 1])
def test_cost_volume_bit_exact(mpv, W, H, D, scales, window, N, view):
    L, R = _images(W, H, D)
    p = ref.params(max_disparity=D, num_scales=scales, num_paths=4, p1=10, trunc=30, ssim_window=N,
                   window=window, block=(0, 0, 0, 0), lr_check=1, lr_tol=1)
    I0, I1 = (L, R) if view == 0 else (np.ascontiguousarray(R[:, ::-1]),
                                       np.ascontiguousarray(L[:, ::-1]))
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(max_disparity=D, num_scales=scales,
                                                       num_paths=4, ssim_window=N, window=window))
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        for level in range(scales):
            lo, Cv, _, _ = ref.view_stage(I0, I1, p, level)
            glo = torch.zeros(lo.shape, dtype=torch.int16, device="cuda")
            gc = torch.full(Cv.shape, -1, dtype=torch.int16, device="cuda")
            mpv.mpv_debug_stage(ctx, l, r, view, level, glo, gc, None, None)
            assert np.array_equal(glo.cpu().numpy().astype(np.int64), lo.astype(np.int64))
            bad = gc.cpu().numpy().view(np.uint16).astype(np.int64) != Cv
            assert not bad.any(), f"level {level}: {bad.sum()} costs differ"
    finally:
        mpv.mpv_destroy(ctx)
