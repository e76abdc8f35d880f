"""The road profile at the edges of its kernel: window lengths of every kind (eta - 1 rows around
multiples of the four rows a thread owns), row counts around whole threads and warps, tall
maps with few staged disparities, sums that need 64-bit keys, and columns' histograms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import ref  # noqa: E402


@pytest.fixture(scope="module")
def mpv():
    from paper_2001_09678_gb300 import build, mpv as m
    build.build()
    m.load()
    return m


# (W, H, D, eta): eta 2 .. 9 (windows of 1 to 8 rows), 10, 17, 256; heights around 4 and 32; D
# around the staged chunks; rows around 3072 (the last with copying
# threads of their own) and 4096; W D above 2^20 (64-bit keys)
CASES = [(40, 61, 20, e) for e in (2, 3, 4, 5, 6, 7, 8, 9, 10, 17, 256)] + [
    (33, 8, 3, 4), (50, 31, 8, 5), (50, 32, 9, 5), (50, 33, 7, 6), (50, 129, 17, 9), (64, 4, 1, 2),
    (1, 40, 5, 8), (90, 4096, 40, 8), (60, 3072, 21, 8), (60, 3073, 21, 8), (70, 1537, 65, 7),
    (9000, 300, 128, 6), (2500, 700, 500, 5)]


@pytest.mark.parametrize("W,H,D,eta", CASES)
def test_road_profile_bit_exact(mpv, W, H, D, eta):
    rng = np.random.default_rng(W * 7 + H + eta)
    # a band of likely rows per disparity, ties among equal counts, rejected pixels
    y = np.arange(H)[:, None]
    U = (y * D // max(H, 1) + rng.integers(-2, 3, (H, W))).clip(0, D - 1).astype(np.uint16)
    U[rng.random((H, W)) < 0.2] = 0xFFFF
    d = torch.from_numpy(U.view(np.int16)).cuda()
    vd = torch.empty((H, D), dtype=torch.int32, device="cuda")
    ud = torch.empty((W, D), dtype=torch.int32, device="cuda")
    prof = torch.empty(D, dtype=torch.int32, device="cuda")
    en = torch.empty(1, dtype=torch.int64, device="cuda")
    ctx = mpv.mpv_create(0)
    try:
        mpv.mpv_road_detect(ctx, d, D, eta, vd, prof, en, udisp=ud)
        torch.cuda.synchronize()
    finally:
        mpv.mpv_destroy(ctx)
    want_vd = ref.vdisparity(U, D)
    assert np.array_equal(vd.cpu().numpy().view(np.uint32), want_vd)
    assert np.array_equal(ud.cpu().numpy().view(np.uint32), ref.udisparity(U, D))
    want_en, want_prof = ref.road_profile(want_vd, eta)
    assert int(en.item()) == want_en
    assert np.array_equal(prof.cpu().numpy(), want_prof)
