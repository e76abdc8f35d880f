"""The Huber loss keeps what its FP32 additions round off: a block's sum is rounded once.

One block (at most 256 elements) adds one FP32 number to a loss of 0, so the result is within one
rounding of the FP32 terms' exact mean, 2^-24, and the 2^-40 that pairs and the reciprocal leave.
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


@pytest.mark.parametrize("count", [1, 2, 31, 33, 64, 100, 255, 256])
def test_loss_rounds_once_per_block(m, count):
    for seed in range(8):
        rng = np.random.default_rng(seed * 300 + count)
        # targets 0 and |p| above delta: the terms p - delta / 2 are exact in FP32
        p = (rng.integers(2 ** 12, 2 ** 21, count) / 2.0 ** 10).astype(np.float32)
        grad, loss = torch.empty(count, device="cuda"), torch.zeros(1, device="cuda")
        m.mpv_cnn_huber(torch.from_numpy(p).cuda(), torch.zeros(count, device="cuda"), 0.5, grad, loss)
        want = np.mean(p.astype(np.float64) - 0.25)
        assert abs(loss.item() - want) <= (2.0 ** -24 + 2.0 ** -40) * want


def test_loss_keeps_non_finite_values(m):
    for bad in (float("inf"), float("nan")):
        p = torch.ones(700, device="cuda")
        p[313] = bad
        grad, loss = torch.empty(700, device="cuda"), torch.zeros(1, device="cuda")
        m.mpv_cnn_huber(p, torch.zeros(700, device="cuda"), 0.5, grad, loss)
        got = loss.item()
        assert got == float("inf") if bad == float("inf") else got != got
