"""The passes on staged data in the bounds-checked build (MPV_DEBUG_BOUNDS): the copies, window
starts, stores and reductions of the rows (agg_rows), the layers (agg_layer) and the
gradient-weighted passes (agg_sweep) are checked at rows of one chunk of 8 pixels and around
whole chunks, numbers of rows around a warp's 4 paths, strides of 16 and 32 labels with padding
labels, windows and single views; the maps must equal the oracle.  Runs in a child process that
loads libmpv_debug.so.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import numpy as np, torch
from oracle import ref
from paper_2001_09678_gb300 import mpv, synth
mpv.load()
lut = np.floor(10 * np.exp(-np.arange(256, dtype=np.float64) / 8.0) + 0.5).astype(np.int32)
sizes = [  # (W, H, D, scales, window, paths, lr)
    (7, 5, 6, 1, 0, 8, 1), (8, 5, 8, 1, 0, 8, 1), (17, 6, 17, 1, 0, 8, 1), (16, 9, 16, 2, 8, 8, 1),
    (33, 11, 32, 2, 20, 8, 1), (41, 15, 40, 2, 32, 8, 0), (39, 23, 36, 3, 12, 4, 1),
    (64, 33, 60, 3, 16, 8, 1), (65, 8, 64, 2, 31, 8, 1),
]
n = 0
for W, H, D, S, win, P, lr in sizes:
    L, R, _ = synth.slanted_pair(W, H, seed=W * 100 + H + D, d_max=max(1.0, D - 2.0))
    for merge, grad in ((0, False), (1, False), (0, True)):
        kw = dict(max_disparity=D, num_scales=S, num_paths=P, p1=10, trunc=30, merge_mode=merge,
                  window=win, lr_check=lr)
        t = lut if grad else None
        want = ref.match(L, R, ref.params(block=(0, 0, 0, 0), lr_tol=1, ssim_window=5 if H // 2 ** (S - 1) >= 5 else 3,
                                          grad_lut=t, **kw))
        ctx = mpv.mpv_create(0)
        mpv.mpv_set_params(ctx, mpv.mpv_default_params(
            ssim_window=5 if H // 2 ** (S - 1) >= 5 else 3, **kw))
        if grad:
            mpv.mpv_set_gradient_penalty(ctx, t)
        l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
        d = torch.full((H, W), -2, dtype=torch.int16, device="cuda")
        mpv.mpv_match(ctx, l, r, d)
        mpv.mpv_sync(ctx)        # raises MpvError(MPV_ERR_INTERNAL) on a failed check
        got = d.cpu().numpy().view(np.uint16)
        assert np.array_equal(got, want), (W, H, D, S, win, P, lr, merge, grad)
        mpv.mpv_destroy(ctx)
        n += 1
print("bounds-checked staged runs ok:", n)
'''


def test_bounds_checked_build_on_staged_passes():
    from paper_2001_09678_gb300 import build
    lib = build.build(debug=True)
    env = dict(os.environ, MPV_LIBRARY=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "bounds-checked staged runs ok: 27" in r.stdout
