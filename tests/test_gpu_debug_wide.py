"""The wide full-range passes in the bounds-checked build (MPV_DEBUG_BOUNDS): every copy of costs,
load of a step's sums and reduction is checked, on 8 and 4 lanes with odd and even numbers of cost
words per lane, and the maps must equal the oracle.  Runs in a child process that loads
libmpv_debug.so.
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
cases = [  # (W, H, D, paths, lr): 8 lanes of 3 to 8 words, then 4 lanes of 5 to 8
    (70, 13, 66, 8, 1), (99, 6, 96, 4, 0), (131, 9, 97, 8, 1), (171, 11, 161, 8, 1),
    (171, 35, 160, 8, 0), (230, 7, 200, 4, 1), (260, 10, 256, 8, 1),
    (1300, 9, 72, 8, 1), (1300, 9, 80, 8, 1), (1300, 7, 91, 8, 1), (1300, 9, 112, 8, 1),
    (1300, 9, 100, 8, 1), (2700, 5, 113, 8, 0), (4000, 6, 99, 4, 1),
]
for W, H, D, P, lr in cases:
    L, R, _ = synth.slanted_pair(W, H, seed=W + D, d_max=0.9 * (D - 1), n_planes=8)
    kw = dict(max_disparity=D, num_scales=1, num_paths=P, p1=10, trunc=30, lr_check=lr)
    want = ref.match(L, R, ref.params(window=0, block=(0, 0, 0, 0), lr_tol=1, ssim_window=5, **kw))
    ctx = mpv.mpv_create(0)
    mpv.mpv_set_params(ctx, mpv.mpv_default_params(**kw))
    l, r = torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda()
    d = torch.full((H, W), -2, dtype=torch.int16, device="cuda")
    mpv.mpv_match(ctx, l, r, d)
    mpv.mpv_sync(ctx)        # raises MpvError(MPV_ERR_INTERNAL) on a failed check
    got = d.cpu().numpy().view(np.uint16)
    assert np.array_equal(got, want), (W, H, D, P, lr, int((got != want).sum()))
    mpv.mpv_destroy(ctx)
print("bounds-checked wide runs ok:", len(cases))
'''


def test_bounds_checked_build_on_wide_levels():
    from paper_2001_09678_gb300 import build
    lib = build.build(debug=True)
    env = dict(os.environ, MPV_LIBRARY=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "bounds-checked wide runs ok: 14" in r.stdout
