"""MF_NORM_MAX streams of different depth types in one process: their first pass is one kernel, so no
stream's launch may change what another's is allowed.  Each stream renders again after the other types
have, and must return the same bits; every non-empty map peaks at exactly 1."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a fresh process: the launch limits are set on a kernel's first use
CHILD = """
import sys
import numpy as np, torch
sys.path.insert(0, {root!r})
import paper_2601_07154_gb300 as mf
from synth.walker import WalkerSpec, walk
window, width, height, n = {window}, {width}, 96, 50
poses = walk(WalkerSpec(n_frames=n, seed=2, turns=True, accel=1.5)).poses_w2c
K = np.array([0.8 * width, 0.8 * width, (width - 1) / 2, (height - 1) / 2])
gen = torch.Generator(device="cuda").manual_seed(1)
depth = torch.rand((n, height, width), device="cuda", generator=gen) * 4 + 0.25
types = [torch.bfloat16, torch.float32, torch.float16]
s = {{t: mf.MotionFocusStream(width, height, window=window, smooth_len=7, mode="heading", depth_dtype=t,
                             map_dtype=torch.bfloat16, normalize="max") for t in types}}
first = {{}}
for t in types + types:
    s[t].reset()
    s[t].push(poses, depth.to(t), K)
    M, G, info, _ = s[t].get_maps()
    full = torch.from_numpy(info["n_valid"] > 0).cuda()
    assert int(full.sum()) > 20 and bool((M.float().amax((1, 2))[full] == 1).all())
    if t in first:
        assert torch.equal(M, first[t][0]) and torch.equal(G, first[t][1])
    first[t] = (M, G)
print("ok")
"""


@pytest.mark.parametrize("window", [8, 16, 32])
@pytest.mark.parametrize("width", [1024, 1023, 1022])
def test_depth_types_take_turns(window, width):
    code = CHILD.format(root=ROOT, window=window, width=width)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
