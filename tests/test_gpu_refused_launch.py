"""A launch that the runtime refuses is reported by the call and leaves no error behind for the caller's
own next check.  The refusal is made on the host: the stream's capture has been invalidated."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes, sys
import numpy as np, torch
sys.path.insert(0, {root!r})
import paper_2601_07154_gb300 as mf
rt = ctypes.CDLL("libcudart.so.13")
st = torch.cuda.Stream()
kw = dict(window=2, smooth_len=3, cuda_stream=st)
pushed = mf.MotionFocusStream(64, 48, **kw)
fresh = mf.MotionFocusStream(64, 48, **kw)
poses, K = np.tile(np.eye(3, 4), (4, 1, 1)), np.array([50.0, 50.0, 32.0, 24.0])
pushed.push(poses, None, K)
M, G = (torch.zeros((4, 48, 64), device="cuda") for _ in range(2))
info = torch.zeros(4 * 64, dtype=torch.uint8, device="cuda")
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.stream(st):
    g.capture_begin()
    try:
        torch.cuda.synchronize()                 # not allowed in a capture: it is invalid from here on
    except Exception:
        pass
    rt.cudaGetLastError()
    for call in (lambda: fresh.push(poses, None, K),
                 lambda: mf.mf_get_maps(pushed.handle, 4, M, G, info, None)):
        try:
            call()
            print("not refused")
        except mf.MFError as e:
            print("refused" if e.status == mf.MF_ERR_CUDA else e, rt.cudaPeekAtLastError())
        rt.cudaGetLastError()
"""


def test_no_error_is_left_behind():
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.stdout.splitlines()[:2] == ["refused 0", "refused 0"], r.stdout + r.stderr[-2000:]
