"""The depth scale of a batch is the exact lower median of its overlap's ratios, at counts around the
selection kernels' CTA and unroll edges, with invalid depths among them, and without any valid pair."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _median(prev, cur):
    ok = (prev > 0) & (cur > 0) & np.isfinite(prev) & np.isfinite(cur)
    if not ok.any():
        return 1.0
    r = np.sort((prev[ok] / cur[ok]).astype(np.float32))
    return float(r[(len(r) - 1) // 2])


@pytest.mark.parametrize("width,height,overlap", [(1, 1, 1), (31, 33, 1), (32, 32, 1), (41, 25, 1), (640, 243, 1),
                                                  (641, 243, 1), (512, 304, 4), (321, 241, 9)])
@pytest.mark.parametrize("storage", [torch.float32, torch.float16])
@pytest.mark.parametrize("spread", [0.0, 0.02, 3.0])
def test_scale_is_the_lower_median(width, height, overlap, storage, spread):
    import paper_2601_07154_gb300 as mf
    rng = np.random.default_rng([width, height, overlap])
    n = overlap + 3
    poses = np.tile(np.eye(3, 4), (n, 1, 1))
    poses[:, 2, 3] = -0.05 * np.arange(n)
    K = np.array([0.8 * width, 0.8 * width, width / 2, height / 2])
    s = mf.MotionFocusStream(width, height, window=2, smooth_len=3, pose_frame="batch_local", overlap=overlap,
                             depth_dtype=storage, map_dtype=torch.float32, depth_align=True)
    for again in range(2):                  # a second clip after a reset: the counters start at 0 again
        planes, want = [], [1.0]
        for b in range(4):
            d = rng.uniform(0.5, 2.0, (n, height, width)) * np.exp(spread * rng.normal(size=(n, height, width)))
            bad = rng.uniform(size=d.shape) < 0.1
            d[bad] = rng.choice([0.0, -1.0, np.nan, np.inf], size=int(bad.sum()))
            if b == 2:
                d[:overlap] = 0.0           # no valid pair: the scale stays
            planes.append(torch.from_numpy(d).to(storage).cuda())
        for b in range(1, 4):
            prev = planes[b - 1][n - overlap:].float().cpu().numpy()
            cur = planes[b][:overlap].float().cpu().numpy()
            want.append(want[-1] * _median(prev, cur))
        for b, d in enumerate(planes):
            s.push(poses, d, K)
            _, _, info, _ = s.get_maps()
            assert np.all(info["depth_scale"] == np.float32(want[b])), (again, b)
        s.reset()
    s.close()
