"""Odd widths: the unit kernel by row phases against the tiled kernel, which drops no point and which
planes that start off the kernel's alignment take.

Both sum the same FP32 terms in the same order, but for terms below 2^-40 of the frame's largest: per
pixel at most 32 of them (2^-35 of the frame's maximum) and at most 32 roundings of the sum that they
can turn (2^-23 of it each).  Then come the roundings to the storage type, three in all where the tiled
kernel's maps are normalised in place (half of 2^-8 in BF16, of 2^-10 in F16, each)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROUND = {torch.float32: 0.0, torch.bfloat16: 3 * 2.0 ** -9, torch.float16: 3 * 2.0 ** -11}
TINY = {torch.float32: 0.0, torch.bfloat16: 0.0, torch.float16: 2.0 ** -24}


def _render(mf, depth, poses, K, dt, offset, **opts):
    n, h, w = depth.shape
    s = mf.MotionFocusStream(w, h, smooth_len=7, depth_dtype=depth.dtype, map_dtype=dt, **opts)
    s.push(poses, depth, K)
    room = torch.full((2, n * h * w + 8), 7.0, dtype=dt, device="cuda")
    M, G = (room[k, offset:offset + n * h * w].view(n, h, w) for k in range(2))
    _, _, info, _ = s.get_maps(out=(M, G))
    s.sync()
    s.close()
    rest = torch.cat([room[:, :offset], room[:, offset + n * h * w:]], 1)
    assert bool((rest == 7.0).all())          # nothing outside the planes is written
    return M.double().cpu().numpy(), G.double().cpu().numpy(), info


@pytest.mark.parametrize("width,height", [(1, 1), (3, 5), (63, 2), (511, 9), (513, 259), (1023, 7), (1027, 130)])
@pytest.mark.parametrize("storage", [("f32", "f32"), ("f32", "f16"), ("bf16", "f32"), ("bf16", "bf16"), ("f16", "f16")])
@pytest.mark.parametrize("window,normalize,mode", [(5, "count", "heading"), (16, "max", "accel"), (31, "count", "accel")])
def test_row_phases_against_tiled(width, height, storage, window, normalize, mode):
    import paper_2601_07154_gb300 as mf
    from synth.walker import WalkerSpec, walk
    types = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
    din, dout = (types[t] for t in storage)
    if normalize == "max" and dout == torch.float16:
        normalize = "count"    # in place, the tiled kernel's F16 maps lose their subnormal range
    n = 45
    poses = walk(WalkerSpec(n_frames=n, seed=width, turns=True, accel=1.5)).poses_w2c
    rng = np.random.default_rng(height)
    depth = rng.uniform(-0.2, 4.0, (n, height, width)).astype(np.float32)
    depth = torch.from_numpy(depth).cuda().to(din)
    K = np.array([0.8 * width + 1, 0.8 * width + 1, (width - 1) / 2, (height - 1) / 2])
    opts = dict(window=window, normalize=normalize, mode=mode)
    M, G, info = _render(mf, depth, poses, K, dout, 0, **opts)
    Mt, Gt, infot = _render(mf, depth, poses, K, dout, 1, **opts)
    for k in info.dtype.names:
        if k == "map_max":
            np.testing.assert_allclose(info[k], infot[k], rtol=1e-5)
        else:
            assert np.array_equal(info[k], infot[k], equal_nan=info[k].dtype.kind == "f"), k
    # an element's own maximum over its frame bounds the dropped terms (1 under "max")
    top = Mt.max(axis=(1, 2), keepdims=True)
    for a, b in ((M, Mt), (G, Gt)):
        tol = 2.0 ** -35 * top + (32 * 2.0 ** -23 + ROUND[dout]) * np.abs(b) + TINY[dout]
        assert np.all(np.abs(a - b) <= tol)
