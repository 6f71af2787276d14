"""Result records, whoever writes them: a frame's last map unit (launches of few units) or a kernel of
their own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _walk(n, seed=3):
    from synth.walker import WalkerSpec, walk
    return np.ascontiguousarray(walk(WalkerSpec(n_frames=n, seed=seed, turns=True, accel=1.5)).poses_w2c)


def _open(mf, width, height, stream, window=8, **kw):
    s = mf.MotionFocusStream(width, height, window=window, smooth_len=7, mode="heading", cuda_stream=stream, **kw)
    K = np.array([0.8 * width, 0.8 * width, (width - 1) / 2, (height - 1) / 2])
    return s, K


@pytest.mark.parametrize("normalize", ["count", "max"])
@pytest.mark.parametrize("width,height", [(320, 240), (321, 240), (1920, 1080)])
def test_a_rendered_frame_can_be_rendered_again(width, height, normalize):
    """The same launches repeated (a captured mf_get_maps replayed) write the same record each time."""
    import paper_2601_07154_gb300 as mf
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(dev)
    n = 21
    s, K = _open(mf, width, height, st, normalize=normalize)
    gen = torch.Generator(device="cuda").manual_seed(7)
    depth = torch.rand((n, height, width), device=dev, generator=gen) * 4 + 0.25
    M, G = (torch.zeros((n, height, width), device=dev) for _ in range(2))
    info = torch.zeros((n, mf._mf.FRAME_INFO_DTYPE.itemsize), dtype=torch.uint8, device=dev)
    torch.cuda.synchronize()
    s.push(_walk(n), depth, K)
    mf.mf_get_maps(s.handle, n - 1, M, G, info, None)   # all but the last frame, at once
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        mf.mf_get_maps(s.handle, 1, M[n - 1:], G[n - 1:], info[n - 1:], None)
    seen = []
    for _ in range(3):
        info[n - 1:].zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        seen.append(info.cpu().numpy().view(mf._mf.FRAME_INFO_DTYPE)[n - 1, 0])
    assert seen[0]["frame_index"] == n - 1 and seen[0]["n_valid"] > 0 and seen[0]["map_max"] > 0
    assert seen[1] == seen[0] and seen[2] == seen[0]
    s.close()
