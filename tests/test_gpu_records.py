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


@pytest.mark.parametrize("width,height,kernel,own", [(320, 240, "auto", 0), (640, 480, "tensor_cores", 1), (1920, 1080, "auto", 1),
                                                     (1921, 1080, "auto", 1)])
@pytest.mark.parametrize("normalize", ["count", "max"])
def test_records_cost_one_kernel_a_call_at_most(width, height, kernel, own, normalize):
    """Frames pushed singly and fetched at once: a map launch each, and one record kernel for all of them
    (none where the map launches write the records); the records are those of one push."""
    import paper_2601_07154_gb300 as mf
    dev = torch.device("cuda", 0)
    n = 20
    s, K = _open(mf, width, height, torch.cuda.Stream(dev), normalize=normalize, map_kernel=kernel)
    poses = _walk(n)
    gen = torch.Generator(device="cuda").manual_seed(7)
    depth = torch.rand((n, height, width), device=dev, generator=gen) * 4 + 0.25
    torch.cuda.synchronize()
    s.push(poses, depth, K)
    want = s.get_maps()
    per_map = 1 if normalize == "count" else 2       # the maximum's pass, or the division in place
    s.reset()
    for k in range(n):
        s.push(poses[k:k + 1], depth[k:k + 1], K)
    before = mf.mf_total_kernel_launches()
    got = s.get_maps()
    assert mf.mf_total_kernel_launches() - before == per_map * n + own
    for a, b in zip(got[:2], want[:2]):
        assert torch.equal(a, b)
    for a, b in zip(got[2:], want[2:]):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    s.close()


@pytest.mark.parametrize("n", [1, 63, 64, 65, 66, 300])
@pytest.mark.parametrize("normalize", ["count", "max"])
def test_either_writer_of_the_records(n, normalize):
    """One map unit a frame, around the number of units up to which the units write the records."""
    import paper_2601_07154_gb300 as mf
    s, K = _open(mf, 64, 16, torch.cuda.Stream(), normalize=normalize)
    poses = _walk(n)
    depth = torch.ones((n, 16, 64), device="cuda")
    torch.cuda.synchronize()
    s.push(poses, depth, K)
    before = mf.mf_total_kernel_launches()
    got = s.get_maps()
    assert mf.mf_total_kernel_launches() - before == (1 if normalize == "count" else 2) + (n > 64)
    s.reset()
    s.push(poses, depth, K)
    one = [s.get_maps(1) for _ in range(n)]
    for k in (2, 3):
        assert np.array_equal(got[k].view(np.uint8), np.concatenate([o[k] for o in one]).view(np.uint8))
    assert n < 30 or (got[2]["n_valid"] > 0).sum() > 0
    s.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 40])
@pytest.mark.parametrize("local", [False, True])
def test_host_poses_by_either_way(n, local):
    """Host poses go with the launch up to 16 of them, else by a copy: the records are those of device poses."""
    import paper_2601_07154_gb300 as mf
    overlap = 0 if not local else 3
    kw = dict(pose_frame="batch_local", overlap=overlap) if local else {}
    K = np.array([256.0, 256.0, 159.5, 119.5])
    poses = _walk(3 * (n + overlap) + 60)
    out = []
    for place in ("host", "device"):
        s = mf.MotionFocusStream(320, 240, window=8, smooth_len=7, mode="heading", cuda_stream=torch.cuda.Stream(), **kw)
        done, infos = 0, []
        for size in (40, n + overlap, n + overlap):
            P = poses[done:done + size].copy()
            done += size - overlap
            s.push(P if place == "host" else torch.from_numpy(P).cuda(), None, K)
            P[:] = np.nan                           # the call has what it needs
            infos.append(s.get_maps(want_maps=False)[2:])
        out.append(infos)
        s.close()
    for a, b in zip(*out):
        for x, y in zip(a, b):
            assert np.array_equal(x.view(np.uint8), y.view(np.uint8))
    assert out[0][-1][0]["n_valid"][-1] > 0
