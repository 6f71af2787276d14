"""Odd widths: a clip's maps and records are the same bits however it is cut into calls, wherever its
planes start and in host or device memory, and 16-bit maps are the FP32 maps rounded once.

At an odd width the rows and frames of a clip start at every alignment, so which kernel, strip and unit
renders a pixel depends on where a launch's planes begin; what a pixel's sum leaves out must not.  The
sizes have strip, group and band edges inside the frame, and the narrow spreads put the limits at which
points are left out there too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

F32, BF16, F16 = torch.float32, torch.bfloat16, torch.float16
N = 40


def _inputs(width, height, seed=5):
    from synth.walker import WalkerSpec, walk
    poses = np.ascontiguousarray(walk(WalkerSpec(n_frames=N, seed=seed, turns=True, accel=1.5)).poses_w2c)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    # representable in every storage type, with depths that are no depth among them
    depth = torch.randint(-4, 129, (N, height, width), device="cuda", generator=gen).float() / 32
    depth.view(-1)[::97] = float("inf")
    depth.view(-1)[::89] = float("nan")
    K = np.array([0.8 * width + 1, 0.8 * width + 1, (width - 1) / 2, (height - 1) / 2])
    return poses, depth, K


def _placed(shape, dt, offset):
    """A plane stack that starts `offset` elements after an aligned address."""
    size = int(np.prod(shape))
    return torch.empty(size + 8, dtype=dt, device="cuda")[offset:offset + size].view(shape)


def _render(s, poses, depth, K, dt, pushes, gets, offsets):
    """M, G, info of a clip pushed and fetched in pieces of those sizes; depth, M and G start at `offsets`."""
    s.reset()
    D = _placed(depth.shape, depth.dtype, offsets[0])
    D.copy_(depth)
    M, G = (_placed(depth.shape, dt, o) for o in offsets[1:])
    info, done, k = [], 0, 0
    while done < N:
        n = min(pushes[k % len(pushes)], N - done)
        s.push(poses[done:done + n], D[done:done + n], K)
        done += n
        k += 1
    done = k = 0
    while done < N:
        n = min(gets[k % len(gets)], N - done)
        info.append(s.get_maps(n, out=(M[done:done + n], G[done:done + n]))[2])
        done += n
        k += 1
    return M, G, np.concatenate(info)


def _same(a, b, dt):
    assert torch.equal(a[0], b[0].to(dt)) and torch.equal(a[1], b[1].to(dt))
    assert np.array_equal(a[2].view(np.uint8), b[2].view(np.uint8))


WAYS = [([N], [N], (0, 0, 0)), ([N], [1], (0, 0, 0)), ([1], [N], (0, 0, 0)), ([7, 2], [3, 5, 1], (1, 0, 0)),
        ([N], [N], (1, 1, 1)), ([N], [N], (2, 3, 1))]


@pytest.mark.parametrize("width,height", [(1, 1), (3, 5), (129, 40), (511, 9), (513, 259), (853, 479), (1027, 131)])
@pytest.mark.parametrize("window", [5, 16, 31])
@pytest.mark.parametrize("normalize", ["count", "max"])
@pytest.mark.parametrize("sigma_rel,mode", [(0.1, "accel"), (0.02, "heading")])
def test_bits_do_not_depend_on_the_route(width, height, window, normalize, sigma_rel, mode):
    import paper_2601_07154_gb300 as mf
    poses, depth, K = _inputs(width, height)
    opts = dict(window=window, normalize=normalize, mode=mode, smooth_len=7, sigma_rel=sigma_rel)
    want = None
    for din, dout in ((F32, F32), (F32, F16), (BF16, F32), (BF16, BF16), (F16, F16)):
        s = mf.MotionFocusStream(width, height, depth_dtype=din, map_dtype=dout, **opts)
        for pushes, gets, offsets in WAYS:
            got = _render(s, poses, depth.to(din), K, dout, pushes, gets, offsets)
            if want is None:
                want = got
                full = torch.from_numpy(got[2]["n_valid"] > 0).cuda()
                top = got[0].amax((1, 2))
                assert int(full.sum()) > 20 and bool((top[full] > 0).any())
                if normalize == "max":  # tiny maxima stay as they are
                    assert bool(((top == 1) | (top < 2.0 ** -20)).all())
            _same(got, want, dout)
        s.close()


@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("normalize", ["count", "max"])
def test_host_memory_and_a_restored_stream(dt, normalize):
    """Staged planes start at every offset, and a restored stream's at others than the original's."""
    import paper_2601_07154_gb300 as mf
    width, height = 513, 259
    poses, depth, K = _inputs(width, height)
    depth = depth.to(dt)
    opts = dict(window=12, normalize=normalize, mode="heading", smooth_len=7, sigma_rel=0.02, depth_dtype=dt, map_dtype=dt)
    a = mf.MotionFocusStream(width, height, **opts)
    want = _render(a, poses, depth, K, dt, [N], [N], (0, 0, 0))
    host = depth.cpu()
    b = mf.MotionFocusStream(width, height, **opts)
    M, G = (torch.empty(depth.shape, dtype=dt, pin_memory=True) for _ in range(2))
    info, cut = [], 23
    b.push(poses[:3], host[:3], K)                 # moves the ring's head
    b.push(poses[3:cut], host[3:cut], K)
    for lo, hi in ((0, 2), (2, 9), (9, cut)):
        info.append(b.get_maps(hi - lo, out=(M[lo:hi], G[lo:hi]))[2])
    c = mf.MotionFocusStream(width, height, **opts)
    c.restore(b.snapshot())
    tails = []
    for s in (b, c):
        s.push(poses[cut:], host[cut:], K)
        tails.append(s.get_maps(out=(M[cut:], G[cut:]))[2])
        _same((M[cut:].cuda(), G[cut:].cuda(), tails[-1]), tuple(t[cut:] for t in want), dt)
    _same((M.cuda(), G.cuda(), np.concatenate(info + tails[:1])), want, dt)
    for s in (a, b, c):
        s.close()
