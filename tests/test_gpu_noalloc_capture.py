"""mf_render_noalloc under stream capture: a replayed graph of its dependent launches gives what the call
itself gives, every time it is replayed, for launches that write their records and for larger ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,n", [(320, 240, 2), (321, 241, 3), (640, 480, 20)])
@pytest.mark.parametrize("normalize", ["count", "max"])
@pytest.mark.parametrize("dt", [torch.float32, torch.float16])
def test_replayed_renders_equal_the_call(width, height, n, normalize, dt):
    import paper_2601_07154_gb300 as mf
    from synth.walker import WalkerSpec, walk
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(dev)
    types = {torch.float32: mf.MF_F32, torch.float16: mf.MF_F16}
    poses = torch.from_numpy(np.ascontiguousarray(
        walk(WalkerSpec(n_frames=n + 20, seed=4, turns=True, accel=1.5)).poses_w2c)).to(dev)
    gen = torch.Generator(device="cuda").manual_seed(3)
    depth = (torch.rand((n, height, width), device=dev, generator=gen) * 4 + 0.25).to(dt)
    K = np.array([0.8 * width, 0.8 * width, (width - 1) / 2, (height - 1) / 2])
    desc = mf.mf_stream_desc_init(width=width, height=height, window=8, smooth_len=7, mode=mf.MF_MODE_HEADING,
                                  depth_dtype=types[dt], map_dtype=types[dt], cuda_stream=st.cuda_stream,
                                  normalize=mf.MF_NORM_MAX if normalize == "max" else mf.MF_NORM_COUNT)

    def outputs():
        M, G = (torch.zeros((n, height, width), dtype=dt, device=dev) for _ in range(2))
        return M, G, torch.zeros((n, 64), dtype=torch.uint8, device=dev)

    def render(out):
        mf.mf_render_noalloc(desc, n + 20, poses, n, depth, K, *out)

    want, got = outputs(), outputs()
    torch.cuda.synchronize()
    render(want)
    torch.cuda.synchronize()
    assert int(want[2].view(torch.int32)[:, 3].min()) > 0      # n_valid
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        render(got)
    for _ in range(3):
        for t in got:
            t.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
