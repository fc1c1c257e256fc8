"""Work shares of the binning warps at their extremes: no visible Gaussian, one in
the last group, one group holding nearly all the cost, more chunks of groups than
the plan's scan holds (chunks doubled), a group of views binned with fewer CTAs
than their scratch is laid out for.  Lists are compared as sets with the oracle's,
exactly; served images with rendered ones to 1e-5 (FP32 sums in another order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    r = m.Renderer(0)
    yield r
    r.close()


def _scene(n, visible):
    """n Gaussians, all behind the camera but those of the index array."""
    small = synth.uniform_scene(1000, seed=n % 1000, precision="fp32").attrs
    a = np.tile(small, ((n + 999) // 1000, 1))[:n]
    a[:, 2] -= 100.0
    a[visible, 2] += 100.0
    return a


CAM = dict(eye=(0.1, 0.2, -2.5), width=200, height=150)


@pytest.mark.parametrize("case", ["none", "last", "first_group", "chunks"])
def test_shares(R, case):
    n = {"none": 5000, "last": 40_001, "first_group": 70_000, "chunks": 2048 * 128 * 32 + 33}[case]
    vis = {"none": [], "last": [n - 1], "first_group": np.arange(0, n, 50),
           "chunks": np.arange(1, n, 997)}[case]
    a = _scene(n, np.asarray(vis, dtype=np.int64))
    if case == "first_group":
        a[:32, 0:3] = 0.0
        a[:32, 3:6] = 3.0            # cover the image
    cam = synth.look_at(CAM["eye"], (0, 0, 0), CAM["width"], CAM["height"], 60.0)
    h = R.load_scene(synth.Scene(a))
    try:
        for _ in range(2):           # the plan's scratch holds the previous frame's
            R.render(h, cam)
            off, gids = R.tile_lists()
    finally:
        R.unload_scene(h)
    g = oracle.preprocess(a, cam)
    ref_off, ref_gids = oracle.bin_tiles(g, cam.width, cam.height)
    assert np.array_equal(off, ref_off)
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    assert np.array_equal(gids[np.lexsort((gids, tile))], ref_gids[np.lexsort((ref_gids, tile))])


def test_grouped_views(R):
    """Served in one group, 90k Gaussians (more than half an SM count of CTAs)."""
    import paper_2603_11531_gb300 as m
    from paper_2603_11531_gb300 import serving
    s = synth.unbounded_scene(90_000, seed=4, precision="fp16")
    cams = synth.orbit_cameras(8, 8.0, 1.0, 320, 240, 60.0)
    h = R.load_scene(s)
    srv = serving.Server(R.ctx, slots=8, max_batch=8)
    try:
        outs = [torch.empty((240, 320, 3), device="cuda") for _ in cams]
        opts = m.render_opts()
        for _ in range(3):
            for t in [srv.submit(h, c, opts, o) for c, o in zip(cams, outs)]:
                srv.wait(t)
        torch.cuda.synchronize()
        for c, o in zip(cams, outs):
            ref = R.render(h, c)["rgb"]
            assert (o - ref).abs().max().item() <= 1e-5
    finally:
        srv.close()
        R.unload_scene(h)
