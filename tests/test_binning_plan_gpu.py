"""Tile lists where the binning work plan changes shape: group and CTA edges of
the Gaussian count (32 per group, 512 per CTA), a last group with one Gaussian,
a workspace reused by a smaller and a larger scene.  Lists are compared as sets
with the oracle's, exactly."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 511, 513, 1024, 1025, 20_001, 77_825])
def test_lists(R, n, precision):
    s = synth.unbounded_scene(n, seed=n, precision=precision)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 250, 170, 60.0)[n % 8]
    h = R.load_scene(s)
    try:
        R.render(h, cam)
        off, gids = R.tile_lists()
    finally:
        R.unload_scene(h)
    g = oracle.preprocess(s.attrs, cam)
    ref_off, ref_gids = oracle.bin_tiles(g, cam.width, cam.height)
    assert np.array_equal(off, ref_off)
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    assert np.array_equal(gids[np.lexsort((gids, tile))], ref_gids[np.lexsort((ref_gids, tile))])
