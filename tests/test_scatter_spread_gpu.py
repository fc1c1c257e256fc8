"""Lists of images with so many tiles that every batch of rows is spread over its
warp (one open sector per CTA and tile, 128 MB of them), and just below that line.
Compared as sets with the oracle's, exactly; the rows are one to a few tiles long."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(3840, 2160), (4111, 2999), (2560, 1440)])
@pytest.mark.parametrize("scale", [0.2, 2.0])
def test_lists(width, height, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    s = synth.unbounded_scene(80_000, seed=9, precision="fp32")
    s.attrs[:, 3:6] *= scale
    cam = synth.orbit_cameras(8, 8.0, 1.0, width, height, 60.0)[3]
    R = m.Renderer(0)
    try:
        h = R.load_scene(s)
        R.render(h, cam)
        off, gids = R.tile_lists()
        R.unload_scene(h)
    finally:
        R.close()
    ref_off, ref_gids = oracle.bin_tiles(oracle.preprocess(s.attrs, cam), width, height)
    assert np.array_equal(off, ref_off)
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    assert np.array_equal(gids[np.lexsort((gids, tile))], ref_gids[np.lexsort((ref_gids, tile))])
