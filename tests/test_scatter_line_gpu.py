"""Tile lists on both sides of the line where the scatter starts to spread every batch
over its warp: 2^22 open sectors, one per binning CTA and tile.  The sizes follow from
the number of SMs (one CTA per SM: n is at least 512 per SM).  Compared as sets with the
oracle's, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [False, True])
@pytest.mark.parametrize("scale", [0.2, 2.0])
def test_lists_at_the_line(over, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    r = m.Renderer(0)
    try:
        sms = m.mgs_ctx_info(r.ctx)[0]
        tiles_x = int((2 ** 22 / sms) ** 0.5)
        tiles_y = 2 ** 22 // (sms * tiles_x) + int(over)
        assert (sms * tiles_x * tiles_y > 2 ** 22) == over
        assert abs(sms * tiles_x * tiles_y - 2 ** 22) <= sms * tiles_x
        width, height = 16 * tiles_x - 5, 16 * tiles_y - 11
        s = synth.unbounded_scene(512 * sms + 1, seed=9, precision="fp32")
        s.attrs[:, 3:6] *= scale
        cam = synth.orbit_cameras(8, 8.0, 1.0, width, height, 60.0)[3]
        r.render(r.load_scene(s), cam)
        off, gids = r.tile_lists()
    finally:
        r.close()
    ref_off, ref_gids = oracle.bin_tiles(oracle.preprocess(s.attrs, cam), width, height)
    assert np.array_equal(off, ref_off)
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    assert np.array_equal(gids[np.lexsort((gids, tile))], ref_gids[np.lexsort((ref_gids, tile))])
