"""Load-time kernels at their edges: the spatial sort's blocks of 4,096 keys (one
key, a full block, one more, equal keys, non-finite means), and the SH decode's
four Gaussians per thread and its accesses on buffers that are not aligned.

Lists are compared as sets with the scene stored as given (the caller's indices:
every Gaussian must be stored exactly once).  Decode bars: tests/test_sh_decode_gpu.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    r = m.Renderer(0)
    yield m, r
    r.close()


def _lists(m, r, attrs, cam, order, on_device):
    h = r.load_scene(torch.from_numpy(attrs).cuda() if on_device else attrs, order=order)
    try:
        img = r.render(h, cam)["rgb"]
        off, gids = r.tile_lists()
    finally:
        r.unload_scene(h)
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    return img, off, gids[np.lexsort((gids, tile))]


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("n,kind", [(2, ""), (31, ""), (4095, ""), (4096, ""), (4097, ""), (8193, "equal"),
                                    (5000, "non-finite"), (100_003, "")])
def test_spatial_sort(env, n, kind, precision):
    m, r = env
    s = synth.unbounded_scene(n, seed=n, precision=precision)
    if kind == "equal":
        s.attrs[:, 0:3] = (0.1, 0.2, 0.3)
    if kind == "non-finite":
        s.attrs[::7, 0] = np.nan
        s.attrs[::11, 2] = np.inf
    cam = synth.orbit_cameras(8, 8.0, 1.0, 200, 130, 60.0)[5]
    a = _lists(m, r, s.attrs, cam, m.MGS_ORDER_AS_GIVEN, False)
    for on_device in (False, True):
        b = _lists(m, r, s.attrs, cam, m.MGS_ORDER_SPATIAL, on_device)
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
        assert float((a[0] - b[0]).abs().max()) <= 1e-5


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("n", [1, 255, 257, 1023, 1025, 5000])
@pytest.mark.parametrize("offset", [0, 1])
def test_decode(env, n, precision, offset):
    m, r = env
    dt = torch.float16 if precision == "fp16" else torch.float32
    md, mv = synth.random_sh_decoders(n)
    h = synth.compressed_sh_features(n, seed=n, precision=precision)
    hb = torch.zeros(6 * n + 8, dtype=dt, device="cuda")
    ab = torch.full((24 * n + 8,), 7.0, dtype=dt, device="cuda")
    hd = hb[offset:offset + 6 * n].view(n, 6)       # offset 1: one element off any vector alignment
    ad = ab[offset:offset + 24 * n].view(n, 24)
    hd.copy_(torch.from_numpy(h))
    m.mgs_decode_sh(r.ctx, hd, md, mv, ad)
    got = ab.float().cpu().numpy()
    rows = got[offset:offset + 24 * n].reshape(n, 24)
    ref = oracle.decode_sh(h.astype(np.float64), md, mv)
    err = np.abs(rows[:, 11:23] - ref)
    assert (err <= (np.abs(ref) * 2.0 ** -11 if precision == "fp16" else 0.0) + 1e-5).all()
    rows[:, 11:23] = 7.0
    assert (got == 7.0).all()                        # nothing else is touched
