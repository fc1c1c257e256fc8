"""Where the rasterisers stop updating T the image must not change: black Gaussians over
a background, whose pixels are T c_bg and nothing else.

Reference: T of the aux render of the same frame, which updates T throughout.  The two
renders multiply the same factors in another order (the lists' order differs from one
frame to the next): n factors, each rounded once on either side, so T differs by 2^-23 n
of itself at most, plus n steps of 2^-149 where a partial product is subnormal, each
scaled by the other partial products and c_bg <= 4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300
    return paper_2603_11531_gb300


def _black(n, opacity, precision):
    s = synth.uniform_scene(n, seed=n, precision="fp32")
    s.attrs[:, 0:3] *= 0.3
    s.attrs[:, 3:6] *= 3.0
    s.attrs[:, 10] = opacity
    s.attrs[:, 11:23] = 0.0
    s.attrs[:, 11:14] = -4.0      # colour max(0, 0.28 * -4 + 0.5) = 0
    if precision == "fp16":
        s.attrs = s.attrs.astype(np.float16)
    return s


@pytest.mark.parametrize("precision,fma", [("fp16", False), ("fp16", True), ("fp32", False)])
@pytest.mark.parametrize("n,opacity", [(127, 0.5), (257, 0.3), (600, 0.2), (1500, 0.1), (6000, 0.9)])
@pytest.mark.parametrize("bg", [(4.0, 0.0, -1.0), (0.1, 0.2, 0.3), (0.0, 0.0, 0.0)])
def test_black_foreground(m, precision, fma, n, opacity, bg):
    s = _black(n, opacity, precision)
    cam = synth.look_at((0.0, 0.0, -2.0), (0, 0, 0), 43, 37, 40.0)
    r = m.Renderer(0)
    try:
        h = r.load_scene(s)
        flags = m.MGS_FLAG_RASTER_FMA if fma else 0
        aux = r.render(h, cam, bg=bg, aux=True, flags=flags)
        plain = r.render(h, cam, bg=bg, flags=flags)["rgb"]
        counted = r.render(h, cam, bg=bg, count=True, flags=flags)["rgb"]
        rgb = torch.empty_like(plain)
        depth = torch.empty(plain.shape[:2], device="cuda")
        m.mgs_render_depth(r.ws, h, cam, m.render_opts(bg=bg, flags=flags), rgb, depth)
        torch.cuda.synchronize()
    finally:
        r.close()
    T = aux["aux"][4].cpu().numpy().astype(np.float64)[..., None]
    if n in (600, 1500):   # T below every freezing bound but one, and far from 0
        assert ((T > 2.0 ** -120) & (T < 2.0 ** -50)).any()
    want = T * np.asarray(np.float32(bg), np.float64)
    tol = 2.0 ** -23 * n * np.abs(want) + 4.0 * n * 2.0 ** -149
    for img in (plain, counted, rgb):
        assert (np.abs(img.cpu().numpy().astype(np.float64) - want) <= tol).all()
