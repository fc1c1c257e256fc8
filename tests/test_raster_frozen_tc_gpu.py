"""Frozen transmittance of the tensor-core sums.

Once every lane of a warp holds partial products of at most 2^-8 for its pixels,
T <= 2^-32 and is no longer updated (checked every 128 list entries, backgrounds up
to 4, not with aux output, which returns T).  Bar: the aux render of the same frame
evaluates the same sums with T updated throughout.  The images may differ by 2^-32
(|c_bg| + 1) for the frozen T, and, as the order within a list differs from one frame
to the next, by the worst rounding of n-term FP32 sums and products: 2^-22 n of the
colour and 2^-23 n of T c_bg.
"""
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


@pytest.mark.parametrize("n", [127, 128, 129, 256, 6000])
@pytest.mark.parametrize("opacity", [0.9, 1.0])          # 1.0: alpha clamped to 0.99
@pytest.mark.parametrize("bg", [(1.0, 0.5, 0.0), (4.0, 0.0, 1.0), (1e6, 1.0, 1.0)])
def test_frozen(R, n, opacity, bg):
    s = synth.uniform_scene(n, seed=n, precision="fp16")
    s.attrs[:, 0:3] *= 0.3
    s.attrs[:, 3:6] *= 3.0
    s.attrs[:, 10] = opacity
    cam = synth.look_at((0.0, 0.0, -2.0), (0, 0, 0), 43, 37, 40.0)
    h = R.load_scene(s)
    try:
        out = R.render(h, cam, bg=bg)["rgb"].cpu().numpy().astype(np.float64)
        cnt = R.render(h, cam, bg=bg, count=True)
        aux = R.render(h, cam, bg=bg, aux=True)
    finally:
        R.unload_scene(h)
    ref = aux["rgb"].cpu().numpy().astype(np.float64)
    T = aux["aux"][4].cpu().numpy().astype(np.float64)[..., None]
    assert n < 256 or (T < 2.0 ** -40).any()
    tol = 2.0 ** -32 * (min(max(bg), 4.0) + 1.0) + 2.0 ** -23 * n * (2.0 * np.abs(ref).max() * (1.0 - T)
                                                                    + T * max(bg))
    for img in (out, cnt["rgb"].cpu().numpy()):
        assert (np.abs(img - ref) <= tol).all()
    want = oracle.render(s.attrs, cam, bg=bg, want_count=True)
    assert np.array_equal(cnt["count"].cpu().numpy(), want["count"])
