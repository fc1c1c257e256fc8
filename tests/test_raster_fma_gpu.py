"""FP32 rasteriser at the edges of its decomposition (8x8 blocks, groups of four
candidates, ring wrap-around, frozen transmittance), against the oracle.

Bar: 1e-4 per pixel for FP32 attributes (tests/test_parity_gpu.py), counts
exact.  The frozen transmittance adds at most 2^-48 * 256.
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


@pytest.mark.parametrize("n,width,height", [(1, 7, 5), (3, 8, 8), (5, 17, 9), (36, 16, 16), (37, 33, 31),
                                            (900, 45, 61)])
@pytest.mark.parametrize("opaque", [False, True])
def test_sizes(R, n, width, height, opaque):
    s = synth.uniform_scene(n, seed=n, precision="fp32")
    if opaque:
        s.attrs[::2, 10] = 1.0     # the 0.99 clamp of alpha is active
    cam = synth.look_at((0.1, 0.2, -2.5), (0, 0, 0), width, height, 60.0)
    h = R.load_scene(s)
    try:
        for kw in ({}, {"count": True}, {"aux": True}):
            out = R.render(h, cam, bg=(0.4, 0.1, 0.2), **kw)
            ref = oracle.render(s.attrs, cam, bg=(0.4, 0.1, 0.2), want_count=True)
            assert np.abs(out["rgb"].cpu().numpy() - ref["rgb"]).max() <= 1e-4
            if "count" in kw:
                assert np.array_equal(out["count"].cpu().numpy(), ref["count"])
    finally:
        R.unload_scene(h)


@pytest.mark.parametrize("bg", [(1.0, 0.5, 0.0), (0.0, 256.0, 1.0), (1e6, 1.0, 1.0)])
def test_frozen_transmittance(R, bg):
    """Thousands of Gaussians in front of every pixel: T falls below every bound,
    with and without a background that allows T to be frozen."""
    s = synth.uniform_scene(6000, seed=3, precision="fp32")
    s.attrs[:, 0:3] *= 0.3
    s.attrs[:, 3:6] *= 3.0
    s.attrs[:, 10] = 0.9
    cam = synth.look_at((0.0, 0.0, -2.0), (0, 0, 0), 48, 40, 40.0)
    h = R.load_scene(s)
    try:
        out = R.render(h, cam, bg=bg)["rgb"].cpu().numpy()
        aux = R.render(h, cam, bg=bg, aux=True)
        T = aux["aux"][4].cpu().numpy()
        assert (T < 2.0 ** -60).any()
        ref = oracle.render(s.attrs, cam, bg=bg, want_count=True)["rgb"]
        scale = max(1.0, max(bg))
        assert np.abs(out - ref).max() <= 1e-4 * scale
        assert np.abs(aux["rgb"].cpu().numpy() - ref).max() <= 1e-4 * scale
    finally:
        R.unload_scene(h)
