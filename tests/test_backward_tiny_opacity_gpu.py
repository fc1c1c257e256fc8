"""Opacities below FP32's smallest normal number: alpha is flushed to 0, and like an
opacity of 0 they get no gradient through alpha (0 times 1 / o, which may be infinite,
is not a gradient).  The other Gaussians' gradients are those without them.

Tolerance: 1e-4 of the largest magnitude (FP32 sums in another atomic order,
tests/test_borrowed_scene_gpu.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth
from test_backward_gpu import R, _gpu_grads  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opacity", [1e-45, 1e-40, 2.9e-39, 1e-38, 1.2e-38, 1e-30])
def test_tiny_opacity(R, opacity):  # noqa: F811
    attrs = synth.uniform_scene(300, seed=5, precision="fp32").attrs
    cam = synth.look_at((0.2, -0.1, -2.6), (0, 0, 0), 48, 40, 60.0)
    dL = np.random.default_rng(0).normal(size=(40, 48, 3))
    attrs[::3, 10] = 0.0
    zero, _ = _gpu_grads(R, attrs, cam, dL, bg=(0.3, 0.2, 0.1))
    attrs[::3, 10] = opacity
    tiny, _ = _gpu_grads(R, attrs, cam, dL, bg=(0.3, 0.2, 0.1))
    assert np.isfinite(tiny["attrs"]).all()
    rest = np.arange(len(attrs)) % 3 != 0
    scale = np.abs(zero["attrs"][rest]).max()
    assert np.abs(tiny["attrs"][rest] - zero["attrs"][rest]).max() <= 1e-4 * scale
    if opacity < 2.0 ** -126:
        assert np.abs(tiny["attrs"][::3, 10]).max() == 0.0
