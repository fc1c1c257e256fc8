"""A pixel that a Gaussian does not include adds nothing to its gradient, also where
the products of the Gaussian's (finite, very large) Eq. 3 weight or colour and the
pixel's (finite) loss gradient leave the FP32 range.

Needles along the view axis close to the camera have weights exp(s_max / d) up to
4e35 and a footprint of a few pixels; the other pixels of their 8x8 blocks belong to
ordinary Gaussians.  Tolerance: 2e-3 of the largest magnitude per parameter kind
(FP32 against the FP64 oracle, tests/test_backward_gpu.py).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth
from test_backward_gpu import R, _compare, _gpu_grads, _ref_grads  # noqa: F401

pytestmark = pytest.mark.gpu


def _needle(exponent, opacity, colour):
    a = np.zeros((1, 24), np.float32)
    a[0, 0:3] = (0.0, 0.0, -2.75)
    a[0, 3:6] = (0.002, 0.002, 0.25 * exponent)
    a[0, 6] = 1.0
    a[0, 10] = opacity
    a[0, 11:14] = colour
    return a


@pytest.mark.parametrize("exponent", [60.0, 78.0, 82.0])   # weights 1e26, 7e33, 4e35
@pytest.mark.parametrize("opacity", [0.9, 0.995])          # 0.995: the 0.99 clamp is active
def test_large_weight(R, exponent, opacity):  # noqa: F811
    base = synth.uniform_scene(300, seed=5, precision="fp32").attrs
    attrs = np.concatenate([base, _needle(exponent, opacity, 0.5)]).astype(np.float32)
    cam = synth.look_at((0.0, 0.0, -3.0), (0, 0, 0), 48, 40, 60.0)
    dL = 1e6 * np.random.default_rng(7).normal(size=(40, 48, 3))
    gpu, _ = _gpu_grads(R, attrs, cam, dL, bg=(0.3, 0.2, 0.1))
    assert np.isfinite(gpu["attrs"]).all()
    _compare(gpu, _ref_grads(attrs, cam, dL, bg=(0.3, 0.2, 0.1)), tol=2e-3)


def test_large_colour(R):  # noqa: F811
    """Colours of 1e30 in a part of the scene: finite gradients for every Gaussian
    that shares no included pixel with them."""
    base = synth.uniform_scene(300, seed=6, precision="fp32").attrs
    attrs = np.concatenate([base, _needle(4.0, 0.9, 1e30)]).astype(np.float32)
    cam = synth.look_at((0.0, 0.0, -3.0), (0, 0, 0), 48, 40, 60.0)
    dL = 1e12 * np.random.default_rng(8).normal(size=(40, 48, 3))
    from oracle import grad as og
    st = og.discrete_structure(attrs, cam)
    gid, pix = st["gid"].numpy(), st["pix"].numpy()
    mine = np.unique(pix[gid == len(base)])
    dL.reshape(-1, 3)[mine] = 0.0     # its own pixels carry no loss
    gpu, _ = _gpu_grads(R, attrs, cam, dL)
    assert np.isfinite(gpu["attrs"]).all()
    assert np.abs(gpu["attrs"][-1]).max() == 0.0
