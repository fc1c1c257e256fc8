"""Rasteriser adjoint at the edges of its decomposition (8x8 blocks, batches of
32 candidates, lists split over CTAs), against the oracle gradient.

Tolerance: 2e-3 of the largest magnitude per parameter kind, the bar of FP32
gradients against the FP64 oracle (tests/test_backward_gpu.py).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import grad as og
from paper_2603_11531_gb300 import synth
from test_backward_gpu import COLS, R, _compare, _gpu_grads, _ref_grads  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,width,height", [
    (1, 7, 5),         # one candidate, less than a block
    (31, 17, 9),       # a batch short of full, ragged tiles and blocks
    (33, 16, 16),      # a batch and one more candidate
    (700, 33, 47),     # many batches per block, eight CTAs per tile
    (900, 641, 490),   # 1271 tiles: two CTAs per tile
])
def test_sizes(R, n, width, height):  # noqa: F811
    s = synth.uniform_scene(n, seed=n, precision="fp32")
    s.attrs[: n // 2, 10] = 0.999      # the 0.99 clamp of alpha is active
    s.attrs[::7, 10] = 0.0             # log2 o = -inf
    cam = synth.look_at((0.2, -0.1, -2.6), (0, 0, 0), width, height, 60.0)
    dL = np.random.default_rng(n).normal(size=(height, width, 3))
    gpu, _ = _gpu_grads(R, s.attrs, cam, dL, bg=(0.3, 0.2, 0.1))
    ref = _ref_grads(s.attrs, cam, dL, bg=(0.3, 0.2, 0.1))
    kinds = dict(COLS)
    live = s.attrs[:, 10] > 0          # o = 0: the kernel defines dL/do as 0
    assert np.all(gpu["attrs"][~live, 10] == 0)
    ref["o"] = np.where(live, ref["o"], 0.0)
    _compare(gpu, ref, tol=2e-3, kinds=kinds)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_pixel_stays_with_its_gaussians(R, bad):  # noqa: F811
    """dL/dC not finite at one pixel: a Gaussian that does not include the pixel
    keeps the gradient it has when that pixel's dL/dC is 0."""
    s = synth.uniform_scene(400, seed=12, precision="fp32")
    cam = synth.look_at((0.2, -0.1, -2.6), (0, 0, 0), 48, 40, 60.0)
    dL = np.random.default_rng(4).normal(size=(40, 48, 3))
    dL[21, 13] = 0.0
    clean, _ = _gpu_grads(R, s.attrs, cam, dL)
    dL[21, 13] = bad
    got, _ = _gpu_grads(R, s.attrs, cam, dL)
    st = og.discrete_structure(s.attrs, cam)
    touched = np.zeros(s.n, bool)
    touched[st["gid"].numpy()[st["pix"].numpy() == 21 * 48 + 13]] = True
    assert touched.any() and (~touched).any()
    assert np.isfinite(got["attrs"][~touched]).all()
    assert not np.isfinite(got["attrs"][touched]).all()
    # FP32 sums in another atomic order: 2^-24 per addition over up to 40 x 48 pixels
    scale = np.abs(clean["attrs"]).max()
    assert np.abs(got["attrs"][~touched] - clean["attrs"][~touched]).max() <= 1e-4 * scale
