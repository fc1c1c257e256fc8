"""MLP biases that need no gradient may be columns or rows: the image is that of flat
biases (1e-5: FP32 sums in another atomic order, tests/test_parity_gpu.py), and the
gradient of the attributes too (1e-4 of the largest)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth
from test_borrowed_scene_gpu import R, _close, _scene  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1])
def test_bias_with_a_unit_axis(R, axis):  # noqa: F811
    from paper_2603_11531_gb300 import autograd as ag
    _, a, mlp = _scene(2000, 4)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 97, 61, 60.0)[3]

    def step(m):
        x = a.clone().requires_grad_(True)
        img = ag.render(R, x, cam, m, use_mlp=True)
        return img.detach(), torch.autograd.grad(img.square().sum(), x)[0]

    ref = step(mlp)
    got = step(tuple(t.unsqueeze(axis) if t.ndim == 1 else t for t in mlp))
    _close(got[0], ref[0], 1e-5)
    _close(got[1], ref[1], 1e-4)
    with pytest.raises(ValueError):
        step((mlp[0], torch.cat([mlp[1], mlp[1]]).unsqueeze(axis), *mlp[2:]))
