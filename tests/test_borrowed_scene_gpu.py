"""Scenes over the caller's memory (training steps): equal to loaded scenes, and
safe when parameters change in place, streams change, or two graphs overlap.

Bars: images 1e-5 (FP32 sums in another atomic order, tests/test_parity_gpu.py);
gradients 1e-4 of the largest magnitude (the same, over a Gaussian's pixels)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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


def _scene(n, seed):
    s = synth.unbounded_scene(n, seed=seed, precision="fp32")
    s.mlp = synth.random_mlp(seed)
    f = lambda b: torch.from_numpy(synth.bf16_bits_to_f32(b).copy()).cuda()  # noqa: E731
    c = lambda x: torch.from_numpy(np.asarray(x, np.float32).copy()).cuda()  # noqa: E731
    mlp = (f(s.mlp.w1), c(s.mlp.b1), f(s.mlp.w2), c(s.mlp.b2), f(s.mlp.w3), c(s.mlp.b3))
    return s, torch.from_numpy(s.attrs).cuda(), mlp


def _close(a, b, tol):
    assert float((a - b).abs().max()) <= tol * max(1.0, float(b.abs().max())), float((a - b).abs().max())


@pytest.mark.parametrize("n", [1, 33, 5000])
@pytest.mark.parametrize("layout", ["plain", "strided", "float64"])
def test_image_equals_loaded_scene(R, n, layout):
    from paper_2603_11531_gb300 import autograd as ag
    s, a, mlp = _scene(n, 3)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 97, 61, 60.0)[3]
    h = R.load_scene(s)
    ref = R.render(h, cam, use_mlp=True)["rgb"]
    R.unload_scene(h)
    if layout == "strided":
        a = torch.cat([a, a], 1)[:, :24]
        mlp = tuple(t.t().contiguous().t() if t.ndim == 2 else t for t in mlp)
    if layout == "float64":
        mlp = tuple(t.double() for t in mlp)
    _close(ag.render(R, a, cam, mlp, use_mlp=True), ref, 1e-5)


def test_parameters_changed_in_place_between_forward_and_backward(R):
    from paper_2603_11531_gb300 import autograd as ag
    _, a0, mlp = _scene(3000, 5)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 96, 64, 60.0)[1]

    def step(spoil, other):
        a = a0.clone().requires_grad_(True)
        m = tuple(t.clone().requires_grad_(True) for t in mlp)
        img = ag.render(R, a, cam, m, use_mlp=True)
        if other:   # a second graph through the same workspace
            ag.render(R, a0 * 1.01, cam, mlp, use_mlp=True)
        if spoil:
            with torch.no_grad():
                a.data.mul_(2.0)
                m[0].data.zero_()
        return torch.autograd.grad(img.square().sum(), [a, *m])

    ref = step(False, False)
    for spoil, other in ((True, False), (False, True), (True, True)):
        for x, y in zip(step(spoil, other), ref):
            _close(x, y, 1e-4)


def test_steps_on_changing_streams(R):
    from paper_2603_11531_gb300 import autograd as ag
    _, a0, mlp = _scene(20000, 6)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 320, 240, 60.0)[2]

    def step():
        a = a0.clone().requires_grad_(True)
        img = ag.render(R, a, cam, mlp, use_mlp=True)
        return torch.autograd.grad(img.square().sum(), a)[0]

    ref = step()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = []
    for k in range(9):
        with torch.cuda.stream(streams[k % 3]):
            outs.append(step())
    torch.cuda.synchronize()
    for o in outs:
        _close(o, ref, 1e-4)


def test_refusals(R):
    from paper_2603_11531_gb300 import autograd as ag
    _, a, mlp = _scene(10, 7)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 32, 32, 60.0)[0]
    for bad in (a.cpu(), a[:, :23]):
        with pytest.raises(ValueError):
            ag.render(R, bad, cam)
    with pytest.raises(TypeError):
        ag.render(R, a.double(), cam)
    with pytest.raises((ValueError, AssertionError)):
        ag.render(R, a, cam, (mlp[0][:, :21], *mlp[1:]), use_mlp=True)
    with pytest.raises((ValueError, AssertionError)):
        ag.render(R, a, cam, (*mlp[:5], mlp[5][:4]), use_mlp=True)
    img = ag.render(R, a.clone().requires_grad_(True), cam)
    img.sum().backward(retain_graph=True)
    with pytest.raises(ValueError):      # the scene is gone after the first backward
        img.sum().backward()
