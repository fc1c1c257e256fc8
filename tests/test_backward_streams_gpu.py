"""A backward pass returns before its kernels are done with the renderer's
workspace; whatever the program does next with that renderer on another stream is
ordered after them.

A bounded busy wait ahead of the backward pass keeps its kernels from starting while
the next call is made, so an unordered call would certainly overtake them.  Both
scenes have the same number of Gaussians.  Bars: those of tests/test_borrowed_scene_gpu.py
(FP32 sums in another atomic order): images 1e-5, gradients 1e-4 of the largest.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu

N, W, H = 4000, 160, 96
WAIT = 40_000_000   # clock cycles: about 20 ms


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    r = m.Renderer(0)
    train = torch.from_numpy(synth.unbounded_scene(N, seed=41, precision="fp32").attrs).cuda()
    shown = r.load_scene(synth.unbounded_scene(N, seed=42, precision="fp32"))
    cams = synth.orbit_cameras(8, 8.0, 1.0, W, H, 60.0)
    yield m, r, train, shown, cams
    r.close()


def _backward_behind_a_wait(r, train, cam, wait):
    from paper_2603_11531_gb300 import autograd as ag
    a = train.clone().requires_grad_(True)
    img = ag.render(r, a, cam)
    loss = img.square().sum()
    if wait:
        torch.cuda._sleep(WAIT)
    return torch.autograd.grad(loss, a)[0]


def _next_call(kind, m, r, shown, cam):
    if kind == "render":
        return r.render(shown, cam)["rgb"]
    if kind == "unchecked":
        return r.render(shown, cam, checked=False)["rgb"]
    if kind == "depth":
        return r.render_depth(shown, cam)["depth"]
    if kind == "to_host":
        host = torch.empty((H, W, 3), pin_memory=True)
        m.mgs_render_to_host(r.ws, shown, cam, m.render_opts(), host)
        torch.cuda.current_stream().synchronize()
        return host.cuda()
    if kind == "captured":
        out = torch.zeros((H, W, 3), device="cuda")
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.current_stream()
        g.capture_begin()
        m.mgs_render(r.ws, shown, cam, m.render_opts(), out)
        g.capture_end()
        g.replay()
        side.synchronize()
        return out
    off, gids = r.tile_lists()   # the backward pass's lists, complete
    tile = np.repeat(np.arange(len(off) - 1), np.diff(off))
    return off, gids[np.lexsort((gids, tile))]


@pytest.mark.parametrize("kind", ["render", "unchecked", "depth", "to_host", "captured", "lists"])
def test_next_call_on_another_stream(env, kind):
    m, r, train, shown, cams = env
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    ref_grad = _backward_behind_a_wait(r, train, cams[1], False)
    ref_next = _next_call("lists" if kind == "lists" else "render" if kind != "depth" else kind,
                          m, r, shown, cams[2])
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        grad = _backward_behind_a_wait(r, train, cams[1], True)
    with torch.cuda.stream(second):
        got = _next_call(kind, m, r, shown, cams[2])
    torch.cuda.synchronize()
    assert float((grad - ref_grad).abs().max()) <= 1e-4 * float(ref_grad.abs().max())
    if kind == "lists":
        assert all(np.array_equal(x, y) for x, y in zip(got, ref_next))
    else:
        assert float((got - ref_next).abs().max()) <= 1e-5 * max(1.0, float(ref_next.abs().max()))
