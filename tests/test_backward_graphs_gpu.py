"""A graph that holds a render of a renderer, launched on another stream right after
that renderer's backward pass, finds the pass's kernels done.

Bars and the busy wait: tests/test_backward_streams_gpu.py."""
import pytest

torch = pytest.importorskip("torch")

from test_backward_streams_gpu import H, W, _backward_behind_a_wait, env  # noqa: F401

pytestmark = pytest.mark.gpu


def test_graph_launch_after_backward(env):  # noqa: F811
    m, r, train, shown, cams = env
    assert not m.mgs_workspace_captured(r.ws)
    ref_grad = _backward_behind_a_wait(r, train, cams[1], False)
    ref = r.render(shown, cams[2])["rgb"]
    out = torch.zeros((H, W, 3), device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(second):
        g.capture_begin()
        m.mgs_render(r.ws, shown, cams[2], m.render_opts(), out)
        g.capture_end()
    assert m.mgs_workspace_captured(r.ws)
    with torch.cuda.stream(first):
        grad = _backward_behind_a_wait(r, train, cams[1], True)
    with torch.cuda.stream(second):
        g.replay()
    torch.cuda.synchronize()
    assert float((grad - ref_grad).abs().max()) <= 1e-4 * float(ref_grad.abs().max())
    assert float((out - ref).abs().max()) <= 1e-5 * max(1.0, float(ref.abs().max()))
