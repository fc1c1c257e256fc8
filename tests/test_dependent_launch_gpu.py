"""Kernels launched as programmatic dependents: back-to-back frames of different
views through one workspace, renders right behind a kernel that writes their
input, and a captured graph give the images of synchronised renders.

Bar: 1e-5 (FP32 sums in another atomic order, tests/test_parity_gpu.py)."""
import pytest

torch = pytest.importorskip("torch")

import paper_2603_11531_gb300 as m
from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = m.Renderer(0)
    yield r
    r.close()


def _scene(precision, n=30_000):
    s = synth.unbounded_scene(n, seed=8, precision=precision)
    s.mlp = synth.random_mlp(8)
    return s, synth.orbit_cameras(16, 8.0, 1.0, 320, 240, 60.0)


def _close(a, b):
    assert float((a - b).abs().max()) <= 1e-5


@pytest.mark.parametrize("precision", ["fp16", "fp32"])
def test_back_to_back_frames(R, precision):
    s, cams = _scene(precision)
    h = R.load_scene(s)
    try:
        opts = m.render_opts(True)
        ref = [R.render(h, c, use_mlp=True)["rgb"] for c in cams]
        outs = [torch.empty_like(ref[0]) for _ in cams]
        for _ in range(5):
            for c, o in zip(cams, outs):
                m.mgs_render(R.ws, h, c, opts, o)
        torch.cuda.synchronize()
        for o, r in zip(outs, ref):
            _close(o, r)
    finally:
        R.unload_scene(h)


def test_input_written_by_the_kernel_before(R):
    s, cams = _scene("fp32", 100_000)
    a = torch.from_numpy(s.attrs).cuda()
    h = R.load_scene(s.attrs)
    ref = R.render(h, cams[3])["rgb"]
    R.unload_scene(h)
    out = torch.empty_like(ref)
    buf = torch.zeros_like(a)
    for _ in range(10):
        buf.zero_()
        buf.add_(a)                # the kernel right before the render
        m.mgs_render_static(buf, cams[3], m.render_opts(), out)
        _close(out, ref)


def test_captured_graph(R):
    s, cams = _scene("fp16")
    h = R.load_scene(s)
    try:
        opts = m.render_opts(True)
        ref = R.render(h, cams[5], use_mlp=True)["rgb"]
        out = torch.zeros_like(ref)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            m.mgs_render(R.ws, h, cams[5], opts, out)
        for _ in range(3):
            out.zero_()
            g.replay()
            torch.cuda.synchronize()
            _close(out, ref)
    finally:
        R.unload_scene(h)


def test_server_uses_graphs(R):
    from paper_2603_11531_gb300 import serving
    s, cams = _scene("fp16")
    h = R.load_scene(s)
    srv = serving.Server(R.ctx, slots=3, max_batch=2)
    try:
        opts = m.render_opts(True)
        ref = [R.render(h, c, use_mlp=True)["rgb"] for c in cams]
        outs = [torch.empty_like(r) for r in ref]
        for _ in range(2):
            for t in [srv.submit(h, c, opts, o) for c, o in zip(cams, outs)]:
                srv.wait(t)
        assert srv.stats()["graphs"]
        for o, r in zip(outs, ref):
            _close(o, r)
    finally:
        srv.close()
        R.unload_scene(h)
