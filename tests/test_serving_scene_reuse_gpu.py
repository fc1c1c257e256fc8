"""A server keeps captured graphs per scene.  A scene that is unloaded gives its handle's
address back, and the next one loaded usually gets it: the server must not take the
new scene's view for one it has a graph of (its launch grids, group costs and tile
lists follow the number of Gaussians).

Bar: the view rendered alone, 1e-5 (FP32 sums in another atomic order, as in
tests/test_serving_gpu.py).  Scenes of one precision, with and without the MLP.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


def test_reused_handle_addresses():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    from paper_2603_11531_gb300.serving import Server
    r = m.Renderer(0)
    srv = Server(r.ctx, slots=1, max_batch=1, hbm_budget_bytes=1 << 30)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 320, 240, 60.0)[1]
    addresses = []
    try:
        for k, (n, mlp) in enumerate([(40000, True), (9000, True), (25000, True), (25000, False),
                                      (1, False), (31000, True), (640, True)]):
            s = synth.unbounded_scene(n, seed=90 + k, precision="fp16")
            h = r.load_scene(s, synth.random_mlp(k) if mlp else None)
            addresses.append(h.value)
            ref = r.render(h, cam, use_mlp=mlp)["rgb"]
            for _ in range(2):   # captured, then relaunched
                out = torch.full((240, 320, 3), float("nan"), device="cuda")
                srv.wait(srv.submit(h, cam, m.render_opts(use_mlp=mlp), out))
                assert float((out - ref).abs().max()) <= 1e-5
            r.unload_scene(h)
        if len(set(addresses)) == len(addresses):
            pytest.skip("no handle address was given twice")
    finally:
        srv.close()
        r.close()
