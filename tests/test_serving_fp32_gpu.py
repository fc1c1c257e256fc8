"""FP32 views served side by side, among FP16 ones: every image equals the view rendered
alone (1e-5: FP32 sums in another order, tests/test_serving_gpu.py).  The batched
rasteriser sums FP32 views with other tile code than a lone view's."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precisions", [("fp32",), ("fp32", "fp16")])
def test_served_equals_alone(precisions):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    from paper_2603_11531_gb300.serving import Server
    r = m.Renderer(0)
    srv = Server(r.ctx, slots=8, max_batch=8, hbm_budget_bytes=2 << 30)
    try:
        scenes = [r.load_scene(synth.unbounded_scene(20000 + 7 * k, seed=50 + k, precision=p))
                  for k, p in enumerate(precisions)]
        opts = m.render_opts(bg=(0.3, 0.2, 0.1))
        reqs = [(scenes[k % len(scenes)], synth.orbit_cameras(24, 8.0, 1.0, 161 + 16 * (k % 5), 97, 60.0)[k])
                for k in range(24)]
        alone = [r.render(h, cam, bg=(0.3, 0.2, 0.1))["rgb"] for h, cam in reqs]
        outs = [torch.full_like(a, float("nan")) for a in alone]
        torch.cuda.synchronize()
        tickets = [srv.submit(h, cam, opts, o) for (h, cam), o in zip(reqs, outs)]
        for t in tickets:
            srv.wait(t)
        for o, a in zip(outs, alone):
            assert float((o - a).abs().max()) <= 1e-5
    finally:
        srv.close()
        r.close()
