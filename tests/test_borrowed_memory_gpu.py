"""A training step's copies of its parameters end with its backward pass, also when the
program keeps the loss and with it the graph."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_mlp", [False, True])
def test_kept_losses_do_not_keep_scenes(use_mlp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    from paper_2603_11531_gb300 import autograd as ag
    n = 100_000
    a = torch.from_numpy(synth.unbounded_scene(n, seed=3, precision="fp32").attrs).cuda()
    a.requires_grad_(True)
    mlp = None
    if use_mlp:
        shapes = [(64, 22), (64,), (64, 64), (64,), (5, 64), (5,)]
        mlp = tuple((0.1 * torch.ones(s, device="cuda")).requires_grad_(True) for s in shapes)
    cam = synth.orbit_cameras(8, 8.0, 1.0, 64, 48, 60.0)[1]
    r = m.Renderer(0)
    kept = []
    try:
        for k in range(6):
            loss = ag.render(r, a, cam, mlp, use_mlp=use_mlp).square().sum()
            loss.backward()
            kept.append(loss)
            torch.cuda.synchronize()
            if k == 1:
                base = torch.cuda.memory_allocated()
        # four more steps: less than half of one step's copy of the attributes
        assert torch.cuda.memory_allocated() - base < n * 96 // 2
    finally:
        r.close()
