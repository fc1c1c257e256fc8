"""A call that fails on the host (here: a workspace larger than the device) reports its
error itself; the calls after it, which check their launches, do not see it again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2603_11531_gb300 import synth

pytestmark = pytest.mark.gpu


def _decode(m, r):
    h = torch.zeros((64, 6), device="cuda")
    attrs = torch.zeros((64, 24), device="cuda")
    m.mgs_decode_sh(r.ctx, h, *synth.random_sh_decoders(1), attrs)


def _backward(m, r):
    from paper_2603_11531_gb300 import autograd as ag
    a = torch.from_numpy(synth.uniform_scene(100, seed=1, precision="fp32").attrs).cuda()
    a.requires_grad_(True)
    cam = synth.look_at((0.2, -0.1, -2.6), (0, 0, 0), 48, 40, 60.0)
    ag.render(r, a, cam).sum().backward()


def _sorted(m, r):
    h = r.load_scene(synth.uniform_scene(100, seed=1, precision="fp32"))
    r.render(h, synth.look_at((0, 0, -3), (0, 0, 0), 48, 40, 60.0), flags=m.MGS_FLAG_SORTED)


def _spatial(m, r):
    r.load_scene(np.zeros((5000, 24), np.float32), order=m.MGS_ORDER_SPATIAL)


@pytest.mark.parametrize("call", [_decode, _backward, _sorted, _spatial])
def test_next_call(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2603_11531_gb300 as m
    r = m.Renderer(0)
    ws = m.mgs_workspace_create(r.ctx)
    try:
        call(m, r)
        with pytest.raises(m.MGSError) as e:
            m.mgs_workspace_reserve(ws, 10 ** 11, 64, 64, 1024)
        assert e.value.status == m.MGS_ERR_OOM
        call(m, r)
        torch.cuda.synchronize()
    finally:
        m.mgs_workspace_destroy(ws)
        r.close()
