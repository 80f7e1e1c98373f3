"""A program that captures bte_collide in a graph of its own: the replays give the call's result, and the
context works on afterwards, through option changes that wait for its own work and drop its graphs."""
import pytest

from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_context_after_a_captured_collide():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte
    c = bte.Context(0)
    c.init_weights([(8, 6.0, 1.0)])
    f = torch.from_numpy(inputs.homogeneous_cells(8, 6.0, 40, seed=1)).cuda()
    Q, s, g = torch.empty_like(f), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    c.collide(f, Q, mode=bte.FP32, stream=s)
    c.sync_status(s)
    ref = Q.clone()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        g.capture_begin()
        c.collide(f, Q, mode=bte.FP32, stream=s)
        g.capture_end()
        Q.zero_()
        g.replay()
    c.sync_status(s)
    assert torch.equal(Q, ref)
    c.set_option("profile_mask", 1)  # waits for the context's work
    c.collide(f, Q, mode=bte.FP32, stream=s)
    c.sync_status(s)
    assert torch.equal(Q, ref)
    c.close()
