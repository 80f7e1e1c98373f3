"""bte_mlp_infer on a stream that is being captured is refused, as it was when it synchronised: a graph
would keep activations that a larger batch frees. The capture and the context stay usable."""
import pytest

from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_infer_is_refused_under_capture():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte
    c = bte.Context(0)
    c.init_weights([(8, 6.0, 1.0)])
    c.mlp_init(0, 128, seed=1)
    f = torch.from_numpy(inputs.homogeneous_cells(8, 6.0, 5, seed=1)).cuda()
    Q = torch.empty_like(f)
    ref = c.mlp_infer(f).clone()  # the activations of this batch exist
    x = torch.zeros(4, device="cuda")
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        g.capture_begin()
        x.add_(1)
        with pytest.raises(bte.BteError):
            c.mlp_infer(f, Q, stream=s)
        g.capture_end()
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 4.0
    c.mlp_infer(f, Q, stream=s)
    c.sync_status(s)
    assert torch.equal(Q, ref)
    c.close()
