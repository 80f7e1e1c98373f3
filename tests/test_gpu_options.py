"""Options and tuning caches mean what they say: an explicit value of dft_split is what
runs, whatever the number of cells."""
import pytest

from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L = 6.0


@pytest.fixture(scope="module")
def bte():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte as b
    return b


@pytest.mark.parametrize("N,cells", [(8, 1024), (12, 256), (16, 160)])
def test_dft_split_four_is_four(bte, N, cells):
    """Enough cells that the default is one CTA per cell. Four CTAs add the moment sums of a cell in
    another order than one, so the projected Q of some cell differs in its last bits; the default
    and an explicit 1 are the same kernel."""
    c = bte.Context(0)
    c.init_weights([(N, L, 1.0)])
    f = torch.from_numpy(inputs.precision_sweep_cells(N, L, cells, seed=3)).cuda()
    assert c.get_option("dft_split") == 0
    Q = {}
    for split in (0, 1, 3, 4):
        c.set_option("dft_split", split)
        Q[split] = c.collide(f, mode=bte.FP32).clone()
    c.sync_status()
    c.close()
    assert torch.equal(Q[0], Q[1]) and torch.equal(Q[3], Q[4])
    assert not torch.equal(Q[4], Q[1])
    assert float((Q[4] - Q[1]).norm() / Q[1].norm()) <= 1e-10
