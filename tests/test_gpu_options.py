"""Options and tuning caches mean what they say: an explicit value of dft_split is what
runs, whatever the number of cells, and a tuned entry is used for the batches it was tuned for."""
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


@pytest.mark.parametrize("N", [16, 24])
def test_tuning_many_cells_leaves_few_cells_alone(bte, N, tmp_path):
    """1 and 20 cells have the same slots but another convolution kernel: tuning one leaves the
    other as in an untuned context, to the last bit, and so does the saved cache."""
    f = torch.from_numpy(inputs.precision_sweep_cells(N, L, 20, seed=8)).cuda()
    ref = bte.Context(0)
    ref.init_weights([(N, L, 1.0)])
    one, many = ref.collide(f[:1], mode=bte.FP32), ref.collide(f, mode=bte.FP32)
    ref.sync_status()
    for tuned, other, expect in ((f, f[:1], one), (f[:1], f, many)):
        c = bte.Context(0)
        c.init_weights([(N, L, 1.0)])
        c.autotune(tuned, reps=1)
        assert torch.equal(c.collide(other, mode=bte.FP32), expect)
        c.sync_status()
        path = tmp_path / "tune.json"
        c.tune_save(path)
        d = bte.Context(0)
        d.init_weights([(N, L, 1.0)])
        assert d.tune_load(path) == 1
        assert torch.equal(d.collide(other, mode=bte.FP32), expect)
        assert torch.equal(d.collide(tuned, mode=bte.FP32), c.collide(tuned, mode=bte.FP32))
        d.sync_status()
        c.close()
        d.close()
    ref.close()
