"""The FP32 operator's error against 64 bits (relative L2 over the batch, the FP64 operator as the
reference: its own error is 1e-14) is no larger than that of the sums over the full spectrum with
TwoSum merges every 16 blocks, in which the roundings of a mode and its mirror average. The bars are
that operator's errors on the same inputs, measured before the sums were taken over half of the modes."""
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


# one call of `cells` cells, or `calls` calls of one (the convolution with pairs in lanes)
@pytest.mark.parametrize("N,lam,cells,calls,bar", [
    (8, 1.0, 1, 24, 4.6169e-7), (8, 1.0, 96, 1, 4.1669e-7), (8, 1.0, 600, 1, 4.2602e-7),
    (12, 0.0, 1, 24, 4.4302e-7), (12, 0.0, 40, 1, 4.6774e-7), (12, 0.0, 320, 1, 5.1025e-7),
    (12, 1.0, 40, 1, 5.4729e-7), (16, 1.0, 1, 24, 7.6861e-7), (16, 1.0, 40, 1, 7.4133e-7),
    (16, 1.0, 600, 1, 7.2136e-7), (16, 0.0, 40, 1, 6.1783e-7), (24, 1.0, 8, 1, 1.0078e-6),
    (24, 1.0, 40, 1, 7.2938e-7), (24, 0.0, 40, 1, 6.2199e-7), (32, 0.0, 8, 1, 6.8471e-7),
    (32, 0.0, 40, 1, 7.3763e-7), (32, 1.0, 40, 1, 8.6997e-7)])
def test_error_is_that_of_the_full_spectrum(bte, N, lam, cells, calls, bar):
    c = bte.Context(0)
    c.init_weights([(N, L, lam)])
    f = torch.from_numpy(inputs.precision_sweep_cells(N, L, cells * calls, seed=500 + N)).cuda()
    E = c.collide(f, mode=bte.FP64_PLAIN)
    Q = torch.empty_like(f)
    for i in range(calls):
        c.collide(f[i * cells:(i + 1) * cells], Q[i * cells:(i + 1) * cells], mode=bte.FP32)
    c.sync_status()
    c.close()
    assert float((Q - E).norm() / E.norm()) <= bar
