"""Device memory that a context holds: scratch is shared by the cached instance layouts and
allocated by the calls that read it."""
import pytest

from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, MB = 6.0, 1 << 20


@pytest.fixture(scope="module")
def bte():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte as b
    return b


def held(since):
    torch.cuda.synchronize()
    return since - torch.cuda.mem_get_info()[0]


def test_the_parts_of_the_layouts_share_their_scratch(bte):
    """33 to 64 cells of N = 16 run 130 x 2 items in 4 parts of 8 KB: 8.5 MB, of which 16 layouts held as
    many. One context: 4.3 MB each of fhat and Qhat, one set of parts, small lists (2 MB granularity)."""
    c = bte.Context(0)
    c.init_weights([(16, L, 1.0)])
    f = torch.from_numpy(inputs.precision_sweep_cells(16, L, 64, seed=1)).cuda()
    Q = torch.empty_like(f)
    c.collide(f, Q, mode=bte.FP32)
    assert c.get_option("debug_conv_path") == 4
    free0 = torch.cuda.mem_get_info()[0]
    for n in range(48, 63):
        c.collide(f[:n], Q[:n], mode=bte.FP32)
    assert c.batch_count() == 16
    c.sync_status()
    assert held(free0) <= 16 * MB
    c.close()


def test_calls_that_read_no_parts_hold_none(bte):
    c = bte.Context(0)
    c.init_weights([(16, L, 1.0)])
    f = torch.from_numpy(inputs.precision_sweep_cells(16, L, 64, seed=1)).cuda()
    c.moments(f[:33])
    free0 = torch.cuda.mem_get_info()[0]
    for n in range(49, 65):
        c.moments(f[:n])
        c.project(f[:n])
    assert held(free0) <= 16 * MB
    c.close()


@pytest.mark.parametrize("mode,N,cells,arrays", [("FP32", 16, 1024, 2), ("FP64_PLAIN", 16, 512, 3)])
def test_transforms_hold_what_they_use(bte, mode, N, cells, arrays):
    """Beside the state, fhat and Qhat (one complex value a grid point), in FP64 one pass's result."""
    c = bte.Context(0)
    c.init_weights([(N, L, 1.0)])
    f = torch.from_numpy(inputs.precision_sweep_cells(N, L, 1, seed=1)).cuda()
    c.collide(f, mode=getattr(bte, mode))  # weight tables
    g = f.repeat(cells, 1)
    Q = torch.empty_like(g)
    free0 = torch.cuda.mem_get_info()[0]
    c.collide(g, Q, mode=getattr(bte, mode))
    c.sync_status()
    each = cells * N ** 3 * (8 if mode == "FP32" else 16)
    assert held(free0) <= arrays * each + 20 * MB
    c.close()
