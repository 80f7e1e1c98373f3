"""Every way in which the FP32 convolution's items run (pairs in lanes, whole, in halves, in more
parts), at the grid sizes that reach it by themselves or with the cut forced, with the way that ran
asserted, against the oracle (1e-5 of the loss term) and bit-identical on repeat. And the FP64 operator on
one cell (cell-major fhat, the lanes over the sum) at N = 16, 24, 32 (1e-12)."""
import numpy as np
import pytest

import oracle
from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, TOL32, TOL64 = 6.0, 1e-5, 1e-12
FEW, WHOLE, HALVES, PARTS = 1, 2, 3, 4


@pytest.fixture(scope="module")
def bte():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte as b
    return b


def error(N, lam, f, Q):
    Qm = oracle.collide(N, L, lam, f, part=1, project=False)
    return (np.linalg.norm(Q - oracle.collide(N, L, lam, f), axis=1) / np.linalg.norm(Qm, axis=1)).max()


# cut: blocks a warp (odd ranges among them), 0 = the batch's own plan on 152 SMs
@pytest.mark.parametrize("N,cells,lam,cut,impl,path", [
    (16, 1, 1.0, 0, 4, FEW), (8, 600, 1.0, 0, 4, WHOLE), (24, 40, 0.0, 0, 4, WHOLE),
    (8, 60, 1.0, 0, 4, HALVES), (12, 40, 0.0, 0, 4, HALVES), (16, 128, 1.0, 20, 4, HALVES), (16, 40, 1.0, 0, 4, PARTS),
    (8, 60, 1.0, 2, 4, PARTS), (12, 40, 0.0, 5, 4, PARTS), (16, 33, 1.0, 7, 4, PARTS), (24, 33, 1.0, 9, 4, PARTS),
    (32, 33, 0.0, 24, 4, PARTS), (16, 33, 1.0, 7, 5, PARTS), (24, 33, 1.0, 30, 5, PARTS)])
def test_items_of_every_kind(bte, N, cells, lam, cut, impl, path):
    f = inputs.precision_sweep_cells(N, L, cells, seed=20 + N)
    pick = [0, cells - 1] if N >= 24 else [0, cells // 2, cells - 1]
    c = bte.Context(0)
    c.init_weights([(N, L, lam)])
    c.set_option("conv_impl", impl)
    c.set_option("debug_conv_parts", cut)
    ft = torch.from_numpy(f).cuda()
    Q = c.collide(ft, mode=bte.FP32).clone()
    assert c.get_option("debug_conv_path") == path
    assert torch.equal(Q, c.collide(ft, mode=bte.FP32))
    c.sync_status()
    with pytest.raises(bte.BteError):
        c.set_option("debug_conv_path", 1)
    c.close()
    assert error(N, lam, f[pick], Q.cpu().numpy()[pick]) <= TOL32


def test_uneven_batch_in_parts(bte):
    """One list over the kinds of N = 12, 16, 24 and 32, every item cut."""
    grids = [(12, L, 0.0), (16, L, 1.0), (24, L, 1.0), (32, L, 0.0)]
    c = bte.Context(0)
    c.init_weights(grids)
    c.set_option("debug_conv_parts", 11)
    cells = [inputs.precision_sweep_cells(N, L, n, seed=N) for (N, _, _), n in zip(grids, (33, 20, 3, 2))]
    inst, off = [], 0
    for t, f in enumerate(cells):
        for _ in range(len(f)):
            inst.append((t, off))
            off += f.shape[1]
    flat = torch.from_numpy(np.concatenate([f.ravel() for f in cells])).cuda()
    Q = c.collide(flat, inst=inst, mode=bte.FP32)
    assert c.get_option("debug_conv_path") == PARTS
    c.sync_status()
    c.close()
    Q, k = Q.cpu().numpy(), 0
    for (N, _, lam), f in zip(grids, cells):
        got = np.stack([Q[o:o + f.shape[1]] for _, o in inst[k:k + len(f)]])
        k += len(f)
        sel = [0, len(f) - 1]
        assert error(N, lam, f[sel], got[sel]) <= TOL32, N


@pytest.mark.parametrize("N,lam", [(16, 1.0), (24, 0.0), (32, 1.0)])
def test_fp64_single_cell_matches_oracle(bte, N, lam):
    f = inputs.precision_sweep_cells(N, L, 1, seed=300 + N)
    c = bte.Context(0)
    c.init_weights([(N, L, lam)])
    Q = c.collide(torch.from_numpy(f).cuda(), mode=bte.FP64_PLAIN).cpu().numpy()
    c.sync_status()
    c.close()
    assert error(N, lam, f, Q) <= TOL64


@pytest.mark.parametrize("N,few", [(8, 56), (12, 22), (16, 11), (24, 9), (32, 10)])
def test_where_few_cells_end(bte, N, few):
    """The last batch with pairs in lanes and the first with cells in lanes, where a call takes as long
    either way (measured with the items cut by their plan); within the bar of one another."""
    f = torch.from_numpy(inputs.precision_sweep_cells(N, L, few + 1, seed=5)).cuda()
    c = bte.Context(0)
    c.init_weights([(N, L, 1.0)])
    Q = c.collide(f[:few], mode=bte.FP32)
    assert c.get_option("debug_conv_path") == FEW
    P = c.collide(f, mode=bte.FP32)
    assert c.get_option("debug_conv_path") != FEW
    c.sync_status()
    c.close()
    Qm = oracle.collide(N, L, 1.0, f[:1].cpu().numpy(), part=1, project=False)
    assert float((P[0] - Q[0]).norm()) <= 2 * TOL32 * np.linalg.norm(Qm)
