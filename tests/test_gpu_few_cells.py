"""The FP32 convolution with pairs in lanes (few cells) against the oracle: one
cell, the largest batch that takes it (conv32_cells_limit) and the first that does
not, every grid size, and an uneven batch of all of them. Tolerance: the FP32
operator's 1e-5 of the loss term."""
import numpy as np
import pytest

import oracle
from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, TOL32 = 6.0, 1e-5


@pytest.fixture(scope="module")
def bte():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte as b
    return b


def error(N, lam, f, Q):
    Qo = oracle.collide(N, L, lam, f)
    Qm = oracle.collide(N, L, lam, f, part=1, project=False)
    return (np.linalg.norm(Q - Qo, axis=1) / np.linalg.norm(Qm, axis=1)).max()


@pytest.mark.parametrize("N,lam,cells", [(8, 1.0, (1, 56, 57)), (12, 0.0, (1, 30, 31)), (16, 1.0, (1, 14, 15)),
                                         (24, 1.0, (1, 9, 10)), (32, 0.0, (1, 9, 10))])
def test_few_cells_match_oracle(bte, N, lam, cells):
    c = bte.Context(0)
    c.init_weights([(N, L, lam)])
    f = inputs.precision_sweep_cells(N, L, max(cells), seed=70 + N)
    pick = [0, max(cells) - 1] if N >= 24 else range(max(cells))
    for n in cells:
        Q = c.collide(torch.from_numpy(f[:n]).cuda(), mode=bte.FP32).cpu().numpy()
        c.sync_status()
        sel = [i for i in pick if i < n]
        assert error(N, lam, f[sel], Q[sel]) <= TOL32, n
    c.close()


def test_few_instances_of_every_grid_match_oracle(bte):
    grids = [(8, L, 1.0), (12, L, 0.0), (16, L, 1.0), (24, L, 1.0)]
    c = bte.Context(0)
    c.init_weights(grids)
    counts = [10, 5, 3, 2]  # shares of the limits: 0.18 + 0.17 + 0.21 + 0.22
    cells = [inputs.precision_sweep_cells(N, L, n, seed=N) for (N, _, _), n in zip(grids, counts)]
    inst, off = [], 3
    for t, f in enumerate(cells):
        for _ in range(len(f)):
            inst.append((t, off))
            off += f.shape[1] + 1  # a gap after each instance
    flat = np.zeros(off)
    for (t, o), row in zip(inst, [r for f in cells for r in f]):
        flat[o:o + row.size] = row
    Q = c.collide(torch.from_numpy(flat).cuda(), inst=inst, mode=bte.FP32).cpu().numpy()
    c.sync_status()
    k = 0
    for (N, _, lam), f in zip(grids, cells):
        got = np.stack([Q[o:o + f.shape[1]] for _, o in inst[k:k + len(f)]])
        k += len(f)
        assert error(N, lam, f, got) <= TOL32, N
    c.close()
