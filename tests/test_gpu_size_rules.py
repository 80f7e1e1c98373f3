"""Where a size or an alignment changes the kernel, both sides of the line:

- the FP32 operator around the cell counts from which a cell's transforms run as one
  CTA (ceil(N^2 / 32) warps a slot, 760 in all: 380, 152 and 95 slots at N = 8, 12, 16)
  and where the convolution's items are cut into many block ranges, against the oracle
  (1e-5 of the loss term; 1e-7 of max f after a Heun step) and bit-identical on repeat;
- surrogate gradients of batches that fill no tile of 64 or 128 rows, against the oracle
  at the bars of the full batches (bf16 operands: 2e-2 per block, 1e-2 on the loss);
- gradients into pages not yet mapped and into mapped ones: the same bytes;
- the surrogate's output at an address that 8 but not 16 divides: the same bytes.
"""
import ctypes

import numpy as np
import pytest

import oracle
from oracle import mlp as omlp
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


def surrogate(bte, N, H):
    c = bte.Context(0)
    c.init_weights([(N, L, 1.0)])
    c.mlp_init(0, H, seed=3)
    c.mlp_set_scales(10.0, 50.0)
    p = (np.random.default_rng(4).standard_normal(omlp.nparams(N ** 3, H)) * 0.05).astype(np.float32)
    c.mlp_set_params(p)
    return c, p


@pytest.mark.parametrize("N,ncells,lam", [(8, 352, 1.0), (8, 384, 1.0), (12, 128, 0.0), (12, 160, 0.0), (16, 40, 1.0),
                                          (16, 64, 1.0), (16, 95, 1.0), (16, 97, 1.0), (24, 33, 1.0), (32, 33, 0.0)])
def test_operator_at_the_edges_of_the_split_rules(bte, N, ncells, lam):
    f = inputs.precision_sweep_cells(N, L, ncells, seed=900 + N)
    pick = [0, ncells // 2, ncells - 1]
    c = bte.Context(0)
    c.init_weights([(N, L, lam)])
    ft = torch.from_numpy(f).cuda()
    Q = c.collide(ft, mode=bte.FP32).clone()
    assert torch.equal(Q, c.collide(ft, mode=bte.FP32))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        c.step(ft, 0.01, 1.0, mode=bte.FP32, stream=s)
    c.sync_status(s)
    c.close()
    Q, g = Q.cpu().numpy()[pick], f[pick]
    norm = np.linalg.norm(oracle.collide(N, L, lam, g, part=1, project=False), axis=1)
    assert (np.linalg.norm(Q - oracle.collide(N, L, lam, g), axis=1) / norm).max() <= TOL32
    if N <= 16:
        ref = oracle.rk2_homogeneous(N, L, lam, g, 0.01, 1.0)
        assert np.abs(ft.cpu().numpy()[pick] - ref).max() <= 1e-7 * np.abs(g).max()


@pytest.mark.parametrize("B", [1, 37, 100, 130])
def test_gradients_of_ragged_batches_match_oracle(bte, B):
    N, H = 8, 128
    M = N ** 3
    c, p = surrogate(bte, N, H)
    f = inputs.homogeneous_cells(N, L, B, seed=B)
    Q = oracle.collide(N, L, 1.0, f)
    loss_o, g_o = omlp.loss_and_grads(p.astype(np.float64), f, Q, (2 * L / N) ** 3, 10.0, 50.0, M, H)
    loss, g = c.mlp_grads(torch.from_numpy(f).cuda(), torch.from_numpy(Q).cuda())
    c.sync_status()
    c.close()
    assert abs(loss - loss_o) <= 1e-2 * loss_o
    o = 0
    for name, n in (("W1", H * M), ("b1", H), ("W2", H * H), ("b2", H), ("W3", M * H), ("b3", M)):
        rel = np.linalg.norm(g[o:o + n] - g_o[o:o + n]) / np.linalg.norm(g_o[o:o + n])
        assert rel <= 2e-2, (name, rel)
        o += n


def test_gradients_do_not_depend_on_the_host_buffer(bte):
    N, H, B = 16, 512, 64
    c, p = surrogate(bte, N, H)
    f = torch.from_numpy(inputs.homogeneous_cells(N, L, B, seed=5)).cuda()
    Q = c.collide(f, mode=bte.FP32)
    _, fresh = c.mlp_grads(f, Q)
    mapped = np.full(p.size + 1, 7.0, dtype=np.float32)[1:]  # pages written, start off a page and a 16-byte boundary
    loss = ctypes.c_double()
    assert c._lib.bte_mlp_grads(c._h, f.data_ptr(), Q.data_ptr(), B, ctypes.byref(loss),
                                mapped.ctypes.data_as(ctypes.c_void_p), None) == 0
    c.close()
    assert np.array_equal(fresh, mapped)


@pytest.mark.parametrize("N", [8, 12, 16])
def test_surrogate_output_does_not_depend_on_its_alignment(bte, N):
    ncells, M = 5, N ** 3
    c, _ = surrogate(bte, N, 128)
    f = torch.from_numpy(inputs.homogeneous_cells(N, L, ncells, seed=7)).cuda()
    even = c.mlp_infer(f).clone()
    odd = c.mlp_infer(f, torch.full((ncells * M + 1,), 3.0, dtype=torch.float64, device="cuda")[1:])
    c.sync_status()
    c.close()
    assert torch.equal(even.flatten(), odd.flatten())
