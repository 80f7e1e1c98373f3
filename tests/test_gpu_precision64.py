"""The FP64 operator's error against extended precision (the weighted sum, its weights and its
transforms in long double) is no larger than that of the sums over the full spectrum with a weight
and an FP64 sum for every ordered pair. The bars are that operator's errors on the same inputs
(raw Q, relative L2 over the cells), one cell a call and in a batch."""
import numpy as np
import pytest

from paper_1211_0540_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")
L = LD(6)


@pytest.fixture(scope="module")
def bte():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1211_0540_gb300 import bte as b
    return b


def gauss_legendre(n):
    x = np.polynomial.legendre.leggauss(n)[0].astype(LD)

    def legendre(x):
        p0, p1 = np.ones_like(x), x.copy()
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / LD(k)
        return p1, n * (x * p1 - p0) / (x * x - 1)

    for _ in range(3):
        p, dp = legendre(x)
        x = x - p / dp
    dp = legendre(x)[1]
    return L * (x + 1) / 2, L / ((1 - x * x) * dp * dp)


def sinc(n, r, scale):
    z = scale * np.sqrt(np.arange(n).astype(LD))[:, None] * r[None, :]
    out = np.ones_like(z)
    out[z != 0] = np.sin(z[z != 0]) / z[z != 0]
    return out


def weights(N, lam, beta, w, r):
    """For beta = 1 the table I[p nq + q], else the function of (zeta', xi') that looks I up."""
    h, nq, hz = N // 2, 3 * (N - 1) ** 2 + 1, PI / (2 * L)
    A = sinc(3 * h * h + 1, r, hz if beta == 1.0 else hz * LD(beta)) * w
    J = (sinc(3 * h * h + 1, r, 2 * hz) * w).sum(1)
    if beta == 1.0:
        return (A @ sinc(nq, r, hz).T).reshape(-1), J
    # |2 m' - beta k'|^2 depends on (|m'|^2, m'.k', |k'|^2)
    table = {}

    def gain(k, m):
        key = (int(m @ m), int(m @ k), int(k @ k))
        if key not in table:
            z = hz * np.sqrt(LD(4 * key[0]) - 4 * LD(beta) * key[1] + LD(beta) ** 2 * key[2]) * r
            s = np.ones_like(z)
            s[z != 0] = np.sin(z[z != 0]) / z[z != 0]
            table[key] = (A[key[2]] * s).sum()
        return table[key]

    return gain, J


def operator(N, lam, f, beta=1.0):
    """Q (not projected) of the rows of f: sqrt(2/pi) (dz)^3 sum [I - J] fhat fhat, I and J by quadrature."""
    h, nq = N // 2, 3 * (N - 1) ** 2 + 1
    r, w = gauss_legendre(400 if beta == 1.0 else 96)  # r^(lam + 2) is smooth enough at 0 for 1e-17
    w = np.sqrt(2 / PI) * (PI / L) ** 3 * w * r ** LD(lam + 2)
    I, J = weights(N, lam, beta, w, r)
    a = np.arange(N) - h
    phase = 2 * PI / N * ((a[:, None] * a[None, :]) % N)
    e = np.empty((N, N), np.clongdouble)
    e.real, e.imag = np.cos(phase), -np.sin(phase)

    def transform(x, e):
        for ax in (1, 2, 3):
            x = np.moveaxis(np.tensordot(e, x, axes=([1], [ax])), 0, ax)
        return x

    fh = (2 * PI) ** LD(-1.5) * (2 * L / N) ** 3 * transform(f.reshape(-1, N, N, N).astype(np.clongdouble), e)
    Qh = np.zeros_like(fh)
    p = (a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2) * nq
    q = [(2 * (m - h) - a) ** 2 for m in range(N)]
    out = [slice(max(0, m - h), min(N, m + h)) for m in range(N)]        # zeta with xi_m's partner on the grid
    other = [slice(max(0, m - h) - m + h, min(N, m + h) - m + h) for m in range(N)]  # that partner
    for m1 in range(N):
        for m2 in range(N):
            for m3 in range(N):
                o = (out[m1], out[m2], out[m3])
                if beta == 1.0:
                    W = I[p[o] + q[m1][o[0], None, None] + q[m2][None, o[1], None] + q[m3][o[2]]]
                else:
                    m = np.array([m1, m2, m3]) - h
                    W = np.array([[[I(np.array([x, y, z]), m) for z in a[o[2]]] for y in a[o[1]]] for x in a[o[0]]])
                W = W - J[(m1 - h) ** 2 + (m2 - h) ** 2 + (m3 - h) ** 2]
                Qh[(slice(None),) + o] += (fh[:, other[m1], other[m2], other[m3]]
                                           * fh[:, m1, m2, m3][:, None, None, None] * W)
    return ((2 * PI) ** LD(-1.5) * (PI / L) ** 3 * transform(Qh, e.conj()).real).reshape(len(f), -1)


@pytest.mark.parametrize("N,lam,beta,cells,batch_bar,single_bar", [
    (8, 0.5, 1.0, 6, 2.3630e-15, 2.2726e-15), (8, 1.0, 1.0, 6, 1.8033e-15, 1.7094e-15),
    (12, 0.5, 1.0, 2, 3.5611e-15, 3.3319e-15), (12, 1.0, 1.0, 2, 2.8949e-15, 2.3209e-15),
    (8, 0.0, 0.8, 6, 1.741e-15, 1.655e-15), (8, 1.0, 0.8, 6, 1.809e-15, 1.725e-15)])
def test_fp64_error_is_that_of_the_full_spectrum(bte, N, lam, beta, cells, batch_bar, single_bar):
    if np.finfo(LD).eps > 2e-19:
        pytest.skip("no extended precision")
    f = inputs.precision_sweep_cells(N, 6.0, 40, seed=77)
    c = bte.Context(0)
    c.init_weights([(N, 6.0, lam, beta)])
    ft = torch.from_numpy(f).cuda()
    batch = c.collide(ft, mode=bte.FP64_PLAIN, raw=True)[:cells].cpu().numpy()
    single = np.concatenate([c.collide(ft[i:i + 1], mode=bte.FP64_PLAIN, raw=True).cpu().numpy()
                             for i in range(cells)])
    c.sync_status()
    c.close()
    E = operator(N, lam, f[:cells], beta)
    for Q, bar in ((batch, batch_bar), (single, single_bar)):
        assert float(np.sqrt(((Q - E) ** 2).sum() / (E ** 2).sum())) <= bar
