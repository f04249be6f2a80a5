"""The coefficient gradient of smooth fields, whose own gradients are small
against their values: a product of two of them is small twice."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import SIPG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg(cuda_device):
    import paper_1911_01492_gb300 as m
    return m


def derivative_row_sum(n):
    """Largest absolute row or column sum of the scaled collocation derivative."""
    t, w = np.polynomial.legendre.leggauss(n)
    x, sw = (t + 1) / 2, np.sqrt(w / 2)
    lam = np.array([1 / np.prod(x[a] - np.delete(x, a)) for a in range(n)])
    D = np.zeros((n, n))
    for a in range(n):
        for b in range(n):
            if a != b:
                D[a, b] = lam[b] / lam[a] / (x[a] - x[b])
        D[a, a] = -D[a].sum()
    D = np.abs(sw[:, None] * D / sw[None, :])
    return max(D.sum(axis=0).max(), D.sum(axis=1).max())


@pytest.mark.parametrize("k", range(1, 9))
def test_gradient_of_nearly_constant_fields(dg, k):
    """u and v are 1 plus delta times a random field: their point derivatives
    come from differences of values near 1, so in FP64 each carries a relative
    error of about 2^-53 R / delta, R the row sum of the derivative; the bound
    allows 8 of those."""
    N, n, delta = 3, k + 1, 2.0 ** -20
    rng = np.random.default_rng(30 + k)
    nd = N ** 3 * n ** 3
    K = np.exp(rng.standard_normal(nd))
    X = np.round(rng.uniform(-1, 1, (2, N ** 3, n ** 3)) * 2 ** 20) / 2 ** 20 * delta
    X[:, :, 0] = 1.0
    u, v = X.reshape(2, -1)
    ref = SIPG(N, k).coeff_grad(K, u, v).reshape(N ** 3, -1)[13]  # the cell without a boundary
    m = dg.Mesh(N, k)
    m.set_coefficient(torch.from_numpy(K).cuda())
    g = m.coeff_grad(torch.from_numpy(u.copy()).cuda(), torch.from_numpy(v.copy()).cuda())
    g = g.cpu().numpy().reshape(N ** 3, -1)[13]
    err = np.linalg.norm(g - ref) / np.linalg.norm(ref)
    assert err < 8 * 2.0 ** -53 * derivative_row_sum(n) / delta
