"""The fixed-point operator with coefficients that vary by orders of magnitude
inside a cell, against extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from extended_reference import ExtendedReference, norm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg(cuda_device):
    import paper_1911_01492_gb300 as m
    return m


def apply(dg, N, k, K, x, nodal=False):
    m = dg.Mesh(N, k)
    m.set_coefficient(torch.from_numpy(np.reshape(K, -1).copy()).cuda())
    f = m.apply_nodal if nodal else m.apply
    return f(torch.from_numpy(np.reshape(x, -1).copy()).cuda()).cpu().numpy()


@pytest.mark.parametrize("k", range(1, 9))
@pytest.mark.parametrize("spread", [0.5, 1.0, 2.0, 4.0])
def test_smooth_vector_rough_coefficient(dg, k, spread):
    """x nearly constant, K = exp(spread N(0,1)) at every point: the terms cancel.
    The error stays below what a change of up to 2^-53 in every mode of x, its own
    rounding in FP64, does to A x."""
    N, n3 = 2 if k > 5 else 3, (k + 1) ** 3
    rng = np.random.default_rng(200 + k)
    K = np.exp(spread * rng.standard_normal(N ** 3 * n3))
    t = rng.uniform(-1, 1, (N ** 3, n3))
    x = 1e-4 * t
    x[:, 0] = 1.0
    R = ExtendedReference(N, k, K)
    unit = norm(R.apply(t * 2.0 ** -53))
    assert norm(apply(dg, N, k, K, x) - R.apply(x)) < unit
