"""A mesh whose geometry changes under its coefficient: refused vertices leave a
curved mesh as the unit cube with the coefficient it has."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import SIPG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg(cuda_device):
    import paper_1911_01492_gb300 as m
    return m


def lattice(N):
    t = np.linspace(0.0, 1.0, N + 1)
    return np.stack(np.meshgrid(t, t, t, indexing="ij"), axis=-1)


@pytest.mark.parametrize("k", range(1, 9))
def test_refused_vertices_leave_the_cube(dg, k):
    N = 3
    rng = np.random.default_rng(20 + k)
    nd = N ** 3 * (k + 1) ** 3
    K, x = np.exp(rng.standard_normal(nd)), rng.uniform(-1, 1, nd)
    X = lattice(N)
    X[1:-1, 1:-1, 1:-1] += rng.uniform(-0.05, 0.05, (N - 1, N - 1, N - 1, 3))
    m = dg.Mesh(N, k)
    m.set_vertices(X)
    m.set_coefficient(torch.from_numpy(K).cuda())
    with pytest.raises(dg.DGError):
        m.set_vertices(-X)                        # every cell inverted
    xd = torch.from_numpy(x).cuda()
    ref = SIPG(N, k).apply(K, x)
    y = m.apply(xd).cpu().numpy()
    assert np.abs(y - ref).max() < 1e-12 * np.abs(ref).max()
    y = m.to_modal(m.apply_nodal(m.to_nodal(xd))).cpu().numpy()
    assert np.abs(y - ref).max() < 1e-12 * np.abs(ref).max()
