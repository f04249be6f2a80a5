"""The FP64 operator's block fixed-point arithmetic at the edges of its number
format: every degree, vectors over the whole exponent range, cells of very
different magnitude side by side, zeros, subnormal numbers and NaN.

Scaling x by a power of two only changes the cells' exponents, so the result
is the scaled one bit for bit as long as it is a normal number.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import SIPG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg(cuda_device):
    import paper_1911_01492_gb300 as m
    return m


def make(dg, N, k, seed, bc="dirichlet"):
    rng = np.random.default_rng(seed)
    K = np.exp(rng.standard_normal(N ** 3 * (k + 1) ** 3))
    m = dg.Mesh(N, k)
    m.set_boundary(bc)
    m.set_coefficient(torch.from_numpy(K).cuda())
    return m, K, rng.uniform(-1, 1, K.size)


def neighbours(N, c):
    crd = (c % N, c // N % N, c // (N * N))
    out = []
    for d, st in enumerate((1, N, N * N)):
        out += [c - st] * (crd[d] > 0) + [c + st] * (crd[d] < N - 1)
    return out


@pytest.mark.parametrize("k", range(1, 9))
def test_power_of_two_scaling_is_exact(dg, k):
    m, _, x = make(dg, 3, k, 70 + k)
    for f in (m.apply, m.apply_nodal):
        y = f(torch.from_numpy(x).cuda()).cpu().numpy()
        for e in (-960, -300, 300, 960):
            ye = f(torch.from_numpy(np.ldexp(x, e)).cuda()).cpu().numpy()
            assert np.array_equal(np.ldexp(ye, -e), y)


@pytest.mark.parametrize("k,N,bc", [(1, 4, "dirichlet"), (2, 3, "flow_x"), (3, 4, "flow_x"),
                                    (4, 3, "dirichlet"), (5, 2, "flow_x"), (8, 2, "dirichlet")])
def test_cells_of_different_magnitude(dg, k, N, bc):
    """Per cell, the error is bounded by the largest input of the cell and its
    face neighbours.  With s that input and R the largest row sum of |A| among
    those columns, FP64 rounding of the sum alone is 2^-53 R s; the bound
    allows 64 of those (three transforms each way and a line operator)."""
    m, K, x = make(dg, N, k, 90 + k, bc)
    nc, n3 = N ** 3, (k + 1) ** 3
    rng = np.random.default_rng(k)
    x = (x.reshape(nc, n3) * 10.0 ** rng.integers(-9, 10, (nc, 1)))
    x[0] = 0.0
    D = SIPG(N, k, bc=bc)
    A = D.assemble(K)
    ref = D.apply(K, x.reshape(-1)).reshape(nc, n3)
    R = np.asarray(abs(A).sum(axis=1)).reshape(nc, n3).max(axis=1)
    y = m.apply(torch.from_numpy(x.reshape(-1)).cuda()).cpu().numpy().reshape(nc, n3)
    big = np.abs(x).max(axis=1)
    for c in range(nc):
        s = max([big[c]] + [big[o] for o in neighbours(N, c)])
        assert np.abs(y[c] - ref[c]).max() <= 64 * 2.0 ** -53 * R[c] * s


def test_far_cells_do_not_matter(dg):
    N, k = 5, 3
    m, _, x = make(dg, N, k, 60)
    n3 = (k + 1) ** 3
    a = np.zeros((N ** 3, n3))
    a[0] = x[:n3] * 1e-30
    b = a.copy()
    b[-1] = x[-n3:] * 1e30
    ya = m.apply(torch.from_numpy(a.reshape(-1)).cuda()).cpu().numpy().reshape(-1, n3)
    yb = m.apply(torch.from_numpy(b.reshape(-1)).cuda()).cpu().numpy().reshape(-1, n3)
    near = [0] + neighbours(N, 0)
    assert np.array_equal(ya[near], yb[near]) and np.all(ya[near] != 0)
    assert not np.any(ya[[c for c in range(N ** 3) if c not in near]])


@pytest.mark.parametrize("k", [1, 2, 3, 5])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_nan_and_infinity_reach_the_cell_and_its_neighbours(dg, k, value):
    N = 3
    m, _, x = make(dg, N, k, 50 + k)
    c, n3 = 13, (k + 1) ** 3
    x[c * n3 + 1] = value
    for f in (m.apply, m.apply_nodal):
        y = f(torch.from_numpy(x).cuda()).cpu().numpy().reshape(-1, n3)
        bad = ~np.isfinite(y)
        hit = sorted([c] + neighbours(N, c))
        assert list(np.flatnonzero(bad.any(axis=1))) == hit
        assert bad[hit].all()


def test_zero_and_subnormal_vectors(dg):
    m, K, x = make(dg, 3, 3, 40)
    z = torch.zeros(m.n_dofs, dtype=torch.float64, device="cuda")
    assert not m.apply(z).any() and not m.apply_nodal(z).any()
    y = m.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    tiny = np.ldexp(x, -1060)      # integers below 2^14 times 2^-1074
    yt = m.apply(torch.from_numpy(tiny).cuda()).cpu().numpy()
    ref = m.apply(torch.from_numpy(np.ldexp(tiny, 1060)).cuda()).cpu().numpy()
    assert np.abs(np.ldexp(yt, 1060) - ref).max() <= 2.0 ** -14 + 1e-15 * np.abs(y).max()
