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


def lines_through(n, p):
    hot = np.zeros((n, n, n), bool)
    hot[p[0], p[1], :] = hot[p[0], :, p[2]] = hot[:, p[1], p[2]] = True
    return hot


def tolerance(n):
    """FP64 rounds each of the terms, the largest of which (the penalty, sigma = 2 n^2
    times a face value) cancel: four of those roundings."""
    return 4 * 2 * n * n * 2.0 ** -53


@pytest.mark.parametrize("k,p", [(1, (0, 1, 0)), (2, (1, 1, 1)), (2, (0, 2, 0)), (3, (1, 2, 1)),
                                 (4, (2, 2, 2)), (5, (0, 2, 1)), (6, (3, 0, 3)), (7, (1, 6, 2)),
                                 (8, (4, 4, 0))])
@pytest.mark.parametrize("s", [1.0, 1e4, 1e9, 1e18])
def test_point_basis_keeps_every_point(dg, k, p, s):
    """Q A Q^T couples a point to its three lines only.  With one large K or one large
    x, the points of the cell off its lines keep FP64's relative precision, and so
    do those of a neighbour off the line that meets them."""
    N, n, c = 3, k + 1, 13
    rng = np.random.default_rng(40 + k)
    shape = (N ** 3, n, n, n)
    off = ~lines_through(n, p)
    x = rng.uniform(-1, 1, shape)
    one = np.ones(shape)

    K = one.copy()
    K[c][p] = s
    for zero in (False, True):        # x zero on the lines through the point: they add nothing
        z = x.copy()
        if zero:
            z[c][~off] = 0.0
        y = apply(dg, N, k, K, z, nodal=True).reshape(shape)
        ref = ExtendedReference(N, k, K).apply_nodal(z).reshape(shape)
        assert norm((y - ref)[c][off]) < tolerance(n) * norm(ref[c][off])

    z = x.copy()
    z[c][p] = s
    y = apply(dg, N, k, one, z, nodal=True).reshape(shape)
    ref = ExtendedReference(N, k, one).apply_nodal(z).reshape(shape)
    assert norm((y - ref)[c][off]) < tolerance(n) * norm(ref[c][off])
    beside = np.ones((n, n, n), bool)
    beside[p[0], p[1], :] = False     # the x-line that continues the point's
    assert norm((y - ref)[c + 1][beside]) < tolerance(n) * norm(ref[c + 1][beside])


@pytest.mark.parametrize("k", [1, 2, 3, 5])
def test_point_basis_diagonal_with_contrast(dg, k):
    """The Jacobi diagonal of the point basis: one step of CG from a unit residual at a
    point off the hot lines is 1 / diagonal there."""
    N, n, c, p = 3, k + 1, 13, (0, 0, 0)
    shape = (N ** 3, n, n, n)
    K = np.ones(shape)
    K[c][p] = 1e18
    R = ExtendedReference(N, k, K)
    at = np.zeros(shape)
    at[c][-1, -1, -1] = 1.0
    diag = float(R.apply_nodal(at).reshape(shape)[c][-1, -1, -1])
    m = dg.Mesh(N, k)
    m.set_coefficient(torch.from_numpy(K.reshape(-1)).cuda())
    b = m.to_modal(torch.from_numpy(at.reshape(-1)).cuda())
    x, st = m.cg_solve(b, rtol=1e-14, maxit=1, precond="jacobi", nodal=True,
                       raise_on_error=False)
    x = m.to_nodal(x).cpu().numpy().reshape(shape)[c][-1, -1, -1]
    assert st["iterations"] == 1 and abs(x * diag - 1) < 1e-10


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6])
def test_solves_from_a_point_source(dg, k):
    """CG vectors that start at one point: cells on both paths, their inner products
    added up."""
    N, n = 4 if k < 4 else 3, k + 1
    rng = np.random.default_rng(k)
    K = np.exp(0.3 * rng.standard_normal(N ** 3 * n ** 3))
    m = dg.Mesh(N, k)
    m.set_coefficient(torch.from_numpy(K).cuda())
    e = torch.zeros(m.n_dofs, dtype=torch.float64, device="cuda")
    e[5 * n ** 3 + 1] = 1.0
    b = m.to_modal(e)
    ref = m.cg_solve(b, rtol=1e-12)[0]
    xb = [torch.zeros_like(b)]
    dg.cg_solve_batched([m], [b], xb, rtol=1e-11, nodal=True)
    for x in (m.cg_solve(b, rtol=1e-12, nodal=True)[0],
              m.cg_solve(b, rtol=1e-12, nodal=True, precond="jacobi")[0],
              m.cg_solve(b, rtol=1e-12, nodal=True, precond="kron")[0], xb[0]):
        assert ((x - ref).norm() / ref.norm()).item() < 1e-6


@pytest.mark.parametrize("k", range(1, 9))
@pytest.mark.parametrize("spread", [0.5, 1.0, 2.0, 4.0])
def test_smooth_vector_rough_coefficient_on_a_vertex_mesh(dg, k, spread):
    """test_smooth_vector_rough_coefficient on the multilinear kernels, whose mesh is
    here the unit cube's own lattice."""
    N, n3 = 2 if k > 5 else 3, (k + 1) ** 3
    rng = np.random.default_rng(200 + k)
    K = np.exp(spread * rng.standard_normal(N ** 3 * n3))
    t = rng.uniform(-1, 1, (N ** 3, n3))
    x = 1e-4 * t
    x[:, 0] = 1.0
    R = ExtendedReference(N, k, K)
    unit = norm(R.apply(t * 2.0 ** -53))
    s = np.linspace(0.0, 1.0, N + 1)
    m = dg.Mesh(N, k)
    m.set_vertices(np.stack(np.meshgrid(s, s, s, indexing="ij"), axis=-1))
    m.set_coefficient(torch.from_numpy(K).cuda())
    y = m.apply(torch.from_numpy(x.reshape(-1)).cuda()).cpu().numpy()
    assert norm(y - R.apply(x)) < unit
