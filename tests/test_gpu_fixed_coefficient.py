"""The fixed-point operator's coefficient data at the edges of their number
format: face coefficients whose mantissa lies at either side of a power of two,
as they come from constant coefficients, over every degree and both bases."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import SIPG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg(cuda_device):
    import paper_1911_01492_gb300 as m
    return m


def relmax(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


def check_constant(dg, N, k, c, bc="dirichlet"):
    rng = np.random.default_rng(1000 * N + k)
    nd = N ** 3 * (k + 1) ** 3
    x = rng.uniform(-1, 1, nd)
    # a constant K scales the operator of K = 1
    ref = c * SIPG(N, k, bc=bc).apply(np.ones(nd), x)
    m = dg.Mesh(N, k)
    m.set_boundary(bc)
    m.set_coefficient(torch.full((nd,), c, dtype=torch.float64, device="cuda"))
    xd = torch.from_numpy(x).cuda()
    assert relmax(m.apply(xd).cpu().numpy(), ref) < 1e-12
    y = m.to_modal(m.apply_nodal(m.to_nodal(xd)))
    assert relmax(y.cpu().numpy(), ref) < 1e-12


@pytest.mark.parametrize("k", range(1, 9))
@pytest.mark.parametrize("N", [2, 4, 5])
def test_constant_coefficient(dg, N, k):
    for c in (2.0, 4.0, 5.0, 8.0, 10.0, 20.0, 100.0):
        check_constant(dg, N, k, c)


@pytest.mark.parametrize("k", range(1, 9))
def test_face_coefficient_just_below_a_power_of_two(dg, k):
    """K = 2 (1 - j 2^-53): h gamma lies j units in the last place, give or take
    the rounding of the means, below a power of two."""
    for j in (0, 1, 2, 4, 30, 1000, 2 ** 16, 2 ** 20, 2 ** 21 - 8, 2 ** 21 + 8, 2 ** 24):
        check_constant(dg, 2, k, 2.0 * (1.0 - j * 2.0 ** -53), bc="flow_x")


@pytest.mark.parametrize("N,k,c", [(8, 3, 2.0), (4, 3, 4.0), (8, 1, 8.0), (5, 2, 5.0),
                                   (5, 3, 10.0)])
def test_solves_with_a_constant_coefficient(dg, N, k, c):
    """FP64 CG in both bases, mixed and batched CG against the solution of
    K = 1, divided by c."""
    def mesh(v):
        m = dg.Mesh(N, k)
        m.set_coefficient(torch.full((m.n_dofs,), v, dtype=torch.float64, device="cuda"))
        return m

    m1, m = mesh(1.0), mesh(c)
    b = m.load_vector(torch.ones(m.n_dofs, dtype=torch.float64, device="cuda"))
    ref = m1.cg_solve(b, rtol=1e-12)[0] / c
    got = [m.cg_solve(b, rtol=1e-12)[0],
           m.cg_solve(b, rtol=1e-12, nodal=True)[0],
           m.cg_solve(b, rtol=1e-12, precond="kron")[0],
           m.cg_solve(b, rtol=1e-10, mode=dg.DG_CG_MIXED_IR)[0]]
    xb = [torch.zeros_like(b)]
    dg.cg_solve_batched([m], [b], xb, rtol=1e-12)
    # the residual's 1e-10 times the condition number, which is below 1e5 here
    for x in got + xb:
        assert ((x - ref).norm() / ref.norm()).item() < 1e-5
