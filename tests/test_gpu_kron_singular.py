"""FP64 Kronecker blocks of a cell without an inverse: a breakdown, not a number."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 5])
@pytest.mark.parametrize("nodal", [False, True])
def test_singular_cell_block_breaks_down(cuda_device, k, nodal):
    """With K = 1e-200 the harmonic means of the interior faces underflow: the
    inner cell's block is singular."""
    import paper_1911_01492_gb300 as dg
    m = dg.Mesh(3, k)
    m.set_coefficient(torch.full((m.n_dofs,), 1e-200, dtype=torch.float64, device="cuda"))
    b = m.load_vector(torch.ones(m.n_dofs, dtype=torch.float64, device="cuda"))
    for _ in range(2):    # the factors are not taken for formed afterwards
        _, st = m.cg_solve(b, rtol=1e-8, maxit=20, precond="kron", nodal=nodal,
                           raise_on_error=False)
        assert st["status"] == dg.DG_ERR_BREAKDOWN
        # reported where the reciprocals are formed, before an iteration uses them
        with pytest.raises(dg.DGError, match="singular"):
            m.cg_solve(b, rtol=1e-8, maxit=20, precond="kron", nodal=nodal)
