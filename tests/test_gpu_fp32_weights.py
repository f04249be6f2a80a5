"""FP32 application: the face weights carry one rounding."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_fp32_error_at_degree_two(cuda_device):
    """A value passes seven line stages (three transforms each way and the line
    operators) of about two roundings, rms 2^-24 / sqrt(3) each: 2.2 of 2^-24 relative
    to the result.  Face weights with five roundings of their own add as much again
    to the face terms, which dominate at this degree."""
    import paper_1911_01492_gb300 as dg
    N, k = 10, 2
    rng = np.random.default_rng(5)
    m = dg.Mesh(N, k)
    K = np.exp(0.3 * rng.standard_normal(m.n_dofs))
    m.set_coefficient(torch.from_numpy(K).cuda())
    x = torch.from_numpy(rng.uniform(-1, 1, m.n_dofs)).cuda().float()
    y, ref = m.apply(x).double(), m.apply(x.double())
    assert ((y - ref).norm() / ref.norm()).item() < 2.6 * 2.0 ** -24
