"""The extended-precision reference against the oracle."""
import numpy as np
import pytest

from oracle import SIPG

from extended_reference import ExtendedReference, norm


@pytest.mark.parametrize("N,k", [(1, 2), (2, 1), (3, 3), (2, 4), (1, 8)])
def test_reference_matches_oracle(N, k):
    rng = np.random.default_rng(N + k)
    K = np.exp(rng.standard_normal(N ** 3 * (k + 1) ** 3))
    x = rng.uniform(-1, 1, K.size)
    R = ExtendedReference(N, k, K)
    assert norm(R.apply(x) - SIPG(N, k).apply(K, x)) < 1e-13 * norm(R.apply(x))
    assert norm(R.to_modal(R.to_nodal(x)) - x) < 1e-17 * norm(x)
