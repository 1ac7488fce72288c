"""The reciprocals of the FP64 pivots are CUDA's rounded divisions.

Of a diagonal A^k, S_k^+ is the diagonal of the reciprocals of A^k's Gamma block, which no update
touches: bit for bit those of IEEE division, for mantissas of every kind and exponents far apart.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0, 40, 400])
def test_reciprocals_of_a_diagonal(spread):
    from paper_2306_00094_gb300 import binding
    w = W.const_1d(N=700, K=2, delta=100 / 700)
    p = binding.Problem.from_workload(binding.Context(), w)
    info = p.decomposition()
    rng = np.random.default_rng(spread)
    diags = []
    for k in range(2):
        n = int(info["n_k"][k])
        d = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-spread, spread + 1, n))
        d[-4:] = 1.0, np.nextafter(2.0, 0.0), np.nextafter(1.0, 2.0), 3.0
        diags.append(d)
        p.set_matrix(k, np.diag(d))
    p.factor(1)
    for k in range(2):
        g = int(info["n_gamma"][k])
        d = diags[k][-g:]
        assert np.array_equal(p.operator(k, 1), np.diag(d))
        assert np.array_equal(p.operator(k, 2), np.diag(1.0 / d))
    p.close()
