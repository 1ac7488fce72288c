"""FP64 digit sweeps at the ends of the exponent range.

Scaling A^k by a power of two scales S_k by it and S_k^+ by its inverse, and every step of the sweep with
them: bit for bit while nothing leaves the normal range (2^1000).  By 2^-1010 the smaller products and
entries are subnormal (the conversion of the digit sums takes its other branch), which moves the rest
by 2^-64 of the largest at most: 1e-12 of the largest entry, the bound of the sweeps' other tests.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _spd(n, rng):
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    a = (q * np.geomspace(1.0, 100.0, n)) @ q.T
    return 0.5 * (a + a.T)


def test_scaled_matrices():
    from paper_2306_00094_gb300 import binding
    p = binding.Problem.from_workload(binding.Context(), W.const_1d(N=380, K=2, delta=40 / 380))
    rng = np.random.default_rng(11)
    mats = [_spd(int(n), rng) for n in p.decomposition()["n_k"]]
    got = {}
    for e in (0, 1000, -1010):
        for k in range(2):
            p.set_matrix(k, np.ldexp(mats[k], e))
        p.factor(1)
        got[e] = [(np.ldexp(p.operator(k, 1), -e), np.ldexp(p.operator(k, 2), e)) for k in range(2)]
    for k in range(2):
        for which in range(2):
            want = got[0][k][which]
            assert np.array_equal(got[1000][k][which], want)
            assert np.abs(got[-1010][k][which] - want).max() <= 1e-12 * np.abs(want).max()
    p.close()
