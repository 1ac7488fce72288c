"""FP32 sweeps by exact digit products on the tensor cores.

S_k and S_k^+ of caller-given SPD matrices (condition number about 100) whose orders and Omega
blocks straddle the 64-wide pivot blocks, the 64-row blocks and the 128-wide tiles, against numpy in
FP64.  Tolerance 1.3e-4 of the largest entry: an elimination of order n < 500 in FP32 errs by about
sqrt(n) cond 2^-24 (the rounding errors of n steps added as random signs).  Scaling rows and
columns by powers of two between 2^-12 and 2^12 scales S by them.  Matrices that are not positive
definite are reported.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1.3e-4


@pytest.fixture(scope="module")
def ctx():
    from paper_2306_00094_gb300 import binding
    return binding.Context()


def _spd(n, rng):
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    a = (q * np.geomspace(1.0, 100.0, n)) @ q.T
    return 0.5 * (a + a.T)


def _schur(a, no):
    return a[no:, no:] - a[no:, :no] @ np.linalg.solve(a[:no, :no], a[:no, no:])


def _problem(ctx, N, delta_cells):
    from paper_2306_00094_gb300 import binding
    w = W.const_1d(N=N, K=2, delta=delta_cells / N)
    p = binding.Problem.from_workload(ctx, w)
    p.set_options(binding.default_options(precision=1))
    d = p.decomposition()
    return p, [int(v) for v in d["n_k"]], [int(v) for v in d["n_gamma"]]


# orders n_k from about 30 to 460, Gamma blocks from 2 to 200
@pytest.mark.parametrize("N,cells", [(50, 2), (118, 10), (124, 3), (126, 2), (128, 2), (230, 30), (252, 3), (256, 64),
                                     (380, 5), (700, 100)])
def test_schur_and_inverse(ctx, N, cells):
    p, nk, ng = _problem(ctx, N, cells)
    rng = np.random.default_rng(N)
    mats = [_spd(n, rng) for n in nk]
    for k in range(2):
        p.set_matrix(k, mats[k])
    p.factor(2)
    for k in range(2):
        s = _schur(mats[k], nk[k] - ng[k])
        assert np.abs(p.operator(k, 1, 1) - s).max() <= TOL * np.abs(s).max()
        sp = np.linalg.inv(s)                      # both parts touch the Dirichlet collar: not floating
        assert np.abs(p.operator(k, 2, 1) - sp).max() <= TOL * np.abs(sp).max()
    p.close()


def test_power_of_two_scaling(ctx):
    p, nk, ng = _problem(ctx, 380, 40)
    rng = np.random.default_rng(7)
    a = [_spd(n, rng) for n in nk]
    d = [2.0 ** rng.integers(-12, 13, n) for n in nk]
    for k in range(2):
        p.set_matrix(k, a[k] * d[k][:, None] * d[k][None, :])
    p.factor(2)
    for k in range(2):
        no = nk[k] - ng[k]
        s = _schur(a[k], no)
        got = p.operator(k, 1, 1) / (d[k][no:, None] * d[k][None, no:])
        assert np.abs(got - s).max() <= TOL * np.abs(s).max()
    p.close()


@pytest.mark.parametrize("where", [0, 63, 64, 130])
def test_not_positive_definite(ctx, where):
    from paper_2306_00094_gb300 import binding
    p, nk, _ = _problem(ctx, 380, 40)
    rng = np.random.default_rng(3)
    a = _spd(nk[0], rng)
    bad = a.copy()
    bad[where, where] -= 500.0
    p.set_matrix(0, bad)
    with pytest.raises(binding.NlfetiError) as e:
        p.factor(2)
    assert e.value.status == binding.E_NOT_SPD
    p.set_matrix(0, a)
    p.factor(2)
    p.close()
