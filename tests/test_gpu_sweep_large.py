"""The digit sweeps where a CTA works through several blocks and segments and parts finish apart.

Four parts of orders 1444, 2052, 2052 and 2916 (Omega blocks of 961 to 2209; none a multiple of 64) get
dense matrices.  Their 12 to 23 tiles a side make 660 blocks of 128 x 128, four or more for every CTA
of the FP32 update: buffers refilled, accumulators reused, the barriers' phases wrapped, the segment
lists rebuilt as parts finish.  For the FP64 update they are more than one chunk of 16 row blocks.

S_k and S_k^+ against numpy in FP64.  The matrices G G^T / n + 0.04 I have a condition number of about
101; an elimination errs by about sqrt(n) cond eps of the largest entry (the rounding errors of n
steps added as random signs).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
COND = 101.0


@pytest.fixture(scope="module")
def setup():
    from paper_2306_00094_gb300 import binding
    N, cells, cut = 86, 4, 35
    mesh = W.make_mesh(2, N, cells)
    kern = W.Kernel(W.KERNEL_CONST_LINF, cells / N)
    kern.scale = W.default_scale(kern, 2)
    mid = mesh.xy[mesh.elems].mean(axis=1) * N > cut
    labels = np.where(W.rect_labels(mesh, 1, 1) < 0, -1, 2 * mid[:, 1] + mid[:, 0]).astype(np.int32)
    w = W.Workload("unequal", mesh, kern, labels, 4, np.zeros((mesh.n_nodes, 1)), 1)
    p = binding.Problem.from_workload(binding.Context(), w)
    d = p.decomposition()
    assert not d["floating"].any()
    orders = [(int(n), int(g)) for n, g in zip(d["n_k"], d["n_gamma"])]
    assert sorted(n for n, _ in orders) == [1444, 2052, 2052, 2916] and len({n - g for n, g in orders}) == 3
    assert all(v % 64 for n, g in orders for v in (n, n - g))
    tiles = [-(-n // 128) for n, _ in orders]
    assert sum(t * (t + 1) // 2 for t in tiles) >= 4 * 152
    rng = np.random.default_rng(5)
    ref = []
    for k, (n, g) in enumerate(orders):
        b = rng.standard_normal((n, n))
        a = b @ b.T / n + 0.04 * np.eye(n)
        a = 0.5 * (a + a.T)
        p.set_matrix(k, a)
        no = n - g
        s = a[no:, no:] - a[no:, :no] @ np.linalg.solve(a[:no, :no], a[:no, no:])
        ref.append((n, s, np.linalg.inv(s)))
    yield binding, p, ref
    p.close()


@pytest.mark.parametrize("mask,factor_tc,eps", [(1, 1, 2.0 ** -53), (2, 1, 2.0 ** -24), (2, 2, 2.0 ** -24)])
def test_schur_and_inverse(setup, mask, factor_tc, eps):
    binding, p, ref = setup
    p.set_options(binding.default_options(precision=mask - 1, factor_tc=factor_tc))
    p.factor(mask)
    for k, (n, s, sp) in enumerate(ref):
        tol = np.sqrt(n) * COND * eps
        assert np.abs(p.operator(k, 1, mask - 1) - s).max() <= tol * np.abs(s).max(), k
        assert np.abs(p.operator(k, 2, mask - 1) - sp).max() <= tol * np.abs(sp).max(), k
