"""Assembly by pair lists: touching, cut by the ball, and wholly inside it.

A^k against the oracle's on meshes where each list is empty, short of a CTA's 16 pairs, or
dominant (delta from 1.5 to 7.3 cells), for the exponents with and without a power function
(s = 0.4, 0.5, 0.75), every ball, and irregular meshes.  Tolerance 1e-12 of the largest entry:
two FP64 codes for the same rule, whose entries sum a few thousand terms of that size at most.
The Dirichlet coupling is checked through a linear solution (in the kernel's null space on a
uniform mesh, so g linear and no load give u linear), to the solver's 1e-8.
"""
import numpy as np
import pytest

import workloads as W
from oracle import feti as ofeti

pytestmark = pytest.mark.gpu


def _make(kind, N, cells, s=0.5, ball=0, irregular=False, k=2):
    delta = cells / N
    kern = W.Kernel(kind, delta, s=s if kind == W.KERNEL_FRACTIONAL else 0.0, ball=ball)
    kern.scale = W.default_scale(kern, 2)
    m = W.collar_cells(delta, N)
    mesh = W.unstructured_mesh(N, m, seed=3) if irregular else W.make_mesh(2, N, m)
    labels = W.graph_labels(mesh, k * k, seed=3) if irregular else W.rect_labels(mesh, k, k)
    return W.Workload("lists", mesh, kern, labels, k * k, W.nodal_loads(mesh, kern.ncomp, 1, 1, "normal"), 1)


FR, PD, L2, LI = W.KERNEL_FRACTIONAL, W.KERNEL_PERIDYNAMIC, W.KERNEL_CONST_L2, W.KERNEL_CONST_LINF
CASES = {
    "frac_s05_1.5": dict(kind=FR, N=7, cells=1.5),
    "frac_s04_4": dict(kind=FR, N=13, cells=4.0, s=0.4),
    "frac_s075_7.3": dict(kind=FR, N=15, cells=7.3, s=0.75),
    "frac_s04_irregular": dict(kind=FR, N=14, cells=3.7, s=0.4, irregular=True),
    "frac_caps": dict(kind=FR, N=13, cells=5.0, s=0.4, ball=4),
    "frac_whole_elements": dict(kind=FR, N=13, cells=4.2, ball=2),
    "pd_1.5": dict(kind=PD, N=7, cells=1.5),
    "pd_5": dict(kind=PD, N=13, cells=5.0),
    "pd_irregular_barycenter": dict(kind=PD, N=14, cells=3.0, ball=1, irregular=True),
    "l2_6.4": dict(kind=L2, N=15, cells=6.4),
    "linf_3.3": dict(kind=LI, N=14, cells=3.3),
    "linf_irregular_4": dict(kind=LI, N=14, cells=4.0, irregular=True),
}


@pytest.fixture(scope="module")
def ctx():
    from paper_2306_00094_gb300 import binding
    return binding.Context()


@pytest.mark.parametrize("name", list(CASES))
def test_matrices(ctx, name):
    from paper_2306_00094_gb300 import binding
    w = _make(**CASES[name])
    p = binding.Problem.from_workload(ctx, w)
    o = ofeti.Feti(w.mesh, w.kernel, w.labels, w.K)
    for k in range(w.K):
        A = p.operator(k, 0)
        assert np.abs(A - o.A[k]).max() <= 1e-12 * np.abs(o.A[k]).max(), k
        assert np.array_equal(A, A.T)
    p.close()


@pytest.mark.parametrize("name", ["frac_s04_4", "frac_caps", "pd_5", "l2_6.4", "linf_3.3"])
def test_linear_solution(ctx, name):
    from paper_2306_00094_gb300 import binding
    w = _make(**CASES[name])
    nc = w.kernel.ncomp
    u = np.repeat(0.3 + 0.7 * w.mesh.xy[:, 0] - 0.4 * w.mesh.xy[:, 1], nc)
    if nc == 2:
        u[1::2] = -0.2 + 0.1 * w.mesh.xy[:, 0] + 0.5 * w.mesh.xy[:, 1]
    p = binding.Problem.from_workload(ctx, w)
    p.factor(1)
    got, _ = p.solve(np.zeros((u.size, 1)), 1, u.reshape(-1, 1))
    assert np.abs(got[:, 0] - u).max() <= 1e-8
    p.close()
