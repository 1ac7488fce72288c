"""Lane layouts of the single-domain CG's SpMV (1, 2, 4 or 8 columns wide, more than one block of 8).

A column gives the same bits whatever it is batched with, for every layout, on a size that is no
multiple of the 32 rows of a unit; and the widest and narrowest batches meet the oracle's solution
to the parity tolerance 1e-8.
"""
import numpy as np
import pytest

import workloads as W
from oracle import problem as oprob

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    from paper_2306_00094_gb300 import binding
    ctx = binding.Context()
    w = W.peridynamic_2d(N=19, k=2, nrhs=32)
    p = binding.Problem.from_workload(ctx, w)
    p.set_options(binding.default_options(tol=1e-12, max_it=20000))
    ref = oprob.Monolithic(w.mesh, w.kernel).solve(w.rhs, w.rhs_kind)
    single = {}
    yield w, p, ref, single
    p.close()


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 8, 9, 17, 32])
def test_columns_do_not_depend_on_the_batch(setup, nrhs):
    w, p, ref, single = setup
    u, _ = p.solve_cg(w.rhs[:, :nrhs], w.rhs_kind)
    err = oprob.rel_nodal_error(u, ref[:, :nrhs], w.mesh, 2)
    assert (err <= 1e-8).all()
    for c in {0, nrhs // 2, nrhs - 1}:
        if c not in single:
            single[c] = p.solve_cg(w.rhs[:, c:c + 1], w.rhs_kind)[0][:, 0]
        assert np.array_equal(single[c], u[:, c])
