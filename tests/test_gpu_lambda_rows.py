"""The PCG's Lambda-space steps past 16384 rows (vector accesses of 4, 2 and 1 columns).

Right-hand side counts that take each vector width, a remainder of a block and more columns than a
block: every column equals its solve alone bit for bit (the first and the last are compared), in
both precisions, and the solutions meet the oracle's single-domain solve to 1e-8, the bound of the
solver's other parity tests.  The problems: one and two components, both past 16384 Lambda rows, nodes with
up to nine copies.
"""
import numpy as np
import pytest

import workloads as W
from oracle import problem as oprob

pytestmark = pytest.mark.gpu

CASES = {
    "scalar": lambda: W.const_l2_2d(N=64, k=8, nrhs=65, delta=0.17),
    "vector": lambda: W.peridynamic_2d(N=54, k=9, nrhs=65, delta_cells=4),
}


@pytest.fixture(scope="module")
def built():
    from paper_2306_00094_gb300 import binding
    ctx = binding.Context()
    out = {}
    for name, mk in CASES.items():
        w = mk()
        p = binding.Problem.from_workload(ctx, w)
        p.factor(3)
        out[name] = (w, p, oprob.Monolithic(w.mesh, w.kernel).solve(w.rhs, w.rhs_kind), {})
    return out


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 6, 12, 64, 65])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_columns_and_parity(built, name, precision, nrhs):
    from paper_2306_00094_gb300 import binding
    w, p, ref, single = built[name]
    assert p.info()["n_lambda"] > 16384
    p.set_options(binding.default_options(precision=precision))
    u, _ = p.solve(w.rhs[:, :nrhs], w.rhs_kind)
    err = oprob.rel_nodal_error(u, ref[:, :nrhs], w.mesh, w.kernel.ncomp)
    assert (err <= 1e-8).all(), err
    for c in {0, nrhs - 1}:
        key = (precision, c)
        if key not in single:
            single[key] = p.solve(w.rhs[:, c:c + 1], w.rhs_kind)[0][:, 0]
        assert np.array_equal(single[key], u[:, c]), c
