"""The PCG's Lambda-space work in thread-block clusters, one cluster per group of columns.

For right-hand side counts that fill, straddle and leave ragged the groups of 1, 2 and 4 columns,
in both precisions: every column equals its solve alone bit for bit, and the solutions meet the
oracle's single-domain solve to 1e-8.  The problems: no floating subdomain at all (no coarse
space), a small coarse space (FP64 coarse solve), one past 16 columns (FP32 parts) and one past 128
(rows shared between the CTAs), and parts whose nodes have up to nine copies.
"""
import numpy as np
import pytest

import workloads as W
from oracle import problem as oprob

pytestmark = pytest.mark.gpu

CASES = {
    "no_coarse": lambda: W.const_l2_2d(N=20, k=2, nrhs=33, delta=0.3),
    "coarse_small": lambda: W.const_l2_2d(N=24, k=4, nrhs=33, delta=2.0 / 24),
    "coarse_27": lambda: W.peridynamic_2d(N=35, k=5, nrhs=33),
    "coarse_147": lambda: W.peridynamic_2d(N=36, k=9, nrhs=33),
    "many_copies": lambda: W.fractional_2d(N=24, k=6, nrhs=33, delta=0.25),
    "one_d": lambda: W.const_1d(N=200, K=4, nrhs=33),
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


@pytest.mark.parametrize("nrhs", [1, 2, 3, 8, 16, 17, 33])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_columns_and_parity(built, name, precision, nrhs):
    from paper_2306_00094_gb300 import binding
    w, p, ref, single = built[name]
    p.set_options(binding.default_options(precision=precision))
    u, _ = p.solve(w.rhs[:, :nrhs], w.rhs_kind)
    err = oprob.rel_nodal_error(u, ref[:, :nrhs], w.mesh, w.kernel.ncomp)
    assert (err <= 1e-8).all(), err
    for c in {0, nrhs - 1}:
        key = (precision, c)
        if key not in single:
            single[key] = p.solve(w.rhs[:, c:c + 1], w.rhs_kind)[0][:, 0]
        assert np.array_equal(single[key], u[:, c]), c


@pytest.mark.parametrize("precond", [1, 2])
def test_tensor_core_input(built, precond):
    """The FP16 input of the tensor-core preconditioner written by the cluster kernel (odd count)."""
    from paper_2306_00094_gb300 import binding
    w, p, ref, _ = built["coarse_27"]
    p.set_options(binding.default_options(precision=1, precond_fp16=precond))
    u, _ = p.solve(w.rhs[:, :11], w.rhs_kind)
    assert (oprob.rel_nodal_error(u, ref[:, :11], w.mesh, 2) <= 1e-8).all()
    p.set_options(binding.default_options(precision=1))
