"""factor_tc names the sweeps whose updates run on the tensor cores: 0 none, 1 both, 2 the Omega sweep.

Read from the kernels of a factorization; and where a sweep is the same, so are its bits: S_k comes
from the Omega sweep alone, S_k^+ from both.
"""
import os
import sys

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _problem():
    from paper_2306_00094_gb300 import binding
    w = W.peridynamic_2d(N=48, k=3, nrhs=1)
    return binding, w, binding.Problem.from_workload(binding.Context(), w)


def _measure():
    from kernel_names import names
    binding, _, p = _problem()
    out = {}
    for tc in (0, 1, 2, "default"):
        p.set_options(binding.default_options(precision=1, **({} if tc == "default" else {"factor_tc": tc})))
        got = names(lambda: p.factor(2), "k_update")
        out[str(tc)] = sorted({"digits" if "k_update_d4" in n else "pipes" for n in got})
    return out


def test_the_sweeps_of_each_setting():
    from kernel_names import child
    assert child(__file__) == {"0": ["pipes"], "1": ["digits"], "2": ["digits", "pipes"], "default": ["digits"]}


def test_the_operators_of_each_setting():
    binding, w, p = _problem()
    got = {}
    for tc in (0, 1, 2):
        p.set_options(binding.default_options(precision=1, factor_tc=tc))
        p.factor(2)
        got[tc] = [(p.operator(k, 1, 1), p.operator(k, 2, 1)) for k in range(w.K)]
    for k in range(w.K):
        assert np.array_equal(got[1][k][0], got[2][k][0])
    assert any(not np.array_equal(got[0][k][0], got[2][k][0]) for k in range(w.K))
    assert any(not np.array_equal(got[1][k][1], got[2][k][1]) for k in range(w.K))
    p.close()


if __name__ == "__main__":
    sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
    import kernel_names
    kernel_names.main(_measure)
