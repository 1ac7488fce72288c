"""factor_tc names the sweeps whose updates run on the tensor cores: 0 none, 1 both, 2 the Omega sweep.

Read from the kernels of a factorization; and where a sweep is the same, so are its bits: S_k comes
from the Omega sweep alone, S_k^+ from both.
"""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import workloads as W

pytestmark = pytest.mark.gpu


def _kernels(p, mask):
    for _ in range(3):                      # the first session of a process records nothing
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            p.factor(mask)
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "k_update" in e.name]
        if names:
            return {"digits" if "k_update_d4" in n else "pipes" for n in names}
    return set()


def test_the_sweeps_of_each_setting():
    from paper_2306_00094_gb300 import binding
    w = W.peridynamic_2d(N=48, k=3, nrhs=1)
    p = binding.Problem.from_workload(binding.Context(), w)
    got = {}
    for tc, kernels in ((0, {"pipes"}), (1, {"digits"}), (2, {"digits", "pipes"})):
        p.set_options(binding.default_options(precision=1, factor_tc=tc))
        assert _kernels(p, 2) == kernels, tc
        got[tc] = [(p.operator(k, 1, 1), p.operator(k, 2, 1)) for k in range(w.K)]
    for k in range(w.K):
        assert np.array_equal(got[1][k][0], got[2][k][0])
    assert any(not np.array_equal(got[0][k][0], got[2][k][0]) for k in range(w.K))
    assert any(not np.array_equal(got[1][k][1], got[2][k][1]) for k in range(w.K))
    p.close()


def test_the_default_is_both_sweeps():
    from paper_2306_00094_gb300 import binding
    p = binding.Problem.from_workload(binding.Context(), W.const_1d(N=200, K=4, nrhs=1))
    p.set_options(binding.default_options(precision=1))
    assert _kernels(p, 2) == {"digits"}
    p.close()
