"""The predicted device bytes of a problem (what the server's admission counts) cover what it holds.

Held: the bytes in torch's allocator, which serves the context, between before the creation and after
the factorization.  The problems have many small parts, where the scratch of the sweeps (panel rows
padded to 128 per part) is most of it, and few larger ones; dense residual matrices, which the
prediction assumes.
"""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "1d_1000_parts_of_13": lambda: W.const_1d(N=8000, K=1000, nrhs=1, delta=2 / 8000),
    "1d_500_parts_of_130": lambda: W.const_1d(N=60000, K=500, nrhs=1, delta=10 / 60000),
    "pd_64_parts": lambda: W.peridynamic_2d(N=96, k=8, nrhs=1),
    "l2_9_parts": lambda: W.const_l2_2d(N=96, k=3, nrhs=1, delta=0.1),
}


def _predict(binding, w, mask):
    """nlf::predict_problem_bytes, which the C interface does not have."""
    f = binding.load()._ZN3nlf21predict_problem_bytesEPK11nlfeti_meshPK13nlfeti_kernelPK13nlfeti_decompi
    f.restype = C.c_size_t
    m, k = w.mesh, w.kernel
    a = [np.ascontiguousarray(x, t) for x, t in ((m.xy, np.float64), (m.elems, np.int32),
                                                 (m.node_is_dirichlet, np.int8), (m.elem_is_dirichlet, np.int8),
                                                 (w.labels, np.int32))]
    xy, el, nd, ed, lab = (x.ctypes.data for x in a)
    mesh = binding.Mesh(m.dim, a[2].size, xy, a[3].size, el, nd, ed)
    kern = binding.Kernel(int(k.type), float(k.delta), float(k.s), float(k.scale), 0)
    return f(C.byref(mesh), C.byref(kern), C.byref(binding.Decomp(int(w.K), lab)), C.c_int(mask))


@pytest.mark.parametrize("mask", [1, 2])
@pytest.mark.parametrize("name", list(CASES))
def test_prediction_covers_what_is_held(name, mask):
    from paper_2306_00094_gb300 import binding
    w = CASES[name]()
    ctx = binding.Context()
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    p = binding.Problem.from_workload(ctx, w)
    p.set_options(binding.default_options(precision=mask - 1, residual_format=1))
    p.factor(mask)
    held = torch.cuda.memory_allocated() - before
    predicted = _predict(binding, w, mask)
    p.close()
    assert held <= predicted, (held, predicted)
