"""bench.py names the interface apply kernel that a tuned shape runs as, and finds its profile by it."""
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("kind,nrhs,rc,ctas,rows,kernel,columns", [
    (0, 16, 16, 2, 8, "apply_self", 16), (0, 64, 16, 2, 8, "apply_self", 16), (0, 16, 16, 2, 4, "apply_tma", 16),
    (0, 16, 16, 1, 8, "apply_tma", 16), (0, 16, 8, 2, 4, "apply_tma", 8), (0, 12, 8, 2, 4, "apply_self", 16),
    (0, 12, 8, 2, 8, "apply_tma", 8), (0, 5, 4, 2, 4, "apply_tma", 8), (0, 1, 1, 2, 4, "apply_tma", 1),
    (1, 16, -1, 1, 4, "apply_mma", None), (1, 17, 16, 2, 8, "apply_self", 16), (2, 12, 8, 2, 4, "apply_tma", 8),
    (2, 3, 2, 2, 4, "apply_tma", 4)])
def test_kernel_of_a_shape(kind, nrhs, rc, ctas, rows, kernel, columns):
    import bench
    got, text = bench.apply_kernel(dict(kind=kind, nrhs=nrhs, rc=rc, ctas_per_sm=ctas, rows_per_warp=rows))
    assert got == kernel and text.startswith(f"k_{kernel} ")
    assert columns is None or f"; {columns} columns per pass" in text
    assert os.path.exists(os.path.join(ROOT, "paper_2306_00094_gb300", "csrc", f"{got}.cuh"))
