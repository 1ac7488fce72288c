"""The set-up refuses a problem whose interface the 32-bit indices of the Lambda-space operators cannot
tell, whichever kernels its iterations take: the rule at its limits, compiled from the header
(such a problem fits no GPU)."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00094_gb300", "csrc")
CUDA = next((d for d in ("/usr/local/cuda/include",) if os.path.isdir(d)), None)
M = 2 ** 31 - 1


@pytest.mark.skipif(shutil.which("g++") is None or CUDA is None, reason="needs g++ and the CUDA headers")
def test_limits(tmp_path):
    cases = [((0, 0, 0, 0), 1), ((M - 1, M, M, M), 1), ((M, 1, 1, 1), 0), ((1, M + 1, 1, 1), 0), ((1, 1, M + 1, 1), 0),
             ((1, 1, 1, M + 1), 0), ((1, 1, 1, 2 ** 33), 0)]
    calls = "".join(f'std::printf("%d\\n", (int)nlf::lambda_indices_fit({", ".join(f"{v}ll" for v in a)}));' for a, _ in cases)
    src = tmp_path / "limits.cpp"
    src.write_text('#include <cstdio>\n#include "internal.hpp"\nint main() {' + calls + "}\n")
    exe = tmp_path / "limits"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", CUDA, "-c", str(src), "-o", f"{exe}.o"], check=True)
    subprocess.run(["g++", f"{exe}.o", "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [want for _, want in cases]


def test_checked_before_any_narrowing():
    src = open(os.path.join(CSRC, "sweep.cu")).read()
    body = src[src.index("void setup_lambda(nlfeti_problem *p)"):]
    assert body.index("lambda_indices_fit") < body.index("lambda_clusters_ok") < re.search(r"k_narrow<<<", body).start()
