"""The warp-aligned tcgen05 instructions are executed by converged warps.

``.sync.aligned`` forms need every thread of the warp at the same instruction, and the compiler need
not bring a warp together after a branch that its lanes took differently.  So a ``__syncwarp()``
stands between any such branch and the next aligned instruction: before every deallocation of tensor
memory (one lane's copies and waits lie before it), and in every loop whose passes load accumulators
and then branch per lane.  Read from the sources: an unconverged warp at such an instruction is
undefined, so this is not found out by running it.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00094_gb300", "csrc")
LOADS = re.compile(r"\b(dg_ld4|dg_ld8|tc_ld16)\(")


def _lines():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read().split("\n")
        yield os.path.basename(path), [ln.split("//")[0] for ln in text]


def _uses(pattern):
    return [(name, i) for name, lines in _lines() for i, ln in enumerate(lines) if re.search(pattern, ln)]


def test_the_instructions_are_found():
    assert len(_uses(r"tcgen05\.dealloc")) >= 4 and len(_uses(LOADS.pattern)) >= 8


@pytest.mark.parametrize("name,line", _uses(r"tcgen05\.dealloc"))
def test_deallocation_by_a_converged_warp(name, line):
    lines = dict(_lines())[name]
    assert any("__syncwarp();" in ln for ln in lines[line - 4:line]), f"{name}:{line + 1}"


@pytest.mark.parametrize("name,line", [(n, i) for n, i in _uses(LOADS.pattern)
                                       if "__device__" not in dict(_lines())[n][i]])
def test_loads_in_a_loop_by_a_converged_warp(name, line):
    """The pass of the loop over accumulator columns (cc or c0) that holds the load: the warp is brought
    together before the load, or where its lanes part later in the pass."""
    lines = dict(_lines())[name]
    head = next(i for i in range(line, -1, -1) if re.search(r"for \(int (cc|c0) = 0;", lines[i]))
    assert line - head < 12, f"{name}:{line + 1}: no loop over accumulator columns"
    depth, body = 0, []
    for ln in lines[head:]:
        depth += ln.count("{") - ln.count("}")
        body.append(ln)
        if depth == 0:
            break
    if any("__syncwarp();" in ln for ln in body[:line - head]):
        return
    # blocks entered by some lanes alone end with the warp brought together
    parts = [i for i, ln in enumerate(body) if "if (__any_sync(" in ln or "} else {" in ln]
    assert parts, f"{name}:{line + 1}"
    for i in parts:
        close = next(k for k in range(i + 1, len(body)) if body[k].rstrip() == " " * (len(body[i]) - len(body[i].lstrip())) + "}")
        assert body[close - 1].strip() == "__syncwarp();", f"{name}:{head + close}"
