"""Every device buffer that a problem or an operator pool holds is used after it was allocated and
uploaded: a buffer that nothing reads counts against the device memory for nothing."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00094_gb300", "csrc")


def _members():
    names = []
    for ln in open(os.path.join(CSRC, "internal.hpp")):
        m = re.match(r"\s*nlf::DevMem ([^;]*);", ln.split("//")[0])
        if m:
            names += [n.strip() for n in m.group(1).split(",")]
    return names


def test_members_are_found():
    assert {"d_Z", "d_l_g_val32", "scratch", "Sh"} <= set(_members())


@pytest.mark.parametrize("name", _members())
def test_used_after_it_is_filled(name):
    fills = re.compile(rf"\b{name}\.alloc\(|\b(upload|f32_copy)\(c, \w+(->|\.){name}\b")
    use = re.compile(rf"(->|\.){name}\b")
    lines = [ln.split("//")[0] for f in glob.glob(os.path.join(CSRC, "*.c*")) for ln in open(f)]
    assert any(use.search(ln) and not fills.search(ln) for ln in lines), name
