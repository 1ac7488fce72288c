"""A chosen shape of the interface apply is the one that runs, and the default is the block that
holds all right-hand sides; read from the names of the kernels that an apply launches."""
import json
import re

import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prob():
    from paper_2306_00094_gb300 import binding
    w = W.const_l2_2d(N=32, k=4, nrhs=1, delta=0.1)
    p = binding.Problem.from_workload(binding.Context(), w)
    p.factor(3)
    p.set_options(binding.default_options(precision=1, batched=1, precond_fp16=1))
    yield binding, p
    p.close()


# operator kind: (operator of the apply, precision)
OPS = {0: (3, 1), 1: (5, 1), 2: (3, 0)}


def _ran(p, kind, nrhs):
    """(kernel, columns per pass, CTAs per SM, rows per warp) of one apply."""
    op, precision = OPS[kind]
    x = np.ones((p.info()["n_u"], nrhs))
    p.apply(op, precision, x)
    names = []
    for _ in range(3):                      # the first session of a process records nothing
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            p.apply(op, precision, x)
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "k_apply_" in e.name]
        if names:
            break
    assert len(names) == 1, names
    kernel, args = re.search(r"(k_apply_\w+)<([^>]*)>", names[0]).groups()
    args = [a.strip() for a in args.split(",")]
    if kernel == "k_apply_self":            # columns, stages, type
        return kernel, int(args[0]), 2, 8
    return kernel, int(args[1]), int(args[3]), int(args[6])


@pytest.mark.parametrize("kind,nrhs,rc,per_sm,rows", [
    (0, 12, 8, 2, 4), (0, 12, 8, 2, 8), (0, 12, 8, 1, 4), (0, 5, 4, 2, 4), (0, 3, 2, 2, 4), (0, 16, 16, 2, 4),
    (0, 16, 16, 2, 8), (0, 33, 16, 2, 4), (1, 12, 8, 2, 4), (1, 17, 16, 2, 4), (2, 5, 4, 2, 4), (2, 12, 8, 2, 4)])
def test_a_chosen_shape_runs(prob, kind, nrhs, rc, per_sm, rows):
    binding, p = prob
    p.set_apply_choice(kind, nrhs, rc, per_sm, rows)
    ran = _ran(p, kind, nrhs)
    p.set_apply_choice(kind, nrhs, 0)
    assert ran[1:] == (rc, per_sm, rows)


@pytest.mark.parametrize("kind,nrhs,block", [(0, 1, 1), (0, 3, 4), (0, 5, 8), (0, 9, 16), (0, 40, 16), (1, 12, 16), (2, 3, 4),
                                             (2, 5, 8), (2, 12, 8)])
def test_the_default_block(prob, kind, nrhs, block):
    binding, p = prob
    assert _ran(p, kind, nrhs)[1:] == (block, 2, 8 if block == 16 else 4)


@pytest.mark.parametrize("nrhs", [5, 12, 16])
def test_the_tuner_keeps_what_it_reports(prob, tmp_path, nrhs):
    binding, p = prob
    path = str(tmp_path / "tune.json")
    fresh = p.autotune(nrhs, path)
    lines = {e["kind"]: e for e in json.load(open(path))["entries"]}
    for again in (False, True):
        entries = p.autotune(nrhs, path) if again else fresh
        for e in entries:
            assert bool(e["from_cache"]) == again
            if e["rc"] == -1:
                continue
            ran = _ran(p, e["kind"], nrhs)[1:]
            if lines[e["kind"]]["rc"] == 0:                  # the default, wider than nrhs
                assert ran[0] > nrhs and ran[1] == 2 and e["rc"] <= nrhs
            else:
                assert (ran[0], ran[2]) == (e["rc"], e["rows_per_warp"])
                if e["kind"] < 2 and e["rc"] >= 8:           # a kernel of its own for one CTA per SM
                    assert ran[1] == e["ctas_per_sm"]
    for kind in (0, 1, 2):
        p.set_apply_choice(kind, nrhs, 0)


def test_entries_of_another_set_of_shapes_are_not_used(prob, tmp_path):
    binding, p = prob
    path = str(tmp_path / "tune.json")
    p.autotune(12, path)
    doc = json.load(open(path))
    assert all(len(e["key"]) == 16 for e in doc["entries"])
    old = "".join("0" if c != "0" else "1" for c in doc["entries"][0]["key"])
    text = open(path).read()
    for e in doc["entries"]:
        text = text.replace(e["key"], old)
    open(path, "w").write(text)
    assert all(e["from_cache"] == 0 for e in p.autotune(12, path))
    for kind in (0, 1, 2):
        p.set_apply_choice(kind, 12, 0)
