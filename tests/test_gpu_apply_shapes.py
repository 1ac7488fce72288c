"""A chosen shape of the interface apply is the one that runs, and the default is the block that
holds all right-hand sides; read from the names of the kernels that an apply launches."""
import json
import os
import re
import sys
import tempfile

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# (operator kind, right-hand sides, columns per pass, CTAs per SM, rows per warp)
CHOSEN = [(0, 12, 8, 2, 4), (0, 12, 8, 2, 8), (0, 12, 8, 1, 4), (0, 5, 4, 2, 4), (0, 3, 2, 2, 4), (0, 16, 16, 2, 4),
          (0, 16, 16, 2, 8), (0, 33, 16, 2, 4), (1, 12, 8, 2, 4), (1, 17, 16, 2, 4), (2, 5, 4, 2, 4), (2, 12, 8, 2, 4)]
# (operator kind, right-hand sides, the default's columns per pass)
DEFAULT = [(0, 1, 1), (0, 3, 4), (0, 5, 8), (0, 9, 16), (0, 40, 16), (1, 12, 16), (2, 3, 4), (2, 5, 8), (2, 12, 8)]
TUNED = [5, 12, 16]


def _problem():
    from paper_2306_00094_gb300 import binding
    w = W.const_l2_2d(N=32, k=4, nrhs=1, delta=0.1)
    p = binding.Problem.from_workload(binding.Context(), w)
    p.factor(3)
    p.set_options(binding.default_options(precision=1, batched=1, precond_fp16=1))
    return p


def _ran(p, kind, nrhs):
    """(columns per pass, CTAs per SM, rows per warp) of one apply."""
    from kernel_names import names
    op, precision = {0: (3, 1), 1: (5, 1), 2: (3, 0)}[kind]
    got = names(lambda: p.apply(op, precision, np.ones((p.info()["n_u"], nrhs))), "k_apply_")
    assert len(got) == 1, got
    kernel, args = re.search(r"(k_apply_\w+)<([^>]*)>", got[0]).groups()
    args = [a.strip() for a in args.split(",")]
    return (int(args[0]), 2, 8) if kernel == "k_apply_self" else (int(args[1]), int(args[3]), int(args[6]))


def _measure():
    p = _problem()
    out = {"chosen": [], "default": [], "tuned": []}
    for kind, nrhs, *shape in CHOSEN:
        p.set_apply_choice(kind, nrhs, *shape)
        out["chosen"].append(_ran(p, kind, nrhs))
        p.set_apply_choice(kind, nrhs, 0)
    out["default"] = [_ran(p, kind, nrhs) for kind, nrhs, _ in DEFAULT]
    for nrhs in TUNED:
        with tempfile.TemporaryDirectory() as d:
            path = os.path.join(d, "tune.json")
            for again in (0, 1):
                entries = p.autotune(nrhs, path)
                lines = {e["kind"]: e["rc"] for e in json.load(open(path))["entries"]}
                out["tuned"] += [dict(e, again=again, cached_rc=lines[e["kind"]],
                                      ran=None if e["rc"] == -1 else _ran(p, e["kind"], nrhs)) for e in entries]
        for kind in (0, 1, 2):
            p.set_apply_choice(kind, nrhs, 0)
    return out


@pytest.fixture(scope="module")
def ran():
    from kernel_names import child
    return child(__file__)


@pytest.mark.parametrize("i", range(len(CHOSEN)), ids=lambda i: "-".join(map(str, CHOSEN[i])))
def test_a_chosen_shape_runs(ran, i):
    assert ran["chosen"][i] == list(CHOSEN[i][2:])


@pytest.mark.parametrize("i", range(len(DEFAULT)), ids=lambda i: "-".join(map(str, DEFAULT[i])))
def test_the_default_block(ran, i):
    block = DEFAULT[i][2]
    assert ran["default"][i] == [block, 2, 8 if block == 16 else 4]


def test_the_tuner_keeps_what_it_reports(ran):
    assert len(ran["tuned"]) == 2 * 3 * len(TUNED)
    for e in ran["tuned"]:
        assert e["from_cache"] == e["again"]
        if e["rc"] == -1:
            continue
        columns, per_sm, rows = e["ran"]
        if e["cached_rc"] == 0:                              # the default, wider than the count
            assert columns > e["nrhs"] >= e["rc"] and per_sm == 2
        else:
            assert (columns, rows) == (e["rc"], e["rows_per_warp"])
            if e["kind"] < 2 and e["rc"] >= 8:               # a kernel of its own for one CTA per SM
                assert per_sm == e["ctas_per_sm"]


def test_entries_of_another_set_of_shapes_are_not_used(tmp_path):
    p = _problem()
    path = str(tmp_path / "tune.json")
    p.autotune(12, path)
    text = open(path).read()
    for e in json.loads(text)["entries"]:
        text = text.replace(e["key"], "".join("0" if c != "0" else "1" for c in e["key"]))
    open(path, "w").write(text)
    assert all(e["from_cache"] == 0 for e in p.autotune(12, path))
    p.close()


if __name__ == "__main__":
    sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
    import kernel_names
    kernel_names.main(_measure)
