"""The kernels that calls of the library launch, read in a child process.

torch's profiler stays attached to the process that used it, and a server that captures graphs in
several threads can then wait forever; the tests' own process never loads it.
"""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _recorded(call):
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.name for e in prof.events()]


def names(call, pattern):
    """Names of the launched kernels that contain pattern (in the child: call() is profiled)."""
    for _ in range(3):                      # the first session of a process records nothing
        got = [n for n in _recorded(call) if pattern in n]
        if got:
            return got
    return []


def child(script):
    """What the main part of a test file prints as JSON, run as a program of its own; skips where the
    profiler records no kernel at all."""
    path = os.pathsep.join([ROOT, *filter(None, [os.environ.get("PYTHONPATH")])])
    r = subprocess.run([sys.executable, script], cwd=ROOT, env=dict(os.environ, PYTHONPATH=path), text=True,
                       capture_output=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    if out is None:
        pytest.skip("the profiler records no kernels here")
    return out


def main(measure):
    """The main part of a test file: prints measure() as JSON (null where nothing is recorded)."""
    import torch
    x = torch.ones(16, device="cuda")
    print(json.dumps(measure() if any(_recorded(lambda: x + 1) for _ in range(3)) else None))
