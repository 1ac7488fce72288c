"""The kernels that calls of the library launch, read in a child process.

torch's profiler stays attached to the process that used it, and a server that captures graphs in
several threads can then wait forever; the tests' own process never loads it.
"""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def names(call, pattern):
    """Names of the launched kernels that contain pattern (in the child: call() is profiled)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):                      # the first session of a process records nothing
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        got = [e.name for e in prof.events() if pattern in e.name]
        if got:
            return got
    return []


def child(script, *args):
    """What the main part of a test file prints as JSON, run as a program of its own."""
    r = subprocess.run([sys.executable, script, *args], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT), text=True,
                       capture_output=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])
