"""Runs Python code in a child process with tests/cuda_shim.c preloaded."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(tmp):
    so = os.path.join(str(tmp), "cuda_shim.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(ROOT, "tests", "cuda_shim.c"), "-ldl"],
                   check=True)
    return so


def run(so, tmp, code, limit=None, redzone=None):
    """(standard output, kernels launched, peak bytes) of `code`, which runs in the repository's root.
    With red zones the second is their log instead: overwritten ones, and the number checked."""
    log = os.path.join(str(tmp), "shim.log")
    if os.path.exists(log):
        os.remove(log)
    env = dict(os.environ, LD_PRELOAD=so, SPI_SHIM_LOG=log, PYTHONPATH=ROOT + os.pathsep + os.path.join(ROOT, "tests"))
    if limit is not None:
        env["SPI_SHIM_LIMIT"] = str(int(limit))
    if redzone is not None:
        env["SPI_SHIM_REDZONE"] = str(int(redzone))
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-500:], r.stderr[-2000:])
    lines = [l.split(None, 1) for l in open(log).read().splitlines()]
    return (r.stdout, [l[1] for l in lines if l[0] == "kernel"] if redzone is None else
            [" ".join(l) for l in lines if l[0] in ("overwritten", "zones")],
            max([int(l[1]) for l in lines if l[0] == "peak"], default=0))
