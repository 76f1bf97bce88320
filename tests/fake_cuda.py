"""Runs a script in a process whose CUDA runtime is fake_cudart.cpp (no GPU): the
library's host code with two devices, failing allocations and recorded launches.
The script finds the library as H, the launches since clear() as launches(), the
fake's calls on F, and prints what the test reads."""
import os
import subprocess
import sys
import textwrap

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BUILD = os.path.join(ROOT, "_build")

PRELUDE = """
import ctypes, sys
sys.path.insert(0, {root!r})
sys.path.insert(0, {root!r} + "/tests")
import numpy as np
import paper_2305_15116_gb300 as H
from paper_2305_15116_gb300 import _capi as C
from inputs import unit_square_mesh, unit_cube_kuhn_mesh
F = ctypes.CDLL({so!r})
F.fake_log.restype = ctypes.c_char_p
F.fake_uploads.restype = ctypes.c_long
F.fake_fail_malloc.argtypes = [ctypes.c_long, ctypes.c_size_t]
F.fake_fail_new.argtypes = [ctypes.c_long]
clear = F.fake_clear_log
X, Y = 1 << 40, 1 << 50  # vectors: addresses that nothing reads

def launches():
    out = []
    for l in F.fake_log().decode().splitlines():
        name, dev, grid, block, smem, cluster = l.split()
        out.append(dict(name=name, dev=int(dev), grid=int(grid), block=int(block), smem=int(smem), cluster=int(cluster)))
    return out

def apply(M, level, dtype=H.F64):
    return C.lib.hyteg_apply(M._h, level, dtype, X, Y, None)
"""


def _shared_object():
    src = os.path.join(ROOT, "tests", "fake_cudart.cpp")
    so = os.path.join(BUILD, "libfakecudart.so")
    if not os.path.exists(so) or os.path.getmtime(so) < os.path.getmtime(src):
        os.makedirs(BUILD, exist_ok=True)
        inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
        tmp = f"{so}.{os.getpid()}"
        subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + inc, src, "-o", tmp], check=True)
        os.replace(tmp, so)
    return so


def run(script):
    """The script's standard output, as lines."""
    so = _shared_object()
    code = PRELUDE.format(root=ROOT, so=so) + textwrap.dedent(script)
    env = dict(os.environ, LD_PRELOAD=so)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.splitlines()
