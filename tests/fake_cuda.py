"""Runs library calls against the stand-in for the CUDA runtime (fake_cudart.cpp)
in a child process, on machines without a GPU."""
import os
import shutil
import subprocess
import sys
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes, os, sys
sys.path.insert(0, {root!r})
from paper_cs_0404008_gb300 import gfpdot as g
L = g.load(auto_build=False)
F = ctypes.CDLL(os.environ["LD_PRELOAD"])
F.fake_events.restype = ctypes.c_char_p
F.fake_used.restype = F.fake_peak.restype = ctypes.c_size_t
F.fake_room.argtypes = [ctypes.c_size_t]
A, B, C = 1 << 40, 1 << 41, 1 << 42       # operands: addresses that nothing reads
CAPTURING = 0x100000                      # a stream being captured

def context():
    h = ctypes.c_void_p()
    assert L.gfp_context_create(0, ctypes.byref(h)) == 0
    F.fake_events()
    return h

def kernels():
    "Names of the kernels launched since the last call, in order."
    ev = F.fake_events().decode().split("\\n")
    return [e.split()[1] for e in ev if e.startswith("launch")]

def count(ks, name):
    return sum(k.startswith(name) for k in ks)

def block(ctx, p, m, k, nb, lda=None, a=A, stream=0):
    return L.gfp_matmul_block(ctx, p, m, k, nb, a, k if lda is None else lda, B, nb, C, nb, stream)
"""


def run(code: str):
    """Runs the statements with PRELUDE's names in a child process."""
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    with tempfile.TemporaryDirectory() as d:
        so = os.path.join(d, "libfakecudart.so")
        r = subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"),
                            os.path.join(ROOT, "tests", "fake_cudart.cpp"), "-o", so], capture_output=True, text=True)
        if r.returncode:
            pytest.skip("no host C++ compiler or CUDA headers: " + r.stderr[-300:])
        r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + code], capture_output=True, text=True,
                           env=dict(os.environ, LD_PRELOAD=so), timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
