"""Runs host code of the library on the CPU against fake_cudart.cpp.

`run(code)` executes a snippet in a child process in which the library's CUDA
runtime calls go to the stand-in; the snippet finds `fake` (the stand-in's
controls), `W`, `B` (workloads, binding) and `np`, and puts what the test wants
to see into the dict `out`."""
import json
import os
import shutil
import subprocess
import sys
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")

PRELUDE = """
import ctypes, json, sys
sys.path.insert(0, {root!r})
fake = ctypes.CDLL({lib!r}, ctypes.RTLD_GLOBAL)
fake.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_double]
fake.fake_launch_cost.argtypes = [ctypes.c_double]
fake.fake_total.argtypes = [ctypes.c_size_t]
fake.fake_fail_launch.argtypes = [ctypes.c_long]
fake.fake_used.restype = fake.fake_peak.restype = ctypes.c_size_t
fake.fake_log.restype = ctypes.c_char_p
import numpy as np
from paper_2302_13907_gb300 import binding as B, workloads as W
out = {{}}
"""


def run(code):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    with tempfile.TemporaryDirectory() as d:
        lib = os.path.join(d, "libfake_cudart.so")
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, SRC, "-o", lib], check=True)
        full = PRELUDE.format(root=ROOT, lib=lib) + code + "\nprint('RESULT ' + json.dumps(out))\n"
        r = subprocess.run([sys.executable, "-c", full], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout[-2000:], r.stderr[-3000:])
    return json.loads([x for x in r.stdout.splitlines() if x.startswith("RESULT ")][-1][7:])
