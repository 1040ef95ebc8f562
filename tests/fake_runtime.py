"""Runs a script against libifmm.so with tests/fake_cudart.cpp preloaded: the
library's host code on a machine without a GPU."""

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
import numpy as np
sys.path.insert(0, {root!r})
fake = ctypes.CDLL({lib!r})
fake.fake_refused.restype = ctypes.c_char_p
fake.fake_in_use.restype = ctypes.c_size_t
fake.fake_limit.argtypes = [ctypes.c_int, ctypes.c_size_t]
def launches(name):
    return fake.fake_launches(name.encode())
def refused():
    return fake.fake_refused().decode()
from paper_1905_10602_gb300 import ifmm
"""


def run(script, tmp_path, env=None):
    from paper_1905_10602_gb300 import build as _build

    _build.build()
    lib = str(tmp_path / "libfake_cudart.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I" + os.path.join(_build.CUDA, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", lib], check=True)
    out = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, lib=lib) + script], capture_output=True,
                         text=True, timeout=600, env=dict(os.environ, LD_PRELOAD=lib, **(env or {})))
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    return out.stdout
