"""Builds tests/kernel_calls.cpp against the library and loads it."""

import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def compile_to(path):
    from paper_1905_10602_gb300 import build as _build

    lib = _build.build()
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I" + os.path.join(_build.CUDA, "include"),
                    "-I" + _build.CSRC, os.path.join(HERE, "kernel_calls.cpp"), "-o", path, lib,
                    "-L" + os.path.join(_build.CUDA, "lib64"), "-lcudart",
                    "-Wl,-rpath," + os.path.dirname(lib)], check=True)
    return path


def load(path):
    return ctypes.CDLL(path)
