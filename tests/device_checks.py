"""Builds and loads the test kernels of ``device_checks.cu`` (test infrastructure, no part of the library)."""
import ctypes as C
import os
import subprocess

from paper_2605_14929_b200 import build as libbuild

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "device_checks.cu")
LIB = os.path.join(HERE, "_build", "libdevice_checks.so")


def build(force: bool = False) -> str:
    deps = [SRC, os.path.join(libbuild.CSRC, "sop_device.cuh"), os.path.join(HERE, "..", "include", "sop.h")]
    if force or not os.path.exists(LIB) or any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps):
        os.makedirs(os.path.dirname(LIB), exist_ok=True)
        subprocess.check_call([libbuild.NVCC] + libbuild.FLAGS + [SRC, "-o", LIB])
    return LIB


def lib() -> C.CDLL:
    return C.CDLL(build())
