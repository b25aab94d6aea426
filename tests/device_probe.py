"""Builds and loads device_probe.cu: the library's internal functions by themselves."""
import ctypes
import os
import subprocess

from paper_2510_08536_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "device_probe.cu")
OUT = os.path.join(HERE, "_build", "libdevice_probe.so")


def load() -> ctypes.CDLL:
    deps = [SRC] + build.HEADERS
    if not os.path.exists(OUT) or any(os.path.getmtime(d) > os.path.getmtime(OUT) for d in deps):
        os.makedirs(os.path.dirname(OUT), exist_ok=True)
        cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", OUT, SRC, "-cudart", "static"]
        p = subprocess.run(cmd, capture_output=True, text=True)
        assert p.returncode == 0, p.stderr
    return ctypes.CDLL(OUT)
