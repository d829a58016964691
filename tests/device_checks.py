"""Builds tests/csrc/device_checks.cu against the library and loads it."""
import ctypes
import os
import subprocess
import tempfile

from paper_1508_03452_gb300 import build as B

_lib = None


def load() -> ctypes.CDLL:
    global _lib
    if _lib is None:
        B.build()
        out = os.path.join(tempfile.mkdtemp(prefix="device_checks_"), "libdevice_checks.so")
        src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "csrc", "device_checks.cu")
        cmd = [B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", src, "-o", out, B.LIB_PATH, "-Xlinker",
               "-rpath=" + os.path.dirname(B.LIB_PATH), "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(r.stderr)
        _lib = ctypes.CDLL(out)
    return _lib
