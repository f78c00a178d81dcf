"""Runs a piece of Python against the library on host_cudart.cpp (no device, no
kernel runs) in a process of its own.  The code finds `rt` (the runtime's
controls), `lib` (the library, with its argument types), `bern`, `np`, `ctypes`,
`launched()` (the kernels noted since the last call), `allocated()` (the sizes allocated since
then) and `empty(n)` (an address
of n zeroed bytes)."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = """
import ctypes, sys
import numpy as np
sys.path.insert(0, %(root)r)
rt = ctypes.CDLL(%(so)r, mode=ctypes.RTLD_GLOBAL)
rt.host_set_alloc_limit.argtypes = [ctypes.c_size_t]
rt.host_fail_copies_after.argtypes = [ctypes.c_long]
rt.host_launched.restype = rt.host_allocated.restype = ctypes.c_char_p
from paper_2211_14438_gb300 import bern
lib = bern.load()
_keep = []
def launched():
    names = rt.host_launched().decode().split()
    rt.host_clear()
    return names
def allocated():
    return [int(x) for x in rt.host_allocated().decode().split()]
def empty(n):
    _keep.append(np.zeros(max(1, n), np.uint8))
    return ctypes.c_void_p(_keep[-1].ctypes.data)
def context():
    h = ctypes.c_void_p()
    assert lib.bern_create(ctypes.byref(h), 0, None) == 0
    return h
"""


def run(tmp_path, code):
    so = str(tmp_path / "libhost_cudart.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", so,
                    os.path.join(HERE, "host_cudart.cpp")], check=True)
    p = subprocess.run([sys.executable, "-c",
                        PRELUDE % dict(root=os.path.dirname(HERE), so=so) + code],
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stdout + p.stderr
    return p.stdout
