"""Runs a piece of Python against the library's host code on a machine without a
GPU: in a process of its own, with tests/_fake_cudart.cpp in place of the CUDA
runtime.  The piece finds `lb` (the package), `fk` (the stand-in's controls),
`np` and `C` (ctypes); it fails by raising."""
import os
import subprocess
import sys
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = """
import ctypes as C, sys
sys.path.insert(0, {root!r})
fk = C.CDLL({fake!r}, mode=C.RTLD_GLOBAL)
for n in ("fk_errors", "fk_launch_name", "fk_launch_items"):
    getattr(fk, n).restype = C.c_char_p
fk.fk_device.restype = fk.fk_launch_dst.restype = C.c_void_p
fk.fk_device.argtypes = [C.c_size_t]
fk.fk_pin.argtypes = [C.c_void_p, C.c_size_t]
import numpy as np
import paper_0807_4471_gb300 as lb
lb.load()

def count(name):
    return fk.fk_count(name.encode())

def launches(part=""):
    return [k for k in range(fk.fk_launches()) if part in fk.fk_launch_name(k).decode()]

def step_items(k):
    "rows of (CTA, lattice, strip, first, end) of step launch k"
    return [tuple(map(int, r.split())) for r in fk.fk_launch_items(k).decode().splitlines()]

def status(call, *args):
    "the status a call raises, LB_OK without one"
    try:
        call(*args)
    except lb.LbError as e:
        return e.status
    return lb.LB_OK
"""
EPILOGUE = """
assert not fk.fk_errors(), fk.fk_errors().decode()
"""

_fake = None


def fake_library():
    """Path of the stand-in, compiled once per process."""
    global _fake
    if _fake is None:
        d = tempfile.mkdtemp(prefix="fake_cudart_")
        out = os.path.join(d, "libcudart.so.13")
        ver = os.path.join(d, "version")
        with open(ver, "w") as fh:
            fh.write("libcudart.so.13 { global: *; };\n")
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                        os.path.join(HERE, "_fake_cudart.cpp"), "-Wl,-soname,libcudart.so.13",
                        "-Wl,--version-script=" + ver, "-o", out], check=True)
        _fake = out
    return _fake


def run(code):
    from paper_0807_4471_gb300 import build
    build.build()
    text = PRELUDE.format(root=ROOT, fake=fake_library()) + code + EPILOGUE
    r = subprocess.run([sys.executable, "-c", text], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return r.stdout
