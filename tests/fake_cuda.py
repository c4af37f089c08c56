"""Run a piece of Python in a child process whose CUDA runtime is tests/fake_cudart.cpp: the library's host
code (plan creation, the engine's admission) without a GPU."""
import json
import os
import subprocess
import sys

from paper_2106_03583_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "fake_cudart.cpp")

PRELUDE = """
import ctypes, json, sys
sys.path[:0] = {paths!r}
import numpy as np
from paper_2106_03583_gb300 import inputs, snac
lib = snac.lib()
fake = ctypes.CDLL(None)
for f in ("fake_used", "fake_peak"):
    getattr(fake, f).restype = ctypes.c_size_t
for f in ("fake_log", "fake_unordered"):
    getattr(fake, f).restype = ctypes.c_char_p
fake.fake_limit.argtypes = [ctypes.c_size_t]
fake.fake_fail_after.argtypes = [ctypes.c_longlong]

def launches():
    return [l.split()[1] for l in fake.fake_log().decode().splitlines() if l.startswith("launch ")]

def create(blocks, precision="fp64", modes=(0, 0), shift=0.0):
    arr, keep = snac._marshal_blocks(blocks)
    o = snac._Options(snac._PREC[precision], 2, 2, 20, 40, 64, -1, 0.0, shift, *modes, 0, 0)
    h = ctypes.c_void_p()
    st = lib.snac_plan_create(ctypes.byref(h), len(blocks), arr, 2, ctypes.byref(o))
    return st, h

def workspace(h):
    n = ctypes.c_size_t()
    assert lib.snac_plan_workspace_bytes(h, ctypes.byref(n)) == 0
    return n.value
"""


def _library():
    build.build()
    out = os.path.join(build.ROOT, "_build", "libfakecudart.so")
    if not os.path.exists(out) or os.path.getmtime(out) < os.path.getmtime(SRC):
        inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
        tmp = f"{out}.{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{inc}", SRC, "-o", tmp], check=True)
        os.replace(tmp, out)
    return out


def run(body: str):
    """The value that ``body`` assigns to ``out`` (plain values)."""
    code = PRELUDE.format(paths=[build.ROOT, HERE]) + body + "\nprint('@' + json.dumps(out))\n"
    env = dict(os.environ, LD_PRELOAD=_library())
    res = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout + res.stderr
    return json.loads([l for l in res.stdout.splitlines() if l.startswith("@")][-1][1:])
