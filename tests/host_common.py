"""The library's host side without a GPU: a child process with tests/host/fake_cudart.c
preloaded in front of the CUDA runtime."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import textwrap

import pytest

from paper_2202_08612_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

PREAMBLE = """
import ctypes, sys
import numpy as np
from paper_2202_08612_gb300 import binding
L = binding.load()
F = ctypes.CDLL(FAKE)
F.fake_log.restype = ctypes.c_char_p
for f in (F.fake_used, F.fake_watched):
    f.restype = ctypes.c_longlong
for f, a in ((F.fake_total, [ctypes.c_longlong]), (F.fake_fail, [ctypes.c_char_p, ctypes.c_longlong]),
             (F.fake_mark, [ctypes.c_char_p] + [ctypes.c_longlong] * 3), (F.fake_watch, [ctypes.c_char_p]), (F.fake_fail_malloc, [ctypes.c_longlong]), (F.fake_is_live, [ctypes.c_void_p])):
    f.argtypes = a
class Dev:
    'A device array of doubles.'
    def __init__(self, *shape):
        self.p = ctypes.c_void_p()
        assert F.cudaMalloc(ctypes.byref(self.p), ctypes.c_size_t(8 * int(np.prod(shape)))) == 0
def launches():
    s = F.fake_log().decode().split()
    F.fake_clear()
    return s
def code(rc):
    return rc, L.mlcc3_last_error().decode()
def context(NO, NV, no, nv, NJ, precision=0, build=True, **params):
    c = ctypes.c_void_p()
    d = binding._Dims(NO, NV, no, nv, NJ, None)
    assert L.mlcc3_create(ctypes.byref(c), ctypes.byref(d), precision, None) == 0
    for k, v in params.items():
        assert L.mlcc3_set_param(c, k.encode(), v) == 0
    inputs = [Dev(NJ, NO + NV, NO + NV), Dev(NV, NO), Dev(NO + NV), Dev(no, nv, NO, NV), Dev(no, nv, NO, NV)]
    if build:
        assert L.mlcc3_build_integrals(c, *[x.p for x in inputs]) == 0, L.mlcc3_last_error()
    launches()
    return c, inputs
"""


def run_host(tmp_path_factory, script: str):
    """Run `script` after PREAMBLE in a child with the fake runtime; its output."""
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    if not os.path.exists(build.LIB) or build._stale():
        build.build()
    fake = os.path.join(tmp_path_factory.getbasetemp(), "libfakecudart.so")
    if not os.path.exists(fake):
        subprocess.run([cc, "-O1", "-w", "-shared", "-fPIC", "-o", fake, os.path.join(HERE, "host", "fake_cudart.c")],
                       check=True)
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, "-c", f"FAKE = {fake!r}\n" + PREAMBLE + textwrap.dedent(script)], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
