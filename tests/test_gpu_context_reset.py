"""The calls that keep no state of the caller's work in a second context of the process: the one behind cudaDeviceReset."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, glob, os, sys
import numpy as np
from paper_2304_11267_b200 import binding as bd, build

lib = bd.load()
names = [l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l]
rt = ctypes.CDLL(names[0])

def check(rc):
    assert rc == 0, rc

def device(a):
    p = ctypes.c_void_p()
    check(rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)))
    check(rt.cudaMemcpy(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes), 1))
    return p

# blocks that ask for an SM to themselves, with one and with two blocks a group
shapes = [(120, 4096), (60, 3 * 8192)]
for turn in range(2):
    for groups, hw in shapes:
        x = np.random.default_rng(groups).standard_normal((1, groups, hw)).astype(np.float16)
        px, py = device(x), device(np.zeros_like(x))
        check(bd.sd_groupnorm_forward(px.value, 0, 0, py.value, 1, groups, hw, groups, 1e-5, bd.F16, 0))
        y = np.empty_like(x)
        check(rt.cudaMemcpy(y.ctypes.data_as(ctypes.c_void_p), py, ctypes.c_size_t(y.nbytes), 2))
        d = x.astype(np.float64)
        want = (d - d.mean(2, keepdims=True)) / np.sqrt(d.var(2, keepdims=True) + 1e-5)
        assert np.abs(y - want).max() < 4e-3, (turn, groups)   # (a rounding to binary16 of values up to 8)
    check(rt.cudaDeviceReset())
print("done")
"""


def test_groupnorm_in_a_second_context():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stderr[-2000:]
