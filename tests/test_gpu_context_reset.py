"""The library after a reset of the device's context: a host code that resets the
device between runs builds new trees and gets the same J.  In a child process
without torch's CUDA state (a reset ends everything of the process that calls it)."""

import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C, sys
import numpy as np
import paper_2310_15235_gb300 as t2
import workloads
lib = t2.load_library()
rt = C.CDLL("libcudart.so.13")
case = workloads.random_case(9000, 60, nb=1, seed=701, clumped=True)
act = np.ascontiguousarray(case["active"], dtype=np.int64)
lo = (C.c_double * 3)(*case["box_lo"])
first = None
for turn in range(3):
    def up(x, dtype):
        x = np.ascontiguousarray(x, dtype=dtype)
        p = C.c_void_p()
        assert rt.cudaMalloc(C.byref(p), C.c_size_t(x.nbytes)) == 0
        assert rt.cudaMemcpy(p, x.ctypes.data_as(C.c_void_p), C.c_size_t(x.nbytes), 1) == 0
        return p
    n = len(case["pos"])
    a = [up(case["pos"], np.float64)] + [up(case[k], np.float32) for k in ("mass", "kappa", "lum", "h")]
    rows, out = up(act, np.int64), up(np.zeros(len(act)), np.float32)
    tree = C.c_void_p()
    rc = lib.trevr2_build(*a, n, 1, lo, float(case["box_size"]), case["bucket"], None, C.byref(tree))
    assert rc == 0, (turn, lib.trevr2_last_error())
    got = []
    for call in (lib.trevr2_J, lib.trevr2_J_noalloc):
        rc = call(tree, rows, len(act), 2, 0.75, None, 1, 0, out, None)
        assert rc == 0, (turn, lib.trevr2_last_error())
        J = np.zeros(len(act), np.float32)
        assert rt.cudaMemcpy(J.ctypes.data_as(C.c_void_p), out, C.c_size_t(J.nbytes), 2) == 0
        got.append(J)
    assert np.all(got[0] > 0)
    first = first or got
    assert all(np.array_equal(x, y) for x, y in zip(got, first)), turn
    assert lib.trevr2_free(tree) == 0
    assert t2.debug_pool_used() == 0
    assert rt.cudaDeviceReset() == 0
    free, total = C.c_size_t(), C.c_size_t()
    assert rt.cudaMemGetInfo(C.byref(free), C.byref(total)) == 0
    print("turn", turn, "free", free.value >> 20, "MiB")
print("done")
"""


def test_build_and_J_after_a_reset():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15235_gb300 import build_lib
    build_lib.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       timeout=240)
    assert r.returncode == 0 and r.stdout.rstrip().endswith("done"), r.stdout + r.stderr
    free = [int(line.split()[3]) for line in r.stdout.splitlines() if line.startswith("turn")]
    assert max(free) - min(free) <= 64, free  # a pool that outlived its context would show
