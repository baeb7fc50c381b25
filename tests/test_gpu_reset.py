"""A program that resets its device's context (cudaDeviceReset: its own context, nothing else) can build and run new
plans afterwards: the library keeps no record of what it has set in the old context.  In a process of its own,
without torch's allocations."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import ctypes
import numpy as np
from paper_1504_02897_gb300 import ddi

lib = ddi.load()
rt = ctypes.CDLL("libcudart.so.13")  # the one the library is linked with


def potential(n, precision, **kw):
    # 384 fine cells along y and the columns' FP64 kernels: both take more than 48 KB of shared memory
    desc = ddi.make_desc(3, n, (-1.0,) * 3, (2.0,) * 3, (0.6, 0.0, 0.8), precision=precision, **kw)
    plan = ctypes.c_void_p()
    st = lib.ddi_plan_create(ctypes.byref(plan), ctypes.byref(desc), None)
    assert st == 0, lib.ddi_last_error()
    rho = np.random.default_rng(1).random(n[::-1]).astype(np.float64 if precision == 0 else np.float32)
    phi = np.empty_like(rho)
    st = lib.ddi_apply_host(plan, rho.ctypes.data_as(ctypes.c_void_p), phi.ctypes.data_as(ctypes.c_void_p), None)
    assert st == 0, lib.ddi_last_error()
    assert lib.ddi_plan_destroy(plan) == 0
    return phi


def all_potentials():
    return [potential((16, 192, 8), p, nr=32, ntheta=16, nphi=16) for p in (0, 1)]


first = all_potentials()
assert rt.cudaDeviceReset() == 0
second = all_potentials()
assert all(np.array_equal(a, b) for a, b in zip(first, second))
print("same")
"""


def test_plans_after_a_context_reset():
    from paper_1504_02897_gb300 import build
    build.build()
    run = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert run.returncode == 0 and run.stdout.split()[-1:] == ["same"], run.stdout + run.stderr
