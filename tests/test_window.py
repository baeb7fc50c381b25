"""The split algorithm's window factor e^{-|k|^2/k0^2} - 1 (csrc/window.cuh) as a mode's thread forms it, compiled
for the host, against FP64.  Two roundings are left, of the heads' FMA and of the tails' addition: half an ulp
each, so the relative error stays below 2^-23 (1 + 2^-10) for the last places that the tails lose."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_02897_gb300", "csrc")
SOURCE = """
#include "window.cuh"
using namespace ddi;
template <typename T> static void run(const double* x, const double* y, const double* z, long n, T* out) {
  for (long i = 0; i < n; ++i)
    out[i] = window_join(window_line(window_entry<T>(x[i]), window_entry<T>(y[i])), window_entry<T>(z[i]));
}
extern "C" void window_f32(const double* x, const double* y, const double* z, long n, float* o) { run(x, y, z, n, o); }
extern "C" void window_f64(const double* x, const double* y, const double* z, long n, double* o) { run(x, y, z, n, o); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("window")
    (d / "w.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I" + CSRC, str(d / "w.cpp"),
                    "-o", str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


@pytest.mark.parametrize("precision,bound", [(1, 2.0 ** -23 * (1 + 2.0 ** -10)), (0, 2.0 ** -51)])
@pytest.mark.parametrize("nf,length,k0", [((512, 512, 512), (48.0, 48.0, 48.0), 0.2), ((64, 32, 48), (12.0, 7.0, 10.0), 1.3),
                                          ((128, 96, 256), (9.0, 9.0, 30.0), 40.0), ((64, 64, 64), (1e-3, 1e-3, 2e-3), 9.6e3)])
def test_window_factor(lib, nf, length, k0, precision, bound):
    rng = np.random.default_rng(3)
    near = [rng.integers(-min(n // 2, 24), min(n // 2, 24), 200000) for n in nf]  # around k = 0
    wide = [rng.integers(-(n // 2), n // 2, 200000) for n in nf]                  # any mode
    l = [np.concatenate(v) for v in zip(near, wide)]
    x2 = [((np.pi / h) * m / k0) ** 2 for h, m in zip(length, l)]  # 2 pi l / (2 len): the padded box's modes
    tab = [np.ascontiguousarray(np.expm1(-v)) for v in x2]
    want = np.expm1(-(x2[0].astype(np.longdouble) + x2[1] + x2[2]))
    out = np.empty(l[0].size, np.float64 if precision == 0 else np.float32)
    f = lib.window_f64 if precision == 0 else lib.window_f32
    f(*(v.ctypes.data_as(ctypes.c_void_p) for v in tab), ctypes.c_long(out.size), out.ctypes.data_as(ctypes.c_void_p))
    on = want != 0
    assert np.all(out[~on] == 0)
    err = np.abs(out[on] - want[on]) / -want[on]
    print(f"largest {float(err.max()):.3g}, r.m.s. {float(np.sqrt(np.mean(err ** 2))):.3g}")
    assert err.max() <= bound
