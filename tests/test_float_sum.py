"""The sum of three floats by which FP32 partials are added (csrc/float_sum.cuh), compiled for the host:
against the exact sum and against FP64 additions one by one.

Tolerance, of the sum of magnitudes: (2 m 2^-24)^3 for a run of m <= 64 values, and per run three FP64
additions of 2^-53 and one into the total."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1408_1782_gb300", "csrc")

SOURCE = """
#include "float_sum.cuh"
extern "C" double merged_sum(const float* x, int n, int groups) {   // value u in group u mod groups
  qbe::FloatSum a[8];
  for (int u = 0; u < n; ++u) a[u % groups].add(x[u]);
  for (int g = 1; g < groups; ++g) a[0].merge(a[g].hi, a[g].mid, a[g].lo);
  return a[0].value();
}
extern "C" double run_sum(const float* x, int n) {
  double s = 0.0;
  for (int u0 = 0; u0 < n; u0 += qbe::FloatSum::kRun) {
    qbe::FloatSum a;
    for (int u = u0; u < n && u < u0 + qbe::FloatSum::kRun; ++u) a.add(x[u]);
    s += a.value();
  }
  return s;
}
"""


@pytest.fixture(scope="module")
def run_sum(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("float_sum")
    src, so = str(d / "s.cpp"), str(d / "libfloatsum.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for fn, n in ((lib.run_sum, 1), (lib.merged_sum, 2)):
        fn.restype = ctypes.c_double
        fn.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * n

    def call(x, groups=0):
        return lib.merged_sum(x.ctypes.data, len(x), groups) if groups else lib.run_sum(x.ctypes.data, len(x))

    return call


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 256, 1024, 4096])
@pytest.mark.parametrize("spread", [0, 12, 30])
def test_no_less_accurate_than_fp64(run_sum, n, spread):
    rng = np.random.default_rng(n + spread)
    worst = fp64 = 0.0
    for _ in range(50):
        x = (rng.standard_normal(n) * np.exp(rng.uniform(-spread, 0, n))).astype(np.float32)
        exact = math.fsum(x.astype(float).tolist())
        size = float(np.abs(x.astype(float)).sum())
        s = 0.0
        for v in x.astype(float):
            s += v
        worst = max(worst, abs(run_sum(x) - exact) / size)
        fp64 = max(fp64, abs(s - exact) / size)
    bound = (2 * min(n, 64) * 2.0 ** -24) ** 3 + math.ceil(n / 64) * 4 * 2.0 ** -53
    assert worst <= bound
    assert worst <= max(fp64, 2.0 ** -53)


@pytest.mark.parametrize("n", [1, 16, 100, 256])
@pytest.mark.parametrize("spread", [0, 12, 30])
def test_merged_sums_no_less_accurate_than_fp64(run_sum, n, spread):
    rng = np.random.default_rng(n + spread)
    for _ in range(50):
        x = (rng.standard_normal(n) * np.exp(rng.uniform(-spread, 0, n))).astype(np.float32)
        exact = math.fsum(x.astype(float).tolist())
        size = float(np.abs(x.astype(float)).sum())
        assert abs(run_sum(x, 8) - exact) <= ((2 * n * 2.0 ** -24) ** 3 + 3 * 2.0 ** -53) * size


def test_infinities_and_nan(run_sum):
    x = np.ones(70, np.float32)
    x[3] = np.inf
    assert run_sum(x) == math.inf
    x[66] = -np.inf
    assert math.isnan(run_sum(x))
    x[:] = 1.0
    x[69] = np.nan
    assert math.isnan(run_sum(x))
    x[69] = -np.inf
    assert run_sum(x, 8) == -math.inf
    x[3] = np.inf
    assert math.isnan(run_sum(x, 8))
