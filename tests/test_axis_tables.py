"""Host tables of an axis: values against libm's at twice the precision, and
the cost of the FP64 ones against the FP32 ones (no GPU)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "hv_passes.cuh"
using namespace rve;
template <typename R> static double fastest(int n) {
  std::vector<Cx<R>> t(n), d(n), a(n);
  double best = 1e9;
  for (int i = 0; i < 40; ++i) {
    const auto t0 = std::chrono::steady_clock::now();
    axis_tables<R>(n, t.data(), d.data(), a.data());
    const std::chrono::duration<double> s = std::chrono::steady_clock::now() - t0;
    if (s.count() < best) best = s.count();
  }
  return best;
}
int main(int, char** argv) {
  const int n = std::atoi(argv[1]);
  std::printf("%.9g %.9g\n", fastest<float>(n), fastest<double>(n));
  std::vector<double2> t(n), d(n), a(n);
  axis_tables<double>(n, t.data(), d.data(), a.data());
  for (int k = 0; k < n; ++k)
    std::printf("%.17g %.17g %.17g %.17g %.17g %.17g\n", t[k].x, t[k].y, d[k].x, d[k].y, a[k].x, a[k].y);
  return 0;
}
"""


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    from paper_2207_10657_gb300 import build
    lib = build.build()
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("tables")
    src, exe = d / "tables.cu", d / "tables"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(src), lib, "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True)

    def run(n):
        out = subprocess.run([str(exe), str(n)], capture_output=True, text=True, check=True).stdout.splitlines()
        return [float(x) for x in out[0].split()], np.array([[float(x) for x in l.split()] for l in out[1:]])
    return run


@pytest.mark.parametrize("n", [2, 6, 90, 512, 1000])
def test_fp64_tables(tables, n):
    _, got = tables(n)
    th = 2 * np.arccos(np.longdouble(-1)) * np.arange(n, dtype=np.longdouble) / n
    c, s, sh, ch = np.cos(th), np.sin(th), np.sin(th / 2), np.cos(th / 2)
    want = np.stack([c, -s, -2 * sh * sh, s, sh, ch], 1)
    want[0, 2:5] = 0
    want[n // 2, 5] = 0
    # one rounding to FP64, and the long double's own error (2^-63 of 1 at
    # most a few times over)
    assert np.all(np.abs(got - want) <= 0.5 * np.spacing(np.abs(want.astype(np.float64))) + 2.0 ** -61)
    assert got[0, 2] == got[0, 3] == got[0, 4] == 0 and got[n // 2, 5] == 0


def test_fp64_tables_cost_no_more_calls(tables):
    """Two libm calls an entry in either precision: the FP64 tables took twice
    the FP32 ones' time with four."""
    (f32, f64), _ = tables(1000)
    assert f64 <= 1.5 * f32, (f32, f64)
