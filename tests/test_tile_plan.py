"""Tiles of the generic passes, planned on the host (no GPU): a program
compiled against the sources and linked with the library prints them."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <utility>
#include "hv_passes.cuh"
using namespace rve;
static void reverse(AxisPlan& p) {
  for (int a = 0, b = p.ns - 1; a < b; ++a, --b) std::swap(p.r[a], p.r[b]);
  finish_plan(p);
}
template <typename R> static void plan(GridDesc g, int wave, bool rev) {
  SpecWork<R> w;
  plan_tiles<R>(g, w, wave);
  if (rev) {  // a schedule that the batched solver's tuner may pick
    reverse(w.px);
    reverse(w.py);
    reverse(w.pz);
  }
  const GenericTiles<R> t(g, w.qx, w.lty, w.ltz, w.px, w.py, w.pz);
  std::printf("%d %d %d %d %d %d %zu %zu %zu\n", w.qx, w.lty, w.ltz, t.xblocks, t.yblocks, t.zblocks, t.xsmem,
              t.ysmem, t.zsmem);
}
// lines of: ndim nx ny nz nq precision wave reversed
int main() {
  int nd, nx, ny, nz, nq, prec, wave, rev;
  while (std::scanf("%d %d %d %d %d %d %d %d", &nd, &nx, &ny, &nz, &nq, &prec, &wave, &rev) == 8) {
    GridDesc g{};
    g.ndim = nd;
    g.nx = nx;
    g.ny = ny;
    g.nz = nd == 3 ? nz : 1;
    g.nxh = nx / 2 + 1;
    g.nxs = spectrum_stride(g.nxh);
    g.nq = nq;
    g.ncomp = (nd == 3 ? 6 : 3) * nq;
    g.nrows = (long long)g.ny * g.nz;
    g.nvox = g.nrows * nx;
    if (prec == 32) plan<float>(g, wave, rev);
    else plan<double>(g, wave, rev);
  }
  return 0;
}
"""
KEYS = ("qx", "lty", "ltz", "xblocks", "yblocks", "zblocks", "xsmem", "ysmem", "zsmem")


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    from paper_2207_10657_gb300 import build
    lib = build.build()
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cu", d / "plan"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, str(src), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(exe)], check=True)

    def run(rows):
        text = "\n".join(" ".join(str(x) for x in r) for r in rows)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [dict(zip(KEYS, map(int, line.split()))) for line in out.splitlines()]
    return run


@pytest.mark.parametrize("dims", [(8, 8, 8), (16, 16, 16), (24, 24, 24), (32, 32, 32), (10, 48, 90), (64, 64), (90, 60),
                                  (512, 512)], ids=lambda d: "x".join(map(str, d)))
def test_tiles_follow_the_share_of_the_launch(planner, dims):
    """A member of a batch keeps tiles of about a block's work however small
    the member is: its launches hold 256 of them.  Alone it is spread out."""
    nd, nc = len(dims), 6 if len(dims) == 3 else 3
    nx, ny, nz = (dims + (1,))[:3]
    row = (nd, nx, ny, nz, 1, 32)
    alone, member = planner([row + (304, 0), row + (2, 0)])
    total = nc * nx * ny * nz  # real values; a complex element holds two
    # x: 2048 complex elements, or half of the member (its share is two
    # blocks), less the rounding to whole (2D: pairs of) voxel rows
    assert 2 * 2048 >= member["qx"] * nc * nx >= min(2048, total // 4)
    # columns: half of the 2048-element tile, or one segment of a sector at
    # least, unless the block's registers hold fewer (1024 elements a line
    # group); two blocks where the grid is smaller than that
    nxh = nx // 2 + 1
    if nd == 3:
        assert (ny << member["lty"]) >= 1024 or member["yblocks"] <= 2 * 2
        assert (nc * nz << member["ltz"]) >= 1024 or member["zblocks"] <= 2 * 2
    else:
        assert (nc * ny << member["ltz"]) >= 1024 or member["zblocks"] <= 2 * 2
    assert member["zblocks"] <= alone["zblocks"] <= max(nxh * (ny if nd == 3 else 1), 1)
    assert alone["xblocks"] >= min(304, nz * ny // 2)


def _smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


def test_every_accepted_grid_fits_a_block(planner):
    """Shared memory of a block (112 KB at most) for every length that a grid
    may have on each axis, alone and with a small share, and for Kuhn
    tetrahedra up to the sizes that rve_create takes."""
    rows = []
    for n in filter(_smooth, range(2, 1025, 2)):
        for prec in (32, 64):
            for wave in (304, 2):
                for o in (2, 64, 1024):
                    tail = (prec, wave, 0)
                    rows += [(2, n, o, 1, 2) + tail, (2, o, n, 1, 2) + tail]
                    if n <= 227:
                        rows.append((3, n, o, 4, 6) + tail)
                    if n <= (341 if prec == 32 else 177):
                        rows.append((3, min(o, 200), 4, n, 6) + tail)
                    rows.append((3, 4, n, 4, 6) + tail)
                    for rev in (0, 1):
                        tail = (prec, wave, rev)
                        rows += [(2, n, o, 1, 1) + tail, (2, o, n, 1, 1) + tail, (3, n, o, 4, 1) + tail,
                                 (3, 4, n, o, 1) + tail, (3, o, 4, n, 1) + tail]
    plans = planner(rows)
    assert len(plans) == len(rows)
    for r, t in zip(rows, plans):
        assert max(t["xsmem"], t["ysmem"], t["zsmem"]) <= 112 * 1024, (r, t)
