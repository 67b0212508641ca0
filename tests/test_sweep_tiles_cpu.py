"""The host's search for the tile of a one-launch 3D sweep: it tries each number
of chunks of an axis once, finds what trying every chunk length finds, and takes
a long thin level no longer than its few different cuts."""
import os
import subprocess

import pytest

from paper_1212_3660_gb300 import build

PROGRAM = """
#include <chrono>
#include <cstdio>
#include "sweep.cuh"
using namespace fks;
static double cost_of(const SweepGeom& G, int nslot, int NT, int PER_SM, int word) {
  const int nt = (G.txp * (G.oy + 4) + 31) & ~31, per = PER_SM * std::max(1, NT / nt) * 152;
  const double blocks = (double)G.ntx * G.nty * G.ntz * nslot;
  const double step = std::max(0.5, std::min(blocks / 152, (double)per / 152) * nt * 19.0 * word / 46000.0);
  return std::ceil(blocks / per) * (G.oz + 2.5) * step;
}
int main() {
  const int NT = 384, PER = 2;
  int nx, ny, nz, nslot;
  while (scanf("%d %d %d %d", &nx, &ny, &nz, &nslot) == 4) {
    const SweepGeom G = sweep_geometry(nx, ny, nz, nslot, NT, PER, 4);
    // every length of the chunks in y and z, for the tile width found
    double best = 1e300;
    for (int oy = 1; oy <= ny && G.txp * (oy + 4) <= NT; ++oy)
      for (int oz = 1; oz <= nz; ++oz) {
        SweepGeom H = G;
        H.oy = oy; H.oz = oz; H.nty = (ny + oy - 1) / oy; H.ntz = (nz + oz - 1) / oz;
        if (H.ntz <= 65535) best = std::min(best, cost_of(H, nslot, NT, PER, 4));
      }
    double us = 1e300;
    for (int r = 0; r < 20; ++r) {
      const auto t0 = std::chrono::steady_clock::now();
      volatile int sink = sweep_geometry(nx, ny, nz, nslot, NT, PER, 4).oz;
      (void)sink;
      us = std::min(us, std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count());
    }
    printf("%d %d %d %d %d %d %d %.17g %.17g %.3f\\n", G.opx, G.oy, G.oz, G.txp, G.ntx, G.nty, G.ntz,
           cost_of(G, nslot, NT, PER, 4), best, us);
  }
}
"""

SHAPES = [(48, 48, 48, 1), (32, 32, 32, 1), (27, 25, 26, 1), (17, 16, 64, 2), (61, 60, 5, 1), (411, 7, 6, 8), (1, 9, 40, 1),
          (2, 4096, 7, 1), (2, 2, 32768, 1), (130000, 1, 1, 1)]


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    d = tmp_path_factory.mktemp("sweeps")
    src, exe = os.path.join(d, "tiles.cu"), os.path.join(d, "tiles")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, src, "-o", exe], check=True)
    out = subprocess.run([exe], input="\n".join("%d %d %d %d" % s for s in SHAPES), capture_output=True, text=True,
                         check=True).stdout.split("\n")
    return {s: [float(v) for v in line.split()] for s, line in zip(SHAPES, out)}


@pytest.mark.parametrize("shape", SHAPES)
def test_tiles_cover_the_level_at_the_least_cost(results, shape):
    opx, oy, oz, txp, ntx, nty, ntz, cost, best, _ = results[shape]
    nx, ny, nz, _ = shape
    assert opx * ntx >= (nx + 1) // 2 and oy * nty >= ny and oz * ntz >= nz
    assert txp * (oy + 4) <= 384 and ntz <= 65535
    assert cost == best


def test_a_long_level_is_searched_as_fast_as_a_cube(results):
    # 724 candidates against about 300: 1.7 times the time; 34 times where every length is tried
    assert results[(2, 2, 32768, 1)][-1] <= 10 * results[(48, 48, 48, 1)][-1]
