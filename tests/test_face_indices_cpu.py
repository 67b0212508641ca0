"""Flat face indices of the complex128 stencil marches (operator apply, defect,
true residual) at the far corner of the largest grids: the face arrays are longer
than the cell arrays, so their indices pass 2^31 on grids of fewer cells. The
index functions are compiled for the host (no GPU) and compared with Python's
integers."""
import os
import subprocess

import pytest

from paper_1212_3660_gb300 import build

PROGRAM = """
#include <cstdio>
#include "stencil.cuh"
int main() {
  int nx, ny, nz;
  while (scanf("%d %d %d", &nx, &ny, &nz) == 3) {
    const int k = nz - 1, j = ny - 1, row = (int)((long long)k * ny + j), c = (int)((long long)row * nx + nx - 1);
    printf("%lld %lld %lld\\n", (long long)fks::x_face(c, row) + 1, (long long)fks::y_face(c, k, nx) + nx,
           (long long)fks::next_face(c, nz > 1 ? nx * ny : nx));
  }
}
"""

# all but the last within ny nz, nx nz or nx ny cells of 2^31
SHAPES = [(4096, 724, 724), (724, 4096, 724), (8, 16384, 16383), (46340, 46341, 1), (2048, 2048, 511), (3, 5, 7)]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("faces")
    src, exe = os.path.join(d, "faces.cu"), os.path.join(d, "faces")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, src, "-o", exe], check=True)
    return exe


def test_last_cell_reads_the_last_face(program):
    out = subprocess.run([program], input="\n".join("%d %d %d" % s for s in SHAPES), capture_output=True, text=True,
                         check=True).stdout.split("\n")
    for (nx, ny, nz), line in zip(SHAPES, out):
        assert nx * ny * nz < 2 ** 31
        last_x = (nx + 1) * ny * nz - 1
        last_y = nx * (ny + 1) * nz - 1
        last_march = nx * ny * (nz + 1) - 1 if nz > 1 else last_y
        assert [int(v) for v in line.split()] == [last_x, last_y, last_march], (nx, ny, nz)
