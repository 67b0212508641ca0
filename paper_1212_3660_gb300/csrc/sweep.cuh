// Tile and chunk of the one-launch 3D sweeps (sweep.cu).
#pragma once
#include <algorithm>
#include <cmath>

namespace fks {

struct SweepGeom {
  int opx, oy, oz;    // pairs, rows and planes a block writes
  int txp;            // pairs of its region, the ring included; its rows are oy + 4
  int ntx, nty, ntz;
};

// The next chunk length after `o` that cuts a side of `n` into fewer chunks
// (n + 1: there is none)
inline int next_chunk(int n, int o) {
  const int cuts = (n + o - 1) / o;
  return cuts > 1 ? (n + cuts - 2) / (cuts - 1) : n + 1;
}

// The least estimated time over the tiles that fit blocks of NT threads, PER_SM
// blocks per SM, `word` bytes a real value. Each number of chunks is tried once
// (about 4 sqrt(ny nz) candidates): 8 us on the host for a level of 2 x 2 x 32768
// cells, 265 when every length is tried.
inline SweepGeom sweep_geometry(int nx, int ny, int nz, int nslot, int NT, int PER_SM, int word) {
  const int np = (nx + 1) / 2;
  SweepGeom best{};
  double cost = 1e300;
  for (int ntx = 1; ntx <= np; ++ntx) {
    const int opx = (np + ntx - 1) / ntx, txp = std::min(opx + (ntx > 2 ? 2 : ntx - 1), np);
    if (txp * 5 > NT) continue;
    if (ntx > 1 && (np + opx - 1) / opx != ntx) continue;
    if (cost < 1e300 && opx < 8) break;
    for (int oy = 1; oy <= ny && txp * (oy + 4) <= NT; oy = next_chunk(ny, oy)) {
      const int nty = (ny + oy - 1) / oy;
      const int nt = (txp * (oy + 4) + 31) & ~31;
      const int per = PER_SM * std::max(1, NT / nt) * 152;
      for (int oz = 1; oz <= nz; oz = next_chunk(nz, oz)) {
        const int ntz = (nz + oz - 1) / oz;
        if (ntz > 65535) continue;
        const double blocks = (double)ntx * nty * ntz * nslot, rounds = std::ceil(blocks / per);
        // a step is 0.5 us of latency, or the SM's share of the traffic (19 words per pair, 46 GB/s)
        const double step = std::max(0.5, std::min(blocks / 152, (double)per / 152) * nt * 19.0 * word / 46000.0);
        const double c = rounds * (oz + 2.5) * step;
        if (c < cost) {
          cost = c;
          best = SweepGeom{opx, oy, oz, txp, ntx, nty, ntz};
        }
      }
    }
  }
  return best;
}

}  // namespace fks
