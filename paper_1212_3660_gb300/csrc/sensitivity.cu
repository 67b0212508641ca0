// Sensitivities of the phasor measurements by the adjoint-state method
// (Section 5, Eq. sensitivity with the adjoint of Eq. adjoint, Algorithm 6), in
// the cell-centred discretisation: with A = K + sigma M, A Phi = b, h = Phi(x_m)
// and A Psi = -e_m (A is complex symmetric, so the adjoint operator is A),
//   dh/dp = Psi^T (dA/dp) Phi.
// For p = ln S_s,c:  sigma M_cc Psi_c Phi_c.
// For p = ln K_c, over the faces of cell c (transmissibility t):
//   interior face to nb:  t K_nb / (K_c + K_nb) (Psi_c - Psi_nb)(Phi_c - Phi_nb)
//     (t = g 2 K_c K_nb / (K_c + K_nb), so dt/dlnK_c = t K_nb / (K_c + K_nb))
//   zero-head boundary face: t Psi_c Phi_c  (t = 2 g K_c; no-flow faces carry t = 0)
// On GB300 this is bound by FP64 arithmetic, not by memory: per cell, shift and
// measurement the differences of Psi, 4 fused multiply-adds per face and a
// complex product. Three things keep the rest small:
//   - dt/dlnK_c of every face (a division) depends neither on the shift nor on
//     the measurement: k_sens_weights forms it once per cell;
//   - a face's difference is formed once for its two cells (the other's is its
//     negative, exactly): along x it comes from the neighbouring lane, along
//     the direction in which a warp marches (y in 2D, z in 3D) from the step
//     before, so a 2D cell takes 2 complex subtractions instead of 4;
//   - the weights times Phi's differences are folded once per cell and shift,
//     for up to SENS_M measurements.
// 512^2, 200 shifts, 8 measurements: 20.0 ms; 26.1 with a thread per cell and
// shift that did all of this itself.
#include "sensitivity.cuh"
#include "stencil.cuh"

namespace fks {

constexpr int SENS_M = 8;       // measurements per pass (their differences below wait in shared memory)
constexpr int SENS_WARPS = 8;
constexpr int SENS_OUT = 31;    // cells per warp; lane 0 is the cell before them

// dt/dlnK_c of cell c's faces: w[a n + c], a in the order x low, x high, y, z
__global__ void k_sens_weights(LevelView<double> L, const double* __restrict__ cond, double* __restrict__ w) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  const Cell p = cell_of((int)c, L.nx, L.ny);
  const Faces<double> f = faces_at(L, p);
  const double kc = cond[c];
  const int64_t sxy = (int64_t)L.nx * L.ny;
  const double t[6] = {f.xl, f.xh, f.yl, f.yh, f.zl, f.zh};
  const bool inner[6] = {p.i > 0, p.i < L.nx - 1, p.j > 0, p.j < L.ny - 1, p.k > 0, p.k < L.nz - 1};
  const int64_t step[6] = {-1, 1, -(int64_t)L.nx, (int64_t)L.nx, -sxy, sxy};
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    if (a >= 4 && L.nz == 1) break;
    double v = t[a];
    if (inner[a]) {
      const double kn = cond[c + step[a]];
      v = t[a] * (kn / (kc + kn));
    }
    w[(int64_t)a * L.n + c] = v;
  }
}

__device__ __forceinline__ z64 shfl_dn(z64 v) {
  return mk(__shfl_down_sync(0xffffffffu, v.re, 1), __shfl_down_sync(0xffffffffu, v.im, 1));
}
__device__ __forceinline__ z64 shfl_up(z64 v) {
  return mk(__shfl_up_sync(0xffffffffu, v.re, 1), __shfl_up_sync(0xffffffffu, v.im, 1));
}
// sign change with integer instructions (a negation that is not an operand of a
// multiply-add takes an issue slot of the FP64 pipe)
__device__ __forceinline__ double neg(double v) {
  return __hiloint2double(__double2hiint(v) ^ 0x80000000, __double2loint(v));
}
__device__ __forceinline__ z64 neg(z64 v) { return mk(neg(v.re), neg(v.im)); }
// acc + d a in four fused multiply-adds
__device__ __forceinline__ z64 cfma(z64 d, z64 a, z64 acc) {
  acc.re = fmaT(d.re, a.re, fmaT(-d.im, a.im, acc.re));
  acc.im = fmaT(d.re, a.im, fmaT(d.im, a.re, acc.im));
  return acc;
}

// The march axis (y in 2D, z in 3D) is cut into strips of `len` steps. A warp
// owns 31 consecutive cells of the list of all strips' first rows (planes), in
// the order strip, row, x, and marches with them; a row may end and the next
// one (or the next strip) begin inside a warp, so narrow grids leave no lanes
// idle (48 x 32 x 32, 113 shifts, 7 measurements: 3.06 ms, 3.68 with two warps
// per row).
template <bool D3>
__global__ void __launch_bounds__(SENS_WARPS * 32, 2)
    k_sensitivity(LevelView<double> L, const double* __restrict__ wt, const z64* __restrict__ phi,
                  const z64* __restrict__ psi, int n_m, int n_f, const z64* __restrict__ sigma, z64* __restrict__ jk,
                  z64* __restrict__ js, int len, int total) {
  __shared__ z64 below[SENS_M][SENS_WARPS * 32];  // psi(c) - psi(c + step) of the march step before
  const int lane = threadIdx.x & 31, t = threadIdx.x, j = blockIdx.y;
  const int nx = L.nx, ny = L.ny, nm = D3 ? L.nz : ny, step = D3 ? nx * ny : nx;
  const int g = (int)(blockIdx.x * SENS_WARPS + (t >> 5)) * SENS_OUT + lane - 1;
  const bool own = g >= 0 && g < total;
  const int strip = own ? g / step : 0, p = own ? g % step : 0, i = p % nx, row = p / nx;
  const int m0 = strip * len, c0 = m0 * step + p;
  // steps of the warp: its last strip may be shorter
  const int steps = __reduce_max_sync(0xffffffffu, own ? min(len, nm - m0) : 0);
  const bool xlo = i > 0, xhi = i < nx - 1;
  const bool ylo = row > 0, yhi = row < ny - 1;
  const int64_t n = L.n;
  const z64* ph = phi + (int64_t)j * n;
  const z64 none = mk(0.0, 0.0), sg = sigma[j];
  // v(c) - v(c + 1), for the lane's cell and, from the lane below, its left face
  auto xdiff = [&](const z64* v, int c, bool in, z64 here, z64* lo, z64* hi) {
    z64 right = shfl_dn(here);
    if (lane == 31 && in && xhi) right = v[c + 1];
    *hi = here - right;
    *lo = neg(shfl_up(*hi));
  };
  for (int mc = 0; mc < n_m; mc += SENS_M) {
    const int nmc = min(SENS_M, n_m - mc);
    int c = c0;
    z64 ph_c = own ? ph[c] : none;
    z64 ph_lo = none;  // phi(c - step) - phi(c)
    if (m0 > 0 && own) {
      ph_lo = ph[c - step] - ph_c;
      for (int q = 0; q < nmc; ++q) {
        const z64* ps = psi + ((int64_t)(mc + q) * n_f + j) * n;
        below[q][t] = ps[c - step] - ps[c];
      }
    }
    for (int m = m0; m < m0 + steps; ++m, c += step) {
      const bool in = own && m < nm, out = in && lane > 0;
      const bool mlo = m > 0, mhi = m + 1 < nm;
      const z64 ph_n = in && mhi ? ph[c + step] : none;
      z64 dl, dh;
      xdiff(ph, c, in, ph_c, &dl, &dh);
      const z64 dm = ph_c - ph_n;
      z64 a[6];
      z64 smphi = none;
      if (out) {
        a[0] = wt[c] * (xlo ? dl : ph_c);
        a[1] = wt[n + c] * (xhi ? dh : ph_c);
        if constexpr (D3) {
          a[2] = wt[2 * n + c] * (ylo ? ph_c - ph[c - nx] : ph_c);
          a[3] = wt[3 * n + c] * (yhi ? ph_c - ph[c + nx] : ph_c);
          a[4] = wt[4 * n + c] * (mlo ? neg(ph_lo) : ph_c);
          a[5] = wt[5 * n + c] * (mhi ? dm : ph_c);
        } else {
          a[2] = wt[2 * n + c] * (mlo ? neg(ph_lo) : ph_c);
          a[3] = wt[3 * n + c] * (mhi ? dm : ph_c);
        }
        smphi = (L.mm[c] * sg) * ph_c;  // sigma M_cc Phi_c
      }
      ph_lo = dm;
      ph_c = ph_n;
      // a measurement's two loads are issued while the one before is summed
      const z64* ps = psi + ((int64_t)mc * n_f + j) * n;
      z64 pc = in ? ps[c] : none, pn = in && mhi ? ps[c + step] : none;
      for (int q = 0; q < nmc; ++q) {
        const int64_t base = ps - psi;
        const z64* next = ps + (int64_t)n_f * n;
        z64 nc = none, nn = none;
        if (q + 1 < nmc) {
          nc = in ? next[c] : none;
          nn = in && mhi ? next[c + step] : none;
        }
        z64 xl, xh;
        xdiff(ps, c, in, pc, &xl, &xh);
        const z64 d = pc - pn, lo = below[q][t];
        below[q][t] = d;
        if (out) {
          z64 acc = cfma(xlo ? xl : pc, a[0], none);
          acc = cfma(xhi ? xh : pc, a[1], acc);
          if constexpr (D3) {
            acc = cfma(ylo ? pc - ps[c - nx] : pc, a[2], acc);
            acc = cfma(yhi ? pc - ps[c + nx] : pc, a[3], acc);
            acc = cfma(mlo ? neg(lo) : pc, a[4], acc);
            acc = cfma(mhi ? d : pc, a[5], acc);
          } else {
            acc = cfma(mlo ? neg(lo) : pc, a[2], acc);
            acc = cfma(mhi ? d : pc, a[3], acc);
          }
          jk[base + c] = acc;
          js[base + c] = smphi * pc;
        }
        ps = next;
        pc = nc;
        pn = nn;
      }
    }
  }
}

size_t sensitivity_work(const LevelHost& L0) { return (size_t)(L0.nz > 1 ? 6 : 4) * L0.n; }

void launch_sensitivity(const LevelHost& L0, const double* cond, const z64* phi, const z64* psi, int n_m, int n_f,
                        const z64* sigma, z64* jk, z64* js, double* work, cudaStream_t s) {
  const LevelView<double> L = view<double>(L0);
  auto up = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
  k_sens_weights<<<(unsigned)up(L0.n, 256), 256, 0, s>>>(L, cond, work);
  // strips of 16 steps while that leaves eight blocks per SM, then of equal length
  const int64_t nm = L0.nz > 1 ? L0.nz : L0.ny, part = L0.n / nm;
  auto blocks = [&](int64_t len) { return up(part * up(nm, len), SENS_OUT * SENS_WARPS); };
  int64_t len = 16;
  while (len > 1 && blocks(len) * n_f < 8 * 152) len /= 2;
  len = up(nm, up(nm, len));
  const dim3 g((unsigned)blocks(len), (unsigned)n_f);
  auto kernel = L0.nz > 1 ? k_sensitivity<true> : k_sensitivity<false>;
  kernel<<<g, SENS_WARPS * 32, 0, s>>>(L, work, phi, psi, n_m, n_f, sigma, jk, js, (int)len, (int)(part * up(nm, len)));
}

}  // namespace fks
