// Structured-grid kernels: operator coefficients, the shifted operator apply,
// and the geometric-multigrid pieces of the inexact inner solve (Section 4,
// Eq. zmmoditer): red-black Gauss-Seidel, residual + restriction,
// interpolation + correction, coarsest-level dense solve.
//
// Every vector kernel takes a batch of sources ("slots") on gridDim.y; vector
// arguments point at slot 0 and consecutive slots are `vs` elements apart.
#include <algorithm>
#include <climits>

#include "grid.cuh"
#include "stencil.cuh"

namespace fks {

__device__ __forceinline__ bool slot_running(const SlotState* st, int slot) {
  return st == nullptr || (st[slot].active && !st[slot].inner_done);
}

// --------------------------------------------------------------------- setup
// Fine-level faces from cell conductivity (harmonic mean on interior faces,
// 2 K A / h on zero-head faces). One thread per face of each orientation.
__global__ void k_faces_from_cond(int nx, int ny, int nz, double hx, double hy, double hz, uint32_t mask,
                                  const double* __restrict__ cond, double* fx, double* fy, double* fz) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t nfx = (int64_t)(nx + 1) * ny * nz, nfy = (int64_t)nx * (ny + 1) * nz;
  int64_t nfz = nz > 1 ? (int64_t)nx * ny * (nz + 1) : 0;
  if (t < nfx) {
    int i = (int)(t % (nx + 1));
    int64_t row = t / (nx + 1);  // k*ny + j
    double g = (hy * hz) / hx;
    int64_t c = row * nx + i;
    double v;
    if (i == 0) v = (mask & 1u) ? 2.0 * cond[c] * g : 0.0;
    else if (i == nx) v = (mask & 2u) ? 2.0 * cond[c - 1] * g : 0.0;
    else { double a = cond[c - 1], b = cond[c]; v = g * (2.0 * a * b / (a + b)); }
    fx[t] = v;
    return;
  }
  t -= nfx;
  if (t < nfy) {
    int i = (int)(t % nx);
    int64_t q = t / nx;
    int j = (int)(q % (ny + 1));
    int k = (int)(q / (ny + 1));
    double g = (hx * hz) / hy;
    int64_t c = ((int64_t)k * ny + j) * nx + i;
    double v;
    if (j == 0) v = (mask & 4u) ? 2.0 * cond[c] * g : 0.0;
    else if (j == ny) v = (mask & 8u) ? 2.0 * cond[c - nx] * g : 0.0;
    else { double a = cond[c - nx], b = cond[c]; v = g * (2.0 * a * b / (a + b)); }
    fy[t] = v;
    return;
  }
  t -= nfy;
  if (t < nfz) {
    int64_t sxy = (int64_t)nx * ny;
    int64_t ij = t % sxy;
    int k = (int)(t / sxy);
    double g = (hx * hy) / hz;
    int64_t c = (int64_t)k * sxy + ij;
    double v;
    if (k == 0) v = (mask & 16u) ? 2.0 * cond[c] * g : 0.0;
    else if (k == nz) v = (mask & 32u) ? 2.0 * cond[c - sxy] * g : 0.0;
    else { double a = cond[c - sxy], b = cond[c]; v = g * (2.0 * a * b / (a + b)); }
    fz[t] = v;
  }
}

// Coarse faces: (sum of the fine faces on the coarse face) x the face's factor
// (fine over coarse centre distance across it: 1/2 on evenly halved axes, 1 on
// axes not coarsened; fac_x/y/z, one per coarse face index along the axis);
// coarse mass: sum of the children. One thread per coarse face / cell. On an
// odd (ragged) axis the last coarse cell has one child: its high face is that
// child's, and the sums skip children past the fine grid.
__global__ void k_coarsen(LevelView<double> F, int rx, int ry, int rz, int cx_, int cy, int cz, double* fx,
                          double* fy, double* fz, double* mm, const double* __restrict__ fac_x,
                          const double* __restrict__ fac_y, const double* __restrict__ fac_z) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t nfx = (int64_t)(cx_ + 1) * cy * cz, nfy = (int64_t)cx_ * (cy + 1) * cz;
  int64_t nfz = cz > 1 || F.nz > 1 ? (int64_t)cx_ * cy * (cz + 1) : 0;
  int64_t ncell = (int64_t)cx_ * cy * cz;
  if (t < nfx) {
    int I = (int)(t % (cx_ + 1));
    int64_t q = t / (cx_ + 1);
    int J = (int)(q % cy), K = (int)(q / cy);
    double s = 0.0;
    const int64_t fi = min(rx * I, F.nx);
    for (int c = 0; c < rz; ++c)
      for (int b = 0; b < ry; ++b) {
        if (rz * K + c >= F.nz || ry * J + b >= F.ny) continue;
        int64_t row = (int64_t)(rz * K + c) * F.ny + (ry * J + b);
        s += F.fx[row * (F.nx + 1) + fi];
      }
    fx[t] = s * fac_x[I];
    return;
  }
  t -= nfx;
  if (t < nfy) {
    int I = (int)(t % cx_);
    int64_t q = t / cx_;
    int J = (int)(q % (cy + 1)), K = (int)(q / (cy + 1));
    double s = 0.0;
    const int64_t fj = min(ry * J, F.ny);
    for (int c = 0; c < rz; ++c)
      for (int a = 0; a < rx; ++a) {
        if (rz * K + c >= F.nz || rx * I + a >= F.nx) continue;
        s += F.fy[((int64_t)(rz * K + c) * (F.ny + 1) + fj) * F.nx + (rx * I + a)];
      }
    fy[t] = s * fac_y[J];
    return;
  }
  t -= nfy;
  if (t < nfz) {
    int64_t sxy = (int64_t)cx_ * cy;
    int64_t ij = t % sxy;
    int K = (int)(t / sxy);
    int I = (int)(ij % cx_), J = (int)(ij / cx_);
    double s = 0.0;
    const int64_t fk = min(rz * K, F.nz);
    for (int b = 0; b < ry; ++b)
      for (int a = 0; a < rx; ++a) {
        if (ry * J + b >= F.ny || rx * I + a >= F.nx) continue;
        s += F.fz[(fk * F.ny + (ry * J + b)) * F.nx + (rx * I + a)];
      }
    fz[t] = s * fac_z[K];
    return;
  }
  t -= nfz;
  if (t < ncell) {
    int I = (int)(t % cx_);
    int64_t q = t / cx_;
    int J = (int)(q % cy), K = (int)(q / cy);
    double s = 0.0;
    for (int c = 0; c < rz; ++c)
      for (int b = 0; b < ry; ++b)
        for (int a = 0; a < rx; ++a) {
          if (rz * K + c >= F.nz || ry * J + b >= F.ny || rx * I + a >= F.nx) continue;
          s += F.mm[((int64_t)(rz * K + c) * F.ny + (ry * J + b)) * F.nx + (rx * I + a)];
        }
    mm[t] = s;
  }
}

__global__ void k_to_f32(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) b[t] = (float)a[t];
}

// The bf16-smoother option's coefficients: a rounded to bf16 (nearest) and the
// same value as fp32 (exact).
__global__ void k_round_bf16(const double* __restrict__ a, __nv_bfloat16* __restrict__ b, float* __restrict__ r,
                             int64_t n) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const __nv_bfloat16 v = __double2bfloat16(a[t]);
  b[t] = v;
  r[t] = __bfloat162float(v);
}

// 1 / (K_cc + tau M_cc) per cell for every distinct tau, computed in fp64.
// (C: the coefficients' storage; the bf16-smoother option computes from the
// bf16-rounded values held as fp32)
template <typename T, typename C>
__global__ void k_invd(LevelView<double, C> L, const z64* __restrict__ taus, int ntau, cx<T>* __restrict__ out) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= L.n) return;
  Cell p = cell_of(c, L.nx, L.ny);
  Faces<double> f = faces_at(L, p);
  double d = fsum(f), m = ldc<double>(L.mm, c);
  for (int q = 0; q < ntau; ++q) {
    z64 D = mk(d + taus[q].re * m, taus[q].im * m);
    double den = abs2(D);
    out[(int64_t)q * L.n + c] = cvt<T>(mk(D.re / den, -D.im / den));
  }
}

// Dense coarsest-level matrix K + tau M (row-major, n x n, zeroed before) for
// every tau: the nonzero entries of row c. col0 (optional, [n_tau][n]) receives
// the first column, contiguous.
template <typename C>
__global__ void k_coarse_dense(LevelView<double, C> L, const z64* __restrict__ taus, z64* __restrict__ A,
                               z64* __restrict__ col0) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  if (c >= L.n) return;
  Cell p = cell_of(c, L.nx, L.ny);
  Faces<double> f = faces_at(L, p);
  double d = fsum(f), m = ldc<double>(L.mm, c);
  int64_t n = L.n, sxy = (int64_t)L.nx * L.ny;
  z64* row = A + (int64_t)q * n * n + c * n;
  row[c] = mk(d + taus[q].re * m, taus[q].im * m);
  if (p.i > 0) row[c - 1] = mk(-f.xl, 0.0);
  if (p.i < L.nx - 1) row[c + 1] = mk(-f.xh, 0.0);
  if (p.j > 0) row[c - L.nx] = mk(-f.yl, 0.0);
  if (p.j < L.ny - 1) row[c + L.nx] = mk(-f.yh, 0.0);
  if (L.nz > 1) {
    if (p.k > 0) row[c - sxy] = mk(-f.zl, 0.0);
    if (p.k < L.nz - 1) row[c + sxy] = mk(-f.zh, 0.0);
  }
  if (col0) col0[(int64_t)q * n + c] = row[0];
}

// --------------------------------------------------------------------- apply
// y = (K + s M) x, one vector per gridDim.z. Bound by the FP64 pipe, as the
// defect: 12 fused multiply-adds for a 3D cell's neighbours, 4 for its
// diagonal, 2 to form it. A thread marches over R cells along z (3D) or y (2D)
// with the neighbours below and above in registers.
template <bool D3>
__global__ void __launch_bounds__(GX * GY) k_apply(LevelView<double> L, z64 s, const z64* __restrict__ x,
                                                   z64* __restrict__ y, int64_t vs, int R) {
  const int nx = L.nx, ny = L.ny, sxy = nx * ny;
  const int i = blockIdx.x * GX + threadIdx.x;
  const int nby = (ny + GY - 1) / GY;
  const int bz = D3 ? blockIdx.y / nby : 0;
  const int j = D3 ? (int)(blockIdx.y - bz * nby) * GY + (int)threadIdx.y : 0;
  const int nm = D3 ? L.nz : ny, step = D3 ? sxy : nx;
  const int m0 = (D3 ? bz : (int)(blockIdx.y * GY + threadIdx.y)) * R, m1 = min(m0 + R, nm);
  if (i >= nx || j >= ny || m0 >= m1) return;
  const z64* v = x + blockIdx.z * vs;
  z64* o = y + blockIdx.z * vs;
  const double* fl = D3 ? L.fz : L.fy;  // the face below cell c along the march
  int c = m0 * step + j * nx + i;
  z64 below = m0 > 0 ? v[c - step] : mk(0.0, 0.0), here = v[c];
  double lo = fl[c];
  for (int m = m0; m < m1; ++m, c += step) {
    const bool top = m + 1 < nm;
    const double hi = fl[next_face(c, step)];
    const z64 above = top ? v[c + step] : mk(0.0, 0.0);
    const int row = D3 ? m * ny + j : m;
    const double mm = L.mm[c], d = fmaT(s.re, mm, L.kd[c]), e = mulT(s.im, mm);
    z64 a = mk(0.0, 0.0);
    if (i > 0) a = axpy(L.fx[x_face(c, row)], v[c - 1], a);
    if (i < nx - 1) a = axpy(L.fx[x_face(c, row) + 1], v[c + 1], a);
    if constexpr (D3) {
      const int64_t fy = y_face(c, m, nx);
      if (j > 0) a = axpy(L.fy[fy], v[c - nx], a);
      if (j < ny - 1) a = axpy(L.fy[fy + nx], v[c + nx], a);
    }
    if (m > 0) a = axpy(lo, below, a);
    if (top) a = axpy(hi, above, a);
    o[c] = mk(fmaT(d, here.re, fmaT(-e, here.im, -a.re)), fmaT(d, here.im, fmaT(e, here.re, -a.im)));
    below = here;
    here = above;
    lo = hi;
  }
}

// --------------------------------------------------------------------- smoother
// One red-black Gauss-Seidel half sweep on the cells of `color`
// (color 0 = red: i + j + k even): z_c = (f_c + sum_nb t z_nb) / (K_cc + tau M_cc).
// `zero_start`: the other colour is taken as zero (first sweep from z = 0).
// Multiple sources (SpMM form): a block holds G sources of the batch as
// threadIdx.z over the same cells (blockDim = (32, 8 / G, G)), so a cell's
// faces and inverse diagonal are fetched from memory once and served to the
// other sources' warps from the SM's L1 (sources in lockstep share tau_k);
// sources whose inner solve has finished return at once. Every source's update
// is the single-source one.
template <typename T, typename C>
__global__ void k_gs(LevelView<T, C> L, const SlotState* st, const cx<T>* __restrict__ invd,
                     const cx<T>* __restrict__ f, cx<T>* __restrict__ z, int64_t vs, int color, int zero_start,
                     int nslot, unsigned mny) {
  pdl_enter();
  const int slot = blockIdx.z * blockDim.z + threadIdx.z;
  if (slot >= nslot || !slot_running(st, slot)) return;
  const int ii = blockIdx.x * GX + threadIdx.x;
  const int row = blockIdx.y * blockDim.y + threadIdx.y;
  if (row >= L.ny * L.nz) return;
  int j, k;
  split_row(row, L.ny, mny, &j, &k);
  const int i = 2 * ii + ((j + k + color) & 1);
  if (i >= L.nx) return;
  const int c = row * L.nx + i;
  const cx<T> id = invd[(int64_t)st[slot].tau * L.n + c];
  cx<T>* zs = z + slot * vs;
  zs[c] = gs_row(L, Cell{i, j, k}, row, c, id, f + slot * vs, (const cx<T>*)zs, zero_start);
}

// The last half sweep of the finest level's post-smoothing fused with the
// defect correction: thread (ii, row) owns cells 2 ii and 2 ii + 1 of the row,
// updates the one of colour `color` as k_gs does, and adds both final values
// e to column k - 1 of the outer iterates (z_k = e on the first cycle, z_k + e
// after), the update of k_correct. z itself is not written: nothing reads the
// finest level's correction after this. Sources as in k_gs.
template <typename T, typename C>
__global__ void k_gs_correct(LevelView<T, C> L, const SlotState* st, const cx<T>* __restrict__ invd,
                             const cx<T>* __restrict__ f, const cx<T>* __restrict__ z, int64_t vs, int color,
                             z64* __restrict__ Zk, int64_t vsZk, int64_t zcol, int nslot, unsigned mny) {
  pdl_enter();
  const int slot = blockIdx.z * blockDim.z + threadIdx.z;
  if (slot >= nslot || !slot_running(st, slot)) return;
  const int ii = blockIdx.x * GX + threadIdx.x;
  const int row = blockIdx.y * blockDim.y + threadIdx.y;
  if (row >= L.ny * L.nz || 2 * ii >= L.nx) return;
  int j, k;
  split_row(row, L.ny, mny, &j, &k);
  const int c0 = row * L.nx + 2 * ii, h = (j + k + color) & 1, i = 2 * ii + h, c = c0 + h;
  const cx<T>* zs = z + slot * vs;
  z64* zk = Zk + slot * vsZk + (int64_t)(st[slot].k - 1) * zcol + c0;
  const bool first = st[slot].cycles == 0, two = 2 * ii + 1 < L.nx;
  const z64 none = mk(0.0, 0.0);
  const z64 o0 = first ? none : zk[0], o1 = first || !two ? none : zk[1];
  cx<T> v = mk(T(0), T(0)), w = v;  // the updated cell, the other
  if (h == 1 || two) w = zs[c0 + 1 - h];
  if (i < L.nx) {
    const cx<T> id = invd[(int64_t)st[slot].tau * L.n + c];
    v = gs_row(L, Cell{i, j, k}, row, c, id, f + slot * vs, zs, 0);
  }
  const z64 e0 = cvt<double>(h ? w : v), e1 = cvt<double>(h ? v : w);
  zk[0] = first ? e0 : (o0 + e0);
  if (two) zk[1] = first ? e1 : (o1 + e1);
}

// --------------------------------------------------------------------- transfer
// Coarse right-hand side = sum over the children of the fine residual f - A z
// (restrict_value).
// Sources as in k_gs (threadIdx.z), so the children's coefficients come from
// memory once per block.
template <typename T, typename C>
__global__ void k_residual_restrict(LevelView<T, C> F, int rx, int ry, int rz, int cnx, int cny, int cnz,
                                    const SlotState* st, const z64* taus, const cx<T>* __restrict__ f,
                                    const cx<T>* __restrict__ z, int64_t vs, cx<T>* __restrict__ fc, int64_t vsc,
                                    int nslot) {
  pdl_enter();
  const int slot = blockIdx.z * blockDim.z + threadIdx.z;
  if (slot >= nslot || !slot_running(st, slot)) return;
  const int I = blockIdx.x * GX + threadIdx.x;
  const int row = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= cnx || row >= cny * cnz) return;
  const int K = row / cny, J = row - K * cny;
  const cx<T> s = cvt<T>(taus[st[slot].tau]);
  fc[slot * vsc + (int64_t)row * cnx + I] = restrict_value(F, rx, ry, rz, I, J, K, s, f + slot * vs, z + slot * vs);
}

// Coarse right-hand side on a 3D level coarsened by 2 in every axis, one
// source per block. The per-coarse-cell loop of k_residual_restrict computes
// its children one after another; here the block's 256 threads first compute
// the fine residuals f - A z of a 32 x 8 x 2 tile, one (i, j) column of two
// planes each (one red cell in complex128, two cells in complex64), into shared
// memory, then one thread per coarse cell adds its children in
// restrict_value's order (z, then y, then x child), skipping those past the
// fine grid, so the sum is bitwise the same (64 x 48 x 48 complex128 9.9 us a
// launch with all cells, 5.5 with the red ones).
template <typename T, typename C>
__global__ void __launch_bounds__(256) k_residual_restrict3(LevelView<T, C> F, int cnx, int cny, int cnz,
                                                            const SlotState* st, const z64* taus,
                                                            const cx<T>* __restrict__ f, const cx<T>* __restrict__ z,
                                                            int64_t vs, cx<T>* __restrict__ fc, int64_t vsc) {
  pdl_enter();
  constexpr int NP = RED_RESIDUAL<T> ? 1 : 2;  // cells per column
  __shared__ cx<T> sr[NP][GY][GX];
  const int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int nby = (F.ny + GY - 1) / GY;
  const int K = blockIdx.y / nby, by = blockIdx.y - K * nby;
  const int i = blockIdx.x * GX + threadIdx.x, j = by * GY + threadIdx.y;
  const cx<T> s = cvt<T>(taus[st[slot].tau]);
  const cx<T>* fs = f + slot * vs;
  const cx<T>* zs = z + slot * vs;
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int k = 2 * K + (NP == 1 ? (i + j) & 1 : q);
    cx<T> r = mk(T(0), T(0));
    if (i < F.nx && j < F.ny && k < F.nz) {
      const int row = k * F.ny + j, c = row * F.nx + i;
      r = residual_row(F, Cell{i, j, k}, row, c, s, fs, zs);
    }
    sr[q][threadIdx.y][threadIdx.x] = r;
  }
  __syncthreads();
  const int t = threadIdx.y * GX + threadIdx.x;
  if (t >= (GX / 2) * (GY / 2)) return;
  const int ti = t % (GX / 2), tj = t / (GX / 2);
  const int I = blockIdx.x * (GX / 2) + ti, J = by * (GY / 2) + tj;
  if (I >= cnx || J >= cny) return;
  cx<T> acc = mk(T(0), T(0));
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = child_first<T>(b + c); a < 2; a += child_step<T>) {
        if (2 * I + a >= F.nx || 2 * J + b >= F.ny || 2 * K + c >= F.nz) continue;
        acc = acc + sr[NP == 1 ? 0 : c][2 * tj + b][2 * ti + a];
      }
  fc[slot * vsc + ((int64_t)K * cny + J) * cnx + I] = acc;
}

// z_fine += P z_coarse on the red cells (the black ones are overwritten by the
// next half sweep before anything reads them)
template <typename T>
__global__ void k_prolong_add(LevelView<T> F, int rx, int ry, int rz, int cnx, int cny, int cnz, uint32_t mask,
                              const SlotState* st, const cx<T>* __restrict__ zc, int64_t vsc,
                              cx<T>* __restrict__ z, int64_t vs) {
  pdl_enter();
  int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  Cell p;
  int c;
  if (!grid_color_cell(F.nx, F.ny, F.nz, 0, &p, &c)) return;
  cx<T>* zs = z + slot * vs;
  zs[c] = zs[c] + prolong_value(p, rx, ry, rz, cnx, cny, cnz, mask, zc + slot * vsc);
}

// z_fine += P z_coarse on a 3D level coarsened by 2 in every axis: a block
// updates 32 x 8 cells in each of the two fine planes of coarse plane K and
// first stages the 18 x 6 x 3 coarse values they interpolate from (planes K -
// 1, K and K + 1) in shared memory, so each coarse value is read once per
// block instead of once per fine cell; the interpolation itself is
// prolong_value_at's, on those values. Only red cells are updated: one of the
// two planes' cells of each column.
template <typename T>
__global__ void __launch_bounds__(256) k_prolong_add3(LevelView<T> F, int cnx, int cny, int cnz, uint32_t mask,
                                                      const SlotState* st, const cx<T>* __restrict__ zc,
                                                      int64_t vsc, cx<T>* __restrict__ z, int64_t vs) {
  pdl_enter();
  constexpr int SX = GX / 2 + 2, SY = GY / 2 + 2;
  __shared__ cx<T> sc[3][SY][SX];
  const int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int nby = (F.ny + GY - 1) / GY;
  const int K = blockIdx.y / nby, by = blockIdx.y - K * nby;
  const int x0 = blockIdx.x * GX, y0 = by * GY;
  const int X0 = x0 / 2 - 1, Y0 = y0 / 2 - 1;
  const cx<T>* zcs = zc + slot * vsc;
  // the cell's own value is loaded before the staging barrier, so its latency
  // overlaps that of the coarse values
  const int i = x0 + threadIdx.x, j = y0 + threadIdx.y;
  cx<T>* zs = z + slot * vs;
  const int k = 2 * K + ((i + j) & 1);
  const bool own = i < F.nx && j < F.ny && k < F.nz;
  const int64_t c = ((int64_t)k * F.ny + j) * F.nx + i;
  const cx<T> z0 = own ? zs[c] : mk(T(0), T(0));
  for (int t = threadIdx.y * GX + threadIdx.x; t < 3 * SY * SX; t += GX * GY) {
    const int q = t / (SY * SX), rem = t - q * (SY * SX);
    const int yy = rem / SX, xx = rem - yy * SX;
    const int X = X0 + xx, Y = Y0 + yy, Z = K - 1 + q;
    const bool in = X >= 0 && X < cnx && Y >= 0 && Y < cny && Z >= 0 && Z < cnz;
    sc[q][yy][xx] = in ? zcs[((int64_t)Z * cny + Y) * cnx + X] : mk(T(0), T(0));
  }
  __syncthreads();
  if (!own) return;
  zs[c] = z0 + prolong_value_at<T>(Cell{i, j, k}, 2, 2, 2, cnx, cny, cnz, mask,
                                   [&](int X, int Y, int Z) { return sc[Z - K + 1][Y - Y0][X - X0]; });
}

// --------------------------------------------------------------------- fused 2D level kernels
// One level of the V-cycle on a 2D grid coarsened in both axes (odd sides
// included: their last coarse cell has one child), in two
// kernels over TX x TY tiles with a halo of H = 4 cells held in shared memory.
// Red-black half sweeps only read the other colour, so every half sweep is
// recomputed on a region that shrinks by one cell per sweep; the tile interior
// then holds exactly the values of the per-sweep kernels.
//   pre : z = four half sweeps from z = 0 (red, black, red, black); write z;
//         coarse f = sum over children of (f - A z)
//   post: z += P z_coarse; four half sweeps (black, red, black, red); write z

// sum over existing neighbours of t_face * z_nb for a 2D cell held at r in a
// shared tile of row length RX (same order as nb_sum)
template <typename T>
__device__ __forceinline__ cx<T> nb_sum_tile(const LevelView<T>& L, Cell p, int r, int RX, const cx<T>* sZ,
                                             cx<T> s0 = cx<T>{T(0), T(0)}) {
  Faces<T> f = faces_at(L, p);
  cx<T> s = s0;
  if (p.i > 0) s = axpy(f.xl, sZ[r - 1], s);
  if (p.i < L.nx - 1) s = axpy(f.xh, sZ[r + 1], s);
  if (p.j > 0) s = axpy(f.yl, sZ[r - RX], s);
  if (p.j < L.ny - 1) s = axpy(f.yh, sZ[r + RX], s);
  return s;
}

template <typename T, int TX, int TY>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? (TX == 32 ? 6 : 8) : 4) k_pre2d(LevelView<T> L, const SlotState* st, const cx<T>* __restrict__ invd,
                                               const z64* taus, const cx<T>* __restrict__ f, cx<T>* __restrict__ z,
                                               int64_t vs, cx<T>* __restrict__ fc, int64_t vsc) {
  pdl_enter();
  constexpr int RX = TX + 2 * FH, RY = TY + 2 * FH;
  extern __shared__ __align__(16) unsigned char pre_smem[];
  cx<T>* sF = (cx<T>*)pre_smem;
  cx<T>* sZ = sF + RX * RY;
  int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int tau = st[slot].tau;
  const cx<T> sft = cvt<T>(taus[tau]);
  const cx<T>* ID = invd + (int64_t)tau * L.n;
  const cx<T>* fs = f + slot * vs;
  const int x0 = blockIdx.x * TX - FH, y0 = blockIdx.y * TY - FH;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int q = tid; q < RX * RY; q += nt) {
    int ry = q / RX, rx = q - ry * RX;
    int gx = x0 + rx, gy = y0 + ry;
    bool in = gx >= 0 && gx < L.nx && gy >= 0 && gy < L.ny;
    sF[q] = in ? fs[gy * L.nx + gx] : mk(T(0), T(0));
  }
  __syncthreads();
  for (int hs = 0; hs < 4; ++hs) {
    const int color = hs & 1;
    const int w = RX - 2 * hs, hgt = RY - 2 * hs;
    const int wh = (w + 1) >> 1;
    for (int q = tid; q < wh * hgt; q += nt) {
      int yy = q / wh;
      int ry = hs + yy;
      int gy = y0 + ry;
      int rx0 = hs + 2 * (q - yy * wh);
      int gx = x0 + rx0;
      if (((gx + gy) & 1) != color) { ++gx; ++rx0; }
      if (rx0 >= RX - hs || gx < 0 || gx >= L.nx || gy < 0 || gy >= L.ny) continue;
      int r = ry * RX + rx0;
      int c = gy * L.nx + gx;
      cx<T> rhs = sF[r];
      if (hs > 0) rhs = nb_sum_tile(L, Cell{gx, gy, 0}, r, RX, sZ, rhs);
      sZ[r] = ID[c] * rhs;
    }
    __syncthreads();
  }
  cx<T>* zs = z + slot * vs;
  for (int q = tid; q < TX * TY; q += nt) {
    int yy = q / TX, xx = q - yy * TX;
    int gx = x0 + FH + xx, gy = y0 + FH + yy;
    if (gx < L.nx && gy < L.ny) zs[gy * L.nx + gx] = sZ[(yy + FH) * RX + xx + FH];
  }
  // residual + restriction to the (TX/2) x (TY/2) coarse cells of the tile. Two
  // lanes per coarse cell, one for each of its rows of children: with one, a
  // quarter of the threads did it all, on half of the SM's FP64 units (512^2
  // complex128, all cells: 29.8 us a launch; two lanes, red cells: 27.2)
  const int cnx = (L.nx + 1) >> 1, cny = (L.ny + 1) >> 1;
  cx<T>* fcs = fc + slot * vsc;
  constexpr int NC = RED_RESIDUAL<T> ? 1 : 2;    // children per lane
  for (int q = tid; q < TX * TY / 2; q += nt) {  // whole warps
    const int h = q & 1, C = q >> 1;
    const int Yl = C / (TX / 2), Xl = C - Yl * (TX / 2);
    const int X = blockIdx.x * (TX / 2) + Xl, Y = blockIdx.y * (TY / 2) + Yl;
    const int gy = 2 * Y + h;
    cx<T> acc = mk(T(0), T(0));
    cx<T> res[NC];
    bool in[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
      const int gx = 2 * X + (NC == 1 ? h : a);
      in[a] = gx < L.nx && gy < L.ny;
      res[a] = acc;
      if (!in[a]) continue;
      const int r = (gy - y0) * RX + (gx - x0);
      const int c = gy * L.nx + gx;
      const T d = sizeof(T) == 8 && L.kd ? L.kd[c] : fsum(faces_at(L, Cell{gx, gy, 0})), m = L.mm[c];
      res[a] = residual_of(sF[r], sZ[r], mk(fmaT(sft.re, m, d), mulT(sft.im, m)),
                           [&](cx<T> s0) { return nb_sum_tile(L, Cell{gx, gy, 0}, r, RX, sZ, s0); });
    }
    // the children in their order: the even lane's, then the odd lane's
#pragma unroll
    for (int a = 0; a < NC; ++a)
      if (in[a]) acc = acc + res[a];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
      const cx<T> other = mk(__shfl_down_sync(0xffffffffu, res[a].re, 1), __shfl_down_sync(0xffffffffu, res[a].im, 1));
      if (__shfl_down_sync(0xffffffffu, (int)in[a], 1)) acc = acc + other;
    }
    if (h == 0 && in[0]) fcs[Y * cnx + X] = acc;
  }
}

// post reads the pre-smoothed z and writes zout (a different buffer): tiles
// read their neighbours' cells as halo, which those tiles overwrite. With Zk
// given (finest level), the result e is instead added to the outer iterate,
// z_k = e on the first cycle and z_k + e after (the update of k_correct).
template <typename T, int TX, int TY>
__global__ void __launch_bounds__(256) k_post2d(LevelView<T> L, uint32_t mask, const SlotState* st,
                                                const cx<T>* __restrict__ invd, const cx<T>* __restrict__ f,
                                                const cx<T>* __restrict__ z, cx<T>* __restrict__ zout, int64_t vs,
                                                const cx<T>* __restrict__ zc, int64_t vsc, z64* __restrict__ Zk,
                                                int64_t vsZk, int64_t zcol) {
  pdl_enter();
  constexpr int RX = TX + 2 * FH, RY = TY + 2 * FH;
  extern __shared__ __align__(16) unsigned char post_smem[];
  cx<T>* sF = (cx<T>*)post_smem;
  cx<T>* sZ = sF + RX * RY;
  int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int tau = st[slot].tau;
  const cx<T>* ID = invd + (int64_t)tau * L.n;
  const cx<T>* fs = f + slot * vs;
  const cx<T>* zs = z + slot * vs;
  cx<T>* zo = zout + slot * vs;
  const cx<T>* zcs = zc + slot * vsc;
  const int cnx = (L.nx + 1) >> 1, cny = (L.ny + 1) >> 1;
  const int x0 = blockIdx.x * TX - FH, y0 = blockIdx.y * TY - FH;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int q = tid; q < RX * RY; q += nt) {
    int ry = q / RX, rx = q - ry * RX;
    int gx = x0 + rx, gy = y0 + ry;
    bool in = gx >= 0 && gx < L.nx && gy >= 0 && gy < L.ny;
    sF[q] = in ? fs[gy * L.nx + gx] : mk(T(0), T(0));
  }
  // z + P zc on the red cells of the region: the first half sweep overwrites the
  // black ones unread
  for (int q = tid; q < (RX / 2) * RY; q += nt) {
    const int ry = q / (RX / 2);
    const int gy = y0 + ry;
    int rx = 2 * (q - ry * (RX / 2));
    if ((x0 + rx + gy) & 1) ++rx;
    const int gx = x0 + rx;
    if (gx < 0 || gx >= L.nx || gy < 0 || gy >= L.ny) continue;
    sZ[ry * RX + rx] = zs[gy * L.nx + gx] + prolong_value(Cell{gx, gy, 0}, 2, 2, 1, cnx, cny, 1, mask, zcs);
  }
  __syncthreads();
  for (int hs = 0; hs < 4; ++hs) {
    const int color = (hs & 1) ? 0 : 1;  // black, red, black, red
    const int sh = hs + 1;
    const int w = RX - 2 * sh, hgt = RY - 2 * sh;
    const int wh = (w + 1) >> 1;
    for (int q = tid; q < wh * hgt; q += nt) {
      int yy = q / wh;
      int ry = sh + yy;
      int gy = y0 + ry;
      int rx0 = sh + 2 * (q - yy * wh);
      int gx = x0 + rx0;
      if (((gx + gy) & 1) != color) { ++gx; ++rx0; }
      if (rx0 >= RX - sh || gx < 0 || gx >= L.nx || gy < 0 || gy >= L.ny) continue;
      int r = ry * RX + rx0;
      int c = gy * L.nx + gx;
      cx<T> rhs = nb_sum_tile(L, Cell{gx, gy, 0}, r, RX, sZ, sF[r]);
      sZ[r] = ID[c] * rhs;
    }
    __syncthreads();
  }
  if (Zk) {
    z64* zk = Zk + slot * vsZk + (int64_t)(st[slot].k - 1) * zcol;
    const bool first = st[slot].cycles == 0;
    for (int q = tid; q < TX * TY; q += nt) {
      int yy = q / TX, xx = q - yy * TX;
      int gx = x0 + FH + xx, gy = y0 + FH + yy;
      if (gx < L.nx && gy < L.ny) {
        const int c = gy * L.nx + gx;
        const z64 ev = cvt<double>(sZ[(yy + FH) * RX + xx + FH]);
        zk[c] = first ? ev : (zk[c] + ev);
      }
    }
    return;
  }
  for (int q = tid; q < TX * TY; q += nt) {
    int yy = q / TX, xx = q - yy * TX;
    int gx = x0 + FH + xx, gy = y0 + FH + yy;
    if (gx < L.nx && gy < L.ny) zo[gy * L.nx + gx] = sZ[(yy + FH) * RX + xx + FH];
  }
}

// --------------------------------------------------------------------- small tiles by pairs
// The same two kernels for 8 x 8 tiles, and in complex64 16 x 16 ones, with a
// pair of cells (2 p, 2 p + 1) of the tile's region per thread: the pair's
// coefficients, right-hand side and iterate are loaded once, together, into
// registers. On the small levels these tiles are for, k_pre2d's time is
// latency: every half sweep waits for its faces and inverse diagonals after
// its barrier (4.4 us a launch in complex64, 7.6 us in complex128). In
// complex128 a 16 x 16 tile stays with k_pre2d, whose half sweeps pack the
// shrinking region's cells into fewer FP64 instructions.
// Cells outside the grid hold zero, which adds t * 0 for a missing neighbour;
// cells whose neighbours the region does not hold get values nothing reads
// (the region shrinks by one cell per half sweep).
template <typename T, int TX>
struct TilePair {
  static constexpr int RX = TX + 2 * FH, PX = RX / 2, NT = PX * RX;
  static constexpr int GUARD = RX + 2;               // cells read around the region
  static constexpr int ZN = RX * RX + 2 * GUARD;
  T x[3], yl[2], yh[2];
  cx<T> id[2], f[2], z[2];
  int ry, r, gx, gy, c;      // region row, region index, left cell and its flat index
  bool in[2];
  __device__ __forceinline__ void load(const LevelView<T>& L, const cx<T>* ID, const cx<T>* fs) {
    const int t = threadIdx.x;
    ry = t / PX;
    const int rx = 2 * (t - ry * PX);
    r = ry * RX + rx;
    gx = (int)blockIdx.x * TX - FH + rx;
    gy = (int)blockIdx.y * TX - FH + ry;
    c = gy * L.nx + gx;
    const bool row = gy >= 0 && gy < L.ny;
    const T* fx = L.fx + c + gy;
    const T* fy = L.fy + c;
    x[0] = x[1] = x[2] = T(0);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      in[h] = row && gx + h >= 0 && gx + h < L.nx;
      id[h] = in[h] ? ID[c + h] : mk(T(0), T(0));
      f[h] = in[h] ? fs[c + h] : mk(T(0), T(0));
      z[h] = mk(T(0), T(0));
      yl[h] = in[h] ? fy[h] : T(0);
      yh[h] = in[h] ? fy[L.nx + h] : T(0);
      if (in[h]) {
        x[h] = fx[h];
        x[h + 1] = fx[h + 1];
      }
    }
  }
  // s + sum t z_nb of cell h, in nb_sum's order; Z points at the region's cell 0
  __device__ __forceinline__ cx<T> nb(const cx<T>* Z, int h, cx<T> s) const {
    const cx<T> far = h ? Z[r + 2] : Z[r - 1];
    const cx<T> own = h ? z[0] : z[1];
    s = axpy(h ? x[1] : x[0], h ? own : far, s);
    s = axpy(h ? x[2] : x[1], h ? far : own, s);
    s = axpy(h ? yl[1] : yl[0], Z[r + h - RX], s);
    s = axpy(h ? yh[1] : yh[0], Z[r + h + RX], s);
    return s;
  }
  // half sweep of `color` on the rows sh .. RX - sh - 1 of the region
  __device__ __forceinline__ void gs(cx<T>* Z, int color, int sh, bool zero) {
    const int h = (gy + color) & 1;  // gx is even
    if (ry < sh || ry >= RX - sh || !(h ? in[1] : in[0])) return;
    cx<T> rhs = h ? f[1] : f[0];
    if (!zero) rhs = nb(Z, h, rhs);
    const cx<T> v = (h ? id[1] : id[0]) * rhs;
    if (h) z[1] = v;
    else z[0] = v;
    Z[r + h] = v;
  }
  __device__ __forceinline__ bool interior() const {
    const int rx = r - ry * RX;
    return ry >= FH && ry < FH + TX && rx >= FH && rx < FH + TX;
  }
};

template <typename T, int TX>
__global__ void __launch_bounds__(TilePair<T, TX>::NT) k_pre2d_pairs(LevelView<T> L, const SlotState* st,
                                                                    const cx<T>* __restrict__ invd, const z64* taus,
                                                                    const cx<T>* __restrict__ f, cx<T>* __restrict__ z,
                                                                    int64_t vs, cx<T>* __restrict__ fc, int64_t vsc) {
  using Tile = TilePair<T, TX>;
  pdl_enter();
  __shared__ cx<T> zmem[Tile::ZN];
  constexpr int NC = RED_RESIDUAL<T> ? 1 : 2;  // the pair's red cell, or both
  __shared__ cx<T> res[TX][NC * TX / 2];
  const int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int tau = st[slot].tau;
  const cx<T> sft = cvt<T>(taus[tau]);
  cx<T>* Z = zmem + Tile::GUARD;
  Tile q;
  q.load(L, invd + (int64_t)tau * L.n, f + slot * vs);
  const bool mine = q.interior();
  T d[NC], m[NC];
#pragma unroll
  for (int a = 0; a < NC; ++a) {
    const int h = NC == 1 ? q.gy & 1 : a;  // gx is even
    d[a] = m[a] = T(0);
    if (mine && (h ? q.in[1] : q.in[0])) {
      m[a] = L.mm[q.c + h];
      if (sizeof(T) == 8 && L.kd) d[a] = L.kd[q.c + h];
    }
  }
  for (int e = threadIdx.x; e < Tile::ZN; e += Tile::NT) zmem[e] = mk(T(0), T(0));
  __syncthreads();
  q.gs(Z, 0, 0, true);
  __syncthreads();
  q.gs(Z, 1, 1, false);
  __syncthreads();
  q.gs(Z, 0, 2, false);
  __syncthreads();
  q.gs(Z, 1, 3, false);
  __syncthreads();
  if (mine) {
    cx<T>* zs = z + slot * vs;
    const int yy = q.ry - FH, xx = q.r - q.ry * Tile::RX - FH;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (q.in[h]) zs[q.c + h] = q.z[h];
#pragma unroll
    for (int a = 0; a < NC; ++a) {
      const int h = NC == 1 ? q.gy & 1 : a;
      if (!(h ? q.in[1] : q.in[0])) continue;
      if (!(sizeof(T) == 8 && L.kd)) {
        const T x0 = h ? q.x[1] : q.x[0], x1 = h ? q.x[2] : q.x[1];
        d[a] = ((x0 + x1) + ((h ? q.yl[1] : q.yl[0]) + (h ? q.yh[1] : q.yh[0]))) + T(0);
      }
      res[yy][NC == 1 ? xx >> 1 : xx + a] =
          residual_of(h ? q.f[1] : q.f[0], h ? q.z[1] : q.z[0], mk(fmaT(sft.re, m[a], d[a]), mulT(sft.im, m[a])),
                      [&](cx<T> s0) { return q.nb(Z, h, s0); });
    }
  }
  __syncthreads();
  const int t = threadIdx.x;
  if (t >= (TX / 2) * (TX / 2)) return;
  const int Yl = t / (TX / 2), Xl = t - Yl * (TX / 2);
  const int X = blockIdx.x * (TX / 2) + Xl, Y = blockIdx.y * (TX / 2) + Yl;
  const int cnx = (L.nx + 1) >> 1, cny = (L.ny + 1) >> 1;
  if (X >= cnx || Y >= cny) return;
  cx<T> acc = mk(T(0), T(0));
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int a = child_first<T>(b); a < 2; a += child_step<T>)
      if (2 * X + a < L.nx && 2 * Y + b < L.ny) acc = acc + res[2 * Yl + b][NC == 1 ? Xl : 2 * Xl + a];
  fc[slot * vsc + (int64_t)Y * cnx + X] = acc;
}

template <typename T, int TX>
__global__ void __launch_bounds__(TilePair<T, TX>::NT)
    k_post2d_pairs(LevelView<T> L, uint32_t mask, const SlotState* st, const cx<T>* __restrict__ invd,
                   const cx<T>* __restrict__ f, const cx<T>* __restrict__ z, cx<T>* __restrict__ zout, int64_t vs,
                   const cx<T>* __restrict__ zc, int64_t vsc, z64* __restrict__ Zk, int64_t vsZk, int64_t zcol) {
  using Tile = TilePair<T, TX>;
  pdl_enter();
  __shared__ cx<T> zmem[Tile::ZN];
  const int slot = blockIdx.z;
  if (!slot_running(st, slot)) return;
  const int tau = st[slot].tau;
  cx<T>* Z = zmem + Tile::GUARD;
  Tile q;
  q.load(L, invd + (int64_t)tau * L.n, f + slot * vs);
  const int cnx = (L.nx + 1) >> 1, cny = (L.ny + 1) >> 1;
  for (int e = threadIdx.x; e < Tile::ZN; e += Tile::NT) zmem[e] = mk(T(0), T(0));
  // the red cell of the pair (the black one is overwritten unread)
  const int h = q.gy & 1;
  cx<T> v = mk(T(0), T(0));
  if (h ? q.in[1] : q.in[0])
    v = z[slot * vs + q.c + h] +
        prolong_value(Cell{q.gx + h, q.gy, 0}, 2, 2, 1, cnx, cny, 1, mask, zc + slot * vsc);
  __syncthreads();
  if (h) q.z[1] = v;
  else q.z[0] = v;
  Z[q.r + h] = v;
  __syncthreads();
  q.gs(Z, 1, 1, false);
  __syncthreads();
  q.gs(Z, 0, 2, false);
  __syncthreads();
  q.gs(Z, 1, 3, false);
  __syncthreads();
  q.gs(Z, 0, 4, false);
  if (!q.interior()) return;
  if (Zk) {
    z64* zk = Zk + slot * vsZk + (int64_t)(st[slot].k - 1) * zcol + q.c;
    const bool first = st[slot].cycles == 0;
#pragma unroll
    for (int b = 0; b < 2; ++b)
      if (q.in[b]) {
        const z64 ev = cvt<double>(q.z[b]);
        zk[b] = first ? ev : (zk[b] + ev);
      }
    return;
  }
  cx<T>* zo = zout + slot * vs + q.c;
#pragma unroll
  for (int b = 0; b < 2; ++b)
    if (q.in[b]) zo[b] = q.z[b];
}

// --------------------------------------------------------------------- tail
// The V-cycle of every level from `lt` down (levels small enough for one CTA)
// in one kernel: one block per slot, level vectors in shared memory,
// coefficients read through the cache. Same operations, in the same order, as
// the per-level kernels.
template <typename T>
__global__ void __launch_bounds__(TAIL_THREADS, 1) k_tail_vcycle(TailParams<T> P, const SlotState* st) {
  pdl_enter();
  int slot = blockIdx.x;
  if (!slot_running(st, slot)) return;
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ LevelView<T> SV[MAX_LEVELS];
  __shared__ const cx<T>* SI[MAX_LEVELS];
  cx<T>* sh = (cx<T>*)tail_smem;
  const int tau = st[slot].tau;
  const cx<T> sft = cvt<T>(P.taus[tau]);
  const int nt = blockDim.x, tid = threadIdx.x;
  // level views: coefficients staged in shared memory (one bulk copy) or read from global
  if (tid < P.nlev) {
    const TailLevel<T>& A = P.lev[tid];
    LevelView<T> v = A.L;
    const cx<T>* id = A.invd + (int64_t)tau * A.L.n;
    if (P.staged) {
      int nfx = (v.nx + 1) * v.ny * v.nz, nfy = v.nx * (v.ny + 1) * v.nz;
      int nfz = v.nz > 1 ? v.nx * v.ny * (v.nz + 1) : 0;
      T* base = (T*)(tail_smem + A.cbyte);
      v.fx = base;
      v.fy = base + nfx;
      v.fz = base + nfx + nfy;
      v.mm = base + nfx + nfy + nfz;
      int realn = nfx + nfy + nfz + v.n;
      realn = (realn + 3) & ~3;
      id = (const cx<T>*)(base + realn);
    }
    SV[tid] = v;
    SI[tid] = id;
  }
  if (P.staged && P.blob) {
    // one flat copy of this tau's coefficients of all tail levels
    const uint4* src = (const uint4*)(P.blob + (size_t)tau * P.blob_bytes);
    uint4* dst = (uint4*)(tail_smem + P.coef0);
    for (int q = tid; q < P.blob_bytes / 16; q += nt) dst[q] = src[q];
  }
  __syncthreads();
  if (P.staged && !P.blob) {
    for (int l = 0; l < P.nlev; ++l) {
      const TailLevel<T>& A = P.lev[l];
      const LevelView<T>& v = SV[l];
      int nfx = (v.nx + 1) * v.ny * v.nz, nfy = v.nx * (v.ny + 1) * v.nz;
      int nfz = v.nz > 1 ? v.nx * v.ny * (v.nz + 1) : 0;
      T* dfx = (T*)v.fx;
      for (int q = tid; q < nfx; q += nt) dfx[q] = A.L.fx[q];
      T* dfy = (T*)v.fy;
      for (int q = tid; q < nfy; q += nt) dfy[q] = A.L.fy[q];
      T* dfz = (T*)v.fz;
      for (int q = tid; q < nfz; q += nt) dfz[q] = A.L.fz[q];
      T* dmm = (T*)v.mm;
      for (int q = tid; q < v.n; q += nt) dmm[q] = A.L.mm[q];
      cx<T>* did = (cx<T>*)SI[l];
      const cx<T>* gid = A.invd + (int64_t)tau * v.n;
      for (int q = tid; q < v.n; q += nt) did[q] = gid[q];
    }
  }
  {
    const TailLevel<T>& A = P.lev[0];
    const cx<T>* fin = P.f_in + slot * P.vs;
    for (int c = tid; c < A.L.n; c += nt) sh[A.off + c] = fin[c];
  }
  __syncthreads();
  auto sweep = [&](int l, int color, int zs) {
    const LevelView<T> L = SV[l];  // a register copy: the loop's shared-memory stores cannot alias it
    cx<T>* F = sh + P.lev[l].off;
    cx<T>* Z = F + L.n;
    const cx<T>* ID = SI[l];
    int work = ((L.nx + 1) >> 1) * L.ny * L.nz;
    for (int t = tid; t < work; t += nt) {
      Cell p;
      int c;
      if (color_cell(L.nx, L.ny, L.nz, color, t, &p, &c)) Z[c] = gs_value(L, p, c, ID[c], F, Z, zs);
    }
    __syncthreads();
  };
  for (int l = 0; l + 1 < P.nlev; ++l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    for (int r = 0; r < 2; ++r) {
      sweep(l, 0, r == 0);
      sweep(l, 1, 0);
    }
    cx<T>* F = sh + A.off;
    cx<T>* Z = F + A.L.n;
    cx<T>* FC = sh + B.off;
    const LevelView<T> LA = SV[l];
    for (int C = tid; C < B.L.n; C += nt) {
      Cell pc = cell_of(C, B.L.nx, B.L.ny);
      FC[C] = restrict_value(LA, A.rx, A.ry, A.rz, pc.i, pc.j, pc.k, sft, F, Z);
    }
    __syncthreads();
  }
  {
    const TailLevel<T>& Cl = P.lev[P.nlev - 1];
    const cx<T>* F = sh + Cl.off;
    cx<T>* Z = sh + Cl.off + Cl.L.n;
    const cx<T>* Ainv = P.Ainv + (int64_t)tau * P.nc * P.nc;
    for (int r = tid; r < P.nc; r += nt) {
      Z[r] = coarse_sum<T>(P.nc, [&](int l) { return Ainv[l * P.nc + r] * F[l]; });
    }
    __syncthreads();
  }
  for (int l = P.nlev - 2; l >= 0; --l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    cx<T>* Z = sh + A.off + A.L.n;
    const cx<T>* ZC = sh + B.off + B.L.n;
    for (int t = tid; t < ((A.L.nx + 1) >> 1) * A.L.ny * A.L.nz; t += nt) {
      Cell p;
      int c;
      if (color_cell(A.L.nx, A.L.ny, A.L.nz, 0, t, &p, &c))
        Z[c] = Z[c] + prolong_value(p, A.rx, A.ry, A.rz, B.L.nx, B.L.ny, B.L.nz, P.mask, ZC);
    }
    __syncthreads();
    for (int r = 0; r < 2; ++r) {
      sweep(l, 1, 0);
      sweep(l, 0, 0);
    }
  }
  {
    const TailLevel<T>& A = P.lev[0];
    cx<T>* zout = P.z_out + slot * P.vs;
    const cx<T>* Z = sh + A.off + A.L.n;
    for (int c = tid; c < A.L.n; c += nt) zout[c] = Z[c];
  }
}

// --------------------------------------------------------------------- 2D tail
// The tail V-cycle for 2D levels halved in both axes, with the cells of every
// level owned in horizontal pairs: thread t owns cells 2t and 2t + 1 of the
// level it is on (one red, one black, as nx is even), and keeps their faces,
// storage, inverse diagonals, right-hand sides and iterates in registers for
// the whole visit of the level; only the iterates go through shared memory,
// for the neighbours. Each cell update performs the operations of gs_value,
// restrict_value and prolong_value in the same order as k_tail_vcycle.
template <typename T>
struct TailPair {
  int i0, j, c0;
  bool own;
  T fxa, fxb, fxc;           // x faces left of c0, between, right of c1
  T yl0, yh0, yl1, yh1;      // y faces of c0 and c1
  T m0, m1;
  cx<T> id0, id1, f0, f1, z0, z1;
};

template <typename T>
__device__ __forceinline__ void tail2d_load(const TailLevel<T>& A, const unsigned char* smem, const cx<T>* F, int t,
                                            int tau, TailPair<T>& q) {
  const int nx = A.L.nx, ny = A.L.ny;
  const int n = nx * ny;
  q.own = 2 * t < n;
  if (!q.own) return;
  q.c0 = 2 * t;
  q.j = q.c0 / nx;
  q.i0 = q.c0 - q.j * nx;
  const int nfx = (nx + 1) * ny, nfy = nx * (ny + 1);
  const T* fx = (const T*)(smem + A.cbyte);
  const T* fy = fx + nfx;
  const T* mm = fy + nfy;
  const cx<T>* id = (const cx<T>*)(fx + ((nfx + nfy + n + 3) & ~3));
  const int rx = q.j * (nx + 1) + q.i0;
  q.fxa = fx[rx];
  q.fxb = fx[rx + 1];
  q.fxc = fx[rx + 2];
  q.yl0 = fy[q.c0];
  q.yl1 = fy[q.c0 + 1];
  q.yh0 = fy[q.c0 + nx];
  q.yh1 = fy[q.c0 + nx + 1];
  q.m0 = mm[q.c0];
  q.m1 = mm[q.c0 + 1];
  q.id0 = id[q.c0];
  q.id1 = id[q.c0 + 1];
  q.f0 = F[q.c0];
  q.f1 = F[q.c0 + 1];
  (void)tau;
}

// half sweep of `color` on the owned cell of that colour
template <typename T>
__device__ __forceinline__ void tail2d_gs(TailPair<T>& q, int nx, int ny, cx<T>* Z, int color, int zs) {
  if (!q.own) return;
  const bool first = ((q.j & 1) == color);  // c0 = (i0 even, j) has colour j & 1
  if (first) {
    cx<T> rhs = q.f0;
    if (!zs) {
      if (q.i0 > 0) rhs = axpy(q.fxa, Z[q.c0 - 1], rhs);
      rhs = axpy(q.fxb, q.z1, rhs);
      if (q.j > 0) rhs = axpy(q.yl0, Z[q.c0 - nx], rhs);
      if (q.j < ny - 1) rhs = axpy(q.yh0, Z[q.c0 + nx], rhs);
    }
    q.z0 = q.id0 * rhs;
    Z[q.c0] = q.z0;
  } else {
    cx<T> rhs = q.f1;
    if (!zs) {
      rhs = axpy(q.fxb, q.z0, rhs);
      if (q.i0 + 1 < nx - 1) rhs = axpy(q.fxc, Z[q.c0 + 2], rhs);
      if (q.j > 0) rhs = axpy(q.yl1, Z[q.c0 + 1 - nx], rhs);
      if (q.j < ny - 1) rhs = axpy(q.yh1, Z[q.c0 + 1 + nx], rhs);
    }
    q.z1 = q.id1 * rhs;
    Z[q.c0 + 1] = q.z1;
  }
}

// f - (K + s M) z on cell h of the owned pair (residual_at with d the sum of the faces)
template <typename T>
__device__ __forceinline__ cx<T> tail2d_residual(const TailPair<T>& q, int nx, int ny, const cx<T>* Z, cx<T> s, int h) {
  const T zero = T(0);
  if (h == 0) {
    Faces<T> fa{q.fxa, q.fxb, q.yl0, q.yh0, zero, zero};
    const T d = fsum(fa);
    return residual_of(q.f0, q.z0, mk(fmaT(s.re, q.m0, d), mulT(s.im, q.m0)), [&](cx<T> nb) {
      if (q.i0 > 0) nb = axpy(q.fxa, Z[q.c0 - 1], nb);
      nb = axpy(q.fxb, q.z1, nb);
      if (q.j > 0) nb = axpy(q.yl0, Z[q.c0 - nx], nb);
      if (q.j < ny - 1) nb = axpy(q.yh0, Z[q.c0 + nx], nb);
      return nb;
    });
  } else {
    Faces<T> fa{q.fxb, q.fxc, q.yl1, q.yh1, zero, zero};
    const T d = fsum(fa);
    return residual_of(q.f1, q.z1, mk(fmaT(s.re, q.m1, d), mulT(s.im, q.m1)), [&](cx<T> nb) {
      nb = axpy(q.fxb, q.z0, nb);
      if (q.i0 + 1 < nx - 1) nb = axpy(q.fxc, Z[q.c0 + 2], nb);
      if (q.j > 0) nb = axpy(q.yl1, Z[q.c0 + 1 - nx], nb);
      if (q.j < ny - 1) nb = axpy(q.yh1, Z[q.c0 + 1 + nx], nb);
      return nb;
    });
  }
}

template <typename T>
__global__ void __launch_bounds__(TAIL_THREADS, 1) k_tail2d(TailParams<T> P, const SlotState* st) {
  pdl_enter();
  const int slot = blockIdx.x;
  if (!slot_running(st, slot)) return;
  extern __shared__ __align__(16) unsigned char t2_smem[];
  cx<T>* sh = (cx<T>*)t2_smem;
  const int tau = st[slot].tau;
  const cx<T> sft = cvt<T>(P.taus[tau]);
  const int nt = blockDim.x, tid = threadIdx.x;
  {
    const uint4* src = (const uint4*)(P.blob + (size_t)tau * P.blob_bytes);
    uint4* dst = (uint4*)(t2_smem + P.coef0);
    for (int q = tid; q < P.blob_bytes / 16; q += nt) dst[q] = src[q];
    const cx<T>* ag = P.Ainv + (int64_t)tau * P.nc * P.nc;
    cx<T>* as = (cx<T>*)(t2_smem + P.ainv_off);
    for (int q = tid; q < P.nc * P.nc; q += nt) as[q] = ag[q];
    const TailLevel<T>& A = P.lev[0];
    const cx<T>* fin = P.f_in + slot * P.vs;
    for (int c = tid; c < A.L.n; c += nt) sh[A.off + c] = fin[c];
  }
  __syncthreads();
  TailPair<T> q;
  // ---- down
  for (int l = 0; l + 1 < P.nlev; ++l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    const int nx = A.L.nx, ny = A.L.ny;
    cx<T>* F = sh + A.off;
    cx<T>* Z = F + A.L.n;
    tail2d_load(A, t2_smem, F, tid, tau, q);
    for (int r = 0; r < 2; ++r) {
      tail2d_gs(q, nx, ny, Z, 0, r == 0);
      __syncthreads();
      tail2d_gs(q, nx, ny, Z, 1, 0);
      __syncthreads();
    }
    // restriction: the pair in row 2J sums its residuals (in complex128 its red
    // cell's is all), the pair in row 2J + 1 adds its own onto that (the child
    // order of restrict_value)
    const int cnx = B.L.nx;
    cx<T>* FC = sh + B.off;
    cx<T>* S = FC + B.L.n;  // the coarse iterate's storage, free until its first sweep
    constexpr int NC = RED_RESIDUAL<T> ? 1 : 2;
    cx<T> res[NC];
    if (q.own) {
#pragma unroll
      for (int a = 0; a < NC; ++a) res[a] = tail2d_residual(q, nx, ny, Z, sft, NC == 1 ? q.j & 1 : a);
      if ((q.j & 1) == 0) {
        cx<T> acc = mk(T(0), T(0));
#pragma unroll
        for (int a = 0; a < NC; ++a) acc = acc + res[a];
        S[(q.j >> 1) * cnx + (q.i0 >> 1)] = acc;
      }
    }
    __syncthreads();
    if (q.own && (q.j & 1)) {
      const int C = (q.j >> 1) * cnx + (q.i0 >> 1);
      cx<T> acc = S[C];
#pragma unroll
      for (int a = 0; a < NC; ++a) acc = acc + res[a];
      FC[C] = acc;
    }
    __syncthreads();
  }
  {
    const TailLevel<T>& Cl = P.lev[P.nlev - 1];
    const cx<T>* F = sh + Cl.off;
    cx<T>* Z = sh + Cl.off + Cl.L.n;
    // the products by all threads, in place of the staged inverse; then two
    // threads per row, one for each part, add them in order
    cx<T>* as = (cx<T>*)(t2_smem + P.ainv_off);
    const int nc = P.nc;
    for (int e = tid; e < nc * nc; e += nt) as[e] = as[e] * F[e / nc];
    __syncthreads();
    for (int e = tid; e < 2 * nc; e += nt) {
      T acc = T(0);
#pragma unroll 4
      for (int l = 0; l < nc; ++l) acc = acc + ((const T*)as)[2 * l * nc + e];
      ((T*)Z)[e] = acc;
    }
    __syncthreads();
  }
  if (P.nlev == 1) {
    const TailLevel<T>& A = P.lev[0];
    cx<T>* zout = P.z_out + slot * P.vs;
    const cx<T>* Z = sh + A.off + A.L.n;
    for (int c = tid; c < A.L.n; c += nt) zout[c] = Z[c];
    return;
  }
  // ---- up
  for (int l = P.nlev - 2; l >= 0; --l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    const int nx = A.L.nx, ny = A.L.ny;
    cx<T>* F = sh + A.off;
    cx<T>* Z = F + A.L.n;
    const cx<T>* ZC = sh + B.off + B.L.n;
    const int cnx = B.L.nx, cny = B.L.ny;
    tail2d_load(A, t2_smem, F, tid, tau, q);
    if (q.own) {
      auto get = [&](int X, int Y, int) { return ZC[Y * cnx + X]; };
      // the red cell of the pair
      const int h = q.j & 1;
      const cx<T> v = Z[q.c0 + h] + prolong_value_at<T>(Cell{q.i0 + h, q.j, 0}, 2, 2, 1, cnx, cny, 1, P.mask, get);
      (h ? q.z1 : q.z0) = v;
      Z[q.c0 + h] = v;
    }
    __syncthreads();
    for (int r = 0; r < 2; ++r) {
      tail2d_gs(q, nx, ny, Z, 1, 0);
      __syncthreads();
      tail2d_gs(q, nx, ny, Z, 0, 0);
      __syncthreads();
    }
  }
  if (q.own) {
    cx<T>* zout = P.z_out + slot * P.vs;
    zout[q.c0] = q.z0;
    zout[q.c0 + 1] = q.z1;
  }
}

// --------------------------------------------------------------------- tail by pairs
// The tail V-cycle for any levels (2D or 3D, odd sides, any coarsening) of at
// most TAILP_THREADS pairs of cells each: thread t owns the pair (2 p, 2 p + 1)
// of one row and keeps its coefficients, right-hand side and iterate in
// registers for the whole visit of the level, so a half sweep is a handful of
// shared-memory reads and 16 multiply-adds per thread. k_tail_vcycle, which
// finds its cells again in every half sweep, sums the residuals of a coarse
// cell one after another and reads the coarsest inverse row by row, was bound
// by those chains: 16 us for 8^3 and 4^3 cells in complex64.
// The residuals go through shared memory and are added per coarse cell in
// restrict_value's order; the coarsest product's terms are formed by all
// threads (from coalesced reads, the inverse being transposed) and added per
// row in order: the bits are k_tail_vcycle's.
// PART 1 and 2 are its way down and its way up, with k_coarse_solve between
// them. In complex128 one SM's FP64 units take 17 us for the product of a
// coarsest level of 105 cells (11 for the terms, 7 for the sums; 30 us the whole
// tail of 45 x 53 x 37), more than two launches and the product over the chip
// (6.4 + 6.5 + 5.5 us).
template <typename T>
struct PairCell {  // the pair's coefficients: x faces left, inside, right; y and z faces below and above each cell
  T x[3], yl[2], yh[2], zl[2], zh[2], m[2];
  cx<T> id[2], f[2], z[2];
  int c0, i0, j, k;
  bool own, right;
};

template <typename T>
__device__ __forceinline__ void pair_load(const TailLevel<T>& A, int tau, const cx<T>* F, int t, PairCell<T>& q) {
  const LevelView<T>& L = A.L;
  const int npx = (L.nx + 1) >> 1;
  const int row = t / npx;
  q.own = row < L.ny * L.nz;
  if (!q.own) return;
  q.i0 = 2 * (t - row * npx);
  q.k = row / L.ny;
  q.j = row - q.k * L.ny;
  q.c0 = row * L.nx + q.i0;
  q.right = q.i0 + 1 < L.nx;
  const cx<T>* id = A.invd + (int64_t)tau * L.n + q.c0;
  const T* fx = L.fx + q.c0 + row;
  const T* fy = L.fy + q.c0 + q.k * L.nx;
  const T* fz = L.fz + q.c0;
  const int sxy = L.nx * L.ny;
  q.x[0] = fx[0];
  q.x[1] = fx[1];
  q.x[2] = q.right ? fx[2] : T(0);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool on = h == 0 || q.right;
    q.id[h] = on ? id[h] : mk(T(0), T(0));
    q.f[h] = on ? F[q.c0 + h] : mk(T(0), T(0));
    q.yl[h] = on ? fy[h] : T(0);
    q.yh[h] = on ? fy[L.nx + h] : T(0);
    q.zl[h] = on && L.nz > 1 ? fz[h] : T(0);
    q.zh[h] = on && L.nz > 1 ? fz[sxy + h] : T(0);
    q.m[h] = on ? L.mm[q.c0 + h] : T(0);
  }
}

// s + sum t z_nb of cell h of the pair, in nb_sum's order; a neighbour outside
// the grid adds t * 0
template <typename T>
__device__ __forceinline__ cx<T> pair_nb(const PairCell<T>& q, const LevelView<T>& L, const cx<T>* Z, int h, cx<T> s) {
  const int c = q.c0 + h, sxy = L.nx * L.ny;
  const cx<T> none = mk(T(0), T(0));
  const cx<T> far = h ? (q.i0 + 2 < L.nx ? Z[c + 1] : none) : (q.i0 > 0 ? Z[c - 1] : none);
  const cx<T> own = h ? q.z[0] : q.z[1];
  s = axpy(h ? q.x[1] : q.x[0], h ? own : far, s);
  s = axpy(h ? q.x[2] : q.x[1], h ? far : own, s);
  s = axpy(h ? q.yl[1] : q.yl[0], q.j > 0 ? Z[c - L.nx] : none, s);
  s = axpy(h ? q.yh[1] : q.yh[0], q.j < L.ny - 1 ? Z[c + L.nx] : none, s);
  if (L.nz > 1) {
    s = axpy(h ? q.zl[1] : q.zl[0], q.k > 0 ? Z[c - sxy] : none, s);
    s = axpy(h ? q.zh[1] : q.zh[0], q.k < L.nz - 1 ? Z[c + sxy] : none, s);
  }
  return s;
}

template <typename T>
__device__ __forceinline__ void pair_gs(PairCell<T>& q, const LevelView<T>& L, cx<T>* Z, int color, bool zero) {
  const int h = (q.j + q.k + color) & 1;
  if (!q.own || (h && !q.right)) return;
  cx<T> rhs = h ? q.f[1] : q.f[0];
  if (!zero) rhs = pair_nb(q, L, Z, h, rhs);
  const cx<T> v = (h ? q.id[1] : q.id[0]) * rhs;
  if (h) q.z[1] = v;
  else q.z[0] = v;
  Z[q.c0 + h] = v;
}

template <typename T, int NT, int PART = 0>
__global__ void __launch_bounds__(NT, 1) k_tail_pairs(TailParams<T> P, const SlotState* st) {
  pdl_enter();
  const int slot = blockIdx.x;
  if (!slot_running(st, slot)) return;
  extern __shared__ __align__(16) unsigned char tp_smem[];
  cx<T>* sh = (cx<T>*)tp_smem;
  cx<T>* R = sh + P.roff;  // residuals of a level, or terms of the coarsest product
  const int tau = st[slot].tau, t = threadIdx.x;
  const cx<T> sft = cvt<T>(P.taus[tau]);
  const cx<T> none = mk(T(0), T(0));
  PairCell<T> q;
  if (PART != 2) {
    const TailLevel<T>& A = P.lev[0];
    const cx<T>* fin = P.f_in + slot * P.vs;
    if (P.nlev > 1) {
      pair_load(A, tau, fin, t, q);
      if (q.own) {
        sh[A.off + q.c0] = q.f[0];
        if (q.right) sh[A.off + q.c0 + 1] = q.f[1];
      }
    } else {
      for (int c = t; c < A.L.n; c += NT) sh[A.off + c] = fin[c];
    }
  }
  for (int l = 0; PART != 2 && l + 1 < P.nlev; ++l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    const LevelView<T>& L = A.L;
    cx<T>* F = sh + A.off;
    cx<T>* Z = F + L.n;
    if (l > 0) pair_load(A, tau, F, t, q);
    q.z[0] = q.z[1] = none;
    pair_gs(q, L, Z, 0, true);
    __syncthreads();
    pair_gs(q, L, Z, 1, false);
    __syncthreads();
    pair_gs(q, L, Z, 0, false);
    __syncthreads();
    pair_gs(q, L, Z, 1, false);
    __syncthreads();
    if (PART == 1 && q.own) {
      const int h = (q.j + q.k) & 1;  // the way up reads the red cells alone
      if (h == 0 || q.right) A.gz[(int64_t)slot * L.n + q.c0 + h] = h ? q.z[1] : q.z[0];
    }
    constexpr int NC = RED_RESIDUAL<T> ? 1 : 2;  // the pair's red cell, or both
#pragma unroll
    for (int a = 0; a < NC; ++a) {
      const int h = NC == 1 ? (q.j + q.k) & 1 : a;
      if (!q.own || (h && !q.right)) continue;
      const T x0 = h ? q.x[1] : q.x[0], x1 = h ? q.x[2] : q.x[1];
      const T yl = h ? q.yl[1] : q.yl[0], yh = h ? q.yh[1] : q.yh[0];
      const T zl = h ? q.zl[1] : q.zl[0], zh = h ? q.zh[1] : q.zh[0], m = h ? q.m[1] : q.m[0];
      const T d = ((x0 + x1) + (yl + yh)) + (zl + zh);
      R[q.c0 + h] = residual_of(h ? q.f[1] : q.f[0], h ? q.z[1] : q.z[0], mk(fmaT(sft.re, m, d), mulT(sft.im, m)),
                                [&](cx<T> s0) { return pair_nb(q, L, Z, h, s0); });
    }
    __syncthreads();
    cx<T>* FC = sh + B.off;
    for (int C = t; C < B.L.n; C += NT) {
      const Cell p = cell_of(C, B.L.nx, B.L.ny);
      cx<T> acc = none;
      for (int c = 0; c < A.rz; ++c)
        for (int b = 0; b < A.ry; ++b)
          for (int a = child_first<T>(A.rx * p.i + A.ry * p.j + b + A.rz * p.k + c); a < A.rx; a += child_step<T>) {
            const int i = A.rx * p.i + a, j = A.ry * p.j + b, k = A.rz * p.k + c;
            if (i < L.nx && j < L.ny && k < L.nz) acc = acc + R[(k * L.ny + j) * L.nx + i];
          }
      FC[C] = acc;
      if (PART == 1) B.gf[(int64_t)slot * B.L.n + C] = acc;
    }
    __syncthreads();
  }
  if (PART == 1) return;
  if (PART == 0) {
    const TailLevel<T>& Cl = P.lev[P.nlev - 1];
    const cx<T>* F = sh + Cl.off;
    cx<T>* Z = sh + Cl.off + Cl.L.n;
    const cx<T>* Ainv = P.Ainv + (int64_t)tau * P.nc * P.nc;
    const int nc = P.nc, cols = min(nc, P.rlen / nc);
    if (P.nlev == 1) __syncthreads();
    // the terms by all threads; then two threads per row, one for each part of
    // the complex sum, add them in order (nc <= NT)
    T acc[2] = {T(0), T(0)};
    for (int l0 = 0; l0 < nc; l0 += cols) {
      const int lc = min(cols, nc - l0);
#pragma unroll 4
      for (int e = t; e < lc * nc; e += NT) R[e] = Ainv[l0 * nc + e] * F[l0 + e / nc];
      __syncthreads();
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (t + h * NT < 2 * nc) {
#pragma unroll 8
          for (int l = 0; l < lc; ++l) acc[h] = acc[h] + ((const T*)R)[2 * l * nc + t + h * NT];
        }
      __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (t + h * NT < 2 * nc) {
        ((T*)Z)[t + h * NT] = acc[h];
        if (P.nlev == 1) ((T*)(P.z_out + slot * P.vs))[t + h * NT] = acc[h];
      }
    __syncthreads();
  }
  for (int l = P.nlev - 2; l >= 0; --l) {
    const TailLevel<T>& A = P.lev[l];
    const TailLevel<T>& B = P.lev[l + 1];
    const LevelView<T>& L = A.L;
    cx<T>* Z = sh + A.off + L.n;
    const cx<T>* ZC = PART == 2 && l == P.nlev - 2 ? B.gz + (int64_t)slot * B.L.n : sh + B.off + B.L.n;
    pair_load(A, tau, PART == 2 ? A.gf + (int64_t)slot * L.n : sh + A.off, t, q);
    q.z[0] = q.z[1] = none;
    const int h = (q.j + q.k) & 1;  // the red cell: the black one is overwritten unread
    if (q.own && (h == 0 || q.right)) {
      const cx<T> v = (PART == 2 ? A.gz + (int64_t)slot * L.n : Z)[q.c0 + h] +
                      prolong_value(Cell{q.i0 + h, q.j, q.k}, A.rx, A.ry, A.rz, B.L.nx, B.L.ny, B.L.nz, P.mask, ZC);
      if (h) q.z[1] = v;
      else q.z[0] = v;
      Z[q.c0 + h] = v;
    }
    __syncthreads();
    for (int r = 0; r < 2; ++r) {
      pair_gs(q, L, Z, 1, false);
      __syncthreads();
      pair_gs(q, L, Z, 0, false);
      __syncthreads();
    }
  }
  if (P.nlev > 1 && q.own) {
    cx<T>* zout = P.z_out + slot * P.vs;
    zout[q.c0] = q.z[0];
    if (q.right) zout[q.c0 + 1] = q.z[1];
  }
}

int tail_pairs_threads(const std::vector<LevelHost>& Ls, int lt, bool fp64) {
  int64_t most = Ls.back().n;  // the coarsest product: a thread per row
  for (size_t l = lt; l + 1 < Ls.size(); ++l)
    most = std::max<int64_t>(most, (int64_t)((Ls[l].nx + 1) / 2) * Ls[l].ny * Ls[l].nz);
  return most <= 512 ? 512 : (most <= 1024 && !fp64 ? 1024 : 0);
}

bool tail2d_ok(const std::vector<LevelHost>& Ls, int lt) {
  const int nl = (int)Ls.size();
  if (Ls[nl - 1].nz != 1) return false;
  for (int l = lt; l + 1 < nl; ++l) {
    const LevelHost& A = Ls[l];
    if (A.nz != 1 || A.rx != 2 || A.ry != 2 || A.nx % 2 || A.ny % 2 || A.n > 2 * TAIL_THREADS) return false;
  }
  return true;
}

// --------------------------------------------------------------------- coarsest
// Gauss-Jordan inversion with partial pivoting of the n x n complex matrices
// K + tau M of the coarsest level (n <= MAX_COARSE), in place: the columns
// already eliminated hold the columns of the inverse that have left the
// identity. With d the pivot, column `col` of the step:
//   pivot row:   p_l = (1/d) a_l,  p_col = 1/d
//   other rows:  a_l - f p_l with f the row's entry in column col; -f p_col there
// The inverse's column of position c is that of the row that was swapped into c.
// 1/d, its two parts divided by two lanes of a warp (an FP64 division is a
// sequence of dependent instructions that costs a whole warp its issue slots)
__device__ __forceinline__ void gj_recip(z64 d, int lane, z64* out) {
  const double den = abs2(d);
  if (lane < 2) ((double*)out)[lane] = den > 0.0 ? (lane ? -d.im : d.re) / den : 0.0;
}

// Pivot candidates are compared as integers (the order of non-negative
// doubles; NaN as 0), which leaves the FP64 pipe to the updates: the larger
// |v|^2 wins, the smaller row on a tie.
__device__ __forceinline__ unsigned long long gj_key(z64 v) {
  const unsigned long long k = (unsigned long long)__double_as_longlong(abs2(v));
  return k > 0x7ff0000000000000ull ? 0ull : k;
}
__device__ __forceinline__ void gj_better(unsigned long long ov, int oi, unsigned long long* v, int* i) {
  if (ov > *v || (ov == *v && oi < *i)) {
    *v = ov;
    *i = oi;
  }
}
__device__ __forceinline__ void gj_warp_best(unsigned long long* v, int* i) {
  for (int d = 16; d > 0; d >>= 1) {
    const unsigned long long ov = __shfl_xor_sync(0xffffffffu, *v, d);
    const int oi = __shfl_xor_sync(0xffffffffu, *i, d);
    gj_better(ov, oi, v, i);
  }
}

// One elimination step over the whole chip. One block per tau, as this was
// before, is bound by one SM's FP64 rate (2 fused multiply-adds a clock) and
// by its reads of the matrix: 260 ms for four 625 x 625 matrices. Here a block
// updates a 32 x 8 tile, read from S and written to D (the two buffers
// alternate, so a step needs no barrier inside the grid). Every block finds
// the pivot itself from the step's column, which the step before left
// contiguous in `cin`. The matrix is banded (5 or 7 diagonals): rows whose
// entry in the column is zero and tiles whose pivot row is zero are copied.
// A tile is 32 columns by 8 rows, one row per warp.
constexpr int GJ_T = 32;
__global__ void __launch_bounds__(256) k_gj_step(const z64* __restrict__ S, z64* __restrict__ D,
                                                 const z64* __restrict__ cin, z64* __restrict__ cout,
                                                 int32_t* __restrict__ piv, int n, int col, int* singular) {
  pdl_enter();
  const int q = blockIdx.z, lane = threadIdx.x, w = threadIdx.y, t = w * 32 + lane;
  const z64* a = S + (int64_t)q * n * n;
  z64* o = D + (int64_t)q * n * n;
  const z64* cc = cin + (int64_t)q * n;
  __shared__ unsigned long long sv[8];
  __shared__ int si[8];
  __shared__ z64 srd;
  const int l = blockIdx.x * GJ_T + lane, r = blockIdx.y * 8 + w;
  // the tile's rows, before the swap (their latency overlaps the search)
  const z64 v = l < n && r < n ? a[(int64_t)r * n + l] : mk(0.0, 0.0);
  const z64 f = r < n ? cc[r] : mk(0.0, 0.0);
  unsigned long long bv = 0ull;
  int bi = INT_MAX;
  for (int e = col + t; e < n; e += 256) gj_better(gj_key(cc[e]), e, &bv, &bi);
  gj_warp_best(&bv, &bi);
  if (lane == 0) {
    sv[w] = bv;
    si[w] = bi;
  }
  __syncthreads();
  bv = sv[0];
  bi = si[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) gj_better(sv[k], si[k], &bv, &bi);
  const int pr = bi;
  if (blockIdx.x == 0 && blockIdx.y == 0 && t == 0) {
    piv[(int64_t)q * n + col] = pr;
    if (bv == 0ull) *singular = 1;
  }
  z64 p = l < n ? a[(int64_t)pr * n + l] : mk(0.0, 0.0);
  if (w == 0) gj_recip(cc[pr], lane, &srd);
  __syncthreads();
  const z64 rd = srd;
  const bool any = __any_sync(0xffffffffu, l == col || p.re != 0.0 || p.im != 0.0);
  if (any && l < n) p = l == col ? rd : rd * p;
  if (l >= n || r >= n) return;
  z64 x = v, fr = f;
  if (r == pr && pr != col) {
    x = a[(int64_t)col * n + l];
    fr = cc[col];
  }
  if (l == col) x = mk(0.0, 0.0);
  if (r == col) x = p;
  else if (any && (fr.re != 0.0 || fr.im != 0.0)) x = x - fr * p;
  o[(int64_t)r * n + l] = x;
  if (l == col + 1) cout[(int64_t)q * n + r] = x;
}

// The same step for matrices of many tiles, in place and in two launches: one
// block per tau finds the pivot, scales its row into `row` and exchanges the
// rows; then the tiles update the rows whose entry in the column is not zero
// and leave the others alone (k_gj_step copies them, and its blocks, several
// rounds of them, each wait for the pivot search and the division: 22 us a
// step of four 729 x 729 matrices).
__global__ void __launch_bounds__(1024) k_gj_pivot(z64* __restrict__ A, z64* __restrict__ row, z64* __restrict__ cin,
                                                   int32_t* __restrict__ piv, int n, int col, int* singular) {
  pdl_enter();
  const int q = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  z64* a = A + (int64_t)q * n * n;
  z64* cc = cin + (int64_t)q * n;
  __shared__ unsigned long long sv[32];
  __shared__ int si[32];
  __shared__ int spr;
  __shared__ z64 srd;
  unsigned long long bv = 0ull;
  int bi = INT_MAX;
  z64 oc = mk(0.0, 0.0);  // the row at position col before the exchange
  if (t < n) {
    oc = a[(int64_t)col * n + t];
    if (t >= col) gj_better(gj_key(cc[t]), t, &bv, &bi);
  }
  gj_warp_best(&bv, &bi);
  if (lane == 0) {
    sv[w] = bv;
    si[w] = bi;
  }
  __syncthreads();
  if (w == 0) {
    bv = lane < (int)(blockDim.x >> 5) ? sv[lane] : 0ull;
    bi = lane < (int)(blockDim.x >> 5) ? si[lane] : INT_MAX;
    gj_warp_best(&bv, &bi);
    gj_recip(cc[bi], lane, &srd);
    __syncwarp();
    if (lane == 0) {
      spr = bi;
      piv[(int64_t)q * n + col] = bi;
      if (bv == 0ull) *singular = 1;
      if (bi != col) cc[bi] = cc[col];  // the exchanged row's factor
    }
  }
  __syncthreads();
  if (t >= n) return;
  const int pr = spr;
  const z64 x = pr == col ? oc : a[(int64_t)pr * n + t];
  const z64 p = t == col ? srd : ((x.re != 0.0 || x.im != 0.0) ? srd * x : x);
  if (pr != col) a[(int64_t)pr * n + t] = oc;
  a[(int64_t)col * n + t] = p;
  row[(int64_t)q * n + t] = p;
}

__global__ void __launch_bounds__(256) k_gj_update(z64* __restrict__ A, const z64* __restrict__ row,
                                                   const z64* __restrict__ cin, z64* __restrict__ cout, int n,
                                                   int col) {
  pdl_enter();
  const int q = blockIdx.z, lane = threadIdx.x, w = threadIdx.y;
  z64* a = A + (int64_t)q * n * n;
  const z64* cc = cin + (int64_t)q * n;
  const int l = blockIdx.x * GJ_T + lane, r0 = blockIdx.y * GJ_T;
  const bool next = (int)blockIdx.x == (col + 1) / GJ_T;  // the tile column that holds the next step's column
  const z64 p = l < n ? row[(int64_t)q * n + l] : mk(0.0, 0.0);
  const bool any = __any_sync(0xffffffffu, p.re != 0.0 || p.im != 0.0);
  if (!any && !next) return;
  z64 f[GJ_T / 8], v[GJ_T / 8];
  bool on[GJ_T / 8];
#pragma unroll
  for (int h = 0; h < GJ_T / 8; ++h) {
    const int r = r0 + w + 8 * h;
    f[h] = r < n && r != col ? cc[r] : mk(0.0, 0.0);
  }
#pragma unroll
  for (int h = 0; h < GJ_T / 8; ++h) {
    const int r = r0 + w + 8 * h;
    on[h] = any && (f[h].re != 0.0 || f[h].im != 0.0);
    v[h] = l < n && r < n && (on[h] || next) ? a[(int64_t)r * n + l] : mk(0.0, 0.0);
  }
#pragma unroll
  for (int h = 0; h < GJ_T / 8; ++h) {
    const int r = r0 + w + 8 * h;
    if (l >= n || r >= n) continue;
    z64 x = v[h];
    if (on[h]) {
      if (l == col) x = mk(0.0, 0.0);
      x = x - f[h] * p;
      a[(int64_t)r * n + l] = x;
    }
    if (l == col + 1) cout[(int64_t)q * n + r] = x;
  }
}

// The inverse in the cycle precision, transposed (Ainv[l][r], so that the
// threads that own the rows of a product read consecutive values) and with its
// columns put back in the order of the rows before pivoting.
template <typename T>
__global__ void __launch_bounds__(256) k_gj_finish(const z64* __restrict__ S, const int32_t* __restrict__ piv,
                                                   cx<T>* __restrict__ out, int n) {
  __shared__ int org[MAX_COARSE];
  __shared__ cx<T> tile[GJ_T][GJ_T + 1];
  const int q = blockIdx.z, lane = threadIdx.x, w = threadIdx.y, t = w * 32 + lane;
  const int32_t* pv = piv + (int64_t)q * n;
  int moved = 0;
  for (int c = t; c < n; c += 256) {
    org[c] = c;
    moved |= pv[c] != c;
  }
  if (__syncthreads_or(moved)) {
    if (t == 0)
      for (int c = 0; c < n; ++c) {
        const int pr = pv[c], k = org[c];
        org[c] = org[pr];
        org[pr] = k;
      }
    __syncthreads();
  }
  const int l0 = blockIdx.x * GJ_T, r0 = blockIdx.y * GJ_T;
#pragma unroll
  for (int h = 0; h < GJ_T / 8; ++h) {
    const int r = r0 + w + 8 * h;
    if (r < n && l0 + lane < n) tile[w + 8 * h][lane] = cvt<T>(S[((int64_t)q * n + r) * n + l0 + lane]);
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < GJ_T / 8; ++h) {
    const int l = l0 + w + 8 * h;
    if (l < n && r0 + lane < n) out[((int64_t)q * n + org[l]) * n + r0 + lane] = tile[lane][w + 8 * h];
  }
}

// Up to GJ_SMALL unknowns: the whole inversion in one block per tau, the
// matrix in shared memory, one warp searching the pivot. A step costs three
// block barriers (about 0.5 us) against the 2.5 us of a launch; from about 40
// unknowns on, the FP64 rate of one SM costs more than the launches.
constexpr int GJ_SMALL = 40;
template <typename T>
__global__ void __launch_bounds__(512) k_gj_small(const z64* __restrict__ A, cx<T>* __restrict__ out, int n,
                                                  int* singular) {
  __shared__ z64 m[GJ_SMALL * GJ_SMALL];
  __shared__ int org[GJ_SMALL];
  __shared__ int spr;
  __shared__ z64 srd;
  const int t = threadIdx.x, q = blockIdx.x, nn = n * n;
  constexpr int PER = (GJ_SMALL * GJ_SMALL + 511) / 512;
  for (int e = t; e < nn; e += 512) m[e] = A[(int64_t)q * nn + e];
  if (t < n) org[t] = t;
  __syncthreads();
  for (int col = 0; col < n; ++col) {
    if (t < 32) {
      unsigned long long bv = 0ull;
      int bi = INT_MAX;
      for (int r = col + t; r < n; r += 32) gj_better(gj_key(m[r * n + col]), r, &bv, &bi);
      gj_warp_best(&bv, &bi);
      gj_recip(m[bi * n + col], t, &srd);
      if (t == 0) {
        spr = bi;
        if (bv == 0ull) *singular = 1;
        const int k = org[col];
        org[col] = org[bi];
        org[bi] = k;
      }
    }
    __syncthreads();
    const int pr = spr;
    const z64 rd = srd;
    z64 x[PER];
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      const int e = t + 512 * h;
      if (e >= nn) break;
      const int r = e / n, l = e - r * n;
      const int sr = r == col ? pr : (r == pr ? col : r);
      const z64 p = l == col ? rd : rd * m[pr * n + l];
      const z64 f = m[sr * n + col];
      x[h] = l == col ? mk(0.0, 0.0) : m[sr * n + l];
      if (r == col) x[h] = p;
      else if (f.re != 0.0 || f.im != 0.0) x[h] = x[h] - f * p;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      const int e = t + 512 * h;
      if (e < nn) m[e] = x[h];
    }
    __syncthreads();
  }
  for (int e = t; e < nn; e += 512) {
    const int l = e / n, r = e - l * n;
    out[((int64_t)q * n + org[l]) * n + r] = cvt<T>(m[r * n + l]);
  }
}

// z = Ainv[tau] f on the coarsest level when it is a level of its own (Ainv
// transposed): a block owns coarse_rows rows. All of its threads form the
// products of those rows, from coalesced reads; then one warp adds each row's
// products in the order of the tail kernels' loop (coarse_sum), so the bits are
// theirs. Complex128 adds in partial sums (a solve of 18 x 22 x 24 cells, 297 of
// them on the coarsest level, 57.5 -> 54.0 ms). The single-block tail reads the
// n x n inverse through one SM.
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_solve(const cx<T>* __restrict__ Ainv, int n, const SlotState* st,
                                                      const cx<T>* __restrict__ f, cx<T>* __restrict__ z,
                                                      int64_t vs) {
  pdl_enter();
  constexpr int RB = coarse_rows<T>();
  extern __shared__ __align__(16) unsigned char cs_smem[];
  cx<T>* pr = (cx<T>*)cs_smem;
  const int slot = blockIdx.y;
  if (!slot_running(st, slot)) return;
  const int r0 = blockIdx.x * RB;
  const cx<T>* a = Ainv + (int64_t)st[slot].tau * n * n;
  const cx<T>* fs = f + slot * vs;
#pragma unroll 4
  for (int e = threadIdx.x; e < n * RB; e += 256) {
    const int l = e / RB, r = r0 + (e - l * RB);
    pr[e] = r < n ? a[(int64_t)l * n + r] * fs[l] : mk(T(0), T(0));
  }
  __syncthreads();
  // two threads per row, one for each part of the complex sum
  const int t = threadIdx.x;
  if constexpr (sizeof(T) == 8) {
    if (coarse_in_parts<T>(n)) {  // a lane per partial sum as well (2 RB COARSE_PARTS = 32 lanes)
      static_assert(2 * coarse_rows<double>() * COARSE_PARTS == 32, "one warp adds");
      if (t >= 32) return;
      const int e = t % (2 * RB);
      T acc = T(0);
#pragma unroll 16
      for (int l = t / (2 * RB); l < n; l += COARSE_PARTS) acc = acc + ((const T*)pr)[2 * l * RB + e];
      acc = acc + __shfl_xor_sync(0xffffffffu, acc, 2 * RB);
      acc = acc + __shfl_xor_sync(0xffffffffu, acc, 4 * RB);
      if (t < 2 * RB && r0 + e / 2 < n) ((T*)(z + slot * vs + r0))[e] = acc;
      return;
    }
  }
  if (t >= 2 * RB || r0 + t / 2 >= n) return;
  T acc = T(0);
#pragma unroll 16
  for (int l = 0; l < n; ++l) acc = acc + ((const T*)pr)[2 * l * RB + t];
  ((T*)(z + slot * vs + r0))[t] = acc;
}

// --------------------------------------------------------------------- defect correction
// z += e (first cycle: z = e), z in fp64, e in the cycle precision.
template <typename T>
__global__ void k_correct(const SlotState* st, cx<double>* __restrict__ z, int64_t zs, int64_t zcol,
                          const cx<T>* __restrict__ e, int64_t es, int64_t n) {
  int slot = blockIdx.y;
  if (!slot_running(st, slot)) return;
  int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n) return;
  z64 ev = cvt<double>(e[slot * es + c]);
  z64* zp = z + slot * zs + (int64_t)(st[slot].k - 1) * zcol + c;
  *zp = st[slot].cycles == 0 ? ev : (*zp + ev);
}

// After the per-slot decisions: with `use_cond`, the last slot to report sets
// the graph's loop condition to "some slot still runs its inner solve"
// (flags[slot] collects the answers, counter[0] counts reports and is reset by
// the last one).
__device__ __forceinline__ void report_slot(int slot, int running, int nslot, int* flags, int* counter,
                                            cudaGraphConditionalHandle cond) {
  flags[slot] = running;
  __threadfence();
  if (atomicAdd(counter, 1) == nslot - 1) {
    __threadfence();
    int any = 0;
    for (int q = 0; q < nslot; ++q) any |= ((volatile int*)flags)[q];
    *counter = 0;
    cudaGraphSetConditional(cond, any ? 1u : 0u);
  }
}

// The inner-solve decision of one slot from ||p||^2 = a and ||v||^2 = b
// (Section 4: stop when ||p_k|| <= eps ||v_k||, or after max_cycles, or after the
// replayed number of cycles). Returns whether the slot keeps cycling.
__device__ __forceinline__ int decide_slot(SlotState& s, int slot, double a, double b, int first, double eps,
                                           int max_cycles, const int32_t* replay_cycles, int m_max, double relax,
                                           double tol) {
  eps = inner_eps(eps, relax, tol, s.rmax);
  s.pnorm2 = a;
  if (first) {
    s.vnorm2 = b;
    s.cycles = 0;
  } else {
    s.cycles += 1;
  }
  bool done;
  if (replay_cycles) done = s.cycles >= replay_cycles[(int64_t)slot * m_max + (s.k - 1)];
  else if (first) done = false;
  else {
    done = a <= eps * eps * s.vnorm2 || s.cycles >= max_cycles;
    if (!(a <= eps * eps * s.vnorm2) && s.cycles >= max_cycles) s.inner_capped = 1;
  }
  s.inner_done = done ? 1 : 0;
  return done ? 0 : 1;
}

struct DecideArgs {
  int on;                        // decide in the last block of each slot
  double eps;
  int max_cycles;
  const int32_t* replay_cycles;  // null unless replaying
  int m_max;
  int use_cond;
  cudaGraphConditionalHandle cond;
  int* flags;
  int* counter;
  int* bcount;                   // per-slot count of finished blocks, reset by the last one
  int nslot;
  double relax, tol;             // relaxed inner tolerance (relax <= 0: eps)
};

// r = v - (K + tau M) z in fp64; f0 = r in the cycle precision; per-block
// partial sums of |r|^2 (and |v|^2 when `with_v`). With D.on the last block of
// each slot sums the partials in a fixed order and takes the inner-solve
// decision (the work of k_inner_decide, without a launch of its own).
// Bound by the FP64 pipe: 12 fused multiply-adds for the neighbours, 4 for the
// diagonal, 2 for the norm per cell of a 3D grid. A thread therefore marches
// over R cells along z (3D) or y (2D), so that the block's reduction (5 warp
// additions and the block's own) is paid once per R cells, and the neighbours
// below and above stay in registers.
template <typename T, bool D3>
__global__ void __launch_bounds__(GX * GY)
    k_defect(LevelView<double> L, SlotState* st, const z64* taus, const z64* __restrict__ diag64,
             const z64* __restrict__ v, int64_t vsv, const z64* __restrict__ z, int64_t vsz, int64_t col, int zero_z,
             cx<T>* __restrict__ f0, int64_t vsf, double* __restrict__ partial, int with_v, int R, DecideArgs D) {
  pdl_enter();
  int slot = blockIdx.z;
  __shared__ double red[2][GX * GY / 32];
  __shared__ int last_blk;
  const int tl = thread_linear();
  if (!slot_running(st, slot)) {
    // a slot that is not cycling still reports "not running"
    if (D.on && D.use_cond && blockIdx.x == 0 && blockIdx.y == 0 && tl == 0)
      report_slot(slot, 0, D.nslot, D.flags, D.counter, D.cond);
    return;
  }
  double r2 = 0.0, v2 = 0.0;
  const int nx = L.nx, ny = L.ny, sxy = nx * ny;
  const int i = blockIdx.x * GX + threadIdx.x;
  const int64_t off = (int64_t)(st[slot].k - 1) * col;
  const int tau = st[slot].tau;
  // the column of cells: (i, j, m0 .. m1) in 3D, (i, m0 .. m1) in 2D
  const int nby = (ny + GY - 1) / GY;
  const int bz = D3 ? blockIdx.y / nby : 0;
  const int j = D3 ? (int)(blockIdx.y - bz * nby) * GY + (int)threadIdx.y : 0;
  const int nm = D3 ? L.nz : ny, step = D3 ? sxy : nx;
  const int m0 = (D3 ? bz : (int)(blockIdx.y * GY + threadIdx.y)) * R;
  const int m1 = (i < nx && j < ny) ? min(m0 + R, nm) : m0;
  const z64* vv = v + slot * vsv + off;
  const z64* zz = z + slot * vsz + off;
  cx<T>* fo = f0 + slot * vsf;
  if (m0 < m1 && zero_z) {
    int c = m0 * step + j * nx + i;
    for (int m = m0; m < m1; ++m, c += step) {
      const z64 r = vv[c];
      fo[c] = cvt<T>(r);
      r2 = fmaT(r.re, r.re, r2);
      r2 = fmaT(r.im, r.im, r2);
      if (with_v) {
        v2 = fmaT(r.re, r.re, v2);
        v2 = fmaT(r.im, r.im, v2);
      }
    }
  } else if (m0 < m1) {
    const z64* dg = diag64 + (int64_t)tau * L.n;
    int c = m0 * step + j * nx + i;
    z64 below = m0 > 0 ? zz[c - step] : mk(0.0, 0.0), here = zz[c];
    // the faces below and above along the march: one load per cell (the face
    // below cell c: fz[c] in 3D, fy[c] in 2D)
    const double* fl = D3 ? L.fz : L.fy;
    double lo = fl[c];
    for (int m = m0; m < m1; ++m, c += step) {
      const bool top = m + 1 < nm;
      const double hi = fl[next_face(c, step)];
      const z64 above = top ? zz[c + step] : mk(0.0, 0.0);
      const int row = D3 ? m * ny + j : m;
      const int64_t fx = x_face(c, row);
      const double xl = L.fx[fx], xh = L.fx[fx + 1];
      z64 a = vv[c];
      const z64 d = dg[c];
      // the neighbours in nb_sum's order, then the diagonal as in minus_product
      if (i > 0) a = axpy(xl, zz[c - 1], a);
      if (i < nx - 1) a = axpy(xh, zz[c + 1], a);
      if constexpr (D3) {
        const int64_t fy = y_face(c, m, nx);
        if (j > 0) a = axpy(L.fy[fy], zz[c - nx], a);
        if (j < ny - 1) a = axpy(L.fy[fy + nx], zz[c + nx], a);
      }
      if (m > 0) a = axpy(lo, below, a);
      if (top) a = axpy(hi, above, a);
      a.re = fmaT(-d.re, here.re, fmaT(d.im, here.im, a.re));
      a.im = fmaT(-d.re, here.im, fmaT(-d.im, here.re, a.im));
      fo[c] = cvt<T>(a);
      r2 = fmaT(a.re, a.re, r2);
      r2 = fmaT(a.im, a.im, r2);
      below = here;
      here = above;
      lo = hi;
    }
  }
  for (int o = 16; o > 0; o >>= 1) r2 += __shfl_down_sync(0xffffffffu, r2, o);
  if (with_v)
    for (int o = 16; o > 0; o >>= 1) v2 += __shfl_down_sync(0xffffffffu, v2, o);
  constexpr int NW = GX * GY / 32;
  int w = tl >> 5, lane = tl & 31;
  if (lane == 0) { red[0][w] = r2; red[1][w] = v2; }
  __syncthreads();
  const int nblk = gridDim.x * gridDim.y;
  if (w == 0) {
    double a = lane < NW ? red[0][lane] : 0.0, b = lane < NW ? red[1][lane] : 0.0;
    for (int o = NW / 2; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (with_v)
      for (int o = NW / 2; o > 0; o >>= 1) b += __shfl_down_sync(0xffffffffu, b, o);
    if (lane == 0) {
      partial[((int64_t)slot * nblk + block_linear()) * 2 + 0] = a;
      partial[((int64_t)slot * nblk + block_linear()) * 2 + 1] = b;
      if (D.on) {
        __threadfence();
        last_blk = atomicAdd(&D.bcount[slot], 1) == nblk - 1;
      }
    }
  }
  if (!D.on) return;
  __syncthreads();
  if (!last_blk) return;
  __threadfence();
  const double* ps = partial + (int64_t)slot * nblk * 2;
  double a = 0.0, b = 0.0;
  for (int q = tl; q < nblk; q += GX * GY) {
    a += __ldcg(ps + 2 * q);
    if (with_v) b += __ldcg(ps + 2 * q + 1);
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    if (with_v) b += __shfl_down_sync(0xffffffffu, b, o);
  }
  __syncthreads();
  if (lane == 0) { red[0][w] = a; red[1][w] = b; }
  __syncthreads();
  if (w != 0) return;
  a = lane < NW ? red[0][lane] : 0.0;
  b = lane < NW ? red[1][lane] : 0.0;
  for (int o = NW / 2; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if (with_v)
    for (int o = NW / 2; o > 0; o >>= 1) b += __shfl_down_sync(0xffffffffu, b, o);
  if (tl == 0) {
    D.bcount[slot] = 0;
    int running = decide_slot(st[slot], slot, a, b, zero_z, D.eps, D.max_cycles, D.replay_cycles, D.m_max, D.relax,
                              D.tol);
    if (D.use_cond) report_slot(slot, running, D.nslot, D.flags, D.counter, D.cond);
  }
}

// Sum the per-block partials in a fixed order and decide whether the inner
// solve of each slot is finished; one block per slot. With `use_cond` the last
// block to finish sets the graph's loop condition to "some slot still runs its
// inner solve" (flags[slot] collects the per-slot answers, counter[0] counts
// finished blocks and is reset by the last one).
__global__ void k_inner_decide(SlotState* st, int nslot, const double* __restrict__ partial, int nblocks,
                               int first, double eps, int max_cycles, const int32_t* replay_cycles, int m_max,
                               int use_cond, cudaGraphConditionalHandle cond, int* flags, int* counter, double relax,
                               double tol) {
  __shared__ double red[32];
  int slot = blockIdx.x;
  SlotState& s = st[slot];
  bool act = s.active && !s.inner_done;
  int running = 0;
  if (act) {
    double a = 0.0, b = 0.0;
    for (int q = threadIdx.x; q < nblocks; q += blockDim.x) {
      a += partial[((int64_t)slot * nblocks + q) * 2 + 0];
      b += partial[((int64_t)slot * nblocks + q) * 2 + 1];
    }
    a = block_sum(a, red);
    b = block_sum(b, red);
    if (threadIdx.x == 0)
      running = decide_slot(s, slot, a, b, first, eps, max_cycles, replay_cycles, m_max, relax, tol);
  }
  if (use_cond && threadIdx.x == 0) report_slot(slot, running, nslot, flags, counter, cond);
}

// K_cc + tau_q M_cc for every distinct tau in fp64 (the diagonal residual_at forms).
__global__ void k_diag64(LevelView<double> L, const z64* __restrict__ taus, int ntau, z64* __restrict__ out) {
  Cell p;
  int c;
  if (!grid_cell(L.nx, L.ny, L.nz, &p, &c)) return;
  const double d = L.kd ? L.kd[c] : fsum(faces_at(L, p));
  const double m = L.mm[c];
  for (int q = 0; q < ntau; ++q) out[(int64_t)q * L.n + c] = mk(fmaT(taus[q].re, m, d), mulT(taus[q].im, m));
}

// K diagonal (sum of each cell's faces), the same sum residual_at forms.
__global__ void k_kdiag(LevelView<double> L, double* __restrict__ kd) {
  Cell p;
  int c;
  if (!grid_cell(L.nx, L.ny, L.nz, &p, &c)) return;
  kd[c] = fsum(faces_at(L, p));
}

// --------------------------------------------------------------------- launchers
static inline unsigned nb(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }
static inline dim3 grid2(int64_t nxw, int64_t rows, int nz) { return dim3(nb(nxw, GX), nb(rows, GY), nz); }
static const dim3 B2(GX, GY);

void launch_faces_from_cond(const LevelHost& L, const double h[3], uint32_t mask, const double* cond,
                            cudaStream_t s) {
  int64_t tot = face_count(L, 0) + face_count(L, 1) + (L.nz > 1 ? face_count(L, 2) : 0);
  k_faces_from_cond<<<nb(tot, 256), 256, 0, s>>>(L.nx, L.ny, L.nz, h[0], h[1], h[2], mask, cond, L.d64[0],
                                                  L.d64[1], L.d64[2]);
}

void launch_coarsen(const LevelHost& F, const LevelHost& C, const double* fac_x, const double* fac_y,
                    const double* fac_z, cudaStream_t s) {
  int64_t tot = face_count(C, 0) + face_count(C, 1) + (C.nz > 1 || F.nz > 1 ? face_count(C, 2) : 0) + C.n;
  k_coarsen<<<nb(tot, 256), 256, 0, s>>>(view<double>(F), F.rx, F.ry, F.rz, C.nx, C.ny, C.nz, C.d64[0], C.d64[1],
                                          C.d64[2], C.d64[3], fac_x, fac_y, fac_z);
}

std::vector<double> coarse_face_factors(const std::vector<double>& w, int r, std::vector<double>* W) {
  const int n = (int)w.size();
  if (r == 1) {
    *W = w;
    return std::vector<double>(n + 1, 1.0);
  }
  const int nc = (n + 1) / 2;
  W->assign(nc, 0.0);
  for (int I = 0; I < nc; ++I) (*W)[I] = w[2 * I] + (2 * I + 1 < n ? w[2 * I + 1] : 0.0);
  std::vector<double> f(nc + 1);
  f[0] = w[0] / (*W)[0];
  for (int I = 1; I < nc; ++I) f[I] = (w[2 * I - 1] + w[2 * I]) / ((*W)[I - 1] + (*W)[I]);
  f[nc] = w[n - 1] / (*W)[nc - 1];
  return f;
}

void launch_to_f32(const double* a, float* b, int64_t n, cudaStream_t s) {
  k_to_f32<<<nb(n, 256), 256, 0, s>>>(a, b, n);
}

template <typename T>
void launch_invd(const LevelHost& L, const z64* taus, int ntau, cx<T>* out, cudaStream_t s, int from_f32) {
  if (from_f32) k_invd<T, float><<<nb(L.n, 256), 256, 0, s>>>(view_as<double, float>(L), taus, ntau, out);
  else k_invd<T, double><<<nb(L.n, 256), 256, 0, s>>>(view<double>(L), taus, ntau, out);
}

template <typename T>
int launch_coarse_inverse(const LevelHost& L, const z64* taus, int ntau, z64* work, z64* work2, cx<T>* inv,
                          int* singular, cudaStream_t s, int from_f32) {
  const int n = (int)L.n;
  const int64_t nn = (int64_t)n * n;
  const bool small = n <= GJ_SMALL;
  // the steps' column buffers, pivot row and pivots live in inv's memory until
  // the finish overwrites it (52 n bytes of its n^2 sizeof(cx<T>) per tau); the
  // pivots move to the other matrix buffer first
  const int64_t tn = (int64_t)ntau * n;
  z64* cb[2] = {(z64*)inv, (z64*)inv + tn};
  z64* prow = cb[1] + tn;
  int32_t* piv = (int32_t*)(prow + tn);
  cudaMemsetAsync(work, 0, sizeof(z64) * nn * ntau, s);
  z64* c0 = small ? nullptr : cb[0];
  const dim3 gd(nb(n, 128), ntau);
  if (from_f32) k_coarse_dense<float><<<gd, 128, 0, s>>>(view_as<double, float>(L), taus, work, c0);
  else k_coarse_dense<double><<<gd, 128, 0, s>>>(view<double>(L), taus, work, c0);
  if (small) {
    k_gj_small<T><<<ntau, 512, 0, s>>>(work, inv, n, singular);
    return 2;
  }
  z64 *src = work, *dst = work2;
  const unsigned nt = nb(n, GJ_T);
  // one launch per step up to about ten blocks per SM (360 unknowns at four taus)
  const bool one = (int64_t)nt * nb(n, 8) * ntau <= 2048;
  for (int col = 0; col < n; ++col) {
    z64 *ci = cb[col & 1], *co = cb[(col + 1) & 1];
    if (one) {
      launch_pdl(k_gj_step, dim3(nt, nb(n, 8), ntau), dim3(32, 8), 0, s, src, dst, ci, co, piv, n, col, singular);
      std::swap(src, dst);
    } else {
      launch_pdl(k_gj_pivot, dim3(ntau), dim3((n + 31) & ~31), 0, s, src, prow, ci, piv, n, col, singular);
      launch_pdl(k_gj_update, dim3(nt, nt, ntau), dim3(32, 8), 0, s, src, prow, ci, co, n, col);
    }
  }
  cudaMemcpyAsync(dst, piv, sizeof(int32_t) * n * ntau, cudaMemcpyDeviceToDevice, s);
  k_gj_finish<T><<<dim3(nt, nt, ntau), dim3(32, 8), 0, s>>>(src, (const int32_t*)dst, inv, n);
  return 2 + (one ? n : 2 * n);
}

void launch_round_bf16(const double* a, __nv_bfloat16* b, float* r, int64_t n, cudaStream_t s) {
  k_round_bf16<<<nb(n, 256), 256, 0, s>>>(a, b, r, n);
}

// Sources per block of the multi-source smoother and restriction: a power of
// two up to 8 (blockDim = (32, 8 / G, G)).
static int spmm_group(int nslot) {
  int g = 1;
  while (g < 8 && 2 * g <= nslot) g *= 2;
  return g;
}

template <typename T>
void launch_gs(const LevelHost& L, const SlotState* st, const cx<T>* invd, const cx<T>* f, cx<T>* z, int64_t vs,
               int nslot, int color, int zero_start, cudaStream_t s, z64* Zk, int64_t vsZk, int64_t zcol, int bf16) {
  const int G = spmm_group(nslot), rb = GY / G;
  const dim3 blk(GX, rb, G), grd(nb((L.nx + 1) / 2, GX), nb((int64_t)L.ny * L.nz, rb), nb(nslot, G));
  const unsigned mny = row_magic(L.ny);
  if constexpr (sizeof(T) == 4) {
    if (bf16) {
      if (Zk)
        launch_pdl(k_gs_correct<T, __nv_bfloat16>, grd, blk, 0, s, view_as<T, __nv_bfloat16>(L), st, invd, f, z, vs, color,
                                                           Zk, vsZk, zcol, nslot, mny);
      else
        launch_pdl(k_gs<T, __nv_bfloat16>, grd, blk, 0, s, view_as<T, __nv_bfloat16>(L), st, invd, f, z, vs, color,
                                                   zero_start, nslot, mny);
      return;
    }
  }
  if (Zk) {
    launch_pdl(k_gs_correct<T, T>, grd, blk, 0, s, view<T>(L), st, invd, f, z, vs, color, Zk, vsZk, zcol, nslot, mny);
    return;
  }
  launch_pdl(k_gs<T, T>, grd, blk, 0, s, view<T>(L), st, invd, f, z, vs, color, zero_start, nslot, mny);
}

template <typename T>
void launch_residual_restrict(const LevelHost& F, const LevelHost& C, const SlotState* st, const z64* taus,
                              const cx<T>* f, const cx<T>* z, int64_t vs, cx<T>* fc, int64_t vsc, int nslot,
                              cudaStream_t s, int bf16) {
  const int G = spmm_group(nslot), rb = GY / G;
  if (G == 1 && F.nz > 1 && F.rx == 2 && F.ry == 2 && F.rz == 2 && (int64_t)nb(F.ny, GY) * C.nz <= 65535) {
    // one source: the tile form (with several, the per-coarse-cell form reads
    // each coefficient once for the block's sources)
    const dim3 g3(nb(F.nx, GX), nb(F.ny, GY) * C.nz, nslot);
    if constexpr (sizeof(T) == 4) {
      if (bf16) {
        launch_pdl(k_residual_restrict3<T, __nv_bfloat16>, g3, B2, 0, s, view_as<T, __nv_bfloat16>(F), C.nx, C.ny,
                   C.nz, st, taus, f, z, vs, fc, vsc);
        return;
      }
    }
    launch_pdl(k_residual_restrict3<T, T>, g3, B2, 0, s, view<T>(F), C.nx, C.ny, C.nz, st, taus, f, z, vs, fc, vsc);
    return;
  }
  const dim3 blk(GX, rb, G), grd(nb(C.nx, GX), nb((int64_t)C.ny * C.nz, rb), nb(nslot, G));
  if constexpr (sizeof(T) == 4) {
    if (bf16) {
      launch_pdl(k_residual_restrict<T, __nv_bfloat16>, grd, blk, 0, s, view_as<T, __nv_bfloat16>(F), F.rx, F.ry, F.rz, C.nx,
                                                                C.ny, C.nz, st, taus, f, z, vs, fc, vsc, nslot);
      return;
    }
  }
  launch_pdl(k_residual_restrict<T, T>, grd, blk, 0, s, view<T>(F), F.rx, F.ry, F.rz, C.nx, C.ny, C.nz, st, taus, f, z, vs, fc,
                                                vsc, nslot);
}

template <typename T>
void launch_prolong_add(const LevelHost& F, const LevelHost& C, uint32_t mask, const SlotState* st, const cx<T>* zc,
                        int64_t vsc, cx<T>* z, int64_t vs, int nslot, cudaStream_t s) {
  if (F.nz > 1 && F.rx == 2 && F.ry == 2 && F.rz == 2 && (int64_t)nb(F.ny, GY) * C.nz <= 65535) {
    const dim3 g(nb(F.nx, GX), nb(F.ny, GY) * C.nz, nslot);
    launch_pdl(k_prolong_add3<T>, g, B2, 0, s, view<T>(F), C.nx, C.ny, C.nz, mask, st, zc, vsc, z, vs);
    return;
  }
  launch_pdl(k_prolong_add<T>, grid2((F.nx + 1) / 2, (int64_t)F.ny * F.nz, nslot), B2, 0, s, view<T>(F), F.rx, F.ry, F.rz, C.nx, C.ny,
                                                                            C.nz, mask, st, zc, vsc, z, vs);
}

// Tiles of 32x32 or 16x16 cells (16x16: more blocks on small grids, a larger
// share of recomputed halo); the caller picks per level.
template <typename T, int TX, int TY>
static size_t fused_smem() {
  return 2 * (size_t)(TX + 2 * FH) * (TY + 2 * FH) * sizeof(cx<T>);
}

bool fused_level_ok(const LevelHost& L) {
  return L.nz == 1 && L.rx == 2 && L.ry == 2 && L.rz == 1;
}

template <typename T>
void fused_prepare() {
  // 8 x 8 and 16 x 16 tiles stay under the 48 KB default
  cudaFuncSetAttribute(k_pre2d<T, 32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem<T, 32, 32>());
  cudaFuncSetAttribute(k_post2d<T, 32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem<T, 32, 32>());
}

template <typename T>
void launch_pre2d(const LevelHost& F, const LevelHost& C, const SlotState* st, const cx<T>* invd, const z64* taus,
                  const cx<T>* f, cx<T>* z, int64_t vs, cx<T>* fc, int64_t vsc, int nslot, int tile, cudaStream_t s) {
  const dim3 g(nb(F.nx, tile), nb(F.ny, tile), nslot);
  const LevelView<T> L = view<T>(F);
  if (tile == 8) {
    launch_pdl(k_pre2d_pairs<T, 8>, g, TilePair<T, 8>::NT, 0, s, L, st, invd, taus, f, z, vs, fc, vsc);
  } else if (tile == 16) {
    if constexpr (sizeof(T) == 4)
      launch_pdl(k_pre2d_pairs<T, 16>, g, TilePair<T, 16>::NT, 0, s, L, st, invd, taus, f, z, vs, fc, vsc);
    else
      launch_pdl(k_pre2d<T, 16, 16>, g, 256, fused_smem<T, 16, 16>(), s, L, st, invd, taus, f, z, vs, fc, vsc);
  } else {
    launch_pdl(k_pre2d<T, 32, 32>, g, 256, fused_smem<T, 32, 32>(), s, L, st, invd, taus, f, z, vs, fc, vsc);
  }
  (void)C;
}

template <typename T>
void launch_post2d(const LevelHost& F, const LevelHost& C, uint32_t mask, const SlotState* st, const cx<T>* invd,
                   const cx<T>* f, const cx<T>* z, cx<T>* zout, int64_t vs, const cx<T>* zc, int64_t vsc, int nslot,
                   int tile, cudaStream_t s, z64* Zk, int64_t vsZk, int64_t zcol) {
  const dim3 g(nb(F.nx, tile), nb(F.ny, tile), nslot);
  const LevelView<T> L = view<T>(F);
  if (tile == 8) {
    launch_pdl(k_post2d_pairs<T, 8>, g, TilePair<T, 8>::NT, 0, s, L, mask, st, invd, f, z, zout, vs, zc, vsc, Zk, vsZk,
               zcol);
  } else if (tile == 16) {
    if constexpr (sizeof(T) == 4)
      launch_pdl(k_post2d_pairs<T, 16>, g, TilePair<T, 16>::NT, 0, s, L, mask, st, invd, f, z, zout, vs, zc, vsc, Zk,
                 vsZk, zcol);
    else
      launch_pdl(k_post2d<T, 16, 16>, g, 256, fused_smem<T, 16, 16>(), s, L, mask, st, invd, f, z, zout, vs, zc, vsc,
                 Zk, vsZk, zcol);
  } else {
    launch_pdl(k_post2d<T, 32, 32>, g, 256, fused_smem<T, 32, 32>(), s, L, mask, st, invd, f, z, zout, vs, zc, vsc, Zk,
               vsZk, zcol);
  }
  (void)C;
}

// The attribute belongs to the kernel, not to a launch, and every context of the
// process shares it: always the same value, so that no operator's setup takes
// shared memory away from the launch or capture that another thread is about to
// make. (A launch's occupancy follows what it asks for itself.)
template <typename T>
void tail_prepare() {
  auto grant = [](auto kernel, size_t bytes) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  grant(k_tail_vcycle<T>, TAIL_SMEM_LIMIT);
  grant(k_tail2d<T>, TAIL_SMEM_LIMIT);
  grant(k_tail_pairs<T, 512>, TAIL_SMEM_LIMIT);
  if constexpr (sizeof(T) == 8) {
    grant(k_tail_pairs<T, 512, 1>, TAIL_SMEM_LIMIT);
    grant(k_tail_pairs<T, 512, 2>, TAIL_SMEM_LIMIT);
  }
  if constexpr (sizeof(T) == 4) grant(k_tail_pairs<T, 1024>, TAIL_SMEM_LIMIT);
  grant(k_coarse_solve<T>, MAX_COARSE * coarse_rows<T>() * sizeof(cx<T>));
}

template <typename T>
void launch_tail(const TailParams<T>& P, size_t smem_bytes, const SlotState* st, int nslot, cudaStream_t s, int part) {
  if (part) {
    if constexpr (sizeof(T) == 8) {
      if (part == 1) launch_pdl(k_tail_pairs<T, 512, 1>, nslot, 512, smem_bytes, s, P, st);
      else launch_pdl(k_tail_pairs<T, 512, 2>, nslot, 512, smem_bytes, s, P, st);
    }
  } else if (P.pairs)
    launch_pdl(k_tail2d<T>, nslot, TAIL_THREADS, smem_bytes, s, P, st);
  else if (P.roff && P.threads == 512)
    launch_pdl(k_tail_pairs<T, 512>, nslot, 512, smem_bytes, s, P, st);
  else if (P.roff) {
    if constexpr (sizeof(T) == 4) launch_pdl(k_tail_pairs<T, 1024>, nslot, 1024, smem_bytes, s, P, st);
  } else
    launch_pdl(k_tail_vcycle<T>, nslot, TAIL_THREADS, smem_bytes, s, P, st);
}

template <typename T>
void launch_coarse_solve(const cx<T>* Ainv, int n, const SlotState* st, const cx<T>* f, cx<T>* z, int64_t vs,
                         int nslot, cudaStream_t s) {
  dim3 g(nb(n, coarse_rows<T>()), nslot);
  launch_pdl(k_coarse_solve<T>, g, 256, (size_t)n * coarse_rows<T>() * sizeof(cx<T>), s, Ainv, n, st, f, z, vs);
}

template <typename T>
void launch_correct(const SlotState* st, z64* z, int64_t zs, int64_t zcol, const cx<T>* e, int64_t es, int64_t n,
                    int nslot, cudaStream_t s) {
  dim3 g(nb(n, 256), nslot);
  k_correct<T><<<g, 256, 0, s>>>(st, z, zs, zcol, e, es, n);
}

// Cells per thread of the complex128 stencil marches: 4 while that leaves 5 blocks per SM
// (then the last wave is a few percent), halved on smaller grids. A function of
// the grid alone, so that a source's norms do not depend on its batch.
int march_len(const LevelHost& L) {
  const int64_t cols = L.nz > 1 ? (int64_t)nb(L.nx, GX) * nb(L.ny, GY) : nb(L.nx, GX);
  int R = 4;
  while (R > 1 && cols * (L.nz > 1 ? nb(L.nz, R) : nb(L.ny, GY * R)) < 5 * 152) R /= 2;
  while (L.nz > 1 && (int64_t)nb(L.ny, GY) * nb(L.nz, R) > 65535) R *= 2;  // gridDim.y
  return R;
}
dim3 march_grid(const LevelHost& L, int R, int nslot) {
  return L.nz > 1 ? dim3(nb(L.nx, GX), nb(L.ny, GY) * nb(L.nz, R), nslot)
                  : dim3(nb(L.nx, GX), nb(L.ny, GY * R), nslot);
}

void launch_apply(const LevelHost& L, z64 sh, const z64* x, z64* y, int64_t vs, int nvec, cudaStream_t s) {
  const int R = march_len(L);
  const dim3 g = march_grid(L, R, nvec);
  if (L.nz > 1) k_apply<true><<<g, B2, 0, s>>>(view<double>(L), sh, x, y, vs, R);
  else k_apply<false><<<g, B2, 0, s>>>(view<double>(L), sh, x, y, vs, R);
}

int defect_blocks(const LevelHost& L) {
  dim3 g = march_grid(L, march_len(L), 1);
  return (int)(g.x * g.y);
}

template <typename T>
void launch_defect_decide(const LevelHost& L, SlotState* st, const z64* taus, const z64* diag64, const z64* v,
                          int64_t vsv, const z64* z, int64_t vsz, int64_t col, int zero_z, cx<T>* f0, int64_t vsf,
                          double* partial, double eps, int max_cycles, const int32_t* replay_cycles, int m_max,
                          int use_cond, cudaGraphConditionalHandle cond, int* flags, int* counter, int* bcount,
                          int nslot, double relax, double tol, cudaStream_t s) {
  DecideArgs D{1, eps, max_cycles, replay_cycles, m_max, use_cond, cond, flags, counter, bcount, nslot, relax, tol};
  const int R = march_len(L);
  const dim3 g = march_grid(L, R, nslot);
  if (L.nz > 1)
    launch_pdl(k_defect<T, true>, g, B2, 0, s, view<double>(L), st, taus, diag64, v, vsv, z, vsz, col, zero_z, f0, vsf,
               partial, zero_z, R, D);
  else
    launch_pdl(k_defect<T, false>, g, B2, 0, s, view<double>(L), st, taus, diag64, v, vsv, z, vsz, col, zero_z, f0,
               vsf, partial, zero_z, R, D);
}

void launch_diag64(const LevelHost& L, const z64* taus, int ntau, z64* out, cudaStream_t s) {
  k_diag64<<<grid2(L.nx, (int64_t)L.ny * L.nz, 1), B2, 0, s>>>(view<double>(L), taus, ntau, out);
}

void launch_kdiag(const LevelHost& L, double* kd, cudaStream_t s) {
  k_kdiag<<<grid2(L.nx, (int64_t)L.ny * L.nz, 1), B2, 0, s>>>(view<double>(L), kd);
}

void launch_inner_decide(SlotState* st, int nslot, const double* partial, int nblocks, int first, double eps,
                         int max_cycles, const int32_t* replay_cycles, int m_max, int use_cond,
                         cudaGraphConditionalHandle cond, int* flags, int* counter, cudaStream_t s, double relax,
                         double tol) {
  k_inner_decide<<<nslot, 512, 0, s>>>(st, nslot, partial, nblocks, first, eps, max_cycles, replay_cycles, m_max,
                                        use_cond, cond, flags, counter, relax, tol);
}

#define INST(T)                                                                                                  \
  template void fused_prepare<T>();                                                                               \
  template void launch_pre2d<T>(const LevelHost&, const LevelHost&, const SlotState*, const cx<T>*, const z64*,    \
                                const cx<T>*, cx<T>*, int64_t, cx<T>*, int64_t, int, int, cudaStream_t);          \
  template void launch_post2d<T>(const LevelHost&, const LevelHost&, uint32_t, const SlotState*, const cx<T>*,     \
                                 const cx<T>*, const cx<T>*, cx<T>*, int64_t, const cx<T>*, int64_t, int, int,    \
                                 cudaStream_t, z64*, int64_t, int64_t);                                           \
  template void tail_prepare<T>();                                                                                \
  template void launch_tail<T>(const TailParams<T>&, size_t, const SlotState*, int, cudaStream_t, int);                \
  template void launch_invd<T>(const LevelHost&, const z64*, int, cx<T>*, cudaStream_t, int);                     \
  template int launch_coarse_inverse<T>(const LevelHost&, const z64*, int, z64*, z64*, cx<T>*, int*, cudaStream_t, \
                                         int);                                                                    \
  template void launch_gs<T>(const LevelHost&, const SlotState*, const cx<T>*, const cx<T>*, cx<T>*, int64_t, int,  \
                             int, int, cudaStream_t, z64*, int64_t, int64_t, int);                                \
  template void launch_residual_restrict<T>(const LevelHost&, const LevelHost&, const SlotState*, const z64*,      \
                                            const cx<T>*, const cx<T>*, int64_t, cx<T>*, int64_t, int,           \
                                            cudaStream_t, int);                                                   \
  template void launch_prolong_add<T>(const LevelHost&, const LevelHost&, uint32_t, const SlotState*,             \
                                      const cx<T>*, int64_t, cx<T>*, int64_t, int, cudaStream_t);                 \
  template void launch_coarse_solve<T>(const cx<T>*, int, const SlotState*, const cx<T>*, cx<T>*, int64_t, int,    \
                                       cudaStream_t);                                                             \
  template void launch_correct<T>(const SlotState*, z64*, int64_t, int64_t, const cx<T>*, int64_t, int64_t, int,  \
                                  cudaStream_t);                                                                  \
  template void launch_defect_decide<T>(const LevelHost&, SlotState*, const z64*, const z64*, const z64*, int64_t, \
                                        const z64*, int64_t, int64_t, int, cx<T>*, int64_t, double*, double, int, \
                                        const int32_t*, int, int, cudaGraphConditionalHandle, int*, int*, int*, int, \
                                        double, double, cudaStream_t);

INST(double)
INST(float)

}  // namespace fks
