// Device helpers for the cell-centred 2d+1-point operator, shared by the grid
// and Krylov kernels.
#pragma once
#include "common.cuh"

namespace fks {

// --------------------------------------------------------------------- indexing
struct Cell {
  int i, j, k;
};

// Cell of flat index c (32-bit: a level has fewer than 2^31 cells).
__device__ __forceinline__ Cell cell_of(int c, int nx, int ny) {
  Cell r;
  int q = c / nx;
  r.i = c - q * nx;
  r.k = q / ny;
  r.j = q - r.k * ny;
  return r;
}

// Launch shape of the grid kernels: block (GX, GY) threads, x along i, y along
// the rows (j, k) of the level, z along the sources.
constexpr int GX = 32, GY = 8;

// Cell of this thread in a (i, row) launch; false past the grid.
__device__ __forceinline__ bool grid_cell(int nx, int ny, int nz, Cell* p, int* c) {
  int i = blockIdx.x * GX + threadIdx.x;
  int row = blockIdx.y * GY + threadIdx.y;
  if (i >= nx || row >= ny * nz) return false;
  int k = row / ny;
  *p = Cell{i, row - k * ny, k};
  *c = row * nx + i;
  return true;
}

// Cell of colour `color` of this thread in a (half-row index, row) launch.
__device__ __forceinline__ bool grid_color_cell(int nx, int ny, int nz, int color, Cell* p, int* c) {
  int ii = blockIdx.x * GX + threadIdx.x;
  int row = blockIdx.y * GY + threadIdx.y;
  if (row >= ny * nz) return false;
  int k = row / ny;
  int j = row - k * ny;
  int i = 2 * ii + ((j + k + color) & 1);
  if (i >= nx) return false;
  *p = Cell{i, j, k};
  *c = row * nx + i;
  return true;
}

__device__ __forceinline__ int block_linear() { return blockIdx.y * gridDim.x + blockIdx.x; }
__device__ __forceinline__ int thread_linear() { return threadIdx.y * GX + threadIdx.x; }

// row = k ny + j without a division: mny = row_magic(ny) (k is first off by one
// at most either way)
inline unsigned row_magic(int ny) { return ny == 1 ? 0xffffffffu : (unsigned)((1ull << 32) / (unsigned)ny) + 1u; }
__device__ __forceinline__ void split_row(int row, int ny, unsigned mny, int* j, int* k) {
  int q = (int)__umulhi((unsigned)row, mny), r = (int)((unsigned)row - (unsigned)q * (unsigned)ny);
  if (r < 0) { r += ny; --q; }
  if (r >= ny) { r -= ny; ++q; }
  *j = r;
  *k = q;
}

// Flat indices of a cell's faces (c = row nx + i, row = k ny + j): the face
// arrays hold up to ny nz (x), nx nz (y) or nx ny (z) entries more than the
// fewer than 2^31 cells, so these take 64 bits. The high faces: + 1, + nx.
__host__ __device__ __forceinline__ int64_t x_face(int c, int row) { return (int64_t)c + row; }
__host__ __device__ __forceinline__ int64_t y_face(int c, int k, int nx) { return c + (int64_t)k * nx; }
// of the cell's faces along the axis that a march takes (`step` cells apart)
__host__ __device__ __forceinline__ int64_t next_face(int c, int step) { return (int64_t)c + step; }

template <typename T>
struct Faces {
  T xl, xh, yl, yh, zl, zh;
};

template <typename T, typename C>
__device__ __forceinline__ Faces<T> faces_at(const LevelView<T, C>& L, Cell p) {
  Faces<T> f;
  int64_t rx = ((int64_t)p.k * L.ny + p.j) * (L.nx + 1) + p.i;
  f.xl = ldc<T>(L.fx, rx);
  f.xh = ldc<T>(L.fx, rx + 1);
  int64_t ry = ((int64_t)p.k * (L.ny + 1) + p.j) * L.nx + p.i;
  f.yl = ldc<T>(L.fy, ry);
  f.yh = ldc<T>(L.fy, ry + L.nx);
  if (L.nz > 1) {
    int64_t rz = ((int64_t)p.k * L.ny + p.j) * L.nx + p.i;
    f.zl = ldc<T>(L.fz, rz);
    f.zh = ldc<T>(L.fz, rz + (int64_t)L.nx * L.ny);
  } else {
    f.zl = T(0);
    f.zh = T(0);
  }
  return f;
}

template <typename T>
__device__ __forceinline__ T fsum(const Faces<T>& f) {
  return ((f.xl + f.xh) + (f.yl + f.yh)) + (f.zl + f.zh);
}

// s0 + sum over existing neighbours of t_face * x_nb (accumulated in this order)
template <typename T, typename C>
__device__ __forceinline__ cx<T> nb_sum(const LevelView<T, C>& L, const Faces<T>& f, Cell p, int64_t c,
                                        const cx<T>* __restrict__ x, cx<T> s0 = cx<T>{T(0), T(0)}) {
  cx<T> s = s0;
  int64_t sxy = (int64_t)L.nx * L.ny;
  if (p.i > 0) s = axpy(f.xl, x[c - 1], s);
  if (p.i < L.nx - 1) s = axpy(f.xh, x[c + 1], s);
  if (p.j > 0) s = axpy(f.yl, x[c - L.nx], s);
  if (p.j < L.ny - 1) s = axpy(f.yh, x[c + L.nx], s);
  if (L.nz > 1) {
    if (p.k > 0) s = axpy(f.zl, x[c - sxy], s);
    if (p.k < L.nz - 1) s = axpy(f.zh, x[c + sxy], s);
  }
  return s;
}

// The same two for the complex64 level kernels, which the instruction rate
// bounds: 32-bit indices (n < 2^31; row = k ny + j, c = row nx + i), every load
// issued before the sum, and a neighbour outside the grid adds t * 0. 128^3:
// half sweep 10.8 -> 9.5 us, the correcting one 22.1 -> 19.6, residual and
// restriction 16.4 -> 14.4; 208 instructions a cell before. complex128, where
// FP64 arithmetic is the bound, keeps the ones above.
template <typename T, typename C>
__device__ __forceinline__ Faces<T> faces_row(const LevelView<T, C>& L, int k, int row, int c) {
  const C* fx = L.fx + ((unsigned)c + (unsigned)row);
  const C* fy = L.fy + ((unsigned)c + (unsigned)(k * L.nx));
  const C* fz = L.fz + c;
  Faces<T> f{ldc<T>(fx, 0), ldc<T>(fx, 1), ldc<T>(fy, 0), ldc<T>(fy, L.nx), T(0), T(0)};
  if (L.nz > 1) {
    f.zl = ldc<T>(fz, 0);
    f.zh = ldc<T>(fz, L.nx * L.ny);
  }
  return f;
}

template <typename T>
struct Star {
  cx<T> xl, xh, yl, yh, zl, zh;
};
template <typename T, typename C>
__device__ __forceinline__ Star<T> star_row(const LevelView<T, C>& L, Cell p, int c, const cx<T>* x) {
  const cx<T> none = mk(T(0), T(0));
  const cx<T>* q = x + c;
  const int sxy = L.nx * L.ny;
  Star<T> v;
  v.xl = p.i > 0 ? q[-1] : none;
  v.xh = p.i < L.nx - 1 ? q[1] : none;
  v.yl = p.j > 0 ? q[-L.nx] : none;
  v.yh = p.j < L.ny - 1 ? q[L.nx] : none;
  v.zl = p.k > 0 ? q[-sxy] : none;
  v.zh = p.k < L.nz - 1 ? q[sxy] : none;
  return v;
}
template <typename T>
__device__ __forceinline__ cx<T> star_sum(const Faces<T>& f, const Star<T>& v, bool d3, cx<T> s) {
  s = axpy(f.xl, v.xl, s);
  s = axpy(f.xh, v.xh, s);
  s = axpy(f.yl, v.yl, s);
  s = axpy(f.yh, v.yh, s);
  if (d3) {
    s = axpy(f.zl, v.zl, s);
    s = axpy(f.zh, v.zh, s);
  }
  return s;
}

// acc - diag x in four fused multiply-adds
template <typename T>
__device__ __forceinline__ cx<T> minus_product(cx<T> acc, cx<T> diag, cx<T> x) {
  acc.re = fmaT(-diag.re, x.re, fmaT(diag.im, x.im, acc.re));
  acc.im = fmaT(-diag.re, x.im, fmaT(-diag.im, x.re, acc.im));
  return acc;
}

// Red-black Gauss-Seidel update of cell c: (f_c + sum_nb t z_nb) / (K_cc + tau M_cc),
// the neighbours taken as zero when `zero_start`.
template <typename T, typename C>
__device__ __forceinline__ cx<T> gs_value(const LevelView<T, C>& L, Cell p, int64_t c, cx<T> id, const cx<T>* f,
                                          const cx<T>* z, int zero_start) {
  cx<T> rhs = f[c];
  if (!zero_start) {
    Faces<T> fc = faces_at(L, p);
    rhs = nb_sum(L, fc, p, c, z, rhs);  // f + sum t z_nb, accumulated from f
  }
  return id * rhs;
}

// gs_value with the row of the cell known
template <typename T, typename C>
__device__ __forceinline__ cx<T> gs_row(const LevelView<T, C>& L, Cell p, int row, int c, cx<T> id, const cx<T>* f,
                                        const cx<T>* z, int zero_start) {
  if constexpr (sizeof(T) == 8) return gs_value(L, p, c, id, f, z, zero_start);
  cx<T> rhs = f[c];
  if (!zero_start) {
    const Faces<T> fa = faces_row(L, p.k, row, c);
    rhs = star_sum(fa, star_row(L, p, c, z), L.nz > 1, rhs);
  }
  return id * rhs;
}

// Cell of colour `color` handled by work item t of a half sweep (false if none).
__device__ __forceinline__ bool color_cell(int nx, int ny, int nz, int color, int t, Cell* p, int* c) {
  int nxh = (nx + 1) >> 1;
  int rows = ny * nz;
  if (t >= nxh * rows) return false;
  int row = t / nxh;
  int k = row / ny;
  int j = row - k * ny;
  int i = 2 * (t - row * nxh) + ((j + k + color) & 1);
  if (i >= nx) return false;
  *p = Cell{i, j, k};
  *c = row * nx + i;
  return true;
}

// The residual that a level restricts. In complex128 only the red cells' is
// formed: the pre-smoothing ends with a black half sweep, which solves every
// black cell's equation, so the black residuals are zero (rounding apart) and
// are neither formed nor added: half of the work of a phase that FP64
// arithmetic bounds (45 x 53 x 37 complex128 66.0 -> 59.2 ms a solve, 64 x 48 x
// 48 172 -> 147). In complex64, where these kernels wait for memory, it would
// give 1 to 2 %, and dropping what rounding leaves at the black cells (1e-7 of
// the iterate) moves x_j by up to 9e-10 on hierarchies that converge slowly
// (185 x 192, x never halved): there all cells stay.
template <typename T>
constexpr bool RED_RESIDUAL = sizeof(T) == 8;

// f - (K + s M) z from the cell's f and z, its diagonal K_cc + s M_cc and a
// functor that accumulates sum t z_nb onto its argument
template <typename T, typename NB>
__device__ __forceinline__ cx<T> residual_of(cx<T> f, cx<T> z, cx<T> diag, NB nb) {
  if constexpr (RED_RESIDUAL<T>) return minus_product(nb(f), diag, z);
  else return f - (diag * z - nb(mk(T(0), T(0))));
}

template <typename T, typename C>
__device__ __forceinline__ cx<T> residual_at(const LevelView<T, C>& L, Cell p, int64_t c, cx<T> s, const cx<T>* f,
                                             const cx<T>* z) {
  const Faces<T> fa = faces_at(L, p);
  const T d = L.kd ? L.kd[c] : fsum(fa);  // same sum either way
  const T m = ldc<T>(L.mm, c);
  return residual_of(f[c], z[c], mk(fmaT(s.re, m, d), mulT(s.im, m)),
                     [&](cx<T> a) { return nb_sum(L, fa, p, c, z, a); });
}

// residual_at with the row of the cell known
template <typename T, typename C>
__device__ __forceinline__ cx<T> residual_row(const LevelView<T, C>& L, Cell p, int row, int c, cx<T> s,
                                              const cx<T>* f, const cx<T>* z) {
  if constexpr (sizeof(T) == 8) return residual_at(L, p, c, s, f, z);
  const Faces<T> fa = faces_row(L, p.k, row, c);
  const Star<T> v = star_row(L, p, c, z);
  const T m = ldc<T>(L.mm, c);
  return residual_of(f[c], z[c], mk(fmaT(s.re, m, fsum(fa)), mulT(s.im, m)),
                     [&](cx<T> a) { return star_sum(fa, v, L.nz > 1, a); });
}

// First child along x that takes part in a restriction, of cells whose other
// coordinates (and first child's x) sum to `sum`; the next is child_step on
template <typename T>
__device__ __forceinline__ int child_first(int sum) { return RED_RESIDUAL<T> ? sum & 1 : 0; }
template <typename T>
constexpr int child_step = RED_RESIDUAL<T> ? 2 : 1;

// Sum over the children of coarse cell (I,J,K) of the fine residual f - (K + s M) z
// (on an odd axis the last coarse cell has one child).
template <typename T, typename C>
__device__ __forceinline__ cx<T> restrict_value(const LevelView<T, C>& F, int rx, int ry, int rz, int I, int J, int K,
                                                cx<T> s, const cx<T>* f, const cx<T>* z) {
  cx<T> acc = mk(T(0), T(0));
  for (int c = 0; c < rz; ++c)
    for (int b = 0; b < ry; ++b)
      for (int a = child_first<T>(rx * I + ry * J + b + rz * K + c); a < rx; a += child_step<T>) {
        Cell p{rx * I + a, ry * J + b, rz * K + c};
        if (p.i >= F.nx || p.j >= F.ny || p.k >= F.nz) continue;
        int64_t cc = ((int64_t)p.k * F.ny + p.j) * F.nx + p.i;
        acc = acc + residual_at(F, p, cc, s, f, z);
      }
  return acc;
}

template <typename T, typename Term>
__device__ __forceinline__ cx<T> coarse_sum(int nc, Term term) {
  cx<T> a[COARSE_PARTS];
#pragma unroll
  for (int p = 0; p < COARSE_PARTS; ++p) a[p] = mk(T(0), T(0));
  if (!coarse_in_parts<T>(nc)) {
#pragma unroll 8
    for (int l = 0; l < nc; ++l) a[0] = a[0] + term(l);
    return a[0];
  }
  for (int l = 0; l < nc; l += COARSE_PARTS)
#pragma unroll
    for (int p = 0; p < COARSE_PARTS; ++p)
      if (l + p < nc) a[p] = a[p] + term(l + p);
  return (a[0] + a[1]) + (a[2] + a[3]);
}

// a positive normal float as T (exact), without the FP64 pipe
template <typename T>
__device__ __forceinline__ T widen(float w) {
  if constexpr (sizeof(T) == 4) {
    return w;
  } else {
    const unsigned u = __float_as_uint(w);
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
  }
}

// (P zc)_c: cell-centred (bi/tri)linear interpolation from the coarser level.
// Per coarsened axis: 3/4 on the parent, 1/4 on the coarse neighbour on the
// child's side; past a zero-head face the ghost is -parent (weight 1/2 on the
// parent), past a no-flow face +parent (weight 1).
// get(X, Y, Z) returns the coarse value at coarse cell (X, Y, Z).
// Post-smoothing starts with the black cells and does not read their old
// values, so only the red ones (i + j + k even) are interpolated.
template <typename T, typename Get>
__device__ __forceinline__ cx<T> prolong_value_at(Cell p, int rx, int ry, int rz, int cnx, int cny, int cnz,
                                                  uint32_t mask, Get get) {
  int idx[3] = {p.i, p.j, p.k};
  int rr[3] = {rx, ry, rz};
  int nn[3] = {cnx, cny, cnz};
  int ti[3][2];
  // the weights are products of 1, 3/4, 1/2 and 1/4, exact in float: they are
  // formed there, and widened with integer instructions (in complex128 their
  // multiplications and zero tests were 20 of the 38 FP64 instructions per cell)
  float tw[3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int par = rr[a] == 2 ? idx[a] >> 1 : idx[a];
    ti[a][0] = par;
    ti[a][1] = par;
    if (rr[a] == 1) {
      tw[a][0] = 1.f;
      tw[a][1] = 0.f;
      continue;
    }
    int nb = (idx[a] & 1) ? par + 1 : par - 1;
    if (nb >= 0 && nb < nn[a]) {
      tw[a][0] = 0.75f;
      ti[a][1] = nb;
      tw[a][1] = 0.25f;
    } else {
      bool dir = nb < 0 ? ((mask >> (2 * a)) & 1u) : ((mask >> (2 * a + 1)) & 1u);
      tw[a][0] = dir ? 0.5f : 1.f;
      tw[a][1] = 0.f;
    }
  }
  cx<T> acc = mk(T(0), T(0));
#pragma unroll
  for (int c2 = 0; c2 < 2; ++c2) {
    const float wz = tw[2][c2];
    if (wz == 0.f) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const float wy = tw[1][b];
      if (wy == 0.f) continue;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float wx = tw[0][a];
        if (wx == 0.f) continue;
        acc = axpy(widen<T>(wx * wy * wz), get(ti[0][a], ti[1][b], ti[2][c2]), acc);
      }
    }
  }
  return acc;
}

template <typename T>
__device__ __forceinline__ cx<T> prolong_value(Cell p, int rx, int ry, int rz, int cnx, int cny, int cnz,
                                               uint32_t mask, const cx<T>* zc) {
  return prolong_value_at<T>(p, rx, ry, rz, cnx, cny, cnz, mask, [&](int X, int Y, int Z) {
    return zc[((int64_t)Z * cny + Y) * cnx + X];
  });
}

}  // namespace fks
