// One red-black Gauss-Seidel sweep (both half sweeps) of a small 3D multigrid
// level in one launch (the inexact inner solve of Section 4, Eq. zmmoditer),
// with the neighbouring stages fused where there are any: the zero start, the
// interpolation of the coarser level's correction before the sweep, and the
// update of the outer iterate z_k after it.
//
// A half sweep of its own (k_gs) costs a launch, about 2.6 us on a level of
// 16^3 or 32^3 cells however little it does. Here a block marches up a chunk
// of planes over a tile of the x-y plane and updates the first colour on plane
// q and the second on plane q - 1 in the same step: four launches per V-cycle
// and level instead of nine (32^3 complex64: 16.7 us against 23.8; 16^3: 14.4
// against 22). On large levels a step's latency (about 1 us) costs more than
// reading the level again from L2: 128^3 22 to 28 us a sweep against 22.4.
//   - A thread owns the pairs of cells (2 p, 2 p + 1) of one row in all planes:
//     one cell of each colour per plane. The neighbours in z are then its own
//     values of the planes below and above, in registers, as is the one inside
//     the pair; the other x neighbour and the two in y come from shared memory,
//     which holds one value per pair and colour.
//   - The first colour is recomputed on a ring of one cell around the tile (one
//     pair in x, one row in y, one plane in z); it only reads old values of the
//     second colour, one cell further out.
//   - Old values of the second colour are never overwritten, in shared memory
//     or in global memory (the result goes to another buffer: neighbouring
//     tiles read this one's cells), so a step needs one block barrier.
//   - The coefficients of the next plane are loaded a step ahead.
// Every update repeats k_gs's arithmetic in its order (a neighbour outside the
// grid adds t * 0 instead of nothing), so the results are bitwise those of the
// half sweeps.
#include "grid.cuh"
#include "stencil.cuh"

namespace fks {

constexpr int SWEEP_THREADS = 384;  // most threads per block
constexpr int SWEEP_BLOCKS = 2;     // blocks per SM

template <typename T>
struct SweepProl {  // the correction of the level below (coarsened by 2 in every axis)
  uint32_t mask;
  int cnx, cny, cnz;
  const cx<T>* zc;
  int64_t vsc;
};

// what a pair of cells needs besides z: the left and the right cell's f,
// 1/diagonal, faces (x: left of the pair, inside, right of it; y: below and
// above each; z: above each)
template <typename T>
struct SweepPair {
  cx<T> f[2], id[2];
  T x[3], yl[2], yh[2], zh[2];
};

template <typename T>
struct alignas(2 * sizeof(cx<T>)) cx2 {
  cx<T> a, b;
};
template <typename T>
struct alignas(2 * sizeof(T)) re2 {
  T a, b;
};

// two consecutive values; one load where the rows start on even offsets
template <bool EVEN, typename T>
__device__ __forceinline__ void pair_c(const cx<T>* p, bool second, cx<T>* o) {
  if constexpr (EVEN) {
    const cx2<T> v = *(const cx2<T>*)p;
    o[0] = v.a;
    o[1] = v.b;
  } else {
    o[0] = p[0];
    o[1] = second ? p[1] : mk(T(0), T(0));
  }
}
template <bool EVEN, typename T, typename C>
__device__ __forceinline__ void pair_r(const C* p, bool second, T* o) {
  if constexpr (EVEN && sizeof(C) == sizeof(T)) {
    const re2<T> v = *(const re2<T>*)p;
    o[0] = v.a;
    o[1] = v.b;
  } else {
    o[0] = ldc<T>(p, 0);
    o[1] = second ? ldc<T>(p, 1) : T(0);
  }
}

template <typename T, typename C, int MODE, bool EVEN>
__global__ void __launch_bounds__(SWEEP_THREADS, SWEEP_BLOCKS)
    k_sweep3(LevelView<T, C> L, SweepGeom G, const SlotState* st, const cx<T>* __restrict__ invd,
             const cx<T>* __restrict__ f, const cx<T>* __restrict__ zin, cx<T>* __restrict__ zout, int64_t vs,
             int color, SweepProl<T> P, z64* __restrict__ Zk, int64_t vsZk, int64_t zcol) {
  pdl_enter();
  constexpr bool ZERO = MODE & SWEEP_ZERO, PROL = MODE & SWEEP_PROLONG, CORR = MODE & SWEEP_CORRECT;
  constexpr int NT = SWEEP_THREADS;
  __shared__ cx<T> sA[2][NT];  // old second colour
  __shared__ cx<T> sB[2][NT];  // new first colour
  const int slot = blockIdx.z;
  if (st && (!st[slot].active || st[slot].inner_done)) return;
  const SlotState* me = st + slot;
  const int nx = L.nx, ny = L.ny, nz = L.nz, sxy = nx * ny, np = (nx + 1) >> 1;
  const int t = threadIdx.x, r = t / G.txp, ii = t - r * G.txp;
  const int bx = blockIdx.x % G.ntx, by = blockIdx.x / G.ntx;
  const int op0 = bx * G.opx;
  const int gp = max(op0 - 1, 0) + ii, gj = by * G.oy - 2 + r;
  const int k0 = blockIdx.y * G.oz, k1 = min(k0 + G.oz, nz);
  // the thread's column: in the grid (its old second colour is read), in the
  // inner ring (its first colour is updated), in the tile (written)
  const bool in = r < G.oy + 4 && gp < np && gj >= 0 && gj < ny;
  const bool upd = in && r >= 1 && r <= G.oy + 2;
  const bool out = in && r >= 2 && r <= G.oy + 1 && gp >= op0 && gp < op0 + G.opx;
  const int i0 = 2 * gp;
  const bool right = EVEN || i0 + 1 < nx;  // the pair has a right cell
  const cx<T> none = mk(T(0), T(0));
  const int c0 = gj * nx + i0;  // left cell in plane 0
  const cx<T>* fs = f + slot * vs;
  const cx<T>* zs = zin + slot * vs;
  const cx<T>* ids = invd + (int64_t)me->tau * L.n;

  // interpolation of the coarse correction (prolong_value_at's weights, order
  // and arithmetic; a neighbour past the boundary has weight 0 there)
  const cx<T>* zc = nullptr;
  int dY = 0;
  T wx[2][2], wy[2];
  if constexpr (PROL) {
    const bool lo = gp > 0, hi = gp + 1 < P.cnx;
    wx[0][0] = lo ? T(0.75) : ((P.mask & 1u) ? T(0.5) : T(1));
    wx[0][1] = lo ? T(0.25) : T(0);
    wx[1][0] = hi ? T(0.75) : ((P.mask & 2u) ? T(0.5) : T(1));
    wx[1][1] = hi ? T(0.25) : T(0);
    const int J = gj >> 1, JN = (gj & 1) ? J + 1 : J - 1;
    const bool yn = JN >= 0 && JN < P.cny;
    wy[0] = yn ? T(0.75) : ((P.mask & ((gj & 1) ? 8u : 4u)) ? T(0.5) : T(1));
    wy[1] = yn ? T(0.25) : T(0);
    dY = yn ? (JN - J) * P.cnx : 0;
    zc = P.zc + slot * P.vsc + J * P.cnx + gp;
  }
  // old value of the second colour's cell of this pair on plane k
  auto old = [&](int k) -> cx<T> {
    if (ZERO || !in || k < 0 || k >= nz) return none;
    const int h = (1 + color + gj + k) & 1;
    if (h && !right) return none;
    cx<T> v = zs[k * sxy + c0 + h];
    if constexpr (PROL) {
      const int K = k >> 1, KN = (k & 1) ? K + 1 : K - 1;
      const bool zn = KN >= 0 && KN < P.cnz;
      const T wz0 = zn ? T(0.75) : ((P.mask & ((k & 1) ? 32u : 16u)) ? T(0.5) : T(1)), wz1 = zn ? T(0.25) : T(0);
      const T wx0 = h ? wx[1][0] : wx[0][0], wx1 = h ? wx[1][1] : wx[0][1];
      const int dX = wx1 == T(0) ? 0 : (h ? 1 : -1);
      const int sc = P.cnx * P.cny;
      const cx<T>* p0 = zc + K * sc;
      const cx<T>* p1 = zn ? zc + KN * sc : p0;
      const T w00 = mulT(wx0, wy[0]), w10 = mulT(wx1, wy[0]), w01 = mulT(wx0, wy[1]), w11 = mulT(wx1, wy[1]);
      cx<T> a = axpy(mulT(w00, wz0), p0[0], none);
      a = axpy(mulT(w10, wz0), p0[dX], a);
      a = axpy(mulT(w01, wz0), p0[dY], a);
      a = axpy(mulT(w11, wz0), p0[dY + dX], a);
      a = axpy(mulT(w00, wz1), p1[0], a);
      a = axpy(mulT(w10, wz1), p1[dX], a);
      a = axpy(mulT(w01, wz1), p1[dY], a);
      a = axpy(mulT(w11, wz1), p1[dY + dX], a);
      v = v + a;
    }
    return v;
  };
  auto coef = [&](int k) -> SweepPair<T> {
    SweepPair<T> s{};
    if (!upd || k < 0 || k >= nz) return s;
    const int c = k * sxy + c0, row = k * ny + gj;
    pair_c<EVEN>(fs + c, right, s.f);
    pair_c<EVEN>(ids + c, right, s.id);
    const C* fx = L.fx + (c + row);
    s.x[0] = ldc<T>(fx, 0);
    s.x[1] = ldc<T>(fx, 1);
    s.x[2] = right ? ldc<T>(fx, 2) : T(0);
    const C* fy = L.fy + (c + k * nx);
    pair_r<EVEN>(fy, right, s.yl);
    pair_r<EVEN>(fy + nx, right, s.yh);
    pair_r<EVEN>(L.fz + (c + sxy), right, s.zh);
    return s;
  };
  // 1/d (f + sum t z_nb) of the cell at position h of its pair; B points at this
  // pair's value of the other colour in shared memory
  auto update = [&](const SweepPair<T>& s, T zl, int h, const cx<T>* B, cx<T> own, cx<T> below, cx<T> above) -> cx<T> {
    const bool have = h ? ii + 1 < G.txp : ii > 0;
    const cx<T> far = have ? B[h ? 1 : -1] : none;
    cx<T> a = axpy(h ? s.x[1] : s.x[0], h ? own : far, h ? s.f[1] : s.f[0]);
    a = axpy(h ? s.x[2] : s.x[1], h ? far : own, a);
    a = axpy(h ? s.yl[1] : s.yl[0], B[-G.txp], a);
    a = axpy(h ? s.yh[1] : s.yh[0], B[G.txp], a);
    a = axpy(zl, below, a);
    a = axpy(h ? s.zh[1] : s.zh[0], above, a);
    return (h ? s.id[1] : s.id[0]) * a;
  };

  int q = k0 - 1;
  int p = (color + gj + q) & 1;  // position of the first colour in the pair on plane q
  cx<T> am = none, ac = none, ap = none;  // old second colour below, on and above plane q
  cx<T> bmm = none, bm = none;            // new first colour on q - 2 and q - 1
  SweepPair<T> cur = coef(q), prev{};
  T zl0 = T(0), zl1 = T(0), pzl = T(0);   // faces below: first and second colour on q, second on q - 1
  if (!ZERO) {
    am = old(q - 1);
    ac = old(q);
    ap = old(q + 1);
    sA[(q + 2) & 1][t] = ac;
  }
  if (upd && q >= 0 && (p == 0 || right)) zl0 = ldc<T>(L.fz, q * sxy + c0 + p);
  __syncthreads();
  for (; q <= k1; ++q) {
    // the next plane's coefficients and the old value above it, a step ahead
    SweepPair<T> nxt{};
    cx<T> an = none;
    if (q < k1) {
      nxt = coef(q + 1);
      an = old(q + 2);
    }
    cx<T> b = none;
    if (upd) {
      if constexpr (ZERO) b = (p ? cur.id[1] : cur.id[0]) * (p ? cur.f[1] : cur.f[0]);
      else b = update(cur, zl0, p, sA[(q + 2) & 1] + t, ac, am, ap);
    }
    sB[(q + 2) & 1][t] = b;
    if (out && q > k0) {
      // second colour on plane q - 1, at position p of the pair there
      const cx<T> e = update(prev, pzl, p, sB[(q + 1) & 1] + t, bm, bmm, b);
      const int c = (q - 1) * sxy + c0;
      if constexpr (CORR) {
        z64* zk = Zk + slot * vsZk + (int64_t)(me->k - 1) * zcol + c;
        const bool first = me->cycles == 0;
        const z64 e0 = cvt<double>(p ? bm : e), e1 = cvt<double>(p ? e : bm);
        zk[0] = first ? e0 : (zk[0] + e0);
        if (right) zk[1] = first ? e1 : (zk[1] + e1);
      } else {
        cx<T>* zo = zout + slot * vs + c;
        if constexpr (EVEN) {
          *(cx2<T>*)zo = cx2<T>{p ? bm : e, p ? e : bm};
        } else {
          zo[0] = p ? bm : e;
          if (right) zo[1] = p ? e : bm;
        }
      }
    }
    if (!ZERO) sA[(q + 1) & 1][t] = ap;
    __syncthreads();
    bmm = bm;
    bm = b;
    am = ac;
    ac = ap;
    ap = an;
    pzl = zl1;
    // the face above a cell is the one below the next plane's cell there, of the other colour
    zl1 = p ? cur.zh[1] : cur.zh[0];
    zl0 = p ? cur.zh[0] : cur.zh[1];
    prev = cur;
    cur = nxt;
    p ^= 1;
  }
}

SweepGeom sweep_geom(const LevelHost& L, int nslot) {
  return sweep_geometry(L.nx, L.ny, L.nz, nslot, SWEEP_THREADS, SWEEP_BLOCKS, (int)sizeof(float));
}

// Cells (times the batch's slots) up to which the march beats the half sweeps:
// 48^3 in complex64 (20.3 us of sweeps per V-cycle against 26.5; 64^3 is even).
// complex128 has none: the recomputed ring costs FP64 time, and they gained on
// some grids and lost on others (solves with the half sweeps and with the march
// on levels up to 2000, 16384 and 131072 cells: 45 x 53 x 37 77.2, 77.6, 78.3 and
// 87.8 ms; 18 x 22 x 24 41.8, 39.0, 38.6 and 38.6; 64 x 48 x 48 73.1, 73.2, 72.5 and
// 68.0).
bool sweep3_ok(const LevelHost& L, int nslot) { return L.nz > 1 && L.n * nslot <= 131072; }

template <typename T, typename C, bool EVEN>
static void launch_c(const LevelHost& L, const SweepGeom& G, int mode, const SlotState* st, const cx<T>* invd,
                     const cx<T>* f, const cx<T>* zin, cx<T>* zout, int64_t vs, int nslot, int color,
                     const SweepProl<T>& P, z64* Zk, int64_t vsZk, int64_t zcol, cudaStream_t s) {
  const dim3 g(G.ntx * G.nty, G.ntz, nslot), b((G.txp * (G.oy + 4) + 31) & ~31);
  auto go = [&](auto kernel) {
    launch_pdl(kernel, g, b, 0, s, view_as<T, C>(L), G, st, invd, f, zin, zout, vs, color, P, Zk, vsZk, zcol);
  };
  switch (mode) {
    case 0: go(k_sweep3<T, C, 0, EVEN>); break;
    case SWEEP_ZERO: go(k_sweep3<T, C, SWEEP_ZERO, EVEN>); break;
    case SWEEP_PROLONG: go(k_sweep3<T, C, SWEEP_PROLONG, EVEN>); break;
    default: go(k_sweep3<T, C, SWEEP_CORRECT, EVEN>);
  }
}

template <typename T>
void launch_sweep3(const LevelHost& L, const SweepGeom& G, const LevelHost* below, uint32_t mask, int mode,
                   const SlotState* st, const cx<T>* invd, const cx<T>* f, const cx<T>* zin, cx<T>* zout, int64_t vs, const cx<T>* zc,
                   int nslot, int color, z64* Zk, int64_t vsZk, int64_t zcol, int bf16, cudaStream_t s) {
  SweepProl<T> P{};
  if (mode & SWEEP_PROLONG) P = SweepProl<T>{mask, below->nx, below->ny, below->nz, zc, below->n};
  auto go = [&](auto c) {
    using C = decltype(c);
    if (L.nx % 2 == 0) launch_c<T, C, true>(L, G, mode, st, invd, f, zin, zout, vs, nslot, color, P, Zk, vsZk, zcol, s);
    else launch_c<T, C, false>(L, G, mode, st, invd, f, zin, zout, vs, nslot, color, P, Zk, vsZk, zcol, s);
  };
  if (bf16) go(__nv_bfloat16{});
  else go(T{});
}

template void launch_sweep3<float>(const LevelHost&, const SweepGeom&, const LevelHost*, uint32_t, int,
                                   const SlotState*, const z32*, const z32*, const z32*, z32*, int64_t, const z32*,
                                   int, int, z64*, int64_t, int64_t, int, cudaStream_t);

}  // namespace fks
