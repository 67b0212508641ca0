// Smoothed-aggregation algebraic multigrid for K + tau M (amg.cu): the host
// setup of one tau's hierarchy and the V-cycle that preconditions the BiCGSTAB
// steps of a CSR operator's inner solve (Section 6).
#pragma once
#include <string>
#include <vector>

#include "common.cuh"

namespace fks {

constexpr int AMG_MAX_LEVELS = 16;
constexpr int64_t AMG_MAX_DENSE = 4096;  // largest coarsest level (dense inverse)

// One level of one tau's hierarchy on the device, values in the cycle precision T.
template <typename T>
struct AmgLevel {
  int64_t n, nc;                  // unknowns of this level and of the next (0 on the coarsest)
  const int64_t* arp;             // A_l (level 0: K + tau M on the entries where K or M is nonzero)
  const int32_t* aci;
  const cx<T>* av;
  const cx<T>* dinv;              // 1 / diag(A_l)
  T omega;                        // Jacobi weight 4 / (3 rho_l)
  const int64_t* prp;             // P_l, n x nc
  const int32_t* pci;
  const cx<T>* pv;
  const int64_t* rrp;             // R_l = P_l^T, nc x n
  const int32_t* rci;
  const cx<T>* rv;
  const cx<T>* cinv;              // coarsest level: dense inverse, row-major n x n
};

// ---------------------------------------------------------------- host setup
struct AmgCsr {                   // complex128 CSR, columns sorted within a row
  int64_t n = 0, m = 0;
  std::vector<int64_t> rp;
  std::vector<int32_t> ci;
  std::vector<z64> v;
};

struct AmgHostLevel {
  AmgCsr A, P, R;
  std::vector<z64> dinv;
  double omega = 0.0;
};

struct AmgHost {
  std::vector<AmgHostLevel> lv;
  std::vector<z64> cinv;          // dense inverse of the coarsest A (row-major)
};

// Aggregates of every level but the coarsest. They depend on the sparsity
// pattern only, so the first tau's build fixes them for every other tau.
struct AmgAgg {
  std::vector<std::vector<int32_t>> agg;
  std::vector<int32_t> count;
};

// The hierarchy of A0 (level 0; its pattern is the strength graph). With
// agg->agg empty the aggregates are computed and stored; otherwise they are
// reused and fix the number of levels. Returns "" or an error message.
std::string amg_build(const AmgCsr& A0, int max_levels, int64_t max_coarse, AmgAgg* agg, AmgHost* out);

// Device copies of a host hierarchy in precision T: every allocation is
// appended to `mem` (the caller frees them, also after an error), one
// AmgLevel per level to `levels`.
template <typename T>
cudaError_t amg_upload(const AmgHost& h, std::vector<void*>& mem, std::vector<AmgLevel<T>>& levels);

// ---------------------------------------------------------------- V-cycle
// Per-level work vectors of a batch ([nslot][n_l] each, cycle precision) and
// the device table of the batch's hierarchies: tab[tau * L + l].
template <typename T>
struct AmgRun {
  const AmgLevel<T>* tab;
  int L, nu;
  int64_t n[AMG_MAX_LEVELS];
  cx<T>* f[AMG_MAX_LEVELS];       // right-hand side of level l >= 1
  cx<T>* x[AMG_MAX_LEVELS];       // iterate
  cx<T>* y[AMG_MAX_LEVELS];       // second Jacobi buffer
  cx<T>* r[AMG_MAX_LEVELS];       // residual, then (l >= 1) the level's result
};

struct BcgScal;
struct SlotState;

#ifdef __CUDACC__
// Per-row arithmetic of the V-cycle, shared by the stage kernels (amg.cu) and
// the cooperative cycle (csr.cu) so that both give the same bits. Vectors are
// read through L2 (__ldcg): in the cooperative kernel other blocks wrote them
// before the last grid barrier.
template <typename T>
__device__ __forceinline__ cx<T> amg_ld(const cx<T>* p) {
  if constexpr (sizeof(T) == 8) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return mk(v.x, v.y);
  } else {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return mk(v.x, v.y);
  }
}

// In complex128 a row takes two lanes, one for the real and one for the
// imaginary part: a warp's FP64 instruction occupies its SM sub-partition for
// 64 clocks whatever it does, and a product's six per entry become three on
// twice the warps. The rows are then dealt to the warps one by one over the
// blocks (warp w of block b is number w * gridDim.x + b), so that a level of a
// few dozen warps spreads over the chip instead of filling the first blocks
// (841 rows: 9.5 us a sweep on four SMs, 5.6 so). complex64 keeps consecutive
// rows in a block, whose vector entries meet in its L1 (64.0 against 68.6 ms
// on 101^2 nodes with three sources). AmgVal is what a lane holds of a complex
// value: all of it (complex64), or its part.
template <typename T>
struct AmgLane {
  static constexpr int LPR = sizeof(T) == 8 ? 2 : 1;
  int64_t first, stride;
  int part;
  __device__ __forceinline__ AmgLane() {
    const int lane = threadIdx.x & 31, wb = blockDim.x >> 5;
    constexpr int RW = 32 / LPR;
    const int64_t w = LPR == 2 ? (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x
                             : (int64_t)blockIdx.x * wb + (threadIdx.x >> 5);
    first = w * RW + lane / LPR;
    stride = (int64_t)gridDim.x * wb * RW;
    part = lane & (LPR - 1);
  }
};
template <typename T>
struct AmgValOf { typedef cx<T> type; };
template <>
struct AmgValOf<double> { typedef double type; };
template <typename T>
using AmgVal = typename AmgValOf<T>::type;

__device__ __forceinline__ z32 amg_get(const z32* p, int) { return amg_ld(p); }
__device__ __forceinline__ double amg_get(const z64* p, int part) { return __ldcg((const double*)p + part); }
__device__ __forceinline__ void amg_put(z32* p, int, z32 v) { *p = v; }
__device__ __forceinline__ void amg_put(z64* p, int part, double v) { ((double*)p)[part] = v; }
__device__ __forceinline__ z32 amg_sub(z32 a, z32 b) { return a - b; }
__device__ __forceinline__ double amg_sub(double a, double b) { return a - b; }
__device__ __forceinline__ z32 amg_add(z32 a, z32 b) { return a + b; }
__device__ __forceinline__ double amg_add(double a, double b) { return a + b; }
__device__ __forceinline__ z32 amg_scale(float s, z32 a) { return s * a; }
__device__ __forceinline__ double amg_scale(double s, double a) { return mulT(s, a); }
// the lane's part of a * b (operator*'s arithmetic), both parts of b given:
// own = b's part here, oth = the other
__device__ __forceinline__ double amg_part(z64 a, double own, double oth, int part) {
  const double t = mulT(a.im, oth);
  return fmaT(a.re, own, __hiloint2double(__double2hiint(t) ^ (part ? 0 : 0x80000000), __double2loint(t)));
}
__device__ __forceinline__ z32 amg_mul(z32 d, z32 v, int) { return d * v; }
__device__ __forceinline__ double amg_mul(z64 d, double v, int part) {
  const double oth = __shfl_xor_sync(3u << ((threadIdx.x & 31) & ~1), v, 1);
  return amg_part(d, v, oth, part);
}

// sum_q v_q x[col_q] over one CSR row, in order. In complex64 the entries of x
// are fetched eight at a time, so that a row waits for few L2 latencies (101^2
// nodes, three sources: 59.9 against 65.1 ms a solve). In complex128, two at a
// time: 174.9 ms on 256^2 nodes, against 207.8 one by one, 179.8 by four and
// 182 by explicit batches of four, which cost the cooperative cycle registers.
template <typename T>
__device__ __forceinline__ AmgVal<T> amg_term(cx<T> a, cx<T> x, int part);
template <>
__device__ __forceinline__ z32 amg_term<float>(z32 a, z32 x, int) { return a * x; }
template <>
__device__ __forceinline__ double amg_term<double>(z64 a, z64 x, int part) {
  return amg_part(a, part ? x.im : x.re, part ? x.re : x.im, part);
}
template <typename T>
__device__ __forceinline__ AmgVal<T> amg_row(const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                             const cx<T>* __restrict__ v, int64_t row, const cx<T>* x, int part) {
  AmgVal<T> acc{};
  int64_t q = rp[row];
  const int64_t e = rp[row + 1];
  if constexpr (sizeof(T) == 8) {
#pragma unroll 2
    for (; q < e; ++q) acc = acc + amg_term<T>(v[q], amg_ld(x + ci[q]), part);
    return acc;
  }
  constexpr int B = 8;
  for (; q + B <= e; q += B) {
    cx<T> xv[B];
#pragma unroll
    for (int b = 0; b < B; ++b) xv[b] = amg_ld(x + ci[q + b]);
#pragma unroll
    for (int b = 0; b < B; ++b) acc = acc + amg_term<T>(v[q + b], xv[b], part);
  }
  if (q < e) {
    cx<T> xv[B];
#pragma unroll
    for (int b = 0; b < B - 1; ++b) xv[b] = amg_ld(x + ci[min(q + b, e - 1)]);
#pragma unroll
    for (int b = 0; b < B - 1; ++b)
      if (q + b < e) acc = acc + amg_term<T>(v[q + b], xv[b], part);
  }
  return acc;
}

// first sweep from zero: omega D^{-1} f at row i (elementwise; its producer computes it)
template <typename T>
__device__ __forceinline__ cx<T> amg_first(const AmgLevel<T>& A, int64_t i, cx<T> f) {
  return A.omega * (A.dinv[i] * f);
}

// The phases of the V-cycle over a lane's rows.
// a later sweep: xo = x + omega D^{-1} (f - A x)
template <typename T>
__device__ __forceinline__ void amg_sweep_rows(const AmgLevel<T>& A, int64_t n, const cx<T>* f,
                                               const cx<T>* x, cx<T>* xo) {
  const AmgLane<T> w;
  for (int64_t i = w.first; i < n; i += w.stride) {
    const AmgVal<T> r = amg_sub(amg_get(f + i, w.part), amg_row<T>(A.arp, A.aci, A.av, i, x, w.part));
    amg_put(xo + i, w.part, amg_add(amg_get(x + i, w.part), amg_scale(A.omega, amg_mul(A.dinv[i], r, w.part))));
  }
}
// r = f - A x
template <typename T>
__device__ __forceinline__ void amg_resid_rows(const AmgLevel<T>& A, int64_t n, const cx<T>* f,
                                               const cx<T>* x, cx<T>* r) {
  const AmgLane<T> w;
  for (int64_t i = w.first; i < n; i += w.stride)
    amg_put(r + i, w.part, amg_sub(amg_get(f + i, w.part), amg_row<T>(A.arp, A.aci, A.av, i, x, w.part)));
}
// fc = P^T r on the next level C, and there (`sweep`) the first sweep xc = omega D^{-1} fc
template <typename T>
__device__ __forceinline__ void amg_restrict_rows(const AmgLevel<T>& A, const AmgLevel<T>& C, 
                                                  int64_t nc, const cx<T>* r, cx<T>* fc, cx<T>* xc, bool sweep) {
  const AmgLane<T> w;
  for (int64_t a = w.first; a < nc; a += w.stride) {
    const AmgVal<T> v = amg_row<T>(A.rrp, A.rci, A.rv, a, r, w.part);
    amg_put(fc + a, w.part, v);
    if (sweep) amg_put(xc + a, w.part, amg_scale(C.omega, amg_mul(C.dinv[a], v, w.part)));
  }
}
// x += P e
template <typename T>
__device__ __forceinline__ void amg_prolong_rows(const AmgLevel<T>& A, int64_t n, cx<T>* x,
                                                 const cx<T>* e) {
  const AmgLane<T> w;
  for (int64_t i = w.first; i < n; i += w.stride)
    amg_put(x + i, w.part, amg_add(amg_get(x + i, w.part), amg_row<T>(A.prp, A.pci, A.pv, i, e, w.part)));
}

// row `row` of the coarsest level's dense inverse times f, by one warp (lanes
// over columns, fixed-order shuffle reduction); the sum is valid in lane 0
template <typename T>
__device__ __forceinline__ cx<T> amg_coarse_row(const AmgLevel<T>& A, int64_t row, const cx<T>* f, int lane) {
  const int64_t n = A.n;
  cx<T> acc = mk(T(0), T(0));
  for (int64_t j = lane; j < n; j += 32) acc = acc + A.cinv[row * n + j] * amg_ld(f + j);
  for (int s = 16; s > 0; s >>= 1) {
    acc.re += __shfl_down_sync(0xffffffffu, acc.re, s);
    acc.im += __shfl_down_sync(0xffffffffu, acc.im, s);
  }
  return acc;
}
#endif

// out0 = V_0(f0) for every slot whose inner solve runs and whose BiCGSTAB
// cycle has not halted (sc may be null); returns the number of launches. The
// first sweep of level 0, R.x[0] = omega_0 D_0^{-1} f0, must already be there:
// the kernel that produces f0 writes it.
template <typename T>
int launch_amg_vcycle(const AmgRun<T>& R, const SlotState* st, const BcgScal* sc, const cx<T>* f0, cx<T>* out0,
                      int nslot, cudaStream_t s);

}  // namespace fks
