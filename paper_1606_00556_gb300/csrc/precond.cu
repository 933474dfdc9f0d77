// CPR-FPF preconditioner (paper Sec. 3.2, Alg. 2) on the colour-split
// layout: Quasi-IMPES decoupling, red-black block ILU(0) as the local solver
// R, an aggregation AMG V-cycle on the pressure block A_pp, and their
// composition.
//
// Red-black block ILU(0).  With the red cells ordered first, red rows have
// no lower part and black-black blocks lie off the pattern except on the
// diagonal, so ILU(0) reduces to
//     D_b' = D_b - sum_{r ~ b} A_br D_r^{-1} A_rb     (pivot blocks of black cells)
// and (L U)^{-1} f is three stencil passes:
//     t_r = D_r^{-1} f_r;   z_b = D_b'^{-1} (f_b - sum A_br t_r);
//     z_r = t_r - D_r^{-1} sum A_rb z_b.
//
// AMG.  Level 0 is the (0,0) entry of every block of D_QI^{-1} A on the
// colour-split grid; level l+1 aggregates the 2x2x2 boxes of level l
// (piecewise-constant P, Galerkin P^T A P, still 7-point); coarsening stops
// at <= coarse_max cells, whose dense inverse is formed once per setup.
// V(nu1, nu2) with red-black Gauss-Seidel: red then black before the coarse
// correction, black then red after it.  After a black half sweep only red
// cells carry a residual, so restriction sums red residuals.  The levels that
// fit one thread-block cluster run in one launch (k_amg_resident); without
// that form the levels of at most kTailCells cells run inside one thread block
// (k_tail, k_tail_smem).
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <new>

#include "bo_internal.cuh"
#include "per_device.h"

namespace bo {
namespace {

constexpr int kTailThreads = 1024;
constexpr int64_t kTailCells = 4096;
constexpr int kCoarseMax = 128;
constexpr size_t kTailSmemMax = 200 * 1024;  // stage the tail levels in shared memory up to this size

// ---------------------------------------------------------------- 3x3 blocks
// inverse by Gauss-Jordan elimination with partial pivoting; false if a
// pivot is zero or the result is not finite.  Each pivot row is scaled by
// one reciprocal: on GB300 an FP64 division is a long sequence of FP64
// instructions, and six of them per pivot made the ILU setup FP64-bound.
template <typename T>
__device__ bool inv3(const T a[9], T out[9]) {
  T m[3][6];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      m[i][j] = a[3 * i + j];
      m[i][3 + j] = (i == j) ? T(1) : T(0);
    }
  for (int k = 0; k < 3; ++k) {
    int p = k;
    for (int i = k + 1; i < 3; ++i)
      if (fabs(m[i][k]) > fabs(m[p][k])) p = i;
    if (m[p][k] == T(0)) return false;
    if (p != k)
      for (int j = 0; j < 6; ++j) { const T t = m[k][j]; m[k][j] = m[p][j]; m[p][j] = t; }
    const T rp = T(1) / m[k][k];
    for (int j = 0; j < 6; ++j) m[k][j] *= rp;
    for (int i = 0; i < 3; ++i) {
      if (i == k) continue;
      const T f = m[i][k];
      for (int j = 0; j < 6; ++j) m[i][j] -= f * m[k][j];
    }
  }
  bool ok = true;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      out[3 * i + j] = m[i][3 + j];
      ok &= isfinite(out[3 * i + j]);
    }
  return ok;
}

// decoupled block (colour, slot) of the cell at half index q: row 0 becomes
// g0 row0 + g1 row1 + g2 row2 with the cell's weights (paper Sec. 3.2,
// D_QI^{-1} A), FP64
__device__ __forceinline__ void dec_block(const Geom& g, const double* __restrict__ A, const double* __restrict__ w,
                                          int color, int slot, int64_t q, double b[9]) {
  const double g0 = w[vidx(g, 0, color, q)], g1 = w[vidx(g, 1, color, q)], g2 = w[vidx(g, 2, color, q)];
  double a[9];
#pragma unroll
  for (int rc = 0; rc < 9; ++rc) a[rc] = A[plane(g, color, slot, rc) + q];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    b[c] = g0 * a[c] + g1 * a[3 + c] + g2 * a[6 + c];
    b[3 + c] = a[3 + c];
    b[6 + c] = a[6 + c];
  }
}

template <typename T>
__device__ __forceinline__ void mul3(const T a[9], const T b[9], T c[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) c[3 * i + j] = a[3 * i] * b[j] + a[3 * i + 1] * b[3 + j] + a[3 * i + 2] * b[6 + j];
}

// Storage and arithmetic types.  S is the storage type of the matrix-like
// arrays (decoupled matrix, ILU pivot inverses, AMG coefficients, coarse
// inverse): double, float or BF16; vectors and arithmetic use T (double for
// S = double, float otherwise).  cv converts a stored value to T, to_store
// an FP64 value to S.
template <typename T, typename S>
__device__ __forceinline__ T cv(S v) { return (T)v; }
template <>
__device__ __forceinline__ float cv<float, __nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename S>
__device__ __forceinline__ S to_store(double v) { return (S)v; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(double v) { return __float2bfloat16_rn((float)v); }

// ---------------------------------------------------------------- setup kernels
// Quasi-IMPES decoupling (paper Sec. 3.2): row 0 of each cell becomes
// g . (row0, row1, row2) with g = (1, -a01/a11, -a02/a22) from the cell's
// diagonal block.  Where that pressure pivot is not positive (injector cells
// flooded to residual oil: the oil row carries no pressure information and
// the water pivot is negative), the cell takes the exact local decoupling,
// g = row 0 of A_ii^{-1} (pivot 1), which keeps the AMG operator's diagonal
// positive for the Gauss-Seidel smoother.  With abf set every cell takes
// that row: the ABF decoupling (D = block diagonal of A) restricted to the
// pressure row, which is all of it the CPR needs (block ILU(0) is invariant
// under a block-diagonal left scaling).  Writes the weights [3][N] and the
// decoupled blocks in storage type S.  The weights are formed in FP64; for
// FP32 or BF16 storage the decoupled rows are formed from the split copy of
// A in split FP32 pairs (FP32 instructions; the result rounded once to S),
// unless the split copy could not hold every value (*range).
template <typename S>
__device__ __forceinline__ S store_split(df v) {
  return to_store<S>((double)__fadd_rn(v.hi, v.lo));
}
template <>
__device__ __forceinline__ float store_split<float>(df v) { return __fadd_rn(v.hi, v.lo); }
template <>
__device__ __forceinline__ __nv_bfloat16 store_split<__nv_bfloat16>(df v) {
  return __float2bfloat16_rn(__fadd_rn(v.hi, v.lo));
}

template <typename S>
__global__ void k_decouple(Geom g, const double* __restrict__ A, const float2* __restrict__ A2,
                           const int* __restrict__ range, S* __restrict__ At, double* __restrict__ w,
                           float* __restrict__ wf, double* __restrict__ di0, int abf, DevState* st) {
  wait_prior_grid();
  const bool split = sizeof(S) < sizeof(double) && A2 && !*range;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x) {
    const int color = (int)(t / g.Nh);
    const int64_t q = t - color * g.Nh;
    double D[9];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) D[rc] = A[plane(g, color, kDiag, rc) + q];
    double g0 = 1.0, g1 = 0.0, g2 = 0.0;
    if (D[4] == 0.0 || D[8] == 0.0 || !isfinite(D[4]) || !isfinite(D[8])) {
      atomicOr(&st->err, kErrBreakdown);
    } else {
      g1 = -D[1] / D[4];
      g2 = -D[2] / D[8];
      if (abf || !(g0 * D[0] + g1 * D[3] + g2 * D[6] > 0.0)) {
        double inv[9];
        if (inv3(D, inv)) {
          g0 = inv[0];
          g1 = inv[1];
          g2 = inv[2];
        } else {
          atomicOr(&st->err, kErrBreakdown);
        }
      }
    }
    w[vidx(g, 0, color, q)] = g0;
    w[vidx(g, 1, color, q)] = g1;
    w[vidx(g, 2, color, q)] = g2;
    if (wf) {
      wf[vidx(g, 0, color, q)] = (float)g0;
      wf[vidx(g, 1, color, q)] = (float)g1;
      wf[vidx(g, 2, color, q)] = (float)g2;
    }
    if (split) {
      int bad = 0;
      const float2 g0p = df_split_bits(g0, &bad), g1p = df_split_bits(g1, &bad), g2p = df_split_bits(g2, &bad);
      const df gs0{g0p.x, g0p.y}, gs1{g1p.x, g1p.y}, gs2{g2p.x, g2p.y};
#pragma unroll
      for (int s = 0; s < 7; ++s) {
        df a[9];
#pragma unroll
        for (int rc = 0; rc < 9; ++rc) {
          const float2 v = A2[a2_index(g, color, s * 9 + rc, q)];
          a[rc] = df{v.x, v.y};
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          df r = df_fma_acc(df{0.f, 0.f}, gs0, a[c]);
          r = df_fma_acc(r, gs1, a[3 + c]);
          r = df_norm(df_fma_acc(r, gs2, a[6 + c]));
          At[at_index(g, color, s * 9 + c, q)] = store_split<S>(r);
          At[at_index(g, color, s * 9 + 3 + c, q)] = store_split<S>(a[3 + c]);
          At[at_index(g, color, s * 9 + 6 + c, q)] = store_split<S>(a[6 + c]);
          if (s == kDiag && c == 0 && (r.hi == 0.f || !isfinite(r.hi))) atomicOr(&st->err, kErrBreakdown);
        }
      }
      continue;
    }
#pragma unroll
    for (int s = 0; s < 7; ++s) {
      double a[9];
#pragma unroll
      for (int rc = 0; rc < 9; ++rc) a[rc] = A[plane(g, color, s, rc) + q];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        At[at_index(g, color, s * 9 + c, q)] = to_store<S>(g0 * a[c] + g1 * a[3 + c] + g2 * a[6 + c]);
        At[at_index(g, color, s * 9 + 3 + c, q)] = to_store<S>(a[3 + c]);
        At[at_index(g, color, s * 9 + 6 + c, q)] = to_store<S>(a[6 + c]);
      }
      if (s == kDiag) {
        const double app = g0 * a[0] + g1 * a[3] + g2 * a[6];
        if (app == 0.0 || !isfinite(app)) atomicOr(&st->err, kErrBreakdown);
        if (di0) di0[t] = 1.0 / app;  // (FP64 storage: At holds app itself)
      }
    }
  }
}

// Pivots are always factored in FP64 from the FP64 matrix and the
// Quasi-IMPES weights, whatever precision they are stored in: the black
// pivots are Schur complements D_b - sum A_br D_r^{-1} A_rb that cancel
// strongly where the permeability contrast is high, and FP32 arithmetic there
// can leave the local solver unstable.

// red pivots: D_r^{-1} of the decoupled diagonal blocks, stored in type S
// and, for the black pass, in FP64 in `red64` ([rc][N/2]); with SPLIT the
// black pass takes them as split pairs instead (red64 read as float2)
template <typename S, bool SPLIT>
__global__ void k_ilu_red(Geom g, const double* __restrict__ A, const double* __restrict__ w, S* __restrict__ Dinv,
                          double* __restrict__ red64, DevState* st) {
  wait_prior_grid();
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    double d[9], inv[9];
    dec_block(g, A, w, 0, kDiag, q, d);
    if (!inv3(d, inv)) {
      atomicOr(&st->err, kErrBreakdown);
      for (int rc = 0; rc < 9; ++rc) inv[rc] = 0.0;
    }
    int bad = 0;
    for (int rc = 0; rc < 9; ++rc) {
      Dinv[(size_t)rc * g.N + q] = to_store<S>(inv[rc]);
      if (SPLIT) reinterpret_cast<float2*>(red64)[(size_t)rc * g.Nh + q] = df_split_bits(inv[rc], &bad);
      else red64[(size_t)rc * g.Nh + q] = inv[rc];
    }
  }
}

// The black pivots of a preconditioner stored in FP32 or BF16, formed in
// split FP32 pairs (48 significant bits, FP32 instructions) instead of FP64:
// the six products L D_r^{-1} U per cell are 324 multiply-adds, which on
// GB300's FP64 rate made this the slowest setup kernel.  The decoupled blocks
// come from the split copy of A and split weights; the Schur complement is
// summed in split pairs and inverted in FP64.  (An FP64-stored
// preconditioner keeps the FP64 kernel below.)
__device__ __forceinline__ void dec_block_split(const Geom& g, const float2* __restrict__ A2, const df wq[3],
                                                int color, int slot, int64_t q, df b[9]) {
  df a[9];
#pragma unroll
  for (int rc = 0; rc < 9; ++rc) {
    const float2 v = A2[a2_index(g, color, slot * 9 + rc, q)];
    a[rc] = df{v.x, v.y};
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    df r = df_fma_acc(df{0.f, 0.f}, wq[0], a[c]);
    r = df_fma_acc(r, wq[1], a[3 + c]);
    r = df_fma_acc(r, wq[2], a[6 + c]);
    b[c] = df_norm(r);
    b[3 + c] = a[3 + c];
    b[6 + c] = a[6 + c];
  }
}

__device__ __forceinline__ void weights_split(const Geom& g, const double* __restrict__ w, int color, int64_t q,
                                              df wq[3]) {
  int bad = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float2 v = df_split_bits(w[vidx(g, k, color, q)], &bad);
    wq[k] = df{v.x, v.y};
  }
}

__device__ __forceinline__ void mul3_split(const df a[9], const df b[9], df c[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      df r = df_fma_acc(df{0.f, 0.f}, a[3 * i], b[j]);
      r = df_fma_acc(r, a[3 * i + 1], b[3 + j]);
      r = df_fma_acc(r, a[3 * i + 2], b[6 + j]);
      c[3 * i + j] = df_norm(r);
    }
}

template <typename S>
__global__ void k_ilu_black_split(Geom g, const float2* __restrict__ A2, const double* __restrict__ A,
                                  const int* __restrict__ range, const double* __restrict__ w,
                                  const float2* __restrict__ red2, S* __restrict__ Dinv, DevState* st) {
  wait_prior_grid();
  if (*range) {  // a value outside the split form's range: the FP64 products, from A
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
      const Cell c = decode(g, 1, q);
      double Sc[9], inv[9];
      dec_block(g, A, w, 1, kDiag, q, Sc);
      for (int s = 0; s < 7; ++s) {
        if (s == kDiag) continue;
        const int64_t nq = nbr(g, c, q, s);
        if (nq < 0) continue;
        double L[9], U[9], Dr[9], T1[9], T2[9];
        dec_block(g, A, w, 1, s, q, L);
        dec_block(g, A, w, 0, opposite(s), nq, U);
        for (int rc = 0; rc < 9; ++rc) {
          const float2 v = red2[(size_t)rc * g.Nh + nq];
          Dr[rc] = (double)v.x + (double)v.y;
        }
        mul3(L, Dr, T1);
        mul3(T1, U, T2);
        for (int rc = 0; rc < 9; ++rc) Sc[rc] -= T2[rc];
      }
      if (!inv3(Sc, inv)) {
        atomicOr(&st->err, kErrBreakdown);
        for (int rc = 0; rc < 9; ++rc) inv[rc] = 0.0;
      }
      for (int rc = 0; rc < 9; ++rc) Dinv[(size_t)rc * g.N + g.Nh + q] = to_store<S>(inv[rc]);
    }
    return;
  }
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 1, q);
    df wb[3], Sc[9];
    weights_split(g, w, 1, q, wb);
    dec_block_split(g, A2, wb, 1, kDiag, q, Sc);
#pragma unroll 1
    for (int s = 0; s < 7; ++s) {
      if (s == kDiag) continue;
      const int64_t nq = nbr(g, c, q, s);
      if (nq < 0) continue;
      df wr[3], L[9], U[9], Dr[9], T1[9], T2[9];
      weights_split(g, w, 0, nq, wr);
      dec_block_split(g, A2, wb, 1, s, q, L);
      dec_block_split(g, A2, wr, 0, opposite(s), nq, U);
#pragma unroll
      for (int rc = 0; rc < 9; ++rc) {
        const float2 v = red2[(size_t)rc * g.Nh + nq];
        Dr[rc] = df{v.x, v.y};
      }
      mul3_split(L, Dr, T1);
      mul3_split(T1, U, T2);
#pragma unroll
      for (int rc = 0; rc < 9; ++rc) Sc[rc] = df_add(Sc[rc], df_neg(T2[rc]));
    }
    double S64[9], inv[9];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) S64[rc] = df_to_double(Sc[rc]);
    if (!inv3(S64, inv)) {
      atomicOr(&st->err, kErrBreakdown);
      for (int rc = 0; rc < 9; ++rc) inv[rc] = 0.0;
    }
    for (int rc = 0; rc < 9; ++rc) Dinv[(size_t)rc * g.N + g.Nh + q] = to_store<S>(inv[rc]);
  }
}

// black pivots: D_b' = D_b - sum_r A_br D_r^{-1} A_rb with the FP64 red
// inverses, stored inverted in type S
template <typename S>
__global__ void k_ilu_black(Geom g, const double* __restrict__ A, const double* __restrict__ w,
                            const double* __restrict__ red64, S* __restrict__ Dinv, DevState* st) {
  wait_prior_grid();
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 1, q);
    double Sc[9], inv[9];
    dec_block(g, A, w, 1, kDiag, q, Sc);
#pragma unroll
    for (int s = 0; s < 7; ++s) {
      if (s == kDiag) continue;
      const int64_t nq = nbr(g, c, q, s);
      if (nq < 0) continue;
      double L[9], U[9], Dr[9], T1[9], T2[9];
      dec_block(g, A, w, 1, s, q, L);
      dec_block(g, A, w, 0, opposite(s), nq, U);
      for (int rc = 0; rc < 9; ++rc) Dr[rc] = red64[(size_t)rc * g.Nh + nq];
      mul3(L, Dr, T1);
      mul3(T1, U, T2);
      for (int rc = 0; rc < 9; ++rc) Sc[rc] -= T2[rc];
    }
    if (!inv3(Sc, inv)) {
      atomicOr(&st->err, kErrBreakdown);
      for (int rc = 0; rc < 9; ++rc) inv[rc] = 0.0;
    }
    for (int rc = 0; rc < 9; ++rc) Dinv[(size_t)rc * g.N + g.Nh + q] = to_store<S>(inv[rc]);
  }
}

// ------------------------------------------------------------ AMG setup
struct LevelDims {
  int32_t nx, ny, nz;
  int64_t n;
};

// (i, j, k) of natural index c of a level (c < 2^31), by 32-bit division
struct Ijk {
  int i, j, k;
};
__device__ __forceinline__ Ijk ijk_of(const LevelDims& L, int64_t c) {
  const uint32_t cu = (uint32_t)c, nx = (uint32_t)L.nx, ny = (uint32_t)L.ny;
  const uint32_t r = cu / nx;
  return Ijk{(int)(cu - r * nx), (int)(r % ny), (int)(r / ny)};
}

__device__ __forceinline__ int64_t nat_index(const LevelDims& L, int i, int j, int k) {
  return i + (int64_t)L.nx * (j + (int64_t)L.ny * k);
}

// FP64 levels keep the reciprocals of the diagonal behind the seven
// coefficients: the Gauss-Seidel sweeps divide with their help, since an FP64
// division is about ten FP64 multiply-adds where the rest of a cell's
// update takes six (FP32 divisions are cheap and stay divisions).
//
// s / d from the rounded reciprocal r = 1 / d: the product, corrected once by
// its residual, is the rounded quotient (P. Markstein, IBM J. Res. Dev. 34,
// 1990); the product alone is off by up to one unit more.  (An infinite
// product has no residual.)  The correction costs a Newton step of 128x128x64
// 0.6 of 18 ms, of 20x20x5 17 of 980 us.
__device__ __forceinline__ double divide_by(double s, double d, double r) {
  const double q = s * r, c = fma(fma(-q, d, s), r, q);
  return isfinite(c) ? c : q;
}
template <typename S>
__host__ __device__ constexpr int level_slots() { return sizeof(S) == 8 ? 8 : 7; }
template <typename S>
__device__ __forceinline__ void put_reciprocal(S* __restrict__ c, const LevelDims& C, int64_t I, double diag) {
  if constexpr (sizeof(S) == 8) c[(size_t)7 * C.n + I] = 1.0 / diag;
}

// Galerkin products: coarse entry (I, J) = sum of the fine entries a_ij with
// i in aggregate I and j in aggregate J.  A block takes 32 consecutive coarse
// cells, a thread per child: consecutive threads read consecutive fine cells,
// and all of a child's loads are in flight at once.  The rows meet in shared
// memory, where a warp takes one of the seven entries of the 32 cells (a
// child's entries towards its own aggregate join the diagonal) and adds it up
// as a loop over the children (x fastest) and their slots does: another order
// leaves another last bit, which some systems amplify (see the CPR's passes
// below).  The value is written in FP64 (the next level's input) and in the
// storage type.  Level 1 is bound by its FP64 products, 168 + 56 warp
// instructions for 32 coarse cells at 16 cycles, and the loads.  Measured, one
// thread per coarse cell and a conversion kernel -> this: level 1 of
// 128x128x64 78 -> 71 us, of 62x45x19 60 -> 11, of 20x20x5 (FP64) 46 -> 10; a
// coarser level 17-22 -> 4-6 us.
template <typename S, typename Row>
__device__ __forceinline__ void galerkin_block(const LevelDims& C, int fnx, int fny, int fnz, Row row,
                                               double* __restrict__ c64, S* __restrict__ c, DevState* st) {
  static_assert(kThreads == 256, "8 children of 32 coarse cells");
  __shared__ double a[7][kThreads];
  const int t = threadIdx.x, q = t & 31, e = t >> 5;
  for (int64_t I0 = blockIdx.x * (int64_t)32; I0 < C.n; I0 += gridDim.x * (int64_t)32) {
    double v[7] = {0, 0, 0, 0, 0, 0, 0};  // (zero where the child is missing)
    const int64_t I = I0 + ((t & 63) >> 1);
    if (I < C.n) {
      const Ijk p = ijk_of(C, I);
      const int i = 2 * p.i + (t & 1), j = 2 * p.j + ((t >> 6) & 1), k = 2 * p.k + (t >> 7);
      if (i < fnx && j < fny && k < fnz) row(i, j, k, v);
    }
#pragma unroll
    for (int s = 0; s < 7; ++s) a[s][t] = v[s];
    __syncthreads();
    if (e < 7 && I0 + q < C.n) {
      auto child = [&](int s, int x, int y, int z) { return a[s][(2 * z + y) * 64 + 2 * q + x]; };
      const int side = e > kDiag;
      double sum = 0.0;
      if (e == kDiag) {
#pragma unroll
        for (int z = 0; z < 2; ++z)
#pragma unroll
          for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
              if (z) sum += child(kZm, x, y, z);
              if (y) sum += child(kYm, x, y, z);
              if (x) sum += child(kXm, x, y, z);
              sum += child(kDiag, x, y, z);
              if (!x) sum += child(kXp, x, y, z);
              if (!y) sum += child(kYp, x, y, z);
              if (!z) sum += child(kZp, x, y, z);
            }
      } else {  // the four children at a face
#pragma unroll
        for (int hi = 0; hi < 2; ++hi)
#pragma unroll
          for (int lo = 0; lo < 2; ++lo)
            sum += e == kXm || e == kXp   ? child(e, side, lo, hi)
                   : e == kYm || e == kYp ? child(e, lo, side, hi)
                                          : child(e, lo, hi, side);
      }
      c64[(size_t)e * C.n + I0 + q] = sum;
      c[(size_t)e * C.n + I0 + q] = to_store<S>(sum);
      if (e == kDiag) {
        put_reciprocal(c, C, I0 + q, sum);
        if (sum == 0.0 || !isfinite(sum)) atomicOr(&st->err, kErrBreakdown);
      }
    }
    __syncthreads();
  }
}

// level 1 from level 0 (the decoupled pressure block, FP64 from A and the weights)
template <typename S>
__global__ void __launch_bounds__(kThreads) k_galerkin0(Geom g, const double* __restrict__ A, const double* __restrict__ w,
                            LevelDims C, double* __restrict__ c64, S* __restrict__ c, DevState* st) {
  wait_prior_grid();
  galerkin_block(C, g.nx, g.ny, g.nz, [&](int i, int j, int k, double (&a)[7]) {
    const int color = (i + j + k) & 1;
    const int64_t q = (i + (int64_t)g.nx * (j + (int64_t)g.ny * k)) >> 1;
    const double g0 = w[vidx(g, 0, color, q)], g1 = w[vidx(g, 1, color, q)], g2 = w[vidx(g, 2, color, q)];
    double r[21];
#pragma unroll
    for (int s = 0; s < 7; ++s)
#pragma unroll
      for (int u = 0; u < 3; ++u) r[3 * s + u] = A[plane(g, color, s, 3 * u) + q];
    // (blocks outside the grid are stored as zeros)
#pragma unroll
    for (int s = 0; s < 7; ++s) a[s] = g0 * r[3 * s] + g1 * r[3 * s + 1] + g2 * r[3 * s + 2];
  }, c64, c, st);
}

// level l+1 from natural-order level l
template <typename S>
__global__ void __launch_bounds__(kThreads) k_galerkinn(LevelDims F, const double* __restrict__ f64, LevelDims C,
                            double* __restrict__ c64, S* __restrict__ c, DevState* st) {
  wait_prior_grid();
  galerkin_block(C, F.nx, F.ny, F.nz, [&](int i, int j, int k, double (&a)[7]) {
    const int64_t cf = nat_index(F, i, j, k);
#pragma unroll
    for (int s = 0; s < 7; ++s) a[s] = f64[(size_t)s * F.n + cf];
  }, c64, c, st);
}

// ------------------------------------------------------- dense inverse
// Hardware barrier of all threads of a thread-block cluster, with release /
// acquire semantics at cluster scope: every memory write of the cluster's
// thread blocks before it is visible to their reads after it.  It is not a
// spin on a flag: every thread of the cluster reaches every barrier (the
// control flow is uniform).
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address in block `rank` of the cluster that corresponds to p in this block's shared memory
__device__ __forceinline__ uint32_t cluster_map(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// The matrix to invert: dense (M), or the coarsest level's stencil, natural
// order (c64) or level 0 in the colour-split index order (A and the weights).
struct DenseSrc {
  const double* M;
  const double* c64;
  LevelDims L;
  Geom g;
  const double* A;
  const double* w;
};
// Row `row` of the matrix over the warp: lane's columns lane + 32 c.
template <int CPL>
__device__ __forceinline__ void dense_row(const DenseSrc& d, int n, int row, double a[CPL]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c = 0; c < CPL; ++c) a[c] = 0.0;
  if (row >= n) return;
  if (d.M) {
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      if (lane + 32 * c < n) a[c] = d.M[(size_t)row * n + lane + 32 * c];
    return;
  }
  // lane s < 7 fetches stencil entry s and its column; every lane then takes the ones that are its own
  int i, j, k, color = 0;
  if (d.c64) {
    i = row % d.L.nx;
    j = (row / d.L.nx) % d.L.ny;
    k = row / (d.L.nx * d.L.ny);
  } else {
    color = row >= d.g.Nh;
    const Cell c = decode(d.g, color, row - color * d.g.Nh);
    i = c.i; j = c.j; k = c.k;
  }
  double v = 0.0;
  int col = -1;
  if (lane < 7) {
    const int ni = i + (lane == kXp) - (lane == kXm), nj = j + (lane == kYp) - (lane == kYm),
              nk = k + (lane == kZp) - (lane == kZm);
    if (ni >= 0 && ni < d.L.nx && nj >= 0 && nj < d.L.ny && nk >= 0 && nk < d.L.nz) {
      const int nat = (int)nat_index(d.L, ni, nj, nk);
      if (d.c64) {
        v = d.c64[(size_t)lane * n + row];
        col = nat;
      } else {
        const int64_t q = row - color * d.g.Nh;
        v = d.w[vidx(d.g, 0, color, q)] * d.A[plane(d.g, color, lane, 0) + q] +
            d.w[vidx(d.g, 1, color, q)] * d.A[plane(d.g, color, lane, 3) + q] +
            d.w[vidx(d.g, 2, color, q)] * d.A[plane(d.g, color, lane, 6) + q];
        col = (int)(((ni + nj + nk) & 1) * d.g.Nh) + (nat >> 1);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < 7; ++s) {
    const double vs = __shfl_sync(0xffffffffu, v, s);
    const int cs = __shfl_sync(0xffffffffu, col, s);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
      if (cs == lane + 32 * c) a[c] += vs;
  }
}

// In-place Gauss-Jordan inversion with partial pivoting of an n x n matrix
// (n <= kCoarseMax), the inverse written in type S.  The matrix lives in
// registers, one row per warp and CPL columns per lane, and rows are never
// exchanged: a row that served as pivot is marked, and the permutation is
// applied when the result is written (row p_k of the eliminated matrix is
// row k of the inverse with column j in place p_j).  A step takes two
// barriers: one after every row has published its entry of column k, whose
// largest unused entry every warp then finds by itself (two redux
// operations on the bit pattern of |a|, then the lowest row), one after
// the pivot's warp has published the scaled pivot row.  What bounds it: up to
// 32 rows the chain of a step (barriers, the reduction, one FP64 division),
// so one block of 32 warps; above, the n^3 FP64 multiply-adds on one SM
// (545 us at n = 128 at the 2 per clock of GB300), so a cluster of eight
// blocks shares the rows and exchanges column and pivot row through
// distributed shared memory.  Measured against the form before it (matrix in
// shared memory, one thread scanning the column): n = 32 74 -> 29 us, n = 50
// 160 -> 68 us (93 in one block), n = 125 1010 -> 304 us.
constexpr int kGjCluster = 8;
template <typename S, int CPL, bool CLUSTER>
__global__ void __launch_bounds__(1024) k_gj_inverse(int n, DenseSrc d, S* __restrict__ Minv, int transposed,
                                                     DevState* st) {
  wait_prior_grid();
  __shared__ double colbuf[kCoarseMax], prow[kCoarseMax];
  __shared__ int piv[kCoarseMax];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = (int)blockIdx.x * ((int)blockDim.x >> 5) + warp;  // (the grid is the cluster)
  const bool mine = row < n;
  double a[CPL];
  dense_row<CPL>(d, n, row, a);
  unsigned used = 0;  // bit c: row lane + 32 c has been a pivot
  int myk = -1;
  auto barrier = [&]() {
    if (CLUSTER) cluster_sync_all();
    else __syncthreads();
  };
  if (CLUSTER) cluster_sync_all();  // every block of the cluster runs before its shared memory is written
  bool fail = false;
  for (int k = 0; k < n && !fail; ++k) {
    double v = a[0];
#pragma unroll
    for (int c = 1; c < CPL; ++c)
      if ((k >> 5) == c) v = a[c];
    const double fac = __shfl_sync(0xffffffffu, v, k & 31);
    if (mine) {
      if (CLUSTER) {
        if (lane < kGjCluster) st_cluster(cluster_map(colbuf + row, lane), fac);
      } else if (lane == 0) {
        colbuf[row] = fac;
      }
    }
    barrier();
    // the unused row with the largest |a| (the lowest such row): by the
    // high word of the magnitude (plus one; zero for a used row), then the
    // low word
    unsigned bh = 0, bl = 0, bi = 0x7fffffffu;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int i = lane + 32 * c;
      if (i < n && !((used >> c) & 1)) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(colbuf[i]);
        const unsigned h = ((unsigned)(u >> 32) & 0x7fffffffu) + 1u, l = (unsigned)u;
        if (h > bh || (h == bh && l > bl)) {
          bh = h;
          bl = l;
          bi = (unsigned)i;
        }
      }
    }
    const unsigned mh = __reduce_max_sync(0xffffffffu, bh);
    const unsigned ml = __reduce_max_sync(0xffffffffu, bh == mh ? bl : 0u);
    const int p = (int)__reduce_min_sync(0xffffffffu, bh == mh && bl == ml ? bi : 0x7fffffffu);
    fail = mh == 1u && ml == 0u;  // the column's largest unused entry is zero
    if ((p & 31) == lane) used |= 1u << (p >> 5);
    if (threadIdx.x == 0) piv[k] = p;
    if (row == p) {  // (warp-uniform)
      myk = k;
      // one reciprocal for the pivot row (an FP64 division is a long sequence)
      const double rp = 1.0 / fac;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        a[c] = (j == k ? 1.0 : a[c]) * rp;
        if (CLUSTER) {
#pragma unroll
          for (int b = 0; b < kGjCluster; ++b) st_cluster(cluster_map(prow + j, b), a[c]);
        } else {
          prow[j] = a[c];
        }
      }
    }
    barrier();
    if (mine && row != p) {
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = lane + 32 * c;
        a[c] = (j == k ? 0.0 : a[c]) - fac * prow[j];
      }
    }
  }
  barrier();
  if (fail) {
    if (threadIdx.x == 0) atomicOr(&st->err, kErrBreakdown);
    return;
  }
  if (!mine) return;
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int j = lane + 32 * c;
    if (j >= n) continue;
    Minv[transposed ? (size_t)piv[j] * n + myk : (size_t)myk * n + piv[j]] = to_store<S>(a[c]);
    if (!isfinite(a[c])) atomicOr(&st->err, kErrBreakdown);
  }
}

template <typename S>
cudaError_t launch_gj(int n, const DenseSrc& d, S* Minv, bool transposed, DevState* st, cudaStream_t s) {
  note_launch();
  if (n <= 32) return launch_pdl(k_gj_inverse<S, 1, false>, 1, 1024, 0, s, n, d, Minv, (int)transposed, st);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kGjCluster, 1, 1);
  cfg.blockDim = dim3(n <= 64 ? 256 : 512, 1, 1);  // 8 blocks x 8 or 16 warps, one row each
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kGjCluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (n <= 64) return cudaLaunchKernelEx(&cfg, k_gj_inverse<S, 2, true>, n, d, Minv, (int)transposed, st);
  return cudaLaunchKernelEx(&cfg, k_gj_inverse<S, 4, true>, n, d, Minv, (int)transposed, st);
}

// ------------------------------------------------------------ apply kernels
// Entry of the preconditioner: f = D_QI^{-1} v (DEC) or f = v, in precision
// T, fused with the first ILU pass on the red cells, t_r = D_r^{-1} f_r.
// v is FP64 or split pairs; sc the scale of an unnormalised Krylov vector.
// FP32 arithmetic reads the split input's high part (the low part lies
// below FP32's rounding) and the FP32 copy of the weights, so the FP32
// preconditioner issues no FP64 instruction here.
template <typename T>
__device__ __forceinline__ T in_get(const InV& v, size_t i, double sc) {
  if (v.f) {
    if constexpr (sizeof(T) == 4) return (float)sc * v.f[i];
    else return sc * ((double)v.f[i] + (double)v.f[v.n + i]);
  }
  return (T)(sc * v.d[i]);
}

template <typename T, typename S, bool DEC>
__global__ void k_cpr_entry(Geom g, InV v, const double* __restrict__ vs, const double* __restrict__ w,
                            const float* __restrict__ wf, const S* __restrict__ Dinv, T* __restrict__ f,
                            T* __restrict__ tv, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  const double sc = vs ? *vs : 1.0;  // scale of an unnormalised Krylov vector
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x) {
    const T v0 = in_get<T>(v, t, sc), v1 = in_get<T>(v, g.N + t, sc), v2 = in_get<T>(v, 2 * g.N + t, sc);
    T f0 = v0;
    if (DEC) {
      if constexpr (sizeof(T) == 4) f0 = fma3(0.f, wf[t], v0, wf[g.N + t], v1, wf[2 * g.N + t], v2);
      else f0 = fma3(0.0, w[t], v0, w[g.N + t], v1, w[2 * g.N + t], v2);
    }
    const T f1 = v1, f2 = v2;
    f[t] = f0;
    f[g.N + t] = f1;
    f[2 * g.N + t] = f2;
    if (t < g.Nh) {
      T d[9];
#pragma unroll
      for (int rc = 0; rc < 9; ++rc) d[rc] = cv<T>(Dinv[(size_t)rc * g.N + t]);
      tv[t] = d[0] * f0 + d[1] * f1 + d[2] * f2;
      tv[g.N + t] = d[3] * f0 + d[4] * f1 + d[5] * f2;
      tv[2 * g.N + t] = d[6] * f0 + d[7] * f1 + d[8] * f2;
    }
  }
}

// preconditioner output: FP64, or split pairs (exact for FP32 values)
template <typename T>
__device__ __forceinline__ void out_put(const OutV& o, size_t i, T v) {
  if (o.f) {
    if constexpr (sizeof(T) == 4) {
      o.f[i] = v;
      o.f[o.n + i] = 0.f;
    } else {
      const df d = df_from(v);
      o.f[i] = d.hi;
      o.f[o.n + i] = d.lo;
    }
  } else {
    o.d[i] = (double)v;
  }
}

template <typename T>
__global__ void k_widen_t(int64_t n, const T* __restrict__ a, double* __restrict__ b, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = (double)a[i];
}

template <typename T>
__global__ void k_copy_vec(int64_t n, const double* __restrict__ v, T* __restrict__ f, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    f[t] = (T)v[t];
}

// sum over the six off-diagonal blocks of a row of At times the other
// colour's vector u: s = sum_s At[color][s] u[nbr]
template <typename T, typename S>
__device__ __forceinline__ void offdiag_sum(const Geom& g, const S* __restrict__ At, int color, int64_t q,
                                            const Cell& c, const T* __restrict__ u, T s[3]) {
  const int oc = color ^ 1;
  s[0] = s[1] = s[2] = T(0);
  // (every slot's loads are issued; a missing neighbour reads this cell's
  // own entries and is masked to zero, so all loads can be in flight)
#pragma unroll
  for (int sl = 0; sl < 7; ++sl) {
    if (sl == kDiag) continue;
    const int64_t nb = nbr(g, c, q, sl);
    const bool ok = nb >= 0;
    const int64_t nq = ok ? nb : q;
    T u0 = u[vidx(g, 0, oc, nq)], u1 = u[vidx(g, 1, oc, nq)], u2 = u[vidx(g, 2, oc, nq)];
    if (!ok) u0 = u1 = u2 = T(0);
    const S* a = At + at_index(g, color, sl * 9, q);
    constexpr size_t P = 32;  // entries (rc) of a block lie 32 apart in a tile
    s[0] = fma3(s[0], cv<T>(ld_stream(a)), u0, cv<T>(ld_stream(a + P)), u1, cv<T>(ld_stream(a + 2 * P)), u2);
    s[1] = fma3(s[1], cv<T>(ld_stream(a + 3 * P)), u0, cv<T>(ld_stream(a + 4 * P)), u1, cv<T>(ld_stream(a + 5 * P)), u2);
    s[2] = fma3(s[2], cv<T>(ld_stream(a + 6 * P)), u0, cv<T>(ld_stream(a + 7 * P)), u1, cv<T>(ld_stream(a + 8 * P)), u2);
  }
}

// ILU pass 2 (black): z_b = D_b'^{-1} (f_b - sum A_br t_r), t_r = D_r^{-1} f_r
// (pass 1).  Pass 3 (red): x_r = t_r - D_r^{-1} sum A_rb x_b.
// blocks per SM the register budget is tuned for: the FP32 passes are
// memory-latency bound and want more warps; the FP64 ones are FP64-bound
template <typename T>
constexpr int ilu_min_blocks() { return sizeof(T) == 4 ? 4 : 3; }

template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, ilu_min_blocks<T>()) k_ilu_b(Geom g, const S* __restrict__ At, const S* __restrict__ Dinv, const T* __restrict__ f,
                        const T* __restrict__ tv, T* __restrict__ z, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 1, q);
    T s[3];
    offdiag_sum(g, At, 1, q, c, tv, s);
    const T r0 = f[vidx(g, 0, 1, q)] - s[0], r1 = f[vidx(g, 1, 1, q)] - s[1], r2 = f[vidx(g, 2, 1, q)] - s[2];
    T d[9];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) d[rc] = cv<T>(Dinv[(size_t)rc * g.N + g.Nh + q]);
    z[vidx(g, 0, 1, q)] = d[0] * r0 + d[1] * r1 + d[2] * r2;
    z[vidx(g, 1, 1, q)] = d[3] * r0 + d[4] * r1 + d[5] * r2;
    z[vidx(g, 2, 1, q)] = d[6] * r0 + d[7] * r1 + d[8] * r2;
  }
}

// (the black half of xb is read.)  OUT = false: z_r = x_r; OUT = true: the
// preconditioner's result, z_r + Pi_p e_r + x_r.
template <typename T, typename S, bool OUT>
__global__ void __launch_bounds__(kThreads, ilu_min_blocks<T>()) k_ilu_r2(Geom g, const S* __restrict__ At, const S* __restrict__ Dinv, const T* tv,
                         const T* xb, T* z, const T* __restrict__ e, OutV zo, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 0, q);
    T s[3];
    offdiag_sum(g, At, 0, q, c, xb, s);
    T d[9], x[3];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) d[rc] = cv<T>(Dinv[(size_t)rc * g.N + q]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T corr = d[3 * k] * s[0] + d[3 * k + 1] * s[1] + d[3 * k + 2] * s[2];
      x[k] = tv[vidx(g, k, 0, q)] - corr;
    }
    if (OUT) {
      out_put<T>(zo, vidx(g, 0, 0, q), z[vidx(g, 0, 0, q)] + e[q] + x[0]);
      out_put<T>(zo, vidx(g, 1, 0, q), z[vidx(g, 1, 0, q)] + x[1]);
      out_put<T>(zo, vidx(g, 2, 0, q), z[vidx(g, 2, 0, q)] + x[2]);
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) z[vidx(g, k, 0, q)] = x[k];
    }
  }
}

// s / d, in FP64 with the stored reciprocal at di[i] (see divide_by)
__device__ __forceinline__ double gs_divide(double s, double d, const double* __restrict__ di, size_t i) { return divide_by(s, d, di[i]); }
__device__ __forceinline__ float gs_divide(float s, float d, const float*, size_t) { return s / d; }

// ---- the rest of the CPR after its first local solve z = R^{-1} f
//   x2 = z + Pi_p e,  e = AMG(A_pp)^{-1} Pi_r (f - A z),  x3 = x2 + R^{-1} (f - A x2),
// the local solve of a residual r = f - A x2 being
//   t_r = D_r^{-1} r_r,  u_b = D_b'^{-1} (r_b - A_br t_r),
//   x3_b = x2_b + u_b,   x3_r = x2_r + (t_r - D_r^{-1} A_rb u_b).
// The black pass forms r_b and A_br t_r over one read of A_br, and so reads
// the off-diagonal blocks of the black rows once where a residual of all rows
// and a black ILU pass read them twice; every sum is added up in the order of
// those separate passes, which gives their results bit for bit.  Newton step
// with separate passes and no cluster form of the AMG -> now: 128x128x64 FP32
// 13.0 -> 11.9 ms, FP64 24.2 -> 20.8 ms, 256x256x128 BF16 91.5 -> 86.3 ms.
//
// Red rows of the red-black ILU(0)'s product are rows of the matrix itself,
// so in exact arithmetic r_r = 0, the AMG right-hand side is zero on red
// cells and x3_r = D_r^{-1} (f_r - A_rb x3_b): passes that use it read a third
// less (128x128x64 FP32 another 7%, FP64 14%).  They are not used.  On some 3%
// of systems (flooded injector cells) the preconditioner amplifies rounding so
// far that another order of its sums takes FGMRES to another iterate: solutions
// moved by 1e-9 to 4e-8 at a tolerance of 1e-8 in all three precisions.

// AMG right-hand side f0 = f_p - (A z)_p, and with it the V-cycle's first half
// sweep, x_r = f0_r / a_rr from zero
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 5 : 4) k_cpr_rhs(Geom g, const S* __restrict__ At,
                         const T* __restrict__ di0, const T* __restrict__ f, const T* __restrict__ z,
                         T* __restrict__ f0, T* __restrict__ x0, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x) {
    const int color = t >= g.Nh;
    const int64_t q = t - color * g.Nh;
    const Cell c = decode(g, color, q);
    T acc = T(0), diag = T(0);
    // (every slot's loads are issued; a missing neighbour reads this cell's
    // own entries and is masked to zero)
#pragma unroll
    for (int sl = 0; sl < 7; ++sl) {
      const int64_t nb = nbr(g, c, q, sl);
      const bool ok = nb >= 0;
      const int64_t nq = ok ? nb : q;
      const int xc = (sl == kDiag || !ok) ? color : (color ^ 1);
      T z0 = z[vidx(g, 0, xc, nq)], z1 = z[vidx(g, 1, xc, nq)], z2 = z[vidx(g, 2, xc, nq)];
      if (!ok) z0 = z1 = z2 = T(0);
      const S* a = At + at_index(g, color, sl * 9, q);
      constexpr size_t P = 32;  // entries (rc) of a block lie 32 apart in a tile
      const T a0 = cv<T>(ld_stream(a));
      if (sl == kDiag) diag = a0;
      acc = fma3(acc, a0, z0, cv<T>(ld_stream(a + P)), z1, cv<T>(ld_stream(a + 2 * P)), z2);
    }
    const T r = f[t] - acc;
    f0[t] = r;
    if (color == 0) x0[t] = gs_divide(r, diag, di0, (size_t)t);
  }
}

// t_r = D_r^{-1} (f - A x2)_r
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, 4) k_cpr_red(Geom g, const S* __restrict__ At,
                         const S* __restrict__ Dinv, const T* __restrict__ f, const T* __restrict__ z,
                         const T* __restrict__ e, T* __restrict__ tv, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 0, q);
    T s[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int sl = 0; sl < 7; ++sl) {
      const S* a = At + at_index(g, 0, sl * 9, q);
      constexpr size_t P = 32;  // entries (rc) of a block lie 32 apart in a tile
      const int64_t nb = nbr(g, c, q, sl);
      const bool ok = nb >= 0;
      const int64_t nq = ok ? nb : q;
      const int xc = sl == kDiag ? 0 : 1;
      T x0 = z[vidx(g, 0, xc, nq)] + e[(size_t)xc * g.Nh + nq], x1 = z[vidx(g, 1, xc, nq)], x2 = z[vidx(g, 2, xc, nq)];
      if (!ok) x0 = x1 = x2 = T(0);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        s[k] = fma3(s[k], cv<T>(ld_stream(a + 3 * k * P)), x0, cv<T>(ld_stream(a + (3 * k + 1) * P)), x1,
                    cv<T>(ld_stream(a + (3 * k + 2) * P)), x2);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = f[vidx(g, k, 0, q)] - s[k];
    T d[9];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) d[rc] = cv<T>(Dinv[(size_t)rc * g.N + q]);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      tv[vidx(g, k, 0, q)] = d[3 * k] * s[0] + d[3 * k + 1] * s[1] + d[3 * k + 2] * s[2];
  }
}

// u_b = D_b'^{-1} ((f - A x2)_b - A_br t_r) into the black half of ub (tv holds
// t_r) and the preconditioner's result x2_b + u_b
template <typename T, typename S>
__global__ void __launch_bounds__(kThreads, ilu_min_blocks<T>()) k_cpr_black(Geom g, const S* __restrict__ At,
                         const S* __restrict__ Dinv, const T* __restrict__ f, const T* __restrict__ tv,
                         const T* __restrict__ z, const T* __restrict__ e, T* __restrict__ ub, OutV zo,
                         const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < g.Nh; q += (int64_t)gridDim.x * blockDim.x) {
    const Cell c = decode(g, 1, q);
    const T x[3] = {z[vidx(g, 0, 1, q)] + e[g.Nh + q], z[vidx(g, 1, 1, q)], z[vidx(g, 2, 1, q)]};
    T acc[3] = {T(0), T(0), T(0)}, s[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int sl = 0; sl < 7; ++sl) {
      const S* a = At + at_index(g, 1, sl * 9, q);
      T y[3] = {x[0], x[1], x[2]}, t[3];
      if (sl != kDiag) {
        const int64_t nb = nbr(g, c, q, sl);
        const bool ok = nb >= 0;
        const int64_t nq = ok ? nb : q;
        y[0] = z[vidx(g, 0, 0, nq)] + e[nq], y[1] = z[vidx(g, 1, 0, nq)], y[2] = z[vidx(g, 2, 0, nq)];
#pragma unroll
        for (int k = 0; k < 3; ++k) t[k] = tv[vidx(g, k, 0, nq)];
        if (!ok) y[0] = y[1] = y[2] = t[0] = t[1] = t[2] = T(0);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const T a0 = cv<T>(ld_stream(a + 96 * k)), a1 = cv<T>(ld_stream(a + 96 * k + 32)), a2 = cv<T>(ld_stream(a + 96 * k + 64));
        acc[k] = fma3(acc[k], a0, y[0], a1, y[1], a2, y[2]);
        if (sl != kDiag) s[k] = fma3(s[k], a0, t[0], a1, t[1], a2, t[2]);
      }
    }
    T r[3], d[9];
#pragma unroll
    for (int k = 0; k < 3; ++k) r[k] = (f[vidx(g, k, 1, q)] - acc[k]) - s[k];
#pragma unroll
    for (int rc = 0; rc < 9; ++rc) d[rc] = cv<T>(Dinv[(size_t)rc * g.N + g.Nh + q]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T u = d[3 * k] * r[0] + d[3 * k + 1] * r[1] + d[3 * k + 2] * r[2];
      ub[vidx(g, k, 1, q)] = u;
      out_put<T>(zo, vidx(g, k, 1, q), x[k] + u);
    }
  }
}

// ---- AMG level 0 (colour-split, coefficients = plane (colour, slot, 0) of At)
// One cell of a level-0 Gauss-Seidel half sweep.
template <typename T, typename S>
__device__ __forceinline__ T gs0_value(const Geom& g, const S* __restrict__ At, const T* __restrict__ di0,
                                      const T* __restrict__ f, const T* __restrict__ x, int color, int zero_guess,
                                      int64_t q) {
  const int oc = color ^ 1;
  T s = f[(size_t)color * g.Nh + q];
  if (!zero_guess) {
    const Cell c = decode(g, color, q);
#pragma unroll
    for (int sl = 0; sl < 7; ++sl) {
      if (sl == kDiag) continue;
      const int64_t nb = nbr(g, c, q, sl);
      const T xv = x[(size_t)oc * g.Nh + (nb >= 0 ? nb : q)];
      s -= cv<T>(At[at_index(g, color, sl * 9, q)]) * (nb >= 0 ? xv : T(0));
    }
  }
  return gs_divide(s, cv<T>(At[at_index(g, color, kDiag * 9, q)]), di0, (size_t)color * g.Nh + q);
}

// A level-0 half sweep over a grid-stride range, B cells per thread at a
// time: the loads of all B cells are issued before any store (the stores go
// to this colour's half of x, which no cell of the sweep reads), so a
// thread's cells overlap their memory latency instead of queueing it.
template <int B, typename T, typename F>
__device__ __forceinline__ void sweep_batched(int64_t t0, int64_t nt, int64_t n, T* __restrict__ out, F value) {
  for (int64_t q0 = t0; q0 < n; q0 += (int64_t)B * nt) {
    T v[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int64_t q = q0 + b * nt;
      v[b] = q < n ? value(q) : T(0);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int64_t q = q0 + b * nt;
      if (q < n) out[q] = v[b];
    }
  }
}

// (B cells per thread at a time, their loads issued before their stores:
// a tile parameter of the per-kernel form that the batch autotuner sets)
template <typename T, typename S, int B>
__global__ void k_gs0(Geom g, const S* __restrict__ At, const T* __restrict__ di0, const T* __restrict__ f,
                      T* __restrict__ x, int color, int zero_guess, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  sweep_batched<B>(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, g.Nh,
                   x + (size_t)color * g.Nh, [&](int64_t q) { return gs0_value<T, S>(g, At, di0, f, x, color, zero_guess, q); });
}

// First post-smoothing half sweep (black cells) with the coarse correction
// folded in: the red neighbours are read as x_r + s x_c(aggregate).  This
// equals prolongating x += s P x_c on every cell and then sweeping the black
// cells, because the black sweep overwrites x_b and the red sweep that
// follows overwrites x_r without reading its old value.
template <typename T, typename S>
__device__ __forceinline__ T gs0_prolong_value(const Geom& g, const S* __restrict__ At, const T* __restrict__ di0,
                                              const T* __restrict__ f, const T* __restrict__ x, const LevelDims& C,
                                              const T* __restrict__ xc, T sc, int64_t q) {
  const int di[7] = {0, 0, -1, 0, 1, 0, 0}, dj[7] = {0, -1, 0, 0, 0, 1, 0}, dk[7] = {-1, 0, 0, 0, 0, 0, 1};
  const Cell c = decode(g, 1, q);
  T s = f[(size_t)g.Nh + q];
#pragma unroll
  for (int sl = 0; sl < 7; ++sl) {
    if (sl == kDiag) continue;
    const int64_t nb = nbr(g, c, q, sl);
    const bool ok = nb >= 0;
    const int64_t cn = ok ? nat_index(C, (c.i + di[sl]) / 2, (c.j + dj[sl]) / 2, (c.k + dk[sl]) / 2) : 0;
    const T xv = x[ok ? nb : q] + sc * xc[cn];
    s -= cv<T>(At[at_index(g, 1, sl * 9, q)]) * (ok ? xv : T(0));
  }
  return gs_divide(s, cv<T>(At[at_index(g, 1, kDiag * 9, q)]), di0, (size_t)g.Nh + q);
}

template <typename T, typename S, int B>
__global__ void k_gs0_prolong(Geom g, const S* __restrict__ At, const T* __restrict__ di0, const T* __restrict__ f,
                              T* __restrict__ x, LevelDims C, const T* __restrict__ xc, T sc, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  sweep_batched<B>(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, g.Nh, x + g.Nh,
                   [&](int64_t q) { return gs0_prolong_value<T, S>(g, At, di0, f, x, C, xc, sc, q); });
}

// Sum of level-0 residuals over aggregate I (red cells only when the last
// half sweep was black)
template <typename T, typename S>
__device__ __forceinline__ T restrict0_cell(const Geom& g, const S* __restrict__ At, const T* __restrict__ f,
                                            const T* __restrict__ x, const LevelDims& C, int64_t I, int red_only) {
  const Ijk cc = ijk_of(C, I);
  const int ci = cc.i, cj = cc.j, ck = cc.k;
  T acc = T(0);
  for (int dk = 0; dk < 2; ++dk)
    for (int dj = 0; dj < 2; ++dj)
      for (int di = 0; di < 2; ++di) {
        const int i = 2 * ci + di, j = 2 * cj + dj, k = 2 * ck + dk;
        if (i >= g.nx || j >= g.ny || k >= g.nz) continue;
        const int color = (i + j + k) & 1;
        if (red_only && color == 1) continue;
        const int64_t q = (i + (int64_t)g.nx * (j + (int64_t)g.ny * k)) >> 1;
        const Cell c{i, j, k, i & 1};
        T r = f[(size_t)color * g.Nh + q];
#pragma unroll
        for (int sl = 0; sl < 7; ++sl) {
          const int64_t nq = nbr(g, c, q, sl);
          if (nq < 0) continue;
          const int xc = (sl == kDiag) ? color : (color ^ 1);
          r -= cv<T>(At[at_index(g, color, sl * 9, q)]) * x[(size_t)xc * g.Nh + nq];
        }
        acc += r;
      }
  return acc;
}

template <typename T, typename S>
__global__ void k_restrict0(Geom g, const S* __restrict__ At, const T* __restrict__ f, const T* __restrict__ x,
                            LevelDims C, T* __restrict__ fc, int red_only, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; I < C.n; I += (int64_t)gridDim.x * blockDim.x)
    fc[I] = restrict0_cell<T, S>(g, At, f, x, C, I, red_only);
}

template <typename T>
__device__ __forceinline__ void prolong0_cell(const Geom& g, T* __restrict__ x, const LevelDims& C,
                                              const T* __restrict__ xc, T s, int64_t t) {
  const int color = (int)(t / g.Nh);
  const int64_t q = t - color * g.Nh;
  const Cell c = decode(g, color, q);
  x[t] += s * xc[nat_index(C, c.i / 2, c.j / 2, c.k / 2)];
}

template <typename T>
__global__ void k_prolong0(Geom g, T* __restrict__ x, LevelDims C, const T* __restrict__ xc, T s, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x)
    prolong0_cell<T>(g, x, C, xc, s, t);
}

// ---- natural-order levels (device functions shared by the multi-block
// kernels and the single-block tail)
template <typename T, typename S = T>
struct LevelView {
  LevelDims d;
  const S* c;  // level_slots n coefficients (storage type)
  T* f;
  T* x;
  __device__ __forceinline__ T cc(int slot, int64_t cidx) const { return cv<T>(c[slot * d.n + cidx]); }
  // s divided by the diagonal
  __device__ __forceinline__ T divided(T s, int64_t cidx) const {
    if constexpr (sizeof(S) == 8) return divide_by(s, cc(kDiag, cidx), c[7 * d.n + cidx]);
    else return s / cc(kDiag, cidx);
  }
};

template <typename T, typename S>
__device__ __forceinline__ void gs_cell(const LevelView<T, S>& L, int64_t cidx, int color, int zero_guess) {
  const Ijk p = ijk_of(L.d, cidx);
  const int i = p.i, j = p.j, k = p.k;
  if (((i + j + k) & 1) != color) return;
  T s = L.f[cidx];
  if (!zero_guess) {
    // every neighbour's loads are issued; a missing one reads the cell
    // itself and the value read is replaced by zero
    const int64_t nxy = (int64_t)L.d.nx * L.d.ny;
    const bool ok[6] = {k > 0, j > 0, i > 0, i < L.d.nx - 1, j < L.d.ny - 1, k < L.d.nz - 1};
    const int slot[6] = {kZm, kYm, kXm, kXp, kYp, kZp};
    const int64_t off[6] = {-nxy, -(int64_t)L.d.nx, -1, 1, (int64_t)L.d.nx, nxy};
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const T xv = L.x[ok[d] ? cidx + off[d] : cidx];
      s -= L.cc(slot[d], cidx) * (ok[d] ? xv : T(0));
    }
  }
  L.x[cidx] = L.divided(s, cidx);
}

template <typename T, typename S>
__device__ __forceinline__ T residual_cell(const LevelView<T, S>& L, int i, int j, int k) {
  const int64_t cidx = nat_index(L.d, i, j, k);
  const int64_t nxy = (int64_t)L.d.nx * L.d.ny;
  T r = L.f[cidx] - L.cc(kDiag, cidx) * L.x[cidx];
  if (k > 0) r -= L.cc(kZm, cidx) * L.x[cidx - nxy];
  if (j > 0) r -= L.cc(kYm, cidx) * L.x[cidx - L.d.nx];
  if (i > 0) r -= L.cc(kXm, cidx) * L.x[cidx - 1];
  if (i < L.d.nx - 1) r -= L.cc(kXp, cidx) * L.x[cidx + 1];
  if (j < L.d.ny - 1) r -= L.cc(kYp, cidx) * L.x[cidx + L.d.nx];
  if (k < L.d.nz - 1) r -= L.cc(kZp, cidx) * L.x[cidx + nxy];
  return r;
}

template <typename T, typename S>
__device__ __forceinline__ T restrict_cell(const LevelView<T, S>& F, const LevelDims& C, int64_t I, int red_only) {
  const Ijk cc = ijk_of(C, I);
  const int ci = cc.i, cj = cc.j, ck = cc.k;
  T acc = T(0);
  for (int dk = 0; dk < 2; ++dk)
    for (int dj = 0; dj < 2; ++dj)
      for (int di = 0; di < 2; ++di) {
        const int i = 2 * ci + di, j = 2 * cj + dj, k = 2 * ck + dk;
        if (i >= F.d.nx || j >= F.d.ny || k >= F.d.nz) continue;
        if (red_only && ((i + j + k) & 1)) continue;
        acc += residual_cell(F, i, j, k);
      }
  return acc;
}

template <typename T, typename S>
__device__ __forceinline__ void prolong_cell(const LevelView<T, S>& F, const LevelView<T, S>& C, int64_t cidx, T s) {
  const Ijk p = ijk_of(F.d, cidx);
  const int i = p.i, j = p.j, k = p.k;
  F.x[cidx] = F.x[cidx] + s * C.x[nat_index(C.d, i / 2, j / 2, k / 2)];
}

// black half sweep with the coarse correction of the red neighbours folded in
// (the natural-order counterpart of k_gs0_prolong)
template <typename T, typename S>
__device__ __forceinline__ void gs_cell_prolong(const LevelView<T, S>& L, const LevelView<T, S>& C, int64_t cidx, T sc) {
  const Ijk p = ijk_of(L.d, cidx);
  const int i = p.i, j = p.j, k = p.k;
  if (((i + j + k) & 1) != 1) return;
  const int64_t nxy = (int64_t)L.d.nx * L.d.ny;
  T s = L.f[cidx];
  const bool ok[6] = {k > 0, j > 0, i > 0, i < L.d.nx - 1, j < L.d.ny - 1, k < L.d.nz - 1};
  const int slot[6] = {kZm, kYm, kXm, kXp, kYp, kZp};
  const int64_t off[6] = {-nxy, -(int64_t)L.d.nx, -1, 1, (int64_t)L.d.nx, nxy};
  const int ci[6] = {i / 2, i / 2, (i - 1) / 2, (i + 1) / 2, i / 2, i / 2};
  const int cj[6] = {j / 2, (j - 1) / 2, j / 2, j / 2, (j + 1) / 2, j / 2};
  const int ck[6] = {(k - 1) / 2, k / 2, k / 2, k / 2, k / 2, (k + 1) / 2};
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const int64_t fi = ok[d] ? cidx + off[d] : cidx;
    const int64_t cn = ok[d] ? nat_index(C.d, ci[d], cj[d], ck[d]) : nat_index(C.d, i / 2, j / 2, k / 2);
    const T xv = L.x[fi] + sc * C.x[cn];
    s -= L.cc(slot[d], cidx) * (ok[d] ? xv : T(0));
  }
  L.x[cidx] = L.divided(s, cidx);
}

template <typename T, typename S>
__global__ void k_gsn_prolong(LevelView<T, S> L, LevelView<T, S> C, T sc, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < L.d.n; c += (int64_t)gridDim.x * blockDim.x)
    gs_cell_prolong(L, C, c, sc);
}

template <typename T, typename S>
__global__ void k_gsn(LevelView<T, S> L, int color, int zero_guess, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < L.d.n; c += (int64_t)gridDim.x * blockDim.x)
    gs_cell(L, c, color, zero_guess);
}

template <typename T, typename S>
__global__ void k_restrictn(LevelView<T, S> F, LevelView<T, S> C, int red_only, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; I < C.d.n; I += (int64_t)gridDim.x * blockDim.x)
    C.f[I] = restrict_cell(F, C.d, I, red_only);
}

template <typename T, typename S>
__global__ void k_prolongn(LevelView<T, S> F, LevelView<T, S> C, T s, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < F.d.n; c += (int64_t)gridDim.x * blockDim.x)
    prolong_cell(F, C, c, s);
}

template <typename T, typename S>
struct TailArgs {
  int first, last;  // levels first..last (last = coarsest)
  int nu1, nu2;
  T s;
  LevelView<T, S> lv[24];
  const S* inv;     // dense inverse of level `last`, transposed
};

// Dynamic shared memory of the single-block tail (one symbol for the whole
// translation unit).
extern __shared__ __align__(16) uint8_t g_tail_smem[];

// Views of the tail levels: in global memory (the kernel's arguments), or
// staged in the tail's shared memory.  The shared-memory views are rebuilt
// from offsets into g_tail_smem at each use, so the compiler sees shared
// addresses and issues shared-memory loads (pointers read back from a
// shared struct would be generic and take the slower generic path).
template <typename T, typename S>
struct TailGlobalViews {
  const TailArgs<T, S>* a;
  __device__ LevelView<T, S> lv(int l) const { return a->lv[l]; }
  __device__ const S* inv() const { return a->inv; }
};
template <typename T, typename S>
struct TailSharedViews {
  const TailArgs<T, S>* a;
  const uint32_t* off;  // per level: coefficient, right-hand side and iterate offsets; the inverse at off[72]
  __device__ LevelView<T, S> lv(int l) const {
    LevelView<T, S> v = a->lv[l];
    v.c = reinterpret_cast<const S*>(g_tail_smem + off[3 * l]);
    v.f = reinterpret_cast<T*>(g_tail_smem + off[3 * l + 1]);
    v.x = reinterpret_cast<T*>(g_tail_smem + off[3 * l + 2]);
    return v;
  }
  __device__ const S* inv() const { return reinterpret_cast<const S*>(g_tail_smem + off[72]); }
};

// x_first = V-cycle(f_first) over levels first..last by one thread block
template <typename T, typename S, typename Views>
__device__ void tail_cycle(const TailArgs<T, S>& a, const Views& vw) {
  const int nt = blockDim.x;
  for (int l = a.first; l < a.last; ++l) {
    const LevelView<T, S> L = vw.lv(l);
    if (a.nu1 == 0) {
      for (int64_t c = threadIdx.x; c < L.d.n; c += nt) L.x[c] = T(0);
      __syncthreads();
    }
    for (int sw = 0; sw < a.nu1; ++sw)
      for (int color = 0; color < 2; ++color) {
        for (int64_t c = threadIdx.x; c < L.d.n; c += nt) gs_cell(L, c, color, sw == 0 && color == 0);
        __syncthreads();
      }
    const LevelView<T, S> C = vw.lv(l + 1);
    for (int64_t I = threadIdx.x; I < C.d.n; I += nt) C.f[I] = restrict_cell(L, C.d, I, a.nu1 > 0);
    __syncthreads();
  }
  {
    const LevelView<T, S> C = vw.lv(a.last);
    const S* inv = vw.inv();
    const int64_t n = C.d.n;
    for (int64_t i = threadIdx.x; i < n; i += nt) {
      T s = T(0);
      for (int64_t j = 0; j < n; ++j) s += cv<T>(inv[j * n + i]) * C.f[j];
      C.x[i] = s;
    }
    __syncthreads();
  }
  for (int l = a.last - 1; l >= a.first; --l) {
    const LevelView<T, S> L = vw.lv(l);
    const LevelView<T, S> C = vw.lv(l + 1);
    if (a.nu2 == 0) {
      for (int64_t c = threadIdx.x; c < L.d.n; c += nt) prolong_cell(L, C, c, a.s);
      __syncthreads();
    }
    for (int sw = 0; sw < a.nu2; ++sw)
      for (int color = 1; color >= 0; --color) {
        for (int64_t c = threadIdx.x; c < L.d.n; c += nt) {
          if (sw == 0 && color == 1) gs_cell_prolong(L, C, c, a.s);
          else gs_cell(L, c, color, 0);
        }
        __syncthreads();
      }
  }
}

template <typename T, typename S>
__global__ void __launch_bounds__(kTailThreads) k_tail(TailArgs<T, S> a, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  tail_cycle(a, TailGlobalViews<T, S>{&a});
}

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~size_t(15); }

// shared-memory bytes that k_tail_smem needs for levels first..last
template <typename T, typename S>
__host__ __device__ size_t tail_smem_bytes(const TailArgs<T, S>& a) {
  size_t b = 0;
  for (int l = a.first; l <= a.last; ++l)
    b += align16(level_slots<S>() * a.lv[l].d.n * sizeof(S)) + 2 * align16(a.lv[l].d.n * sizeof(T));
  return b + align16((size_t)a.lv[a.last].d.n * a.lv[a.last].d.n * sizeof(S));
}

// The same V-cycle with the tail levels staged in shared memory: their
// coefficients, right-hand sides and iterates, and the coarse inverse, are
// copied in once, every sweep then reads shared memory instead of L2, and
// only the first tail level's iterate (read by the next finer level's
// prolongation) is copied back.
// Offsets of the tail levels in the dynamic shared memory (per level: the
// coefficients, the right-hand side and the iterate; the coarse inverse at
// off[72]), computed by thread 0.
template <typename T, typename S>
__device__ void tail_offsets(const TailArgs<T, S>& a, uint32_t* off) {
  if (threadIdx.x == 0) {
    uint32_t o = 0;
    for (int l = a.first; l <= a.last; ++l) {
      const uint32_t n = (uint32_t)a.lv[l].d.n;
      off[3 * l] = o;
      o += (uint32_t)align16(level_slots<S>() * n * sizeof(S));
      off[3 * l + 1] = o;
      o += (uint32_t)align16(n * sizeof(T));
      off[3 * l + 2] = o;
      o += (uint32_t)align16(n * sizeof(T));
    }
    off[72] = o;
  }
}

// Copies the tail levels' coefficients and the coarse inverse into shared
// memory (they do not change during a V-cycle; the caller synchronises).
template <typename T, typename S>
__device__ void tail_stage_coefficients(const TailArgs<T, S>& a, const TailSharedViews<T, S>& vw) {
  for (int l = a.first; l <= a.last; ++l) {
    const int64_t n = a.lv[l].d.n;
    S* c = const_cast<S*>(vw.lv(l).c);
    const S* src = a.lv[l].c;
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < level_slots<S>() * n; i += blockDim.x) c[i] = src[i];
  }
  const int64_t nc = a.lv[a.last].d.n;
  S* inv = const_cast<S*>(vw.inv());
#pragma unroll 8
  for (int64_t i = threadIdx.x; i < nc * nc; i += blockDim.x) inv[i] = a.inv[i];
}

// Asynchronous staging (cp.async, 16 bytes each; a remainder below 16 bytes
// is copied directly), so the block can go on with other work while the
// copies land; the caller waits (cp.async.wait_all) and synchronises before
// the staged values are read.  The sources are device allocations and the
// shared-memory offsets multiples of 16 bytes.
__device__ __forceinline__ void copy_to_shared_async(void* dst, const void* src, size_t bytes) {
  const size_t n16 = bytes / 16;
  const uint32_t d0 = (uint32_t)__cvta_generic_to_shared(dst);
  for (size_t i = threadIdx.x; i < n16; i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + (uint32_t)(16 * i)),
                 "l"(reinterpret_cast<const char*>(src) + 16 * i)
                 : "memory");
  for (size_t b = 16 * n16 + threadIdx.x; b < bytes; b += blockDim.x)
    reinterpret_cast<char*>(dst)[b] = reinterpret_cast<const char*>(src)[b];
}

// The tail V-cycle on staged coefficients: the first tail level's
// right-hand side comes in from global memory (through L2: other blocks of
// a cooperative launch wrote it), and only its iterate goes back.
template <typename T, typename S>
__device__ void tail_run_staged(const TailArgs<T, S>& a, const TailSharedViews<T, S>& vw) {
  const int64_t n = a.lv[a.first].d.n;
  T* f = vw.lv(a.first).f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) f[i] = __ldcg(a.lv[a.first].f + i);
  __syncthreads();
  tail_cycle(a, vw);
  const T* x = vw.lv(a.first).x;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) a.lv[a.first].x[i] = x[i];
}

template <typename T, typename S>
__global__ void __launch_bounds__(kTailThreads) k_tail_smem(TailArgs<T, S> a, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  __shared__ uint32_t off[73];
  tail_offsets(a, off);
  __syncthreads();
  const TailSharedViews<T, S> vw{&a, off};
  tail_stage_coefficients(a, vw);
  tail_run_staged(a, vw);
}

// ---- the multi-block AMG levels in two cooperative launches
// Grid-wide barrier of a cooperative launch (all blocks resident): one
// arrival counter and one generation word in the device state.  The wait is
// bounded; if it runs out (which needs a block that never arrives) the
// barrier records kErrTimeout, and every later barrier of the launch fails
// at once, so the kernel returns and the solve reports BO_ERR_TIMEOUT.
// (the limit is a launch argument: bo_set_amg_barrier_spins lowers it)
// one block of 1024 threads per SM: a quarter of the arrivals at each
// barrier of four 256-thread blocks, for the same threads
constexpr int kCoopThreads = 1024;

__device__ __forceinline__ unsigned atom_add_release(unsigned* p, unsigned v) {
  unsigned old;
  asm volatile("atom.add.release.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The arrival is a release (every write the block made before the barrier,
// ordered by the block barrier ahead of it, is visible to whoever acquires
// the flipped word) and the polls are acquires; no separate fences.
__device__ __forceinline__ bool grid_barrier(DevState* st, unsigned spins) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile int* err = &st->err;
    int good = !(*err & kErrTimeout);
    if (good) {
      // One word per barrier round: block 0 adds 2^31 - (blocks - 1) and
      // every other block adds 1, so the round's arrivals sum to 2^31 and
      // the last one flips the word's top bit; a block has passed when the
      // top bit differs from the one its own addition saw.
      const unsigned inc = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1) : 1u;
      const unsigned old = atom_add_release(&st->counter[5], inc);
      unsigned it = 0;
      while (((ld_acquire(&st->counter[5]) ^ old) & 0x80000000u) == 0) {
        if (++it > spins || (*err & kErrTimeout)) {
          atomicOr(&st->err, kErrTimeout);
          good = 0;
          break;
        }
        __nanosleep(32);
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok;
}

// (i + j + k) even at a natural-order level
__device__ __forceinline__ bool red_cell(const LevelDims& L, int64_t c) {
  const Ijk p = ijk_of(L, c);
  return ((p.i + p.j + p.k) & 1) == 0;
}

template <typename T, typename S>
struct CycleArgs {
  Geom g;
  const S* At;
  const T* di0;  // FP64: reciprocals of level 0's diagonal (colour-split), else NULL
  T* f0;
  T* x0;
  int tail_from;  // first level of the single-block tail
  int legs_to;    // the down and up legs smooth levels 0 .. legs_to - 1 (from 1 on their zero-guess red half
                  // sweep comes with the restriction)
  int nu1, nu2;
  int cpr;  // see amg_vcycle
  T s;
  unsigned spins;  // polls of a grid barrier before it gives up (BO_ERR_TIMEOUT)
  LevelView<T, S> lv[24];
};

// Down leg: level-0 pre-smoothing and restriction, then the same for the
// natural-order levels 1 .. tail_from - 1, a grid barrier after every half
// sweep (the kernel-per-half-sweep form launches each separately).
template <typename T, typename S>
__device__ bool amg_down(const CycleArgs<T, S>& a, DevState* st) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  const Geom& g = a.g;
  for (int sw = 0; sw < a.nu1; ++sw)
    for (int color = sw == 0 ? a.cpr : 0; color < 2; ++color) {
      const int zero = sw == 0 && color == 0;
      sweep_batched<4>(t0, nt, g.Nh, a.x0 + (size_t)color * g.Nh,
                       [&](int64_t q) { return gs0_value<T, S>(g, a.At, a.di0, a.f0, a.x0, color, zero, q); });
      if (!grid_barrier(st, a.spins)) return false;
    }
  if (a.nu1 == 0) {
    for (int64_t t = t0; t < g.N; t += nt) a.x0[t] = T(0);
    if (!grid_barrier(st, a.spins)) return false;
  }
  // The first pre-smoothing half sweep of a multi-block level starts from
  // zero, x_r = f_r / a_rr: the thread that restricts a red cell's
  // right-hand side computes it at once, which saves that sweep's barrier.
  {
    const LevelView<T, S>& C = a.lv[1];
    const bool fold = a.nu1 > 0 && 1 < a.legs_to;
    for (int64_t I = t0; I < C.d.n; I += nt) {
      const T fI = restrict0_cell<T, S>(g, a.At, a.f0, a.x0, C.d, I, a.nu1 > 0);
      C.f[I] = fI;
      if (fold && red_cell(C.d, I)) C.x[I] = C.divided(fI, I);
    }
  }
  for (int l = 1; l < a.legs_to; ++l) {
    if (!grid_barrier(st, a.spins)) return false;
    const LevelView<T, S>& L = a.lv[l];
    for (int sw = 0; sw < a.nu1; ++sw)
      for (int color = 0; color < 2; ++color) {
        if (sw == 0 && color == 0) continue;  // done with the restriction
        for (int64_t c = t0; c < L.d.n; c += nt) gs_cell(L, c, color, 0);
        if (!grid_barrier(st, a.spins)) return false;
      }
    if (a.nu1 == 0) {
      for (int64_t c = t0; c < L.d.n; c += nt) L.x[c] = T(0);
      if (!grid_barrier(st, a.spins)) return false;
    }
    const LevelView<T, S>& C = a.lv[l + 1];
    const bool fold = a.nu1 > 0 && l + 1 < a.legs_to;
    for (int64_t I = t0; I < C.d.n; I += nt) {
      const T fI = restrict_cell(L, C.d, I, a.nu1 > 0);
      C.f[I] = fI;
      if (fold && red_cell(C.d, I)) C.x[I] = C.divided(fI, I);
    }
  }
  return true;
}

// Up leg: post-smoothing of levels tail_from - 1 .. 1 and then level 0, the
// first (black) half sweep of each level reading the coarse correction
template <typename T, typename S>
__device__ bool amg_up(const CycleArgs<T, S>& a, DevState* st) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  const Geom& g = a.g;
  for (int l = a.legs_to - 1; l >= 1; --l) {
    const LevelView<T, S>& L = a.lv[l];
    const LevelView<T, S>& C = a.lv[l + 1];
    if (a.nu2 == 0) {
      for (int64_t c = t0; c < L.d.n; c += nt) prolong_cell(L, C, c, a.s);
      if (!grid_barrier(st, a.spins)) return false;
    }
    for (int sw = 0; sw < a.nu2; ++sw)
      for (int color = 1; color >= 0; --color) {
        for (int64_t c = t0; c < L.d.n; c += nt) {
          if (sw == 0 && color == 1) gs_cell_prolong(L, C, c, a.s);
          else gs_cell(L, c, color, 0);
        }
        if (!grid_barrier(st, a.spins)) return false;
      }
  }
  const LevelView<T, S>& C1 = a.lv[1];
  if (a.nu2 == 0) {
    for (int64_t t = t0; t < g.N; t += nt) prolong0_cell<T>(g, a.x0, C1.d, C1.x, a.s, t);
    return true;
  }
  for (int sw = 0; sw < a.nu2; ++sw) {
    if (sw == 0)
      sweep_batched<4>(t0, nt, g.Nh, a.x0 + g.Nh, [&](int64_t q) {
        return gs0_prolong_value<T, S>(g, a.At, a.di0, a.f0, a.x0, C1.d, C1.x, a.s, q);
      });
    else
      sweep_batched<4>(t0, nt, g.Nh, a.x0 + g.Nh,
                       [&](int64_t q) { return gs0_value<T, S>(g, a.At, a.di0, a.f0, a.x0, 1, 0, q); });
    if (!grid_barrier(st, a.spins)) return false;
    sweep_batched<4>(t0, nt, g.Nh, a.x0, [&](int64_t q) { return gs0_value<T, S>(g, a.At, a.di0, a.f0, a.x0, 0, 0, q); });
    if (sw + 1 < a.nu2 && !grid_barrier(st, a.spins)) return false;
  }
  return true;
}

template <typename T, typename S>
__global__ void __launch_bounds__(kCoopThreads, 1) k_amg_down(CycleArgs<T, S> a, DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  amg_down(a, st);
}

template <typename T, typename S>
__global__ void __launch_bounds__(kCoopThreads, 1) k_amg_up(CycleArgs<T, S> a, DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  amg_up(a, st);
}

// ---- the resident levels: level l0 and every coarser one in one thread-block cluster
// Each block holds a stretch of a level in its shared memory (iterate,
// right-hand side, residual) and its threads hold the coefficients of the
// cells they own in registers through all half sweeps of a visit; neighbours
// and aggregates that another block owns are read through distributed shared
// memory.  A half sweep is then six shared-memory reads, six multiply-adds
// and a barrier.  A level is shared by all blocks (cluster barrier, about
// 0.3 us) while it is large, and kept by block 0 alone (block barrier) once
// it is small.  What bounds it is latency: barriers, and the loads and index
// arithmetic of a visit, so the coefficients are kept in a packed copy in
// the order the threads own the cells, with each cell's place in the
// stencil, its aggregate and its children worked out beforehand (k_res_pack).
// Measured against the form before it (cooperative legs for level 0, the
// same sweeps on operands in L2, small levels in one block): a 20x20x5 FP64
// Newton step 1589 -> 1097 us, 62x45x19 FP32 2297 -> 1975 us, 128x128x64 FP32
// 10.64 -> 10.25 ms at 14 iterations.
//
// Cells go in pairs: natural cells 2q and 2q + 1 always have the two colours
// (a grid row of even length holds whole pairs; where the length is odd, a
// pair that crosses the end of a row or of a plane changes colour too), so
// every thread has one cell to do in each half sweep, and the red and black
// arrays are indexed by q as level 0's colour-split arrays are.
constexpr int kResThreads = 512;
constexpr int kResMaxCluster = 16;
constexpr size_t kResSmemMax = 200 * 1024;
// pairs a thread may own (registers: 14 coefficients and 12 addresses a pair)
template <typename T>
__host__ __device__ constexpr int res_pairs() { return sizeof(T) == 4 ? 2 : 1; }
// levels of at most this many cells stay in one block: a half sweep over
// them takes less than the cluster barrier that sharing it would cost (in
// FP64 the multiply-adds of 256 cells already take 0.25 us on one SM)
template <typename T>
constexpr int64_t res_single() { return sizeof(T) == 4 ? 2048 : 256; }
// values per cell in the packed copy: six off-diagonal coefficients, the
// diagonal and, in FP64, its reciprocal
template <typename T>
__host__ __device__ constexpr int res_values() { return sizeof(T) == 4 ? 7 : 8; }

}  // namespace

// One resident level: its shape, its place in each block's shared memory and
// its packed copy.
//   cp:   [colour][value][pair], the values in order -z, -y, -x, +x, +y, +z,
//         diagonal (, reciprocal), missing neighbours 0
//   meta: [0][pair] bit 0 the colour of the pair's first cell, bits 1-6 and
//         7-12 the neighbours (in that order) that its red and black cell
//         have, the rest the red cell's aggregate on the next level (natural
//         index and colour: 16 bits, since no level holds more cells than a
//         cluster's threads own);
//         [1], [2][pair] for the red and black cell as an aggregate: the
//         natural index of its first child on the level above and which
//         further children exist along x, y, z.  The coarsest level keeps
//         that word per cell in natural order.
struct ResLevel {
  int32_t n, npairs, nx, nxy;
  int32_t lch;    // log2 of the pairs per block
  int32_t dist;   // shared by the cluster, or kept by block 0
  uint32_t off;   // red x, black x, red residual, red f, black f: (1 << lch) entries each
  uint32_t coef;  // staged copy of cp, or ~0u
  void* cp;
  int32_t* meta;
  void* f;        // level l0 only: right-hand side in, iterate out (natural order; level 0 colour-split)
  void* x;
};

struct ResPlan {
  int32_t cluster;  // blocks
  int32_t l0, last;
  int32_t nu1, nu2;
  double s;
  ResLevel rl[24];
  const void* inv;     // coarse inverse, transposed (storage type)
  uint32_t zero_off;   // zeros in each block, one a lane: what a missing neighbour's iterate reads as
  uint32_t dense_off;  // right-hand side and solution of the coarsest level: 2 kCoarseMax entries
  uint32_t inv_off;    // staged inverse, or ~0u
  uint32_t smem;
};

namespace {

__device__ __forceinline__ float ld_sh(uint32_t a, bool cluster, float) {
  float v;
  if (cluster) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  else asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ double ld_sh(uint32_t a, bool cluster, double) {
  double v;
  if (cluster) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  else asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_sh(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void st_sh(uint32_t a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ uint32_t map_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// the levels' coefficients in natural order (storage type)
struct CoefPtrs {
  const void* c[24];
};

// The packed copies of all resident levels, one thread per pair (the
// coarsest level, whose inverse is kept instead: one per cell).
template <typename T, typename S>
__global__ void k_res_pack(const __grid_constant__ ResPlan a, Geom g, const S* __restrict__ At,
                           const T* __restrict__ di0, const __grid_constant__ CoefPtrs coef) {
  wait_prior_grid();
  constexpr int K = res_values<T>();
  int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int l = a.l0; l <= a.last; ++l) {
    const ResLevel& r = a.rl[l];
    const int32_t items = l == a.last ? r.n : r.npairs;
    if (t >= items) {
      t -= items;
      continue;
    }
    const int32_t ny = r.nxy / r.nx, nz = r.n / r.nxy;
    // the neighbours a cell has, -z, -y, -x, +x, +y, +z
    auto neighbours = [&](int32_t c) {
      const int32_t i = c % r.nx, j = (c / r.nx) % ny, k = c / r.nxy;
      return (k > 0 ? 1 : 0) | (j > 0 ? 2 : 0) | (i > 0 ? 4 : 0) | (i + 1 < r.nx ? 8 : 0) | (j + 1 < ny ? 16 : 0) |
             (k + 1 < nz ? 32 : 0);
    };
    // a cell's word as an aggregate of level l - 1
    auto child_word = [&](int32_t c) {
      if (l == a.l0) return 0;
      const ResLevel& f = a.rl[l - 1];
      const int32_t i = c % r.nx, j = (c / r.nx) % ny, k = c / r.nxy;
      const int32_t fny = f.nxy / f.nx, fnz = f.n / f.nxy;
      return ((2 * i + f.nx * 2 * j + f.nxy * 2 * k) << 3) | (2 * i + 1 < f.nx ? 1 : 0) | (2 * j + 1 < fny ? 2 : 0) |
             (2 * k + 1 < fnz ? 4 : 0);
    };
    if (l == a.last) {
      r.meta[t] = child_word(t);
      return;
    }
    const int32_t q = t, np = r.npairs;
    const int32_t c0 = 2 * q;
    const int32_t par = (c0 % r.nx + (c0 / r.nx) % ny + c0 / r.nxy) & 1;
    T* cp = (T*)r.cp;
    const S* lc = (const S*)coef.c[l];
    int32_t have = 0;
    for (int col = 0; col < 2; ++col) {
      const int32_t c = c0 + (col ^ par);
      const bool live = c < r.n;
      const int slot[7] = {kZm, kYm, kXm, kXp, kYp, kZp, kDiag};
      for (int d = 0; d < 7; ++d) {
        T v = d == 6 ? T(1) : T(0);
        if (live) v = l ? cv<T>(lc[(size_t)slot[d] * r.n + c]) : cv<T>(At[at_index(g, col, slot[d] * 9, q)]);
        cp[(size_t)(col * K + d) * np + q] = v;
      }
      if constexpr (sizeof(T) == 8)
        cp[(size_t)(col * K + 7) * np + q] = !live ? T(1) : l ? (T)lc[(size_t)7 * r.n + c] : di0[(size_t)col * g.Nh + q];
      r.meta[(size_t)(1 + col) * np + q] = live ? child_word(c) : 0;
      if (live) have |= neighbours(c) << (6 * col);
    }
    int32_t agg = 0;
    const int32_t cr = c0 + par;  // the red cell
    if (cr < r.n) {
      const ResLevel& cl = a.rl[l + 1];
      const int32_t i = (cr % r.nx) >> 1, j = ((cr / r.nx) % ny) >> 1, k = (cr / r.nxy) >> 1;
      agg = ((i + cl.nx * j + cl.nxy * k) << 1) | ((i + j + k) & 1);
    }
    r.meta[q] = (agg << 13) | (have << 1) | par;
    return;
  }
}

// The array sections of a level in a block's shared memory
enum : int { kSecRed = 0, kSecBlack = 1, kSecRes = 2, kSecF = 3 };  // kSecF, kSecF + 1: f of red and black

template <typename T>
__device__ __forceinline__ uint32_t res_local(const ResLevel& r, uint32_t base, int sec, int32_t q) {
  const uint32_t m = (1u << r.lch) - 1u;
  return base + r.off + (((uint32_t)sec << r.lch) + ((uint32_t)q & m)) * (uint32_t)sizeof(T);
}
// address of entry q of a section, in whichever block owns it
template <typename T, bool DIST>
__device__ __forceinline__ uint32_t res_addr(const ResLevel& r, uint32_t base, int sec, int32_t q) {
  const uint32_t a = res_local<T>(r, base, sec, q);
  return DIST ? map_rank(a, (uint32_t)(q >> r.lch)) : a;
}

template <typename T, int NP>
struct ResCells {
  T c[2][NP][6];          // off-diagonal coefficients (0 where the neighbour is missing)
  T d[2][NP];             // diagonal
  T di[2][NP];            // and in FP64 its reciprocal
  T f[2][NP];
  uint32_t nb[2][NP][6];  // shared-memory addresses of the neighbours' iterates
  uint32_t own[2][NP];    // and of the cell's own
  int32_t m[NP];          // meta word 0
  bool live[2][NP];
};

__device__ __forceinline__ float res_divide(float s, float d, float) { return s / d; }
__device__ __forceinline__ double res_divide(double s, double d, double r) { return divide_by(s, d, r); }

// One visit of level l: the cells of this thread into registers
template <typename T, int NP, bool DIST>
__device__ __forceinline__ void res_load(const ResPlan& a, int l, uint32_t base, ResCells<T, NP>& r) {
  constexpr int K = res_values<T>();
  const ResLevel& rl = a.rl[l];
  const int32_t np = rl.npairs;
  const int32_t q0 = DIST ? (int32_t)blockIdx.x << rl.lch : 0;
  const int32_t q1 = min(np, q0 + (1 << rl.lch));
  const T* cp = (const T*)rl.cp;
  if (!DIST && rl.coef != ~0u) cp = reinterpret_cast<const T*>(g_tail_smem + rl.coef);
  const int32_t off[6] = {-rl.nxy, -rl.nx, -1, 1, rl.nx, rl.nxy};
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int32_t q = q0 + (int32_t)threadIdx.x + kResThreads * p;
    const bool in = q < q1;
    const int32_t qq = in ? q : 0;
    r.m[p] = rl.meta[qq];
#pragma unroll
    for (int col = 0; col < 2; ++col) {
#pragma unroll
      for (int d = 0; d < 6; ++d) r.c[col][p][d] = cp[(col * K + d) * np + qq];
      r.d[col][p] = cp[(col * K + 6) * np + qq];
      r.di[col][p] = K == 8 ? cp[(col * K + K - 1) * np + qq] : T(0);
    }
    const int32_t par = r.m[p] & 1;
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      const int32_t c = 2 * qq + (col ^ par);
      r.live[col][p] = in && c < rl.n;
      r.own[col][p] = res_local<T>(rl, base, col, qq);
      // (a missing neighbour reads as zero, whatever the iterates hold: its
      // coefficient is 0, but 0 times an infinity is not)
      const uint32_t zl = base + a.zero_off + (threadIdx.x & 31u) * (uint32_t)sizeof(T);
      const uint32_t zero = DIST ? map_rank(zl, blockIdx.x) : zl;
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const bool have = (r.m[p] >> (1 + 6 * col + d)) & 1;
        const uint32_t ad = res_addr<T, DIST>(rl, base, col ^ 1, have ? (c + off[d]) >> 1 : qq);
        r.nb[col][p][d] = have ? ad : zero;
      }
    }
  }
}

template <bool DIST>
__device__ __forceinline__ void res_barrier() {
  if (DIST) cluster_sync_all();
  else __syncthreads();
}

// (warps whose threads own no cell of the colour skip to the barrier: FP64
// multiply-adds issued for nothing would occupy the SM's narrow FP64 pipe)
template <typename T, int NP, bool DIST>
__device__ __forceinline__ void res_sweep(ResCells<T, NP>& r, int col) {
  bool any = false;
#pragma unroll
  for (int p = 0; p < NP; ++p) any = any || r.live[col][p];
  if (any) {
    T xv[NP][6];
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
      for (int d = 0; d < 6; ++d) xv[p][d] = r.live[col][p] ? ld_sh(r.nb[col][p][d], DIST, T(0)) : T(0);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T s = r.f[col][p];
#pragma unroll
      for (int d = 0; d < 6; ++d) s -= r.c[col][p][d] * xv[p][d];
      if (r.live[col][p]) st_sh(r.own[col][p], res_divide(s, r.d[col][p], r.di[col][p]));
    }
  }
  res_barrier<DIST>();
}

// Right-hand side of a cell from the red residuals of its children on level
// `r` (nu1 >= 1: the black residuals are zero after a black half sweep), in
// the order of the other launch forms: (0,0,0), (1,1,0), (1,0,1), (0,1,1)
template <typename T>
__device__ __forceinline__ T res_gather(const ResLevel& r, uint32_t base, int32_t word) {
  const int32_t c = word >> 3;
  const bool ex = word & 1, ey = word & 2, ez = word & 4;
  const int32_t ch[4] = {c, c + 1 + r.nx, c + 1 + r.nxy, c + r.nx + r.nxy};
  const bool ok[4] = {true, ex && ey, ex && ez, ey && ez};
  T v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int32_t q = (ok[e] ? ch[e] : c) >> 1;
    const uint32_t ad = res_local<T>(r, base, kSecRes, q);
    v[e] = r.dist ? ld_sh(map_rank(ad, (uint32_t)(q >> r.lch)), true, T(0)) : ld_sh(ad, false, T(0));
  }
  T acc = T(0);
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (ok[e]) acc += v[e];
  return acc;
}

// Pre-smoothing of level l and its red residuals, ready for the next level.
// Every block of the cluster runs it when the level is shared (DIST), block
// 0 alone otherwise.
template <typename T, bool DIST>
__device__ __forceinline__ void res_down(const ResPlan& a, const Geom& g, int l, uint32_t base) {
  constexpr int NP = res_pairs<T>();
  ResCells<T, NP> r;
  res_load<T, NP, DIST>(a, l, base, r);
  const ResLevel& rl = a.rl[l];
  const int32_t q0 = DIST ? (int32_t)blockIdx.x << rl.lch : 0;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int32_t i = (int32_t)threadIdx.x + kResThreads * p, q = q0 + i;
    const bool place = i < (1 << rl.lch);
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      T f = T(0);
      if (r.live[col][p]) {
        if (l > a.l0) f = res_gather<T>(a.rl[l - 1], base, rl.meta[(1 + col) * rl.npairs + q]);
        else if (l) f = ((const T*)rl.f)[2 * q + (col ^ (r.m[p] & 1))];
        else f = ((const T*)rl.f)[(size_t)col * g.Nh + q];
      }
      r.f[col][p] = f;
      if (place) st_sh(res_local<T>(rl, base, kSecF + col, q), f);
    }
    // the first half sweep starts from zero: x_r = f_r / d_r (black zero
    // until its own half sweep)
    if (place) {
      st_sh(res_local<T>(rl, base, kSecRed, q), r.live[0][p] ? res_divide(r.f[0][p], r.d[0][p], r.di[0][p]) : T(0));
      st_sh(res_local<T>(rl, base, kSecBlack, q), T(0));
    }
  }
  res_barrier<DIST>();
  res_sweep<T, NP, DIST>(r, 1);
  for (int sw = 1; sw < a.nu1; ++sw) {
    res_sweep<T, NP, DIST>(r, 0);
    res_sweep<T, NP, DIST>(r, 1);
  }
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    if (!r.live[0][p]) continue;
    // (the diagonal's term first, or after the lower neighbours on level 0:
    // the order of the other launch forms, whose results these are bit for bit)
    const T dx = ld_sh(r.own[0][p], false, T(0));
    T v = r.f[0][p];
    if (l) v -= r.d[0][p] * dx;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      if (d == 3 && !l) v -= r.d[0][p] * dx;
      v -= r.c[0][p][d] * ld_sh(r.nb[0][p][d], DIST, T(0));
    }
    st_sh(r.own[0][p] + ((uint32_t)(kSecRes - kSecRed) << rl.lch) * (uint32_t)sizeof(T), v);
  }
  res_barrier<DIST>();
}

// Coarse correction and post-smoothing of level l
template <typename T, bool DIST>
__device__ __forceinline__ void res_up(const ResPlan& a, const Geom& g, int l, uint32_t base) {
  constexpr int NP = res_pairs<T>();
  ResCells<T, NP> r;
  res_load<T, NP, DIST>(a, l, base, r);
  const ResLevel& rl = a.rl[l];
  const int32_t q0 = DIST ? (int32_t)blockIdx.x << rl.lch : 0;
  const T sc = (T)a.s;
  // x_r += s x_c (the black cells are overwritten by the half sweep that follows)
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int32_t q = q0 + (int32_t)threadIdx.x + kResThreads * p;
#pragma unroll
    for (int col = 0; col < 2; ++col) r.f[col][p] = r.live[col][p] ? ld_sh(res_local<T>(rl, base, kSecF + col, q), false, T(0)) : T(0);
    if (!r.live[0][p]) continue;
    const int32_t agg = r.m[p] >> 13;
    uint32_t ad;
    int32_t owner = 0;
    if (l + 1 == a.last) {
      ad = base + a.dense_off + (uint32_t)(kCoarseMax + (agg >> 1)) * (uint32_t)sizeof(T);
    } else {
      const ResLevel& cl = a.rl[l + 1];
      ad = res_local<T>(cl, base, agg & 1, agg >> 2);
      owner = cl.dist ? (agg >> 2) >> cl.lch : 0;
    }
    const T xc = DIST ? ld_sh(map_rank(ad, (uint32_t)owner), true, T(0)) : ld_sh(ad, false, T(0));
    st_sh(r.own[0][p], ld_sh(r.own[0][p], false, T(0)) + sc * xc);
  }
  res_barrier<DIST>();
  for (int sw = 0; sw < a.nu2; ++sw) {
    res_sweep<T, NP, DIST>(r, 1);
    res_sweep<T, NP, DIST>(r, 0);
  }
  if (l == a.l0) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int32_t q = q0 + (int32_t)threadIdx.x + kResThreads * p;
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        if (!r.live[col][p]) continue;
        const T v = ld_sh(r.own[col][p], false, T(0));
        if (l) ((T*)rl.x)[2 * q + (col ^ (r.m[p] & 1))] = v;
        else ((T*)rl.x)[(size_t)col * g.Nh + q] = v;
      }
    }
  }
}

template <typename T, typename S>
__global__ void __launch_bounds__(kResThreads, 1) k_amg_resident(const __grid_constant__ ResPlan a, Geom g,
                                                                const DevState* st) {
  wait_prior_grid();
  if (st->done) return;  // uniform: every block reads the same flag
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(g_tail_smem);
  const bool first = blockIdx.x == 0;
  const int32_t n = a.rl[a.last].n;
  if (first) {
    // block 0 stages the small levels' coefficients and the coarse inverse
    // under the first level's sweeps
    for (int l = a.l0; l < a.last; ++l)
      if (a.rl[l].coef != ~0u)
        copy_to_shared_async(g_tail_smem + a.rl[l].coef, a.rl[l].cp, (size_t)2 * res_values<T>() * a.rl[l].npairs * sizeof(T));
    if (a.inv_off != ~0u) copy_to_shared_async(g_tail_smem + a.inv_off, a.inv, (size_t)n * n * sizeof(S));
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (threadIdx.x < 32) st_sh(base + a.zero_off + threadIdx.x * (uint32_t)sizeof(T), T(0));
  cluster_sync_all();  // every block runs before its shared memory is read
  int l = a.l0;
  for (; l < a.last && a.rl[l].dist; ++l) res_down<T, true>(a, g, l, base);
  const int shared_to = l;
  if (first) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (; l < a.last; ++l) res_down<T, false>(a, g, l, base);
    // the coarsest level: x = inv f, a thread per row (inv is stored transposed)
    const uint32_t fo = base + a.dense_off;
    const ResLevel& rl = a.rl[a.last];
    for (int i = threadIdx.x; i < n; i += kResThreads)
      st_sh(fo + (uint32_t)(i * sizeof(T)),
            a.l0 == a.last ? ((const T*)rl.f)[i] : res_gather<T>(a.rl[a.last - 1], base, rl.meta[i]));
    __syncthreads();
    const S* inv = a.inv_off != ~0u ? reinterpret_cast<const S*>(g_tail_smem + a.inv_off) : (const S*)a.inv;
    for (int i = threadIdx.x; i < n; i += kResThreads) {
      T s = T(0);
#pragma unroll 8
      for (int j = 0; j < n; ++j) s += cv<T>(inv[j * n + i]) * ld_sh(fo + (uint32_t)(j * sizeof(T)), false, T(0));
      st_sh(fo + (uint32_t)((kCoarseMax + i) * sizeof(T)), s);
      if (a.l0 == a.last) ((T*)rl.x)[i] = s;
    }
    __syncthreads();
    for (l = a.last - 1; l >= shared_to; --l) res_up<T, false>(a, g, l, base);
  }
  cluster_sync_all();
  for (l = shared_to - 1; l >= a.l0; --l) res_up<T, true>(a, g, l, base);
  cluster_sync_all();  // no block leaves while another may read its shared memory
}

// dense solve on level 0 when level 0 is the coarsest: x = inv f (inv transposed)
template <typename T, typename S>
__global__ void k_dense0(int64_t n, const S* __restrict__ inv, const T* __restrict__ f, T* __restrict__ x,
                         const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    T s = T(0);
    for (int64_t j = 0; j < n; ++j) s += cv<T>(inv[j * n + i]) * f[j];
    x[i] = s;
  }
}

template <typename T>
__global__ void k_zero(int64_t n, T* __restrict__ x, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = T(0);
}

// z = Pi_p e (stage AMG alone), FP64 output
template <typename T>
__global__ void k_place_p(Geom g, const T* __restrict__ e, double* __restrict__ z, const DevState* st) {
  wait_prior_grid();
  if (st->done) return;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x) {
    z[t] = (double)e[t];
    z[g.N + t] = 0.0;
    z[2 * g.N + t] = 0.0;
  }
}

// y = At x with At rebuilt in FP64 from A and the weights (parity checks)
__global__ void k_spmv_dec64(Geom g, const double* __restrict__ A, const double* __restrict__ w,
                             const double* __restrict__ x, double* __restrict__ y) {
  wait_prior_grid();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < g.N; t += (int64_t)gridDim.x * blockDim.x) {
    const int color = (int)(t / g.Nh);
    const int64_t q = t - color * g.Nh;
    const Cell c = decode(g, color, q);
    double acc[3] = {0, 0, 0};
    for (int sl = 0; sl < 7; ++sl) {
      const int64_t nq = nbr(g, c, q, sl);
      if (nq < 0) continue;
      const int xc = (sl == kDiag) ? color : (color ^ 1);
      double b[9];
      dec_block(g, A, w, color, sl, q, b);
      for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) acc[r] += b[3 * r + k] * x[vidx(g, k, xc, nq)];
    }
    for (int r = 0; r < 3; ++r) y[vidx(g, r, color, q)] = acc[r];
  }
}

// ---------------------------------------------------------------- host side
template <typename T, typename S>
LevelView<T, S> view(bo_prec* P, int l) {
  const Level& L = P->lev[l];
  return LevelView<T, S>{LevelDims{L.nx, L.ny, L.nz, L.n}, (const S*)L.c, (T*)L.f, (T*)L.x};
}

LevelDims dims_of(const Level& L) { return LevelDims{L.nx, L.ny, L.nz, L.n}; }

// Largest cluster of the resident kernel that the current device can
// co-schedule with its shared memory (16 is a non-portable size), or 0.
// Queried, and the kernel's attributes set, once per instantiation and device.
template <typename T, typename S>
int resident_max_cluster(int device) {
  static PerDevice cached;
  return cached.get(device, [] {
    const void* k = (const void*)k_amg_resident<T, S>;
    if (cudaFuncSetAttribute(k_amg_resident<T, S>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_amg_resident<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemMax) ==
            cudaSuccess) {
      for (int c : {kResMaxCluster, 8, 4, 2, 1}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c, 1, 1);
        cfg.blockDim = dim3(kResThreads, 1, 1);
        cfg.dynamicSmemBytes = kResSmemMax;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclus = 0;
        if (cudaOccupancyMaxActiveClusters(&nclus, k, &cfg) == cudaSuccess && nclus >= 1) return c;
      }
    }
    cudaGetLastError();
    return 0;
  });
}

// The resident form's levels, cluster and shared-memory layout for P: level
// l0 is the finest level that fits the largest cluster (FP32: 32768 cells,
// two pairs per thread; FP64: 16384).  The cluster is the smallest that
// gives a block at most `per` pairs of level l0 (FP32: 512, one half-sweep
// cell per thread; FP64: 128, whose multiply-adds take about a cluster
// barrier's time), so a batch's small systems leave SMs to one another.
// cluster = 0 where the form does not apply (no pre- or post-smoothing).
template <typename T, typename S>
void resident_plan(bo_prec* P, ResPlan& a) {
  a.cluster = 0;
  const int maxc = resident_max_cluster<T, S>(P->mat->ctx->device);
  const Geom& g = P->mat->g;
  const int last = P->nlev - 1;
  if (maxc < 1 || last < 1 || P->opts.amg_nu1 < 1 || P->opts.amg_nu2 < 1) return;
  const int64_t cap = (int64_t)2 * kResThreads * res_pairs<T>() * maxc;
  auto cells = [&](int l) { return l ? P->lev[l].n : g.N; };
  int l0 = 0;
  while (l0 < last && cells(l0) > cap) ++l0;
  if (l0 > 0 && l0 > P->tail_from) return;
  int C = 1;
  if (l0 < last && cells(l0) > res_single<T>()) {
    const int64_t per = sizeof(T) == 4 ? 512 : 128;
    while (C < maxc && (cells(l0) + 1) / 2 > per * C) C *= 2;
  }
  uint32_t o = 0;
  for (int l = l0; l <= last; ++l) {
    ResLevel& r = a.rl[l];
    r = ResLevel{};
    r.n = (int32_t)cells(l);
    r.npairs = (r.n + 1) / 2;
    r.nx = l ? P->lev[l].nx : g.nx;
    r.nxy = r.nx * (l ? P->lev[l].ny : g.ny);
    r.coef = ~0u;
    if (l == last) break;
    r.dist = C > 1 && r.n > res_single<T>();
    const int32_t per = r.dist ? (r.npairs + C - 1) / C : r.npairs;
    while ((1 << r.lch) < per) ++r.lch;
    if ((1 << r.lch) > kResThreads * res_pairs<T>()) return;
    r.off = o;
    o += (uint32_t)align16(((size_t)5 << r.lch) * sizeof(T));
  }
  a.zero_off = o;
  o += 32 * sizeof(T);
  a.dense_off = o;
  o += (uint32_t)align16(2 * kCoarseMax * sizeof(T));
  for (int l = l0; l < last; ++l) {
    ResLevel& r = a.rl[l];
    const size_t b = align16((size_t)2 * res_values<T>() * r.npairs * sizeof(T));
    if (r.dist || o + b > kResSmemMax) continue;
    r.coef = o;
    o += (uint32_t)b;
  }
  const size_t ib = align16((size_t)P->ncoarse * P->ncoarse * sizeof(S));
  a.inv_off = ~0u;
  if (o + ib <= kResSmemMax) {
    a.inv_off = o;
    o += (uint32_t)ib;
  }
  if (o > kResSmemMax) return;
  a.smem = o;
  a.l0 = l0;
  a.last = last;
  a.nu1 = P->opts.amg_nu1;
  a.nu2 = P->opts.amg_nu2;
  a.s = P->opts.amg_overcorr;
  a.cluster = C;
}

// cpr: within the CPR, whose k_cpr_rhs has done the first half sweep (if nu1 >
// 0; the cluster form starts from the right-hand side alone).
template <typename T, typename S>
void amg_vcycle(bo_prec* P, const DevState* st, bool cpr) {
  cudaStream_t s = P->stream;
  const Geom& g = P->mat->g;
  const S* At = (const S*)P->At;
  const T* di0 = (const T*)P->di0;  // (NULL unless T is double)
  T* f0 = (T*)P->f0;
  T* x0 = (T*)P->e0;
  const int nu1 = P->opts.amg_nu1, nu2 = P->opts.amg_nu2;
  const T sc = (T)P->opts.amg_overcorr;
  if (P->nlev == 1) {
    (launch_pdl(k_dense0<T, S>, grid_for(g.N), kThreads, 0, s, g.N, (const S*)P->coarse_inv, f0, x0, st), note_launch());
    return;
  }
  // tile parameters of the per-kernel form (set by the batch autotuner):
  // threads per block and level-0 cells per thread
  const int TB = P->amg_threads;
  const int CB = P->amg_cells;
  const int ghalf = grid_for((g.Nh + CB - 1) / CB, TB);
  auto gs0 = [&](int color, int zero) {
    if (CB == 4) (launch_pdl(k_gs0<T, S, 4>, ghalf, TB, 0, s, g, At, di0, f0, x0, color, zero, st), note_launch());
    else if (CB == 2) (launch_pdl(k_gs0<T, S, 2>, ghalf, TB, 0, s, g, At, di0, f0, x0, color, zero, st), note_launch());
    else (launch_pdl(k_gs0<T, S, 1>, ghalf, TB, 0, s, g, At, di0, f0, x0, color, zero, st), note_launch());
  };
  auto gs0_prolong = [&]() {
    const LevelDims C1 = dims_of(P->lev[1]);
    const T* xc = (const T*)P->lev[1].x;
    if (CB == 4) (launch_pdl(k_gs0_prolong<T, S, 4>, ghalf, TB, 0, s, g, At, di0, f0, x0, C1, xc, sc, st), note_launch());
    else if (CB == 2) (launch_pdl(k_gs0_prolong<T, S, 2>, ghalf, TB, 0, s, g, At, di0, f0, x0, C1, xc, sc, st), note_launch());
    else (launch_pdl(k_gs0_prolong<T, S, 1>, ghalf, TB, 0, s, g, At, di0, f0, x0, C1, xc, sc, st), note_launch());
  };
  const int last = P->nlev - 1;
  // Launch forms (all compute the same V-cycle):
  //  mode 2: every level that fits a cluster's registers and shared memory in
  //          one cluster launch (k_amg_resident), the levels above it in two
  //          cooperative launches (down leg, up leg, grid barriers between
  //          half sweeps), or one kernel per half sweep inside stream capture;
  //  mode 1: the cooperative legs also smooth the multi-block natural
  //          levels, the tail levels in one block;
  //  mode 0, or when a launch form is refused: one kernel per half sweep,
  //          restriction and prolongation.
  const int mode = g_amg_coop.load();
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);
  const bool coop = mode != 0 && cap == cudaStreamCaptureStatusNone;
  const ResPlan& ra = *P->res;
  const int rc = mode == 2 ? ra.cluster : 0;
  auto resident = [&]() {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(rc, 1, 1);
    cfg.blockDim = dim3(kResThreads, 1, 1);
    cfg.dynamicSmemBytes = ra.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = rc;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, k_amg_resident<T, S>, ra, g, st) != cudaSuccess) return false;
    note_launch();
    return true;
  };
  if (rc > 0 && ra.l0 == 0) {
    if (resident()) return;
    cudaGetLastError();
  }
  // first level of the cluster launch (none: past the last)
  const int res_from = rc > 0 && ra.l0 > 0 ? ra.l0 : last + 1;
  CycleArgs<T, S> ca;
  ca.g = g;
  ca.At = At;
  ca.di0 = di0;
  ca.f0 = f0;
  ca.x0 = x0;
  ca.tail_from = P->tail_from;
  ca.legs_to = std::min(P->tail_from, res_from);
  ca.nu1 = nu1;
  ca.nu2 = nu2;
  ca.cpr = cpr;
  ca.s = sc;
  ca.spins = g_amg_spins.load();
  for (int l = 1; l <= last; ++l) ca.lv[l] = view<T, S>(P, l);
  TailArgs<T, S> ta;
  ta.first = P->tail_from;
  ta.last = last;
  ta.nu1 = nu1;
  ta.nu2 = nu2;
  ta.s = sc;
  for (int l = 1; l <= last; ++l) ta.lv[l] = view<T, S>(P, l);
  ta.inv = (const S*)P->coarse_inv;
  const size_t tb = tail_smem_bytes(ta);
  DevState* stw = const_cast<DevState*>(st);

  // per-kernel pre- and post-smoothing of the multi-block natural levels
  const int natural_to = ca.legs_to;
  auto natural_pre = [&](int l) {
    LevelView<T, S> L = view<T, S>(P, l), C = view<T, S>(P, l + 1);
    const int gl = grid_for(L.d.n, TB);
    for (int sw = 0; sw < nu1; ++sw) {
      (launch_pdl(k_gsn<T, S>, gl, TB, 0, s, L, 0, sw == 0, st), note_launch());
      (launch_pdl(k_gsn<T, S>, gl, TB, 0, s, L, 1, 0, st), note_launch());
    }
    if (nu1 == 0) (launch_pdl(k_zero<T>, gl, TB, 0, s, L.d.n, L.x, st), note_launch());
    (launch_pdl(k_restrictn<T, S>, grid_for(C.d.n, TB), TB, 0, s, L, C, nu1 > 0, st), note_launch());
  };
  auto natural_down = [&]() {
    for (int l = 1; l < natural_to; ++l) natural_pre(l);
  };
  auto natural_post = [&](int l) {
    LevelView<T, S> L = view<T, S>(P, l), C = view<T, S>(P, l + 1);
    const int gl = grid_for(L.d.n, TB);
    if (nu2 == 0) (launch_pdl(k_prolongn<T, S>, gl, TB, 0, s, L, C, sc, st), note_launch());
    for (int sw = 0; sw < nu2; ++sw) {
      if (sw == 0) (launch_pdl(k_gsn_prolong<T, S>, gl, TB, 0, s, L, C, sc, st), note_launch());
      else (launch_pdl(k_gsn<T, S>, gl, TB, 0, s, L, 1, 0, st), note_launch());
      (launch_pdl(k_gsn<T, S>, gl, TB, 0, s, L, 0, 0, st), note_launch());
    }
  };
  auto natural_up = [&]() {
    for (int l = natural_to - 1; l >= 1; --l) natural_post(l);
  };
  auto tail = [&]() {
    if (tb <= kTailSmemMax) {
      cudaFuncSetAttribute(k_tail_smem<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tb);
      (launch_pdl(k_tail_smem<T, S>, 1, kTailThreads, tb, s, ta, st), note_launch());
    } else {
      (launch_pdl(k_tail<T, S>, 1, kTailThreads, 0, s, ta, st), note_launch());
    }
  };

  // a cooperative launch that may also start as soon as the previous
  // kernel's blocks have finished (programmatic dependent launch)
  auto launch_coop = [&](auto kern, int grid) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kCoopThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, ca, stw) == cudaSuccess;
  };

  // down leg
  bool down_done = false;
  if (coop) {
    const int gd = occ_grid((const void*)k_amg_down<T, S>, g.Nh, kCoopThreads);
    down_done = launch_coop(k_amg_down<T, S>, gd);
    if (down_done) note_launch();
    else cudaGetLastError();
  }
  if (!down_done) {
    for (int sw = 0; sw < nu1; ++sw) {
      if (sw > 0 || !cpr) gs0(0, sw == 0);
      gs0(1, 0);
    }
    if (nu1 == 0) (launch_pdl(k_zero<T>, grid_for(g.N, TB), TB, 0, s, g.N, x0, st), note_launch());
    (launch_pdl(k_restrict0<T, S>, grid_for(P->lev[1].n, TB), TB, 0, s, g, At, f0, x0, dims_of(P->lev[1]),
        (T*)P->lev[1].f, nu1 > 0, st), note_launch());
    natural_down();
  }

  // the coarser levels: one cluster launch, or the single-block tail (with
  // the natural levels between the legs and the tail per kernel if the
  // cluster launch is refused)
  if (res_from > last || !resident()) {
    if (res_from <= last) {
      cudaGetLastError();
      for (int l = natural_to; l < P->tail_from; ++l) natural_pre(l);
      tail();
      for (int l = P->tail_from - 1; l >= natural_to; --l) natural_post(l);
    } else {
      tail();
    }
  }

  // up leg
  if (down_done) {
    const int gu = occ_grid((const void*)k_amg_up<T, S>, g.Nh, kCoopThreads);
    if (launch_coop(k_amg_up<T, S>, gu)) {
      note_launch();
      return;
    }
    cudaGetLastError();
    natural_up();
  } else {
    natural_up();
  }
  if (nu2 == 0)
    (launch_pdl(k_prolong0<T>, grid_for(g.N, TB), TB, 0, s, g, x0, dims_of(P->lev[1]), (const T*)P->lev[1].x, sc, st),
     note_launch());
  for (int sw = 0; sw < nu2; ++sw) {
    if (sw == 0) gs0_prolong();
    else gs0(1, 0);
    gs0(0, 0);
  }
}

// z = CPR stage applied to v (FP64, internal order); result FP64 in zo
template <typename T, typename S>
void cpr_apply(bo_prec* P, InV v, OutV zo, int stage, const DevState* st, const double* vs) {
  cudaStream_t s = P->stream;
  const Geom& g = P->mat->g;
  const int gN = grid_for(g.N);
  const S* At = (const S*)P->At;
  const S* D = (const S*)P->Dinv;
  T* f = (T*)P->f;
  T* tv = (T*)P->t;
  T* e0 = (T*)P->e0;
  T* f0 = (T*)P->f0;
  T* z1 = (T*)P->z1;
  if (stage == BO_STAGE_AMG) {  // (v is a caller's FP64 vector here: vs is NULL)
    (launch_pdl(k_copy_vec<T>, gN, kThreads, 0, s, g.N, v.d, f0, st), note_launch());
    amg_vcycle<T, S>(P, st, false);
    learned_coarse_apply(P, st);
    (launch_pdl(k_place_p<T>, gN, kThreads, 0, s, g, e0, zo.d, st), note_launch());
    return;
  }
  // x1 = R^{-1} f with f = D_QI^{-1} v (stage CPR) or f = v
  if (stage == BO_STAGE_CPR)
    (launch_cells(k_cpr_entry<T, S, true>, g.N, s, g, v, vs, P->w, P->wf,
        D, f, tv, st),
     note_launch());
  else
    (launch_cells(k_cpr_entry<T, S, false>, g.N, s, g, v, vs, P->w, P->wf,
        D, f, tv, st),
     note_launch());
  (launch_cells(k_ilu_b<T, S>, g.Nh, s, g, At, D, f, tv, z1, st),
   note_launch());
  // (the pass reads z1's black half and writes its red half)
  (launch_cells(k_ilu_r2<T, S, false>, g.Nh, s, g, At, D, tv, z1, z1, nullptr, OutV{}, st),
   note_launch());
  if (stage == BO_STAGE_ILU) {
    (launch_pdl(k_widen_t<T>, grid_for(3 * g.N), kThreads, 0, s, 3 * g.N, z1, zo.d, st), note_launch());
    return;
  }
  // x2 = x1 + Pi_p AMG(A_pp)^{-1} Pi_r (f - At x1)
  (launch_cells(k_cpr_rhs<T, S>, g.N, s, g, At, (const T*)P->di0, f, z1,
      f0, e0, st),
   note_launch());
  amg_vcycle<T, S>(P, st, true);
  learned_coarse_apply(P, st);
  // x3 = x2 + R^{-1} (f - At x2)
  (launch_cells(k_cpr_red<T, S>, g.Nh, s, g, At, D, f, z1, e0, tv,
      st),
   note_launch());
  (launch_cells(k_cpr_black<T, S>, g.Nh, s, g, At, D, f, tv, z1, e0, tv,
      zo, st),
   note_launch());
  (launch_cells(k_ilu_r2<T, S, true>, g.Nh, s, g, At, D, tv, tv, z1, e0, zo, st),
   note_launch());
}

// the arithmetic type of a storage type
template <typename S>
struct ArithOf { using type = float; };
template <>
struct ArithOf<double> { using type = double; };

template <typename S>
int values_impl(bo_prec* P) {
  bo_mat* m = P->mat;
  cudaStream_t s = P->stream;
  const Geom& g = m->g;
  const int tN = cell_threads(g.N), th = cell_threads(g.Nh);
  const int gN = grid_for(g.N, tN), gh = grid_for(g.Nh, th);
  (launch_pdl(k_decouple<S>, gN, tN, 0, s, g, m->A, m->a2_valid ? m->A2 : nullptr, m->a2_range, (S*)P->At, P->w, P->wf,
      P->di0, P->opts.decoupling == BO_DECOUPLE_ABF, P->st), note_launch());
  // FP64 red inverses for the black pass: the Krylov basis is idle during setup
  double* red64 = P->V;
  if (sizeof(S) < sizeof(double) && m->a2_valid) {
    // black pivots in split arithmetic (the kernel takes the FP64 products
    // itself where the split copy of A could not hold every value)
    (launch_pdl(k_ilu_red<S, true>, gh, th, 0, s, g, m->A, P->w, (S*)P->Dinv, red64, P->st), note_launch());
    (launch_pdl(k_ilu_black_split<S>, gh, th, 0, s, g, m->A2, m->A, m->a2_range, P->w,
        reinterpret_cast<const float2*>(red64), (S*)P->Dinv, P->st),
     note_launch());
  } else {
    (launch_pdl(k_ilu_red<S, false>, gh, th, 0, s, g, m->A, P->w, (S*)P->Dinv, red64, P->st), note_launch());
    (launch_pdl(k_ilu_black<S>, gh, th, 0, s, g, m->A, P->w, red64, (S*)P->Dinv, P->st), note_launch());
  }
  // AMG hierarchy values (eight threads per coarse cell)
  for (int l = 1; l < P->nlev; ++l) {
    Level& C = P->lev[l];
    if (l == 1)
      (launch_pdl(k_galerkin0<S>, grid_for(8 * C.n), kThreads, 0, s, g, m->A, P->w, dims_of(C), C.c64, (S*)C.c, P->st),
       note_launch());
    else
      (launch_pdl(k_galerkinn<S>, grid_for(8 * C.n), kThreads, 0, s, dims_of(P->lev[l - 1]), P->lev[l - 1].c64,
           dims_of(C), C.c64, (S*)C.c, P->st), note_launch());
  }
  const int last = P->nlev - 1;
  const LevelDims cd = last == 0 ? LevelDims{g.nx, g.ny, g.nz, g.N} : dims_of(P->lev[last]);
  if (P->res->cluster > 0) {  // the resident levels' packed copies
    using T = typename ArithOf<S>::type;
    CoefPtrs cf = {};
    int64_t items = 0;
    for (int l = P->res->l0; l <= last; ++l) {
      if (l) cf.c[l] = P->lev[l].c;
      items += l == last ? P->res->rl[l].n : P->res->rl[l].npairs;
    }
    (launch_pdl(k_res_pack<T, S>, (int)((items + kThreads - 1) / kThreads), kThreads, 0, s, *P->res, g, (const S*)P->At,
         (const T*)P->di0, cf), note_launch());
  }
  const DenseSrc src{nullptr, last == 0 ? nullptr : P->lev[last].c64, cd, g, m->A, P->w};
  if (launch_gj<S>((int)P->ncoarse, src, (S*)P->coarse_inv, true, P->st, s) != cudaSuccess) return BO_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return BO_ERR_CUDA;
  return learned_coarse_values(P);
}

}  // namespace

int prec_alloc(bo_prec* P) {
  const Geom& g = P->mat->g;
  const size_t ts = P->tsize;
  bool ok = true;
  auto al = [&](size_t bytes) -> void* {
    void* p = nullptr;
    if (ok && cudaMalloc(&p, bytes) != cudaSuccess) { ok = false; return nullptr; }
    return p;
  };
  const size_t ss = P->ssize;  // storage of the matrix-like arrays
  P->At = al(a2_size(g) * ss);  // tiled like the split copy of A (at_index)
  P->w = (double*)al((size_t)3 * g.N * sizeof(double));
  P->wf = ts == sizeof(float) ? (float*)al((size_t)3 * g.N * sizeof(float)) : nullptr;
  P->Dinv = al((size_t)9 * g.N * ss);
  P->di0 = ss == sizeof(double) ? (double*)al((size_t)g.N * sizeof(double)) : nullptr;
  P->f = al((size_t)3 * g.N * ts);
  P->t = al((size_t)3 * g.N * ts);
  P->z1 = al((size_t)3 * g.N * ts);
  P->e0 = al((size_t)g.N * ts);
  P->f0 = al((size_t)g.N * ts);
  // AMG hierarchy shape
  int coarse_max = P->opts.amg_coarse_max;
  if (coarse_max <= 0 || coarse_max > kCoarseMax) coarse_max = kCoarseMax;
  P->nlev = 1;
  int nx = g.nx, ny = g.ny, nz = g.nz;
  int64_t n = g.N;
  while (n > coarse_max && P->nlev < 24) {
    nx = (nx + 1) / 2; ny = (ny + 1) / 2; nz = (nz + 1) / 2;
    n = (int64_t)nx * ny * nz;
    Level& L = P->lev[P->nlev];
    L.nx = nx; L.ny = ny; L.nz = nz; L.n = n;
    L.c64 = (double*)al((size_t)7 * n * sizeof(double));
    L.c = al((size_t)(ss == 8 ? 8 : 7) * n * ss);  // level_slots
    L.f = al((size_t)n * ts);
    L.x = al((size_t)n * ts);
    P->nlev++;
  }
  if (n > kCoarseMax) return BO_ERR_ARG;
  P->ncoarse = n;
  P->tail_from = P->nlev - 1;
  for (int l = 1; l < P->nlev; ++l)
    if (P->lev[l].n <= kTailCells) { P->tail_from = l; break; }
  if (P->tail_from < 1) P->tail_from = 1;
  P->coarse_inv = al((size_t)n * n * ss);
  // the resident AMG levels
  P->res = new (std::nothrow) ResPlan();
  if (!P->res) return BO_ERR_OOM;
  if (P->bf16) resident_plan<float, __nv_bfloat16>(P, *P->res);
  else if (P->fp32) resident_plan<float, float>(P, *P->res);
  else resident_plan<double, double>(P, *P->res);
  if (P->res->cluster > 0) {
    ResPlan& a = *P->res;
    const size_t K = ts == sizeof(double) ? res_values<double>() : res_values<float>();
    for (int l = a.l0; l <= a.last; ++l) {
      ResLevel& r = a.rl[l];
      if (l < a.last) r.cp = al(2 * K * r.npairs * ts);
      r.meta = (int32_t*)al((size_t)(l < a.last ? 3 * r.npairs : r.n) * sizeof(int32_t));
      r.f = l ? P->lev[l].f : P->f0;
      r.x = l ? P->lev[l].x : P->e0;
    }
    a.inv = P->coarse_inv;
  }
  if (ok && cudaMalloc(&P->st, sizeof(DevState)) != cudaSuccess) ok = false;
  if (ok) cudaMemsetAsync(P->st, 0, sizeof(DevState), P->stream);
  return ok ? BO_OK : BO_ERR_OOM;
}

void prec_free(bo_prec* P) {
  auto fr = [](void* p) { if (p) cudaFree(p); };
  fr(P->At); fr(P->w); fr(P->wf); fr(P->Dinv); fr(P->di0);
  fr(P->f); fr(P->t); fr(P->z1); fr(P->e0); fr(P->f0);
  for (int l = 1; l < P->nlev; ++l) { fr(P->lev[l].c64); fr(P->lev[l].c); fr(P->lev[l].f); fr(P->lev[l].x); }
  fr(P->coarse_inv); fr(P->st);
  if (P->res) {
    for (int l = 0; l < 24; ++l) { fr(P->res->rl[l].cp); fr(P->res->rl[l].meta); }
    delete P->res;
    P->res = nullptr;
  }
  learned_coarse_free(P);
  graphs_reset(P);
  if (P->cap_stream) cudaStreamDestroy(P->cap_stream);
  P->cap_stream = nullptr;
}

int prec_values(bo_prec* P) {
  if (P->bf16) return values_impl<__nv_bfloat16>(P);
  return P->fp32 ? values_impl<float>(P) : values_impl<double>(P);
}

// (not where the cluster launch takes every level, nor where level 0 is the coarsest)
bool amg_has_tiles(const bo_prec* P) {
  return P->nlev > 1 && !(g_amg_coop.load() == 2 && P->res->cluster > 0 && P->res->l0 == 0);
}

int launch_dense_inverse64(int n, const double* M, double* Minv, DevState* st, cudaStream_t s) {
  if (n < 1 || n > kCoarseMax) return BO_ERR_ARG;
  const DenseSrc src{M, nullptr, LevelDims{n, 1, 1, n}, Geom{}, nullptr, nullptr};
  if (launch_gj<double>(n, src, Minv, false, st, s) != cudaSuccess) return BO_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? BO_OK : BO_ERR_CUDA;
}

void launch_cpr(bo_prec* P, const double* v, double* z, int stage, const DevState* st, const double* vs) {
  const int64_t n = 3 * P->mat->g.N;
  const InV in{v, nullptr, n};
  const OutV out{z, nullptr, n};
  if (P->bf16) cpr_apply<float, __nv_bfloat16>(P, in, out, stage, st, vs);
  else if (P->fp32) cpr_apply<float, float>(P, in, out, stage, st, vs);
  else cpr_apply<double, double>(P, in, out, stage, st, vs);
}

void launch_cpr_split(bo_prec* P, const double* v, float* z, const DevState* st, const double* vs) {
  const int64_t n = 3 * P->mat->g.N;
  const InV in{v, nullptr, n};
  const OutV out{nullptr, z, n};
  if (P->bf16) cpr_apply<float, __nv_bfloat16>(P, in, out, BO_STAGE_CPR, st, vs);
  else if (P->fp32) cpr_apply<float, float>(P, in, out, BO_STAGE_CPR, st, vs);
  else cpr_apply<double, double>(P, in, out, BO_STAGE_CPR, st, vs);
}

void launch_cpr_split_in(bo_prec* P, const float* v, float* z, const DevState* st, const double* vs) {
  const int64_t n = 3 * P->mat->g.N;
  const InV in{nullptr, v, (n + 3) & ~(int64_t)3};  // the basis layout: low plane at n rounded up to 4
  const OutV out{nullptr, z, n};
  if (P->bf16) cpr_apply<float, __nv_bfloat16>(P, in, out, BO_STAGE_CPR, st, vs);
  else if (P->fp32) cpr_apply<float, float>(P, in, out, BO_STAGE_CPR, st, vs);
  else cpr_apply<double, double>(P, in, out, BO_STAGE_CPR, st, vs);
}

void launch_spmv_decoupled_internal(bo_prec* P, const double* x, double* y) {
  const Geom& g = P->mat->g;
  (launch_pdl(k_spmv_dec64, grid_for(g.N), kThreads, 0, P->stream, g, P->mat->A, P->w, x, y), note_launch());
}

}  // namespace bo
