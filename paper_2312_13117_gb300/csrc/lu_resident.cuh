// Dense complex LU with partial pivoting of a matrix that stays in shared memory
// for the whole factorisation, templated on the element type.
//
// A node of order n with l probe columns takes (n + l)(n | 1) elements: up to
// n = 110 at l = 10 in complex128 and n = 160 at l = 8 in complex64 fit one SM.
// The blocked routines of lu_core.cuh hold the matrix in global memory and give a
// column four block barriers and several global round trips; here a column takes
// two barriers and no global access:
//   * warp 0 looks ahead: it updates column j + 1 first, finds its pivot, forms the
//     reciprocal and scales the column, while the other warps apply column j to
//     the columns right of it;
//   * the rank-1 update runs over tiles of RW rows x 4 (or 2) x CU columns, one warp
//     each. In FP64 a warp's multiply-add occupies its scheduler's FP64 unit for
//     64 clocks, so lanes without an element cost as much as busy ones: the tile
//     is narrow in both directions (padding below 4 of 75 rows and columns on
//     average at n = 100), and the tiles are handed out by a shared counter, which
//     keeps the four schedulers' units level to within one tile;
//   * the pivots' reciprocals are kept, so that the back substitution multiplies.
//     A complex division costs about 30 FP64 instructions.
// The pivot rule is that of lu_core.cuh (largest |Re| + |Im|, lowest row on ties)
// and every element receives its updates in the same order.
#pragma once

#include "lu_core.cuh"

namespace resident {

__host__ __device__ inline int lead(int n) { return n | 1; }  // odd: row swaps touch distinct banks

// Shared control words of one factorisation.
struct Ctl {
  int info;  // 0, or 1 + the first column whose pivot was exactly zero
  int tile;  // next tile of the running update
};

// Bytes of shared memory of a node: matrix and probe columns, reciprocals, pivots.
__host__ __device__ inline size_t node_bytes(int n, int l, size_t elem) {
  return (((size_t)lead(n) * (n + l) + n) * elem + (size_t)n * sizeof(int) + 15) & ~(size_t)15;
}

// One warp: pivot of column j (rows j..n-1, up to date), the swap inside the
// column, the pivot's reciprocal, and the multipliers below it.
template <typename T2>
__device__ __forceinline__ void pivot_column(T2* __restrict__ col, int n, int j, int* __restrict__ piv,
                                             T2* __restrict__ rinv, Ctl& ctl) {
  using R = decltype(l1abs(T2{}));
  const int lane = threadIdx.x & 31;
  R bv = R(-1);
  int bi = n;
  for (int i = j + lane; i < n; i += 32) {
    const R v = l1abs(col[i]);
    if (v > bv) { bv = v; bi = i; }
  }
  lucore::warp_argmax(bv, bi);
  int p = __shfl_sync(0xffffffffu, bi, 0);
  if (p >= n) p = j;
  const T2 pv = col[p], top = col[j];
  const bool zero = cis_zero(pv);
  const T2 rp = crecip(pv);  // not finite for a zero pivot, as a division by it would be
  __syncwarp();
  for (int i = j + 1 + lane; i < n; i += 32) {
    const T2 v = i == p ? top : col[i];
    col[i] = zero ? v : cmul(v, rp);
  }
  if (lane == 0) {
    col[j] = pv;
    piv[j] = p;
    rinv[j] = rp;
    if (zero && ctl.info == 0) ctl.info = j + 1;
  }
  __syncwarp();
}

// LU of the n x n leading block of M (column-major, leading dimension ld, shared
// memory) with ncols >= n columns; every thread of the CTA calls it, after a
// barrier that follows the last write to M. Row swaps reach all columns. Returns
// with the CTA synchronised; ctl.info, piv and rinv are then set.
template <typename T2>
__device__ __forceinline__ void factor(T2* __restrict__ M, int n, int ncols, int ld, int* __restrict__ piv,
                                       T2* __restrict__ rinv, Ctl& ctl) {
  constexpr bool kDouble = sizeof(T2) == 16;
  constexpr int RW = kDouble ? 8 : 16;    // tile rows: one conflict-free phase of a shared access
  constexpr int CW = 32 / RW;             // columns a warp touches at once
  constexpr int CU = 4;                   // of those, per tile
  constexpr int TC = CW * CU;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x, nwarp = nthr >> 5;
  const int lr = lane & (RW - 1), lc = lane / RW;
  if (warp == 0) {
    if (lane == 0) ctl.info = 0;
    __syncwarp();
    pivot_column(M, n, 0, piv, rinv, ctl);
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int p = piv[j];
    if (p != j)
      for (int c = tid; c < ncols; c += nthr)
        if (c != j) {
          const T2 t = M[(size_t)c * ld + j];
          M[(size_t)c * ld + j] = M[(size_t)c * ld + p];
          M[(size_t)c * ld + p] = t;
        }
    if (tid == 0) ctl.tile = 0;
    __syncthreads();
    const T2* lj = M + (size_t)j * ld;
    // a zero pivot leaves the columns right of it as they are (its multipliers are all zero)
    const bool zero = cis_zero(lj[j]);
    const int r_lo = j + 1, m = n - r_lo;
    if (warp == 0 && j + 1 < n) {
      T2* cj = M + (size_t)(j + 1) * ld;
      const T2 u = cj[j];
      if (!zero)
        for (int i = r_lo + lane; i < n; i += 32) {
          T2 v = cj[i];
          cfms(v, lj[i], u);
          cj[i] = v;
        }
      __syncwarp();
      pivot_column(cj, n, j + 1, piv, rinv, ctl);
    }
    const int c_lo = j + 2, mc = ncols - c_lo;
    if (m > 0 && mc > 0 && !zero) {
      const int ntr = (m + RW - 1) / RW, nt = ntr * ((mc + TC - 1) / TC);
      int t = warp;
      for (;;) {
        if (kDouble) {
          if (lane == 0) t = atomicAdd(&ctl.tile, 1);
          t = __shfl_sync(0xffffffffu, t, 0);
        }
        if (t >= nt) break;
        const int tc = t / ntr, tr = t - tc * ntr;
        const int i = r_lo + tr * RW + lr, c0 = c_lo + tc * TC + lc;
        const bool row_ok = i < n;
        const T2 l = row_ok ? lj[i] : czero<T2>();
        T2 v[CU], u[CU];
#pragma unroll
        for (int q = 0; q < CU; ++q) {
          const int c = c0 + q * CW;
          if (row_ok && c < ncols) {
            v[q] = M[(size_t)c * ld + i];
            u[q] = M[(size_t)c * ld + j];
          }
        }
#pragma unroll
        for (int q = 0; q < CU; ++q) {
          const int c = c0 + q * CW;
          if (row_ok && c < ncols) {
            cfms(v[q], l, u[q]);
            M[(size_t)c * ld + i] = v[q];
          }
        }
        if (!kDouble) t += nwarp;
      }
    }
    __syncthreads();
  }
}

// U X = Y in place for the l columns after the n x n block: a half warp owns a
// column and takes 16 rows at a time, so no barrier is needed.
template <typename T2>
__device__ __forceinline__ void back(T2* __restrict__ M, int n, int l, int ld, const T2* __restrict__ rinv) {
  const int lane = threadIdx.x & 15, nhalf = blockDim.x >> 4;
  const unsigned mask = 0xffffu << (threadIdx.x & 16);
  for (int c = threadIdx.x >> 4; c < l; c += nhalf) {
    T2* y = M + (size_t)(n + c) * ld;
    for (int j = n - 1; j >= 0; --j) {
      const T2 x = cmul(y[j], rinv[j]);
      const T2* uj = M + (size_t)j * ld;
      __syncwarp(mask);
      if (lane == 0) y[j] = x;
      for (int i = lane; i < j; i += 16) {
        T2 v = y[i];
        cfms(v, uj[i], x);
        y[i] = v;
      }
      __syncwarp(mask);
    }
  }
}

}  // namespace resident
