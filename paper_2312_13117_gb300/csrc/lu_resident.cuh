// Dense complex LU with partial pivoting (FP64) of a matrix that stays in shared
// memory for the whole factorisation.
//
// A node of order n with l probe columns takes (n + l)(n | 1) elements: up to
// n = 110 at l = 10 fit one SM.
// The blocked routines of lu_core.cuh hold the matrix in global memory and give a
// column four block barriers and several global round trips; here a column takes
// two barriers and no global access:
//   * warp 0 looks ahead: it updates column j + 1 first, finds its pivot, forms the
//     multipliers and scales the column, while the other warps apply column j to
//     the columns right of it;
//   * the rank-1 update runs over tiles of RW rows x 4 x CU columns, one warp
//     each. A warp's multiply-add occupies its scheduler's FP64 unit for
//     64 clocks, so lanes without an element cost as much as busy ones: the tile
//     is narrow in both directions (padding below 4 of 75 rows and columns on
//     average at n = 100), and the tiles are handed out by a shared counter, which
//     keeps the four schedulers' units level to within one tile;
//   * the back substitution's quotients (Smith) share the parts of the division that
//     depend on the pivot alone, and a quotient's two real divisions run in two lanes:
//     11 FP64 instructions of a warp instead of some 40.
// The pivot rule is that of lu_core.cuh (largest |Re| + |Im|, lowest row on ties)
// and every element receives the same operations in the same order as there.
#pragma once

#include "lu_core.cuh"

namespace resident {

__host__ __device__ inline int lead(int n) { return n | 1; }  // odd: row swaps touch distinct banks

// Shared control words of one factorisation.
struct Ctl {
  int info;  // 0, or 1 + the first column whose pivot was exactly zero
  int tile;  // next tile of the running update
};

// Bytes of shared memory of a node: matrix and probe columns, divisors, pivots.
__host__ __device__ inline size_t node_bytes(int n, int l) {
  return (((size_t)lead(n) * (n + l) + n) * sizeof(double2) + (size_t)n * sizeof(int) + 15) & ~(size_t)15;
}

// One warp: pivot of column j (rows j..n-1, up to date), the swap inside the
// column, the pivot's divisor (Smith), and the multipliers below it.
__device__ __forceinline__ void pivot_column(double2* __restrict__ col, int n, int j, int* __restrict__ piv,
                                             double2* __restrict__ divisor, Ctl& ctl) {
  const int lane = threadIdx.x & 31;
  double bv = -1.0;
  int bi = n;
  for (int i = j + lane; i < n; i += 32) {
    const double v = l1abs(col[i]);
    if (v > bv) { bv = v; bi = i; }
  }
  lucore::warp_argmax(bv, bi);
  int p = __shfl_sync(0xffffffffu, bi, 0);
  if (p >= n) p = j;
  const double2 pv = col[p], top = col[j];
  const bool zero = cis_zero(pv);
  const Smith sd(pv);
  const double2 rp = sd.reciprocal();  // not finite for a zero pivot, as a division by it would be
  __syncwarp();
  for (int i = j + 1 + lane; i < n; i += 32) {
    const double2 v = i == p ? top : col[i];
    col[i] = zero ? v : Smith::multiplier(v, rp);
  }
  if (lane == 0) {
    col[j] = pv;
    piv[j] = p;
    divisor[j] = make_double2(sd.t, sd.d);
    if (zero && ctl.info == 0) ctl.info = j + 1;
  }
  __syncwarp();
}

// LU of the n x n leading block of M (column-major, leading dimension ld, shared
// memory) with ncols >= n columns; every thread of the CTA calls it, after a
// barrier that follows the last write to M. Row swaps reach all columns. Returns
// with the CTA synchronised; ctl.info, piv and divisor are then set.
__device__ __forceinline__ void factor(double2* __restrict__ M, int n, int ncols, int ld, int* __restrict__ piv,
                                       double2* __restrict__ divisor, Ctl& ctl) {
  constexpr int RW = 8;                   // tile rows: one conflict-free phase of a shared access
  constexpr int CW = 32 / RW;             // columns a warp touches at once
  constexpr int CU = 4;                   // of those, per tile
  constexpr int TC = CW * CU;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
  const int lr = lane & (RW - 1), lc = lane / RW;
  if (warp == 0) {
    if (lane == 0) ctl.info = 0;
    __syncwarp();
    pivot_column(M, n, 0, piv, divisor, ctl);
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int p = piv[j];
    if (p != j)
      for (int c = tid; c < ncols; c += nthr)
        if (c != j) {
          const double2 t = M[(size_t)c * ld + j];
          M[(size_t)c * ld + j] = M[(size_t)c * ld + p];
          M[(size_t)c * ld + p] = t;
        }
    if (tid == 0) ctl.tile = 0;
    __syncthreads();
    const double2* lj = M + (size_t)j * ld;
    // a zero pivot leaves the columns right of it as they are (its multipliers are all zero)
    const bool zero = cis_zero(lj[j]);
    const int r_lo = j + 1, m = n - r_lo;
    if (warp == 0 && j + 1 < n) {
      double2* cj = M + (size_t)(j + 1) * ld;
      const double2 u = cj[j];
      if (!zero)
        for (int i = r_lo + lane; i < n; i += 32) {
          double2 v = cj[i];
          cfms(v, lj[i], u);
          cj[i] = v;
        }
      __syncwarp();
      pivot_column(cj, n, j + 1, piv, divisor, ctl);
    }
    const int c_lo = j + 2, mc = ncols - c_lo;
    if (m > 0 && mc > 0 && !zero) {
      const int ntr = (m + RW - 1) / RW, nt = ntr * ((mc + TC - 1) / TC);
      for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&ctl.tile, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= nt) break;
        const int tc = t / ntr, tr = t - tc * ntr;
        const int i = r_lo + tr * RW + lr, c0 = c_lo + tc * TC + lc;
        const bool row_ok = i < n;
        const double2 l = row_ok ? lj[i] : make_double2(0.0, 0.0);
        double2 v[CU], u[CU];
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
      }
    }
    __syncthreads();
  }
}

// U X = Y in place for the l columns after the n x n block, in the blocked routine's order
// (cta_back_blocked of lu_core.cuh): W lanes own a column, so no barrier is needed.
template <int W>
__device__ __forceinline__ void back_w(double2* __restrict__ M, int n, int l, int ld,
                                       const double2* __restrict__ divisor) {
  constexpr int NB = lucore::NB;
  const int lane = threadIdx.x & (W - 1), part = lane & 1;
  const unsigned mask = (W == 32 ? 0xffffffffu : (1u << W) - 1u) << (threadIdx.x & 31 & ~(W - 1));
  for (int c = threadIdx.x / W; c < l; c += blockDim.x / W) {
    double2* y = M + (size_t)(n + c) * ld;
    for (int k0 = (n - 1) / NB * NB; k0 >= 0; k0 -= NB) {
      const int kend = min(n, k0 + NB);
      for (int j = kend - 1; j >= k0; --j) {
        const double2* uj = M + (size_t)j * ld;
        const double2 td = divisor[j];
        const double q = Smith(uj[j], td.x, td.y).part(y[j], part);  // even lanes: real, odd: imaginary
        const double2 x = make_double2(__shfl_sync(mask, q, 0, W), __shfl_sync(mask, q, 1, W));
        if (lane == 0) y[j] = x;
        for (int i = k0 + lane; i < j; i += W) {
          double2 v = y[i];
          cfms(v, uj[i], x);
          y[i] = v;
        }
        __syncwarp(mask);
      }
      for (int i = lane; i < k0; i += W) {
        double2 v = y[i];
        for (int j = k0; j < kend; ++j) cfms(v, M[(size_t)j * ld + i], y[j]);
        y[i] = v;
      }
      __syncwarp(mask);
    }
  }
}
// 16 lanes a column while that leaves no scheduler more than one warp (l <= 8), else 8, which
// halves the instructions of the quotients.
__device__ __forceinline__ void back(double2* __restrict__ M, int n, int l, int ld,
                                     const double2* __restrict__ divisor) {
  if (l <= 8) back_w<16>(M, n, l, ld, divisor);
  else back_w<8>(M, n, l, ld, divisor);
}

}  // namespace resident
