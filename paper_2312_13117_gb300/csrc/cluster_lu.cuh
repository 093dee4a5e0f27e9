// FP64 LU of one matrix by a thread-block cluster.
//
// Where few matrices are to be factored, one CTA each leaves most SMs idle, so the CTAs of a
// cluster share one: the LU of order 512 takes 52 ms on one SM, on the FP64 pipe, and 18.7 on 4
// (7.6 of it the panels, which one CTA factors). Every CTA of a cluster reaches every barrier
// below.
#pragma once

#include "lu_core.cuh"

namespace lucore {

struct Interchanges {
  int row[2 * NB], src[2 * NB];  // a panel's interchanges: row[i] takes the old row src[i]
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}

__device__ __forceinline__ double2 shfl2(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// A panel's interchanges on all other columns and U12 = L11^{-1} A12 on those right of it:
// a warp takes four columns, lane t the rows k0 + t and piv[k0 + t].
__device__ inline void swap_and_trsm(double2* M, int n, int ncols, int k0, int kb, const int* piv, LuSmem& lu,
                                     Interchanges& sw, int rank, int size) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 2 * NB) {  // follow one row back through the interchanges
    const int t = tid & (NB - 1);
    int r = t >= kb ? 0 : (tid < NB ? k0 + t : piv[k0 + t]);
    sw.row[tid] = r;
    for (int j = kb - 1; j >= 0; --j) {
      const int p = piv[k0 + j];
      r = r == k0 + j ? p : (r == p ? k0 + j : r);
    }
    sw.src[tid] = r;
  }
#pragma unroll
  for (int u = 0; u < NB * NB / THREADS; ++u) {
    const int e = tid + u * THREADS, i = e & (NB - 1), t = e / NB;
    lu.Ls[e] = i < kb && t < kb && i > t ? M[(size_t)(k0 + t) * n + k0 + i] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const bool live = lane < kb;
  const int s0 = sw.src[lane], r1 = sw.row[NB + lane], s1 = sw.src[NB + lane];
  constexpr int CW = 4;
  for (int g = (rank * THREADS + tid) >> 5; g * CW < ncols; g += size * (THREADS / 32)) {
    double2 x[CW], y[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      const int c = g * CW + q;
      const bool in = live && c < ncols && (c < k0 || c >= k0 + kb);
      x[q] = in ? M[(size_t)c * n + s0] : make_double2(0.0, 0.0);
      y[q] = in ? M[(size_t)c * n + s1] : make_double2(0.0, 0.0);
    }
    __syncwarp();
    // rows below the panel's, before the panel's own (a row piv[k0 + t] may be one of those:
    // both then hold the same value)
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      const int c = g * CW + q;
      if (live && r1 >= k0 + kb && c < ncols && (c < k0 || c >= k0 + kb)) M[(size_t)c * n + r1] = y[q];
    }
    if ((g + 1) * CW > k0 + kb)
      for (int t = 0; t < kb - 1; ++t) {
        const double2 lt = lu.Ls[t * NB + lane];
#pragma unroll
        for (int q = 0; q < CW; ++q) {
          const double2 xt = shfl2(x[q], t);
          if (g * CW + q >= k0 + kb && lane > t) cfms(x[q], lt, xt);
        }
      }
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      const int c = g * CW + q;
      if (live && c < ncols && (c < k0 || c >= k0 + kb)) M[(size_t)c * n + k0 + lane] = x[q];
    }
  }
}

// LU of the n x n leading block of M with ncols >= n columns (cta_lu's, to the bit) by a cluster
// of `size` CTAs: the first factors the panels, all share the interchanges, the triangular solves
// and the trailing updates. Returns 0, or 1 + the first column whose pivot was exactly zero
// (*flag: its way to the other CTAs).
__device__ inline int cluster_lu(double2* M, int n, int ncols, int* piv, int* flag, LuSmem& lu, Interchanges& sw,
                                 int rank, int size) {
  if (threadIdx.x == 0) lu.info_sh = 0;
  __syncthreads();
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    if (rank == 0) {
      cta_lu_panel(M, n, k0 + kb, k0, kb, piv, lu, k0);
      if (threadIdx.x == 0) *flag = lu.info_sh;
    }
    cluster_sync();
    swap_and_trsm(M, n, ncols, k0, kb, piv, lu, sw, rank, size);
    cluster_sync();
    if (k0 + kb >= n) break;
    cta_lu_update_simt<double2, 2>(M, n, ncols, k0, kb, lu, rank, size);
    cluster_sync();
  }
  return *flag;
}

}  // namespace lucore
