// Node solves for small problems (n <= 32, l <= 16): one warp per node.
//
// The same work as the CTA kernels (assembly of T(z_j), LU with partial
// pivoting on [T | V], back substitution), but a whole node lives in one
// warp's slice of shared memory with lane i owning row i, so every step is
// warp-synchronous: no block barriers, and an SM holds many nodes at once.
// Pivot rule as everywhere: largest |Re| + |Im| in the column, lowest row on
// ties.
#include "pmcim_internal.cuh"

namespace {

constexpr int WARPS = 4;
constexpr int SN = 32;  // largest n
constexpr int SL = 16;  // largest l

struct SmallSmem {  // then WARPS matrices of `rows` rows of `ldc` entries
  ProblemDev P[WARPS];
  double2 fz[WARPS][PMCIM_MAX_TERMS];
  double2 divisor[WARPS][SN];  // Smith's ratio and denominator of the pivots
};
constexpr size_t kSmallHead = (sizeof(SmallSmem) + 15) & ~size_t(15);
// Row length for n + l columns: odd, so that eight rows lie in distinct banks.
__host__ __device__ inline int small_ldc(int n, int l) { return (n + l) | 1; }

template <bool BIE>
__global__ void __launch_bounds__(WARPS * 32) k_factor_solve_small(NodeArgs a, int matrix_elems) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmallSmem& sm = *reinterpret_cast<SmallSmem*>(smem_raw);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lr = lane & 7, lc = lane >> 3;  // a tile of 8 rows x 4 columns
  double2* M = reinterpret_cast<double2*>(smem_raw + kSmallHead) + (size_t)w * matrix_elems;
  double2* divisor = sm.divisor[w];
  ProblemDev& P = sm.P[w];
  for (;;) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(a.counter, 1);
    idx = __shfl_sync(0xffffffffu, idx, 0);
    if (idx >= a.n_items) break;
    const NodeItem it = a.items[idx];
    const RegionDev rg = a.regions[it.region];
    {
      const int* s = reinterpret_cast<const int*>(a.probs + rg.prob);
      int* d = reinterpret_cast<int*>(&P);
      for (int i = lane; i < (int)(sizeof(ProblemDev) / sizeof(int)); i += 32) d[i] = s[i];
    }
    __syncwarp();
    const int n = P.n, l = P.l, ncols = n + l, LDC = small_ldc(n, l);
    double2 z, wgt;
    node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &wgt);
    if (lane < P.K) sm.fz[w][lane] = eval_f(P.term[lane], z);
    __syncwarp();
    const size_t nn = (size_t)n * n;
    // assemble [T(z_j) | V] (T(z_j)^H for a certificate's step with rg.herm), row `lane`
    if (lane < n) {
      double2* row = M + lane * LDC;
      for (int c = 0; c < n; ++c) {
        double2 v = make_double2(0.0, 0.0);
        const size_t e = rg.herm ? (size_t)lane * n + c : (size_t)c * n + lane;
        for (int k = 0; k < P.K; ++k) {
          const TermDesc& t = P.term[k];
          if (t.dense) cfma(v, sm.fz[w][k], P.A[(size_t)t.mat_index * nn + e]);
          else if (c == lane && t.kind != PMCIM_F_HELMHOLTZ_DLP) cfma(v, sm.fz[w][k], t.id);
        }
        if (rg.herm) v.y = -v.y;
        row[c] = v;
      }
      for (int c = 0; c < l; ++c) row[n + c] = P.V[(size_t)c * n + lane];
    }
    __syncwarp();
    if (BIE && P.bie) {
      const bie::Wave W = bie::wave_of(z);
      add_layer(P.bie, n, layer_coefficient(P), W, lane, 32, [&](int i, int j, double2 v) {
        double2& m = rg.herm ? M[j * LDC + i] : M[i * LDC + j];  // T^H: entry (j, i) is conj(T_ij)
        m = cadd(m, rg.herm ? cconj(v) : v);
      });
      __syncwarp();
    }
    int info = 0;
    for (int j = 0; j < n; ++j) {
      double bv = -1.0;
      int bi = n;
      if (lane >= j && lane < n) {
        bv = l1abs(M[lane * LDC + j]);
        bi = lane;
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_down_sync(0xffffffffu, bv, o);
        const int oi = __shfl_down_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      int p = __shfl_sync(0xffffffffu, bi, 0);
      if (p >= n) p = j;
      if (p != j)
        for (int c = lane; c < ncols; c += 32) {
          const double2 t = M[j * LDC + c];
          M[j * LDC + c] = M[p * LDC + c];
          M[p * LDC + c] = t;
        }
      __syncwarp();
      const double2 pv = M[j * LDC + j];
      const Smith sd(pv);
      const double2 rp = sd.reciprocal();  // not finite for a zero pivot, as a division by it would be
      if (lane == 0) divisor[j] = make_double2(sd.t, sd.d);
      if (pv.x == 0.0 && pv.y == 0.0) {
        if (info == 0) info = j + 1;
        __syncwarp();
        continue;
      }
      if (lane > j && lane < n) M[lane * LDC + j] = Smith::multiplier(M[lane * LDC + j], rp);
      __syncwarp();
      // rank-1 update in tiles of 8 rows x 4 columns: a lane without an element costs the FP64
      // unit as much as a busy one, and a row per lane leaves most idle in the end
      for (int r0 = j + 1; r0 < n; r0 += 8) {
        const int r = r0 + lr;
        const double2 lij = r < n ? M[r * LDC + j] : make_double2(0.0, 0.0);
        for (int c0 = j + 1 + lc; c0 < ncols; c0 += 16) {
          double2 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (r < n && c0 + 4 * q < ncols) v[q] = M[r * LDC + c0 + 4 * q];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (r < n && c0 + 4 * q < ncols) {
              cfms(v[q], lij, M[j * LDC + c0 + 4 * q]);
              M[r * LDC + c0 + 4 * q] = v[q];
            }
        }
      }
      __syncwarp();
    }
    // back substitution U X = Y on the l right-hand columns
    for (int j = n - 1; j >= 0; --j) {
      // lanes c and c + 16: the real and the imaginary part of column c's quotient (l <= 16)
      const int c = lane & (SL - 1), im = lane / SL;
      double q = 0.0;
      if (c < l) {
        const double2 td = divisor[j];
        q = Smith(M[j * LDC + j], td.x, td.y).part(M[j * LDC + n + c], im);
      }
      __syncwarp();
      if (c < l) (im ? M[j * LDC + n + c].y : M[j * LDC + n + c].x) = q;
      __syncwarp();
      if (lane < j)
        for (int c = 0; c < l; ++c) cfms(M[lane * LDC + n + c], M[lane * LDC + j], M[j * LDC + n + c]);
      __syncwarp();
    }
    if (lane < n) {
      double2* Xo = a.X + rg.x_off + (size_t)it.j * n * l;
      for (int c = 0; c < l; ++c) Xo[(size_t)c * n + lane] = M[lane * LDC + n + c];
    }
    if (lane == 0) a.node_info[rg.node_off + it.j] = info;
    __syncwarp();
  }
}

}  // namespace

bool small_kernel_fits(int n, int l) { return n <= SN && l <= SL; }

namespace {
constexpr size_t kSmallMax = kSmallHead + (size_t)WARPS * SN * ((SN + SL) | 1) * sizeof(double2);
}  // namespace

cudaError_t prepare_factor_small() {
  cudaError_t e = cudaFuncSetAttribute(k_factor_solve_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmallMax);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_factor_solve_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmallMax);
}

// Launch only; prepare_factor_small() must have set the shared-memory limit. max_n, max_l: the
// largest among the items, which set how many nodes an SM holds (n = 24, l = 1: 20; at the
// largest sizes 8). The FP64 unit bounds the kernel: quotients that share the pivot's part of the
// division (a complex division is some 90 FP64 instructions of a warp) and the narrow update tiles
// took a call of 3072 nodes of n = 24, l = 1 from 1.26 to 0.83 ms, 0.80 with products by rounded
// reciprocals, which are another rounding.
cudaError_t launch_factor_solve_small(const NodeArgs& a, int max_n, int max_l, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int elems = max_n * small_ldc(max_n, max_l);
  const size_t smem = kSmallHead + (size_t)WARPS * elems * sizeof(double2);
  int per = (int)((227 * 1024 + 1024) / (smem + 1024));
  if (per > 5) per = 5;
  int grid = per * (sms > 0 ? sms : 1);
  const int need = (a.n_items + WARPS - 1) / WARPS;
  if (grid > need) grid = need;
  if (a.bie) k_factor_solve_small<true><<<grid, WARPS * 32, smem, s>>>(a, elems);
  else k_factor_solve_small<false><<<grid, WARPS * 32, smem, s>>>(a, elems);
  return cudaGetLastError();
}
