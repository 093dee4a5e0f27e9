// Plain FP64 path: per-node assembly of T(z_j), blocked complex LU with partial
// pivoting, and the l-column solve, plus verification by sigma_min(T(lambda)).
//
// The paper solves T(z_j) x_j = f at every quadrature node with a dense direct
// solver (Eq. 2.4; Appendix, linearsolver = MATLAB backslash) and suggests
// solving all nodes in parallel (Sec. 3.2, remark on deeper parallelism).
// Here one CTA owns one node at a time (persistent grid, one workspace slot per
// CTA, two CTAs per SM): GB300 issues only ~2 DFMA per SM per clock, so a
// node-per-CTA schedule keeps every SM's FP64 pipe busy without cross-CTA
// synchronisation, and the trailing updates (the O(n^3) part) run from shared
// memory tiles with a 4x4 complex register block per thread.
//
// The probe block V is appended to T as l extra columns, so the row swaps and
// trailing updates of the factorisation also perform P and L^-1 on V; only the
// back substitution with U remains.
//
// Pivot rule: the row maximising |Re| + |Im| in the column, lowest row index on
// ties (the BLAS izamax convention of LAPACK zgetrf).
#include "cluster_lu.cuh"

namespace {

using namespace lucore;

// ---------------------------------------------------------------------------
// Persistent kernel: node g -> X_g = T(z_g)^{-1} V.
// ---------------------------------------------------------------------------
// Shared memory of the node kernel: the LU tiles plus the node's problem.
struct NodeSmem {
  LuSmem lu;
  ProblemDev P;
  bie::Wave wave;
  int item;
};

// RI: the trailing update's register block (4: 64 x 64 tiles; 2: 32 x 32 tiles).
template <int RI, bool BIE>
__global__ void __launch_bounds__(THREADS, 2) k_factor_solve_fp64(NodeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  NodeSmem& sm = *reinterpret_cast<NodeSmem*>(smem_raw);
  const int tid = threadIdx.x;
  double2* M = reinterpret_cast<double2*>(a.work + (size_t)blockIdx.x * a.slot_bytes);
  int* piv = a.piv + (size_t)blockIdx.x * a.max_n;

  for (;;) {
    // largest-first list, handed out by an atomic counter (no waiting on other CTAs)
    if (tid == 0) sm.item = atomicAdd(a.counter, 1);
    __syncthreads();
    const int idx = sm.item;
    if (idx >= a.n_items) break;
    const NodeItem it = a.items[idx];
    const RegionDev rg = a.regions[it.region];
    load_problem(&sm.P, a.probs + rg.prob);
    __syncthreads();
    const ProblemDev& P = sm.P;
    const int n = P.n, l = P.l, ncols = n + l;
    double2 z, w;
    node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &w);
    if (tid < P.K) sm.lu.fz[tid] = eval_f(P.term[tid], z);
    if (BIE && tid == 0) sm.wave = bie::wave_of(z);
    __syncthreads();

    // assemble [T(z_j) | V]
    const size_t nn = (size_t)n * n;
    // a circulant boundary-integral term: its n distinct entries K_{m,0}, formed once per
    // node in the slot's probe-block columns (V is written there below)
    double2* circ = M + nn;
    const bool use_circ = BIE && P.bie_circ;
    if (use_circ) {
      for (int m = tid; m < n; m += THREADS) circ[m] = bie::dlp_entry(P.bie, n, m, 0, sm.wave);
      __syncthreads();
    }
    for (int col = 0; col < n; ++col) {
      for (int row = tid; row < n; row += THREADS) {
        const size_t e = (size_t)col * n + row;
        double2 v = make_double2(0.0, 0.0);
        for (int k = 0; k < P.K; ++k) {
          const TermDesc& t = P.term[k];
          if (t.dense) {
            cfma(v, sm.lu.fz[k], P.A[(size_t)t.mat_index * nn + e]);
          } else if (use_circ && t.kind == PMCIM_F_HELMHOLTZ_DLP) {
            const int m = row >= col ? row - col : row - col + n;
            cfma(v, t.id, circ[m]);
          } else if (row == col && t.kind != PMCIM_F_HELMHOLTZ_DLP) {
            cfma(v, sm.lu.fz[k], t.id);
          }
        }
        M[e] = v;
      }
    }
    if (BIE && P.bie && !use_circ) {
      __syncthreads();
      add_layer(P.bie, n, layer_coefficient(P), sm.wave, tid, THREADS,
                [&](int i, int j, double2 v) { M[(size_t)j * n + i] = cadd(M[(size_t)j * n + i], v); });
    }
    if (use_circ) __syncthreads();  // circ is read above and overwritten by V below
    for (size_t e = tid; e < (size_t)n * l; e += THREADS) M[nn + e] = P.V[e];
    __syncthreads();

    const int info = cta_lu<double2, RI>(M, n, ncols, piv, sm.lu);
    cta_back_blocked(M, n, l, sm.lu);

    double2* Xo = a.X + rg.x_off + (size_t)it.j * n * l;
    for (size_t e = tid; e < (size_t)n * l; e += THREADS) Xo[e] = M[nn + e];
    if (tid == 0) a.node_info[rg.node_off + it.j] = info;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Verification: sigma_min(T(lambda)) by inverse iteration on (T^H T)^{-1}
// using the LU of T(lambda) (pmCIMb step 3).
// ---------------------------------------------------------------------------
struct VerifySmem {
  LuSmem lu;
  ProblemDev P;
  bie::Wave wave;
  double red[THREADS / 32];
  Interchanges swaps;
};

// ---------------------------------------------------------------------------
// The inverse iteration's triangular solves with one right-hand side, by the whole cluster in
// 32-row blocks. The inverses of the diagonal blocks are formed once per value, so that a
// block's unknowns are a product instead of a chain of 32 dependent steps. The first CTA takes
// columns 0..32/size-1 of each block, and so on: each keeps its own sums
//   acc[rank][i] = sum over its solved columns of A[i, t] y_t
// (a row always by the same thread), and a block's right-hand side is in - sum_rank acc[rank]:
// one cluster barrier per block. What bounds it: 2 n^2 multiply-adds an iteration on the FP64
// pipe and then the barrier and L2 latency of 4 n / 32 blocks. One CTA with one or two barriers a
// row took 3.7 ms an iteration at n = 512, substitution in 32-row blocks 1.2, this 0.33 with 4 CTAs.
// ---------------------------------------------------------------------------
// The inverses of L's (type 0) and U's (type 1) diagonal blocks, column-major and zero-padded
// to 32 x 32: dinv + (type * blocks + block) * NB * NB. A warp takes four columns.
__device__ void invert_diagonals(const double2* M, int n, double2* dinv, int rank, int size) {
  constexpr int CW = 4;
  const int lane = threadIdx.x & 31, blocks = (n + NB - 1) / NB;
  for (int g = (rank * THREADS + (int)threadIdx.x) >> 5; g < 2 * blocks * (NB / CW); g += size * (THREADS / 32)) {
    const int type = g / (blocks * (NB / CW)), blk = g / (NB / CW) % blocks, c0 = g % (NB / CW) * CW;
    const int k0 = blk * NB, kb = min(NB, n - k0);
    const double2* D = M + (size_t)k0 * n + k0;
    double2 x[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q) x[q] = make_double2(lane == c0 + q && c0 + q < kb ? 1.0 : 0.0, 0.0);
    if (type == 0) {
      for (int t = c0; t < kb - 1; ++t) {
        const double2 d = lane > t && lane < kb ? D[(size_t)t * n + lane] : make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < CW; ++q) cfms(x[q], d, shfl2(x[q], t));
      }
    } else {
      const double2 rd = lane < kb ? crecip(D[(size_t)lane * n + lane]) : make_double2(0.0, 0.0);
      for (int t = min(c0 + CW, kb) - 1; t >= 0; --t) {
        const double2 d = lane < t ? D[(size_t)t * n + lane] : make_double2(0.0, 0.0);
#pragma unroll
        for (int q = 0; q < CW; ++q) {
          if (lane == t) x[q] = cmul(x[q], rd);
          cfms(x[q], d, shfl2(x[q], t));
        }
      }
    }
    double2* out = dinv + (size_t)(type * blocks + blk) * NB * NB;
#pragma unroll
    for (int q = 0; q < CW; ++q) out[(c0 + q) * NB + lane] = x[q];
  }
}

// out = A^{-1} (scale * in) with A = M's triangle, or its conjugate transpose (HERM), in the
// order of the blocks that FORWARD gives. dinv: that triangle's inverse diagonal blocks.
// size divides 32. Every thread of the cluster; in and out are not the same.
template <bool HERM, bool FORWARD>
__device__ void cluster_solve(const double2* M, int n, const double2* dinv, const double2* in, double scale,
                              double2* out, double2* acc, VerifySmem& sm, int rank, int size) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int blocks = (n + NB - 1) / NB, cw = NB / size, t0 = rank * cw;
  double2* mine = acc + (size_t)rank * n;
  double2* part = sm.lu.Us;  // [warp][row]
  const double2 zero = make_double2(0.0, 0.0);
  const auto at = [&](int i, int t) {  // A[i, t]
    return HERM ? cconj(M[(size_t)i * n + t]) : M[(size_t)t * n + i];
  };
  for (int i = tid; i < n; i += THREADS) mine[i] = zero;
  constexpr int G = 8;  // columns whose entries are in flight
  for (int step = 0; step < blocks; ++step) {
    const int blk = FORWARD ? step : blocks - 1 - step;
    const int k0 = blk * NB, kb = min(NB, n - k0);
    // what does not depend on the block's unknowns is loaded before the barrier
    const double2* Dk = dinv + (size_t)blk * NB * NB;
    double2 d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = 4 * wid + u;
      d[u] = HERM ? cconj(Dk[lane * NB + t]) : Dk[t * NB + lane];
    }
    // this thread's rows: 32-row chunks wid, wid + 8, ... among those still to be solved
    const int first = FORWARD ? blk + 1 : 0, last = FORWARD ? blocks : blk;
    int chunk = first + ((wid - first) & 7);
    int i = chunk * NB + lane;
    bool in_rows = chunk < last && i < n;
    double2 m[G], a = in_rows ? mine[i] : zero;
#pragma unroll
    for (int u = 0; u < G; ++u) m[u] = in_rows && u < cw && t0 + u < kb ? at(i, k0 + t0 + u) : zero;
    cluster_sync();
    // this warp's four entries of the block's right-hand side: eight lanes each
    const int tv = 4 * wid + (lane >> 3), r = lane & 7;
    double2 v = zero;
    if (tv < kb) {
      if (r < size) {
        const double2 s = acc[(size_t)r * n + k0 + tv];
        v = make_double2(-s.x, -s.y);
      }
      if (r == 0) v = cadd(v, cscale(in[k0 + tv], scale));
    }
    for (int o = size >> 1; o > 0; o >>= 1) {
      v.x += __shfl_down_sync(0xffffffffu, v.x, o);
      v.y += __shfl_down_sync(0xffffffffu, v.y, o);
    }
    double2 y = zero;
#pragma unroll
    for (int u = 0; u < 4; ++u) cfma(y, d[u], shfl2(v, 8 * u));
    part[wid * NB + lane] = y;
    __syncthreads();
    // y_t of this CTA's columns, in every warp: four lanes a column, eight columns at a time
    for (int g = 0; g < cw; g += G) {
      const int t = t0 + g + (lane >> 2), q = lane & 3;
      y = g + (lane >> 2) < cw ? cadd(part[q * NB + t], part[(q + 4) * NB + t]) : zero;
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        y.x += __shfl_xor_sync(0xffffffffu, y.x, o);
        y.y += __shfl_xor_sync(0xffffffffu, y.y, o);
      }
      if (wid == 0 && q == 0 && g + (lane >> 2) < cw && t < kb) out[k0 + t] = y;
      double2 yt[G];
#pragma unroll
      for (int u = 0; u < G; ++u) yt[u] = shfl2(y, 4 * u);
      for (int c = chunk; c < last; c += THREADS / 32) {
        if (c != chunk || g != 0) {
          i = c * NB + lane;
          in_rows = i < n;
          a = in_rows ? mine[i] : zero;
#pragma unroll
          for (int u = 0; u < G; ++u)
            m[u] = in_rows && g + u < cw && t0 + g + u < kb ? at(i, k0 + t0 + g + u) : zero;
        }
#pragma unroll
        for (int u = 0; u < G; ++u)
          if (u < cw) cfma(a, m[u], yt[u]);
        if (in_rows) mine[i] = a;
      }
    }
  }
  cluster_sync();
}

__device__ double vec_norm(const double2* x, int n, VerifySmem& sm) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += THREADS) s += cabs2(x[i]);
  return sqrt(block_sum(s, sm.red));
}

template <bool BIE>
__global__ void __launch_bounds__(THREADS, 2) k_verify_fp64(ValueArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  VerifySmem& sm = *reinterpret_cast<VerifySmem*>(smem_raw);
  const int tid = threadIdx.x;
  const int size = a.cluster, rank = cluster_rank(), slot = blockIdx.x / size;
  double2* M = a.work + (size_t)slot * a.max_n * a.max_n;
  int* piv = a.piv + (size_t)slot * a.max_n;
  double2* y = a.vec + (size_t)slot * verify_vec_len(a.max_n);

  for (int it = slot; it < a.m; it += gridDim.x / size) {
    load_problem(&sm.P, a.probs + a.prob_of[it]);
    __syncthreads();
    const ProblemDev& P = sm.P;
    const int n = P.n;
    const size_t nn = (size_t)n * n;
    double2 *x = y + n, *acc = x + n, *dinv = acc + (size_t)size * n;
    double2* dinvU = dinv + (size_t)(n + NB - 1) / NB * NB * NB;
    const double2 lam = a.lam[it];
    if (tid < P.K) sm.lu.fz[tid] = eval_f(P.term[tid], lam);
    if (BIE && tid == 0) sm.wave = bie::wave_of(lam);
    __syncthreads();
    if (BIE && P.bie) {
      for (size_t e = (size_t)rank * THREADS + tid; e < nn; e += size * THREADS) M[e] = make_double2(0.0, 0.0);
      cluster_sync();
      add_layer(P.bie, n, layer_coefficient(P), sm.wave, rank * THREADS + tid, size * THREADS,
                [&](int i, int j, double2 v) { M[(size_t)j * n + i] = v; });
      cluster_sync();
    }
    for (int col = rank; col < n; col += size) {
      for (int row = tid; row < n; row += THREADS) {
        const size_t e = (size_t)col * n + row;
        double2 v = BIE && P.bie ? M[e] : make_double2(0.0, 0.0);
        for (int k = 0; k < P.K; ++k) {
          const TermDesc& t = P.term[k];
          if (t.dense) cfma(v, sm.lu.fz[k], P.A[(size_t)t.mat_index * nn + e]);
          else if (row == col && t.kind != PMCIM_F_HELMHOLTZ_DLP) cfma(v, sm.lu.fz[k], t.id);
        }
        M[e] = v;
      }
    }
    cluster_sync();
    double fro = 0.0;
    if (rank == 0) {
      for (size_t e = tid; e < nn; e += THREADS) fro += cabs2(M[e]);
      fro = sqrt(block_sum(fro, sm.red));
    }
    const int info = cluster_lu(M, n, n, piv, reinterpret_cast<int*>(dinvU + (size_t)(n + NB - 1) / NB * NB * NB),
                                sm.lu, sm.swaps, rank, size);

    // Inverse iteration on T^H T; T = P^T L U, and as w = T^{-H} x is only needed as P w, the
    // interchanges drop out. Every CTA forms the norms, from the same numbers in the same order.
    double smin = 0.0, scale = 0.0;
    if (info == 0) {
      invert_diagonals(M, n, dinv, rank, size);
      // deterministic start vector
      if (rank == 0)
        for (int i = tid; i < n; i += THREADS) x[i] = make_double2(1.0 + 0.5 * sin(0.7 * i), cos(1.3 * i));
      cluster_sync();
      scale = 1.0 / vec_norm(x, n, sm);
      double rho_prev = 0.0, rho = 0.0;
      for (int iter = 0; iter < 30; ++iter) {
        cluster_solve<true, true>(M, n, dinvU, x, scale, y, acc, sm, rank, size);   // U^H
        cluster_solve<true, false>(M, n, dinv, y, 1.0, x, acc, sm, rank, size);     // L^H: P w
        rho = vec_norm(x, n, sm);
        cluster_solve<false, true>(M, n, dinv, x, 1.0, y, acc, sm, rank, size);     // L
        cluster_solve<false, false>(M, n, dinvU, y, 1.0, x, acc, sm, rank, size);   // U: T^{-1} w
        scale = 1.0 / vec_norm(x, n, sm);
        if (iter > 0 && fabs(rho - rho_prev) <= 1e-12 * rho) break;
        rho_prev = rho;
      }
      smin = 1.0 / rho;
    }
    if (rank != 0) {
      cluster_sync();  // the first CTA has done with the slot (below)
      continue;
    }
    if (tid == 0) {
      a.sigma[it] = smin;
      double thr = a.tol_verify * fmax(1.0, fro / sqrt((double)n));
      a.accept[it] = (smin <= thr) ? 1 : 0;
    }
    if (a.vec_out)  // the inverse iteration's last unit vector (zero when the LU met an exact zero pivot)
      for (int i = tid; i < n; i += THREADS)
        a.vec_out[(size_t)it * a.max_n + i] = info == 0 ? cscale(x[i], scale) : make_double2(0.0, 0.0);
    cluster_sync();
  }
}

}  // namespace

int factor_slots_fp64(int n, int l) {
  (void)n;
  (void)l;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return 2 * (sms > 0 ? sms : 1);
}

cudaError_t prepare_factor_fp64() {
  const void* fns[4] = {(const void*)k_factor_solve_fp64<4, false>, (const void*)k_factor_solve_fp64<2, false>,
                        (const void*)k_factor_solve_fp64<4, true>, (const void*)k_factor_solve_fp64<2, true>};
  for (const void* f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NodeSmem));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Launch only; prepare_factor_fp64() must have set the shared-memory limit (it
// is not called here so that the launch can be captured into a graph).
cudaError_t launch_factor_solve_fp64(const NodeArgs& a, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  const size_t smem = sizeof(NodeSmem);
  int grid = a.slots < a.n_items ? a.slots : a.n_items;
  if (a.bie) {
    if (a.fp64_tile == 32) k_factor_solve_fp64<2, true><<<grid, THREADS, smem, s>>>(a);
    else k_factor_solve_fp64<4, true><<<grid, THREADS, smem, s>>>(a);
  } else {
    if (a.fp64_tile == 32) k_factor_solve_fp64<2, false><<<grid, THREADS, smem, s>>>(a);
    else k_factor_solve_fp64<4, false><<<grid, THREADS, smem, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t launch_verify_fp64(const ValueArgs& a, cudaStream_t s) {
  if (a.m <= 0) return cudaSuccess;
  const size_t smem = sizeof(VerifySmem);
  const void* fn = a.bie ? (const void*)k_verify_fp64<true> : (const void*)k_verify_fp64<false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int clusters = a.slots < a.m ? a.slots : a.m;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)a.cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * a.cluster));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  e = a.bie ? cudaLaunchKernelEx(&cfg, k_verify_fp64<true>, a) : cudaLaunchKernelEx(&cfg, k_verify_fp64<false>, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// ===========================================================================
// Node solves without device allocation.
//
// Some callers cannot allocate device memory while they run: a host
// application that owns every byte of device memory through its own pool, or a
// latency-bound service loop that must not stall on the device-wide
// synchronisation that cudaFree implies. For them this entry point solves
// T(z_j) X_j = V at caller-given points with all inputs and outputs in caller
// buffers and the factorisation workspace in a fixed array compiled into the
// library. It makes no allocation of any kind.
//
// The array below is held by every GPU that loads the library until the
// process exits. It is shared by all calls and keeps the last call's contents;
// nothing in it needs clearing, because the kernel writes every workspace
// element (assembled matrix, probe columns, pivots) before it reads it. Calls
// that overlap on the GPU (two streams, two threads) race on the array.
// ===========================================================================
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(32) << 20;  // 32 MiB
static __device__ __align__(256) double2 g_noalloc_scratch[kNoAllocScratchBytes / sizeof(double2)];

struct PointArgs {
  ProblemDesc prob;
  const double2* A;
  const double2* V;
  int l;
  const double2* z;   // m points
  int m;
  double2* X;         // m * n * l
  int32_t* info;      // m, may be NULL
  double2* work;      // slots * n * (n + l), inside g_noalloc_scratch
  int32_t* piv;       // slots * n, inside g_noalloc_scratch
};

// Same per-node work as k_factor_solve_fp64, at an explicit point z_j.
__global__ void __launch_bounds__(THREADS, 2) k_factor_solve_points_fp64(PointArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LuSmem& sm = *reinterpret_cast<LuSmem*>(smem_raw);
  const int tid = threadIdx.x;
  const ProblemDesc& P = a.prob;
  const int n = P.n, l = a.l, ncols = n + l;
  double2* M = a.work + (size_t)blockIdx.x * n * ncols;
  int* piv = a.piv + (size_t)blockIdx.x * n;
  for (int node = blockIdx.x; node < a.m; node += gridDim.x) {
    const double2 z = a.z[node];
    if (tid < P.K) sm.fz[tid] = eval_f(P.term[tid], z);
    __syncthreads();
    const size_t nn = (size_t)n * n;
    // the flattened element index keeps every thread busy for any n
    for (size_t e = tid; e < nn; e += THREADS) {
      const size_t row = e % n, col = e / n;
      double2 v = make_double2(0.0, 0.0);
      for (int k = 0; k < P.K; ++k) {
        const TermDesc& t = P.term[k];
        if (t.dense) cfma(v, sm.fz[k], a.A[(size_t)t.mat_index * nn + e]);
        else if (row == col) cfma(v, sm.fz[k], t.id);
      }
      M[e] = v;
    }
    for (size_t e = tid; e < (size_t)n * l; e += THREADS) M[nn + e] = a.V[e];
    __syncthreads();
    const int info = cta_lu(M, n, ncols, piv, sm);
    cta_back_subst(M, n, l, sm);
    double2* Xo = a.X + (size_t)node * n * l;
    for (size_t e = tid; e < (size_t)n * l; e += THREADS) Xo[e] = M[nn + e];
    if (tid == 0 && a.info) a.info[node] = info;
    __syncthreads();
  }
}

}  // namespace

extern "C" int pmcim_solve_points_noalloc(int32_t n, int32_t K, const pmcim_fterm* f, const uint8_t* dense,
                                          const double* A, int32_t m, const double* z, int32_t l,
                                          const double* V, double* X, int32_t* info, void* cuda_stream) {
  if (n < 1 || K < 1 || K > PMCIM_MAX_TERMS || l < 1 || l > PMCIM_MAX_L || m < 0) return PMCIM_EINVAL;
  if (!f || !dense || !V || (m > 0 && (!z || !X))) return PMCIM_EINVAL;
  // the workspace of one CTA slot must fit the fixed array
  const size_t slot_bytes = (size_t)n * (n + l) * sizeof(double2) + (size_t)n * sizeof(int32_t);
  if (slot_bytes > kNoAllocScratchBytes) return PMCIM_ENOTSUP;
  ProblemDesc desc{};
  desc.n = n;
  desc.K = K;
  int nd = 0;
  for (int k = 0; k < K; ++k) {
    if (f[k].kind != PMCIM_F_MONOMIAL && f[k].kind != PMCIM_F_EXP_NEG) return PMCIM_EINVAL;
    if (f[k].kind == PMCIM_F_MONOMIAL && (f[k].degree < 0 || f[k].degree > 16)) return PMCIM_EINVAL;
    TermDesc& t = desc.term[k];
    t.kind = f[k].kind;
    t.degree = f[k].degree;
    t.tau = f[k].tau;
    t.id = make_double2(f[k].id_re, f[k].id_im);
    t.dense = dense[k] ? 1 : 0;
    t.mat_index = dense[k] ? nd++ : -1;
  }
  desc.n_dense = nd;
  if (nd > 0 && !A) return PMCIM_EINVAL;
  if (m == 0) return PMCIM_OK;

  // The device address of the array, looked up on every call with the calling
  // thread's device current. The lookup allocates nothing; it is not cached,
  // because a context torn down and created again (cudaDeviceReset by the host
  // application) can place the array at a new address.
  void* base = nullptr;
  if (cudaGetSymbolAddress(&base, g_noalloc_scratch) != cudaSuccess || !base) return PMCIM_ECUDA;
  int slots = factor_slots_fp64(n, l);
  const size_t fit = kNoAllocScratchBytes / slot_bytes;
  if ((size_t)slots > fit) slots = (int)fit;
  if (slots > m) slots = m;

  PointArgs a;
  a.prob = desc;
  a.A = reinterpret_cast<const double2*>(A);
  a.V = reinterpret_cast<const double2*>(V);
  a.l = l;
  a.z = reinterpret_cast<const double2*>(z);
  a.m = m;
  a.X = reinterpret_cast<double2*>(X);
  a.info = info;
  a.work = reinterpret_cast<double2*>(base);
  a.piv = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(base) + (size_t)slots * n * (n + l) * sizeof(double2));
  const size_t smem = sizeof(LuSmem);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (cudaFuncSetAttribute(k_factor_solve_points_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return PMCIM_ECUDA;
  k_factor_solve_points_fp64<<<slots, THREADS, smem, s>>>(a);
  if (cudaGetLastError() != cudaSuccess) return PMCIM_ECUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return PMCIM_ECUDA;
  return PMCIM_OK;
}
