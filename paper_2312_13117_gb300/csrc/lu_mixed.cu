// Precision form of the node solves: FP32 LU with FP64 iterative refinement.
//
// The method's cost is the linear solve at every quadrature node (Eq. 2.4;
// Sec. 2.1 cost remark). On GB300 the FP32 pipe issues 64 times as many FMAs
// per clock as the FP64 pipe, so the O(n^3) factorisation runs in FP32 and
// FP64 is kept for what needs it: the residual R = V - T(z_j) X, formed from
// the FP64 coefficients A_k, and the accumulated solution X.
//
// Per node:
//   1. assemble T(z_j), rounded to complex64, append V;
//   2. FP32 blocked LU with partial pivoting (also eliminates V), back
//      substitution -> X_0 (promoted to FP64);
//   3. sweeps s = 1..max: R = V - T(z_j) X in FP64; delta = LU^-1 (R / |R|max)
//      in FP32, scaled back; X += delta. Stop when the estimated remaining
//      error |delta_s|^2 / |delta_{s-1}| (|delta_0| = |X_0|) is below
//      tol_ir |X| (max norms);
//   4. no convergence within max sweeps (or growth) -> the node is solved
//      again by the FP64 LU and flagged.
//
// A launch's nodes go through these steps together, one kernel per step, each
// node's factors staying in a slot of its own in device memory:
//   k_mixed_factor    steps 1-2 up to the triangular factors, two CTAs per SM;
//   k_mixed_solve     the back substitution, and each sweep's correction;
//   k_oz_digits,      (oz_refine.cu) the residuals of all active nodes as one
//   k_oz_residual     product with the coefficients, which all nodes of a problem
//                     share: the coefficient digits are read once for 32 solution
//                     columns of any nodes;
//   k_mixed_fallback  step 4.
// The kernels of a sweep read the list of nodes that still refine, which the sweep
// before appended to; with none left they return at once. Every step is bound by
// latency when one node has an SM to itself (block barriers, global round trips),
// so what counts is how many nodes an SM works on at a time; in one kernel per node
// the residual's tensor memory and operand stages allowed one. The trailing updates
// run on the FMA pipes, or, for regions marked lu_tc, as complex products on the
// tensor cores: 3xTF32 (tc_update.cuh) or BF16 3M (tc_update_bf16.cuh).
// node_info: bits 0-23 = 0 or 1 + first zero-pivot column, bits 24-28 = sweeps
// run, bit 29 = a tensor-core wait ran out, bit 30 = FP64 fallback.
#include <algorithm>

#include "ozaki.cuh"
#include "tc_update_bf16.cuh"
#include "lu32.cuh"
#include "cluster_lu.cuh"

namespace {

using namespace lucore;

// Residual tiles: 128 rows x 16 columns per pass, depth 16; thread (tx, ty) owns
// rows tx + 64 i (i < 2) and columns ty + 4 q (q < 4) of the tile. The FP64
// pipe issues so slowly that shared-memory traffic is no constraint here; the
// small register block leaves room for the rest of the refinement loop.
constexpr int RT_ROWS = 128;
constexpr int RT_COLS = 16;
constexpr int RT_K = 16;
constexpr int RT_RI = RT_ROWS / 64;  // rows per thread
static_assert(RT_K * RT_COLS == THREADS, "one X-slice element per thread");
static_assert((RT_K * RT_ROWS) % THREADS == 0 && THREADS % RT_ROWS == 0, "tile copy mapping");

struct ResSmem {
  double2 As[2][RT_K * RT_ROWS];  // A_k tiles [kk][row], double-buffered
  double2 Xs[RT_K * RT_COLS];     // f_k X tile [kk][col]
};

__device__ __forceinline__ void cp_async_16(void* dst, const void* src, bool ok) {
  // 16 bytes global -> shared; zero-filled (nothing read) when !ok
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// wait until at most the most recent group is still in flight
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Issue the copies of A_k rows r0.., columns k0..k0+RT_K-1 into dst [kk][row];
// thread (pr, pk) copies rows pr of columns pk + (THREADS / RT_ROWS) u. Out of
// range elements are zero-filled from a valid address.
__device__ __forceinline__ void res_tile_async(double2* dst, const double2* __restrict__ Ak, int n, int r0, int k0,
                                               int pr, int pk) {
#pragma unroll
  for (int u = 0; u < RT_K * RT_ROWS / THREADS; ++u) {
    const int kk = pk + (THREADS / RT_ROWS) * u;
    const bool ok = r0 + pr < n && k0 + kk < n;
    cp_async_16(dst + kk * RT_ROWS + pr, ok ? Ak + (size_t)(k0 + kk) * n + r0 + pr : Ak, ok);
  }
}

// A CTA's node context.
struct NodeCtx {
  ProblemDev P;
  double2 fz[PMCIM_MAX_TERMS];
  float2 fz32[PMCIM_MAX_TERMS];  // f_k(z) rounded to complex64
  double2 fid;                   // sum over identity terms of f_k(z) id_k
  float2 fid32;
  double red[THREADS / 32];
  int item;
};

struct FactorSmem {
  NodeCtx c;
  uint64_t mbar_tc[2];    // tensor-core completion, one per accumulator
  uint32_t tmem_base;     // TMEM_FACTOR columns
  int tc_bad;             // a tensor-core wait ran out: FMA pipes from then on
  // last: the operand stage of the trailing update starts at lu32.Ls and runs over the
  // end of the struct
  LuSmemT<float2> lu32;
};
constexpr size_t kFactorHead = offsetof(FactorSmem, lu32) + offsetof(LuSmemT<float2>, Ls);

// Bytes of the scratch that starts at lu32.Ls: the operand stage of the tensor-core
// updates, or else the FMA pipes' tiles and the largest panel's scratch.
inline size_t factor_scratch_bytes(int max_n, bool tc) {
  if (tc) return tcu::STAGE_BYTES;
  size_t b = sizeof(LuSmemT<float2>) - offsetof(LuSmemT<float2>, Ls);
  for (int rows : {max_n, 256, 512, 1024, 2048})
    if (rows <= max_n && rows <= lu32::ROWS_MAX) b = std::max(b, lu32::panel_scratch_bytes(rows));
  return (b + 127) & ~size_t(127);
}

template <bool RES64>
struct SolveSmem {
  union {
    lu32::SolveSmem32 s;    // triangular solves
    ResSmem res;            // residual tiles on the FP64 pipe
  };
  NodeCtx c;
};
template <>
struct SolveSmem<false> {
  lu32::SolveSmem32 s;
  NodeCtx c;
};
// The right-hand sides of a node stay in shared memory up to this size, behind SolveSmem
// (three CTAs per SM).
constexpr size_t kSolveYBytes = 46 * 1024;

struct FallbackSmem {
  LuSmemT<double2> lu64;
  Interchanges swaps;
  NodeCtx c;
};

// Phase clock: thread 0 adds the cycles since the last mark to counter p.
struct PhaseClock {
  unsigned long long* c;
  long long t;
  __device__ explicit PhaseClock(unsigned long long* base) : c(base), t(0) { t = (long long)clock64(); }
  __device__ void mark(int p) {
    if (c && gtid() == 0) {
      const long long u = (long long)clock64();
      c[p] += (unsigned long long)(u - t);
      t = u;
    }
  }
  // the CTA's lifetime since t0 (global_ns)
  __device__ void wall(unsigned long long t0) {
    if (c && gtid() == 0) c[PH_CTA_WALL_NS] += global_ns() - t0;
  }
};

// The FP32 blocked LU: register panels (lu32.cuh; columns of more rows than they hold in
// global memory), the trailing updates on the tensor cores (tc: 1 = 3xTF32, 2 = BF16 3M; while
// no wait has run out) or on the FMA pipes (0). Row interchanges in LINPACK's order (none on
// the L columns left of a panel); each panel's permutation goes to lists for the forward
// solves.
__device__ int cta_lu32(float2* __restrict__ M, int n, int ncols, int* __restrict__ piv, int* __restrict__ lists,
                        LuSmemT<float2>& sm, tcu::Ctx& cx, int tc, PhaseClock& pc) {
  if (gtid() == 0) sm.info_sh = 0;
  gsync();
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    const int kend = k0 + kb, rows = n - k0;
    int* list = lists + (size_t)(k0 / NB) * SWAP_LIST_INTS;
    if (rows <= lu32::ROWS_MAX) {
      const int r = lu32::panel_r(rows);
      if (r == 1) lu32::panel<1>(M, n, k0, kb, piv, list, cx.stage, &sm.info_sh);
      else if (r == 2) lu32::panel<2>(M, n, k0, kb, piv, list, cx.stage, &sm.info_sh);
      else if (r == 4) lu32::panel<4>(M, n, k0, kb, piv, list, cx.stage, &sm.info_sh);
      else lu32::panel<8>(M, n, k0, kb, piv, list, cx.stage, &sm.info_sh);
      pc.mark(PH_PANEL);
      if (kend >= ncols) continue;
      lu32::swap_trsm(M, n, ncols, k0, kb, lu32::panel_smem(cx.stage, rows), reinterpret_cast<float2*>(cx.stage));
    } else {
      cta_lu_panel(M, n, ncols, k0, kb, piv, sm, k0);
      if (gtid() == 0) compose_swaps(piv, k0, kend, list);
      gsync();
      pc.mark(PH_PANEL);
      if (kend >= ncols) continue;
      cta_lu_trsm(M, n, ncols, k0, kb, sm);
    }
    pc.mark(PH_TRSM);
    if (kend >= n) continue;
    if (tc == 2 && !*cx.bad) tcb::update(M, n, ncols, k0, kb, cx);
    else if (tc == 1 && !*cx.bad) tcu::update(M, n, ncols, k0, kb, cx);
    else cta_lu_update_simt(M, n, ncols, k0, kb, sm);
    pc.mark(PH_UPDATE);
  }
  gsync();
  return sm.info_sh;
}

__device__ double block_max(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  gsync();
  if ((gtid() & 31) == 0) red[gtid() >> 5] = v;
  gsync();
  double t = 0.0;
  for (int k = 0; k < THREADS / 32; ++k) t = fmax(t, red[k]);
  return t;
}

// R = V - sum_k f_k(z) A_k X  (FP64), R and X column-major n x l.
// R = V - id X - f_M M X in FP64 (the refinement residual), M an n x n column-major
// matrix (NULL: none). With two or more dense terms M is T(z_j) itself, assembled
// in FP64 once per node by the factor step (f_M = 1, id = 0), so that a sweep
// multiplies X by one matrix instead of one per term; with a single dense term M
// is that term's A_k.
__device__ void residual_fp64(const double2* __restrict__ X, double2* __restrict__ R, const NodeCtx& cx,
                              ResSmem& rs, const double2* __restrict__ M, double2 fM, double2 id) {
  const ProblemDev& P = cx.P;
  const int n = P.n, l = P.l;
  const int tid = gtid();
  const int tx = tid & 63, ty = tid >> 6;
  const int pr = tid % RT_ROWS, pk = tid / RT_ROWS;  // tile element (row, k) this thread fetches first
  const int xk = tid % RT_K, xc = tid / RT_K;        // X slice element (k, column)
  for (int c0 = 0; c0 < l; c0 += RT_COLS) {
    for (int r0 = 0; r0 < n; r0 += RT_ROWS) {
      double2 acc[RT_RI][4];
#pragma unroll
      for (int i = 0; i < RT_RI; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int row = r0 + tx + 64 * i, c = c0 + ty + 4 * q;
          double2 v = make_double2(0.0, 0.0);
          if (row < n && c < l) {
            v = P.V[(size_t)c * n + row];
            cfms(v, id, X[(size_t)c * n + row]);
          }
          acc[i][q] = v;
        }
      if (M) {
        // tiles of M stream through two shared buffers with cp.async: the copy
        // of the next tile is in flight while the current one is multiplied
        const double2* xcol = X + (size_t)(c0 + xc) * n;
        const bool xc_ok = c0 + xc < l;
        double2 px = (xk < n && xc_ok) ? xcol[xk] : make_double2(0.0, 0.0);
        gsync();  // both buffers are free
        res_tile_async(rs.As[0], M, n, r0, 0, pr, pk);
        cp_async_commit();
        int b = 0;
        for (int k0 = 0; k0 < n; k0 += RT_K, b ^= 1) {
          gsync();  // the previous step's multiplications are done
          rs.Xs[xk * RT_COLS + xc] = cmul(fM, px);
          if (k0 + RT_K < n) {
            res_tile_async(rs.As[b ^ 1], M, n, r0, k0 + RT_K, pr, pk);
            px = (k0 + RT_K + xk < n && xc_ok) ? xcol[k0 + RT_K + xk] : make_double2(0.0, 0.0);
          }
          cp_async_commit();
          cp_async_wait_prior();  // this tile's copies have landed (the next may be in flight)
          gsync();
          const double2* As = rs.As[b];
#pragma unroll 4
          for (int kk = 0; kk < RT_K; ++kk) {
            double2 av[RT_RI], xv[4];
#pragma unroll
            for (int i = 0; i < RT_RI; ++i) av[i] = As[kk * RT_ROWS + tx + 64 * i];
#pragma unroll
            for (int q = 0; q < 4; ++q) xv[q] = rs.Xs[kk * RT_COLS + ty + 4 * q];
#pragma unroll
            for (int i = 0; i < RT_RI; ++i)
#pragma unroll
              for (int q = 0; q < 4; ++q) cfms(acc[i][q], av[i], xv[q]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < RT_RI; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int row = r0 + tx + 64 * i, c = c0 + ty + 4 * q;
          if (row < n && c < l) R[(size_t)c * n + row] = acc[i][q];
        }
    }
  }
  cp_async_wait_all();
  gsync();
}

// The same for one column (l = 1), as a matrix-vector product: the tiled form
// above would multiply RT_COLS - 1 zero columns as well. Each thread owns four
// rows of a 4 x THREADS row block and streams the columns of M (coalesced over
// rows, several columns in flight); f_M x is staged in shared memory.
__device__ void residual_fp64_col(const double2* __restrict__ X, double2* __restrict__ R, const NodeCtx& cx,
                                  ResSmem& rs, const double2* __restrict__ M, double2 fM, double2 id) {
  const ProblemDev& P = cx.P;
  const int n = P.n;
  const int tid = gtid();
  constexpr int XCH = 2 * RT_K * RT_ROWS;  // f_M x entries per shared-memory chunk
  double2* xs = &rs.As[0][0];
  for (int r0 = 0; r0 < n; r0 += 4 * THREADS) {
    double2 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = r0 + tid + i * THREADS;
      double2 v = make_double2(0.0, 0.0);
      if (row < n) {
        v = P.V[row];
        cfms(v, id, X[row]);
      }
      acc[i] = v;
    }
    if (M) {
      for (int c0 = 0; c0 < n; c0 += XCH) {
        const int cn = min(XCH, n - c0);
        gsync();  // the previous chunk is no longer read
        for (int e = tid; e < cn; e += THREADS) xs[e] = cmul(fM, X[c0 + e]);
        gsync();
#pragma unroll 4
        for (int c = 0; c < cn; ++c) {
          const double2 xv = xs[c];
          const double2* __restrict__ mc = M + (size_t)(c0 + c) * n;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = r0 + tid + i * THREADS;
            if (row < n) cfms(acc[i], mc[row], xv);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = r0 + tid + i * THREADS;
      if (row < n) R[row] = acc[i];
    }
  }
  gsync();
}

// T(z_j) in FP64 into T (n x n, column-major), the matrix of the refinement
// residuals, and rounded to complex64 into M32 (leading dimension n), the FP32
// LU's matrix: the dense terms in one pass over the elements, four elements per
// thread at a time so that their coefficient loads overlap, then the identity
// terms on the diagonal. herm: T(z_j)^H instead (the coefficients read transposed,
// the sum conjugated; used by the certificates' bordered steps).
__device__ void assemble_fp64(const NodeCtx& cx, double2* __restrict__ T, float2* __restrict__ M32, bool herm) {
  const ProblemDev& P = cx.P;
  const int n = P.n;
  const size_t nn = (size_t)n * n;
  for (size_t e0 = gtid(); e0 < nn; e0 += 4 * (size_t)THREADS) {
    double2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = make_double2(0.0, 0.0);
    for (int k = 0; k < P.K; ++k) {
      const TermDesc& t = P.term[k];
      if (!t.dense) continue;
      const double2* __restrict__ A = P.A + (size_t)t.mat_index * nn;
      double2 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const size_t e = e0 + (size_t)u * THREADS;
        const size_t src = herm ? (e % n) * n + e / n : e;
        a[u] = e < nn ? A[src] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) cfma(v[u], cx.fz[k], a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t e = e0 + (size_t)u * THREADS;
      if (e < nn) {
        if (herm) v[u].y = -v[u].y;
        T[e] = v[u];
        M32[e] = make_float2((float)v[u].x, (float)v[u].y);
      }
    }
  }
  gsync();
  double2 id = cx.fid;
  if (herm) id.y = -id.y;
  for (int i = gtid(); i < n; i += THREADS) {
    const size_t e = (size_t)i * n + i;
    const double2 t = cadd(T[e], id);
    T[e] = t;
    M32[e] = make_float2((float)t.x, (float)t.y);
  }
  gsync();
}

// The FP32 LU's matrix of a boundary-integral node from the FP64 T(z_j) that
// k_bie_assemble left: the matrix, or the first column of a circulant one, rounded once in
// stage (n values of shared memory) where it fits.
__device__ void round_bie(const double2* __restrict__ T, float2* __restrict__ M32, int n, bool column_only,
                          float2* __restrict__ stage, int stage_elems) {
  const size_t nn = (size_t)n * n;
  if (!column_only) {
#pragma unroll 4
    for (size_t e = gtid(); e < nn; e += THREADS) M32[e] = make_float2((float)T[e].x, (float)T[e].y);
    return;
  }
  const bool fits = n <= stage_elems;
  if (fits)
    for (int m = gtid(); m < n; m += THREADS) stage[m] = make_float2((float)T[m].x, (float)T[m].y);
  gsync();
  const int warp = gtid() >> 5, lane = gtid() & 31;
  for (int col = warp; col < n; col += THREADS / 32)
    for (int row = lane; row < n; row += 32) {
      const int m = row >= col ? row - col : row - col + n;
      M32[(size_t)col * n + row] = fits ? stage[m] : make_float2((float)T[m].x, (float)T[m].y);
    }
}

// T(z_j) for the FP32 LU: FP32 arithmetic on the complex64 copy of the A_k
// (the LU only has to approximate T(z_j) to FP32 accuracy; the refinement
// residuals use the FP64 coefficients). It keeps the factor step off the FP64
// pipe. The flattened element index with eight elements per thread in flight
// keeps the loads of each term overlapped; the identity terms are added to the
// diagonal afterwards (a test per element would cost a 64-bit division).
__device__ void assemble32(const NodeCtx& cx, float2* __restrict__ M32) {
  const ProblemDev& P = cx.P;
  const int n = P.n;
  const size_t nn = (size_t)n * n;
  constexpr int U = 8;
  const float2 fid = cx.fid32;
  for (size_t e0 = gtid(); e0 < nn; e0 += (size_t)U * THREADS) {
    float2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = make_float2(0.f, 0.f);
    for (int k = 0; k < P.K; ++k) {
      const TermDesc& t = P.term[k];
      if (!t.dense) continue;
      const float2* __restrict__ A = P.A32 + (size_t)t.mat_index * nn;
      float2 a[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const size_t e = e0 + (size_t)u * THREADS;
        a[u] = e < nn ? A[e] : make_float2(0.f, 0.f);
      }
      const float2 f = cx.fz32[k];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u].x = fmaf(f.x, a[u].x, fmaf(-f.y, a[u].y, v[u].x));
        v[u].y = fmaf(f.x, a[u].y, fmaf(f.y, a[u].x, v[u].y));
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t e = e0 + (size_t)u * THREADS;
      if (e < nn) M32[e] = v[u];
    }
  }
  if (fid.x != 0.f || fid.y != 0.f) {
    gsync();
    for (int i = gtid(); i < n; i += THREADS) {
      float2& d = M32[(size_t)i * n + i];
      d.x += fid.x;
      d.y += fid.y;
    }
  }
}

// T(z_j) in FP64 for the fallback: columns rank, rank + size, ...
__device__ void assemble(const NodeCtx& cx, double2* M64, int rank, int size) {
  const ProblemDev& P = cx.P;
  const int n = P.n;
  const size_t nn = (size_t)n * n;
  for (int col = rank; col < n; col += size) {
    for (int row = gtid(); row < n; row += THREADS) {
      const size_t e = (size_t)col * n + row;
      double2 v = make_double2(0.0, 0.0);
      for (int k = 0; k < P.K; ++k) {
        const TermDesc& t = P.term[k];
        if (t.dense) cfma(v, cx.fz[k], P.A[(size_t)t.mat_index * nn + e]);
        else if (row == col) cfma(v, cx.fz[k], t.id);
      }
      M64[e] = v;
    }
  }
}

// Node item -> problem, node point and, with FZ, the scalar functions in the CTA's context.
template <bool FZ>
__device__ void load_node(const MixedArgs& a, int q, NodeCtx& c, RegionDev& rg, NodeItem& it) {
  it = a.items[q];
  rg = a.regions[it.region];
  {
    const int* src = reinterpret_cast<const int*>(a.probs + rg.prob);
    int* dst = reinterpret_cast<int*>(&c.P);
    for (int i = gtid(); i < (int)(sizeof(ProblemDev) / sizeof(int)); i += THREADS) dst[i] = src[i];
  }
  gsync();
  if (!FZ) return;
  double2 z, w;
  node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &w);
  if (gtid() < c.P.K) {
    const double2 f = eval_f(c.P.term[gtid()], z);
    c.fz[gtid()] = f;
    c.fz32[gtid()] = make_float2((float)f.x, (float)f.y);
  }
  gsync();
  if (gtid() == 0) {
    double2 id = make_double2(0.0, 0.0);
    for (int k = 0; k < c.P.K; ++k)
      if (!c.P.term[k].dense && c.P.term[k].kind != PMCIM_F_HELMHOLTZ_DLP)
        id = cadd(id, cmul(c.fz[k], c.P.term[k].id));
    c.fid = id;
    c.fid32 = make_float2((float)id.x, (float)id.y);
  }
  gsync();
}

// The next index of a work list of `total` entries, -1 past its end or once the launch has
// failed; every thread gets it.
__device__ __forceinline__ int next_index(const MixedArgs& a, int counter, int total, NodeCtx& c) {
  gsync();  // the previous item is no longer read
  if (gtid() == 0) {
    const int k = atomicAdd(a.ctl + counter, 1);
    c.item = k < total && *reinterpret_cast<volatile int32_t*>(a.err) == 0 ? k : -1;
  }
  gsync();
  return c.item;
}

constexpr uint32_t TMEM_FACTOR = 256;  // columns per CTA, two CTAs per SM
static_assert(tcu::TMEM_COLS <= TMEM_FACTOR && 2 * tcb::ACC_COLS <= TMEM_FACTOR, "TMEM columns");

// Steps 1-2: node after node, each into its own slot.
// BIE: the instantiation for launches with a boundary-integral term (bie.cuh); the
// other leaves its code out. TC: a region of the launch updates on the tensor cores.
template <bool BIE, bool TC>
__global__ void __launch_bounds__(THREADS, 2) k_mixed_factor(MixedArgs a, int scratch_bytes) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  FactorSmem& sm = *reinterpret_cast<FactorSmem*>(smem_raw);
  const int tid = gtid();
  NodeCtx& c = sm.c;
  PhaseClock pc(a.phase ? a.phase + (size_t)blockIdx.x * PMCIM_PHASES : nullptr);
  const unsigned long long t_start = global_ns();
  if (TC && tid < 32) tcu::tmem_alloc_cols(&sm.tmem_base, TMEM_FACTOR);
  if (tid == 0) {
    tcu::mbar_init(&sm.mbar_tc[0]);
    tcu::mbar_init(&sm.mbar_tc[1]);
    sm.tc_bad = 0;
  }
  tcu::fence_async_smem();
  tcu::fence_before();
  __syncthreads();
  tcu::fence_after();
  tcu::Ctx cx{smem_raw + kFactorHead, sm.mbar_tc, TC ? sm.tmem_base : 0u, {0u, 0u}, &sm.tc_bad, a.tc_wait_cycles};
  for (;;) {
    const int q = next_index(a, MIXED_CTL_FACTOR, a.count, c);
    if (q < 0) break;
    char* slot = a.work + (size_t)q * a.slot_bytes;
    float2* M32 = reinterpret_cast<float2*>(slot);
    NodeItem it;
    RegionDev rg;
    load_node<true>(a, q, c, rg, it);
    const ProblemDev& P = c.P;
    const int n = P.n, l = P.l, ncols = n + l;
    const size_t nn = (size_t)n * n, nl = (size_t)n * l;
    pc.mark(PH_SETUP);
    // T(z_j) in FP64 for the residuals on the FP64 pipe, and rounded; T(z_j)^H likewise
    if (BIE && P.bie && !rg.herm)
      round_bie(a.t64 + (size_t)q * a.t64_stride, M32, n, mixed_column_only(a, P),
                reinterpret_cast<float2*>(cx.stage), scratch_bytes / (int)sizeof(float2));
    else if (rg.herm || (P.n_dense >= 2 && !a.oz))
      assemble_fp64(c, a.t64 + (size_t)q * a.t64_stride, M32, rg.herm != 0);
    else
      assemble32(c, M32);
    for (size_t e = tid; e < nl; e += THREADS) M32[nn + e] = make_float2((float)P.V[e].x, (float)P.V[e].y);
    gsync();
    if (rg.border > 0) {  // the bordered matrix of a certificate: column s of T(z_j) replaced
      const double2* bc = a.border + rg.v_off;
      float2* col = M32 + (size_t)(rg.border - 1) * n;
      for (int i = tid; i < n; i += THREADS) col[i] = make_float2((float)bc[i].x, (float)bc[i].y);
      gsync();
    }
    pc.mark(PH_ASSEMBLE);
    const int bad_before = sm.tc_bad;
    int* lists = reinterpret_cast<int*>(slot + mixed_lists_offset(n, l));
    int* piv = lists + (size_t)((n + NB - 1) / NB) * SWAP_LIST_INTS;
    const int info = cta_lu32(M32, n, ncols, piv, lists, sm.lu32, cx, TC ? rg.lu_tc : 0, pc);
    if (tid == 0) {
      MixedState st{};
      st.info = info;
      st.lost = sm.tc_bad != bad_before ? MIXED_LOST_LU : 0;
      // a boundary-integral node's residual takes the whole of T(z_j) as its one dense term
      st.id = BIE && P.bie ? make_double2(0.0, 0.0) : c.fid;
      a.state[q] = st;
    }
  }
  if (TC) {
    // a commit whose wait ran out may still be in flight: wait once more, with the
    // default limit whatever the update's own limit was, before the columns are given back
    if (sm.tc_bad) {
      // returns at once for a barrier with no commit outstanding
      tcu::wait_parity(&sm.mbar_tc[0], cx.phase[0] ^ 1u, tcu::WAIT_CYCLES);
      tcu::wait_parity(&sm.mbar_tc[1], cx.phase[1] ^ 1u, tcu::WAIT_CYCLES);
    }
    tcu::fence_before();
    __syncthreads();
    tcu::fence_after();
    if (tid < 32) tcu::tmem_dealloc_cols(sm.tmem_base, TMEM_FACTOR);
  }
  pc.wall(t_start);
}

// Thread 0: a finished node's info word.
__device__ __forceinline__ void finish_node(const MixedArgs& a, const RegionDev& rg, const NodeItem& it,
                                            const MixedState& st, bool ok) {
  a.node_info[rg.node_off + it.j] =
      st.info | (min(st.sweeps, 31) << 24) | (st.lost ? (1 << 29) : 0) | (ok ? 0 : (1 << 30));
}

// The back substitution (sw = 0, every node) or sweep sw's correction (the active nodes). A
// bordered node's sweeps all run in the launch of the first: they are not bounded by
// MIXED_MAX_SWEEPS, and their residuals need no other kernel.
// RES64: a node of the launch forms its residuals on the FP64 pipe.
template <bool RES64>
__global__ void __launch_bounds__(THREADS, 3) k_mixed_solve(MixedArgs a, int sw, int y_bytes) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SolveSmem<RES64>& sm = *reinterpret_cast<SolveSmem<RES64>*>(smem_raw);
  const int tid = gtid();
  NodeCtx& c = sm.c;
  const int total = sw == 0 ? a.count : a.ctl[MIXED_CTL_ACTIVE + sw];
  if (total == 0) return;
  PhaseClock pc(a.phase ? a.phase + (size_t)blockIdx.x * PMCIM_PHASES : nullptr);
  const unsigned long long t_start = global_ns();
  for (;;) {
    const int k = next_index(a, sw == 0 ? MIXED_CTL_FIRST : MIXED_CTL_SWEEP + sw, total, c);
    if (k < 0) break;
    const int q = sw == 0 ? k : a.act[(size_t)(sw & 1) * a.slots + k];
    char* slot = a.work + (size_t)q * a.slot_bytes;
    float2* M32 = reinterpret_cast<float2*>(slot);
    NodeItem it;
    RegionDev rg;
    load_node<RES64>(a, q, c, rg, it);
    const ProblemDev& P = c.P;
    const int n = P.n, l = P.l;
    const size_t nn = (size_t)n * n, nl = (size_t)n * l;
    double2* R = reinterpret_cast<double2*>(slot + mixed_residual_offset(n, l));
    const int* lists = reinterpret_cast<const int*>(slot + mixed_lists_offset(n, l));
    float2* Y = nl * sizeof(float2) <= (size_t)y_bytes ? reinterpret_cast<float2*>(smem_raw + sizeof(SolveSmem<RES64>))
                                                       : M32 + nn;
    double2* X = a.X + rg.x_off + (size_t)it.j * nl;
    MixedState st = a.state[q];
    const bool oz = mixed_node_oz(a, P, rg);
    bool ok = st.info == 0, done = false;
    if (sw == 0) {
      if (ok) {
        // X_0 = U^-1 (L^-1 P V) in FP32 (the LU eliminated V)
        double xm = 0.0;
        if (Y != M32 + nn) {
          for (size_t e = tid; e < nl; e += THREADS) Y[e] = M32[nn + e];
          gsync();
        }
        lu32::back(M32, Y, n, l, sm.s);
        for (size_t e = tid; e < nl; e += THREADS) {
          const float2 y = Y[e];
          const double2 x = make_double2((double)y.x, (double)y.y);
          X[e] = x;
          xm = fmax(xm, fmax(fabs(x.x), fabs(x.y)));
        }
        st.dprev = block_max(xm, c.red);
      }
      // max_sweeps == 0: the FP32 solve alone (a direction for a certificate), no refinement
      // and no FP64 re-solve
      done = a.max_sweeps == 0;
      pc.mark(PH_FIRST_SOLVE);
    } else {
      for (int s = sw;; ++s) {
        if (oz) {
          ok = (st.lost & MIXED_LOST_RESIDUAL) == 0;  // R is not valid where a wait ran out
        } else if (RES64) {
          // the matrix the residual multiplies: T(z_j) assembled once, or the one dense term
          const double2* M = nullptr;
          double2 fM = make_double2(1.0, 0.0), id = make_double2(0.0, 0.0);
          if (P.n_dense >= 2 || rg.herm || P.bie) {
            M = a.t64 + (size_t)q * a.t64_stride;
          } else {
            id = c.fid;
            for (int t = 0; t < P.K; ++t)
              if (P.term[t].dense) {
                M = P.A + (size_t)P.term[t].mat_index * nn;
                fM = c.fz[t];
              }
          }
          ResSmem& res = *reinterpret_cast<ResSmem*>(smem_raw);
          if (l == 1) residual_fp64_col(X, R, c, res, M, fM, id);
          else residual_fp64(X, R, c, res, M, fM, id);
        }
        if (ok && rg.border > 0) {
          // bordered system M u = b, M = T(z_j) + (c - T(z_j) e_s) e_s^T with b = -T(z_j) e_s:
          // R = b - T X - (c + b) X_s (l = 1)
          const double2 xs = X[rg.border - 1];
          const double2* bc = a.border + rg.v_off;
          for (size_t e = tid; e < nl; e += THREADS) cfms(R[e], cadd(bc[e], P.V[e]), xs);
        }
        pc.mark(PH_RESIDUAL);
        double rm = 0.0;
        if (ok) {
          for (size_t e = tid; e < nl; e += THREADS) rm = fmax(rm, fmax(fabs(R[e].x), fabs(R[e].y)));
          rm = block_max(rm, c.red);
          done = rm == 0.0;
        }
        if (ok && !done) {
          const double inv = 1.0 / rm;
          // right-hand side R / |R|max; the forward solve applies the row interchanges
          for (size_t e = tid; e < nl; e += THREADS) {
            const double2 rv = R[e];
            Y[e] = make_float2((float)(rv.x * inv), (float)(rv.y * inv));
          }
          gsync();
          lu32::forward(M32, Y, n, l, sm.s, lists);
          lu32::back(M32, Y, n, l, sm.s);
          double dm = 0.0, xmx = 0.0;
          for (size_t e = tid; e < nl; e += THREADS) {
            const float2 d = Y[e];
            double2 x = X[e];
            const double dx = (double)d.x * rm, dy = (double)d.y * rm;
            x.x += dx;
            x.y += dy;
            X[e] = x;
            dm = fmax(dm, fmax(fabs(dx), fabs(dy)));
            xmx = fmax(xmx, fmax(fabs(x.x), fabs(x.y)));
          }
          dm = block_max(dm, c.red);
          xmx = block_max(xmx, c.red);
          st.sweeps = s;
          if (!(dm < st.dprev) && s > 1) ok = false;  // no contraction
          else if (dm * dm <= a.tol_ir * xmx * st.dprev) done = true;
          else if (s >= a.max_sweeps) ok = false;
          st.dprev = dm;
        }
        pc.mark(PH_CORRECTION);
        if (done || !ok || rg.border == 0) break;
      }
    }
    const bool refine = a.max_sweeps > 0;
    if ((done || !ok) && rg.border > 0) {
      // the certificate's vector y = e_s + (u - u_s e_s): T(z_j) y = -u_s c
      gsync();
      if (tid == 0) X[rg.border - 1] = make_double2(1.0, 0.0);
    }
    if (tid == 0) {
      a.state[q] = st;
      if (!ok && refine && rg.border == 0) {
        a.fallback[atomicAdd(a.ctl + MIXED_CTL_FALLBACK_COUNT, 1)] = q;
      } else if (done || !ok) {
        finish_node(a, rg, it, st, ok);
      } else {  // active in the next sweep
        const int nx = sw + 1;
        a.act[(size_t)(nx & 1) * a.slots + atomicAdd(a.ctl + MIXED_CTL_ACTIVE + nx, 1)] = q;
        if (oz) {
          const int ncg = (l + 7) / 8;
          const int u = a.ubase[rg.prob] + atomicAdd(mixed_ucount(a, nx) + rg.prob, ncg);
          for (int g = 0; g < ncg; ++g) a.units[(size_t)(nx & 1) * a.unit_cap + u + g] = q * 8 + g;
        }
      }
    }
  }
  pc.wall(t_start);
}

// Step 4: the nodes that did not converge, by the FP64 LU. The chunk's other nodes are
// done, so the FP64 matrices take the slots' place. One such node of order 1024 is 0.36 s of an
// SM, and nothing else runs meanwhile; so as long as there are few of them (at most `few`, which
// leaves two CTAs per SM) the CTAs of a cluster share one (0.07 s), and else, where all SMs are
// busy anyway, a CTA has one of its own, without barriers across SMs. The two kernels of a chunk
// read the number of such nodes and one of them returns at once. Both round alike.
template <bool CLUSTER>
__global__ void __launch_bounds__(THREADS, 2) k_mixed_fallback(MixedArgs a, size_t bytes, int size, int few) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  FallbackSmem& sm = *reinterpret_cast<FallbackSmem*>(smem_raw);
  NodeCtx& c = sm.c;
  const int total = a.ctl[MIXED_CTL_FALLBACK_COUNT];
  if (total == 0 || (total <= few) != CLUSTER || *reinterpret_cast<volatile int32_t*>(a.err)) return;
  PhaseClock pc(a.phase ? a.phase + (size_t)blockIdx.x * PMCIM_PHASES : nullptr);
  const unsigned long long t_start = global_ns();
  const int rank = CLUSTER ? cluster_rank() : 0, slot = (int)blockIdx.x / size, slots = (int)gridDim.x / size;
  for (int it_no = slot;; it_no += slots) {
    int k = it_no;
    if (!CLUSTER) k = next_index(a, MIXED_CTL_FALLBACK, total, c);
    if (k < 0 || k >= total) break;
    const int q = a.fallback[k];
    NodeItem it;
    RegionDev rg;
    load_node<true>(a, q, c, rg, it);
    const ProblemDev& P = c.P;
    const int n = P.n, l = P.l;
    const size_t nn = (size_t)n * n, nl = (size_t)n * l;
    double2* M64 = reinterpret_cast<double2*>(a.work + (size_t)slot * bytes);
    int* piv = reinterpret_cast<int*>(M64 + nn + nl);
    double2* X = a.X + rg.x_off + (size_t)it.j * nl;
    if (P.bie) {  // T(z_j) as k_bie_assemble left it
      const double2* T64 = a.t64 + (size_t)q * a.t64_stride;
      const bool column = mixed_column_only(a, P);
      for (int col = rank; col < n; col += size)
        for (int row = gtid(); row < n; row += THREADS)
          M64[(size_t)col * n + row] =
              T64[!column ? (size_t)col * n + row : (size_t)(row >= col ? row - col : row - col + n)];
    } else {
      assemble(c, M64, rank, size);
    }
    for (size_t e = (size_t)rank * THREADS + gtid(); e < nl; e += (size_t)size * THREADS) M64[nn + e] = P.V[e];
    int info;
    if (CLUSTER) {
      cluster_sync();
      info = cluster_lu(M64, n, n + l, piv, piv + n, sm.lu64, sm.swaps, rank, size);
    } else {
      gsync();
      info = cta_lu(M64, n, n + l, piv, sm.lu64);
    }
    // each CTA its share of the columns
    const int c0 = l * rank / size, c1 = l * (rank + 1) / size;
    if (c1 > c0) cta_back_blocked(M64, n, c1 - c0, sm.lu64, c0);
    for (size_t e = (size_t)n * c0 + gtid(); e < (size_t)n * c1; e += THREADS) X[e] = M64[nn + e];
    if (gtid() == 0 && rank == 0) {
      MixedState st = a.state[q];
      st.info = info;
      finish_node(a, rg, it, st, false);
    }
    pc.mark(PH_FALLBACK);
    if (CLUSTER) cluster_sync();  // the matrix is no longer read
  }
  pc.wall(t_start);
}

}  // namespace

// Slot layout: [FP32 matrix n x (n + l)] [FP64 residual n x l] [the panels' row
// permutations, SWAP_LIST_INTS ints each] [pivots].
size_t mixed_slot_bytes(int n, int l) {
  const size_t ints = (size_t)((n + NB - 1) / NB) * SWAP_LIST_INTS + n;
  return (mixed_lists_offset(n, l) + ints * sizeof(int) + 255) & ~(size_t)255;
}
// Bytes a slot area needs at the least: one FP64 fallback.
size_t mixed_fallback_bytes(int n, int l) {
  return (((size_t)n * (n + l) * sizeof(double2) + (size_t)(n + 1) * sizeof(int)) + 255) & ~(size_t)255;
}

namespace {
const void* factor_kernel(bool bie, bool tc) {
  if (bie) return tc ? (const void*)k_mixed_factor<true, true> : (const void*)k_mixed_factor<true, false>;
  return tc ? (const void*)k_mixed_factor<false, true> : (const void*)k_mixed_factor<false, false>;
}
}  // namespace

static_assert(2 * (kFactorHead + tcu::STAGE_BYTES + 1024) <= 228 * 1024, "two CTAs per SM");
static_assert(lu32::panel_scratch_bytes(lu32::ROWS_MAX) <= tcu::STAGE_BYTES && lu32::panel_scratch_bytes(1024) <= tcu::STAGE_BYTES &&
                  lu32::panel_scratch_bytes(256) <= tcu::STAGE_BYTES && lu32::panel_scratch_bytes(512) <= tcu::STAGE_BYTES,
              "a panel fits the operand stage");
static_assert(3 * (sizeof(SolveSmem<false>) + kSolveYBytes + 1024) <= 228 * 1024, "three CTAs per SM");

cudaError_t prepare_factor_mixed() {
  for (int i = 0; i < 4; ++i) {
    cudaError_t e = cudaFuncSetAttribute(factor_kernel(i & 1, i & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kFactorHead + tcu::STAGE_BYTES));
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaFuncSetAttribute(k_mixed_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(SolveSmem<true>));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_mixed_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(sizeof(SolveSmem<false>) + kSolveYBytes));
  if (e != cudaSuccess) return e;
  for (const void* f : {(const void*)k_mixed_fallback<false>, (const void*)k_mixed_fallback<true>}) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FallbackSmem));
    if (e != cudaSuccess) return e;
  }
  return prepare_oz_refine();
}

namespace {
__global__ void k_round_c64(const double2* __restrict__ src, float2* __restrict__ dst, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = make_float2((float)src[i].x, (float)src[i].y);
}
}  // namespace

cudaError_t round_coefficients_c64(const double2* src, float2* dst, size_t count, cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const size_t blocks = (count + 255) / 256;
  k_round_c64<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(src, dst, count);
  return cudaGetLastError();
}

// One chunk's kernels in order (no synchronisation, so that they can be captured);
// prepare_factor_mixed() must have set the shared-memory limits. *launched: kernels.
cudaError_t launch_factor_solve_mixed(const MixedArgs& a, int sms, cudaStream_t s, int* launched) {
  *launched = 0;
  if (a.count <= 0) return cudaSuccess;
  const int rounds = mixed_rounds(a.max_sweeps, a.border != nullptr);
  if (rounds > MIXED_MAX_SWEEPS) return cudaErrorInvalidValue;  // (ctl has no counters for more)
  cudaError_t e = cudaMemsetAsync(a.ctl, 0, mixed_ctl_zero_ints(a.n_probs, rounds) * sizeof(int), s);
  if (e != cudaSuccess) return e;
  auto grid = [&](int per_sm) { return per_sm * sms < a.count ? per_sm * sms : a.count; };
  if (a.bie && a.t64) {
    e = launch_bie_assemble(a, sms, s, launched);
    if (e != cudaSuccess) return e;
  }
  {
    const int scratch = (int)factor_scratch_bytes(a.max_n, a.tc != 0);
    const size_t smem = kFactorHead + scratch;
    const int g = grid(2);
    if (a.bie && a.tc) k_mixed_factor<true, true><<<g, THREADS, smem, s>>>(a, scratch);
    else if (a.bie) k_mixed_factor<true, false><<<g, THREADS, smem, s>>>(a, scratch);
    else if (a.tc) k_mixed_factor<false, true><<<g, THREADS, smem, s>>>(a, scratch);
    else k_mixed_factor<false, false><<<g, THREADS, smem, s>>>(a, scratch);
    ++*launched;
  }
  for (int sw = 0; sw <= rounds; ++sw) {
    if (sw > 0 && a.oz) {
      e = launch_oz_residual(a, sw, sms, s, launched);
      if (e != cudaSuccess) return e;
    }
    // (the FP64-pipe residual's tiles leave no room for the right-hand sides)
    const size_t nl = (size_t)a.max_n * a.max_l * sizeof(float2);
    const int y = !a.res64 && nl <= kSolveYBytes ? (int)nl : 0;
    if (a.res64) k_mixed_solve<true><<<grid(3), THREADS, sizeof(SolveSmem<true>), s>>>(a, sw, 0);
    else k_mixed_solve<false><<<grid(3), THREADS, sizeof(SolveSmem<false>) + y, s>>>(a, sw, y);
    ++*launched;
  }
  if (a.max_sweeps > 0 && !a.border) {
    const size_t per = mixed_fallback_bytes(a.max_n, a.max_l);
    const size_t mats = a.work_bytes / per;
    if (mats < 1) return cudaErrorInvalidValue;
    // CTAs of a cluster: a power of two that leaves each 16 rows
    int size = 1;
    while (size < 8 && 32 * size <= a.max_n) size *= 2;
    const int few = size > 1 ? (int)std::min<size_t>(mats, (size_t)(2 * sms / size)) : 0;
    if (few > 0) {
      cudaLaunchAttribute at;
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = (unsigned)size;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(std::min(few, a.count) * size));
      cfg.blockDim = dim3(THREADS);
      cfg.dynamicSmemBytes = sizeof(FallbackSmem);
      cfg.stream = s;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      e = cudaLaunchKernelEx(&cfg, k_mixed_fallback<true>, a, per, size, few);
      if (e != cudaSuccess) return e;
      ++*launched;
    }
    if (few < a.count) {
      const size_t g = std::min(mats, (size_t)grid(2));
      k_mixed_fallback<false><<<(unsigned)g, THREADS, sizeof(FallbackSmem), s>>>(a, per, 1, few);
      ++*launched;
    }
  }
  return cudaGetLastError();
}
