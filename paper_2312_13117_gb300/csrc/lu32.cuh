// The FP32 LU's panel, row interchanges, triangular solve and block solves (complex64,
// one CTA of 256 threads per node; lu_mixed.cu). Same pivots as lu_core.cuh (largest
// |Re| + |Im|, lowest row on ties, rows counted in their interchanged order); the order
// of an element's updates is the same too.
//
// What bounds a small or middle node is not arithmetic but instructions and barriers
// around it (at n = 256 the multiply-adds are a third of all instructions, and a column
// took four block barriers). So:
//   * a panel's rows are held in registers, R rows of W = 32 / R columns per thread, and
//     stay where they are: a row carries its position, and an interchange exchanges two
//     positions. A column takes one barrier: every warp publishes its best row together
//     with its key, and all threads pick the winner among the eight;
//   * the panel's permutation then falls out of the positions, and is applied to the
//     columns right of the panel by the triangular solve, which holds the panel's rows of
//     a column in one warp anyway.
// Against sub-panels factored in shared memory with separate interchanges, milliseconds of a
// CTA per node: n = 256 panels 0.89 -> 0.37 (interchanges included), n = 1024 panels,
// interchanges and triangular solves 9.3 -> 5.9, a sweep's solves (l = 16) 2.4 -> 2.0.
#pragma once

#include "lu_core.cuh"

namespace lu32 {

using namespace lucore;

constexpr int ROWS_MAX = 2048;  // rows of a panel in registers (R = 8)

// Shared words of the panel, besides its scratch.
struct PanelSmem {
  float2 row[2][THREADS / 32][NB];  // the warps' candidate rows, by column parity
  float2 l11[NB * NB], us[NB * NB / 2];
  uint2 cand[2][THREADS / 32];      // key, position
  int cnt, nbelow;
  int dst[2 * NB], src[2 * NB];     // the permutation: position dst receives row src
  int topsrc[NB];                   // row that comes to each of the panel's first rows
  int bdst[NB], bsrc[NB];           // rows below that receive one of the panel's first rows
};

// Rows per thread of a panel of `rows` rows.
__host__ __device__ constexpr int panel_r(int rows) { return rows <= 256 ? 1 : rows <= 512 ? 2 : rows <= 1024 ? 4 : 8; }
// Scratch of a panel: the finished entries by row, W columns (at least the 32 x 32 block of
// swap_trsm), then the row at each position, then PanelSmem.
__host__ __device__ constexpr size_t panel_entries(int rows) {
  const size_t p = (size_t)(NB / panel_r(rows)) * rows;
  return p > (size_t)NB * (rows < NB ? rows : NB) ? p : (size_t)NB * (rows < NB ? rows : NB);
}
__host__ __device__ constexpr size_t panel_scratch_bytes(int rows) {
  return ((panel_entries(rows) * sizeof(float2) + (size_t)rows * sizeof(int) + 15) & ~size_t(15)) + sizeof(PanelSmem);
}
__device__ __forceinline__ PanelSmem& panel_smem(unsigned char* scratch, int rows) {
  return *reinterpret_cast<PanelSmem*>(scratch + panel_scratch_bytes(rows) - sizeof(PanelSmem));
}

// Order of the pivot rule: 0 for a NaN, else 1 + the bits of |Re| + |Im|.
__device__ __forceinline__ unsigned pivot_key(float2 a) {
  const float v = l1abs(a);
  return v >= 0.f ? __float_as_uint(v) + 1u : 0u;
}

// Columns j0 .. j1-1 of a sub-panel, whose rows have at most WR columns left; v[i][c] is
// column j + c of the thread's row i, so a step's update also shifts the row left.
template <int R, int W, int WR>
__device__ __forceinline__ void panel_steps(float2 (&v)[R][W], int (&pos)[R], int j0, int j1, int m, int p0,
                                            float2* __restrict__ P, int pld, PanelSmem& ps,
                                            int* __restrict__ piv, int* __restrict__ info) {
  const int tid = gtid(), lane = tid & 31, warp = tid >> 5;
  for (int j = j0; j < j1; ++j) {
    const int b = j & 1;
    unsigned bk = 0;
    int bpos = 0x7fffffff, bi = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const unsigned k = pos[i] >= j && pos[i] < m ? pivot_key(v[i][0]) : 0u;
      if (k > bk || (k == bk && k != 0u && pos[i] < bpos)) {
        bk = k;
        bpos = pos[i];
        bi = i;
      }
    }
    const unsigned wk = __reduce_max_sync(0xffffffffu, bk);
    const int wp = __reduce_min_sync(0xffffffffu, bk == wk ? bpos : 0x7fffffff);
    if (wk == 0u) {
      if (lane == 0) ps.cand[b][warp] = make_uint2(0u, 0u);
    } else if (bk == wk && bpos == wp) {
      ps.cand[b][warp] = make_uint2(wk, (unsigned)wp);
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (bi == i) {
#pragma unroll
          for (int c = 0; c < WR; ++c) ps.row[b][warp][c] = v[i][c];
        }
    }
    gsync();
    const uint2 cd = lane < THREADS / 32 ? ps.cand[b][lane] : make_uint2(0u, 0u);
    const unsigned key = __reduce_max_sync(0xffffffffu, cd.x);
    int pp = (int)__reduce_min_sync(0xffffffffu, cd.x == key ? cd.y : 0x7fffffffu);
    const float2* u;
    if (key != 0u) {
      u = ps.row[b][__ffs(__ballot_sync(0xffffffffu, cd.x == key && (int)cd.y == pp)) - 1];
    } else {  // every entry is NaN (the same in every thread): the pivot is the row at position j
      pp = j;
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (pos[i] == j) {
#pragma unroll
          for (int c = 0; c < WR; ++c) ps.row[b][0][c] = v[i][c];
        }
      gsync();
      u = ps.row[b][0];
    }
    const float2 pv = u[0];
    const bool zero = cis_zero(pv);
    const float2 rp = crecip(pv);
    if (tid == 0) {
      piv[p0 + j] = p0 + pp;
      if (zero && *info == 0) *info = p0 + j + 1;
    }
    float2 l[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      l[i] = zero ? make_float2(0.f, 0.f) : cmul(v[i][0], rp);
      if (pos[i] == pp) {  // the pivot row: its entries from here on are U's
        pos[i] = j;
#pragma unroll
        for (int c = 0; c < WR; ++c)
          if (j + c < W) P[(j + c) * pld + i * THREADS + tid] = v[i][c];
      } else {
        if (pos[i] == j) pos[i] = pp;
        if (pos[i] > j && pos[i] < m) P[j * pld + i * THREADS + tid] = zero ? v[i][0] : l[i];
      }
    }
    // finished rows shift along with the others; their entries are no longer read
#pragma unroll
    for (int c = 1; c < WR; ++c) {
      const float2 uc = u[c];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        float2 x = v[i][c];
        cfms(x, l[i], uc);
        v[i][c - 1] = x;
      }
    }
  }
}

// Factors the panel k0 .. k0+kb-1 of M (n rows, column-major, leading dimension n) in
// sub-panels of W = NB / R columns, n - k0 <= 256 R; left-looking inside the panel: a
// sub-panel's columns get the permutation and the updates of the earlier ones as they are
// loaded. Returns with the CTA synchronised, the panel's rows in their interchanged order
// in M, its permutation in list (global, for the forward solves) and in ps.topsrc / bdst /
// bsrc (for swap_trsm). scratch: panel_scratch_bytes.
template <int R>
__device__ __noinline__ void panel(float2* __restrict__ M, int n, int k0, int kb, int* __restrict__ piv,
                                   int* __restrict__ list, unsigned char* __restrict__ scratch,
                                   int* __restrict__ info) {
  constexpr int W = NB / R;
  const int tid = gtid(), lane = tid & 31, warp = tid >> 5;
  const size_t ld = (size_t)n;
  const int m0 = n - k0;
  float2* P = reinterpret_cast<float2*>(scratch);
  int* perm = reinterpret_cast<int*>(P + panel_entries(m0));  // row at each position (relative to k0)
  PanelSmem& ps = panel_smem(scratch, m0);
  if (W < NB)
    for (int r = tid; r < m0; r += THREADS) perm[r] = r;
  if (tid == 0) ps.cnt = 0;
  gsync();
  for (int off = 0; off < kb; off += W) {
    const int sb = min(W, kb - off), p0 = k0 + off, m = m0 - off;
    float2 v[R][W];
    int pos[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = tid + i * THREADS;
      pos[i] = r < m ? r : 0x40000000;
      const int src = r < m ? (W < NB ? perm[off + r] : r) : 0;
#pragma unroll
      for (int c = 0; c < W; ++c)
        v[i][c] = r < m && c < sb ? M[(size_t)(p0 + c) * ld + k0 + src] : make_float2(0.f, 0.f);
    }
    if (W < NB && off > 0) {
      // U rows of the earlier sub-panels in these columns: L11 x = rows k0 .. p0-1
      constexpr int CPW = (W + 7) / 8;  // columns of a warp
      float2 x[CPW];
      float2* l11 = ps.l11;
      for (int e = tid; e < off * NB; e += THREADS) {
        const int i = e & (NB - 1), t = e / NB;
        if (i < off) l11[e] = M[(size_t)(k0 + t) * ld + k0 + i];
      }
#pragma unroll
      for (int q = 0; q < CPW; ++q) {
        const int c = warp + 8 * q;
        x[q] = lane < off && c < sb ? M[(size_t)(p0 + c) * ld + k0 + perm[lane]] : make_float2(0.f, 0.f);
      }
      gsync();  // every load of these columns is done, l11 is complete
      for (int t = 0; t < off - 1; ++t) {
        const float2 lt = l11[t * NB + lane];
#pragma unroll
        for (int q = 0; q < CPW; ++q) {
          float2 xt;
          xt.x = __shfl_sync(0xffffffffu, x[q].x, t);
          xt.y = __shfl_sync(0xffffffffu, x[q].y, t);
          if (lane > t && lane < off) cfms(x[q], lt, xt);
        }
      }
#pragma unroll
      for (int q = 0; q < CPW; ++q) {
        const int c = warp + 8 * q;
        if (c < W && lane < off) {
          ps.us[lane * W + c] = x[q];
          if (c < sb) M[(size_t)(p0 + c) * ld + k0 + lane] = x[q];
        }
      }
      gsync();
#pragma unroll 2
      for (int t = 0; t < off; ++t) {
        float2 lt[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const int r = tid + i * THREADS;
          lt[i] = r < m ? M[(size_t)(k0 + t) * ld + p0 + r] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int c = 0; c < W; ++c) {
          const float2 u = ps.us[t * W + c];
#pragma unroll
          for (int i = 0; i < R; ++i) cfms(v[i][c], lt[i], u);
        }
      }
    }
    constexpr int Q = W / 4;
    panel_steps<R, W, W>(v, pos, 0, min(sb, Q), m, p0, P, m0, ps, piv, info);
    panel_steps<R, W, W - Q>(v, pos, Q, min(sb, 2 * Q), m, p0, P, m0, ps, piv, info);
    panel_steps<R, W, W - 2 * Q>(v, pos, 2 * Q, min(sb, 3 * Q), m, p0, P, m0, ps, piv, info);
    panel_steps<R, W, W - 3 * Q>(v, pos, 3 * Q, sb, m, p0, P, m0, ps, piv, info);
    // the finished rows to their positions (a thread reads its own entries of P)
    int id[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = tid + i * THREADS;
      id[i] = r < m ? (W < NB ? perm[off + r] : r) : 0;
      if (r < m) {
#pragma unroll
        for (int c = 0; c < W; ++c)
          if (c < sb) M[(size_t)(p0 + c) * ld + p0 + pos[i]] = P[c * m0 + i * THREADS + tid];
        if (pos[i] != r) {
          const int e = atomicAdd(&ps.cnt, 1);
          ps.dst[e] = pos[i];
          ps.src[e] = r;
        }
      }
    }
    gsync();
    if (W < NB) {
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (tid + i * THREADS < m) perm[off + pos[i]] = id[i];
      // the sub-panel's interchanges on the panel's columns left of it
      const int cnt = ps.cnt;
      constexpr int GU = (2 * W * (NB - W) + THREADS - 1) / THREADS;
      float2 g[GU > 0 ? GU : 1];
#pragma unroll
      for (int q = 0; q < GU; ++q) {
        const int e = tid + q * THREADS, c = e / (2 * W), k = e % (2 * W);
        if (c < off && k < cnt) g[q] = M[(size_t)(k0 + c) * ld + p0 + ps.src[k]];
      }
      gsync();
#pragma unroll
      for (int q = 0; q < GU; ++q) {
        const int e = tid + q * THREADS, c = e / (2 * W), k = e % (2 * W);
        if (c < off && k < cnt) M[(size_t)(k0 + c) * ld + p0 + ps.dst[k]] = g[q];
      }
      gsync();
      if (tid == 0) ps.cnt = 0;
      gsync();
    }
  }
  if (W < NB) {  // the panel's permutation
    for (int r = tid; r < m0; r += THREADS)
      if (perm[r] != r) {
        const int e = atomicAdd(&ps.cnt, 1);
        ps.dst[e] = r;
        ps.src[e] = perm[r];
      }
    gsync();
  }
  const int cnt = ps.cnt;
  if (tid < NB) ps.topsrc[tid] = tid;
  if (tid == 0) ps.nbelow = 0;
  gsync();
  if (tid < cnt) {
    const int d = ps.dst[tid], s = ps.src[tid];
    list[1 + tid] = k0 + d;
    list[1 + 2 * NB + tid] = k0 + s;
    if (d < kb) {
      ps.topsrc[d] = s;
    } else {  // such a row receives one of the panel's first rows (interchange j moves row j there)
      const int e = atomicAdd(&ps.nbelow, 1);
      ps.bdst[e] = d;
      ps.bsrc[e] = s;
    }
  }
  if (tid == 0) list[0] = cnt;
  gsync();
}

// The panel's interchanges and U12 = L11^{-1} A12 on columns k0+kb .. ncols-1 in one pass:
// lane i of a warp holds row k0 + i of a column. CW columns per warp at a time, the next
// group's loads issued before this group's substitution.
__device__ inline void swap_trsm(float2* __restrict__ M, int n, int ncols, int k0, int kb, const PanelSmem& ps,
                                 float2* __restrict__ Ls) {
  constexpr int CW = 4, STRIDE = (THREADS / 32) * CW;
  const int tid = gtid(), lane = tid & 31, wid = tid >> 5;
  const size_t ld = (size_t)n;
  const int kend = k0 + kb;
  for (int e = tid; e < kb * NB; e += THREADS) {
    const int i = e & (NB - 1), t = e / NB;
    Ls[e] = i < kb ? M[(size_t)(k0 + t) * ld + k0 + i] : make_float2(0.f, 0.f);  // L11[i][t]
  }
  gsync();
  const int ts = ps.topsrc[lane], nb = ps.nbelow;
  const bool far = lane < kb && ts >= kb;  // this position's row comes from below the panel
  const int bd = lane < nb ? ps.bdst[lane] : 0, bs = lane < nb ? ps.bsrc[lane] : 0;
  float2 xt[CW], xf[CW];
  auto load = [&](int c0) {
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      const int c = c0 + q;
      xt[q] = lane < kb && c < ncols ? M[(size_t)c * ld + k0 + lane] : make_float2(0.f, 0.f);
      xf[q] = far && c < ncols ? M[(size_t)c * ld + k0 + ts] : make_float2(0.f, 0.f);
    }
  };
  load(kend + wid * CW);
  for (int c0 = kend + wid * CW; c0 < ncols; c0 += STRIDE) {
    float2 x[CW];
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      float2 s, d;
      s.x = __shfl_sync(0xffffffffu, xt[q].x, ts & 31);
      s.y = __shfl_sync(0xffffffffu, xt[q].y, ts & 31);
      d.x = __shfl_sync(0xffffffffu, xt[q].x, bs);
      d.y = __shfl_sync(0xffffffffu, xt[q].y, bs);
      x[q] = far ? xf[q] : s;
      __syncwarp();  // the column's rows are all read before any is written
      if (lane < nb && c0 + q < ncols) M[(size_t)(c0 + q) * ld + k0 + bd] = d;
    }
    load(c0 + STRIDE);
    for (int t = 0; t < kb - 1; ++t) {
      const float2 lt = Ls[t * NB + lane];
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        float2 y;
        y.x = __shfl_sync(0xffffffffu, x[q].x, t);
        y.y = __shfl_sync(0xffffffffu, x[q].y, t);
        if (lane > t) cfms(x[q], lt, y);  // (lanes past kb hold zeros of L11)
      }
    }
#pragma unroll
    for (int q = 0; q < CW; ++q)
      if (lane < kb && c0 + q < ncols) M[(size_t)(c0 + q) * ld + k0 + lane] = x[q];
  }
  gsync();
}

// ---------------------------------------------------------------------------
// Triangular solves with the factors on l columns Y (leading dimension n; shared or global
// memory), in 32-row blocks: the diagonal block one warp per column pair (lane = row),
// then the rows outside it by all threads.
// ---------------------------------------------------------------------------
struct SolveSmem32 {
  alignas(16) float2 Ls[NB * NB];             // diagonal block, [t][i]
  alignas(16) float2 S[NB * PMCIM_MAX_L];     // the block's solution, [t][column], stride l rounded up to 8
};

// Y[i] -= sum_t M[i, k0 + t] S[t] on rows r0 .. r1-1; CH columns per task, a row's columns
// spread over several tasks where l > CH. Eight of the row's entries are in flight.
template <int CH>
__device__ __forceinline__ void update_rows(const float2* __restrict__ M, float2* __restrict__ Y, int n, int l, int k0,
                                            int kb, int r0, int r1, const SolveSmem32& sm, int ldS) {
  const int rows = r1 - r0, nch = (l + CH - 1) / CH;
  if (rows <= 0) return;
  int ch = gtid() / rows, r = gtid() - ch * rows;
  const int dch = THREADS / rows, dr = THREADS - dch * rows;
  for (; ch < nch;) {
    const int i = r0 + r, c0 = ch * CH;
    const float2* mrow = M + (size_t)k0 * n + i;
    float2 acc[CH];
#pragma unroll
    for (int q = 0; q < CH; ++q) acc[q] = c0 + q < l ? Y[(size_t)(c0 + q) * n + i] : make_float2(0.f, 0.f);
    for (int t0 = 0; t0 < kb; t0 += 8) {
      float2 m[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) m[u] = t0 + u < kb ? mrow[(size_t)(t0 + u) * n] : make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float4* s4 = reinterpret_cast<const float4*>(sm.S + (t0 + u) * ldS + c0);
#pragma unroll
        for (int q = 0; q < CH; q += 2) {
          const float4 s = s4[q / 2];
          cfms(acc[q], m[u], make_float2(s.x, s.y));
          cfms(acc[q + 1], m[u], make_float2(s.z, s.w));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < CH; ++q)
      if (c0 + q < l) Y[(size_t)(c0 + q) * n + i] = acc[q];
    ch += dch;
    r += dr;
    if (r >= rows) {
      r -= rows;
      ++ch;
    }
  }
}

__device__ __forceinline__ void load_diagonal(const float2* __restrict__ M, int n, int k0, int kb, SolveSmem32& sm) {
#pragma unroll
  for (int e = gtid(); e < NB * NB; e += THREADS) {
    const int i = e & (NB - 1), t = e / NB;
    sm.Ls[e] = i < kb && t < kb ? M[(size_t)(k0 + t) * n + k0 + i] : make_float2(0.f, 0.f);
  }
}

// Division by one pivot (Smith, cdiv to the bit: its products are rounded before they are
// added): the ratio of the pivot's parts and the denominator are formed once, two real
// divisions are left per quotient.
struct Divisor {
  float t, d;
  bool re;  // |Re| >= |Im|
  __device__ explicit Divisor(float2 b) : re(fabsf(b.x) >= fabsf(b.y)) {
    const float u = re ? b.x : b.y, v = re ? b.y : b.x;
    t = v / u;
    d = __fadd_rn(__fmul_rn(v, t), u);
  }
  __device__ __forceinline__ float2 divide(float2 a) const {
    const float p = __fmul_rn(a.x, t), q = __fmul_rn(a.y, t);
    const float x = re ? __fadd_rn(q, a.x) : __fadd_rn(p, a.y);
    const float y = re ? __fadd_rn(-p, a.y) : __fadd_rn(q, -a.x);
    return make_float2(x / d, y / d);
  }
};

// The diagonal block's solve; lower: unit lower triangle, else upper, whose unknowns are
// quotients by the pivots (a multiplication by a rounded reciprocal would be one rounding
// more per unknown). S rows past kb and columns past l become zero.
template <bool LOWER>
__device__ __forceinline__ void solve_diagonal(float2* __restrict__ Y, int n, int l, int k0, int kb, SolveSmem32& sm,
                                               int ldS) {
  const int lane = gtid() & 31, wid = gtid() >> 5;
  const Divisor pivot(!LOWER && lane < kb ? sm.Ls[lane * NB + lane] : make_float2(1.f, 0.f));
  for (int c = wid; c < ldS; c += 2 * (THREADS / 32)) {
    const int c2 = c + THREADS / 32;
    float2 a = lane < kb && c < l ? Y[(size_t)c * n + k0 + lane] : make_float2(0.f, 0.f);
    float2 b = lane < kb && c2 < l ? Y[(size_t)c2 * n + k0 + lane] : make_float2(0.f, 0.f);
    for (int s = 0; s < kb; ++s) {
      const int t = LOWER ? s : kb - 1 - s;
      const float2 lt = sm.Ls[t * NB + lane];
      if (!LOWER && lane == t) {
        a = pivot.divide(a);
        b = pivot.divide(b);
      }
      float2 ta, tb;
      ta.x = __shfl_sync(0xffffffffu, a.x, t);
      ta.y = __shfl_sync(0xffffffffu, a.y, t);
      tb.x = __shfl_sync(0xffffffffu, b.x, t);
      tb.y = __shfl_sync(0xffffffffu, b.y, t);
      if (LOWER ? lane > t : lane < t) {
        cfms(a, lt, ta);
        cfms(b, lt, tb);
      }
    }
    if (lane < kb && c < l) Y[(size_t)c * n + k0 + lane] = a;
    if (lane < kb && c2 < l) Y[(size_t)c2 * n + k0 + lane] = b;
    sm.S[lane * ldS + c] = a;
    if (c2 < ldS) sm.S[lane * ldS + c2] = b;
  }
}

__device__ __forceinline__ void update_any(const float2* __restrict__ M, float2* __restrict__ Y, int n, int l, int k0,
                                           int kb, int r0, int r1, const SolveSmem32& sm, int ldS) {
  // sixteen columns a task where the rows alone fill the CTA (the factors are then read once),
  // else eight
  if (l > 8 && r1 - r0 >= THREADS) update_rows<16>(M, Y, n, l, k0, kb, r0, r1, sm, ldS);
  else update_rows<8>(M, Y, n, l, k0, kb, r0, r1, sm, ldS);
}
__device__ __forceinline__ int solve_lds(int l) { return l > 8 ? (l + 15) / 16 * 16 : 8; }

// U x = y.
__device__ inline void back(const float2* __restrict__ M, float2* __restrict__ Y, int n, int l, SolveSmem32& sm) {
  const int ldS = solve_lds(l);
  for (int k0 = (n - 1) / NB * NB; k0 >= 0; k0 -= NB) {
    const int kb = min(NB, n - k0);
    load_diagonal(M, n, k0, kb, sm);
    gsync();
    solve_diagonal<false>(Y, n, l, k0, kb, sm, ldS);
    gsync();
    update_any(M, Y, n, l, k0, kb, 0, k0, sm, ldS);
    gsync();
  }
}

// L y = b, each panel's permutation (lists + p SWAP_LIST_INTS, global memory) applied to y
// before its columns of L.
__device__ inline void forward(const float2* __restrict__ M, float2* __restrict__ Y, int n, int l, SolveSmem32& sm,
                               const int* __restrict__ lists) {
  const int ldS = solve_lds(l), lane = gtid() & 31, wid = gtid() >> 5;
  for (int k0 = 0; k0 < n; k0 += NB) {
    const int kb = min(NB, n - k0);
    {
      // a warp per column: all its rows are read before any is written
      const int* L = lists + (size_t)(k0 / NB) * SWAP_LIST_INTS;
      const int cnt = L[0];
      const int d0 = lane < cnt ? L[1 + lane] : 0, s0 = lane < cnt ? L[1 + 2 * NB + lane] : 0;
      const int d1 = lane + 32 < cnt ? L[33 + lane] : 0, s1 = lane + 32 < cnt ? L[33 + 2 * NB + lane] : 0;
      for (int c = wid; c < l; c += THREADS / 32) {
        float2* y = Y + (size_t)c * n;
        const float2 a = y[s0], b = y[s1];
        __syncwarp();
        if (lane < cnt) y[d0] = a;
        if (lane + 32 < cnt) y[d1] = b;
      }
    }
    load_diagonal(M, n, k0, kb, sm);
    gsync();
    solve_diagonal<true>(Y, n, l, k0, kb, sm, ldS);
    gsync();
    update_any(M, Y, n, l, k0, kb, k0 + kb, n, sm, ldS);
    gsync();
  }
}

}  // namespace lu32
