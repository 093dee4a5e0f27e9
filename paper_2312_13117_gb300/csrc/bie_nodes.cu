// T(z_j) of boundary-integral nodes for the precision forms: the matrix in FP64, and
// its exact digits for the residuals on the tensor cores.
//
// The entries are FP64 Bessel evaluations (bie.cuh), about 220 FP64 operations each at
// 2 per SM and clock, n (n - 1) / 2 of them per node where every pair of points has its
// own distance: that bounds the assembly (n = 256: 1.7 ms of one SM). It is a kernel of
// its own, in pieces of 4096 pairs, so that all SMs share it evenly however few nodes there are.
// Where the matrix is circulant (a circle) a node has n distinct entries and only they
// are formed and kept.
//
// The residual V - T(z_j) X on the FP64 unit is 8 n^2 l operations a sweep, more than the
// whole assembly of a circulant node. As digits it is tensor work like that of the other
// problems (oz_refine.cu); making the digits is integer arithmetic on the entries' bits.
// Measured on whole calls with FP32 LUs, n = 256, l = 8: a circle, 6400 nodes, 118 -> 46.8 ms;
// an ellipse, 768 nodes, 63.2 -> 23.2 ms.
#include "ozaki.cuh"

namespace {

using namespace ozk;

constexpr int BT = 256;
constexpr int PIECE = 4096;  // pairs of an assembly item
constexpr int CIRC = 1024;   // largest circulant matrix that is written from its first column

// rint(x 2^shift) as an integer (ties away from zero), |result| <= 2^55, by the bits of x.
__device__ __forceinline__ long long scaled_integer(double x, int shift) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  const int sh = 1075 - ex - shift;  // x = m 2^(ex - 1075)
  if (ex == 0 || ex == 0x7ff || sh > 53) return 0;  // (an overflowed entry has no digits)
  const long long m = (b & 0xfffffffffffffll) | (1ll << 52);
  const long long r = sh > 0 ? (m + (1ll << (sh - 1))) >> sh : m << -sh;
  return b < 0 ? -r : r;
}

// High word of |x|: ordered as |x|, and its exponent field gives the row exponent.
__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }
// The exponent e with |x| < 2^e for values up to high word h (0 for zero rows).
__device__ __forceinline__ int exponent_of_hi(int h) { return h >> 20 ? (h >> 20) - 1022 : 0; }

__global__ void __launch_bounds__(BT, 2) k_bie_assemble(MixedArgs a, int pieces) {
  __shared__ ProblemDev P;
  __shared__ double2 fz[PMCIM_MAX_TERMS];
  __shared__ bie::Wave wave;
  __shared__ double2 first[CIRC];
  for (long long w = blockIdx.x; w < (long long)a.count * pieces; w += gridDim.x) {
    // (pieces outermost: the CTAs share the first pieces of all nodes, the only ones of circulant nodes)
    const int q = (int)(w % a.count), piece = (int)(w / a.count);
    const NodeItem it = a.items[q];
    const RegionDev rg = a.regions[it.region];
    const ProblemDev& G = a.probs[rg.prob];
    if (!G.bie || rg.herm) continue;  // the same in every thread
    const int n = G.n, pairs = n * (n / 2);
    const bool column = mixed_column_only(a, G);
    if (column ? piece > 0 : piece * PIECE >= pairs) continue;
    __syncthreads();
    load_problem(&P, &G);
    __syncthreads();
    double2 z, wt;
    node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &wt);
    if (threadIdx.x < P.K) fz[threadIdx.x] = eval_f(P.term[threadIdx.x], z);
    if (threadIdx.x == 0) wave = bie::wave_of(z);
    __syncthreads();
    const double2 cb = layer_coefficient(P);
    double2 id = make_double2(0.0, 0.0);
    for (int k = 0; k < P.K; ++k)
      if (!P.term[k].dense && P.term[k].kind != PMCIM_F_HELMHOLTZ_DLP) id = cadd(id, cmul(fz[k], P.term[k].id));
    const size_t nn = (size_t)n * n;
    double2* T = a.t64 + (size_t)q * a.t64_stride;
    auto store = [&](int i, int j, double2 v) {
      const size_t e = (size_t)j * n + i;
      for (int k = 0; k < P.K; ++k)
        if (P.term[k].dense) cfma(v, fz[k], P.A[(size_t)P.term[k].mat_index * nn + e]);
      T[e] = v;
    };
    if (column) {
      for (int m = threadIdx.x; m < n; m += BT) {
        double2 v = cmul(cb, bie::dlp_entry(P.bie, n, m, 0, wave));
        T[m] = m == 0 ? cadd(v, id) : v;
      }
      continue;
    }
    if (P.bie_circ && n <= CIRC) {  // n distinct entries: every piece forms them and writes its share
      for (int m = threadIdx.x; m < n; m += BT) first[m] = cmul(cb, bie::dlp_entry(P.bie, n, m, 0, wave));
      __syncthreads();
      for (int e = 2 * piece * PIECE + threadIdx.x; e < min(n * n, 2 * (piece + 1) * PIECE); e += BT) {
        const int j = e / n, i = e - j * n;
        const double2 v = first[i >= j ? i - j : i - j + n];
        store(i, j, i == j ? cadd(v, id) : v);
      }
      continue;
    }
    for (int p = piece * PIECE + threadIdx.x; p < min(pairs, (piece + 1) * PIECE); p += BT) {
      int i, j;
      if (!bie::pair_of(n, p, &i, &j)) continue;
      double2 x, y;
      bie::dlp_pair(P.bie, n, i, j, wave, &x, &y);
      store(i, j, cmul(cb, x));
      store(j, i, cmul(cb, y));
    }
    if (piece == 0)
      for (int j = threadIdx.x; j < n; j += BT) store(j, j, cadd(cmul(cb, bie::dlp_diagonal(P.bie, n, j)), id));
  }
}

// Row exponents and digit tiles [kc][digit][re, im] of one 128-row block of a node's T(z_j)
// (the layout of k_coeff_digits).
__global__ void __launch_bounds__(BT) k_bie_digits(MixedArgs a, int max_rb) {
  __shared__ int emax[TM];
  const int tid = threadIdx.x;
  for (long long w = blockIdx.x; w < (long long)a.count * max_rb; w += gridDim.x) {
    const int q = (int)(w / max_rb), rb = (int)(w % max_rb);
    const NodeItem it = a.items[q];
    const RegionDev rg = a.regions[it.region];
    const ProblemDev& P = a.probs[rg.prob];
    if (!P.bie || rg.herm || rb >= row_blocks(P.n)) continue;  // the same in every thread
    const int n = P.n, kcn = k_chunks(n);
    const bool column = mixed_column_only(a, P);
    const double2* T = a.t64 + (size_t)q * a.t64_stride;
    __syncthreads();  // emax of the previous item
    if (tid < TM) emax[tid] = 0;
    __syncthreads();
    {
      const int r = tid & (TM - 1), i = rb * TM + r;
      int h = 0;
      if (i < n) {
        if (column)  // every row holds the same values
          for (int m = tid / TM; m < n; m += BT / TM) h = max(h, max(abs_hi(T[m].x), abs_hi(T[m].y)));
        else
#pragma unroll 4
          for (int j = tid / TM; j < n; j += BT / TM) {
            const double2 v = T[(size_t)j * n + i];
            h = max(h, max(abs_hi(v.x), abs_hi(v.y)));
          }
      }
      atomicMax(&emax[r], h);
    }
    __syncthreads();
    if (tid < TM) {
      emax[tid] = exponent_of_hi(emax[tid]);
      a.texp[(size_t)q * a.texp_stride + rb * TM + tid] = emax[tid];
    }
    __syncthreads();
    unsigned char* base = a.tdig + (size_t)q * a.tdig_stride + (size_t)rb * kcn * BIE_DIGITS * A_STAGE;
    for (int task = tid; task < TM * kcn * (KC / 8); task += BT) {
      const int r = task & (TM - 1), j0 = task / TM * 8, i = rb * TM + r;
      const int shift = 7 * BIE_DIGITS - 1 - emax[r];
      long long Nr[8], Ni[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + u;
        double2 v = make_double2(0.0, 0.0);
        if (i < n && j < n) v = column ? T[i >= j ? i - j : i - j + n] : T[(size_t)j * n + i];
        Nr[u] = scaled_integer(v.x, shift);
        Ni[u] = scaled_integer(v.y, shift);
      }
      unsigned char* st = base + (size_t)(j0 / KC) * BIE_DIGITS * A_STAGE + tile_off(r, j0 % KC);
#pragma unroll 1
      for (int t = BIE_DIGITS - 1; t >= 0; --t) {
        uint32_t pr[4], pi[4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const int v0 = next_digit(Nr[u], t), v1 = next_digit(Nr[u + 1], t);
          const int v2 = next_digit(Ni[u], t), v3 = next_digit(Ni[u + 1], t);
          pr[u / 2] = (uint32_t)bf16_of_int(v0) | ((uint32_t)bf16_of_int(v1) << 16);
          pi[u / 2] = (uint32_t)bf16_of_int(v2) | ((uint32_t)bf16_of_int(v3) << 16);
        }
        *reinterpret_cast<uint4*>(st + (size_t)t * A_STAGE) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
        *reinterpret_cast<uint4*>(st + (size_t)t * A_STAGE + A_TILE) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
      }
    }
  }
}

}  // namespace

size_t bie_digit_bytes(int n) { return (size_t)row_blocks(n) * k_chunks(n) * BIE_DIGITS * A_STAGE; }

cudaError_t launch_bie_assemble(const MixedArgs& a, int sms, cudaStream_t s, int* launched) {
  const int pieces = (a.max_n * (a.max_n / 2) + PIECE - 1) / PIECE, rb = row_blocks(a.max_n);
  auto grid = [&](long long items, int per_sm) {
    return (unsigned)(items < (long long)per_sm * sms ? items : (long long)per_sm * sms);
  };
  k_bie_assemble<<<grid((long long)a.count * pieces, 2), BT, 0, s>>>(a, pieces);
  ++*launched;
  if (a.tdig) {
    k_bie_digits<<<grid((long long)a.count * rb, 4), BT, 0, s>>>(a, rb);
    ++*launched;
  }
  return cudaGetLastError();
}
