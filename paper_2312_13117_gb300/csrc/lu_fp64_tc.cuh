// Trailing updates of the FP64 LU on the 5th-generation tensor cores.
//
// A22 -= L21 U12 for an outer block of 64 columns. GB300 has 2 FP64 multiply-adds per SM and
// clock, so the update's n^3 / 3 complex multiply-adds were nearly all of a node's time. Here
// each row of L21 and each column of U12 becomes integers of 55 bits under a common power of
// two, cut into seven balanced base-256 digits (exact in BF16), and a product is the sum over
// the 34 digit pairs with s + t <= 7 (the idea of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication",
// Numer. Algorithms 59, 2012). A digit order q = s + t adds at most 7 pairs x 2 (complex) x 64
// products of at most 2^14, an integer below 2^24: the FP32 accumulators are exact. They are
// summed as int64, and C takes one FP64 multiply-add per real number and outer block in place
// of 128.
//
// The inner index is balanced first: U's row k is divided, and L's column k multiplied, by the
// power of two above the row's largest entry, so that a row scale of the matrix (which U's rows
// carry) costs no bits. Against 64-bit mantissas, a block of a Gaussian matrix of order 256 is
// off by 2.4e-17 rms (elements of 0.17) where the chain of FMAs that this replaces is off by
// 6.4e-17; with s + t <= 6 (28 pairs) it would be 1.3e-16. Entries beyond 2^+-400 and
// infinities or NaN leave the block to the FMA pipes.
//
// A tile is 128 rows by 16 columns, real and imaginary parts side by side (N = 32):
//   D_q += Lr[s] [Ur | Ui][t] + Li[s] [-Ui | Ur][t], q = s + t,
// eight orders of 32 TMEM columns, 256 in all; two CTAs share an SM. As the orders' columns and
// U12's digits both follow one another, one MMA of up to 224 columns multiplies a digit of L21
// by all of U12's (an MMA per pair took 137 clocks each, at N = 32). The digits go through
// global scratch in the MMA's operand layout. A tile needs 224 KB of L21's and 56 KB of U12's,
// and the next one the same of L21's: they come from L2 through a ring of 8 KB stages, whose
// depth and the copies' latency bound the tiles, U12's through a ring of four 14 KB chunks. One
// thread copies, one issues, and all eight warps drain a tile, beside the other CTA's MMAs.
// At n = 1024 a node's 2672 tiles take 11.5 us each to issue, 5 more until the products are
// complete, and 5 to drain; the digits take 4.6 ms of the node's 65.
//
// Every wait is bounded. When one runs out the copies and MMAs in flight are waited for, and
// the rest of this block and the CTA's later blocks use the FMA pipes.
#pragma once
#include "ozaki.cuh"

namespace ozlu {

using lucore::THREADS;

constexpr int KO = 64;                 // columns of an outer block
constexpr int S = 7;                   // digits
constexpr int BITS = 55;
constexpr int TM = 128, CN = 16;
constexpr int RING = 6;
constexpr int A_STAGE = 2 * TM * 16 * 2;       // digit s of 16 inner indices: real, imaginary
constexpr int A_STEPS = KO / 16 * S;           // stages of a tile
constexpr int B_PART = 2 * CN * 16 * 2;        // one digit and form of 16 inner indices
constexpr int B_CHUNK = 2 * S * B_PART;        // [form][digit]
constexpr int B_RING = KO / 16;
constexpr int B_BLOCK = B_RING * B_CHUNK;
constexpr int STAGE_BYTES = RING * A_STAGE + B_BLOCK;  // 104 KB
constexpr int ORDERS = S + 1;
constexpr uint32_t TMEM_COLS = 256;  // ORDERS * 2 * CN
constexpr int MAX_EXP = 400;

struct Shared {
  uint64_t full[RING], empty[RING], b_full[B_RING], b_empty[B_RING], acc, last;
  uint32_t tmem;
  int bad;
  uint32_t a_issued, b_issued;  // copies issued, for the settling wait
  int ek[KO];
  int red[THREADS];
};

// The counters of the barriers' phases: copies (the copying thread's), stages multiplied (the
// issuing thread's), tiles (every thread's).
struct State {
  uint32_t a_issued = 0, a_used = 0, b_issued = 0, b_used = 0, acc = 0;
  bool on = true;
};

inline __host__ __device__ int row_blocks(int n) { return (n + TM - 1) / TM; }
inline __host__ __device__ int col_blocks(int ncols) { return (ncols + CN - 1) / CN; }
// Scratch of a matrix: L21's digits, U12's, then the exponents of rows and columns.
inline __host__ __device__ size_t scratch_bytes(int n, int l) {
  const size_t b = (size_t)row_blocks(n) * A_STEPS * A_STAGE + (size_t)col_blocks(n + l) * B_BLOCK +
                   ((size_t)row_blocks(n) * TM + (size_t)col_blocks(n + l) * CN) * sizeof(int);
  return (b + 127) & ~(size_t)127;
}

__device__ __forceinline__ int expo_field(double2 v) {
  return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff) >> 20;
}
// rint(x 2^shift) (ties away from zero), |result| <= 2^BITS, by the bits of x.
__device__ __forceinline__ long long scaled_integer(double x, int shift) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  const int sh = 1075 - ex - shift;
  if (ex == 0 || sh > 53) return 0;
  const long long m = (b & 0xfffffffffffffll) | (1ll << 52);
  const long long r = sh > 0 ? (m + (1ll << (sh - 1))) >> sh : m << -sh;
  return b < 0 ? -r : r;
}
__device__ __forceinline__ int next_digit(long long& N, int s) {
  if (s == 0) return (int)N;
  const int d = (int)(signed char)(N & 255);
  N = (N - d) >> 8;
  return d;
}
__device__ __forceinline__ uint32_t pack2(int a, int b) {
  return (uint32_t)ozk::bf16_of_int(a) | ((uint32_t)ozk::bf16_of_int(b) << 16);
}

// Operand descriptor: K-major, no swizzle, core matrices 128 B apart along K, 8-row groups 256 B.
__device__ __forceinline__ uint64_t desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t cols, uint32_t acc) {
  // kind::f16, F32 accumulator, BF16 A and B, both K-major, M = 128, N = cols
  const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | ((cols >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr)
      : "memory");
}

// Before the first update: barriers and TMEM (all threads).
__device__ __forceinline__ void begin(Shared& sh) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < RING; ++i) {
      tcu::mbar_init(&sh.full[i]);
      tcu::mbar_init(&sh.empty[i]);
    }
    for (int i = 0; i < B_RING; ++i) {
      tcu::mbar_init(&sh.b_full[i]);
      tcu::mbar_init(&sh.b_empty[i]);
    }
    tcu::mbar_init(&sh.acc);
    tcu::mbar_init(&sh.last);
    sh.bad = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) tcu::tmem_alloc_cols(&sh.tmem, TMEM_COLS);
  tcu::fence_before();
  __syncthreads();
  tcu::fence_after();
}
// After the last one (all threads; no MMA is in flight).
__device__ __forceinline__ void end(Shared& sh) {
  tcu::fence_before();
  __syncthreads();
  tcu::fence_after();
  if (threadIdx.x < 32) tcu::tmem_dealloc_cols(sh.tmem, TMEM_COLS);
}

// The digits of L21 (rows kend..n-1) and U12 (columns kend..ncols-1). False (in every thread)
// when an exponent is out of range.
__device__ bool make_digits(const double2* M, int n, int ncols, int k0, unsigned char* A, unsigned char* B, int* er,
                            int* ec, Shared& sh) {
  const int tid = threadIdx.x, kend = k0 + KO;
  const size_t ld = (size_t)n;
  const int rows = row_blocks(n - kend) * TM, cols = col_blocks(ncols - kend) * CN;
  bool fine = true;
  {
    const double2* row = M + k0 + (tid & (KO - 1));
    int m = 0;
#pragma unroll 8
    for (int j = kend + tid / KO; j < ncols; j += THREADS / KO) m = max(m, expo_field(row[(size_t)j * ld]));
    sh.red[tid] = m;
    __syncthreads();
    if (tid < KO) {
      for (int g = 1; g < THREADS / KO; ++g) m = max(m, sh.red[g * KO + tid]);
      fine = m == 0 || abs(m - 1022) <= MAX_EXP;
      sh.ek[tid] = m ? m - 1022 : 0;
    }
    __syncthreads();
  }
  constexpr int NONE = -(1 << 20);
  for (int r = tid; r < rows; r += THREADS) {
    const bool in = kend + r < n;
    const double2* Lr = M + (size_t)k0 * ld + (in ? kend + r : 0);
    int e = NONE;
#pragma unroll 8
    for (int k = 0; k < KO; ++k) {
      const int f = in ? expo_field(Lr[(size_t)k * ld]) : 0;
      if (f) e = max(e, f - 1022 + sh.ek[k]);
      fine = fine && f != 2047;
    }
    if (e == NONE) e = 0;
    fine = fine && abs(e) <= MAX_EXP;
    er[r] = e;
    unsigned char* dst = A + (size_t)(r / TM) * A_STEPS * A_STAGE + (r % TM >> 3) * 256 + (r & 7) * 16;
#pragma unroll 1
    for (int k = 0; k < KO; k += 8) {
      long long Nr[8], Ni[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double2 v = in ? Lr[(size_t)(k + u) * ld] : make_double2(0.0, 0.0);
        Nr[u] = scaled_integer(v.x, sh.ek[k + u] + BITS - e);
        Ni[u] = scaled_integer(v.y, sh.ek[k + u] + BITS - e);
      }
      unsigned char* d = dst + (size_t)(k / 16) * S * A_STAGE + (k & 8) * 16;
#pragma unroll 1
      for (int s = S - 1; s >= 0; --s) {
        uint32_t pr[4], pi[4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          const int r0 = next_digit(Nr[u], s), r1 = next_digit(Nr[u + 1], s);
          const int i0 = next_digit(Ni[u], s), i1 = next_digit(Ni[u + 1], s);
          pr[u / 2] = pack2(r0, r1);
          pi[u / 2] = pack2(i0, i1);
        }
        *reinterpret_cast<uint4*>(d + s * A_STAGE) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
        *reinterpret_cast<uint4*>(d + s * A_STAGE + A_STAGE / 2) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
      }
    }
  }
  // eight lanes a column, eight inner indices each (a warp's columns are in or out together
  // of the loop: cols is a multiple of 16)
  const int k = (tid & 7) * 8;
  for (int j = tid >> 3; j < cols; j += THREADS / 8) {
    const bool in = kend + j < ncols;
    const double2* U = M + (size_t)(in ? kend + j : 0) * ld + k0 + k;
    double2 v[8];
    int e = NONE;
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = in ? U[u] : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int f = expo_field(v[u]);
      if (f) e = max(e, f - 1022 - sh.ek[k + u]);
    }
    for (int o = 1; o < 8; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (e == NONE) e = 0;
    fine = fine && abs(e) <= MAX_EXP;
    if ((tid & 7) == 0) ec[j] = e;
    long long Nr[8], Ni[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      Nr[u] = scaled_integer(v[u].x, BITS - e - sh.ek[k + u]);
      Ni[u] = scaled_integer(v[u].y, BITS - e - sh.ek[k + u]);
    }
    // operand rows: [re 0-7 | im 0-7 | re 8-15 | im 8-15] of the block's columns
    const int c = j % CN;
    unsigned char* d = B + (size_t)(j / CN) * B_BLOCK + (size_t)(k / 16) * B_CHUNK + (c >> 3) * 512 +
                       (k & 8) * 16 + (c & 7) * 16;
#pragma unroll 1
    for (int s = S - 1; s >= 0; --s) {
      uint32_t pr[4], pi[4], ni[4];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        const int r0 = next_digit(Nr[u], s), r1 = next_digit(Nr[u + 1], s);
        const int i0 = next_digit(Ni[u], s), i1 = next_digit(Ni[u + 1], s);
        pr[u / 2] = pack2(r0, r1);
        pi[u / 2] = pack2(i0, i1);
        ni[u / 2] = pack2(-i0, -i1);
      }
      unsigned char* f0 = d + s * B_PART;
      unsigned char* f1 = f0 + S * B_PART;
      *reinterpret_cast<uint4*>(f0) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<uint4*>(f0 + 256) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
      *reinterpret_cast<uint4*>(f1) = make_uint4(ni[0], ni[1], ni[2], ni[3]);
      *reinterpret_cast<uint4*>(f1 + 256) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
    }
  }
  ozk::fence_proxy_async_all();  // the digits, and the stage's earlier use, before the bulk copies
  return __syncthreads_and(fine) != 0;
}

// An update's tiles, row blocks outermost, and the copying thread's place in them.
struct Tiles {
  const unsigned char *A, *B;
  int rbn, cbn;
  uint32_t next_a, next_b;  // copies issued
};

__device__ __forceinline__ bool copy_a(Tiles& q, unsigned char* stage, Shared& sh, State& st, long long limit) {
  const uint32_t slot = st.a_issued % RING, turn = st.a_issued / RING;
  if (turn > 0 && !tcu::wait_parity(&sh.empty[slot], (turn - 1) & 1u, limit)) return false;
  const uint32_t tile = q.next_a / A_STEPS;
  ozk::expect_tx(&sh.full[slot], A_STAGE);
  ozk::bulk_g2s(stage + slot * A_STAGE, q.A + (size_t)(tile / q.cbn * A_STEPS + q.next_a % A_STEPS) * A_STAGE, A_STAGE,
                &sh.full[slot]);
  ++st.a_issued;
  ++q.next_a;
  return true;
}
__device__ __forceinline__ bool copy_b(Tiles& q, unsigned char* stage, Shared& sh, State& st, long long limit) {
  const uint32_t slot = st.b_issued % B_RING, turn = st.b_issued / B_RING;
  if (turn > 0 && !tcu::wait_parity(&sh.b_empty[slot], (turn - 1) & 1u, limit)) return false;
  const uint32_t tile = q.next_b / B_RING;
  ozk::expect_tx(&sh.b_full[slot], B_CHUNK);
  ozk::bulk_g2s(stage + RING * A_STAGE + slot * B_CHUNK,
                q.B + (size_t)(tile % q.cbn) * B_BLOCK + (size_t)(q.next_b % B_RING) * B_CHUNK, B_CHUNK,
                &sh.b_full[slot]);
  ++st.b_issued;
  ++q.next_b;
  return true;
}

// The copies of the tiles up to this one, and the ring's next ones. False when a wait ran out.
__device__ bool copy_tile(Tiles& q, int tile, unsigned char* stage, Shared& sh, State& st, long long limit) {
  const uint32_t end = min((uint32_t)(q.rbn * q.cbn * A_STEPS), (uint32_t)(tile + 1) * A_STEPS + RING);
  while (q.next_a < end) {
    if (q.next_a % S == 0 && q.next_b * S == q.next_a && !copy_b(q, stage, sh, st, limit)) return false;
    if (!copy_a(q, stage, sh, st, limit)) return false;
  }
  return true;
}

// One tile's MMAs. False when a wait ran out.
__device__ bool issue_tile(unsigned char* stage, Shared& sh, State& st, long long limit) {
  const uint32_t tmem = sh.tmem;
  const uint64_t a_desc = desc(tcu::smem_u32(stage)), b_desc = desc(tcu::smem_u32(stage + RING * A_STAGE));
#pragma unroll 1
  for (int ks = 0; ks < B_RING; ++ks) {
    const uint32_t bs = st.b_used % B_RING;
    if (!tcu::wait_parity(&sh.b_full[bs], (st.b_used / B_RING) & 1u, limit)) return false;
    // (descriptor addresses count 16 bytes, and stay below their field's 2^14)
    const uint64_t b0 = b_desc + bs * (B_CHUNK / 16), b1 = b0 + S * (B_PART / 16);
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
      const uint32_t slot = st.a_used % RING;
      if (!tcu::wait_parity(&sh.full[slot], (st.a_used / RING) & 1u, limit)) return false;
      tcu::fence_after();
      const uint64_t a0 = a_desc + slot * (A_STAGE / 16), a1 = a0 + A_STAGE / 32;
      const uint32_t d = tmem + (uint32_t)(s * 2 * CN), cols = (uint32_t)(2 * CN * min(S, ORDERS - s));
      // the first product of an order overwrites the last tile's: order 7's is that of s = 1, t = 6
      if (ks == 0 && s == 1) {
        mma(d, a0, b0, cols - 2 * CN, 1u);
        mma(tmem + (ORDERS - 1) * 2 * CN, a0, b0 + (S - 1) * (B_PART / 16), 2 * CN, 0u);
      } else {
        mma(d, a0, b0, cols, ks != 0 || s != 0);
      }
      mma(d, a1, b1, cols, 1u);
      tcu::commit(&sh.empty[slot]);
      ++st.a_used;
    }
    tcu::commit(&sh.b_empty[bs]);
    ++st.b_used;
  }
  tcu::commit(&sh.acc);
  return true;
}

// A22 -= L21 U12 for the outer block k0..k0+63; scratch: scratch_bytes(n, ncols - n) bytes,
// 128-byte aligned. False (in every thread) when the block's numbers are out of the digits'
// range; A22 is then unchanged.
__device__ bool update(double2* M, int n, int ncols, int k0, unsigned char* scratch, unsigned char* stage, Shared& sh,
                       State& st, long long limit) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int kend = k0 + KO;
  const size_t ld = (size_t)n;
  const int rbn = row_blocks(n - kend), cbn = col_blocks(ncols - kend);
  unsigned char* A = scratch;
  unsigned char* B = A + (size_t)row_blocks(n) * A_STEPS * A_STAGE;
  int* er = reinterpret_cast<int*>(B + (size_t)col_blocks(ncols) * B_BLOCK);
  int* ec = er + row_blocks(n) * TM;
  if (!make_digits(M, n, ncols, k0, A, B, er, ec, sh)) return false;

  Tiles q{A, B, rbn, cbn, 0u, 0u};
  const int half = wid >> 2;
  const uint32_t t_addr = sh.tmem + ((uint32_t)(wid & 3) << 21) + (uint32_t)(half * 16);
  int tile = 0;
  for (; tile < cbn * rbn; ++tile) {
    const int rb = tile / cbn, cb = tile % cbn;
    if (tid == 0 && !issue_tile(stage, sh, st, limit)) *reinterpret_cast<volatile int*>(&sh.bad) = 1;
    if (tid == 32 && !copy_tile(q, tile, stage, sh, st, limit)) *reinterpret_cast<volatile int*>(&sh.bad) = 1;
    __syncwarp();  // (these warps' other lanes do not poll beside them)
    const int r = rb * TM + (wid & 3) * 32 + lane, c0 = cb * CN + half * 8;
    const bool in = kend + r < n;
    double2* C = M + (size_t)(kend + c0) * ld + kend + r;
    double2 c[8];
    int e[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      c[u] = in && kend + c0 + u < ncols ? C[(size_t)u * ld] : make_double2(0.0, 0.0);
      e[u] = ec[c0 + u];
    }
    const int e_row = er[r];
    bool ok = true;
    for (const long long t0 = clock64();;) {
      if (tcu::wait_parity(&sh.acc, st.acc & 1u, 0)) break;
      if (*reinterpret_cast<volatile int*>(&sh.bad) || clock64() - t0 > 4 * limit) {
        ok = false;
        break;
      }
    }
    if (!__syncthreads_and(ok)) break;
    __syncwarp();
    ++st.acc;
    tcu::fence_after();
    long long wr[8], wi[8];
    int hr[8], hi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) wr[u] = wi[u] = 0;
#pragma unroll
    for (int o = 0; o < ORDERS; ++o) {
      uint32_t g[16];
      tmem_ld16(t_addr + (uint32_t)(o * 2 * CN), g);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int gr = __float2int_rn(__uint_as_float(g[u])), gi = __float2int_rn(__uint_as_float(g[8 + u]));
        if (o < S - 1) {  // below 2^62 in units of order S - 2
          wr[u] = wr[u] * 256 + gr;
          wi[u] = wi[u] * 256 + gi;
        } else if (o == S - 1) {
          hr[u] = gr;
          hi[u] = gi;
        } else {  // the last two orders round into them
          wr[u] += (hr[u] * 256ll + gr + 32768) >> 16;
          wi[u] += (hi[u] * 256ll + gi + 32768) >> 16;
        }
      }
    }
    tcu::fence_before();
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      // digit d_s stands for d_s 256^(6 - s) 2^(e - BITS) on both sides
      const double sc = __hiloint2double((e_row + e[u] + 8 * S - 2 * BITS + 1023) << 20, 0);
      c[u].x = fma(-(double)wr[u], sc, c[u].x);
      c[u].y = fma(-(double)wi[u], sc, c[u].y);
      if (in && kend + c0 + u < ncols) C[(size_t)u * ld] = c[u];
    }
    __syncthreads();
    tcu::fence_after();
  }
  if (tile == cbn * rbn) return true;

  // a wait ran out: settle what is in flight, then the rest on the FMA pipes
  if (tid == 32) {
    sh.a_issued = st.a_issued;
    sh.b_issued = st.b_issued;
  }
  __syncthreads();
  if (tid == 0) {
    for (uint32_t i = st.b_used; i != sh.b_issued; ++i)
      tcu::wait_parity(&sh.b_full[i % B_RING], (i / B_RING) & 1u);
    for (uint32_t i = st.a_used; i != sh.a_issued; ++i) tcu::wait_parity(&sh.full[i % RING], (i / RING) & 1u);
    tcu::commit(&sh.last);
    tcu::wait_parity(&sh.last, 0);
  }
  st.on = false;
  __syncthreads();
  tcu::fence_after();
  for (; tile < cbn * rbn; ++tile) {
    const int r0 = kend + tile / cbn * TM, c0 = kend + tile % cbn * CN;
    for (int x = tid; x < TM * CN; x += THREADS) {
      const int i = r0 + x % TM, j = c0 + x / TM;
      if (i >= n || j >= ncols) continue;
      double2 v = M[(size_t)j * ld + i];
      for (int k = k0; k < kend; ++k) cfms(v, M[(size_t)k * ld + i], M[(size_t)j * ld + k]);
      M[(size_t)j * ld + i] = v;
    }
  }
  __syncthreads();
  return true;
}

}  // namespace ozlu
