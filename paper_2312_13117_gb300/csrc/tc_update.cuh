// Trailing update of the FP32 LU on the 5th-generation tensor cores.
//
// In the right-looking blocked LU (the factorisation step of every node solve,
// Eq. 2.4) almost all arithmetic is the update A22 -= L21 U12 after each
// 32-column panel. Here it runs as tcgen05.mma of kind::tf32 with the
// accumulators in tensor memory (TMEM):
//
//   * a complex product is four real ones, D_re = Lr Ur - Li Ui and
//     D_im = Li Ur + Lr Ui; the minus sign is the MMA's negate-A bit;
//   * each FP32 operand x is split into x_big = tf32(x) and
//     x_small = x - x_big ("3xTF32", see split), and every real product is
//     big*big + big*small + small*big, accumulated in FP32. The dropped
//     small*small term is below 2^-22 |x||y|, so the update has FP32-level
//     accuracy, which is what the FP64 refinement around the LU assumes;
//   * one tile is 128 rows (the MMA's M, one TMEM lane per row) by 32 columns;
//     D_re sits in TMEM columns 0..31 and D_im in 32..63 of one of two
//     accumulator buffers. The L21 tile is staged once per 128-row block and
//     reused across its column tiles;
//   * the column tiles of a row block are software-pipelined over two U12
//     buffers and two accumulators: while the tensor cores multiply tile t+1,
//     the threads stage the operands of tile t+2 and subtract tile t from C;
//     the C values of a tile are loaded before its MMAs are waited for;
//   * operands are K-major in the canonical no-swizzle layout: 8-row x 16-byte
//     core matrices, element (r, k) at (r/8)*SBO + (k/4)*LBO + (r%8)*16 + (k%4)*4
//     with LBO = 128 and SBO = 1024 bytes (32 TF32 values per row).
//
// Thread 0 issues the MMAs and commits them to an mbarrier; every wait on it is
// bounded. A wait that runs out sets the caller's flag and the rest of that
// panel's update is skipped; the CTA's later panels use the FMA pipes. The LU is
// then inexact, which the FP64 refinement around it either absorbs (it only
// needs an approximate inverse) or answers by solving the node again in FP64.
#pragma once
#include <cstddef>
#include <cstdint>

#include "lu_core.cuh"

namespace tcu {

constexpr int TM = 128;                  // tile rows = MMA M = TMEM lanes
constexpr int TN = 32;                   // tile columns = MMA N
constexpr int TK = 32;                   // panel width (complex) = lucore::NB
constexpr int LBO = 128;                 // bytes between core matrices along K
constexpr int SBO = (TK / 4) * 128;      // bytes between 8-row groups
constexpr int A_BYTES = TM * TK * 4;     // one real TF32 operand of L21: 16 KB
constexpr int B_BYTES = TN * TK * 4;     // one real TF32 operand of U12: 4 KB
constexpr int B_SET = 4 * B_BYTES;       // [Ur_big][Ui_big][Ur_small][Ui_small]
// [Lr_big][Li_big][Lr_small][Li_small] [U12 set 0] [U12 set 1]
constexpr int STAGE_BYTES = 4 * A_BYTES + 2 * B_SET;  // 96 KB
constexpr uint32_t ACC_COLS = 2 * TN;    // D_re, D_im of one tile
constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;  // two accumulators
constexpr long long WAIT_CYCLES = 1ll << 30;  // about half a second at 2 GHz

static_assert(TK == lucore::NB, "the tensor-core tile is one panel deep");
static_assert(lucore::THREADS == 256, "staging and epilogue assume 8 warps");

struct Ctx {
  unsigned char* stage;  // STAGE_BYTES of shared memory, 128-byte aligned
  uint64_t* mbar;        // two shared mbarriers (one per accumulator), count 1
  uint32_t tmem;         // TMEM address of the TMEM_COLS allocated columns
  uint32_t phase[2];     // parity of each barrier's next commit (the same in every thread)
  int* bad;              // shared flag: a wait ran out
  long long wait_cycles; // limit of one completion wait inside update()
  struct Wide* wide;     // shared barriers of update_wide
  uint32_t step;         // its next step (the same in every thread)
  const void* maps;      // tensor maps of the launch's matrices for blocks of L21 and of U12
  int slot;              // this matrix in them
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: start address, LBO, SBO, descriptor version 1,
// base offset 0, no swizzle.
__device__ __forceinline__ uint64_t desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(LBO >> 4) << 16) | ((uint64_t)(SBO >> 4) << 32) |
         (1ull << 46);
}

// Instruction descriptor of kind::tf32: F32 accumulator, TF32 A and B, both
// K-major, N = TN, M = TM, optional negation of A.
__device__ __forceinline__ uint32_t idesc(uint32_t neg_a) {
  return (1u << 4) | (2u << 7) | (2u << 10) | (neg_a << 13) | ((uint32_t)(TN >> 3) << 17) |
         ((uint32_t)(TM >> 4) << 24);
}

// Two TF32 parts of x: the nearest (ties away; integer arithmetic, as cvt.rna.tf32 runs at a
// quarter of its rate or less) and the rest, of which the tensor cores take the upper 11 bits
// (one less than its 12). A NaN stays in the rest.
__device__ __forceinline__ void split(float x, uint32_t& big, uint32_t& small) {
  big = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  small = __float_as_uint(x - __uint_as_float(big));
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t da, uint64_t db, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(da), "l"(db), "r"(id), "r"(acc));
}

__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ bool wait_parity(uint64_t* bar, uint32_t parity, long long limit = WAIT_CYCLES) {
  const uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Two 16-column loads of this warp's 32 TMEM lanes (the real and the imaginary
// part of 16 tile columns) and the wait for them, in one statement so that no
// use of the registers can move above the wait.
__device__ __forceinline__ void tmem_ld_pair(uint32_t a_re, uint32_t a_im, float (&re)[16], float (&im)[16]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a_re), "r"(a_im)
      : "memory");
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    re[c] = __uint_as_float(r[c]);
    im[c] = __uint_as_float(r[16 + c]);
  }
}

// Allocation of a power of two of columns, 32..512, by one whole warp, before a barrier that
// the warps using the columns also pass.
__device__ __forceinline__ void tmem_alloc_cols(uint32_t* dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_cols(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}

// Core-matrix offset (bytes) of the 16-byte group holding elements (r, 4q..4q+3).
__device__ __forceinline__ int core_off(int r, int q) { return (r >> 3) * SBO + q * LBO + (r & 7) * 16; }

__device__ __forceinline__ void st_v4(unsigned char* base, int off, const uint32_t (&v)[4]) {
  *reinterpret_cast<uint4*>(base + off) = make_uint4(v[0], v[1], v[2], v[3]);
}

// Stage L21 rows r0..r0+127 (columns k0..k0+kb-1) of the column-major matrix M
// (leading dimension ld, n rows). Thread t takes row t % 128 and the k-quads
// q = t / 128 + 2 i: a warp reads 32 consecutive rows of one column at a time.
__device__ __forceinline__ void stage_L(const float2* __restrict__ M, size_t ld, int n, int r0, int k0, int kb,
                                        unsigned char* st) {
  const int tid = lucore::gtid();
  const int r = tid & (TM - 1);
  const bool row_ok = r0 + r < n;
  float2 v[4][4];  // all 16 loads in flight before the first shared store
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int k = 4 * ((tid >> 7) + 2 * i) + t;
      v[i][t] = (row_ok && k < kb) ? M[(size_t)(k0 + k) * ld + r0 + r] : make_float2(0.f, 0.f);
    }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int q = (tid >> 7) + 2 * i;
    uint32_t rb[4], ib[4], rs[4], is[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      split(v[i][t].x, rb[t], rs[t]);
      split(v[i][t].y, ib[t], is[t]);
    }
    const int off = core_off(r, q);
    st_v4(st + 0 * A_BYTES, off, rb);
    st_v4(st + 1 * A_BYTES, off, ib);
    st_v4(st + 2 * A_BYTES, off, rs);
    st_v4(st + 3 * A_BYTES, off, is);
  }
}

// Stage U12 rows k0..k0+kb-1 of columns c0..c0+31 (bounded by ncols) into the
// U12 set at bset. Thread t takes column t % 32 and k-quad t / 32: four
// consecutive values of a column.
__device__ __forceinline__ void stage_U(const float2* __restrict__ M, size_t ld, int ncols, int c0, int k0, int kb,
                                        unsigned char* bset) {
  const int tid = lucore::gtid();
  const int c = tid & (TN - 1), q = tid >> 5;
  const bool col_ok = c0 + c < ncols;
  float2 v[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int k = 4 * q + t;
    v[t] = (col_ok && k < kb) ? M[(size_t)(c0 + c) * ld + k0 + k] : make_float2(0.f, 0.f);
  }
  uint32_t rb[4], ib[4], rs[4], is[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    split(v[t].x, rb[t], rs[t]);
    split(v[t].y, ib[t], is[t]);
  }
  const int off = core_off(c, q);
  st_v4(bset + 0 * B_BYTES, off, rb);
  st_v4(bset + 1 * B_BYTES, off, ib);
  st_v4(bset + 2 * B_BYTES, off, rs);
  st_v4(bset + 3 * B_BYTES, off, is);
}

// Thread 0: the 48 MMAs of one tile (3 split pairs x 4 real products x 4 K-steps
// of 8) from the L21 stage and U12 set b into accumulator b, then the commit
// to barrier b.
__device__ __forceinline__ void issue_tile(const Ctx& cx, int b) {
  const uint32_t sa = smem_u32(cx.stage), sb = sa + 4 * A_BYTES + (uint32_t)(b * B_SET);
  const uint32_t id_p = idesc(0), id_n = idesc(1);
  const uint32_t d_re = cx.tmem + (uint32_t)b * ACC_COLS, d_im = d_re + (uint32_t)TN;
  // (A split, B split): big*big, big*small, small*big
  const int pa[3] = {0, 0, 2}, pb[3] = {0, 2, 0};
  uint32_t acc = 0;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const uint32_t ar = sa + (pa[p] + 0) * A_BYTES, ai = sa + (pa[p] + 1) * A_BYTES;
    const uint32_t br = sb + (pb[p] + 0) * B_BYTES, bi = sb + (pb[p] + 1) * B_BYTES;
#pragma unroll
    for (int ks = 0; ks < TK / 8; ++ks) {
      const uint32_t o = (uint32_t)(ks * 2 * LBO);  // 8 TF32 = two core matrices along K
      mma(d_re, desc(ar + o), desc(br + o), id_p, acc);
      mma(d_re, desc(ai + o), desc(bi + o), id_n, 1u);
      mma(d_im, desc(ai + o), desc(br + o), id_p, acc);
      mma(d_im, desc(ar + o), desc(bi + o), id_p, 1u);
      acc = 1u;
    }
  }
  commit(cx.mbar + b);
}

// Shared-memory writes of the staging threads made visible to the tensor cores,
// and the group synchronised (tcgen05 ordering on both sides of the barrier).
__device__ __forceinline__ void stage_barrier() {
  fence_async_smem();
  fence_before();
  lucore::gsync();
  fence_after();
}

// Hint to bring the 128-byte line holding p into L2 (no register, no wait).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// L2 prefetch of what tile tt of the row block at r0 will load: its C values (32
// columns x 128 rows: one line per thread) and its U12 operand (32 columns x 32
// rows: two lines per column). Only addresses inside the matrix are touched.
__device__ __forceinline__ void prefetch_tile(const float2* M, size_t ld, int n, int ncols, int k0, int kend,
                                              int r0, int tt) {
  const int tid = lucore::gtid();
  const int c0 = kend + tt * TN;
  const int col = c0 + (tid >> 3), row = r0 + 16 * (tid & 7);
  if (col < ncols && row < n) prefetch_l2(M + (size_t)col * ld + row);
  if (tid < 2 * TN) {
    const int uc = c0 + (tid >> 1), ur = k0 + 16 * (tid & 1);
    if (uc < ncols && ur < kend) prefetch_l2(M + (size_t)uc * ld + ur);
  }
}

// L2 prefetch of the L21 rows r0..r0+127 of panel columns k0..k0+31 (one line per thread).
__device__ __forceinline__ void prefetch_L(const float2* M, size_t ld, int n, int k0, int kend, int r0) {
  const int tid = lucore::gtid();
  const int col = k0 + (tid >> 3), row = r0 + 16 * (tid & 7);
  if (col < kend && row < n) prefetch_l2(M + (size_t)col * ld + row);
}

// A22 -= L21 U12 for the panel k0..k0+kb-1 on the tensor cores. All threads of
// the group call it; it returns with the group synchronised and no MMA in
// flight, unless a wait ran out (then *cx.bad is set and the rest of the
// panel's update is skipped).
__device__ inline void update(float2* __restrict__ M, int n, int ncols, int k0, int kb, Ctx& cx) {
  const int tid = lucore::gtid(), warp = tid >> 5, lane = tid & 31;
  const size_t ld = (size_t)n;
  const int kend = k0 + kb;
  const int quad = warp & 3, half = warp >> 2;  // TMEM lanes 32*quad.., tile columns 16*half..
  const uint32_t lane_base = cx.tmem + ((uint32_t)(32 * quad) << 16);
  unsigned char* bset0 = cx.stage + 4 * A_BYTES;
  const int T = (ncols - kend + TN - 1) / TN;  // column tiles of a row block
  for (int r0 = kend; r0 < n; r0 += TM) {
    stage_L(M, ld, n, r0, k0, kb, cx.stage);
    stage_U(M, ld, ncols, kend, k0, kb, bset0);
    stage_barrier();
    if (tid == 0) issue_tile(cx, 0);
    const int row = r0 + 32 * quad + lane;
    for (int t = 0; t < T; ++t) {
      const int b = t & 1;
      const int c0 = kend + t * TN;
      // the lines of the tile two steps ahead (in this row block or the next) into L2
      if (t + 2 < T) prefetch_tile(M, ld, n, ncols, k0, kend, r0, t + 2);
      else if (r0 + TM < n && t + 2 - T < T) prefetch_tile(M, ld, n, ncols, k0, kend, r0 + TM, t + 2 - T);
      if (t + 3 == T && r0 + TM < n) prefetch_L(M, ld, n, k0, kend, r0 + TM);
      // this tile's C values, loaded while its MMAs run; issued first, so that their
      // latency overlaps that of the U12 loads below
      float2 cv[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int col = c0 + 16 * half + c;
        cv[c] = (row < n && col < ncols) ? M[(size_t)col * ld + row] : make_float2(0.f, 0.f);
      }
      // operands of tile t+1: its U12 set was last read by tile t-1's MMAs, complete
      if (t + 1 < T) stage_U(M, ld, ncols, c0 + TN, k0, kb, bset0 + (b ^ 1) * B_SET);
      const bool ok = wait_parity(cx.mbar + b, cx.phase[b], cx.wait_cycles);
      cx.phase[b] ^= 1u;
      if (!ok) atomicExch(cx.bad, 1);
      stage_barrier();  // tile t+1 staged; tile t-1's accumulator read by every thread
      if (*cx.bad) return;
      if (t + 1 < T && tid == 0) issue_tile(cx, b ^ 1);
      float re[16], im[16];
      const uint32_t acc = lane_base + (uint32_t)b * ACC_COLS;
      tmem_ld_pair(acc + (uint32_t)(16 * half), acc + (uint32_t)(TN + 16 * half), re, im);
      if (row < n) {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int col = c0 + 16 * half + c;
          if (col < ncols) M[(size_t)col * ld + row] = make_float2(cv[c].x - re[c], cv[c].y - im[c]);
        }
      }
      fence_before();  // this accumulator read is ordered before the next barrier
    }
    lucore::gsync();  // every epilogue store of the row block done before the next staging
  }
}

// ---------------------------------------------------------------------------
// The update of an outer block of up to 128 columns, A22 -= L21 U12 with K = 128.
//
// A rank-32 update reads and writes the whole trailing matrix for every panel (179 MB per
// node at n = 1024, 4.4 of 6.8 TB/s with its operands for two nodes per SM). Here a tile of
// 128 rows x 128 columns gathers the products of up to four panels in TMEM before it touches
// C. Measured, update phase of a node's LU with two nodes on the SM: n = 1024 12.3 -> 7.6 ms,
// n = 2048 92 -> 54 ms.
//
// With both operands in shared memory the products are bound by its bandwidth (128 B per
// clock: an MMA of M = 128, N = 64, K = 8 reads 6 KB, 48 clocks, for 32 clocks of
// arithmetic, and the staged operands have to be written there too). So the block of L21 goes
// to TMEM, and [Re | Im] of 64 columns lie side by side, D = Lr [Ur | Ui] + Li [-Ui | Ur] with
// N = 128: an MMA reads 4 KB for 64 clocks. A step is 16 inner indices of 64 columns, 12 MMAs.
// The blocks come by tensor copies into raw buffers (two steps ahead for L21, one for U12;
// plain loads have only the 28 KB of L1 that two CTAs' shared memory leaves for data in
// flight, and bulk copies of single columns cost some 40 clocks each to issue), and two teams
// split them: warps 4-7 L21 (into two TMEM buffers), warps 1-3 U12 (into both forms in two
// shared-memory buffers). Issuing an MMA blocks its thread while the queue is full, so warp 0
// does nothing else. All eight read the accumulators.
// ---------------------------------------------------------------------------
constexpr int OUTER = 128;                             // columns of an outer block
constexpr int WK = 16;                                 // inner indices of a step
constexpr int WN = 64;                                 // columns of a tile
constexpr int WSTEPS = OUTER / WK;                     // steps of a tile
constexpr int WB_BYTES = 2 * WN * WK * 4;              // one form and split part of U12: 8 KB
constexpr int WB_SET = 4 * WB_BYTES;                   // [form 0: big, small][form 1: big, small]
constexpr int WSBO = (WK / 4) * 128;                   // bytes between 8-row groups
constexpr int WRAW_L = 2, WRAW_U = 1;                  // raw buffers
constexpr int WL_RAW = TM * WK * 8, WU_RAW = WN * WK * 8;  // raw blocks: [k][row] 16 KB, [column][k] 8 KB
constexpr uint32_t WA_COLS = 4 * WK;                   // TMEM: [Lr big][Li big][Lr small][Li small]
constexpr uint32_t WIDE_COLS = 2 * WN + 2 * WA_COLS;   // accumulator, then two blocks of L21
constexpr int WIDE_STAGE = 2 * WB_SET + WRAW_L * WL_RAW + WRAW_U * WU_RAW;  // 104 KB
constexpr int WTEAM_U = 96, WTEAM_L = 128;             // warps 1-3, warps 4-7
constexpr int MAP_BYTES = 128;                          // a tensor map
static_assert(WTEAM_L == TM && WTEAM_L + WTEAM_U + 32 == lucore::THREADS, "teams");
struct Wide {
  uint64_t full[2];   // an arrival of every thread of the teams: step k is staged (k & 1)
  uint64_t empty[2];  // its products have ended
  uint64_t rawl[WRAW_L], rawu[WRAW_U];  // raw blocks have landed (step k: k % WRAW_*)
  uint64_t last;      // after a wait ran out: all products have ended
};

__device__ __forceinline__ void wide_init(Wide& w) {
  for (int i = 0; i < 2; ++i) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&w.full[i])), "r"(WTEAM_U + WTEAM_L)
                 : "memory");
    mbar_init(&w.empty[i]);
  }
  for (int i = 0; i < WRAW_L; ++i) mbar_init(&w.rawl[i]);
  for (int i = 0; i < WRAW_U; ++i) mbar_init(&w.rawu[i]);
  mbar_init(&w.last);
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Block of matrix z at column y, row x, zeros outside the matrix (x even: 16-byte boundaries).
__device__ __forceinline__ void tensor_copy(void* dst, const void* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}
// Wait for a phase; false (and *bad set) when it runs out, or once any wait of the CTA has.
__device__ __forceinline__ bool wait_unless_bad(uint64_t* bar, uint32_t parity, long long limit, int* bad) {
  const uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (*reinterpret_cast<volatile int*>(bad)) return false;
    if (clock64() - t0 > limit) {
      atomicExch(bad, 1);
      return false;
    }
  }
}
__device__ __forceinline__ uint64_t desc_wide(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(LBO >> 4) << 16) | ((uint64_t)(WSBO >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ int wide_off(int r, int q) { return (r >> 3) * WSBO + q * LBO + (r & 7) * 16; }

// The same product with A in tensor memory.
__device__ __forceinline__ void mma_ta(uint32_t d, uint32_t a, uint64_t db, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(db), "r"(id), "r"(acc));
}
// Sixteen columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(addr)
      : "memory");
}

// Thread 0: the products of a tile's steps. False when a wait ran out: nothing is in flight
// then.
__device__ inline bool issue_wide(const Ctx& cx) {
  const uint32_t id = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(2 * WN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  const int pa[3] = {0, 0, 2}, pb[3] = {0, 1, 0};  // (A split, B split): big*big, big*small, small*big
  Wide& w = *cx.wide;
  for (int i = 0; i < WSTEPS; ++i) {
    const uint32_t k = cx.step + i;
    if (!wait_unless_bad(&w.full[k & 1], (k >> 1) & 1u, cx.wait_cycles, cx.bad)) {
      commit(&w.last);
      wait_parity(&w.last, 0u, WAIT_CYCLES);
      return false;
    }
    fence_after();
    uint32_t acc = i > 0 ? 1u : 0u;
    const uint32_t ta = cx.tmem + 2 * WN + (k & 1) * WA_COLS, sb = smem_u32(cx.stage) + (k & 1) * WB_SET;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const uint32_t ar = ta + pa[p] * WK, ai = ar + WK;
      const uint32_t b0 = sb + pb[p] * WB_BYTES, b1 = b0 + 2 * WB_BYTES;
#pragma unroll
      for (int ks = 0; ks < WK / 8; ++ks) {
        const uint32_t o = (uint32_t)(ks * 2 * LBO);
        mma_ta(cx.tmem, ar + 8 * ks, desc_wide(b0 + o), id, acc);
        mma_ta(cx.tmem, ai + 8 * ks, desc_wide(b1 + o), id, 1u);
        acc = 1u;
      }
    }
    commit(&w.empty[k & 1]);
  }
  return true;
}

// The products of step k have ended (and so have all earlier ones).
__device__ __forceinline__ bool wide_wait(const Ctx& cx, uint32_t k) {
  const bool ok = wait_unless_bad(&cx.wide->empty[k & 1], (k >> 1) & 1u, cx.wait_cycles, cx.bad);
  fence_after();
  return ok;
}

// A tile of the update: rows r0 .., columns c0 ... ; r0 >= n: none.
struct WideTile {
  int r0, c0;
};

// Raw copies of step `step` (block i of a tile), by one thread.
__device__ __forceinline__ void copy_l(int n, int k0, WideTile tl, int i, uint32_t step, const Ctx& cx) {
  if (tl.r0 >= n) return;
  const uint32_t b = step % WRAW_L;
  mbar_expect(&cx.wide->rawl[b], WL_RAW);
  tensor_copy(cx.stage + 2 * WB_SET + b * WL_RAW, cx.maps, tl.r0, k0 + i * WK, cx.slot, &cx.wide->rawl[b]);
}
__device__ __forceinline__ void copy_u(int n, int k0, WideTile tl, int i, uint32_t step, const Ctx& cx) {
  if (tl.r0 >= n) return;
  const uint32_t b = step % WRAW_U;
  mbar_expect(&cx.wide->rawu[b], WU_RAW);
  tensor_copy(cx.stage + 2 * WB_SET + WRAW_L * WL_RAW + b * WU_RAW, static_cast<const char*>(cx.maps) + MAP_BYTES,
              k0 + i * WK, tl.c0, cx.slot, &cx.wide->rawu[b]);
}
// True in every thread of a team (named barrier id, count threads) when ok is true in all.
template <int ID, int COUNT>
__device__ __forceinline__ bool team_all(bool ok) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((int)ok), "n"(ID), "n"(COUNT)
      : "memory");
  return r != 0;
}
// After a wait ran out: the copies of steps from .. upto - 1 have landed (default limit).
template <int RAW>
__device__ __forceinline__ void settle_raw(uint64_t* bars, uint32_t from, uint32_t upto) {
  for (uint32_t k = from; k < upto; ++k) wait_parity(&bars[k % RAW], (k / RAW) & 1u);
}

// Warps 4-7: L21's blocks of tile tl; thread t holds row t and TMEM lane t. The copies run
// WRAW_L steps ahead, into the next tile nx; first: none is issued yet. False (the same in the
// whole team) when a wait ran out: its copies have landed then.
static __device__ __noinline__ bool stage_wide_l(int n, int k0, WideTile tl, WideTile nx, bool first, int t,
                                                 const Ctx& cx) {
  const uint32_t lane_base = cx.tmem + 2 * WN + ((uint32_t)(t & ~31) << 16);
  if (first && t == 0)
    for (int i = 0; i < WRAW_L; ++i) copy_l(n, k0, tl, i, cx.step + i, cx);
  for (int i = 0; i < WSTEPS; ++i) {
    const uint32_t step = cx.step + i, b = step & 1, rb = step % WRAW_L;
    bool ok = wait_unless_bad(&cx.wide->rawl[rb], (step / WRAW_L) & 1u, cx.wait_cycles, cx.bad);
    float2 v[WK];
    const float2* raw = reinterpret_cast<const float2*>(cx.stage + 2 * WB_SET + rb * WL_RAW) + t;
#pragma unroll
    for (int q = 0; q < WK; ++q) v[q] = raw[q * TM];
    ok = ok && (step < 2 || wide_wait(cx, step - 2));  // the TMEM buffer's last products have ended
    if (!team_all<2, WTEAM_L>(ok)) {                    // (every thread has read the raw block)
      const int left = WSTEPS - i;                      // this tile's blocks, then the next one's
      settle_raw<WRAW_L>(cx.wide->rawl, step, step + (nx.r0 < n ? WRAW_L : min(WRAW_L, left)));
      return false;
    }
    if (t == 0) {
      if (i + WRAW_L < WSTEPS) copy_l(n, k0, tl, i + WRAW_L, step + WRAW_L, cx);
      else copy_l(n, k0, nx, i + WRAW_L - WSTEPS, step + WRAW_L, cx);
    }
    uint32_t big[WK], small[WK];
    const uint32_t ta = lane_base + b * WA_COLS;
#pragma unroll
    for (int q = 0; q < WK; ++q) split(v[q].x, big[q], small[q]);
    tmem_st16(ta, big);
    tmem_st16(ta + 2 * WK, small);
#pragma unroll
    for (int q = 0; q < WK; ++q) split(v[q].y, big[q], small[q]);
    tmem_st16(ta + WK, big);
    tmem_st16(ta + 3 * WK, small);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    fence_before();
    mbar_arrive(&cx.wide->full[b]);
  }
  return true;
}

// Warps 1-3: U12's blocks of tile tl, in units of four inner indices of a column.
static __device__ __noinline__ bool stage_wide_u(int n, int k0, WideTile tl, WideTile nx, bool first, int t,
                                                 const Ctx& cx) {
  constexpr int UNITS = WN * WK / 4, ROUNDS = (UNITS + WTEAM_U - 1) / WTEAM_U;
  if (first && t == 0)
    for (int i = 0; i < WRAW_U; ++i) copy_u(n, k0, tl, i, cx.step + i, cx);
  for (int i = 0; i < WSTEPS; ++i) {
    const uint32_t step = cx.step + i, b = step & 1, rb = step % WRAW_U;
    bool ok = wait_unless_bad(&cx.wide->rawu[rb], (step / WRAW_U) & 1u, cx.wait_cycles, cx.bad);
    float4 v[ROUNDS][2];
    const float4* raw = reinterpret_cast<const float4*>(cx.stage + 2 * WB_SET + WRAW_L * WL_RAW + rb * WU_RAW);
#pragma unroll
    for (int u = 0; u < ROUNDS; ++u) {
      const int e = t + u * WTEAM_U;  // column e / 4, inner indices 4 (e % 4) ..
      v[u][0] = e < UNITS ? raw[2 * e] : make_float4(0.f, 0.f, 0.f, 0.f);
      v[u][1] = e < UNITS ? raw[2 * e + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    ok = ok && (step < 2 || wide_wait(cx, step - 2));  // the forms' last products have ended
    if (!team_all<3, WTEAM_U>(ok)) {                    // (every thread has read the raw block)
      const int left = WSTEPS - i;
      settle_raw<WRAW_U>(cx.wide->rawu, step, step + (nx.r0 < n ? WRAW_U : min(WRAW_U, left)));
      return false;
    }
    if (t == 0) {
      if (i + WRAW_U < WSTEPS) copy_u(n, k0, tl, i + WRAW_U, step + WRAW_U, cx);
      else copy_u(n, k0, nx, i + WRAW_U - WSTEPS, step + WRAW_U, cx);
    }
    unsigned char* bst = cx.stage + b * WB_SET;
#pragma unroll
    for (int u = 0; u < ROUNDS; ++u) {
      const int e = t + u * WTEAM_U;
      if (e < UNITS) {
        const float re4[4] = {v[u][0].x, v[u][0].z, v[u][1].x, v[u][1].z};
        const float im4[4] = {v[u][0].y, v[u][0].w, v[u][1].y, v[u][1].w};
        uint32_t rb4[4], ib[4], rs[4], is[4], nb[4], ns[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          split(re4[q], rb4[q], rs[q]);
          split(im4[q], ib[q], is[q]);
          nb[q] = ib[q] ^ 0x80000000u;
          ns[q] = is[q] ^ 0x80000000u;
        }
        const int re = wide_off(e >> 2, e & 3), im = wide_off(WN + (e >> 2), e & 3);
        st_v4(bst + 0 * WB_BYTES, re, rb4);
        st_v4(bst + 0 * WB_BYTES, im, ib);
        st_v4(bst + 1 * WB_BYTES, re, rs);
        st_v4(bst + 1 * WB_BYTES, im, is);
        st_v4(bst + 2 * WB_BYTES, re, nb);
        st_v4(bst + 2 * WB_BYTES, im, rb4);
        st_v4(bst + 3 * WB_BYTES, re, ns);
        st_v4(bst + 3 * WB_BYTES, im, rs);
      }
    }
    fence_async_smem();
    mbar_arrive(&cx.wide->full[b]);
  }
  return true;
}

// The update of outer block k0 .. k0+127 of an n x ncols matrix (n even, k0 a multiple of 128). Returns with the CTA synchronised and neither an MMA nor a copy in
// flight; when a wait ran out *cx.bad is set and the rest of the update is skipped.
static __device__ __noinline__ void update_wide(float2* __restrict__ M, int n, int ncols, int k0, Ctx& cx) {
  const int tid = lucore::gtid(), warp = tid >> 5, lane = tid & 31;
  const size_t ld = (size_t)n;
  const int kend = k0 + OUTER;
  const int quad = warp & 3, half = warp >> 2;
  const uint32_t lane_base = cx.tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(half * (WN / 2));
  // L21 and U12 were written by plain stores and are read by bulk copies
  asm volatile("fence.proxy.async;" ::: "memory");
  lucore::gsync();
  bool first = true;
  bool done = false;  // this thread's team has staged the tile, and issued the next one's first copies
  for (WideTile tl{kend, kend}; tl.r0 < n;) {
    WideTile nx{tl.r0, tl.c0 + WN};
    if (nx.c0 >= ncols) nx = WideTile{tl.r0 + TM, kend};
    if (warp == 0) {
      if (lane == 0) issue_wide(cx);
      __syncwarp();
    } else if (warp < 4) {
      done = stage_wide_u(n, k0, tl, nx, first, tid - 32, cx);
    } else {
      // this tile's C lines into L2 while its products run
#pragma unroll
      for (int u = 0; u < WN * TM / 16 / WTEAM_L; ++u) {
        const int e = tid - 128 + u * WTEAM_L, col = tl.c0 + (e >> 3), row = tl.r0 + 16 * (e & 7);
        if (col < ncols && row < n) prefetch_l2(M + (size_t)col * ld + row);
      }
      done = stage_wide_l(n, k0, tl, nx, first, tid - 128, cx);
    }
    first = false;
    cx.step += WSTEPS;
    lucore::gsync();
    const int staged = *reinterpret_cast<volatile int*>(cx.bad) == 0;
    lucore::gsync();  // every thread has read it before the next wait can set it
    if (staged) wide_wait(cx, cx.step - 1);
    lucore::gsync();
    if (*reinterpret_cast<volatile int*>(cx.bad)) {  // (not set again before the next barrier)
      if (done && nx.r0 < n) {
        if (warp < 4) settle_raw<WRAW_U>(cx.wide->rawu, cx.step, cx.step + WRAW_U);
        else settle_raw<WRAW_L>(cx.wide->rawl, cx.step, cx.step + WRAW_L);
      }
      lucore::gsync();
      return;
    }
    const int row = tl.r0 + 32 * quad + lane;
#pragma unroll 1
    for (int h = 0; h < WN / 2; h += 16) {
      const int cb = tl.c0 + half * (WN / 2) + h;
      float2 cv[16];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        cv[c] = row < n && cb + c < ncols ? M[(size_t)(cb + c) * ld + row] : make_float2(0.f, 0.f);
      float re[16], im[16];
      tmem_ld_pair(lane_base + (uint32_t)h, lane_base + (uint32_t)(WN + h), re, im);
      if (row < n) {
#pragma unroll
        for (int c = 0; c < 16; ++c)
          if (cb + c < ncols) M[(size_t)(cb + c) * ld + row] = make_float2(cv[c].x - re[c], cv[c].y - im[c]);
      }
    }
    fence_before();  // the accumulators are read before the next tile's first products
    lucore::gsync();
    fence_after();
    tl = nx;
  }
}

}  // namespace tcu
