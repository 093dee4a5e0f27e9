// Refinement residuals of all active nodes of a chunk on the tensor cores.
//
// R_j = V - id_j X_j - sum_d A_d (f_d(z_j) X_j) with the exact digit products of
// ozaki.cuh. The coefficients A_d are the same for every node of a problem, so the
// products of all nodes are one matrix product per term, A_d [Y_1 | Y_2 | ...]:
// a tile takes 128 rows and up to four groups of 8 solution columns of any active
// nodes (N = 64 accumulator columns, real and imaginary parts side by side in each
// group). Against a product per node (N = 32, half of it padding at 8 columns, one
// CTA per node) the coefficient digits are read once for 32 columns and an MMA has
// twice the columns for the same operand A, whose shared-memory reads (4 KB, 32
// clocks) bound it at N = 32.
//
// One persistent CTA per SM, warp-specialised:
//   warp 0        bulk copies: coefficient digits through a ring of NA 16 KB stages,
//                 the digits of f_d X (14 KB per group and 32 inner indices) two deep;
//   warp 1        MMAs into all 512 TMEM columns: 8 digit orders x 64 columns;
//   warps 4-19    drains, after every 256 inner indices. A warp owns 32 rows and one
//                 column group, and forms what ozk::residual forms, in the same order and
//                 to the same bits: Horner's rule over the orders in double-float, then
//                 one FP64 update of R (kept in registers) per 256 inner indices, which
//                 overlaps the next products.
// A boundary-integral node has a matrix of its own: its tiles hold its own groups only,
// and the digits are those of T(z_j) (bie_nodes.cu). Its rows hold numbers of very
// different sizes (H_1 grows like e^{-Im w}), and its residuals take the place of FP64
// ones, so it gets 8 digits (55 bits of a row's largest number) and the pairs of total
// order <= 10, in 9 accumulators and at most three groups a tile. Errors of such a residual
// relative to |X|, n = 34, z = 2 - 2.8 i: 5.1e-16 (plain FP64 1.1e-15, 7 digits 7.9e-14);
// 100 disks of 64 nodes at n = 256, l = 8 take 46.6 ms in all (45.3 with 7 digits).
// A wait for operands is bounded by tc_wait_cycles: when one runs out the CTA's nodes
// are marked, and solved again in FP64. A wait between the warps is bounded by
// handoff_wait_cycles: when one runs out the launch fails (MixedArgs::err).
#include "ozaki.cuh"

namespace {

using namespace ozk;

constexpr int CG = 8;                     // solution columns of a group
// The digits of a form of products: dense terms (ozaki.cuh), or a boundary-integral node's T(z_j).
template <bool BIE>
struct Form {
  static constexpr int S = BIE ? 8 : ozk::S, QMAX = BIE ? 10 : ozk::QMAX, NQ = QMAX - 1;
  static constexpr int SHIFT = 7 * S - 1;   // a number's integer is rint(x 2^(SHIFT - exponent))
  static constexpr int SCALE = 2 * SHIFT - 7 * (2 * S - QMAX);  // weight of the last order, 2^(e + g - SCALE)
  static constexpr int MAXG = BIE ? 3 : 4;  // groups of a tile
  static constexpr int STAGE = 2 * CG * KC * 2 * 2 * S;  // a group's digits of 32 inner indices: 14 or 16 KB
  static constexpr int PART = STAGE / 2;                 // [real rows][imaginary rows]
};
static_assert(Form<false>::SHIFT == DIGIT_SHIFT && Form<false>::SCALE == DRAIN_SCALE, "the coefficients' digits");
static_assert(Form<true>::S == BIE_DIGITS, "T(z_j)'s digits");
static_assert(Form<true>::NQ * 16 * Form<true>::MAXG <= 512 && Form<false>::NQ * 16 * Form<false>::MAXG <= 512,
              "TMEM columns");
static_assert(8 * 2 * KD * 64 * 64 <= (1 << 24), "tensor-core partial sums must stay exact in FP32");
constexpr int RA = 6;                     // A stages
constexpr int RB2 = 2;                    // B stages
constexpr int DRAIN_WARP0 = 4, DRAIN_WARPS = 16;
constexpr int GEMM_THREADS = 32 * (DRAIN_WARP0 + DRAIN_WARPS);
constexpr int DIGIT_THREADS = 256;

// Byte offset of digit t, form f (0: [Yr | Yi], 1: [-Yi | Yr]), part p (of `part` bytes) (0: the real
// accumulator rows, 1: the imaginary ones), column c, inner index k of a group's stage.
// Consecutive 8-row blocks of a tile's operand are `part` bytes apart in every (t, f).
__device__ __forceinline__ int stage_off(int part, int t, int f, int p, int c, int k) {
  return p * part + (t * 2 + f) * 512 + (k >> 3) * 128 + c * 16 + (k & 7) * 2;
}

// 2^e, exact for every e that a double holds.
__device__ __forceinline__ double pow2(int e) {
  return (e >= -1022 && e <= 1023) ? __hiloint2double((e + 1023) << 20, 0) : scalbn(1.0, e);
}

// Matrices a problem's residual multiplies: its dense terms, or T(z_j).
__device__ __forceinline__ int terms_of(const ProblemDev& P) { return P.bie ? 1 : P.n_dense; }

// Digits of f_d X of the active nodes, one CTA per node and dense term; CTA 0 also
// counts the residual tiles before each problem, by form.
__global__ void __launch_bounds__(DIGIT_THREADS) k_oz_digits(MixedArgs a, int sw, int max_dense) {
  __shared__ double red[DIGIT_THREADS];
  __shared__ int g[CG];
  __shared__ double2 f_sh;
  const int tid = threadIdx.x;
  const int active = a.ctl[MIXED_CTL_ACTIVE + sw];
  if (blockIdx.x == 0 && tid < 32) {
    const int* uc = mixed_ucount(a, sw);
    for (int f = 0; f < 2; ++f) {
      int* tiles = mixed_tiles(a, f != 0);
      int base = 0;
      for (int p0 = 0; p0 < a.n_probs; p0 += 32) {
        const int p = p0 + tid;
        int v = 0;
        if (p < a.n_probs && (a.probs[p].bie != nullptr) == (f != 0)) {
          // problems share their tiles among nodes; a boundary-integral node has its own
          const int ncg = (a.probs[p].l + CG - 1) / CG;
          constexpr int GB = Form<true>::MAXG, GD = Form<false>::MAXG;
          v = (f ? uc[p] / ncg * ((ncg + GB - 1) / GB) : (uc[p] + GD - 1) / GD) * row_blocks(a.probs[p].n);
        }
        const int own = v;
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(0xffffffffu, v, o);
          if (tid >= o) v += x;
        }
        if (p < a.n_probs) tiles[p] = base + v - own;
        base += __shfl_sync(0xffffffffu, v, 31);
      }
      if (tid == 0) tiles[a.n_probs] = base;
    }
  }
  for (int w = blockIdx.x; w < active * max_dense; w += gridDim.x) {
    const int q = a.act[(size_t)(sw & 1) * a.slots + w / max_dense], dd = w % max_dense;
    const NodeItem it = a.items[q];
    const RegionDev rg = a.regions[it.region];
    const ProblemDev& P = a.probs[rg.prob];
    if (dd >= terms_of(P) || !mixed_node_oz(a, P, rg)) continue;  // the same in every thread
    const int n = P.n, l = P.l, kcn = k_chunks(n), ncg = (l + CG - 1) / CG;
    const int digits = P.bie ? Form<true>::S : Form<false>::S, stage = P.bie ? Form<true>::STAGE : Form<false>::STAGE;
    __syncthreads();  // f_sh and g of the previous node
    if (tid == 0) {
      if (P.bie) {
        f_sh = make_double2(1.0, 0.0);
      } else {
        int k = 0;
        for (int d = -1; k < P.K; ++k)
          if (P.term[k].dense && ++d == dd) break;
        double2 z, wt;
        node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &wt);
        f_sh = eval_f(P.term[k], z);
      }
    }
    __syncthreads();
    const double2 f = f_sh;
    const double2* X = a.X + rg.x_off + (size_t)it.j * n * l;
    for (int cg = 0; cg < ncg; ++cg) {
      {
        const int c = cg * CG + (tid & (CG - 1));
        double m = 0.0;
        if (c < l)
          for (int j = tid / CG; j < n; j += DIGIT_THREADS / CG) {
            const double2 y = y_product(f, X[(size_t)c * n + j]);
            m = fmax(m, fmax(fabs(y.x), fabs(y.y)));
          }
        for (int o = CG; o < 32; o <<= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        __syncthreads();  // red and g of the previous group
        if ((tid & 31) < CG) red[(tid >> 5) * CG + (tid & (CG - 1))] = m;
        __syncthreads();
        if (tid < CG) {
          double mm = 0.0;
          for (int k = 0; k < DIGIT_THREADS / 32; ++k) mm = fmax(mm, red[k * CG + tid]);
          g[tid] = exponent_of(mm);
          a.gexp[(size_t)q * a.gexp_stride + (dd * ncg + cg) * CG + tid] = g[tid];
        }
        __syncthreads();
      }
      unsigned char* dst = a.ysl + (size_t)q * a.ysl_stride + (size_t)(dd * ncg + cg) * kcn * stage;
      for (int task = tid; task < CG * kcn * (KC / 8); task += DIGIT_THREADS) {
        const int cc = task & (CG - 1), j0 = (task / CG) * 8, c = cg * CG + cc;
        const int shift = 7 * digits - 1 - g[cc];
        const bool normal = shift >= -1022 && shift <= 1023;  // 2^shift is a normal number
        const double up = normal ? pow2(shift) : 0.0;
        long long Nr[8], Ni[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          double2 y = make_double2(0.0, 0.0);
          if (c < l && j0 + u < n) y = y_product(f, X[(size_t)c * n + j0 + u]);
          Nr[u] = __double2ll_rn(normal ? y.x * up : scalbn(y.x, shift));
          Ni[u] = __double2ll_rn(normal ? y.y * up : scalbn(y.y, shift));
        }
        unsigned char* st = dst + (size_t)(j0 / KC) * stage;
#pragma unroll 1
        for (int t = digits - 1; t >= 0; --t) {
          uint32_t pr[4], pi[4], nr[4];
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            const int r0 = next_digit(Nr[u], t), r1 = next_digit(Nr[u + 1], t);
            const int i0 = next_digit(Ni[u], t), i1 = next_digit(Ni[u + 1], t);
            pr[u / 2] = (uint32_t)bf16_of_int(r0) | ((uint32_t)bf16_of_int(r1) << 16);
            pi[u / 2] = (uint32_t)bf16_of_int(i0) | ((uint32_t)bf16_of_int(i1) << 16);
            nr[u / 2] = (uint32_t)bf16_of_int(-i0) | ((uint32_t)bf16_of_int(-i1) << 16);
          }
          const int k = j0 % KC;
          *reinterpret_cast<uint4*>(st + stage_off(stage / 2, t, 0, 0, cc, k)) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
          *reinterpret_cast<uint4*>(st + stage_off(stage / 2, t, 0, 1, cc, k)) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
          *reinterpret_cast<uint4*>(st + stage_off(stage / 2, t, 1, 0, cc, k)) = make_uint4(nr[0], nr[1], nr[2], nr[3]);
          *reinterpret_cast<uint4*>(st + stage_off(stage / 2, t, 1, 1, cc, k)) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
        }
      }
    }
  }
}

template <bool BIE>
struct GemmSmem {
  alignas(1024) unsigned char a[RA][A_STAGE];
  alignas(1024) unsigned char b[RB2][Form<BIE>::MAXG * Form<BIE>::STAGE];
  uint64_t a_full[RA], a_empty[RA], b_full[RB2], b_empty[RB2], acc_full, acc_empty, last;
  uint32_t a_issued, b_issued;  // copies issued, for the settling wait
  uint32_t tmem;
  int bad;  // a wait ran out
};

// A tile: row block rb of problem p, groups units[0 .. ng).
struct Tile {
  int p, rb, ng;
  const int* units;
};

// Walks this CTA's tiles (blockIdx.x, + gridDim.x, ...) in order.
template <bool BIE>
struct TileWalk {
  const MixedArgs& a;
  const int* tiles;
  const int* uc;
  int sw, t, p;
  __device__ TileWalk(const MixedArgs& a_, int sw_)
      : a(a_), tiles(mixed_tiles(a_, BIE)), uc(mixed_ucount(a_, sw_)), sw(sw_), t((int)blockIdx.x), p(0) {}
  __device__ bool next(Tile& out) {
    if (t >= tiles[a.n_probs]) return false;
    while (tiles[p + 1] <= t) ++p;
    const int rbn = row_blocks(a.probs[p].n), loc = t - tiles[p];
    constexpr int MAXG = Form<BIE>::MAXG;
    int u0 = loc / rbn * MAXG, end = uc[p];
    if (BIE) {  // a node's groups are consecutive
      const int ncg = (a.probs[p].l + CG - 1) / CG, per = (ncg + MAXG - 1) / MAXG, node = loc / rbn / per;
      u0 = node * ncg + loc / rbn % per * MAXG;
      end = (node + 1) * ncg;
    }
    out.p = p;
    out.rb = loc % rbn;
    out.ng = min(MAXG, end - u0);
    out.units = a.units + (size_t)(sw & 1) * a.unit_cap + a.ubase[p] + u0;
    t += gridDim.x;
    return true;
  }
};

__device__ __forceinline__ void init_count(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tcu::smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(tcu::smem_u32(bar))
               : "memory");
}

enum { LOST_OPERANDS = 1, LOST_HANDOFF = 2 };  // which wait of the CTA ran out first

// Wait for a phase; false once any wait of the CTA has run out.
__device__ __forceinline__ bool wait_or_bad(uint64_t* bar, uint32_t parity, long long limit, int* bad,
                                            int which = LOST_OPERANDS) {
  const uint32_t addr = tcu::smem_u32(bar);
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (*reinterpret_cast<volatile int*>(bad)) return false;
    if (clock64() - t0 > limit) {
      atomicCAS(bad, 0, which);
      return false;
    }
  }
}

// Shared-memory descriptors: K-major, no swizzle, LBO 128 B; 8-row blocks SBO apart.
__device__ __forceinline__ uint64_t desc_sbo(uint32_t addr, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
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

// warp 0, one lane
template <bool BIE>
__device__ void copy_role(const MixedArgs& a, int sw, GemmSmem<BIE>& sm) {
  constexpr int S = Form<BIE>::S, MAXG = Form<BIE>::MAXG, STAGE = Form<BIE>::STAGE;
  TileWalk<BIE> walk(a, sw);
  Tile t;
  uint32_t na = 0, nb = 0;
  bool ok = true;
  while (ok && walk.next(t)) {
    const ProblemDev& P = a.probs[t.p];
    const int rbn = row_blocks(P.n), kcn = k_chunks(P.n), ncg = (P.l + CG - 1) / CG;
    const unsigned char* src[MAXG];
    for (int g = 0; g < t.ng; ++g)
      src[g] = a.ysl + (size_t)(t.units[g] >> 3) * a.ysl_stride + (size_t)(t.units[g] & 7) * kcn * STAGE;
    const unsigned char* digits = BIE ? a.tdig + (size_t)(t.units[0] >> 3) * a.tdig_stride : P.Adig;
    for (int dd = 0; dd < terms_of(P) && ok; ++dd) {
      const unsigned char* asrc = digits + ((size_t)dd * rbn + t.rb) * kcn * S * A_STAGE;
      for (int kc = 0; kc < kcn && ok; ++kc) {
        const uint32_t bi = nb % RB2, bk = nb / RB2;
        ok = bk == 0 || wait_or_bad(&sm.b_empty[bi], (bk - 1) & 1u, a.tc_wait_cycles, &sm.bad);
        if (!ok) break;
        expect_tx(&sm.b_full[bi], (uint32_t)t.ng * STAGE);
        for (int g = 0; g < t.ng; ++g)
          bulk_g2s(sm.b[bi] + g * STAGE, src[g] + ((size_t)dd * ncg * kcn + kc) * STAGE, STAGE, &sm.b_full[bi]);
        ++nb;
        for (int s = 0; s < S; ++s) {
          const uint32_t ai = na % RA, ak = na / RA;
          ok = ak == 0 || wait_or_bad(&sm.a_empty[ai], (ak - 1) & 1u, a.tc_wait_cycles, &sm.bad);
          if (!ok) break;
          expect_tx(&sm.a_full[ai], A_STAGE);
          bulk_g2s(sm.a[ai], asrc + ((size_t)kc * S + s) * A_STAGE, A_STAGE, &sm.a_full[ai]);
          ++na;
        }
      }
    }
  }
  sm.a_issued = na;
  sm.b_issued = nb;
}

// warp 1, one lane
template <bool BIE>
__device__ void mma_role(const MixedArgs& a, int sw, GemmSmem<BIE>& sm) {
  constexpr int S = Form<BIE>::S, QMAX = Form<BIE>::QMAX, MAXG = Form<BIE>::MAXG, PART = Form<BIE>::PART;
  TileWalk<BIE> walk(a, sw);
  Tile t;
  uint32_t na = 0, nb = 0, blk = 0;
  bool ok = true;
  while (ok && walk.next(t)) {
    const ProblemDev& P = a.probs[t.p];
    const int kcn = k_chunks(P.n);
    // kind::f16, F32 accumulator, BF16 A and B, K-major, M = 128, N = 16 per group
    const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(t.ng * 2) << 17) | ((uint32_t)(TM >> 4) << 24);
    for (int dd = 0; dd < terms_of(P) && ok; ++dd)
      for (int kc0 = 0; kc0 < kcn && ok; kc0 += KD / KC) {
        ok = blk == 0 || wait_or_bad(&sm.acc_empty, (blk - 1) & 1u, a.handoff_wait_cycles, &sm.bad, LOST_HANDOFF);
        if (!ok) break;
        tcu::fence_after();
        uint32_t used = 0;
        const int kc1 = min(kcn, kc0 + KD / KC);
        for (int kc = kc0; kc < kc1 && ok; ++kc) {
          const uint32_t bi = nb % RB2;
          ok = wait_or_bad(&sm.b_full[bi], (nb / RB2) & 1u, a.tc_wait_cycles, &sm.bad);
          for (int s = 0; s < S && ok; ++s) {
            const uint32_t ai = na % RA;
            ok = wait_or_bad(&sm.a_full[ai], (na / RA) & 1u, a.tc_wait_cycles, &sm.bad);
            if (!ok) break;
            tcu::fence_after();
            const uint32_t ab = tcu::smem_u32(sm.a[ai]), bb = tcu::smem_u32(sm.b[bi]);
            for (int u = 0; u + s + 2 <= QMAX && u < S; ++u) {
              const int qi = s + u;  // digit order q - 2
              const uint32_t d = sm.tmem + (uint32_t)(qi * 16 * MAXG);
#pragma unroll
              for (int ks = 0; ks < KC / 16; ++ks) {
                const uint32_t o = (uint32_t)(ks * 256);  // 16 BF16 = two core matrices along K
                mma(d, desc_sbo(ab + o, 512), desc_sbo(bb + u * 1024 + o, PART), id, (used >> qi) & 1u);
                mma(d, desc_sbo(ab + A_TILE + o, 512), desc_sbo(bb + u * 1024 + 512 + o, PART), id, 1u);
                used |= 1u << qi;
              }
            }
            tcu::commit(&sm.a_empty[ai]);
            ++na;
          }
          if (ok) {
            tcu::commit(&sm.b_empty[bi]);
            ++nb;
          }
        }
        if (ok) tcu::commit(&sm.acc_full);
        ++blk;
      }
  }
  // every product has ended before the CTA gives its memory back
  tcu::commit(&sm.last);
  tcu::wait_parity(&sm.last, 0u, tcu::WAIT_CYCLES);
}

// warps 4-19
template <bool BIE>
__device__ void drain_role(const MixedArgs& a, int sw, GemmSmem<BIE>& sm) {
  constexpr int NQ = Form<BIE>::NQ, MAXG = Form<BIE>::MAXG;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quad = warp & 3, gi = (warp - DRAIN_WARP0) >> 2;
  const uint32_t base = sm.tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(16 * gi);
  TileWalk<BIE> walk(a, sw);
  Tile t;
  uint32_t blk = 0;
  while (walk.next(t)) {
    const ProblemDev& P = a.probs[t.p];
    const int n = P.n, l = P.l, rbn = row_blocks(n), kcn = k_chunks(n), ncg = (l + CG - 1) / CG;
    const bool mine = gi < t.ng;
    const int row = t.rb * TM + 32 * quad + lane;
    const int unit = mine ? t.units[gi] : 0, q = unit >> 3, cg = unit & 7;
    const NodeItem it = a.items[q];
    const RegionDev rg = a.regions[it.region];
    const double2* X = a.X + rg.x_off + (size_t)it.j * n * l + (size_t)cg * CG * n + row;
    double2* R = reinterpret_cast<double2*>(a.work + (size_t)q * a.slot_bytes + mixed_residual_offset(n, l)) +
                 (size_t)cg * CG * n + row;
    const int cols = min(CG, l - cg * CG);
    if constexpr (BIE) {
      // exact sums of the orders' upper and lower part over all inner indices
      constexpr int NHI = NQ - 4;
      long long hi[2 * CG], lo[2 * CG];  // hi 2^28 + lo, in units of the last order
#pragma unroll
      for (int c = 0; c < 2 * CG; ++c) hi[c] = lo[c] = 0;
      for (int kc0 = 0; kc0 < kcn; kc0 += KD / KC) {
        const bool ok = wait_or_bad(&sm.acc_full, blk & 1u, a.handoff_wait_cycles, &sm.bad, LOST_HANDOFF);
        if (!__all_sync(0xffffffffu, ok)) return;  // sm.bad is set
        ++blk;
        tcu::fence_after();
        if (mine) {
#pragma unroll
          for (int h = 0; h < NQ; ++h) {
            uint32_t v[16];
            tmem_ld16(base + (uint32_t)(h * 16 * MAXG), v);
#pragma unroll
            for (int c = 0; c < 2 * CG; ++c) {
              const long long d = (long long)__float2int_rn(__uint_as_float(v[c]));
              if (h < NHI) hi[c] += d * (1 << (7 * (NHI - 1 - h)));
              else lo[c] += d * (1 << (7 * (NQ - 1 - h)));
            }
          }
        }
        tcu::fence_before();
        __syncwarp();
        if (lane == 0) arrive(&sm.acc_empty);
      }
      if (mine && row < n) {
        const int er = a.texp[(size_t)q * a.texp_stride + t.rb * TM + 32 * quad + lane];
        const int* ge = a.gexp + (size_t)q * a.gexp_stride + cg * CG;
#pragma unroll
        for (int c = 0; c < CG; ++c) {
          if (c < cols) {
            double2 v = P.V[(size_t)(cg * CG + c) * n + row];
            const int e = er + ge[c] - Form<true>::SCALE;
            const double s1 = -pow2(e), s2 = -pow2(e + 28);
            v.x = fma(s2, (double)hi[c], fma(s1, (double)lo[c], v.x));
            v.y = fma(s2, (double)hi[CG + c], fma(s1, (double)lo[CG + c], v.y));
            R[(size_t)c * n] = v;
          }
        }
      }
      continue;
    }
    double r[2 * CG];  // R's columns of the group: real parts, imaginary parts
    if (mine && row < n) {
      const double2 id = a.state[q].id;
      const bool has_id = id.x != 0.0 || id.y != 0.0;
#pragma unroll
      for (int c = 0; c < CG; ++c) {
        double2 v = make_double2(0.0, 0.0);
        if (c < cols) {
          v = P.V[(size_t)(cg * CG + c) * n + row];
          if (has_id) cfms(v, id, X[(size_t)c * n]);
        }
        r[c] = v.x;
        r[CG + c] = v.y;
      }
    }
    for (int dd = 0; dd < terms_of(P); ++dd) {
      // the product's scale in each column, 2^(row exponent + column exponent - 61)
      int ge[CG];
      int er = 0;
      if (mine && row < n) {
        er = P.Aexp[((size_t)dd * rbn + t.rb) * TM + 32 * quad + lane];
#pragma unroll
        for (int c = 0; c < CG; ++c)
          ge[c] = a.gexp[(size_t)q * a.gexp_stride + (dd * ncg + cg) * CG + c] + er - DRAIN_SCALE;
      }
      for (int kc0 = 0; kc0 < kcn; kc0 += KD / KC) {
        const bool ok = wait_or_bad(&sm.acc_full, blk & 1u, a.handoff_wait_cycles, &sm.bad, LOST_HANDOFF);
        if (!__all_sync(0xffffffffu, ok)) return;  // sm.bad is set
        ++blk;
        tcu::fence_after();
        DF H[2 * CG];
        if (mine) {
          // Horner's rule over the orders in double-float, as ozk::residual's
#pragma unroll
          for (int c = 0; c < 2 * CG; ++c) H[c] = DF{0.f, 0.f};
#pragma unroll 1
          for (int h = 0; h < NQ; ++h) {
            uint32_t v[16];
            tmem_ld16(base + (uint32_t)(h * 16 * MAXG), v);
#pragma unroll
            for (int c = 0; c < 2 * CG; ++c)
              H[c] = df_add_f(DF{H[c].hi * 128.f, H[c].lo * 128.f}, __uint_as_float(v[c]));
          }
        }
        tcu::fence_before();
        __syncwarp();
        if (lane == 0) arrive(&sm.acc_empty);
        // (the FP64 part while the next block's products run)
        if (mine && row < n) {
#pragma unroll
          for (int c = 0; c < CG; ++c) {
            const double sc = pow2(ge[c]);
            r[c] = fma(-sc, (double)H[c].hi, fma(-sc, (double)H[c].lo, r[c]));
            r[CG + c] = fma(-sc, (double)H[CG + c].hi, fma(-sc, (double)H[CG + c].lo, r[CG + c]));
          }
        }
      }
    }
    if (mine && row < n) {
#pragma unroll
      for (int c = 0; c < CG; ++c)
        if (c < cols) R[(size_t)c * n] = make_double2(r[c], r[CG + c]);
    }
  }
}

template <bool BIE>
__global__ void __launch_bounds__(GEMM_THREADS, 1) k_oz_residual(MixedArgs a, int sw) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  GemmSmem<BIE>& sm = *reinterpret_cast<GemmSmem<BIE>*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if ((int)blockIdx.x >= mixed_tiles(a, BIE)[a.n_probs] || *reinterpret_cast<volatile int32_t*>(a.err)) return;
  const long long t0 = clock64();
  const unsigned long long w0 = global_ns();
  if (warp == 2) tcu::tmem_alloc_cols(&sm.tmem, 512);
  if (tid == 0) {
    for (int i = 0; i < RA; ++i) {
      init_count(&sm.a_full[i], 1);
      init_count(&sm.a_empty[i], 1);
    }
    for (int i = 0; i < RB2; ++i) {
      init_count(&sm.b_full[i], 1);
      init_count(&sm.b_empty[i], 1);
    }
    init_count(&sm.acc_full, 1);
    init_count(&sm.acc_empty, DRAIN_WARPS);
    init_count(&sm.last, 1);
    sm.a_issued = sm.b_issued = 0;
    sm.bad = 0;
  }
  tcu::fence_async_smem();
  tcu::fence_before();
  __syncthreads();
  tcu::fence_after();
  if (warp == 0) {
    if (lane == 0) copy_role(a, sw, sm);
  } else if (warp == 1) {
    if (lane == 0) mma_role(a, sw, sm);
  } else if (warp >= DRAIN_WARP0) {
    drain_role(a, sw, sm);
  }
  __syncwarp();
  tcu::fence_before();
  __syncthreads();
  tcu::fence_after();
  if (sm.bad) {
    // let every issued copy land (bounded by the default limit), so that nothing
    // asynchronous touches this CTA's shared memory after it ends
    if (tid == 0) {
      for (uint32_t k = sm.a_issued > RA ? sm.a_issued - RA : 0; k < sm.a_issued; ++k)
        tcu::wait_parity(&sm.a_full[k % RA], (k / RA) & 1u, tcu::WAIT_CYCLES);
      for (uint32_t k = sm.b_issued > RB2 ? sm.b_issued - RB2 : 0; k < sm.b_issued; ++k)
        tcu::wait_parity(&sm.b_full[k % RB2], (k / RB2) & 1u, tcu::WAIT_CYCLES);
      if (sm.bad == LOST_HANDOFF) atomicExch(a.err, 1);
    }
    // the nodes of this CTA's tiles have no valid residual
    TileWalk<BIE> walk(a, sw);
    Tile t;
    while (walk.next(t))
      if (tid < t.ng) atomicOr(&a.state[t.units[tid] >> 3].lost, MIXED_LOST_RESIDUAL);
  }
  __syncthreads();
  if (warp == 2) tcu::tmem_dealloc_cols(sm.tmem, 512);
  if (a.phase && tid == 0) {
    unsigned long long* c = a.phase + (size_t)blockIdx.x * PMCIM_PHASES;
    c[PH_RESIDUAL] += (unsigned long long)(clock64() - t0);
    c[PH_CTA_WALL_NS] += global_ns() - w0;
  }
}

}  // namespace

// terms: dense terms, 0 for a boundary-integral node
size_t oz_slot_bytes(int n, int l, int terms) {
  const size_t groups = (size_t)((l + CG - 1) / CG) * k_chunks(n);
  return terms > 0 ? terms * groups * Form<false>::STAGE : groups * Form<true>::STAGE;
}

cudaError_t prepare_oz_refine() {
  cudaError_t e = cudaFuncSetAttribute(k_oz_residual<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(GemmSmem<false>));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_oz_residual<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(GemmSmem<true>));
}

cudaError_t launch_oz_residual(const MixedArgs& a, int sw, int sms, cudaStream_t s, int* launched) {
  static_assert(sizeof(GemmSmem<false>) <= 227 * 1024 && sizeof(GemmSmem<true>) <= 227 * 1024, "one CTA per SM");
  const int nd = a.gexp_stride / PMCIM_MAX_L;
  const long long w = (long long)a.count * nd;
  k_oz_digits<<<(unsigned)(w < 4 * sms ? w : 4 * sms), DIGIT_THREADS, 0, s>>>(a, sw, nd);
  ++*launched;
  if (a.oz_dense) {
    k_oz_residual<false><<<sms, GEMM_THREADS, sizeof(GemmSmem<false>), s>>>(a, sw);
    ++*launched;
  }
  if (a.tdig) {
    k_oz_residual<true><<<sms, GEMM_THREADS, sizeof(GemmSmem<true>), s>>>(a, sw);
    ++*launched;
  }
  return cudaGetLastError();
}
