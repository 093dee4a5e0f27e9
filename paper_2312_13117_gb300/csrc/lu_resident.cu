// FP64 node solves with the node's matrix resident in shared memory.
//
// The same work as k_factor_solve_fp64 (assembly of T(z_j), LU with partial
// pivoting on [T | V], back substitution), for nodes whose matrix and probe
// columns fit an SM's shared memory (lu_resident.cuh): one CTA per node, as many
// CTAs per SM as fit. The FP64 unit (2 multiply-adds per SM and clock) bounds
// these nodes: n = 100, l = 10 needs 0.42 ms of one SM. Measured on whole calls:
// 3600 nodes of n = 100, l = 10 (indicator) 20.8 ms against 47.8 ms through the
// blocked kernel, 512 nodes of n = 64, l = 8 (moments) 1.23 against 3.47 ms.
#include "lu_resident.cuh"

namespace {

using namespace resident;

struct Head {
  Ctl ctl;
  int item;
  ProblemDev P;
  double2 fz[PMCIM_MAX_TERMS];
  bie::Wave wave;
};
constexpr size_t kHeadBytes = (sizeof(Head) + 15) & ~size_t(15);

template <bool BIE>
__global__ void __launch_bounds__(512) k_factor_solve_resident(NodeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Head& sm = *reinterpret_cast<Head*>(smem_raw);
  double2* M = reinterpret_cast<double2*>(smem_raw + kHeadBytes);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  for (;;) {
    if (tid == 0) sm.item = atomicAdd(a.counter, 1);
    __syncthreads();
    const int idx = sm.item;
    if (idx >= a.n_items) break;
    const NodeItem it = a.items[idx];
    const RegionDev rg = a.regions[it.region];
    load_problem(&sm.P, a.probs + rg.prob);
    __syncthreads();
    const ProblemDev& P = sm.P;
    const int n = P.n, l = P.l, ncols = n + l, ld = lead(n);
    double2* divisor = M + (size_t)ld * ncols;
    int* piv = reinterpret_cast<int*>(divisor + n);
    double2 z, w;
    node_weight(rg.cre, rg.cim, rg.r, rg.N, it.j, &z, &w);
    if (tid < P.K) sm.fz[tid] = eval_f(P.term[tid], z);
    // a circulant boundary-integral term's n distinct entries, in the divisors' place
    const bool use_circ = BIE && P.bie_circ;
    if (BIE) {
      if (tid == 0) sm.wave = bie::wave_of(z);
      __syncthreads();
      if (use_circ)
        for (int m = tid; m < n; m += blockDim.x) divisor[m] = bie::dlp_entry(P.bie, n, m, 0, sm.wave);
    }
    __syncthreads();
    const size_t nn = (size_t)n * n;
    for (int col = warp; col < n; col += nwarp)
      for (int row = lane; row < n; row += 32) {
        double2 v = make_double2(0.0, 0.0);
        for (int k = 0; k < P.K; ++k) {
          const TermDesc& t = P.term[k];
          if (t.dense) cfma(v, sm.fz[k], P.A[(size_t)t.mat_index * nn + (size_t)col * n + row]);
          else if (use_circ && t.kind == PMCIM_F_HELMHOLTZ_DLP)
            cfma(v, t.id, divisor[row >= col ? row - col : row - col + n]);
          else if (row == col && t.kind != PMCIM_F_HELMHOLTZ_DLP) cfma(v, sm.fz[k], t.id);
        }
        M[(size_t)col * ld + row] = v;
      }
    if (BIE && P.bie && !use_circ) {
      __syncthreads();
      add_layer(P.bie, n, layer_coefficient(P), sm.wave, tid, blockDim.x,
                [&](int i, int j, double2 v) { M[(size_t)j * ld + i] = cadd(M[(size_t)j * ld + i], v); });
    }
    for (int c = warp; c < l; c += nwarp)
      for (int row = lane; row < n; row += 32) M[(size_t)(n + c) * ld + row] = P.V[(size_t)c * n + row];
    __syncthreads();
    factor(M, n, ncols, ld, piv, divisor, sm.ctl);
    back(M, n, l, ld, divisor);
    __syncthreads();
    double2* Xo = a.X + rg.x_off + (size_t)it.j * n * l;
    for (int c = warp; c < l; c += nwarp)
      for (int row = lane; row < n; row += 32) Xo[(size_t)c * n + row] = M[(size_t)(n + c) * ld + row];
    if (tid == 0) a.node_info[rg.node_off + it.j] = sm.ctl.info;
    __syncthreads();
  }
}

constexpr size_t kSmBytes = 227 * 1024;  // shared memory of an SM that CTAs can have

}  // namespace

size_t resident_bytes(int n, int l) { return kHeadBytes + node_bytes(n, l); }

// CTAs per SM that ask for this much shared memory, 0 when one does not fit. An SM gives
// each CTA 1 KB more than it asks for.
int resident_ctas(size_t bytes) {
  if (bytes > kSmBytes) return 0;
  const size_t k = (kSmBytes + 1024) / (bytes + 1024);
  return (int)(k < 8 ? k : 8);
}

cudaError_t prepare_factor_resident() {
  cudaError_t e = cudaFuncSetAttribute(k_factor_solve_resident<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_factor_solve_resident<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmBytes);
}

// bytes: the largest resident_bytes among the items.
cudaError_t launch_factor_solve_resident(const NodeArgs& a, size_t bytes, cudaStream_t s) {
  if (a.n_items <= 0) return cudaSuccess;
  const int ctas = resident_ctas(bytes);
  if (ctas < 1) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int grid = ctas * (sms > 0 ? sms : 1);
  if (grid > a.n_items) grid = a.n_items;
  // a CTA alone on its SM needs 16 warps to keep the FP64 units busy
  const int threads = ctas == 1 ? 512 : 256;
  if (a.bie) k_factor_solve_resident<true><<<grid, threads, bytes, s>>>(a);
  else k_factor_solve_resident<false><<<grid, threads, bytes, s>>>(a);
  return cudaGetLastError();
}
