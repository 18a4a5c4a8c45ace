// FP64 CUDA-core tensor contraction as a batched GEMM over strided views.
//
// Every contraction of the XTRG compression (the environment substeps of
// Fig. VMPO(c), the two-site overlap C_E of Eq. LSEProd and the transfer
// contractions of the traces) is a batched GEMM whose row, column and
// contraction indices are up to three-level strided views of the stored
// tensors (struct Idx3), so no permutation pass is needed between steps.
//
// This is the FP64 path; it also serves the canonicalisation and the traces
// of the tensor-core path.  What bounds it: a GB300 SM retires two FP64 FMAs
// a clock (64 times fewer than FP32), so a 32 x 32 x 16 tile step keeps the
// pipe busy for 8192 clocks and neither shared memory nor L2 matters; the
// time is the FMAs issued by the busiest SM.  Hence
//  - small tiles (32 x 32) with the contraction split over a cluster of up to
//    8 CTAs, so that every SM gets the same share also when the output has
//    few tiles (the partial tiles are summed in rank order through
//    distributed shared memory: no workspace, the same result every run);
//  - a warp owns 4 rows x 32 columns: rows past M cost nothing in steps of 4
//    (the transfers have 1, 5 or 25 of them), and the two operands are
//    exchanged when that wastes fewer lanes.
//  - the next K-block is loaded into registers before the tile's FMAs, and a
//    symmetric result computes only one triangle of its tiles.
// Measured: all transfers of one observables row at L = 64, D* = 256 (31
// GFLOP, 25 ms at the pipe's rate): 245 ms with 64 x 64 tiles and no split,
// 38.5 ms with small split tiles, 35.8 ms with the last item, 29.0 ms with one
// CTA an SM (see the launch), 28.0 ms with the present rule for the split.
#include "common.cuh"

#include <cooperative_groups.h>

namespace {

namespace cg = cooperative_groups;

constexpr int BM = 32, BN = 32, BK = 16, NT = 256;
constexpr int LDA = BM + 2, LDB = BN + 2;   // even: 16-byte reads of a row pair
constexpr int SPLIT_MAX = 8;                // portable cluster size

// idx_off with 32-bit divisions (every index of a view is below 2^31)
__device__ __forceinline__ long long off32(const Idx3& d, unsigned idx) {
  if (d.n0 == 1 && d.n1 == 1) return (long long)idx * d.s2;
  const unsigned t = idx / (unsigned)d.n0, i0 = idx - t * (unsigned)d.n0;
  const unsigned i2 = t / (unsigned)d.n1, i1 = t - i2 * (unsigned)d.n1;
  return (long long)i2 * d.s2 + (long long)i1 * d.s1 + (long long)i0 * d.s0;
}

// One 32 x 32 output tile over K range [k_begin, k_end) of this cluster rank.
template <bool SPLIT>
__global__ void __launch_bounds__(NT) gemm_kernel(GemmF64 g, int a_kfast, int b_kfast, int splits,
                                                  int k_per) {
  __shared__ __align__(16) double As[BK][LDA];
  __shared__ __align__(16) double Bs[BK][LDB];
  __shared__ long long offAm[BM], offBn[BN];

  // a symmetric result: the tiles above the diagonal are mirrored (every rank of
  // a cluster has the same tile)
  if (g.sym && blockIdx.x > blockIdx.y) return;
  const bool mirror = g.sym && blockIdx.x < blockIdx.y;
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int rank = SPLIT ? (int)(blockIdx.z % splits) : 0;
  const long long b = SPLIT ? blockIdx.z / splits : blockIdx.z;
  const int k_begin = SPLIT ? rank * k_per : 0;
  const int k_end = SPLIT ? min(g.K, k_begin + k_per) : g.K;
  const double* A = g.A + b * g.sab;
  const double* B = g.B + b * g.sbb;

  if (tid < BM) {
    const int m = m0 + tid;
    offAm[tid] = (m < g.M) ? off32(g.am, m) : 0;
  } else if (tid < BM + BN) {
    const int n = n0 + tid - BM;
    offBn[tid - BM] = (n < g.N) ? off32(g.bn, n) : 0;
  }

  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const bool live = m0 + 4 * warp < g.M;   // this warp's rows (uniform in the warp)

  // this thread's two elements of each operand's K-block; a block is loaded
  // into registers while the one before it is multiplied
  const int ami = a_kfast ? tid / BK : tid % BM, aki = a_kfast ? tid % BK : tid / BM;
  const int bni = b_kfast ? tid / BK : tid % BN, bki = b_kfast ? tid % BK : tid / BN;
  const int ams = a_kfast ? NT / BK : 0, aks = a_kfast ? 0 : NT / BM;   // step to the second
  const int bns = b_kfast ? NT / BK : 0, bks = b_kfast ? 0 : NT / BN;
  double va[2], vb[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int mi = ami + q * ams, ka = k0 + aki + q * aks;
      const int ni = bni + q * bns, kb = k0 + bki + q * bks;
      va[q] = (m0 + mi < g.M && ka < k_end) ? A[offAm[mi] + off32(g.ak, ka)] : 0.0;
      vb[q] = (n0 + ni < g.N && kb < k_end) ? B[offBn[ni] + off32(g.bk, kb)] : 0.0;
    }
  };
  __syncthreads();
  if (k_begin < k_end) load(k_begin);
  for (int k0 = k_begin; k0 < k_end; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      As[aki + q * aks][ami + q * ams] = va[q];
      Bs[bki + q * bks][bni + q * bns] = vb[q];
    }
    __syncthreads();
    if (k0 + BK < k_end) load(k0 + BK);
    if (live) {
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        const double2 a01 = *reinterpret_cast<const double2*>(&As[kk][4 * warp]);
        const double2 a23 = *reinterpret_cast<const double2*>(&As[kk][4 * warp + 2]);
        const double bb = Bs[kk][lane];
        acc[0] = fma(a01.x, bb, acc[0]);
        acc[1] = fma(a01.y, bb, acc[1]);
        acc[2] = fma(a23.x, bb, acc[2]);
        acc[3] = fma(a23.y, bb, acc[3]);
      }
    }
  }

  double* C = g.C + b * g.scb;
  if (!SPLIT) {
    const int n = n0 + lane;
    if (n >= g.N) return;
    const long long on = off32(g.cn, n);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + 4 * warp + i;
      if (m >= g.M) break;
      const long long o = off32(g.cm, m) + on;
      double v = g.alpha * acc[i];
      if (g.beta != 0.0) v += g.beta * C[o];
      C[o] = v;
      if (mirror) C[off32(g.cm, n) + off32(g.cn, m)] = v;
    }
    return;
  }
  // sum of the ranks' tiles: rank r takes every splits-th row
  __shared__ double Cs[BM][BN];
  cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
  for (int i = 0; i < 4; ++i) Cs[4 * warp + i][lane] = acc[i];
  cluster.sync();
  const int n = n0 + lane;
  for (int row = rank + splits * warp; row < BM; row += splits * (NT / 32)) {
    const int m = m0 + row;
    if (m < g.M && n < g.N) {
      double s = 0.0;
      for (int q = 0; q < splits; ++q) s += *cluster.map_shared_rank(&Cs[row][lane], q);
      const long long o = off32(g.cm, m) + off32(g.cn, n);
      double v = g.alpha * s;
      if (g.beta != 0.0) v += g.beta * C[o];
      C[o] = v;
      if (mirror) C[off32(g.cm, n) + off32(g.cn, m)] = v;
    }
  }
  cluster.sync();   // peers may still be reading this CTA's tile
}

int innermost_unit(const Idx3& d) {
  // the fastest-varying sub-index of the view has unit stride
  if (d.n0 > 1) return d.s0 == 1;
  if (d.n1 > 1) return d.s1 == 1;
  return d.s2 == 1;
}

inline long long up_to(long long x, long long q) { return (x + q - 1) / q * q; }

// Dynamic shared memory that keeps an SM to one CTA (see the launch).
constexpr int ALONE_SMEM = 120 * 1024;
PerDevice<int> g_sms;

}  // namespace

cudaError_t gemm_f64(const GemmF64& g0, cudaStream_t st) {
  if (g0.M <= 0 || g0.N <= 0 || g0.batch <= 0) return cudaSuccess;
  if (g0.K <= 0 || g0.batch > 65535) return cudaErrorInvalidValue;
  GemmF64 g = g0;
  // C^T = B^T A^T when its rows and columns round up to less work
  if (up_to(g.N, 4) * up_to(g.M, BN) < up_to(g.M, 4) * up_to(g.N, BN)) {
    g.M = g0.N; g.N = g0.M;
    g.A = g0.B; g.am = g0.bn; g.ak = g0.bk; g.sab = g0.sbb;
    g.B = g0.A; g.bk = g0.ak; g.bn = g0.am; g.sbb = g0.sab;
    g.cm = g0.cn; g.cn = g0.cm;
  }
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
  if (grid.y > 65535) return cudaErrorInvalidValue;
  int sms = 152;
  cudaError_t e = g_sms.get(
      [](int dev) {
        int n = 0;
        if (cudaFuncSetAttribute(gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 ALONE_SMEM) != cudaSuccess)
          cudaGetLastError();
        return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0
                   ? n : 152;
      },
      &sms);
  if (e != cudaSuccess) return e;
  // Split of the contraction: the fewest K-steps on the busiest SM.  A split
  // adds its start and the exchange of its partial tile, about two K-steps
  // (16 x 32 x 32 FMAs at 2 a clock, 4 us each); a step is one K-block of 16.
  // It adds them once: with several CTAs an SM the others compute meanwhile
  // (counted for each of them: observables row 29.0 ms, once: 28.0 ms).
  if (g.sym && g.M != g.N) return cudaErrorInvalidValue;
  const long long tiles = g.sym ? (long long)grid.x * (grid.x + 1) / 2 * g.batch
                                : (long long)grid.x * grid.y * g.batch;
  const int kb = (g.K + BK - 1) / BK;
  int splits = 1;
  long long best = 0;
  for (int s = 1; s <= SPLIT_MAX && (s == 1 || (s <= kb && g.batch * s <= 65535)); s *= 2) {
    const long long cost = (tiles * s + sms - 1) / sms * ((kb + s - 1) / s) + (s > 1 ? 2 : 0);
    if (s == 1 || cost < best) {
      best = cost;
      splits = s;
    }
  }
  const int a_kfast = innermost_unit(g.ak) && !innermost_unit(g.am);
  const int b_kfast = innermost_unit(g.bk) && !innermost_unit(g.bn);
  note_launch();
  if (splits == 1) {
    gemm_kernel<false><<<grid, NT, 0, st>>>(g, a_kfast, b_kfast, 1, g.K);
    return cudaGetLastError();
  }
  grid.z = (unsigned)(g.batch * splits);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = (unsigned)splits;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // When every CTA could have an SM to itself it gets one: the CTAs of a cluster
  // are otherwise put two to an SM, which then takes twice as long (observables
  // row: 35.8 ms, 29.0 ms with this).  Short ones are launch-bound either way
  // and keep their small footprint for the kernels of other streams.
  const int blocks = (kb + splits - 1) / splits;
  if (tiles * splits <= sms && blocks >= 4) cfg.dynamicSmemBytes = ALONE_SMEM;
  return cudaLaunchKernelEx(&cfg, gemm_kernel<true>, g, a_kfast, b_kfast, splits, blocks * BK);
}
