// Layout and precision conversions of the tensor-core path: FP64 tensors to
// BF16 split planes through strided views, and the FP64 reduction of split-K
// partial sums (alone, or fused with the planes of the result in both
// orientations).
#include <cuda_bf16.h>

#include "mixed_ops.cuh"
#include "plane_layout.h"
#include "planes.cuh"

namespace {

inline int grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  if (b < 1) b = 1;
  return (int)b;
}

// out[b][r][k] (row stride ld, batch stride obs, plane stride ops) =
// split(src[b*sbs + off(rv, r) + off(kv, k)]); padding columns k in [K, ld) = 0.
//
// Bound by HBM: sizeof(S) read and 2 * planes written per element.  Tiles of
// 32 rows x 64 columns: the reads run along whichever index is contiguous in
// src (kfast: k, else the rows), the planes pass through shared memory, and
// each thread writes eight consecutive columns of a row per plane, 16 bytes.
// Every row starts 16-byte aligned: the launch refuses other layouts.
// Measured on 2^26 FP64 elements, 3 planes (0.94 GB moved): 152 us, 91 % of
// the measured copy rate; 862 us with an element a thread, its 64-bit divisions
// and FP64 conversions.
constexpr int TP_R = 32, TP_K = 64;
template <typename S>
struct PlaneJob {
  const S* src;
  Idx3 rv, kv;
  long long sbs;
  int rows, K, tiles_r, tiles_k;
  long long tiles;
  __nv_bfloat16* out;
  long long ld, obs, ops;
  int kfast;        // reads along k
};

// One matrix, or with PAIR two in one launch (a small product's operands);
// clear (may be null) is set to zero.  With run_if, runs only if *run_if >
// thresh or is not finite.
template <typename S, bool PAIR>
__global__ void __launch_bounds__(256)
    to_planes_kernel(const PlaneJob<S> j0, const PlaneJob<S> j1, int planes, int* clear,
                     const double* __restrict__ run_if, double thresh) {
  if (run_if && *run_if <= thresh) return;
  __shared__ __align__(16) unsigned short tp[3][TP_R][TP_K + 8];
  const int tid = threadIdx.x;
  if (clear && blockIdx.x == 0 && tid == 0) *clear = 0;
  for (long long tt = blockIdx.x; tt < j0.tiles + j1.tiles; tt += gridDim.x) {
    const PlaneJob<S>& j = !PAIR || tt < j0.tiles ? j0 : j1;
    const long long t = !PAIR || tt < j0.tiles ? tt : tt - j0.tiles;
    const int per = j.tiles_r * j.tiles_k;
    const int b = (int)(t / per), w = (int)(t - (long long)b * per);
    const int r0 = w / j.tiles_k * TP_R, k0 = w % j.tiles_k * TP_K;
    const S* sb = j.src + b * j.sbs;
    S x[8];
    if (j.kfast) {
      const int k = k0 + tid % 64, y = tid / 64;
      const long long ok = k < j.K ? off32(j.kv, k) : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + y + 4 * u;
        x[u] = (r < j.rows && k < j.K) ? sb[off32(j.rv, r) + ok] : S(0);
      }
    } else {
      const int r = r0 + tid % 32, y = tid / 32;
      const long long orr = r < j.rows ? off32(j.rv, r) : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + y + 8 * u;
        x[u] = (r < j.rows && k < j.K) ? sb[orr + off32(j.kv, k)] : S(0);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      unsigned short c[3];
      cut(x[u], c);
      const int y = j.kfast ? tid / 64 + 4 * u : tid % 32;
      const int z = j.kfast ? tid % 64 : tid / 32 + 8 * u;
      tp[0][y][z] = c[0];
      tp[1][y][z] = c[1];
      tp[2][y][z] = c[2];
    }
    __syncthreads();
    const int y = tid / 8, z = tid % 8 * 8, r = r0 + y, k = k0 + z;
    if (r < j.rows && k < j.ld) {
      __nv_bfloat16* d = j.out + b * j.obs + (long long)r * j.ld + k;
      // unrolled: without, 2^26 elements take 160 us
#pragma unroll
      for (int q = 0; q < 3; ++q, d += j.ops)
        if (q < planes) *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(&tp[q][y][z]);
    }
    __syncthreads();
  }
}

// the fastest-varying sub-index of a view has unit stride
int unit_stride(const Idx3& d) {
  if (d.n0 > 1) return d.s0 == 1;
  if (d.n1 > 1) return d.s1 == 1;
  return d.s2 == 1;
}

template <typename S>
PlaneJob<S> plane_job(const S* src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K, int batch,
                      __nv_bfloat16* out, long long ld, long long obs, long long ops) {
  PlaneJob<S> j{};
  if ((long long)rows * ld * batch <= 0) return j;
  // rows that follow one another across the batch are rows of one matrix: a tile
  // holds 32 of them, whatever the size of the batch's matrices (500 of 1 x 4096:
  // 111 -> 14 us; 2000 of 1 x 1 10.4 -> 5.1 us)
  if (batch > 1 && rv.n1 == 1 && rv.n0 == 1 && sbs == rows * rv.s2 && obs == rows * ld &&
      (long long)rows * batch <= 0x7fffffffLL) {
    rows *= batch;
    batch = 1;
  }
  j.src = src; j.rv = rv; j.kv = kv; j.sbs = sbs; j.rows = rows; j.K = K;
  j.tiles_r = (rows + TP_R - 1) / TP_R;
  j.tiles_k = (int)((ld + TP_K - 1) / TP_K);
  j.tiles = (long long)j.tiles_r * j.tiles_k * batch;
  j.out = out; j.ld = ld; j.obs = obs; j.ops = ops;
  j.kfast = unit_stride(kv) || !unit_stride(rv);
  return j;
}

// Whether every row of every plane starts on 16 bytes (and so ends on them:
// a thread stores eight columns from any multiple of 8 below ld).
template <typename S>
bool rows_aligned(const PlaneJob<S>& j) {
  return (uintptr_t)j.out % 16 == 0 && j.ld % 8 == 0 && j.obs % 8 == 0 && j.ops % 8 == 0;
}

template <typename S>
cudaError_t launch_to_planes(const PlaneJob<S>& j0, const PlaneJob<S>& j1, int planes, int* clear,
                             cudaStream_t st, const double* run_if = nullptr, double thresh = 0.0) {
  const long long tiles = j0.tiles + j1.tiles;
  if (tiles <= 0) return cudaSuccess;
  if (!rows_aligned(j0) || !rows_aligned(j1)) return cudaErrorInvalidValue;
  // two matrices share a launch while they leave room on the chip; larger ones
  // gain nothing by it, and the kernel of one has its view in constants (1024 x
  // 65536: 152 us a matrix, 180 us in a pair)
  if (j0.tiles > 0 && j1.tiles > 0 && tiles > 152 * 16) {
    const cudaError_t e = launch_to_planes(j0, PlaneJob<S>{}, planes, clear, st, run_if, thresh);
    return e != cudaSuccess ? e : launch_to_planes(j1, PlaneJob<S>{}, planes, nullptr, st, run_if, thresh);
  }
  const unsigned grid = (unsigned)(tiles < 152 * 16 ? tiles : 152 * 16);
  note_launch();
  if (j1.tiles == 0)
    to_planes_kernel<S, false><<<grid, 256, 0, st>>>(j0, j1, planes, clear, run_if, thresh);
  else
    to_planes_kernel<S, true><<<grid, 256, 0, st>>>(j0, j1, planes, clear, run_if, thresh);
  return cudaGetLastError();
}

// FP64 sum of FP32 partials; the conversions are integer operations (FP64-pipe
// conversions alone bound this kernel: 13 us on 2.7 M elements)
__global__ void reduce_partials_kernel(const float* __restrict__ part, int splits, long long n,
                                       double* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    double s = f32_to_f64(part[e]);
#pragma unroll 8
    for (int i = 1; i < splits; ++i) s += f32_to_f64(part[i * n + e]);
    out[e] = s;
  }
}

// One 32 x 32 tile of C = sum of the split-K partials: the FP64 result, its
// three BF16 planes in both orientations (row-major [m][ldn] and transposed
// [n][ldm], the K-major operands of C x and C^T x), and the tile's sum of
// squares added into *ss.  The transposed planes go through shared memory so
// that both the reads and the writes are coalesced; padding columns of both
// plane layouts are written as zero.
__global__ void reduce_partials_planes_kernel(const float* __restrict__ part, int splits, int m,
                                              int n, double* __restrict__ out,
                                              __nv_bfloat16* __restrict__ prm, long long ldn,
                                              __nv_bfloat16* __restrict__ ptr, long long ldm,
                                              long long ps, double* ss) {
  // the three planes of the tile, kept for the transposed writes (FP64
  // arithmetic is slow on this GPU: the partials are summed in FP32 with a
  // compensation term, which keeps the sum to about FP64 accuracy for the
  // few splits, and the planes are cut from that pair in FP32)
  __shared__ __nv_bfloat16 tp[3][32][34];
  __shared__ double red[8];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;   // 32 x 8 threads
  const int n0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
  const long long mn = (long long)m * n;
  double acc = 0.0;
  // the thread's four rows side by side and four partials at a time: sixteen
  // loads in flight (a row after the other waited out the latency of every
  // partial: 26 us at 256 x 256 x 32 splits, now 10)
  float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
  const int c = n0 + tx;
  {
    const float* src[4];
    bool in[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = m0 + ty + 8 * u;
      in[u] = r < m && c < n;
      src[u] = part + (in[u] ? (long long)r * n + c : 0);
    }
    for (int i0 = 0; i0 < splits; i0 += 4) {
      float x[4][4];
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          x[v][u] = (in[u] && i0 + v < splits) ? src[u][(long long)(i0 + v) * mn] : 0.f;
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // two-sum: hi + lo = old hi + part exactly, errors gathered in lo
          const float t = hi[u] + x[v][u];
          const float bp = t - hi[u];
          lo[u] += (hi[u] - (t - bp)) + (x[v][u] - bp);
          hi[u] = t;
        }
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int y = ty + 8 * u, r = m0 + y;
    if (r < m && c < n) {
      const double v = (double)hi[u] + (double)lo[u];
      out[(long long)r * n + c] = v;
      acc = fma(v, v, acc);
    }
    const __nv_bfloat16 p0 = __float2bfloat16_rn(hi[u]);
    const float r1 = (hi[u] - __bfloat162float(p0)) + lo[u];
    const __nv_bfloat16 p1 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 p2 = __float2bfloat16_rn(r1 - __bfloat162float(p1));
    tp[0][y][tx] = p0;
    tp[1][y][tx] = p1;
    tp[2][y][tx] = p2;
    if (r < m && c < ldn) {
      const long long o = (long long)r * ldn + c;
      prm[o] = p0;
      prm[o + ps] = p1;
      prm[o + 2 * ps] = p2;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (tx == 0) red[ty] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += red[i];
    atomicAdd(ss, t);
  }
  for (int y = ty; y < 32; y += 8) {
    const int r = n0 + y, ct = m0 + tx;   // row r of C^T, column ct
    if (r < n && ct < ldm) {
      const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
      const bool in = ct < m;
      const long long o = (long long)r * ldm + ct;
      ptr[o] = in ? tp[0][tx][y] : z;
      ptr[o + ps] = in ? tp[1][tx][y] : z;
      ptr[o + 2 * ps] = in ? tp[2][tx][y] : z;
    }
  }
}


}  // namespace

cudaError_t to_planes(const double* src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K,
                      int batch, __nv_bfloat16* out, long long ld, long long obs, int planes,
                      long long ops, cudaStream_t st) {
  return launch_to_planes(plane_job(src, rv, kv, sbs, rows, K, batch, out, ld, obs, ops),
                          PlaneJob<double>{}, planes, nullptr, st);
}

cudaError_t to_planes_pair(const double* a, int rows_a, int Ka, __nv_bfloat16* out_a, const double* b,
                           int rows_b, int Kb, __nv_bfloat16* out_b, int batch, int planes,
                           int* clear, cudaStream_t st) {
  const PlaneLayout la = plane_layout(rows_a, Ka, batch), lb = plane_layout(rows_b, Kb, batch);
  return launch_to_planes(
      plane_job(a, idx_plain(Ka), idx_plain(1), (long long)rows_a * Ka, rows_a, Ka, batch, out_a,
                la.ld, la.batch_stride, la.plane_stride),
      plane_job(b, idx_plain(Kb), idx_plain(1), (long long)rows_b * Kb, rows_b, Kb, batch, out_b,
                lb.ld, lb.batch_stride, lb.plane_stride),
      planes, clear, st);
}

cudaError_t to_planes_if(const double* src, Idx3 rv, Idx3 kv, int rows, int K, __nv_bfloat16* out,
                         long long ld, int planes, long long ops, const double* run_if,
                         double thresh, cudaStream_t st) {
  if (!run_if) return cudaErrorInvalidValue;
  return launch_to_planes(plane_job(src, rv, kv, 0, rows, K, 1, out, ld, 0, ops), PlaneJob<double>{},
                          planes, nullptr, st, run_if, thresh);
}

cudaError_t to_planes_f32(const float* src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K,
                          int batch, __nv_bfloat16* out, long long ld, long long obs, int planes,
                          long long ops, cudaStream_t st) {
  return launch_to_planes(plane_job(src, rv, kv, sbs, rows, K, batch, out, ld, obs, ops),
                          PlaneJob<float>{}, planes, nullptr, st);
}

cudaError_t reduce_partials(const float* part, int splits, long long n, double* out,
                            cudaStream_t st) {
  note_launch();
  reduce_partials_kernel<<<grid_for(n), 256, 0, st>>>(part, splits, n, out);
  return cudaGetLastError();
}


cudaError_t reduce_partials_planes(const float* part, int splits, int m, int n, double* out,
                                   __nv_bfloat16* prm, long long ldn, __nv_bfloat16* ptr,
                                   long long ldm, long long ps, double* ss, cudaStream_t st) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  dim3 grid((unsigned)((n + 31) / 32), (unsigned)((m + 31) / 32));
  note_launch();
  reduce_partials_planes_kernel<<<grid, 256, 0, st>>>(part, splits, m, n, out, prm, ldn, ptr, ldm,
                                                      ps, ss);
  return cudaGetLastError();
}
