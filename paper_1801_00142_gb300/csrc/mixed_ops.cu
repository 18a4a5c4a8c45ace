// Layout and precision conversions of the tensor-core path: FP64 tensors to
// BF16 split planes through strided views, and the FP64 reduction of split-K
// partial sums (alone, or fused with the planes of the result in both
// orientations).
#include <cuda_bf16.h>

#include "mixed_ops.cuh"
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
// Rows start 16-byte aligned (ld is a multiple of 8, as are obs and ops where
// 16-byte stores are chosen, see the launch).
// Measured on 2^26 FP64 elements, 3 planes (0.94 GB moved): 157 us, 88 % of
// the measured copy rate; 862 us with an element a thread, its 64-bit divisions
// and FP64 conversions.
constexpr int TP_R = 32, TP_K = 64;
template <typename S>
__global__ void __launch_bounds__(256)
    to_planes_kernel(const S* __restrict__ src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K,
                     int tiles_r, int tiles_k, long long tiles, __nv_bfloat16* __restrict__ out,
                     long long ld, long long obs, int planes, long long ops, int kfast, int vec,
                     const double* __restrict__ run_if, double thresh) {
  if (run_if && *run_if <= thresh) return;
  __shared__ __align__(16) unsigned short tp[3][TP_R][TP_K + 8];
  const int tid = threadIdx.x;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int b = (int)(t / (tiles_r * tiles_k)), w = (int)(t - (long long)b * (tiles_r * tiles_k));
    const int r0 = w / tiles_k * TP_R, k0 = w % tiles_k * TP_K;
    const S* sb = src + b * sbs;
    S x[8];
    if (kfast) {
      const int k = k0 + tid % 64, y = tid / 64;
      const long long ok = k < K ? off32(kv, k) : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + y + 4 * u;
        x[u] = (r < rows && k < K) ? sb[off32(rv, r) + ok] : S(0);
      }
    } else {
      const int r = r0 + tid % 32, y = tid / 32;
      const long long orr = r < rows ? off32(rv, r) : 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = k0 + y + 8 * u;
        x[u] = (r < rows && k < K) ? sb[orr + off32(kv, k)] : S(0);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      unsigned short c[3];
      cut(x[u], c);
      const int y = kfast ? tid / 64 + 4 * u : tid % 32;
      const int z = kfast ? tid % 64 : tid / 32 + 8 * u;
      tp[0][y][z] = c[0];
      tp[1][y][z] = c[1];
      tp[2][y][z] = c[2];
    }
    __syncthreads();
    const int y = tid / 8, z = tid % 8 * 8, r = r0 + y, k = k0 + z;
    if (r < rows && k < ld) {
      __nv_bfloat16* d = out + b * obs + (long long)r * ld + k;
      for (int q = 0; q < planes; ++q, d += ops) {
        if (vec) {
          *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(&tp[q][y][z]);
        } else {
          for (int u = 0; u < 8; ++u) d[u] = __ushort_as_bfloat16(tp[q][y][z + u]);
        }
      }
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
cudaError_t launch_to_planes(const S* src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K,
                             int batch, __nv_bfloat16* out, long long ld, long long obs, int planes,
                             long long ops, cudaStream_t st, const double* run_if = nullptr,
                             double thresh = 0.0) {
  if ((long long)rows * ld * batch <= 0) return cudaSuccess;
  const int tiles_r = (rows + TP_R - 1) / TP_R, tiles_k = (int)((ld + TP_K - 1) / TP_K);
  const long long tiles = (long long)tiles_r * tiles_k * batch;
  const int vec = ((uintptr_t)out % 16) == 0 && ld % 8 == 0 && obs % 8 == 0 && ops % 8 == 0;
  const int kfast = unit_stride(kv) || !unit_stride(rv);
  const long long grid = tiles < 152 * 16 ? tiles : 152 * 16;
  note_launch();
  to_planes_kernel<S><<<(unsigned)grid, 256, 0, st>>>(src, rv, kv, sbs, rows, K, tiles_r, tiles_k,
                                                      tiles, out, ld, obs, planes, ops, kfast, vec, run_if,
                                                      thresh);
  return cudaGetLastError();
}

__global__ void reduce_partials_kernel(const float* __restrict__ part, int splits, long long n,
                                       double* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll 8
    for (int i = 0; i < splits; ++i) s += (double)part[i * n + e];
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
  return launch_to_planes<double>(src, rv, kv, sbs, rows, K, batch, out, ld, obs, planes, ops, st);
}

cudaError_t to_planes_if(const double* src, Idx3 rv, Idx3 kv, int rows, int K, __nv_bfloat16* out,
                         long long ld, int planes, long long ops, const double* run_if,
                         double thresh, cudaStream_t st) {
  if (!run_if) return cudaErrorInvalidValue;
  return launch_to_planes<double>(src, rv, kv, 0, rows, K, 1, out, ld, 0, planes, ops, st, run_if,
                                  thresh);
}

cudaError_t to_planes_f32(const float* src, Idx3 rv, Idx3 kv, long long sbs, int rows, int K,
                          int batch, __nv_bfloat16* out, long long ld, long long obs, int planes,
                          long long ops, cudaStream_t st) {
  return launch_to_planes<float>(src, rv, kv, sbs, rows, K, batch, out, ld, obs, planes, ops, st);
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
