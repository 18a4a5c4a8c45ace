// Truncation of the tensor-core path: one warm-started subspace step,
// orthonormalised by scaled CholeskyQR2.
//
// The two-site update keeps the dominant rank-k subspace of C_E (Fig.
// VMPO(d)).  The FP64 path computes it exactly by Jacobi SVD; here, where
// C_E itself carries FP32-level errors, one step of subspace iteration from
// the previous sweep's basis is used instead: left-to-right,
//   Y = C_E V_prev (+ eta R),  U = orth(Y),  C_i = U,  C_{i+1} = U^T C_E,
// and mirrored right-to-left.  V_prev are the orthonormal rows of the current
// C_{i+1} (right-canonical guess, or V^T of the previous right-to-left pass),
// padded with pseudo-random columns when the bond grows.  The tiny random
// term eta R keeps every column of Y away from exact zero; directions it adds
// carry weight below eta^2 relative.
//
// orth() is a scaled CholeskyQR2 of the whole block (tensor-core Gram, one-CTA
// FP32 Cholesky, all-SM triangular solve; see below), the second pass to first
// order where that suffices.  A pivot that shows a column to be numerically
// dependent on those before it drops the column: its output is zero (dead)
// and the noise gives it a fresh direction in the next sweep (CQ_TAU1,
// CQ_TAU2).  Completing the bases that fail the second pass by block
// Gram-Schmidt instead took 1.7 ms each at k = 256, for 45 of the 504 updates of
// a doubling at L = 64, D* = 256 (868 ms, 790 without).  The caller checks
// max |U^T U - I| over the live columns and takes the exact split when the FP32
// products lost orthogonality.
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "mixed_ops.cuh"
#include "planes.cuh"
#include "subspace_split.cuh"
#include "tc_gemm.cuh"

namespace {

inline int grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  if (b < 1) b = 1;
  return (int)b;
}

// counter-based pseudo-random value in [-1, 1) (splitmix64 finaliser)
__device__ inline float hash_uniform(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  return (float)(unsigned)(x >> 40) * (1.f / 8388608.f) - 1.f;   // 24 bits, no FP64
}

// Q[r][j] (rows x k) = src(j, r) for j < kold (src FP64 with strides), else
// pseudo-random.  src(j, r) = S[j*sj + r*sr].
__global__ void warm_start_kernel(const double* __restrict__ S, long long sj, long long sr,
                                  int kold, int rows, int k, unsigned long long seed0,
                                  const unsigned long long* __restrict__ base,
                                  float* __restrict__ Q) {
  const unsigned long long seed = seed0 ^ (*base * 0x9E3779B97F4A7C15ull);
  const long long total = (long long)rows * k;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(e / k), j = (int)(e % k);
    Q[e] = j < kold ? (float)S[j * sj + r * sr] : hash_uniform(seed * 0x100000001B3ull + e);
  }
}

// Y += eta R with eta = 1e-5 * rms(C_E), rms from ||C_E||^2 on the device
__global__ void add_noise_kernel(float* __restrict__ Y, long long n, const double* __restrict__ tot,
                                 double inv_mn, unsigned long long seed0,
                                 const unsigned long long* __restrict__ base) {
  const unsigned long long seed = seed0 ^ (*base * 0x9E3779B97F4A7C15ull);
  const float eta = (float)(1e-5 * sqrt(*tot * inv_mn));
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    Y[e] += eta * hash_uniform(seed ^ (0xD1B54A32D192ED03ull * (e + 1)));
}

__global__ void copy_f2d_kernel(const float* __restrict__ a, long long n, double* __restrict__ b) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    b[e] = (double)a[e];
}

// out[c][r] = in[r][c] (rows x cols -> cols x rows), FP32 -> FP64
__global__ void transpose_f2d_kernel(const float* __restrict__ a, int rows, int cols,
                                     double* __restrict__ b) {
  const long long total = (long long)rows * cols;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(e / rows), r = (int)(e % rows);
    b[e] = (double)a[(long long)r * cols + c];
  }
}

// sum of squares in FP64 (grid-stride, one atomic per CTA)
__global__ void sumsq_f64_kernel(const double* __restrict__ a, long long n, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    s = fma(a[e], a[e], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x / 32); ++i) t += red[i];
    atomicAdd(out, t);
  }
}

constexpr int MAX_K = SUBSPACE_BLOCK_K;

// C[m][n] (row stride ldc) = sum over s of part[s][m][n]
__global__ void sum_partials_kernel(const float* __restrict__ part, int splitk, int M, int N,
                                    float* __restrict__ C, long long ldc) {
  const long long MN = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < MN;
       e += (long long)gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int s = 0; s < splitk; ++s) acc += part[s * MN + e];
    C[(e / N) * ldc + e % N] = acc;
  }
}

#define RET(x)                                 \
  do {                                         \
    cudaError_t _e = (x);                      \
    if (_e != cudaSuccess) return _e;          \
  } while (0)

// C (M x N, FP32 row-major, ldc) = A B^T on the tensor cores (3 planes, 6
// products).  Each operand is either given as BF16 planes already (p: row
// stride pld, plane stride pps) or as an FP32 view split by to_planes_f32.
struct View {
  const float* f;
  Idx3 rv, kv;
  const __nv_bfloat16* p;
  long long pld, pps;
};

View planes_view(const __nv_bfloat16* p, long long pld, long long pps) {
  return View{nullptr, idx_plain(0), idx_plain(0), p, pld, pps};
}
View f32_view(const float* f, Idx3 rv, Idx3 kv) { return View{f, rv, kv, nullptr, 0, 0}; }

cudaError_t tc_product(const View& a, const View& b, int M, int N, int K, float* C, long long ldc,
                       const SubspaceBuffers& buf, cudaStream_t st) {
  const long long ld = tc_ld(K);
  const long long psa = (long long)M * ld, psb = (long long)N * ld;
  if (psa > buf.psa || psb > buf.psb) return cudaErrorInvalidValue;
  TcOperand A{buf.pa, 3, M, K, ld, 0, buf.psa, 1};
  TcOperand B{buf.pb, 3, N, K, ld, 0, buf.psb, 1};
  if (a.p) A = TcOperand{a.p, 3, M, K, a.pld, 0, a.pps, 1};
  else RET(to_planes_f32(a.f, a.rv, a.kv, 0, M, K, 1, buf.pa, ld, 0, 3, buf.psa, st));
  // a Gram (the same FP32 view on both sides) converts its operand once
  const bool same = !a.p && !b.p && a.f == b.f && M == N && !memcmp(&a.rv, &b.rv, sizeof(Idx3)) &&
                    !memcmp(&a.kv, &b.kv, sizeof(Idx3));
  if (b.p) B = TcOperand{b.p, 3, N, K, b.pld, 0, b.pps, 1};
  else if (same) B = A;
  else RET(to_planes_f32(b.f, b.rv, b.kv, 0, N, K, 1, buf.pb, ld, 0, 3, buf.psb, st));
  TcOutput o;
  memset(&o, 0, sizeof o);
  o.alpha = 1.0;
  // products with few output tiles (the k x k Grams, the k-wide factors)
  // split K so that about one wave of CTAs runs, partials summed after
  const int kb = (K + 63) / 64, tiles = ((M + 127) / 128) * ((N + 127) / 128);
  int splitk = 1;
  if (buf.part && tiles < 76) {
    int sk = 152 / tiles;
    sk = sk < kb ? sk : kb;
    sk = sk < 32 ? sk : 32;
    const int per = (kb + sk - 1) / sk;
    sk = (kb + per - 1) / per;
    if ((size_t)sk * M * N <= buf.part_floats) splitk = sk;
  }
  if (splitk == 1) {
    o.mode = TC_OUT_F32;
    o.f32 = C;
    o.cm = idx_plain(ldc);
    o.cn = idx_plain(1);
    return tc_gemm(A, B, M, N, K, 1, 6, 1, o, buf.err, st);
  }
  o.mode = TC_OUT_PARTIAL;
  o.f32 = buf.part;
  RET(tc_gemm(A, B, M, N, K, 1, 6, splitk, o, buf.err, st));
  note_launch();
  sum_partials_kernel<<<grid_for((long long)M * N), 256, 0, st>>>(buf.part, splitk, M, N, C, ldc);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Fast path of the orthonormalisation: scaled CholeskyQR2.
//
// Y = C_E V_prev + eta R has columns of very different norms (they follow
// the singular values of C_E), but once the warm start has converged they
// are close to orthogonal.  With the column scaling D = diag(1/||y_j||) the
// Gram G = D Y^T Y D is then well conditioned, and two CholeskyQR passes
// (G = L L^T, U = Y D L^{-T}) give an orthonormal U to FP32 level.  The
// Gram runs on the tensor cores (tc_product, 24-bit products, unbiased
// FP32 accumulation), the k x k Cholesky on one CTA in FP32 (blocked
// right-looking, packed lower triangle in shared memory), and the
// triangular solve on every SM (one warp per row, blocks of 32 columns).
// A column whose scaled pivot falls below tau is numerically dependent on
// the columns before it (a warm start far from converged, a growing bond) and
// is dropped; a column whose norm is zero is dead: their output columns are
// zero.
//
// Thresholds of the scaled pivot, the squared part of a unit column that is
// orthogonal to those before it.  First pass: the Gram's own error, up to 1e-6
// at k = 256.  Second pass: its columns are nearly orthonormal, and one with a
// small pivot is the remainder of a column that only just passed the first.
// That remainder still carries weight; dividing it by its norm raises the 3e-6
// of FP32 to 3e-6 / sqrt(pivot), which has to stay below the 1e-4 the caller
// accepts: 0.01 leaves a factor of three.  At 0.25 the second pass dropped 3 %
// more columns than the first had, and one sweep over random states (L = 8, D* =
// 50 to 128, 400 of them) discarded 15 % more weight than with Gram-Schmidt (+- 5 %);
// at 0.01 0.998 +- 0.045 of it, and at 1e-30 no less, but exact splits set in.
constexpr float CQ_TAU1 = 1e-6f, CQ_TAU2 = 0.01f;
constexpr int CQ_NT = 384;        // threads of the factor kernel (12 warps: up to 170 registers)
constexpr int CQ_SOLVE_NT = 256;  // threads of the solve kernel (8 warps, one row each)

__device__ __forceinline__ int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// shared memory of the factor kernel: the packed lower triangle, the
// transposed panel copy Pt[32][MAX_K], the scaling and the reciprocal pivots
constexpr int CQ_LD = 36;   // row stride of the factored diagonal block copy (16-byte rows)

size_t cholqr_factor_smem(int k) {
  const size_t packed = ((size_t)k * (k + 1) / 2 + 3) / 4 * 4;
  return (packed + (size_t)32 * MAX_K + 32 * CQ_LD + 2 * MAX_K) * 4;
}

// G (k x k FP32 row-major, symmetric; lower triangle read) -> Lout (packed
// lower Cholesky factor of D G D), dout (the scaling d_j; 0 for a dead
// column), linv_out (1 / L_jj, 0 for a dead column).  A column whose scaled
// pivot falls below tau (its part orthogonal to the columns before it is below
// sqrt(tau) of its norm: numerically dependent) is dropped as dead and counted
// in flag[4]; *flag = 1 if G is not finite (never cleared here).  Right-looking,
// 32-wide panels: the diagonal block in registers of warp 0 (lane = row, shuffles),
// the rows below it one per thread against that block, then the trailing
// update in 4 x 4 register blocks from the transposed panel copy (float4
// reads, conflict-free).  Measured at k = 64: 34 us with a column at a time and
// a row's loads at a time, 22 us so.  With run_if set, runs only if *run_if != 0 and
// *flag == 0.
__global__ void __launch_bounds__(CQ_NT, 1)
    cholqr_factor(const float* __restrict__ G, int k, float tau, float* __restrict__ Lout, float* __restrict__ dout, float* __restrict__ linv_out,
                  int* flag, const int* run_if) {
  if (run_if && (*run_if == 0 || *flag)) return;
  if (run_if && threadIdx.x == 0) atomicAdd(const_cast<int*>(run_if) + 1, 1);
  extern __shared__ __align__(16) float cq[];
  const int np = k * (k + 1) / 2;
  float* A = cq;                                    // packed lower triangle
  float* Pt = cq + ((np + 3) / 4 * 4);              // panel, transposed: Pt[t * MAX_K + row]
  float* Ld = Pt + 32 * MAX_K;                      // factored diagonal block, Ld[r * CQ_LD + c]
  float* d = Ld + 32 * CQ_LD;                       // scaling
  float* li = d + MAX_K;                            // 1 / L_jj
  __shared__ float red[32];
  __shared__ int bad, ndefl;
  __shared__ float4 colb[32];   // four columns of the diagonal-block step
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  float gm = 0.f;
  for (int j = tid; j < k; j += CQ_NT) {
    const float g = G[(long long)j * k + j];
    gm = fmaxf(gm, (g == g) ? g : 3.0e38f);
  }
  for (int o = 16; o > 0; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  if (lane == 0) red[warp] = gm;
  if (tid == 0) {
    bad = 0;
    ndefl = 0;
  }
  __syncthreads();
  if (tid < 32) {
    float v = tid < CQ_NT / 32 ? red[tid] : 0.f;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (tid == 0) red[0] = v;
  }
  __syncthreads();
  const float gmax = red[0];
  for (int j = tid; j < k; j += CQ_NT) {
    const float g = G[(long long)j * k + j];
    d[j] = (g > 1e-30f * gmax && g < 3.0e38f) ? 1.f / sqrtf(g) : 0.f;
  }
  __syncthreads();
  // packed load, a warp per row (coalesced reads of G), three rows at a time:
  // all their loads are issued before any is used, so a warp waits out the
  // memory latency once per three rows
  constexpr int LR = 3;
  for (int i0 = warp; i0 < k; i0 += LR * (CQ_NT / 32)) {
    float g[LR][MAX_K / 32];
#pragma unroll
    for (int v = 0; v < LR; ++v) {
      const int i = i0 + v * (CQ_NT / 32);
#pragma unroll
      for (int t = 0; t < MAX_K / 32; ++t) {
        const int j = lane + 32 * t;
        g[v][t] = (i < k && j <= i) ? G[(long long)i * k + j] : 0.f;
      }
    }
#pragma unroll
    for (int v = 0; v < LR; ++v) {
      const int i = i0 + v * (CQ_NT / 32);
      const float di = i < k ? d[i] : 0.f;
#pragma unroll
      for (int t = 0; t < MAX_K / 32; ++t) {
        const int j = lane + 32 * t;
        if (i < k && j <= i) {
          const float x = g[v][t] * di * d[j];
          A[pk(i, j)] = (x == x) ? x : 0.f;
          if (x != x) bad = 1;
        }
      }
    }
  }
  __syncthreads();
  for (int p0 = 0; p0 < k; p0 += 32) {
    const int pw = min(32, k - p0);
    // (a) the diagonal block: lane r holds row p0 + r (columns p0..p0+31)
    if (warp == 0) {
      float r[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) r[c] = (lane < pw && c <= lane) ? A[pk(p0 + lane, p0 + c)] : 0.f;
      // dead columns of the block (zero scaling) as one bit per lane; pivots
      // that break down, collected the same way (the pivot is warp-uniform)
      const unsigned deadm = __ballot_sync(0xffffffffu, lane < pw && d[p0 + lane] == 0.f);
      unsigned brokem = 0;
      float myinv = 0.f;
      // Four columns at a time: their 4 x 4 diagonal block comes to every lane
      // by ten shuffles and is factored by all of them alike, each lane solves
      // its row's four entries against it, and these go through shared memory
      // once, read back as float4 broadcasts by the trailing update.  (A column
      // at a time the chain pivot - scaling - store - read ran 32 times, 400
      // clocks each.)  Entries above the diagonal hold values nobody reads.
#pragma unroll
      for (int jb = 0; jb < 8; ++jb) {
        const int j0 = 4 * jb;
        if (j0 < pw) {
          float l[4][4], iv[4], x[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c <= i; ++c) l[i][c] = __shfl_sync(0xffffffffu, r[j0 + c], j0 + i);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float piv = l[c][c];
            const bool dead = ((deadm >> (j0 + c)) & 1u) || j0 + c >= pw;
            const bool broke = !dead && !(piv > tau);
            const float rs = rsqrtf(piv);
            const bool good = !(dead || broke);
            l[c][c] = good ? piv * rs : 1.f;
            iv[c] = good ? rs : 0.f;
            if (broke) brokem |= 1u << (j0 + c);
#pragma unroll
            for (int i = c + 1; i < 4; ++i) l[i][c] *= iv[c];
#pragma unroll
            for (int i = c + 1; i < 4; ++i)
#pragma unroll
              for (int k = c + 1; k <= i; ++k) l[i][k] = fmaf(-l[i][c], l[k][c], l[i][k]);
            if (lane == j0 + c) myinv = iv[c];
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            float v = r[j0 + c];
#pragma unroll
            for (int k = 0; k < c; ++k) v = fmaf(-x[k], l[c][k], v);
            x[c] = v * iv[c];
            r[j0 + c] = lane == j0 + c ? l[c][c] : (lane > j0 + c ? x[c] : r[j0 + c]);
          }
          if (j0 < 28) {
            colb[lane] = make_float4(x[0], x[1], x[2], x[3]);
            __syncwarp();
            // trailing part of the block: r[c] -= sum of L_lane,. L_c,.
#pragma unroll
            for (int c = j0 + 4; c < 32; ++c) {
              const float4 y = colb[c];
              r[c] = fmaf(-x[0], y.x, r[c]);
              r[c] = fmaf(-x[1], y.y, r[c]);
              r[c] = fmaf(-x[2], y.z, r[c]);
              r[c] = fmaf(-x[3], y.w, r[c]);
            }
            __syncwarp();
          }
        }
      }
      if (lane < pw) li[p0 + lane] = myinv;
      if (lane == 0 && brokem) ndefl += __popc(brokem);
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        if (lane < pw && c <= lane) A[pk(p0 + lane, p0 + c)] = r[c];
        Ld[lane * CQ_LD + c] = (lane < pw && c <= lane) ? r[c] : 0.f;
      }
    }
    __syncthreads();
    // (b) rows below the block: L_ip = A_ip L_pp^{-T}, one thread per row;
    // the rows of L_pp are read as float4 broadcasts and each dot product
    // runs in four partial sums (short dependency chains)
    for (int i = p0 + pw + tid; i < k; i += CQ_NT) {
      float x[32];
      const int base = pk(i, p0);
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        if (t < pw) {
          float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int q4 = 0; q4 < 8; ++q4) {
            if (4 * q4 < t) {
              const float4 l = *reinterpret_cast<const float4*>(Ld + t * CQ_LD + 4 * q4);
              // entries q >= t of row t are zero in Ld (and x[q] for q >= t
              // is not yet defined): only q < t is taken
              s4[0] = fmaf(x[4 * q4], l.x, s4[0]);
              if (4 * q4 + 1 < t) s4[1] = fmaf(x[4 * q4 + 1], l.y, s4[1]);
              if (4 * q4 + 2 < t) s4[2] = fmaf(x[4 * q4 + 2], l.z, s4[2]);
              if (4 * q4 + 3 < t) s4[3] = fmaf(x[4 * q4 + 3], l.w, s4[3]);
            }
          }
          x[t] = (A[base + t] - ((s4[0] + s4[1]) + (s4[2] + s4[3]))) * li[p0 + t];
        }
      }
#pragma unroll
      for (int t = 0; t < 32; ++t)
        if (t < pw) {
          A[base + t] = x[t];
          Pt[t * MAX_K + i] = x[t];
        }
    }
    __syncthreads();
    // (c) trailing update A_ic -= sum_t L_it L_ct for p0+pw <= c <= i
    const int r0 = p0 + pw, n = k - r0;
    if (n > 0) {
      const int nb = (n + 3) / 4, nblk = nb * (nb + 1) / 2;
      for (int bidx = tid; bidx < nblk; bidx += CQ_NT) {
        int bi = (int)((sqrtf(8.f * (float)bidx + 1.f) - 1.f) * 0.5f);
        while (bi * (bi + 1) / 2 > bidx) --bi;
        while ((bi + 1) * (bi + 2) / 2 <= bidx) ++bi;
        const int bc = bidx - bi * (bi + 1) / 2;
        const int i0 = r0 + 4 * bi, c0 = r0 + 4 * bc;
        float acc[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
        // i0, c0 are multiples of 4 below MAX_K: whole float4 reads.  Rows
        // of Pt past k hold stale values; they only reach the entries of acc
        // with i >= k or c >= k, which are not stored.
#pragma unroll 8
        for (int t = 0; t < pw; ++t) {
          const float4 a = *reinterpret_cast<const float4*>(Pt + t * MAX_K + i0);
          const float4 b = *reinterpret_cast<const float4*>(Pt + t * MAX_K + c0);
          const float pi[4] = {a.x, a.y, a.z, a.w}, pc[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(pi[u], pc[v], acc[u][v]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const int i = i0 + u, c = c0 + v;
            if (i < k && c <= i) A[pk(i, c)] -= acc[u][v];
          }
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < np; e += CQ_NT) Lout[e] = A[e];
  for (int j = tid; j < k; j += CQ_NT) {
    dout[j] = d[j];
    linv_out[j] = li[j];
  }
  if (tid == 0 && bad) atomicExch(flag, 1);
  if (tid == 0 && ndefl) atomicAdd(flag + 4, ndefl);
}

// BF16 planes of U and U^T (3 planes each; both null: not wanted).
struct SolvePlanes {
  __nv_bfloat16* rm;   // [plane][rows][ldk], plane stride ps_rm
  long long ldk, ps_rm;
  __nv_bfloat16* tr;   // [plane][k][ldr], plane stride ps_tr
  long long ldr, ps_tr;
};

// U[r] = (Y[r] o d) L^{-T} for every row r (one warp per row; rows ldy / ldu
// apart, so a column block of a wider matrix works in place): with u L^T = z,
// u_j = (z_j - sum_{i<j} u_i L_ji) / L_jj, in blocks of 32 columns (earlier
// blocks first, then a sequential solve inside the block).  Does nothing if
// *flag is set (the factor met a non-finite Gram) or, with run_if set, if *run_if is
// 0.  U may be Y itself (ldu = ldy): each row is read by the lanes that
// write it, column j before U[r][j].  With planes, U's and U^T's BF16 planes
// are written too, the operands of the next two products (the eight rows of
// a CTA are one 16-byte store per column of U^T).
__global__ void __launch_bounds__(CQ_SOLVE_NT)
    cholqr_solve(const float* Y, long long ldy, int rows, int k,
                 const float* __restrict__ Lp, const float* __restrict__ dv,
                 const float* __restrict__ linv, const int* __restrict__ flag,
                 const int* __restrict__ run_if, float* U, long long ldu, SolvePlanes pl) {
  if (*flag || (run_if && *run_if == 0)) return;
  extern __shared__ __align__(16) float Ls[];
  constexpr int WPB = CQ_SOLVE_NT / 32;
  static_assert(WPB == 8, "eight rows a CTA: one 16-byte store per column and plane");
  __shared__ __align__(16) unsigned short tp[3][MAX_K][WPB];
  const int np = k * (k + 1) / 2;
  // the packed factor (16-byte aligned in global memory), 16 bytes per load
  const int n4 = np / 4;
#pragma unroll 4
  for (int e = threadIdx.x; e < n4; e += CQ_SOLVE_NT)
    reinterpret_cast<float4*>(Ls)[e] = reinterpret_cast<const float4*>(Lp)[e];
  for (int e = 4 * n4 + threadIdx.x; e < np; e += CQ_SOLVE_NT) Ls[e] = Lp[e];
  __syncthreads();
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  for (int r0 = blockIdx.x * WPB; r0 < rows; r0 += gridDim.x * WPB) {
    const int r = r0 + warp;
    const bool in = r < rows;
    float x[MAX_K / 32];
#pragma unroll
    for (int qb = 0; qb < MAX_K / 32; ++qb) {
      x[qb] = 0.f;
      if (qb * 32 < k) {
        const int j = qb * 32 + lane;
        float s = (in && j < k) ? Y[(long long)r * ldy + j] * dv[j] : 0.f;
        // earlier blocks
#pragma unroll
        for (int q = 0; q < MAX_K / 32; ++q) {
          if (q < qb) {
#pragma unroll 8
            for (int t = 0; t < 32; ++t) {
              const float xt = __shfl_sync(0xffffffffu, x[q], t);
              if (j < k) s = fmaf(-xt, Ls[pk(j, q * 32 + t)], s);
            }
          }
        }
        // inside the block (1 / L_jj read before the chain: a load inside it,
        // one per step, put the memory latency on the chain 32 times)
        const float lij = (j < k) ? linv[j] : 0.f;
        float xj = 0.f;
#pragma unroll
        for (int t = 0; t < 32; ++t) {
          if (qb * 32 + t < k) {
            if (lane == t) xj = s * lij;
            const float xt = __shfl_sync(0xffffffffu, xj, t);
            if (lane > t && j < k) s = fmaf(-xt, Ls[pk(j, qb * 32 + t)], s);
          }
        }
        x[qb] = xj;
        if (in && j < k) U[(long long)r * ldu + j] = xj;
        if (pl.rm && j < pl.ldk) {
          unsigned short w[3] = {0, 0, 0};
          if (j < k) cut(xj, w);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            if (in) pl.rm[q * pl.ps_rm + (long long)r * pl.ldk + j] = __ushort_as_bfloat16(w[q]);
            tp[q][j][warp] = w[q];
          }
        }
      }
    }
    if (pl.rm) {
      __syncthreads();
      // rows past the last one were zero, as the padding of U^T has to be
      if (r0 < pl.ldr)
        for (int e = threadIdx.x; e < 3 * k; e += CQ_SOLVE_NT) {
          const int q = e / k, j = e - q * k;
          *reinterpret_cast<uint4*>(pl.tr + q * pl.ps_tr + (long long)j * pl.ldr + r0) =
              *reinterpret_cast<const uint4*>(tp[q][j]);
        }
      __syncthreads();
    }
  }
}

// shared-memory opt-in of the two CholeskyQR kernels, once per device
PerDevice<cudaError_t> g_cholqr_setup;

cudaError_t cholqr_setup() {
  cudaError_t r = cudaSuccess;
  cudaError_t e = g_cholqr_setup.get(
      [](int) {
        cudaError_t x = cudaFuncSetAttribute(cholqr_factor,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)cholqr_factor_smem(MAX_K));
        if (x == cudaSuccess)
          x = cudaFuncSetAttribute(cholqr_solve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)((size_t)MAX_K * (MAX_K + 1) / 2 * 4));
        return x;
      },
      &r);
  return e != cudaSuccess ? e : r;
}

// Two scaled CholeskyQR passes on the column block Yb (rows x w, row stride
// ldy): Yb -> U1 (in tmp, row stride w) -> Yb.  A non-finite Gram raises
// b.chol_flag[0] and leaves Yb as it was.
cudaError_t cholqr2_block(float* Yb, long long ldy, int rows, int w, float* tmp,
                          const SubspaceBuffers& b, cudaStream_t st) {
  const size_t fsm = cholqr_factor_smem(w), ssm = (size_t)w * (w + 1) / 2 * 4;
  const int wpb = CQ_SOLVE_NT / 32;
  int grid = (rows + wpb - 1) / wpb;
  if (grid > 152) grid = 152;
  const float* src = Yb;
  long long lds = ldy;
  float* dst = tmp;
  long long ldd = w;
  for (int pass = 0; pass < 2; ++pass) {
    // G = Yb^T Yb (w x w) on the tensor cores
    RET(tc_product(f32_view(src, idx_plain(1), idx_plain(lds)),
                   f32_view(src, idx_plain(1), idx_plain(lds)), w, w, rows, b.out, w, b, st));
    note_launch();
    cholqr_factor<<<1, CQ_NT, fsm, st>>>(b.out, w, pass == 0 ? CQ_TAU1 : CQ_TAU2,
                                         b.chol_L, b.chol_d, b.chol_li, b.chol_flag, nullptr);
    RET(cudaGetLastError());
    note_launch();
    cholqr_solve<<<grid, CQ_SOLVE_NT, ssm, st>>>(src, lds, rows, w, b.chol_L, b.chol_d, b.chol_li,
                                                 b.chol_flag, nullptr, dst, ldd, SolvePlanes{});
    RET(cudaGetLastError());
    src = tmp;
    lds = w;
    dst = Yb;
    ldd = ldy;
  }
  return cudaSuccess;
}

// Yb[r][c] -= Z[r][c] (Yb row stride ldy, Z row stride w), unless *flag
__global__ void subtract_block_kernel(float* __restrict__ Yb, long long ldy,
                                      const float* __restrict__ Z, int rows, int w,
                                      const int* __restrict__ flag) {
  if (*flag) return;
  const long long total = (long long)rows * w;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / w, c = e % w;
    Yb[r * ldy + c] -= Z[e];
  }
}

// The second CholeskyQR pass to first order.  After the first pass the Gram
// of U1 is G2 = I + E with E small; its Cholesky factor is L = I + Phi(E) +
// O(E^2), Phi(E) the strictly lower part of E plus half its diagonal, so
// U2 = U1 L^{-T} = U1 (I - Phi(E)^T) + O(E^2) and U2^T U2 = I + O(E^2).
// Writes B = I - Phi(E) (k x k: U2 = U1 B^T is one tensor-core product);
// dead columns (zero columns of U1) keep B's row e_j and get zeros elsewhere.
// If a live |E_ij| exceeds emax (or is not finite), or a column that is not zero
// has lost half its norm (G2_jj < 1/2: the first order cannot restore it), sets
// *need_full: the full second pass runs instead (and counts itself in
// need_full[1]).
// G comes as the partials of its split contraction: summed here, with the
// sum written to G for the full second pass; B as its BF16 planes.
__global__ void __launch_bounds__(256)
    cholqr_linear_kernel(const float* __restrict__ part, int splits, int k, float emax,
                         float* __restrict__ G, __nv_bfloat16* __restrict__ B, long long ldb,
                         long long psb, int* need_full) {
  __shared__ float dn[32], dc[32];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int n0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const long long kk = (long long)k * k;
  // the thread's four entries and, in two warps, a diagonal entry of the
  // tile's rows or columns, summed side by side
  long long at[5];
  bool in[5];
  const int di = (ty ? c0 : n0) + tx;
  at[4] = (long long)di * k + di;
  in[4] = ty < 2 && di < k;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int n = n0 + ty + 8 * u, c = c0 + tx;
    at[u] = (long long)n * k + c;
    in[u] = n < k && c < k;
  }
  float g[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int s = 0; s < splits; ++s)
#pragma unroll
    for (int u = 0; u < 5; ++u)
      if (in[u]) g[u] += part[s * kk + at[u]];
  if (ty < 2) (ty ? dc : dn)[tx] = g[4];
  __syncthreads();
  bool big = false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int n = n0 + ty + 8 * u, c = c0 + tx;
    if (n >= k || c >= ldb) continue;
    const float gn = dn[ty + 8 * u], gc = dc[tx];
    float v = 0.f;
    if (c < k) {
      if (!(gn >= 0.5f)) {
        v = (n == c) ? 1.f : 0.f;
        if (n == c && gn != 0.f) big = true;
      } else if (gc >= 0.5f) {
        const float E = (n == c) ? gn - 1.f : g[u];
        if (!(fabsf(E) <= emax)) big = true;
        v = (n == c) ? 1.f - 0.5f * E : (n > c ? -E : 0.f);
      }
      G[(long long)n * k + c] = g[u];
    }
    unsigned short w[3];
    cut(v, w);
#pragma unroll
    for (int q = 0; q < 3; ++q) B[q * psb + (long long)n * ldb + c] = __ushort_as_bfloat16(w[q]);
  }
  if (__syncthreads_or(big) && threadIdx.x == 0) atomicExch(need_full, 1);
}

// Largest |E_ij| of the first-order second pass; above it the full second
// CholeskyQR pass runs.  The neglected O(E^2) terms (up to about 4 k E^2 in
// the max norm, typically ~1e-5 at k = 256) stay below the orthonormality
// check's bound; removing them by one more first-order correction of the
// checked basis was measured not to change the free energy.
constexpr float CQ_LINEAR_EMAX = 1e-3f;

// An orthonormal basis of the columns of Y (rows x k, FP32) for k wider than
// one column block, in place: block classical Gram-Schmidt over column blocks,
// each projected twice against the blocks before it on the tensor cores (S =
// Q^T Y_b, Y_b -= Q S) and then orthonormalised by scaled CholeskyQR2; a
// non-finite Gram leaves Y as it was, which the caller's check turns into the
// exact split.  b.Q is overwritten.
cudaError_t orthonormalise_blocks(float* Y, int rows, int k, const SubspaceBuffers& b,
                                  cudaStream_t st) {
  if (k > SUBSPACE_MAX_K) return cudaErrorInvalidValue;
  RET(cholqr_setup());
  const int B = b.orth_block;
  if (B < 32 || B > MAX_K || B % 32) return cudaErrorInvalidValue;
  for (int j0 = 0; j0 < k; j0 += B) {
    const int w = k - j0 < B ? k - j0 : B;
    float* Yb = Y + j0;
    for (int pass = 0; pass < 2 && j0 > 0; ++pass) {
      // S (j0 x w, in b.out) = Q^T Y_b with Q = Y[:, :j0]
      RET(tc_product(f32_view(Y, idx_plain(1), idx_plain(k)), f32_view(Yb, idx_plain(1), idx_plain(k)),
                     j0, w, rows, b.out, w, b, st));
      // Z (rows x w, in b.Q) = Q S
      RET(tc_product(f32_view(Y, idx_plain(k), idx_plain(1)), f32_view(b.out, idx_plain(1), idx_plain(w)),
                     rows, w, j0, b.Q, w, b, st));
      note_launch();
      subtract_block_kernel<<<grid_for((long long)rows * w), 256, 0, st>>>(Yb, k, b.Q, rows, w,
                                                                           b.chol_flag);
      RET(cudaGetLastError());
    }
    RET(cholqr2_block(Yb, k, rows, w, b.Q, b, st));
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// The truncation up to one column block (k <= b.orth_block), a chain of
// kernels each bound by its launch and latency at the bonds met here: every
// tensor-core product leaves its split-K partials, and the kernel after it
// sums them and writes the next product's operand planes, so that no pass
// only sums, converts, copies or clears.  U_hat is the basis kept as planes of
// its transpose (U^T left-to-right, V^T right-to-left) behind C_E's planes, so
// that one product gives both the centre and the Gram of the check.

// warm start as planes: out[j][r] = src(j, r) = S[j * sj + r * sr] for j <
// kold, else pseudo-random (k rows of ld columns).  Clears the scalars of the
// update (zero_words words at zero, and the two flags).
__global__ void __launch_bounds__(256)
    warm_planes_kernel(const double* __restrict__ S, long long sj, long long sr, int kold, int rows,
                       int k, unsigned long long seed0,
                       const unsigned long long* __restrict__ base, __nv_bfloat16* __restrict__ out,
                       long long ld, long long ps, int* zero, int zero_words, int* flags) {
  __shared__ __align__(16) unsigned short tp[3][32][72];
  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    if (tid < zero_words) zero[tid] = 0;
    if (tid == 64) flags[0] = 0;
    if (tid == 65) flags[2] = 0;
  }
  const unsigned long long seed = seed0 ^ (*base * 0x9E3779B97F4A7C15ull);
  const int j0 = blockIdx.y * 32, r0 = blockIdx.x * 64;
  const bool rfast = sr == 1;
  double x[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int j = j0 + (rfast ? tid / 64 + 4 * u : tid % 32);
    const int r = r0 + (rfast ? tid % 64 : tid / 32 + 8 * u);
    x[u] = (j < kold && r < rows) ? S[j * sj + r * sr] : 0.0;
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int y = rfast ? tid / 64 + 4 * u : tid % 32, z = rfast ? tid % 64 : tid / 32 + 8 * u;
    const int j = j0 + y, r = r0 + z;
    unsigned short w[3];
    if (j >= kold && r < rows)
      cut(hash_uniform(seed * 0x100000001B3ull + (unsigned long long)r * k + j), w);
    else
      cut(x[u], w);
    tp[0][y][z] = w[0];
    tp[1][y][z] = w[1];
    tp[2][y][z] = w[2];
  }
  __syncthreads();
  const int y = tid / 8, z = tid % 8 * 8, j = j0 + y, r = r0 + z;
  if (j < k && r < ld)
#pragma unroll
    for (int q = 0; q < 3; ++q)
      *reinterpret_cast<uint4*>(out + q * ps + (long long)j * ld + r) =
          *reinterpret_cast<const uint4*>(&tp[q][y][z]);
}

// The source of one basis factor (rows x k, row-major FP32): the sum of a
// product's partials, or a finished array chosen on the device.
struct BasisSrc {
  const float* part;
  int splits;
  const float* alt1;   // taken instead if *flag1 != 0
  const int* flag1;
  const float* alt2;   // taken instead if *flag2 != 0 (and not alt1)
  const int* flag2;
};

// F = source (+ noise eta R with eta = 1e-5 rms(C_E)); written as FP32 (f32,
// may be null), FP64 row-major (f64) or transposed (f64t), and as planes of
// F^T [plane][k][ldr] (zero padding).  Tiles of 64 rows x 32 columns.
__global__ void __launch_bounds__(256)
    basis_kernel(BasisSrc src, int rows, int k, const double* __restrict__ tot, double inv_mn,
                 unsigned long long seed0, const unsigned long long* __restrict__ base, float* f32,
                 double* f64, double* f64t, __nv_bfloat16* __restrict__ out, long long ldr,
                 long long ps) {
  __shared__ float v[32][65];   // [column][row]
  const int tid = threadIdx.x, tx = tid % 32, ty = tid / 32;
  const int r0 = blockIdx.x * 64, j0 = blockIdx.y * 32;
  const float* alt = nullptr;
  if (src.flag1 && *src.flag1) alt = src.alt1;
  else if (src.flag2 && *src.flag2) alt = src.alt2;
  const long long n = (long long)rows * k;
  float a[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = r0 + ty + 8 * u, j = j0 + tx;
    a[u] = 0.f;
    if (alt && r < rows && j < k) a[u] = alt[(long long)r * k + j];
  }
  if (!alt) {
#pragma unroll 2
    for (int s = 0; s < src.splits; ++s)
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + ty + 8 * u, j = j0 + tx;
        if (r < rows && j < k) a[u] += src.part[s * n + (long long)r * k + j];
      }
  }
  if (tot) {
    const unsigned long long seed = seed0 ^ (*base * 0x9E3779B97F4A7C15ull);
    const float eta = (float)(1e-5 * sqrt(*tot * inv_mn));
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const long long e = (long long)(r0 + ty + 8 * u) * k + j0 + tx;
      a[u] += eta * hash_uniform(seed ^ (0xD1B54A32D192ED03ull * (unsigned long long)(e + 1)));
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = r0 + ty + 8 * u, j = j0 + tx;
    const bool in = r < rows && j < k;
    v[tx][ty + 8 * u] = in ? a[u] : 0.f;
    if (in && f32) f32[(long long)r * k + j] = a[u];
    if (in && f64) f64[(long long)r * k + j] = (double)a[u];
  }
  __syncthreads();
  {
    const int y = tid / 8, z = tid % 8 * 8, j = j0 + y, r = r0 + z;
    if (j < k && r < ldr) {
      __align__(16) unsigned short w[3][8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        unsigned short c[3];
        cut(v[y][z + u], c);
        w[0][u] = c[0];
        w[1][u] = c[1];
        w[2][u] = c[2];
      }
#pragma unroll
      for (int q = 0; q < 3; ++q)
        *reinterpret_cast<uint4*>(out + q * ps + (long long)j * ldr + r) =
            *reinterpret_cast<const uint4*>(w[q]);
    }
  }
  if (f64t)
    for (int e = tid; e < 32 * 64; e += 256) {
      const int j = j0 + e / 64, r = r0 + e % 64;
      if (j < k && r < rows) f64t[(long long)j * rows + r] = (double)v[e / 64][e % 64];
    }
}

// The last product: its partials (R x Cc) hold the centre and, in the columns
// from c_gram on (left-to-right) or the rows from r_gram on, the Gram of the
// kept basis.  Writes the centre in FP64 (row stride ldo), adds its sum of
// squares, raises the orthonormality defect over the live columns; the last
// CTA to finish sets the defect to +inf when no column is live, raises the
// discarded weight of an accepted split into *disc_max (may be null) and
// clears ||C_E||^2 for the next update.
struct CentreOut {
  double* out;
  int ldo, r_gram, c_gram, k;
  double* dscal;   // [1] sum of squares, [2] defect
  int* live;       // [0] a live column seen, [1] CTAs finished
  double* ce_ss;
  double thresh;
  double* disc_max;
};
__global__ void __launch_bounds__(256)
    centre_kernel(const float* __restrict__ part, int splits, int R, int Cc, CentreOut o) {
  __shared__ float dr[32], dc[32];
  __shared__ double red[8];
  __shared__ float redf[8];
  __shared__ int last;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const long long n = (long long)R * Cc;
  const bool grams = r0 + 31 >= o.r_gram || c0 + 31 >= o.c_gram;   // some Gram entry in this tile
  const int ro = o.r_gram < R ? o.r_gram : 0, co = o.c_gram < Cc ? o.c_gram : 0;
  // the thread's four entries and, in two warps of a tile with Gram entries,
  // the diagonal entry of the Gram index of the tile's rows (ty = 0) or columns
  // (ty = 1), summed side by side
  long long at[5];
  bool in[5];
  const int di = ty == 0 ? r0 + tx - ro : c0 + tx - co;
  at[4] = (long long)(di + ro) * Cc + di + co;
  in[4] = grams && ty < 2 && di >= 0 && di < o.k;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = r0 + ty + 8 * u, c = c0 + tx;
    at[u] = (long long)r * Cc + c;
    in[u] = r < R && c < Cc;
  }
  float v4[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
  for (int s = 0; s < splits; ++s)
#pragma unroll
    for (int u = 0; u < 5; ++u)
      if (in[u]) v4[u] += part[s * n + at[u]];
  if (grams && ty < 2) (ty ? dc : dr)[tx] = v4[4];
  if (grams) __syncthreads();
  double acc = 0.0;
  float mx = 0.f;
  int live = 0;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = r0 + ty + 8 * u, c = c0 + tx;
    if (r >= R || c >= Cc) continue;
    const float v = v4[u];
    if (r < o.r_gram && c < o.c_gram) {
      const double d = (double)v;
      o.out[(long long)r * o.ldo + c] = d;
      acc = fma(d, d, acc);
    } else {
      const int i = r - ro, j = c - co;
      const float gi = dr[ty + 8 * u], gj = dc[tx];
      if (i == j && gi >= 0.5f) live = 1;
      if (!(gi < 0.5f || gj < 0.5f)) {
        const float d = fabsf(v - (i == j ? 1.f : 0.f));
        mx = fmaxf(mx, d != d ? 1e30f : d);
      }
    }
  }
  for (int s = 16; s > 0; s >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, s);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
  }
  if (tx == 0) {
    red[ty] = acc;
    redf[ty] = mx;
  }
  const int any_live = __syncthreads_or(live);
  if (threadIdx.x == 0) {
    double t = 0.0;
    float m = 0.f;
    for (int i = 0; i < 8; ++i) {
      t += red[i];
      m = fmaxf(m, redf[i]);
    }
    if (t != 0.0) atomicAdd(o.dscal + 1, t);
    // non-negative doubles order like their bit patterns
    if (m > 0.f)
      atomicMax(reinterpret_cast<unsigned long long*>(o.dscal + 2),
                (unsigned long long)__double_as_longlong((double)m));
    if (any_live) atomicOr(o.live, 1);
    __threadfence();
    last = atomicAdd(o.live + 1, 1) == (int)(gridDim.x * gridDim.y) - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    const double tot = __ldcg(o.ce_ss), kept = __ldcg(o.dscal + 1);
    double defect = __ldcg(o.dscal + 2);
    if (__ldcg(o.live) == 0) {
      defect = INFINITY;
      o.dscal[2] = defect;
    }
    const double disc = tot > 0.0 ? fmax(0.0, 1.0 - kept / tot) : 0.0;
    if (o.disc_max && defect <= o.thresh)
      atomicMax(reinterpret_cast<unsigned long long*>(o.disc_max),
                (unsigned long long)__double_as_longlong(disc));
    *o.ce_ss = 0.0;
  }
}

// A B^T on the tensor cores (3 planes, 6 products) as split-K partials in
// b.part; *splits: their number.  Products with few output tiles split K so
// that about one wave of CTAs runs.
cudaError_t tc_partials(const TcOperand& A, const TcOperand& B, int M, int N, int K, int* splits,
                        const SubspaceBuffers& b, cudaStream_t st) {
  const int kb = (K + 63) / 64, tiles = ((M + 127) / 128) * ((N + 127) / 128);
  int sk = 1;
  if (tiles < 76) {
    sk = 152 / tiles;
    sk = sk < kb ? sk : kb;
    sk = sk < 32 ? sk : 32;
    const int per = (kb + sk - 1) / sk;
    sk = (kb + per - 1) / per;
    while (sk > 1 && (size_t)sk * M * N > b.part_floats) --sk;
  }
  if ((size_t)sk * M * N > b.part_floats) return cudaErrorInvalidValue;
  TcOutput o;
  memset(&o, 0, sizeof o);
  o.alpha = 1.0;
  o.mode = TC_OUT_PARTIAL;
  o.f32 = b.part;
  *splits = sk;
  return tc_gemm(A, B, M, N, K, 1, 6, sk, o, b.err, st);
}

TcOperand plane_op(const __nv_bfloat16* p, int rows, int k, long long ld, long long ps) {
  return TcOperand{p, 3, rows, k, ld, 0, ps, 1};
}

cudaError_t narrow_split(int m, int n, int k, int dir_right, const double* warm, int kold,
                         double* left, double* right, unsigned long long seed,
                         const SubspaceBuffers& b, cudaStream_t st, double* disc_max,
                         double thresh) {
  RET(cholqr_setup());
  // the basis has `rows` rows on the side of the isometry, the other side is
  // `other`; ce: C_E with that side as rows, behind it the basis' transpose
  const int rows = dir_right ? m : n, other = dir_right ? n : m;
  const long long ldr = tc_ld(rows), ldo = tc_ld(other), ldk = tc_ld(k);
  const __nv_bfloat16* ce = dir_right ? b.ce_rm : b.ce_tr;      // rows x other
  __nv_bfloat16* cet = dir_right ? b.ce_tr : b.ce_rm;           // other x rows
  __nv_bfloat16* hat = cet + (long long)other * ldr;            // k x rows: the basis, transposed
  if ((long long)(other + k) * ldr > b.ce_ps || (long long)rows * ldk > b.psa ||
      (long long)k * ldr > b.psb || (long long)k * ldo > b.psb || (long long)k * ldk > b.psb)
    return cudaErrorInvalidValue;
  const size_t fsm = cholqr_factor_smem(k), ssm = (size_t)k * (k + 1) / 2 * 4;
  const int wpb = CQ_SOLVE_NT / 32;
  const int sgrid = (rows + wpb - 1) / wpb < 152 ? (rows + wpb - 1) / wpb : 152;
  const dim3 bgrid((unsigned)((ldr + 63) / 64), (unsigned)((k + 31) / 32));
  float* G = b.out;
  int* need_full = b.chol_flag + 2;
  int sp = 1;
  // warm start Q^T (k x other): the current C_{i+1} rows or C_i columns
  note_launch();
  warm_planes_kernel<<<dim3((unsigned)((ldo + 63) / 64), (unsigned)((k + 31) / 32)), 256, 0, st>>>(
      warm, dir_right ? n : 1, dir_right ? 1 : kold, kold, other, k, seed, b.seed_base, b.pb, ldo,
      b.psb, b.zero, b.zero_words, b.chol_flag);
  RET(cudaGetLastError());
  // Y = C_E Q (rows x k) + noise, and the planes of Y^T
  RET(tc_partials(plane_op(ce, rows, other, ldo, b.ce_ps), plane_op(b.pb, k, other, ldo, b.psb), rows,
                  k, other, &sp, b, st));
  note_launch();
  basis_kernel<<<bgrid, 256, 0, st>>>(BasisSrc{b.part, sp, nullptr, nullptr, nullptr, nullptr}, rows,
                                      k, b.ce_ss, 1.0 / ((double)m * n), seed + 7, b.seed_base, b.Y,
                                      nullptr, nullptr, hat, ldr, b.ce_ps);
  RET(cudaGetLastError());
  // pass 1: G = Y^T Y, scaled Cholesky, Y <- U1 in place (skipped if G is not finite)
  const TcOperand H = plane_op(hat, k, rows, ldr, b.ce_ps);
  RET(tc_partials(H, H, k, k, rows, &sp, b, st));
  note_launch();
  sum_partials_kernel<<<grid_for((long long)k * k), 256, 0, st>>>(b.part, sp, k, k, G, k);
  note_launch();
  cholqr_factor<<<1, CQ_NT, fsm, st>>>(G, k, CQ_TAU1, b.chol_L, b.chol_d, b.chol_li, b.chol_flag,
                                       nullptr);
  RET(cudaGetLastError());
  note_launch();
  cholqr_solve<<<sgrid, CQ_SOLVE_NT, ssm, st>>>(b.Y, k, rows, k, b.chol_L, b.chol_d, b.chol_li,
                                                b.chol_flag, nullptr, b.Y, k,
                                                SolvePlanes{b.pa, ldk, b.psa, hat, ldr, b.ce_ps});
  RET(cudaGetLastError());
  // pass 2 to first order: G = U1^T U1 = I + E, U2 = U1 (I - Phi(E)^T)
  RET(tc_partials(H, H, k, k, rows, &sp, b, st));
  note_launch();
  const unsigned kt = (unsigned)((ldk + 31) / 32);
  cholqr_linear_kernel<<<dim3(kt, kt), 256, 0, st>>>(b.part, sp, k, CQ_LINEAR_EMAX, G, b.pb, ldk,
                                                     b.psb, need_full);
  RET(cudaGetLastError());
  // the full second pass, only if E was too large: U1 -> b.Q
  note_launch();
  cholqr_factor<<<1, CQ_NT, fsm, st>>>(G, k, CQ_TAU2, b.chol_L, b.chol_d, b.chol_li, b.chol_flag,
                                       need_full);
  RET(cudaGetLastError());
  note_launch();
  cholqr_solve<<<sgrid, CQ_SOLVE_NT, ssm, st>>>(b.Y, k, rows, k, b.chol_L, b.chol_d, b.chol_li,
                                                b.chol_flag, need_full, b.Q, k, SolvePlanes{});
  RET(cudaGetLastError());
  RET(tc_partials(plane_op(b.pa, rows, k, ldk, b.psa), plane_op(b.pb, k, k, ldk, b.psb), rows, k, k,
                  &sp, b, st));
  // the basis: FP64 factor (U, or V transposed) and planes of its transpose
  // (after a non-finite Gram, Y itself: the check then
  // hands the update to the exact split, which reports them)
  note_launch();
  basis_kernel<<<bgrid, 256, 0, st>>>(BasisSrc{b.part, sp, b.Y, b.chol_flag, b.Q, need_full}, rows, k,
                                      nullptr, 0.0, 0ull, b.seed_base, nullptr,
                                      dir_right ? left : nullptr, dir_right ? nullptr : right, hat,
                                      ldr, b.ce_ps);
  RET(cudaGetLastError());
  // centre and Gram in one product: [U^T C_E | U^T U], or [C_E V ; V^T V]
  CentreOut o;
  o.k = k;
  o.dscal = b.dscal;
  o.live = b.live;
  o.ce_ss = b.ce_ss;
  o.thresh = thresh;
  o.disc_max = disc_max;
  const TcOperand X = plane_op(cet, other + k, rows, ldr, b.ce_ps);
  const int R = dir_right ? k : other + k, Cc = dir_right ? other + k : k;
  RET(dir_right ? tc_partials(H, X, R, Cc, rows, &sp, b, st)
                : tc_partials(X, H, R, Cc, rows, &sp, b, st));
  o.out = dir_right ? right : left;
  o.ldo = dir_right ? n : k;
  o.r_gram = dir_right ? R : other;
  o.c_gram = dir_right ? other : Cc;
  note_launch();
  centre_kernel<<<dim3((unsigned)((Cc + 31) / 32), (unsigned)((R + 31) / 32)), 256, 0, st>>>(
      b.part, sp, R, Cc, o);
  return cudaGetLastError();
}

}  // namespace

size_t subspace_plane_elems_a(int cap) { return 3 * (size_t)(4 * cap) * tc_ld(4 * cap); }
size_t subspace_plane_elems_b(int cap) { return 3 * (size_t)(4 * cap) * tc_ld(4 * cap); }
// C_E's planes with room for the basis' transpose behind them
size_t subspace_plane_elems_ce(int cap) { return 3 * (size_t)(5 * cap) * tc_ld(4 * cap); }

namespace {
// max over live columns of |Q^T Q - I| (dead columns, norm < 1/2, are skipped)
// into b.dscal[2] (as FP64).  Q^T Q by the tensor cores, 6 products.
__global__ void orth_defect_kernel(const float* __restrict__ G, int k, double* out) {
  __shared__ float red[32];
  float mx = 0.f;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < k * k; e += gridDim.x * blockDim.x) {
    const int i = e / k, j = e % k;
    const float gi = G[(long long)i * k + i], gj = G[(long long)j * k + j];
    if (gi < 0.5f || gj < 0.5f) continue;
    const float d = fabsf(G[e] - (i == j ? 1.f : 0.f));
    mx = fmaxf(mx, d != d ? 1e30f : d);
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < (int)(blockDim.x / 32); ++i) t = fmaxf(t, red[i]);
    // non-negative doubles order like their bit patterns (*out starts at +0)
    atomicMax(reinterpret_cast<unsigned long long*>(out),
              (unsigned long long)__double_as_longlong((double)t));
  }
}

cudaError_t orth_check(const float* Q, int rows, int k, const SubspaceBuffers& b, cudaStream_t st) {
  RET(tc_product(f32_view(Q, idx_plain(1), idx_plain(k)), f32_view(Q, idx_plain(1), idx_plain(k)),
                 k, k, rows, b.out, k, b, st));
  note_launch();
  const int g = (k * k + 4095) / 4096;
  orth_defect_kernel<<<g < 152 ? g : 152, 1024, 0, st>>>(b.out, k, b.dscal + 2);
  return cudaGetLastError();
}

}  // namespace

size_t subspace_buffer_floats(int cap) {
  const size_t m = 4 * (size_t)cap;
  return m * cap /*Q*/ + m * cap /*Y*/ + m * m /*out*/;
}

namespace {
// discarded weight 1 - ||centre||^2 / ||C_E||^2 of an accepted split
// (orthonormality defect <= thresh) raised into *disc_max
__global__ void split_finish_kernel(const double* __restrict__ ce_ss, const double* __restrict__ dscal,
                                    double thresh, double* disc_max) {
  const double tot = *ce_ss, defect = dscal[2];
  const double disc = tot > 0.0 ? fmax(0.0, 1.0 - dscal[1] / tot) : 0.0;
  if (defect <= thresh)
    atomicMax(reinterpret_cast<unsigned long long*>(disc_max),
              (unsigned long long)__double_as_longlong(disc));
}

// After the orthonormality check (G = Q^T Q): the defect is set to +inf if no
// column of Q is live, or if an orthonormalisation met a non-finite Gram, so
// that the exact split runs.
__global__ void split_guard_kernel(const float* __restrict__ G, int k, const int* __restrict__ flag,
                                   double* defect) {
  __shared__ int live;
  if (threadIdx.x == 0) live = 0;
  __syncthreads();
  for (int j = threadIdx.x; j < k; j += blockDim.x)
    if (G[(long long)j * k + j] >= 0.5f) live = 1;
  __syncthreads();
  if (threadIdx.x == 0 && (!live || *flag)) *defect = INFINITY;
}

cudaError_t split_guard(int k, const SubspaceBuffers& b, cudaStream_t st) {
  note_launch();
  split_guard_kernel<<<1, 256, 0, st>>>(b.out, k, b.chol_flag, b.dscal + 2);
  return cudaGetLastError();
}
}  // namespace

const double* subspace_defect(const SubspaceBuffers& b) { return b.dscal + 2; }

namespace {
__global__ void bump_kernel(unsigned long long* p) { *p += 1; }
}  // namespace

cudaError_t subspace_next_seed(const SubspaceBuffers& b, cudaStream_t st) {
  note_launch();
  bump_kernel<<<1, 1, 0, st>>>(b.seed_base);
  return cudaGetLastError();
}

cudaError_t subspace_split(const double* CE, int m, int n, int k, int dir_right,
                           const double* warm, int kold, double* left, double* right,
                           unsigned long long seed, const SubspaceBuffers& b, cudaStream_t st,
                           double* disc_max, double thresh) {
  (void)CE;
  if (k > SUBSPACE_MAX_K || k > m || k > n) return cudaErrorInvalidValue;
  if (k <= b.orth_block)
    return narrow_split(m, n, k, dir_right, warm, kold, left, right, seed, b, st, disc_max, thresh);
  const double inv_mn = 1.0 / ((double)m * n);
  const long long ldn = tc_ld(n), ldm = tc_ld(m);
  const View ce = planes_view(b.ce_rm, ldn, b.ce_ps);    // C_E   (m rows, K = n)
  const View cet = planes_view(b.ce_tr, ldm, b.ce_ps);   // C_E^T (n rows, K = m)
  RET(cudaMemsetAsync(b.zero, 0, b.zero_words * sizeof(int), st));
  RET(cudaMemsetAsync(b.chol_flag, 0, sizeof(int), st));
  if (dir_right) {
    // warm start: rows of the current C_{i+1} (kold x n) -> Q (n x k)
    note_launch();
    warm_start_kernel<<<grid_for((long long)n * k), 256, 0, st>>>(warm, n, 1, kold, n, k, seed,
                                                                  b.seed_base, b.Q);
    // Y = C_E Q (m x k): A = C_E (m rows, K = n), B = Q^T (k rows, K = n)
    RET(tc_product(ce, f32_view(b.Q, idx_plain(1), idx_plain(k)), m, k, n, b.Y, k, b, st));
    note_launch();
    add_noise_kernel<<<grid_for((long long)m * k), 256, 0, st>>>(b.Y, (long long)m * k, b.ce_ss,
                                                                 inv_mn, seed + 7, b.seed_base);
    RET(cudaGetLastError());
    float* U = b.Y;
    RET(orthonormalise_blocks(U, m, k, b, st));
    RET(orth_check(U, m, k, b, st));
    RET(split_guard(k, b, st));
    // C_i = U (m x k); C_{i+1} = U^T C_E (k x n)
    note_launch();
    copy_f2d_kernel<<<grid_for((long long)m * k), 256, 0, st>>>(U, (long long)m * k, left);
    // U^T C_E (k x n): A = U^T (k rows, K = m), B = C_E^T (n rows, K = m)
    RET(tc_product(f32_view(U, idx_plain(1), idx_plain(k)), cet, k, n, m, b.out, n, b, st));
    note_launch();
    copy_f2d_kernel<<<grid_for((long long)k * n), 256, 0, st>>>(b.out, (long long)k * n, right);
    RET(cudaGetLastError());
  } else {
    // warm start: columns of the current C_i (m x kold) -> Q (m x k)
    note_launch();
    warm_start_kernel<<<grid_for((long long)m * k), 256, 0, st>>>(warm, 1, kold, kold, m, k, seed,
                                                                  b.seed_base, b.Q);
    // Z = C_E^T Q (n x k): A = C_E^T (n rows, K = m), B = Q^T (k rows, K = m)
    RET(tc_product(cet, f32_view(b.Q, idx_plain(1), idx_plain(k)), n, k, m, b.Y, k, b, st));
    note_launch();
    add_noise_kernel<<<grid_for((long long)n * k), 256, 0, st>>>(b.Y, (long long)n * k, b.ce_ss,
                                                                 inv_mn, seed + 7, b.seed_base);
    RET(cudaGetLastError());
    float* V = b.Y;
    RET(orthonormalise_blocks(V, n, k, b, st));
    RET(orth_check(V, n, k, b, st));
    RET(split_guard(k, b, st));
    // C_{i+1} = V^T (k x n); C_i = C_E V (m x k)
    note_launch();
    transpose_f2d_kernel<<<grid_for((long long)n * k), 256, 0, st>>>(V, n, k, right);
    // C_E V (m x k): A = C_E (m rows, K = n), B = V^T (k rows, K = n)
    RET(tc_product(ce, f32_view(V, idx_plain(1), idx_plain(k)), m, k, n, b.out, k, b, st));
    note_launch();
    copy_f2d_kernel<<<grid_for((long long)m * k), 256, 0, st>>>(b.out, (long long)m * k, left);
    RET(cudaGetLastError());
  }
  // ||centre||^2 for the discarded weight 1 - ||centre||^2 / ||C_E||^2
  double* centre = dir_right ? right : left;
  const long long nc = dir_right ? (long long)k * n : (long long)m * k;
  note_launch();
  sumsq_f64_kernel<<<grid_for(nc) < 304 ? grid_for(nc) : 304, 256, 0, st>>>(centre, nc,
                                                                            b.dscal + 1);
  RET(cudaGetLastError());
  if (disc_max) {
    note_launch();
    split_finish_kernel<<<1, 1, 0, st>>>(b.ce_ss, b.dscal, thresh, disc_max);
    RET(cudaGetLastError());
  }
  return cudaMemsetAsync(b.ce_ss, 0, sizeof(double), st);
}

const __nv_bfloat16* subspace_basis_planes(const SubspaceBuffers& b, int m, int n, int k,
                                           int dir_right, long long* ld, long long* ps) {
  if (k > b.orth_block || k > SUBSPACE_MAX_K) return nullptr;
  *ld = tc_ld(dir_right ? m : n);
  *ps = b.ce_ps;
  return dir_right ? b.ce_tr + (long long)n * *ld : b.ce_rm + (long long)m * *ld;
}
