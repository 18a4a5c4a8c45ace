// FP64 singular value split of Fig. VMPO(d): pivoted QR, then one-sided
// (Hestenes) Jacobi on the transposed triangular factor.
//
// The generalised overlap C_E (Eq. LSEProd) is factorised C_E = U Lambda V^T
// and truncated by *number*: the largest min(D*, numerical rank) singular
// values are kept (Sec. II D: truncation by discarded weight is avoided; only
// singular values at or below rel_tol * sigma_max, i.e. numerically zero, are
// dropped).  Left-to-right the left factor is U and the right factor
// Lambda V^T; right-to-left Lambda goes with U (App. D.1).
//
// Let A (q x p) be the matrix with the side of the wanted isometry as its
// columns: A = M^T for U, A = M for V.
//  1. Pivoted QR, A P = Q R, by modified Gram-Schmidt on the columns of A;
//     only R^T (p x r) is formed, Q is never needed.  It ends early at rank r
//     when what is left has a Frobenius norm below a tenth of rel_tol *
//     sigma_max (those singular values are numerically zero), or, when kcap
//     cuts the spectrum, as soon as what is left, E, no longer counts.  E is
//     orthogonal to Q, so A^T A = R^T R + E^T E: leaving it out loses at most
//     |E|^2 of captured weight, and turns the kept subspace by |E|^2 over the
//     gap of the squares at the cut, where rounding turns it by eps sigma_max
//     over the gap.  Hence |E|^2 <= 1e-12 of the weight left after kcap columns
//     and <= eps sigma_max sigma_k (the latter is the tighter one on flat
//     spectra: with the first alone, values 1e-5 apart at the cut and one of
//     9e-7 behind it gave factors off by 4e-9, now 3e-11; thermal states meet
//     both a column or two apart).
//  2. One-sided Jacobi orthogonalises the r columns of R^T: R^T J = X Sigma
//     with X the wanted singular vectors.  The triangular factor of a pivoted
//     QR is close to having orthogonal rows, and the rotations resolve small
//     singular values to high relative accuracy (which the series
//     initialisation needs: its higher-order terms sit 1e-10 .. 1e-15 below
//     the leading one).  Jacobi on C_E itself takes 12 to 40 sweeps over
//     min(m, n) columns; on R^T it takes 4 to 6 over r of them.
//  3. The kept columns X_k = (R^T J)_k / sigma_k are one factor, the other one
//     is M projected on them: U^T M or M V.  The Jacobi sweeps leave the columns
//     orthogonal to about 1e-15 only, which in the plain projection puts 1e-15
//     sigma_1 into the row of every small sigma_j and takes away the relative
//     accuracy of step 2.  So the projection T is followed by T - L T, L the
//     strictly lower part of the Gram X^T X (columns in falling order of sigma):
//     what is left of the larger ones' rows goes out of each row, the pseudo-
//     inverse of X to first order.  Energy of the series initialisation at L = 8,
//     tau0 = 2^-26, against exact: 4e-8 without, 7e-16 with (the Hamiltonian is
//     1e-8 of that state); it costs 1 % of a doubling at L = 32, D* = 40.
//
// GPU mapping: one kernel per split, half a warp per column (step 1) or a warp
// per column pair of a round-robin round (step 2); columns live in L2 (read past
// L1).  Steps and rounds are separated by a barrier over all CTAs.  What
// bounds it is latency: a step moves a few columns, does a hundred FP64
// operations per lane pair and meets the barrier.  Small problems run in one
// thread-block cluster of up to 16 CTAs, whose hardware barrier takes a
// fraction of a microsecond; larger ones, which need more than 16 SMs' worth
// of FP64 (two FMAs a clock each), run as a cooperative grid with a bounded
// barrier (on expiry the kernel records a timeout and every CTA leaves).
// Measured, one FP64 doubling at L = 32, D* = 40, one sweep (62 splits of up
// to 160 x 160): 1095 ms with Jacobi on C_E, 116 ms with this split (an average
// split of its bulk takes 0.66 ms: 90 QR steps and some 400 rounds).
#include <math.h>

#include "common.cuh"

namespace {

constexpr int WPB = 8;                  // warps per CTA
constexpr int NT = WPB * 32;
constexpr int CL_MAX = 16;              // CTAs of the largest cluster (opt-in size)
constexpr long long SPIN_LIMIT = 1LL << 22;
constexpr int REGS = 8;                 // columns up to 32 * REGS rows stay in registers

struct SvdArgs {
  const double* M;
  int m, n, kcap, mode, max_sweeps;
  int p, q, rmax;        // isometry side, other side, min(p, q)
  long long sc, si;      // A[i][c] = M[c * sc + i * si], i < q, c < p
  double tol2, rel_tol;
  double *A, *W, *nrm;   // A: p columns of length q; W: rmax columns of length p; nrm: 2 x max_cols
  int max_cols;
  double* sig;
  int* perm;
  double *left, *right;
  unsigned* bar;      // [0] arrivals, [1] generation
  int* cnt;           // [0..2] rotations per sweep (ring), [3..5] unconverged pairs per check (ring)
  int* out;           // [0] k, [1] rank, [2] sweeps, [3] status (0 ok, 1 timeout, 2 not converged)
  double* stats;      // [0] total weight, [1] discarded fraction, [2] sigma_max,
                      // [3] ||M||_F^2 (accumulated while loading), [4] columns of the QR
  // device-decided mode (all null otherwise): run only if *run_if > thresh
  // or is not finite; keep exactly min(kcap, p, q); report into acc
  const double* run_if;
  double thresh;
  SvdDeviceAcc acc;
};

// Grid barrier with a bounded wait.  Returns false if the wait expired or
// another CTA already recorded a timeout (then every CTA returns).
__device__ bool grid_barrier(const SvdArgs& a) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* vb = a.bar;
    volatile int* st = a.out + 3;
    if (*st == 1) {
      ok = 0;
    } else {
      unsigned gen = vb[1];
      __threadfence();
      unsigned arrived = atomicAdd(a.bar, 1u);
      if (arrived == gridDim.x - 1) {
        vb[0] = 0;
        __threadfence();
        atomicAdd(a.bar + 1, 1u);
      } else {
        long long it = 0;
        while (vb[1] == gen) {
          if (++it > SPIN_LIMIT || *st == 1) {
            atomicExch(a.out + 3, 1);
            if (a.acc.status) atomicMax(a.acc.status, 1);
            ok = 0;
            break;
          }
          if (it > 64) __nanosleep(32);
        }
      }
      __threadfence();
    }
  }
  __syncthreads();
  return ok != 0;
}

// Barrier over all CTAs of the launch (one cluster, or the whole grid).
template <bool CLUSTER>
__device__ __forceinline__ bool all_sync(const SvdArgs& a) {
  if (!CLUSTER) return grid_barrier(a);
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
  return true;
}

__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// FP32 value of x 2^(1023 - e0), e0 a biased exponent, by integer operations
__device__ __forceinline__ float scaled_float(double x, int e0) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ff) - e0 + 127;
  const unsigned m = ((h & 0xfffffu) << 3) | (l >> 29);
  const unsigned v = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : ((unsigned)e << 23) | m);
  return __uint_as_float((h & 0x80000000u) | v);
}
// a normal FP32 value as FP64
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u >> 3) & 0x0fffffffu) + 0x38000000u)),
                          (int)(u << 29));
}

// Whether ga^2 > tol2 al be (al, be squared norms, ga their Gram entry):
// mantissas in FP32, exponents apart.
__device__ __forceinline__ bool above_tol(double al, double be, double ga, float tol2) {
  const int eg = biased_exp(ga), ea = biased_exp(al), eb = biased_exp(be);
  if (eg == 0 || ea == 0 || eb == 0) return false;
  const float g = scaled_float(ga, eg);
  const int de = 2 * eg - ea - eb;   // cos^2 = g^2 / (mantissas of al, be) 2^de
  return de > -140 && g * g * exp2f((float)(de < 100 ? de : 100)) >
                          tol2 * scaled_float(al, ea) * scaled_float(be, eb);
}

// The rotation that zeroes the Gram entry ga, as three shears
//   x -= tau y,  y += s x,  x -= tau y,   tau = tan(theta / 2), s = 2 tau / (1 + tau^2):
// three FMAs an element where the plain form takes four operations, and no
// square root.  A warp gets one FP64 instruction through in 64 clocks whatever
// it is (measured; an ALU instruction takes 5), so the angle, t = tan(theta) =
// sign(z) / (|z| + sqrt(1 + z^2)), z = (be - al) / (2 ga), comes from FP32 (its
// error of 1e-7 leaves 1e-7 ga behind, which a later visit removes), the
// conversions are integer operations, and s follows from tau to FP64 accuracy
// by one third-order step.  false: the angle is below FP32's range.
__device__ __forceinline__ bool rotation(double al, double be, double ga, double& t, double& tau,
                                         double& s) {
  const int eg = biased_exp(ga);
  const float z = 0.5f * scaled_float(be - al, eg) / scaled_float(ga, eg);
  const float t32 = fabsf(z) > 1e9f
                        ? 0.5f / z
                        : copysignf(1.f / (fabsf(z) + sqrtf(fmaf(z, z, 1.f))), z);
  if (!(fabsf(t32) > 1e-37f)) return false;
  const float cf = rsqrtf(fmaf(t32, t32, 1.f)), tf = t32 * cf / (1.f + cf);
  t = widen(t32);
  tau = widen(tf);
  const double w = fma(tau, tau, 1.0), y0 = widen(1.f / fmaf(tf, tf, 1.f)), e = fma(-w, y0, 1.0);
  s = widen(2.f * tf) * fma(y0, fma(e, e, e), y0);
  return true;
}

// One pair of W's columns: rotated if its Gram entry is above tol * norms.
__device__ __forceinline__ int rotate_pair(const SvdArgs& a, int jp, int jq, double gfloor,
                                           int lane) {
  const int p = a.p;
  double* wp = a.W + (long long)jp * p;
  double* wq = a.W + (long long)jq * p;
  const double al = __ldcg(a.nrm + jp), be = __ldcg(a.nrm + jq);
  double t, tau, s;
  if (p <= 32 * REGS) {
    double x[REGS], y[REGS], ga = 0.0;
#pragma unroll
    for (int u = 0; u < REGS; ++u) {
      const int e = lane + 32 * u;
      x[u] = e < p ? __ldcg(wp + e) : 0.0;
      y[u] = e < p ? __ldcg(wq + e) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < REGS; ++u)
      if (32 * u < p) ga = fma(x[u], y[u], ga);
    ga = warp_sum(ga);
    if (!above_tol(al, be, ga, (float)a.tol2) || (gfloor > 0.0 && !(fabs(ga) > gfloor))) return 0;
    if (!rotation(al, be, ga, t, tau, s)) return 0;
#pragma unroll
    for (int u = 0; u < REGS; ++u) {
      const int e = lane + 32 * u;
      if (32 * u < p) {
        x[u] = fma(-tau, y[u], x[u]);
        y[u] = fma(s, x[u], y[u]);
        x[u] = fma(-tau, y[u], x[u]);
        if (e < p) {
          __stcg(wp + e, x[u]);
          __stcg(wq + e, y[u]);
        }
      }
    }
    if (lane == 0) {
      const double na = fma(-t, ga, al), nb = fma(t, ga, be);
      __stcg(a.nrm + jp, na > 0.0 ? na : 0.0);
      __stcg(a.nrm + jq, nb > 0.0 ? nb : 0.0);
    }
  } else {
    double ga0 = 0.0;
#pragma unroll 4
    for (int e = lane; e < p; e += 32) ga0 = fma(__ldcg(wp + e), __ldcg(wq + e), ga0);
    const double ga = warp_sum(ga0);
    if (!above_tol(al, be, ga, (float)a.tol2) || (gfloor > 0.0 && !(fabs(ga) > gfloor))) return 0;
    if (!rotation(al, be, ga, t, tau, s)) return 0;
#pragma unroll 4
    for (int e = lane; e < p; e += 32) {
      const double y = __ldcg(wq + e), x = fma(-tau, y, __ldcg(wp + e)), yn = fma(s, x, y);
      __stcg(wq + e, yn);
      __stcg(wp + e, fma(-tau, yn, x));
    }
    if (lane == 0) {
      const double na = fma(-t, ga, al), nb = fma(t, ga, be);
      __stcg(a.nrm + jp, na > 0.0 ? na : 0.0);
      __stcg(a.nrm + jq, nb > 0.0 ? nb : 0.0);
    }
  }
  return 1;
}

// C[i][j] = sum_t P(i, t) Q(t, j) over all CTAs, 16 x 16 tiles.
__device__ void project(const double* P, long long pi, long long pt, const double* Q, long long qt,
                        long long qj, double* C, long long ci, long long cj, int ni, int nj,
                        int nt) {
  __shared__ double Ps[16][17], Qs[16][17];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int tj = (nj + 15) / 16, tiles = (ni + 15) / 16 * tj;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int i0 = tile / tj * 16, j0 = tile % tj * 16;
    double acc = 0.0;
    for (int t0 = 0; t0 < nt; t0 += 16) {
      // consecutive threads take the index that is contiguous in memory
      const int a_i = pt == 1 ? ty : tx, a_t = pt == 1 ? tx : ty;
      const int b_j = qj == 1 ? tx : ty, b_t = qj == 1 ? ty : tx;
      Ps[a_t][a_i] = (i0 + a_i < ni && t0 + a_t < nt) ? __ldcg(P + (i0 + a_i) * pi + (t0 + a_t) * pt) : 0.0;
      Qs[b_t][b_j] = (j0 + b_j < nj && t0 + b_t < nt) ? __ldcg(Q + (t0 + b_t) * qt + (j0 + b_j) * qj) : 0.0;
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 16; ++t) acc = fma(Ps[t][ty], Qs[t][tx], acc);
      __syncthreads();
    }
    if (i0 + ty < ni && j0 + tx < nj) C[(i0 + ty) * ci + (j0 + tx) * cj] = acc;
  }
}

// C(i, j) = T(i, j) - sum_{t < i} E[i][t] T(t, j) over all CTAs, 16 x 16 tiles;
// E has rows of k, T and C are k x nj.
__device__ void take_out_lower(const double* E, int k, const double* T, long long ti, long long tj,
                               double* C, long long ci, long long cj, int nj) {
  __shared__ double Es[16][17], Ts[16][17];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int tw = (nj + 15) / 16, tiles = (k + 15) / 16 * tw;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int i0 = tile / tw * 16, j0 = tile % tw * 16;
    const int i = i0 + ty, j = j0 + tx;
    double acc = 0.0;
    for (int t0 = 0; t0 <= i0; t0 += 16) {
      const int b_j = tj == 1 ? tx : ty, b_t = tj == 1 ? ty : tx;
      Es[tx][ty] = (i < k && t0 + tx < i) ? __ldcg(E + (long long)i * k + t0 + tx) : 0.0;
      Ts[b_t][b_j] = (j0 + b_j < nj && t0 + b_t < k) ? __ldcg(T + (t0 + b_t) * ti + (j0 + b_j) * tj) : 0.0;
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 16; ++t) acc = fma(Es[t][ty], Ts[t][tx], acc);
      __syncthreads();
    }
    if (i < k && j < nj) C[i * ci + j * cj] = __ldcg(T + i * ti + j * tj) - acc;
  }
}

constexpr int LGQ = 16;    // lanes of a column in the QR step
constexpr int REGQ = 16;   // columns up to LGQ * REGQ rows stay in registers there

__device__ __forceinline__ double group_sum(double v) {   // over LGQ lanes
#pragma unroll
  for (int o = LGQ / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <bool CLUSTER>
__global__ void __launch_bounds__(NT) svd_split_kernel(SvdArgs a) {
  // device-decided mode: every CTA leaves before the first barrier
  if (a.run_if && *a.run_if <= a.thresh) return;
  const int lane = threadIdx.x & 31;
  // consecutive work items go to different SMs
  const int gw = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int TW = gridDim.x * WPB;
  const long long gt = blockIdx.x * (long long)NT + threadIdx.x;
  const long long GT = (long long)gridDim.x * NT;
  const int p = a.p, q = a.q;

  // load A's columns and their squared norms
  double ss = 0.0;
  for (int c = gw; c < p; c += TW) {
    double* col = a.A + (long long)c * q;
    double s2 = 0.0;
#pragma unroll 4
    for (int i = lane; i < q; i += 32) {
      const double x = a.M[c * a.sc + i * a.si];
      __stcg(col + i, x);
      s2 = fma(x, x, s2);
    }
    s2 = warp_sum(s2);
    if (lane == 0) __stcg(a.nrm + c, s2);
    ss += s2;
  }
  if (lane == 0 && ss != 0.0) atomicAdd(a.stats + 3, ss);
  if (!all_sync<CLUSTER>(a)) return;
  const double fro = __ldcg(a.stats + 3);
  if (!(fro <= 1.7976931348623157e308)) {   // a non-finite entry: reported, nothing emitted
    if (gt == 0) {
      a.out[0] = 1;
      a.out[1] = 0;
      a.out[2] = 0;
      a.stats[0] = a.stats[2] = fro;
      a.stats[1] = a.stats[4] = 0.0;
      if (a.run_if && a.acc.runs) atomicAdd(a.acc.runs, 1ull);
      if (a.run_if && a.acc.status) atomicMax(a.acc.status, 3);
    }
    return;
  }

  // ---- 1. pivoted QR (modified Gram-Schmidt), rows of R into W's columns;
  // half a warp per column: an SM gets an FP64 instruction through in 19
  // clocks and a warp in 64, so the sums over lanes and the scalars count
  int r = 0;
  double scale = 1.0, rem = 0.0;
  float mx0 = 0.f, remcut = -1.f, remf = 0.f;   // weights relative to 2^(e0 - 1023) in FP32
  const int e0 = biased_exp(fro);
  const float nstop = (float)(0.01 * a.rel_tol * a.rel_tol);
  const int grp = lane / LGQ, gl = lane % LGQ;
  for (int j = 0; j < a.rmax; ++j) {
    const double* nr = a.nrm + (j & 1) * (long long)a.max_cols;
    double* nw = a.nrm + ((j + 1) & 1) * (long long)a.max_cols;
    // pivot: the column with the largest norm left, ties to the lowest column
    // (finished ones hold -1; positive doubles order like their bits); every
    // warp scans the same values, so all take the same branches
    long long best = -1;
    int piv = 0x7fffffff;
    remf = 0.f;
#pragma unroll 4
    for (int c = lane; c < p; c += 32) {
      const double v = __ldcg(nr + c);
      const long long bits = __double_as_longlong(v);
      if (bits > 0) remf += scaled_float(v, e0);
      if (bits > best) {
        best = bits;
        piv = c;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long v = __shfl_xor_sync(0xffffffffu, best, o);
      const int c = __shfl_xor_sync(0xffffffffu, piv, o);
      remf += __shfl_xor_sync(0xffffffffu, remf, o);
      if (v > best || (v == best && c < piv)) {
        best = v;
        piv = c;
      }
    }
    const double bn = __longlong_as_double(best);
    if (j == 0 && best > 0) {
      mx0 = scaled_float(bn, e0);
      // W is scaled by a power of two to norms of at most about 1
      scale = ldexp(1.0, -(ilogb(bn) / 2));
    }
    if (best <= 0 || remf <= nstop * mx0) break;
    // sigma_max and sigma_k as the first pivot and the one after kcap columns show them
    if (j == a.kcap) remcut = fminf(1e-12f * remf, 2.2e-16f * sqrtf(mx0 * scaled_float(bn, e0)));
    if (j > a.kcap && remf <= remcut) break;
    // 1 / |pivot|: FP32 for the mantissa (in [1, 4), even exponent), then one
    // third-order step
    const int eb = biased_exp(bn), h = (eb - 1023) >> 1;   // bn = m 4^h
    double rinv;
    if (eb > 0) {
      const double m = __hiloint2double(__double2hiint(bn) - (h << 21), __double2loint(bn));
      const double y0 = widen(rsqrtf(scaled_float(m, 1023)));
      const double e = fma(-m * y0, y0, 1.0);
      const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);
      rinv = __hiloint2double(__double2hiint(y) - (h << 20), __double2loint(y));
    } else {
      rinv = rsqrt(bn);   // subnormal
    }
    const double ws = rinv * scale, binv = rinv * rinv;
    const double* xp = a.A + (long long)piv * q;
    double* wrow = a.W + (long long)j * p;
    double x[REGQ];
    if (q <= LGQ * REGQ) {
#pragma unroll
      for (int u = 0; u < REGQ; ++u) x[u] = gl + LGQ * u < q ? __ldcg(xp + gl + LGQ * u) : 0.0;
    }
    for (int c0 = gw * (32 / LGQ); c0 < p; c0 += TW * (32 / LGQ)) {
      const int c = c0 + grp;
      const bool in = c < p;
      const long long nc = in ? __double_as_longlong(__ldcg(nr + c)) : -1;
      const bool work = nc >= 0 && c != piv;
      double* xc = a.A + (long long)(in ? c : 0) * q;
      double dot = 0.0, s2 = 0.0;
      if (q <= LGQ * REGQ) {
        double y[REGQ];
#pragma unroll
        for (int u = 0; u < REGQ; ++u)
          y[u] = (work && gl + LGQ * u < q) ? __ldcg(xc + gl + LGQ * u) : 0.0;
#pragma unroll
        for (int u = 0; u < REGQ; ++u)
          if (LGQ * u < q) dot = fma(x[u], y[u], dot);
        dot = group_sum(dot);
        const double f = dot * binv;
#pragma unroll
        for (int u = 0; u < REGQ; ++u)
          if (LGQ * u < q) {
            y[u] = fma(-f, x[u], y[u]);
            s2 = fma(y[u], y[u], s2);
            if (work && gl + LGQ * u < q) __stcg(xc + gl + LGQ * u, y[u]);
          }
      } else {
        if (work)
          for (int e = gl; e < q; e += LGQ) dot = fma(__ldcg(xp + e), __ldcg(xc + e), dot);
        dot = group_sum(dot);
        const double f = dot * binv;
        if (work)
          for (int e = gl; e < q; e += LGQ) {
            const double y = fma(-f, __ldcg(xp + e), __ldcg(xc + e));
            s2 = fma(y, y, s2);
            __stcg(xc + e, y);
          }
      }
      s2 = group_sum(s2);
      if (in && gl == 0) {
        __stcg(wrow + c, c == piv ? bn * ws : (work ? dot * ws : 0.0));
        __stcg(nw + c, work ? s2 : -1.0);
      }
    }
    r = j + 1;
    remf = 0.f;   // what is left is known at the next step's scan only
    if (!all_sync<CLUSTER>(a)) return;
  }
  // (a finite fro has e0 below 2047, so the factor is finite)
  rem = (double)remf * __longlong_as_double((long long)(e0 > 0 ? e0 : 1) << 52);
  // the norms become those of W's columns: every warp has read them
  if (!all_sync<CLUSTER>(a)) return;

  // ---- 2. one-sided Jacobi on W (p x r)
  const int nn = r + (r & 1), mod = nn - 1, npairs = nn / 2;
  int sweeps = 0;
  bool converged = r < 2;
  for (int s = 0; s < a.max_sweeps; ++s) {
    // squared column norms afresh: the rotations update them with rounding
    for (int j = gw; j < r; j += TW) {
      const double* w = a.W + (long long)j * p;
      double s2 = 0.0;
#pragma unroll 4
      for (int e = lane; e < p; e += 32) {
        const double x = __ldcg(w + e);
        s2 = fma(x, x, s2);
      }
      s2 = warp_sum(s2);
      if (lane == 0) __stcg(a.nrm + j, s2);
    }
    if (gt == 0) {
      a.cnt[(s + 1) % 3] = 0;
      a.cnt[3 + (s + 1) % 3] = 0;
    }
    if (!all_sync<CLUSTER>(a)) return;
    if (converged) break;
    // Pairs of columns below the resolution of the whole problem could rotate
    // without end: past 30 sweeps (never met) Gram entries beneath eps^2
    // ||W||^2 are left alone
    const double gfloor = s < 30 ? 0.0 : 4.930380657631324e-32 * fro * scale * scale;
    // after a sweep that rotated fewer than one pair in 16, all cosines at once
    // (24 us at r = 90 against 120 for a sweep): a converged state needs no
    // more rounds, and one with more rotations behind it never was converged
    const bool settled = s > 0 && __ldcg(a.cnt + (s - 1) % 3) * 16LL < (long long)r * (r - 1) / 2;
    if (settled) {
      int off = 0;
      const int np = r * (r - 1) / 2;
      for (int e = gw; e < np; e += TW) {
        int i = (int)((1.f + sqrtf(1.f + 8.f * (float)e)) * 0.5f);
        while (i * (i - 1) / 2 > e) --i;
        while ((i + 1) * i / 2 <= e) ++i;
        const int jj = e - i * (i - 1) / 2;
        const double* wi = a.W + (long long)i * p;
        const double* wj = a.W + (long long)jj * p;
        double ga = 0.0;
#pragma unroll 4
        for (int x = lane; x < p; x += 32) ga = fma(__ldcg(wi + x), __ldcg(wj + x), ga);
        ga = warp_sum(ga);
        off += above_tol(__ldcg(a.nrm + i), __ldcg(a.nrm + jj), ga, (float)a.tol2) &&
               (!(gfloor > 0.0) || fabs(ga) > gfloor);
      }
      if (lane == 0 && off) atomicAdd(a.cnt + 3 + s % 3, off);
      if (!all_sync<CLUSTER>(a)) return;
      if (__ldcg(a.cnt + 3 + s % 3) == 0) {
        converged = true;
        break;
      }
    }
    int myrot = 0;
    for (int rd = 0; rd < mod; ++rd) {
      for (int i = gw; i < npairs; i += TW) {
        int jp, jq;
        if (i == 0) { jp = rd; jq = nn - 1; }
        else { jp = (rd + i) % mod; jq = (rd - i + mod) % mod; }
        if (jp > jq) { int t = jp; jp = jq; jq = t; }
        if (jq >= r) continue;
        myrot += rotate_pair(a, jp, jq, gfloor, lane);
      }
      if (rd == mod - 1 && lane == 0 && myrot) atomicAdd(a.cnt + s % 3, myrot);
      if (!all_sync<CLUSTER>(a)) return;
    }
    sweeps = s + 1;
    converged = __ldcg(a.cnt + s % 3) == 0;
  }

  // ---- 3. singular values, their order, the kept number
  for (int j = (int)gt; j < a.rmax; j += (int)GT) {
    const double s2 = j < r ? __ldcg(a.nrm + j) : 0.0;
    int rk = 0;
    if (j < r) {
      // non-negative doubles order like their bits
      const long long b2 = __double_as_longlong(s2);
#pragma unroll 8
      for (int i = 0; i < r; ++i) {
        const long long x = __double_as_longlong(__ldcg(a.nrm + i));
        rk += x > b2 || (x == b2 && i < j);
      }
    } else {
      rk = j;
    }
    a.perm[rk] = j;
    a.sig[j] = sqrt(s2) / scale;   // exact division: scale is a power of two
  }
  if (!all_sync<CLUSTER>(a)) return;
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    double mx = 0.0;
    for (int j = lane; j < r; j += 32) mx = fmax(mx, __ldcg(a.nrm + j));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const double smx = sqrt(mx);
    int cnt = 0;
    const double thr = a.rel_tol * a.rel_tol * mx;
    for (int j = lane; j < r; j += 32) cnt += __ldcg(a.nrm + j) > thr;
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    int k = cnt < a.kcap ? cnt : a.kcap;
    if (a.run_if) k = a.kcap < a.rmax ? a.kcap : a.rmax;
    if (k < 1) k = 1;
    double keptw = 0.0, dropw = 0.0;
    for (int j = lane; j < r; j += 32) {
      const double w = __ldcg(a.nrm + __ldcg(a.perm + j));
      if (j < k) keptw += w;
      else dropw += w;
    }
    keptw = warp_sum(keptw);
    dropw = warp_sum(dropw) + rem * scale * scale;
    if (lane == 0) {
      a.out[0] = k;
      a.out[1] = cnt;
      a.out[2] = sweeps;
      if (!converged) a.out[3] = 2;
      a.stats[0] = (keptw + dropw) / scale / scale;
      a.stats[1] = keptw + dropw > 0.0 ? dropw / (keptw + dropw) : 0.0;
      a.stats[2] = smx / scale;
      a.stats[4] = r;
      if (a.run_if) {
        if (a.acc.disc_max)
          atomicMax(reinterpret_cast<unsigned long long*>(a.acc.disc_max),
                    (unsigned long long)__double_as_longlong(a.stats[1]));
        if (a.acc.runs) atomicAdd(a.acc.runs, 1ull);
        if (a.acc.status && !converged) atomicMax(a.acc.status, 2);
        if (a.acc.status && !isfinite(smx)) atomicMax(a.acc.status, 3);
      }
    }
  }
  if (!all_sync<CLUSTER>(a)) return;

  // ---- 4. the isometry, then M projected on it (columns in falling order of sigma)
  const int k = __ldcg(a.out);
  for (int rr = gw; rr < k; rr += TW) {
    const int j = __ldcg(a.perm + rr);
    const double s2 = j < r ? __ldcg(a.nrm + j) : 0.0;
    const double inv = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
    const double* w = a.W + (long long)j * p;
    for (int x = lane; x < p; x += 32) {
      const double v = s2 > 0.0 ? __ldcg(w + x) * inv : 0.0;
      if (a.mode == SPLIT_RIGHT) __stcg(a.left + (long long)x * k + rr, v);
      else __stcg(a.right + (long long)rr * a.n + x, v);
    }
  }
  if (!all_sync<CLUSTER>(a)) return;
  // the Gram of the isometry takes A's place (k^2 <= p q), the projection W's (of
  // the capacity of M, as k <= m, n); both were read before the barrier
  if (a.mode == SPLIT_RIGHT) {   // Sigma V^T = U^T M
    project(a.left, 1, k, a.left, k, 1, a.A, k, 1, k, k, a.m);
    project(a.left, 1, k, a.M, a.n, 1, a.W, a.n, 1, k, a.n, a.m);
    if (!all_sync<CLUSTER>(a)) return;
    take_out_lower(a.A, k, a.W, a.n, 1, a.right, a.n, 1, a.n);
  } else {                       // U Sigma = M V, as its transpose
    project(a.right, a.n, 1, a.right, 1, a.n, a.A, k, 1, k, k, a.n);
    project(a.M, a.n, 1, a.right, 1, a.n, a.W, k, 1, a.m, k, a.n);
    if (!all_sync<CLUSTER>(a)) return;
    take_out_lower(a.A, k, a.W, 1, k, a.left, 1, k, a.m);
  }
}

cudaLaunchConfig_t cluster_config(int ctas, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// CTAs of the cooperative launch and of the largest cluster (once per device,
// thread-safe; no kernel runs for it)
struct SvdSetup {
  cudaError_t err;
  int max_ctas, max_cluster;
};
PerDevice<SvdSetup> g_svd_setup;

SvdSetup svd_setup() {
  SvdSetup s{cudaSuccess, 0, 0};
  cudaError_t e = g_svd_setup.get(
      [](int dev) {
        SvdSetup r{cudaSuccess, 0, 0};
        int sms = 0, per = 0;
        r.err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (r.err == cudaSuccess)
          r.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, svd_split_kernel<false>, NT, 0);
        r.max_ctas = sms * (per < 1 ? per : 1);
        if (r.err == cudaSuccess && r.max_ctas < 1) r.err = cudaErrorLaunchOutOfResources;
        if (cudaFuncSetAttribute(svd_split_kernel<true>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
          cudaGetLastError();
        for (int c = CL_MAX; c >= 2 && !r.max_cluster; c /= 2) {
          cudaLaunchAttribute attr[1];
          cudaLaunchConfig_t cfg = cluster_config(c, 0, attr);
          int n = 0;
          if (cudaOccupancyMaxActiveClusters(&n, svd_split_kernel<true>, &cfg) == cudaSuccess && n >= 1)
            r.max_cluster = c;
          else
            cudaGetLastError();
        }
        return r;
      },
      &s);
  if (e != cudaSuccess) s.err = e;
  return s;
}

cudaError_t svd_launch(const double* M, int m, int n, int kcap, double rel_tol, SplitMode mode,
                       double* left, double* right, const SvdBuffers& buf, cudaStream_t st,
                       const double* run_if, double thresh, const SvdDeviceAcc& acc,
                       bool cleared = false) {
  const int p = mode == SPLIT_RIGHT ? m : n, q = mode == SPLIT_RIGHT ? n : m;
  const int rmax = p < q ? p : q;
  if (m < 1 || n < 1 || kcap < 1 || (size_t)m * n > buf.max_elems || p > buf.max_cols)
    return cudaErrorInvalidValue;
  cudaError_t e;
  const SvdSetup setup = svd_setup();
  if (setup.err != cudaSuccess) return setup.err;
  SvdArgs a;
  a.M = M; a.m = m; a.n = n; a.p = p; a.q = q; a.rmax = rmax;
  a.sc = mode == SPLIT_RIGHT ? n : 1;
  a.si = mode == SPLIT_RIGHT ? 1 : n;
  a.kcap = kcap; a.mode = (int)mode; a.max_sweeps = 60;
  const double tol = sqrt((double)(p > q ? p : q)) * 2.220446049250313e-16;
  a.tol2 = tol * tol;
  a.rel_tol = rel_tol;
  a.A = buf.V; a.W = buf.W; a.nrm = buf.nrm; a.max_cols = buf.max_cols;
  a.sig = buf.sig; a.perm = buf.perm;
  a.left = left; a.right = right;
  a.bar = (unsigned*)buf.counter;      // 2 words
  a.cnt = buf.counter + 2;             // 6 words
  a.out = buf.kept;                    // 4 words
  a.stats = buf.stats;
  a.run_if = run_if;
  a.thresh = thresh;
  a.acc = acc;
  if (!cleared) {
    if ((e = cudaMemsetAsync(buf.counter, 0, 8 * sizeof(int), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(buf.kept, 0, 4 * sizeof(int), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(buf.stats, 0, 4 * sizeof(double), st)) != cudaSuccess) return e;
  }
  note_launch();
  // One cluster while its SMs finish a step in about the time of a grid
  // barrier: a QR step costs 3 p q FP64 operations, 32 a clock on 16 SMs.
  // The cluster is as small as keeps a Jacobi round (5 p operations per pair)
  // near 600 clocks, for a faster barrier.
  if (setup.max_cluster >= 2 && (long long)p * q <= 40000) {
    int ctas = 2;
    while (ctas < setup.max_cluster && (long long)rmax / 2 * 5 * p > 1200LL * ctas) ctas *= 2;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = cluster_config(ctas, st, attr);
    return cudaLaunchKernelEx(&cfg, svd_split_kernel<true>, a);
  }
  int grid = p < setup.max_ctas ? p : setup.max_ctas;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((void*)svd_split_kernel<false>, dim3(grid), dim3(NT), args, 0,
                                     st);
}

}  // namespace

cudaError_t svd_split_f64_if(const double* M, int m, int n, int kcap, SplitMode mode,
                             double* left, double* right, const SvdBuffers& buf, cudaStream_t st,
                             const double* run_if, double thresh, const SvdDeviceAcc& acc,
                             bool cleared) {
  if (!run_if) return cudaErrorInvalidValue;
  return svd_launch(M, m, n, kcap, 0.0, mode, left, right, buf, st, run_if, thresh, acc, cleared);
}

cudaError_t svd_split_f64(const double* M, int m, int n, int kcap, double rel_tol, SplitMode mode,
                          double* left, double* right, const SvdBuffers& buf, cudaStream_t st,
                          SvdResult* res, bool* converged) {
  *converged = true;
  cudaError_t e = svd_launch(M, m, n, kcap, rel_tol, mode, left, right, buf, st, nullptr, 0.0,
                             SvdDeviceAcc{nullptr, nullptr, nullptr});
  if (e != cudaSuccess) return e;
  int out[4];
  double stats[5];
  if ((e = cudaMemcpyAsync(out, buf.kept, sizeof out, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(stats, buf.stats, sizeof stats, cudaMemcpyDeviceToHost, st)) !=
      cudaSuccess)
    return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  if (out[3] == 1) return cudaErrorLaunchTimeout;
  if (out[3] == 2) *converged = false;
  res->k = out[0];
  res->rank = out[1];
  res->sweeps = out[2];
  res->discarded = stats[1];
  res->sigma_max = stats[2];
  res->columns = (int)stats[4];
  return cudaSuccess;
}
