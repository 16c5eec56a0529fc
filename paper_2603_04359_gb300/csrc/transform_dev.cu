// Device (float64) construction of the block-CAT transform (Sec. 4, Eq. 7 and Eq. 10) for k <= 128.
//
// For every k x k block, with Sigma_x = L L^T and Sigma_w = R R^T (Cholesky):
//   G = Sigma_w # Sigma_x^{-1} = L^{-T} (L^T Sigma_w L)^{1/2} L^{-1}           (Eq. 7)
//   C = L^T Sigma_w L = X X^T with X = L^T R.  One-sided Jacobi rotations make the columns of X orthogonal,
//   W = X J with w_i = sigma_i u_i, so C^{1/2} = sum_i w_i w_i^T / sigma_i and
//   G = Y Y^T with y_i = L^{-T} w_i sigma_i^{-1/2}.  The same rotations on Y give w2_i = lambda_i^{1/2} u_i:
//   M = G^{1/2} = sum_i w2_i w2_i^T lambda_i^{-1/2},  M^{-1} = sum_i w2_i w2_i^T lambda_i^{-3/2},
//   T = H_k M,  (T^{-1})^T = H_k M^{-1}                                          (Eq. 10)
// C and G are never formed: the eigenvalues come from factors, which keeps the small ones accurate.
//
// This GPU issues about two float64 fmas per cycle and SM, so the count of float64 operations is what a
// kernel takes.  The rotations are nearly all of them (k^2 / 2 pairs a sweep on vectors of k): one-sided
// (no second factor to rotate), in the scaled form of Gentleman (two fmas per element instead of four
// operations; the columns' scales are kept apart and folded in once a sweep), their angles in float32 (a
// sweep is repeated until the columns are orthogonal; each rotation is made orthogonal in float64).  A
// block's rows are split over a cluster of four CTAs, which exchange k / 2 partial inner products a round,
// so that 32 blocks keep 128 SMs busy.  Measured, 4096 channels at k = 128: 9.9 ms (rotations 5.1 and 3.4 in
// 11 and 7 sweeps of ~0.47, Cholesky 0.8, products 0.6) against 271 ms for the host's Jacobi on 16 cores.  A
// round takes ~3.6 us, ~1.5 of them fmas; the rest is the exchange across the cluster (four CTAs are the best: two
// double the fmas, eight do not fit the SMs).
//
// The host path (transform_host.cpp) stays for what this one does not decide: k = 256, the diagonal kind, a few
// blocks of k = 16 and 32 (transform_dev_supported), and any layer with a block whose condition numbers may exceed 1e11 (a bound from the traces of a block
// and its inverse) or that is not positive definite: the flags then send the whole layer there.
#include <cmath>

#include "common.cuh"
#include "gemm_pair.cuh"

namespace cat {
namespace {

constexpr int kThreads = 256;
constexpr int kCluster = 4;
constexpr int kMaxSweeps = 30;
constexpr double kMaxCond = 1e11;

// flags[0]: a Cholesky factor or its condition; [1]: the first rotations; [2]: the second ones
__device__ __forceinline__ void raise(int* flag) { atomicOr(flag, 1); }

// 2^e as a double, |e| <= 1000
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// CTA (block b, which): Cholesky factor of Sigma_x (sums / n, which = 0) or Sigma_w (1), scaled by 2^-e, e a
// multiple of 4 near the trace's exponent, and for Sigma_x the factor's inverse.
template <int K>
__global__ void __launch_bounds__(kThreads)
    chol_kernel(const double* __restrict__ sx, double inv_n, const double* __restrict__ sw, double* __restrict__ lx,
                double* __restrict__ lw, double* __restrict__ lxi, int* __restrict__ exps, int* __restrict__ flags) {
  extern __shared__ double sm[];
  constexpr int LD = K + 1;
  double* S = sm;                 // lower: the factor; strictly above the diagonal: its inverse, transposed
  double* dinv = sm + K * LD;     // 1 / diagonal
  double* red = dinv + K;         // column sums of squares of the inverse
  __shared__ double s_tr;
  __shared__ int s_bad;
  const int b = blockIdx.x, which = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* in = (which ? sw : sx) + (size_t)b * K * K;
  const double f = which ? 1.0 : inv_n;
  if (tid == 0) {
    double tr = 0.0;
#pragma unroll 16
    for (int i = 0; i < K; ++i) tr += in[i * K + i] * f;
    s_tr = tr;
    s_bad = !(tr > 1e-280 && tr < 1e280);
  }
  __syncthreads();
  if (s_bad) {                    // uniform over the CTA
    if (tid == 0) raise(flags);
    return;
  }
  const int e = (ilogb(s_tr) >> 2) * 4;
  const double fs = f * pow2(-e);
  if (tid == 0) exps[2 * b + which] = e;
  for (int q = tid; q < K * K; q += kThreads) {
    const int i = q / K, j = q % K;
    if (j <= i) S[i * LD + j] = 0.5 * (in[i * K + j] + in[j * K + i]) * fs;
  }
  __syncthreads();
  for (int j = 0; j < K; ++j) {
    if (tid == 0) {
      double d = S[j * LD + j];
      if (!(d > 0.0) || !(d < 1e300)) {
        s_bad = 1;
        d = 1.0;
      }
      // d^{-1/2} by Newton steps from float32 (d is at most the scaled trace; tiny pivots by the library)
      double r = (double)rsqrtf((float)d);
      r = r * (1.5 - 0.5 * d * r * r);
      r = r * (1.5 - 0.5 * d * r * r);
      if (!(d > 1e-30)) r = 1.0 / sqrt(d);
      S[j * LD + j] = d * r;
      dinv[j] = r;
    }
    __syncthreads();
    if (s_bad) break;             // uniform: read after the barrier, set before it
    for (int i = j + 1 + tid; i < K; i += kThreads) S[i * LD + j] *= dinv[j];
    __syncthreads();
    for (int i = j + 1 + warp; i < K; i += kThreads / 32) {
      const double lij = S[i * LD + j];
      for (int l = j + 1 + lane; l <= i; l += 32) S[i * LD + l] -= lij * S[l * LD + j];
    }
    __syncthreads();
  }
  if (s_bad) {
    if (tid == 0) raise(flags);
    return;
  }
  // inverse of the factor, one column per thread: x_i = -(sum_{c <= j < i} L_ij x_j) / L_ii
  if (tid < K) {
    const int c = tid;
    double sq = dinv[c] * dinv[c];
    for (int i = 1; i < K; ++i) {
      double s4[4] = {0.0, 0.0, 0.0, 0.0};         // four chains: the sums are a matter of latency
      for (int j0 = 0; j0 < i; j0 += 4)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int j = j0 + e;
          if (j < i) s4[e] += S[i * LD + j] * (j < c ? 0.0 : (j == c ? dinv[c] : S[c * LD + j]));
        }
      if (i > c) {
        const double x = -((s4[0] + s4[1]) + (s4[2] + s4[3])) * dinv[i];
        S[c * LD + i] = x;
        sq += x * x;
      }
    }
    red[c] = sq;
  }
  __syncthreads();
  if (tid == 0) {
    double ti = 0.0;
    for (int i = 0; i < K; ++i) ti += red[i];
    // cond <= tr(A) tr(A^{-1}) <= k^2 cond
    if (!(s_tr * pow2(-e) * ti <= kMaxCond)) raise(flags);
  }
  double* out = (which ? lw : lx) + (size_t)b * K * K;
  for (int q = tid; q < K * K; q += kThreads) {
    const int i = q / K, j = q % K;
    out[q] = j <= i ? S[i * LD + j] : 0.0;
    if (!which) lxi[(size_t)b * K * K + q] = j > i ? 0.0 : (j == i ? dinv[i] : S[j * LD + i]);
  }
}

// C[b] = A[b]^T B[b], column j times sig2[b][j]^{-1/4} when sig2 is given; CTA: a 32 x 32 tile of block b.
__global__ void __launch_bounds__(kThreads)
    tn_kernel(const double* __restrict__ A, const double* __restrict__ B, const double* __restrict__ sig2, int K,
              double* __restrict__ C) {
  __shared__ double as[32][33], bs[32][33];
  const int b = blockIdx.x, i0 = blockIdx.y * 32, j0 = blockIdx.z * 32, tid = threadIdx.x;
  const double* Ab = A + (size_t)b * K * K;
  const double* Bb = B + (size_t)b * K * K;
  const int tx = tid & 15, ty = tid >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int l0 = 0; l0 < K; l0 += 32) {
    for (int q = tid; q < 32 * 32; q += kThreads) {
      const int l = q >> 5, c = q & 31;
      as[l][c] = (l0 + l < K && i0 + c < K) ? Ab[(size_t)(l0 + l) * K + i0 + c] : 0.0;
      bs[l][c] = (l0 + l < K && j0 + c < K) ? Bb[(size_t)(l0 + l) * K + j0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < 32; ++l) {
      const double a0 = as[l][ty], a1 = as[l][ty + 16], b0 = bs[l][tx], b1 = bs[l][tx + 16];
      acc[0][0] += a0 * b0;
      acc[0][1] += a0 * b1;
      acc[1][0] += a1 * b0;
      acc[1][1] += a1 * b1;
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int i = i0 + ty + 16 * u, j = j0 + tx + 16 * v;
      if (i >= K || j >= K) continue;
      C[((size_t)b * K + i) * K + j] = sig2 ? acc[u][v] / sqrt(sqrt(sig2[(size_t)b * K + j])) : acc[u][v];
    }
}

// a double stored at the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ void st_cluster(double* p, uint32_t rank, double v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

// One-sided Jacobi rotations of the columns of X[b] (K x K, in place) until they are orthogonal; sig2 gets
// the squared norms.  Cluster of four CTAs per block, K / 4 rows each.  A round rotates K / 2 disjoint
// column pairs (round robin).  Eight warps hold the rows (a warp its own, lane = pair): inner products, then the
// rotations.  Two more warps (thread = pair) add up the partial inner products, exchange them and find the
// angles; what an angle needs besides the inner product is worked out before the exchange, and the scales and
// norms are updated while the others rotate, so a round's chain of float64 latencies is short.  Every CTA adds
// up the same partial inner products in the same order, so all four take the same decisions.
template <int K>
struct JacCfg {
  static constexpr int RPC = K / kCluster, PAIRS = K / 2;
  static constexpr int NW = RPC < 8 ? RPC : 8, RW = RPC / NW;   // warps with rows, rows per warp
  static constexpr int PL = PAIRS > 32 ? PAIRS / 32 : 1;        // pairs per lane
  static constexpr int WARPS = 8 + PL;
  static constexpr size_t SMEM =
      (size_t)(RPC * K + NW * PAIRS + 2 * kCluster * PAIRS + kCluster * K + 3 * K + 2 * PAIRS) * sizeof(double);
};

template <int K>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(JacCfg<K>::WARPS * 32)
    jacobi_kernel(double* __restrict__ X, double* __restrict__ sig2, const int* __restrict__ skip_if, int n_skip,
                  int* __restrict__ flag) {
  using C = JacCfg<K>;
  constexpr int RPC = C::RPC, PAIRS = C::PAIRS, NW = C::NW, RW = C::RW, PL = C::PL, NT = C::WARPS * 32;
  extern __shared__ double sm[];
  double* xs = sm;                                // [RPC][K]
  double* part = xs + RPC * K;                    // [NW][PAIRS]
  double* inbox = part + NW * PAIRS;              // [2][kCluster][PAIRS]
  double* inbox_n = inbox + 2 * kCluster * PAIRS; // [kCluster][K]
  double* nrm = inbox_n + kCluster * K;           // squared norms of the (scaled) columns
  double* scl = nrm + K;                          // column scales and their reciprocals
  double* isc = scl + K;
  double* m1 = isc + K;                           // [PAIRS] multipliers of the round
  double* m2 = m1 + PAIRS;
  __shared__ int s_big;
  const int b = blockIdx.x / kCluster, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_rank();
  for (int i = 0; i < n_skip; ++i)
    if (skip_if[i]) return;                       // raised by earlier launches: the same for the whole grid
  double* Xb = X + (size_t)b * K * K + (size_t)rank * RPC * K;
  for (int q = tid; q < RPC * K; q += NT) xs[q] = Xb[q];
  for (int c = tid; c < K; c += NT) scl[c] = isc[c] = 1.0;
  if (tid == 0) s_big = 0;
  cluster_sync();
  // the round's pair i: column K - 1 with r for i = 0, r + i with r - i modulo K - 1 for the others
  auto pair_of = [](int i, int r, int* p, int* q) {
    *p = i == 0 ? K - 1 : r + i - (r + i >= K - 1 ? K - 1 : 0);
    *q = i == 0 ? r : r - i + (r - i < 0 ? K - 1 : 0);
  };
  bool done = false;
  uint32_t round = 0;
  auto fold = [&] {                               // the scales into the columns, and the columns' norms
    for (int q = tid; q < RPC * K; q += NT) xs[q] *= scl[q % K];
    __syncthreads();
    for (int c = tid; c < K; c += NT) {
      double s = 0.0;
#pragma unroll 4
      for (int r = 0; r < RPC; ++r) s += xs[r * K + c] * xs[r * K + c];
      for (uint32_t p = 0; p < kCluster; ++p) st_cluster(&inbox_n[rank * K + c], p, s);
      scl[c] = isc[c] = 1.0;
    }
    cluster_sync();
    for (int c = tid; c < K; c += NT)
      nrm[c] = ((inbox_n[c] + inbox_n[K + c]) + inbox_n[2 * K + c]) + inbox_n[3 * K + c];
    __syncthreads();
  };
  for (int sweep = 0; sweep < kMaxSweeps && !done; ++sweep) {
    fold();
    if (warp < 8) {
      // ---------------------------------------------------------------- rows: warp w holds w RW .. w RW + RW - 1
      const bool work = warp < NW && (PAIRS >= 32 || lane < PAIRS);
      double* xw = xs + (work ? warp * RW * K : 0);
      for (int r = 0; r < K - 1; ++r, ++round) {
        int p[PL], q[PL];
        double x[PL][RW], y[PL][RW];
#pragma unroll
        for (int u = 0; u < PL; ++u) {
          pair_of((lane + 32 * u) % PAIRS, r, &p[u], &q[u]);
          double s = 0.0;
#pragma unroll
          for (int i = 0; i < RW; ++i) {
            x[u][i] = xw[i * K + p[u]];
            y[u][i] = xw[i * K + q[u]];
            s += x[u][i] * y[u][i];
          }
          if (work) part[warp * PAIRS + lane + 32 * u] = s;
        }
        __syncthreads();
        cluster_sync();
        __syncthreads();                          // the multipliers are there
        if (work) {
#pragma unroll
          for (int u = 0; u < PL; ++u) {
            const double u1 = m1[lane + 32 * u], u2 = m2[lane + 32 * u];
#pragma unroll
            for (int i = 0; i < RW; ++i) {
              xw[i * K + p[u]] = x[u][i] - u1 * y[u][i];
              xw[i * K + q[u]] = y[u][i] + u2 * x[u][i];
            }
          }
        }
        __syncwarp();                             // the next round's pairs lie in other lanes of this warp
      }
    } else {
      // ---------------------------------------------------------------- angles: thread = pair
      const int pr = tid - 256;
      const bool work = pr < PAIRS;
      for (int r = 0; r < K - 1; ++r, ++round) {
        int p, q;
        pair_of(work ? pr : 0, r, &p, &q);
        __syncthreads();                          // the partial inner products, and the last round's scales and norms
        double* in = inbox + (round & 1u) * (kCluster * PAIRS);
        if (work) {
          double s[NW];
#pragma unroll
          for (int g = 0; g < NW; ++g) s[g] = part[g * PAIRS + pr];
#pragma unroll
          for (int w = NW / 2; w > 0; w /= 2)
#pragma unroll
            for (int g = 0; g < w; ++g) s[g] += s[g + w];
          for (uint32_t c = 0; c < kCluster; ++c) st_cluster(&in[rank * PAIRS + pr], c, s[0]);
        }
        // what the angle needs besides the inner product; rs scales its operands to about 1
        const double sp = scl[p], sq = scl[q], ip = isc[p], iq = isc[q], aa = nrm[p], bb = nrm[q];
        const double big = aa > bb ? aa : bb;
        const double rs = pow2(1023 - (int)((__double_as_longlong(big) >> 52) & 0x7FF));
        const double ss = sp * sq, sr = ss * rs, k1 = sq * ip, k2 = sp * iq;
        const float df = (float)((bb - aa) * rs), root = sqrtf((float)(aa * rs)) * sqrtf((float)(bb * rs));
        __syncwarp();
        cluster_sync();                           // round r + 2 writes this inbox only after round r + 1's barrier
        double t = 0.0, ab = 0.0;
        if (work) {
          const double dot = (in[pr] + in[PAIRS + pr]) + (in[2 * PAIRS + pr] + in[3 * PAIRS + pr]);
          const float abf = (float)(dot * sr);
          if (!(fabsf(abf) <= 1e-16f * root)) {
            // the columns are orthogonal to 1e-8 of their norms at every rotation of the last sweep: what that sweep
            // leaves is the square of it
            if (!(fabsf(abf) <= 1e-8f * root)) s_big = 1;
            const float zeta = df / (2.0f * abf);
            const float t32 = copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(1.0f + zeta * zeta));
            if (isfinite(t32)) t = (double)t32;
            ab = dot * ss;
          }
          m1[pr] = t * k1;
          m2[pr] = t * k2;
        }
        __syncthreads();                          // the others rotate; meanwhile:
        if (work && t != 0.0) {
          // c = (1 + t^2)^{-1/2} by Newton steps from float32, 1 / c = (1 + t^2) c
          const double x = 1.0 + t * t;
          double c = (double)rsqrtf((float)x);
          c = c * (1.5 - 0.5 * x * c * c);
          c = c * (1.5 - 0.5 * x * c * c);
          const double ci = x * c;
          scl[p] = sp * c;
          scl[q] = sq * c;
          isc[p] = ip * ci;
          isc[q] = iq * ci;
          nrm[p] = aa - t * ab;
          nrm[q] = bb + t * ab;
        }
      }
    }
    __syncthreads();
    done = s_big == 0;
    __syncthreads();
    if (tid == 0) s_big = 0;
    __syncthreads();
  }
  fold();
  if (tid == 0) {
    double lo = nrm[0], hi = nrm[0];
    for (int c = 1; c < K; ++c) {
      lo = nrm[c] < lo ? nrm[c] : lo;
      hi = nrm[c] > hi ? nrm[c] : hi;
    }
    double sum = 0.0;
    for (int c = 0; c < K; ++c) sum += nrm[c];     // a NaN anywhere
    if (!done || !(lo > 0.0) || !(hi <= kMaxCond * lo) || !(sum < 1e300)) raise(flag);
  }
  for (int q = tid; q < RPC * K; q += NT) Xb[q] = xs[q];
  if (rank == 0)
    for (int c = tid; c < K; c += NT) sig2[(size_t)b * K + c] = nrm[c];
  cluster_sync();                                 // no CTA leaves while another may still write to it
}

// T[b] = H M and Aw[b] = H M^{-1} (with_h), or M and M^{-1}: CTA (block, panel of PW columns).
template <int K>
__global__ void __launch_bounds__(kThreads)
    compose_kernel(const double* __restrict__ W, const double* __restrict__ lam, const int* __restrict__ exps, int with_h,
                   float* __restrict__ T, float* __restrict__ Aw, const int* __restrict__ flags) {
  constexpr int PW = K < 32 ? K : 32, RS = kThreads / PW, R = K / RS > 0 ? K / RS : 1, EC = 16;
  extern __shared__ double sm[];
  double* mo = sm;                  // [2][K][PW]
  double* wt = sm + 2 * K * PW;     // [K][EC + 1]
  double* f1 = wt + K * (EC + 1);   // [EC] lambda^{-1/2}
  double* f2 = f1 + EC;             // [EC] lambda^{-3/2}
  if (flags[0] | flags[1] | flags[2]) return;     // the host path writes this layer's T
  const int b = blockIdx.x, j0 = blockIdx.y * PW, tid = threadIdx.x;
  const double* Wb = W + (size_t)b * K * K;
  const int j = tid % PW, r0 = tid / PW;
  double a1[R], a2[R];
#pragma unroll
  for (int u = 0; u < R; ++u) a1[u] = a2[u] = 0.0;
  for (int e0 = 0; e0 < K; e0 += EC) {
    for (int q = tid; q < K * EC; q += kThreads) wt[(q / EC) * (EC + 1) + q % EC] = Wb[(size_t)(q / EC) * K + e0 + q % EC];
    if (tid < EC) {
      const double l = lam[(size_t)b * K + e0 + tid], s = sqrt(l);
      f1[tid] = 1.0 / s;
      f2[tid] = 1.0 / (s * l);
    }
    __syncthreads();
#pragma unroll 4
    for (int e = 0; e < EC; ++e) {
      const double w = wt[(j0 + j) * (EC + 1) + e], w1 = w * f1[e], w2 = w * f2[e];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int i = r0 + RS * u;
        if (i < K) {
          a1[u] += wt[i * (EC + 1) + e] * w1;
          a2[u] += wt[i * (EC + 1) + e] * w2;
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < R; ++u) {
    const int i = r0 + RS * u;
    if (i < K) {
      mo[i * PW + j] = a1[u];
      mo[(K + i) * PW + j] = a2[u];
    }
  }
  __syncthreads();
  if (with_h) {                     // fast Walsh-Hadamard transform down every column
    for (int len = 1; len < K; len <<= 1) {
      for (int q = tid; q < K * PW; q += kThreads) {          // K / 2 butterflies per column, two matrices
        const int c = q % PW, h = (q / PW) % (K / 2), mat = q / (PW * (K / 2));
        const int i = (h / len) * 2 * len + h % len;
        double* p = mo + ((size_t)mat * K + i) * PW + c;
        const double x = p[0], y = p[len * PW];
        p[0] = x + y;
        p[len * PW] = x - y;
      }
      __syncthreads();
    }
  }
  // the blocks were scaled by 2^-ex and 2^-ew (multiples of 4): M by 2^((ew - ex) / 4)
  const int de = (exps[2 * b + 1] - exps[2 * b]) / 4;
  const double h = with_h ? 1.0 / sqrt((double)K) : 1.0;
  const double s1 = h * pow2(de), s2 = h * pow2(-de);
  for (int q = tid; q < K * PW; q += kThreads) {
    const int i = q / PW, c = q % PW;
    const size_t o = ((size_t)b * K + i) * K + j0 + c;
    T[o] = (float)(mo[i * PW + c] * s1);
    Aw[o] = (float)(mo[(K + i) * PW + c] * s2);
  }
}

template <int K>
cudaError_t build_k(int64_t nb, const double* sx, int64_t n_calib, const double* sw, int with_h, float* T, float* Aw,
                    double* work, int* ints, cudaStream_t s) {
  constexpr size_t kChol = (size_t)(K * (K + 1) + 2 * K) * 8;
  constexpr size_t kJac = JacCfg<K>::SMEM;
  constexpr int kJacThreads = JacCfg<K>::WARPS * 32;
  constexpr int PW = K < 32 ? K : 32;
  constexpr size_t kComp = (size_t)(2 * K * PW + K * 17 + 32) * 8;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(chol_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChol)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(jacobi_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJac)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(compose_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kComp)) != cudaSuccess) return e;
  const size_t blk = (size_t)nb * K * K;
  double *b0 = work, *b1 = work + blk, *b2 = work + 2 * blk, *b3 = work + 3 * blk, *sig = work + 4 * blk;
  int *flags = ints, *exps = ints + 4;
  if ((e = cudaMemsetAsync(flags, 0, 4 * sizeof(int), s)) != cudaSuccess) return e;
  const unsigned g = (unsigned)nb, tl = (unsigned)((K + 31) / 32);
  auto launched = [&] {
    note_launch();
    return cudaGetLastError();
  };
  chol_kernel<K><<<dim3(g, 2), kThreads, kChol, s>>>(sx, 1.0 / (double)n_calib, sw, b0, b1, b2, exps, flags);
  if ((e = launched()) != cudaSuccess) return e;
  tn_kernel<<<dim3(g, tl, tl), kThreads, 0, s>>>(b0, b1, nullptr, K, b3);            // X = L^T R
  if ((e = launched()) != cudaSuccess) return e;
  jacobi_kernel<K><<<kCluster * g, kJacThreads, kJac, s>>>(b3, sig, flags, 1, flags + 1);
  if ((e = launched()) != cudaSuccess) return e;
  tn_kernel<<<dim3(g, tl, tl), kThreads, 0, s>>>(b2, b3, sig, K, b0);                // Y = L^{-T} W sigma^{-1/2}
  if ((e = launched()) != cudaSuccess) return e;
  jacobi_kernel<K><<<kCluster * g, kJacThreads, kJac, s>>>(b0, sig, flags, 2, flags + 2);
  if ((e = launched()) != cudaSuccess) return e;
  compose_kernel<K><<<dim3(g, K / PW), kThreads, kComp, s>>>(b0, sig, exps, with_h, T, Aw, flags);
  return launched();
}

}  // namespace

// A few small blocks are built faster on the host (16 cores), where each has a core to itself: the whole preparation of a
// layer with 2, 4, 8 and 16 blocks, us host/device: k = 16 570/770 580/770 830/790 1170/800, k = 32 1345/1450 1400/1425 1640/1500
// 2040/1510.
bool transform_dev_supported(int k, int64_t nb) {
  return k <= 128 && nb <= 0x0FFFFFFF && nb >= (k == 16 ? 8 : (k == 32 ? 5 : 1));
}

// Stream-ordered scratch of one build: doubles, then ints (4 flags, two exponents per block).
size_t transform_dev_bytes(int k, int64_t nb) {
  return ((size_t)4 * nb * k * k + (size_t)nb * k) * sizeof(double) + (size_t)(4 + 2 * nb) * sizeof(int);
}

// T [nb][k][k] and Aw = (T^{-1})^T from the sums Sigma_x (over n_calib tokens) and Sigma_w; work: scratch of
// transform_dev_bytes.  *flags: three device ints; if any is nonzero once the stream is synchronized, T and
// Aw were not written and the layer is for the host path.
cudaError_t launch_build_transform(int k, int64_t nb, const double* sx, int64_t n_calib, const double* sw, int with_h,
                                   float* T, float* Aw, void* work, const int** flags, cudaStream_t s) {
  double* w = static_cast<double*>(work);
  int* ints = reinterpret_cast<int*>(w + (size_t)4 * nb * k * k + (size_t)nb * k);
  *flags = ints;
  switch (k) {
    case 16: return build_k<16>(nb, sx, n_calib, sw, with_h, T, Aw, w, ints, s);
    case 32: return build_k<32>(nb, sx, n_calib, sw, with_h, T, Aw, w, ints, s);
    case 64: return build_k<64>(nb, sx, n_calib, sw, with_h, T, Aw, w, ints, s);
    case 128: return build_k<128>(nb, sx, n_calib, sw, with_h, T, Aw, w, ints, s);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace cat
