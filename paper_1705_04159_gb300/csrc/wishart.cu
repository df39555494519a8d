// wishart.cu -- the Normal-Wishart draw of one side's hyperparameters from its
// row mean and scatter (Algorithm 1), in FP64, by one cluster of CTAs.
//
// With n rows, mean xbar and centred scatter S, W*^-1 = W0^-1 + S + beta0 n /
// (beta0 + n) (mu0 - xbar)(mu0 - xbar)^T, nu* = nu0 + n, beta* = beta0 + n,
// Lambda = (C A)(C A)^T with C = chol(W*) and Bartlett's A, mu = mu* +
// chol(beta* Lambda)^-T z.  Exact identities keep the FP64 work to about
// K^3 / 6 multiply-adds per step:
//  * C = chol(W*) without forming W* = (W*^-1)^-1: with J the reversal
//    permutation and L_M = chol(J W*^-1 J), W*^-1 = (J L_M J)(J L_M J)^T with
//    J L_M J upper triangular, so W* = (J L_M^-T J)(J L_M^-T J)^T and
//    C = J L_M^-T J, i.e. C[i][j] = T[K-1-j][K-1-i] with T = L_M^-1
//    (lower triangular with a positive diagonal, hence the Cholesky factor);
//  * L_M = L' D^1/2 with L' unit lower triangular, so T = D^-1/2 L'^-1, and
//    neither the factorisation nor the substitution has a root in its chain;
//  * chol(beta* Lambda) = sqrt(beta*) B for B = C A (lower triangular with a
//    positive diagonal and Lambda = B B^T), so mu = mu* + B^-T z / sqrt(beta*)
//    and Lambda mu = B (B^T mu* + z / sqrt(beta*)).
//
// What bounds it: on a GB300 a quarter of an SM takes 64 cycles for one FP64
// warp instruction, whatever the number of active lanes, and as long for a
// dependent one.  So the work is spread over warps and SMs by instruction, the
// lanes are filled, and the chains (a pivot to the next, a solved entry to the
// next) are kept short.  The phases, with a cluster barrier between them:
//   1. CTA 0 factors J W*^-1 J = L' D L'^T, the other CTAs draw Bartlett's A;
//   2. a warp per column j of T: forward substitution with L', then at once
//      row K-1-j of B = C A, which needs no other column of T;
//   3. a warp per row of Lambda = B B^T and of Lambda mu; one warp solves for mu.
// One draw alone (five kernels of one or K CTAs before: factorisation,
// substitution, B, Lambda, mu): 45 -> 22 us at K = 10, 90 -> 34 at K = 32, 182 ->
// 70 at K = 64, of which now the factorisation 13 and 34 us, the substitution
// and B 5.7 and 13.5, Lambda and mu 5 and 9.5.
#include <cuda_runtime.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "hyper.cuh"

namespace gb {
namespace {

constexpr int kWishThreads = 256, kWishWarps = kWishThreads / 32;
constexpr int kNpl = kMaxK / 32;
constexpr unsigned kFull = 0xffffffffu;

// CTAs of the cluster: one column of T a quarter SM for K <= 64, two up to 128.
// Past eight the size is not portable, and a device whose GPCs offer fewer SMs (a
// partition of one) takes the largest half that fits (wish_cluster); the warps then
// take their columns in several rounds.
int wish_ctas(int K) { return K <= 16 ? 4 : K <= 32 ? 8 : 16; }

// The column of T that a warp begins with: one a quarter SM (warps 0 - 3), then
// the rest in reverse order, a short column to a long one; 8 nc further in each
// round.
__device__ __forceinline__ int first_column(int cta, int nc, int warp) {
  return warp < 4 ? cta + nc * warp : 8 * nc - 1 - (cta + nc * (warp - 4));
}

__host__ __device__ inline int wish_packed(int K) { return (K * (K + 1) / 2 + 1) & ~1; }
// the matrix, then B; A, then B scaled; a row of C per warp; (row, column) of the packed elements
int wish_smem(int K) {
  return (int)sizeof(double) * (2 * wish_packed(K) + kWishWarps * K) + (int)sizeof(uint16_t) * wish_packed(K);
}
// First element of column j of the lower triangle, packed by columns from the
// last on, so that the columns past any j are the elements before its first.
__device__ __forceinline__ int col_off(int K, int j) { return (K - 1 - j) * (K - j) / 2; }

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// 1 / d = r (1 + t) for d > 0: r the reciprocal to FP32 accuracy, t = e + e^2
// with e = 1 - d r, which leaves an error of e^3 = 2^-66 before rounding.  x / d
// is then (x r) + (x r) t, whose first product is off the chain; a division
// in the pivots' chain would be more than twice as long.
// Returns false if d is not a positive normal number (or one too large): the
// test is on the bits, an FP64 comparison would be a link of the chain.
__device__ __forceinline__ bool reciprocal(double d, double& r, double& t) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  if ((unsigned)(hi - 0x00100000) >= 0x7fd00000u - 0x00100000u) return false;
  // the mantissa m in [1, 2), its reciprocal in FP32, both as bits
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, lo);
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(f)
      : "f"(__int_as_float(0x3f800000 | ((hi & 0x000fffff) << 3) | ((unsigned)lo >> 29))));
  const int fb = __float_as_int(f), ex = (hi >> 20) - 1023;
  const int h = (fb >> 3) + ((1023 - 127) << 20);
  const double rm = __hiloint2double(h, (int)((unsigned)fb << 29));
  const double e = fma(-m, rm, 1.0);
  t = fma(e, e, e);
  r = __hiloint2double(h - (ex << 20), (int)((unsigned)fb << 29));
  return true;
}

// M = L' D L'^T in place by one CTA: M holds the lower triangle (col_off), ij
// the row and column of its elements; D goes to dg, its place in M is not
// written.  Right-looking: at step c warp w < 4 updates rows c + 1 + 32 w and
// on of column c + 1, scales them and publishes them unscaled (us) and scaled
// (ls); every one of these warps forms the pivot for itself, which costs an
// instruction on its own quarter of the SM and saves a barrier.  The other
// warps update the columns after it by 32 packed elements at a time; one
// barrier a step.  So a step takes the longer of the chain (six FP64
// instructions and some 300 cycles of shared memory, barrier and integer
// work) and the trailing elements at 16 cycles per 32.  Returns false (to warp
// 0) if a pivot is not positive.
__device__ bool ldl_factor(double* M, const uint16_t* ij, int K, double* dg, double (*us)[kMaxK],
                           double (*ls)[kMaxK], int warp, int lane) {
  bool ok = true;
  const int v = lane + 32 * warp;
  // rows j + v of column j, given their elements x and the pivot
  auto publish = [&](int j, double x, double d) {
    double r, t;
    if (!reciprocal(d, r, t)) {
      ok = ok && d > 0.0;
      r = 1.0 / (d > 0.0 ? d : 1.0);
      t = 0.0;
    }
    const double y = x * r;
    const double l = fma(y, t, y);
    if (v == 0) dg[j] = d;
    if (j + v < K) {
      us[j & 1][j + v] = x;
      ls[j & 1][j + v] = l;
      if (v > 0) M[col_off(K, j) + v] = l;
    }
  };
  if (32 * warp < K) {
    const double d = M[col_off(K, 0)];
    publish(0, v < K ? M[col_off(K, 0) + v] : 0.0, d);
  }
  for (int c = 0; c + 1 < K; ++c) {
    const int j = c + 1, nm = (K - j + 31) >> 5;  // warps of column j
    __syncthreads();
    const double *u = us[c & 1], *l = ls[c & 1];
    if (warp < nm) {
      const double* col = M + col_off(K, j);
      const double uj = u[j];
      const double d = fma(-l[j], uj, col[0]);
      const double x = warp == 0 && lane == 0 ? d : j + v < K ? fma(-l[j + v], uj, col[v]) : 0.0;
      publish(j, x, d);
    } else if (nm > 1 || warp != 4) {  // one chain has its quarter SM to itself
      const int n = col_off(K, j);
      const int w = nm > 1 ? warp - nm : warp - 1 - (warp > 4), nw = nm > 1 ? kWishWarps - nm : kWishWarps - 2;
      const int st = 32 * nw;
      int e = 32 * w + lane;
      for (; e - lane + 3 * st + 32 <= n; e += 4 * st) {  // four loads in flight
        double x[4], y[4], z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int q = ij[e + i * st];
          x[i] = l[q & 255];
          y[i] = u[q >> 8];
          z[i] = M[e + i * st];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) M[e + i * st] = fma(-x[i], y[i], z[i]);
      }
      for (; e < n; e += st) {
        const int q = ij[e];
        M[e] = fma(-l[q & 255], u[q >> 8], M[e]);
      }
    }
  }
  __syncthreads();
  return ok;
}

// Bartlett's lower-triangular A for Wishart(., nu), packed by rows, by
// nthreads threads: A_kl ~ N(0, 1) for k > l (normal number k (k - 1) / 2 + l
// of counter base (0, t, ., WISHART), Box-Muller in FP32 like the row
// normals: these decide nothing discrete) and A_kk = sqrt(chi^2(nu - k)),
// chi^2(m) = 2 Gamma(m / 2) by Marsaglia-Tsang in FP64 with the attempt
// number as the counter's third word (counter (k, t, a, GAMMA)); the
// acceptance test decides which attempt is kept, so it runs in FP64 like the
// reference.  The attempt cap flags kStatusRng.
__device__ void bartlett(double* A, int K, double nu, uint2 key, uint32_t t, int side, int cap, int* status,
                         int thread, int nthreads) {
  const uint32_t sw_w = stream_word(kStreamWishart, side);
  const uint32_t sw_g = stream_word(kStreamGamma, side);
  for (int k = thread; k < K; k += nthreads) {
    const double shape = 0.5 * (nu - (double)k);
    const double s = shape < 1.0 ? shape + 1.0 : shape;
    const double d = s - 1.0 / 3.0;
    const double c = 1.0 / sqrt(9.0 * d);
    double g = -1.0;
    for (int a = 0; a < cap && g < 0.0; ++a) {
      const uint4 w = philox(make_uint4((uint32_t)k, t, (uint32_t)a, sw_g), key);
      double zn, zs;
      normal2_f64(w.x, w.y, zn, zs);
      double v = 1.0 + c * zn;
      if (v <= 0.0) continue;
      v = v * v * v;
      const double u = unit_f64(w.z);
      if (log(u) < 0.5 * zn * zn + d - d * v + d * log(v)) {
        g = d * v;
        if (shape < 1.0) g *= pow(unit_f64(w.w), 1.0 / shape);
      }
    }
    if (g < 0.0) {
      atomicOr(status, kStatusRng);
      g = s;
    }
    A[k * (k + 1) / 2 + k] = sqrt(2.0 * g);
  }
  // below the diagonal, from the last threads on
  for (int e = nthreads - 1 - thread; e < K * (K - 1) / 2; e += nthreads) {
    int k = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)e)) * 0.5f);
    while (k * (k - 1) / 2 > e) --k;
    while ((k + 1) * k / 2 <= e) ++k;
    const int l = e - k * (k - 1) / 2;
    A[k * (k + 1) / 2 + l] = (double)normal_at_f32(key, 0u, t, sw_w, (uint32_t)e);
  }
}

// n doubles of global memory written by another CTA to shared memory
__device__ __forceinline__ void copy_in(double* dst, const double* src, int n) {
  for (int e0 = threadIdx.x; e0 < n; e0 += 8 * kWishThreads) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = e0 + u * kWishThreads < n ? __ldcg(src + e0 + u * kWishThreads) : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u * kWishThreads < n) dst[e0 + u * kWishThreads] = v[u];
  }
}

__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  return s;
}

// Column j of L'^-1 by one warp, K - j <= 32 G entries from row j on, lane l
// holding entries l + 32 m; scaled by rs, in reverse order, it is row
// K - 1 - j of C, C[i][m] = T[K-1-m][j].  The number of groups is a template
// argument because an FP64 instruction whose lanes are all masked still takes
// its 64 cycles (with four groups and masks, 340 cycles a step instead of 120
// at K = 16).
template <int G>
__device__ __forceinline__ void unit_solve(const double* M, int K, int j, const double* rs, double* out,
                                           int lane) {
  const int len = K - j;
  double x[G];
#pragma unroll
  for (int m = 0; m < G; ++m) x[m] = lane + 32 * m == 0 ? 1.0 : 0.0;
#pragma unroll
  for (int mi = 0; mi < G; ++mi) {
    const int c1 = mi < G - 1 ? 32 : len - 32 * mi;
    // entry q > i of column j + i of L' at col_off(j + i) - i + q
    const double* col = M + col_off(K, j + 32 * mi) - 32 * mi + lane;
    int st = K - j - 32 * mi;
#pragma unroll 4
    for (int c = 0; c < c1; ++c) {
      const double xi = __shfl_sync(kFull, x[mi], c);
      const double l = lane > c && lane < c1 ? col[32 * mi] : 0.0;
      x[mi] = fma(-l, xi, x[mi]);
#pragma unroll
      for (int m = mi + 1; m < G; ++m) x[m] = fma(m < G - 1 || lane + 32 * m < len ? -col[32 * m] : 0.0, xi, x[m]);
      col -= st--;
    }
  }
#pragma unroll
  for (int m = 0; m < G; ++m) {
    const int q = lane + 32 * m;
    if (q < len) out[len - 1 - q] = x[m] * rs[j + q];
  }
}

// The packed element e as (row, column), K - 1 less each.
__device__ __forceinline__ void unpack(int e, int& ri, int& rj) {
  int q = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((q + 1) * (q + 2) / 2 <= e) ++q;
  while (q * (q + 1) / 2 > e) --q;
  rj = q;
  ri = q - (e - q * (q + 1) / 2);
}

// The lower triangle of A (K x K) packed into M by columns, and its element table.
__device__ void load_lower(const double* A, int K, double* M, uint16_t* ij) {
  for (int e = threadIdx.x; e < K * (K + 1) / 2; e += kWishThreads) {
    int ri, rj;
    unpack(e, ri, rj);
    M[e] = A[(K - 1 - ri) * K + K - 1 - rj];
    ij[e] = (uint16_t)((K - 1 - ri) | (K - 1 - rj) << 8);
  }
}

// Ainv = A^-1 = T^T T, T = chol(A)^-1, by the same phases: the factor, a warp
// per column of T, a warp per row of the product (scr: 2 K K + K + 1 doubles).
// One CTA in global memory before: 75 us at K = 32, 663 at K = 100; a burst of
// six small jobs, each of which waits for its W0^-1, 14.0 -> 13.5 ms.
__global__ void __launch_bounds__(kWishThreads, 1) spd_inverse(const double* A, double* Ainv, int K, double* scr,
                                                               int* status) {
  extern __shared__ __align__(16) double wsm[];
  __shared__ double s_dg[kMaxK], s_rr[kMaxK], s_part[4][kMaxK];
  const int np = K * (K + 1) / 2, nc = gridDim.x, cta = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* M = wsm;
  double* cbuf = M + 2 * wish_packed(K) + warp * K;
  uint16_t* ij = reinterpret_cast<uint16_t*>(M + 2 * wish_packed(K) + kWishWarps * K);
  double *gL = scr, *gT = scr + K * K, *gD = gT + K * K, *gok = gD + K;
  const int j0 = first_column(cta, nc, warp);
  if (cta == 0) {
    load_lower(A, K, M, ij);
    __syncthreads();
    const bool ok = ldl_factor(M, ij, K, s_dg, s_part, s_part + 2, warp, lane);
    if (tid == 0) {
      *gok = ok ? 1.0 : 0.0;
      if (!ok) atomicOr(status, kStatusNotPD);
    }
    for (int e = tid; e < np; e += kWishThreads) gL[e] = M[e];
    for (int k = tid; k < K; k += kWishThreads) gD[k] = s_dg[k];
  }
  cluster_sync();
  if (__ldcg(gok) == 0.0) return;
  copy_in(M, gL, np);
  for (int k = tid; k < K; k += kWishThreads) s_rr[k] = rsqrt(__ldcg(gD + k));
  __syncthreads();
  for (int j = j0; j < K; j += 8 * nc) {
    switch ((K - j + 31) >> 5) {
      case 1: unit_solve<1>(M, K, j, s_rr, cbuf, lane); break;
      case 2: unit_solve<2>(M, K, j, s_rr, cbuf, lane); break;
      case 3: unit_solve<3>(M, K, j, s_rr, cbuf, lane); break;
      default: unit_solve<4>(M, K, j, s_rr, cbuf, lane);
    }
    __syncwarp();
    for (int q = lane; q < K - j; q += 32) gT[col_off(K, j) + q] = cbuf[K - 1 - j - q];
    __syncwarp();
  }
  cluster_sync();
  copy_in(M, gT, np);
  __syncthreads();
  for (int j = j0; j < K; j += 8 * nc) {
    // row i = K - 1 - j: entry (i, l), l <= i, is sum over k >= i of T[k][i] T[k][l]
    const int i = K - 1 - j;
    const double* ti = M + col_off(K, i);
    for (int l0 = 0; l0 <= i; l0 += 32) {
      const int l = l0 + lane;
      if (l <= i) {
        const double* tl = M + col_off(K, l) + i - l;
        double s = 0.0, u = 0.0;
        int k = 0;
        for (; k + 2 <= K - i; k += 2) {
          s = fma(ti[k], tl[k], s);
          u = fma(ti[k + 1], tl[k + 1], u);
        }
        if (k < K - i) s = fma(ti[k], tl[k], s);
        Ainv[i * K + l] = Ainv[l * K + i] = s + u;
      }
    }
  }
}

// Checks that A is SPD; on success writes chol(A) in FP32 to lout (lower
// triangle packed by rows: element (i, j) at i (i + 1) / 2 + j).
__global__ void __launch_bounds__(kWishThreads, 1) spd_check(const double* A, int K, int* status, float* lout) {
  extern __shared__ __align__(16) double wsm[];
  __shared__ double s_dg[kMaxK], s_part[4][kMaxK];
  __shared__ int s_ok;
  double* M = wsm;
  uint16_t* ij = reinterpret_cast<uint16_t*>(M + 2 * wish_packed(K) + kWishWarps * K);
  load_lower(A, K, M, ij);
  __syncthreads();
  const bool ok = ldl_factor(M, ij, K, s_dg, s_part, s_part + 2, threadIdx.x >> 5, threadIdx.x & 31);
  if (threadIdx.x == 0) {
    s_ok = ok;
    if (!ok) atomicOr(status, kStatusNotPD);
  }
  __syncthreads();
  if (!s_ok) return;
  for (int k = threadIdx.x; k < K; k += kWishThreads) s_dg[k] = sqrt(s_dg[k]);
  __syncthreads();
  for (int e = threadIdx.x; e < K * (K + 1) / 2; e += kWishThreads) {
    const int i = ij[e] & 255, j = ij[e] >> 8;
    lout[i * (i + 1) / 2 + j] = (float)(i == j ? s_dg[j] : M[e] * s_dg[j]);
  }
}

// Scratch (doubles): L' packed (from 0), A packed (from K K), B packed (from
// 2 K K), D (K, from 4 K K), 1 at 5 K K once the factorisation succeeded (0:
// the draw is left out).
__global__ void __launch_bounds__(kWishThreads, 1) wishart_draw(const HyperArgs a) {
  extern __shared__ __align__(16) double wsm[];
  __shared__ double s_dg[kMaxK], s_rr[kMaxK], s_mus[kMaxK], s_w[kMaxK], s_z[kMaxK], s_part[kWishWarps][kMaxK];
  const int K = a.K, KK = K * K, KA = K + 1, np = K * (K + 1) / 2;
  const int nc = gridDim.x, cta = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* M = wsm;
  double* U = M + wish_packed(K);
  double* cbuf = U + wish_packed(K) + warp * K;
  uint16_t* ij = reinterpret_cast<uint16_t*>(U + wish_packed(K) + kWishWarps * K);
  double* gL = a.scr;
  double* gA = gL + KK;
  double* gB = gA + KK;
  double* gD = gL + 4 * KK;
  double* gok = gL + 5 * KK;
  // the warp's columns j of T, and rows K - 1 - j of B and Lambda, start here
  const int j0 = first_column(cta, nc, warp);
  const double n = (double)a.n;
  const uint2 key = seed_key(a.seed);
  const uint32_t t = *a.tp;
  for (int k = tid; k < K; k += kWishThreads) {
    const double d = a.mu0[k] - a.xbar[k];
    s_w[k] = d;
    s_z[k] = d * a.wmean;
  }
  __syncthreads();

  // ---- 1
  if (cta == 0) {
    // element (i, j): (J W*^-1 J)[i][j] = W*^-1[K-1-i][K-1-j]
    constexpr int kLoads = 8;
    for (int e0 = tid; e0 < np; e0 += kLoads * kWishThreads) {
      double wv[kLoads], sv[kLoads];
      int src[kLoads];
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        const int e = e0 + u * kWishThreads;
        int ri, rj;
        unpack(e, ri, rj);
        src[u] = rj << 8 | ri;
        wv[u] = e < np ? a.W0inv[rj * K + ri] : 0.0;
        sv[u] = e < np ? a.S[rj * K + ri] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        const int e = e0 + u * kWishThreads;
        const int ri = src[u] & 255, rj = src[u] >> 8;
        if (e < np) {
          M[e] = fma(s_z[rj], s_w[ri], wv[u] + sv[u]);
          ij[e] = (uint16_t)((K - 1 - ri) | (K - 1 - rj) << 8);
        }
      }
    }
    __syncthreads();
    const bool ok = ldl_factor(M, ij, K, s_dg, s_part, s_part + 2, warp, lane);
    if (tid == 0) {
      *gok = ok ? 1.0 : 0.0;
      if (!ok) atomicOr(a.status, kStatusNotPD);
    }
    for (int e = tid; e < np; e += kWishThreads) gL[e] = M[e];
    for (int k = tid; k < K; k += kWishThreads) gD[k] = s_dg[k];
  } else {
    bartlett(gA, K, a.nu0 + n, key, t, a.side, a.gamma_cap, a.status, (cta - 1) * kWishThreads + tid,
             (nc - 1) * kWishThreads);
  }
  cluster_sync();
  if (__ldcg(gok) == 0.0) return;

  // ---- 2
  if (cta != 0) copy_in(M, gL, np);
  copy_in(U, gA, np);
  for (int k = tid; k < K; k += kWishThreads) s_rr[k] = rsqrt(cta == 0 ? s_dg[k] : __ldcg(gD + k));
  // for later: z / sqrt(beta*) and mu*, by the threads with the least to do here
  const double bstar = a.beta0 + n;
  for (int k = kWishThreads - 1 - tid; k < K; k += kWishThreads) {
    s_z[k] = (double)normal_at_f32(key, 0u, t, stream_word(kStreamHyperMu, a.side), (uint32_t)k) / sqrt(bstar);
    s_mus[k] = (a.beta0 * a.mu0[k] + n * a.xbar[k]) / bstar;
  }
  __syncthreads();
  for (int j = j0; j < K; j += 8 * nc) {
    const int len = K - j;
    switch ((len + 31) >> 5) {
      case 1: unit_solve<1>(M, K, j, s_rr, cbuf, lane); break;
      case 2: unit_solve<2>(M, K, j, s_rr, cbuf, lane); break;
      case 3: unit_solve<3>(M, K, j, s_rr, cbuf, lane); break;
      default: unit_solve<4>(M, K, j, s_rr, cbuf, lane);
    }
    const int i = len - 1;
    __syncwarp();
    // row i of B: sum over m = l .. i of C[i][m] A[m][l], four chains
#pragma unroll
    for (int g = 0; g < kNpl; ++g) {
      const int l = lane + 32 * g;
      if (32 * g > i) break;
      double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
      for (int m0 = 32 * g; m0 <= i; m0 += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int m = m0 + u;
          if (m <= i && l <= m) s[u] = fma(cbuf[m], U[m * (m + 1) / 2 + l], s[u]);
        }
      }
      if (l <= i) {
        const double v = (s[0] + s[1]) + (s[2] + s[3]);
        gB[i * (i + 1) / 2 + l] = v;
        a.lchol[i * (i + 1) / 2 + l] = (float)v;
      }
    }
    __syncwarp();
  }
  cluster_sync();

  // ---- 3
  double* B = M;
  copy_in(B, gB, np);
  __syncthreads();
  // w = B^T mu* + z / sqrt(beta*), a warp per eighth of the rows
  {
    double s[kNpl];
#pragma unroll
    for (int g = 0; g < kNpl; ++g) s[g] = 0.0;
    for (int i = warp; i < K; i += kWishWarps) {
      const double mi = s_mus[i];
#pragma unroll
      for (int g = 0; g < kNpl; ++g)
        if (lane + 32 * g <= i) s[g] = fma(B[i * (i + 1) / 2 + lane + 32 * g], mi, s[g]);
    }
#pragma unroll
    for (int g = 0; g < kNpl; ++g)
      if (lane + 32 * g < K) s_part[warp][lane + 32 * g] = s[g];
  }
  const bool last = cta == nc - 1;
  if (last)
    for (int k = tid; k < K; k += kWishThreads) s_rr[k] = 1.0 / B[k * (k + 1) / 2 + k];
  __syncthreads();
  for (int k = tid; k < K; k += kWishThreads) {
    double s = s_z[k];
#pragma unroll
    for (int q = 0; q < kWishWarps; ++q) s += s_part[q][k];
    s_w[k] = s;
  }
  if (last)  // the rows of B over their diagonals, for mu
    for (int i = warp; i < K; i += kWishWarps)
      for (int k = lane; k < i; k += 32) U[i * (i + 1) / 2 + k] = B[i * (i + 1) / 2 + k] * s_rr[i];
  __syncthreads();
  // mu: B^T x = z / sqrt(beta*) from the bottom by the last warp, lane l holding entries
  // l + 32 m of x B_ii, so that the chain is one shuffle and one multiply-add
  if (last && warp == kWishWarps - 1) {
    double z[kNpl];
#pragma unroll
    for (int m = 0; m < kNpl; ++m) z[m] = lane + 32 * m < K ? s_z[lane + 32 * m] : 0.0;
#pragma unroll
    for (int mi = kNpl - 1; mi >= 0; --mi) {
      if (32 * mi >= K) continue;
#pragma unroll 4
      for (int c = min(31, K - 1 - 32 * mi); c >= 0; --c) {
        const int i = 32 * mi + c;
        const double* bi = U + i * (i + 1) / 2 + lane;
        const double zi = __shfl_sync(kFull, z[mi], c);
        if (lane < c) z[mi] = fma(-bi[32 * mi], zi, z[mi]);
#pragma unroll
        for (int m = 0; m < mi; ++m) z[m] = fma(-bi[32 * m], zi, z[m]);
      }
    }
#pragma unroll
    for (int m = 0; m < kNpl; ++m) {
      const int k = lane + 32 * m;
      if (k < K) a.mu[k] = fma(z[m], s_rr[k], s_mus[k]);
    }
    if (lane == 0) a.lamaug[K * KA + K] = 0.f;
  }
  for (int wj = j0; wj < K; wj += 8 * nc) {
    const int i = K - 1 - wj;
    const double* bi = B + i * (i + 1) / 2;
    double b0 = 0.0;
#pragma unroll
    for (int g = 0; g < kNpl; ++g) {
      const int j = lane + 32 * g;
      if (32 * g > i) break;
      if (j <= i) b0 = fma(bi[j], s_w[j], b0);
      const double* bj = B + j * (j + 1) / 2;
      const int kn = min(i, 32 * g + 31);
      double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
      for (int k0 = 0; k0 <= kn; k0 += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = k0 + u;
          if (k <= j && j <= i) s[u] = fma(bi[k], bj[k], s[u]);
        }
      }
      if (j <= i) {
        const double v = (s[0] + s[1]) + (s[2] + s[3]);
        a.lam[i * K + j] = v;
        a.lam[j * K + i] = v;
        a.lamaug[i * KA + j] = (float)v;
        a.lamaug[j * KA + i] = (float)v;
      }
    }
    b0 = warp_sum(b0);
    if (lane == 0) {
      a.lamaug[K * KA + i] = (float)b0;
      a.lamaug[i * KA + K] = (float)b0;
    }
  }
}

}  // namespace

namespace {

// The launch of kern on one cluster of `ctas` CTAs.
template <typename... P>
int cluster_config(void (*kern)(P...), int K, int ctas, cudaStream_t st, cudaLaunchConfig_t* cfg,
                   cudaLaunchAttribute* at) {
  BPMF_TRY(allow_smem(kern, wish_smem(kMaxK)));
  BPMF_CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  *cfg = {};
  cfg->gridDim = dim3((unsigned)ctas);
  cfg->blockDim = dim3(kWishThreads);
  cfg->dynamicSmemBytes = wish_smem(K);
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = cfg->gridDim.x;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  return BPMF_OK;
}

template <typename... P, typename... A>
int launch_cluster(void (*kern)(P...), int K, int ctas, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  BPMF_TRY(cluster_config(kern, K, ctas, st, &cfg, &at));
  BPMF_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, args...));
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

}  // namespace

int wish_cluster(int K, int* ctas) {
  for (int n = wish_ctas(K); n >= 2; n /= 2) {  // a draw needs two: the factorisation's and Bartlett's
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    int fit = 0;
    BPMF_TRY(cluster_config(wishart_draw, K, n, nullptr, &cfg, &at));
    if (cudaOccupancyMaxActiveClusters(&fit, wishart_draw, &cfg) == cudaSuccess && fit > 0) {
      *ctas = n;
      return BPMF_OK;
    }
    cudaGetLastError();
  }
  set_error("wishart: the device holds no cluster of two CTAs for K = %d", K);
  return BPMF_ECUDA;
}

int launch_wishart(const HyperArgs& a, int ctas, cudaStream_t st, int64_t* launches) {
  BPMF_TRY(launch_cluster(wishart_draw, a.K, ctas, st, a));
  if (launches) *launches += 1;
  return BPMF_OK;
}

int launch_spd_inverse_f64(const double* A, double* Ainv, int K, int ctas, double* scratch, int* status,
                           cudaStream_t st) {
  return launch_cluster(spd_inverse, K, ctas, st, A, Ainv, K, scratch, status);
}

int launch_check_spd_f64(const double* A, int K, int* status, float* lout, cudaStream_t st) {
  const int smem = wish_smem(K);
  BPMF_TRY(allow_smem(spd_check, wish_smem(kMaxK)));
  spd_check<<<1, kWishThreads, smem, st>>>(A, K, status, lout);
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

}  // namespace gb
