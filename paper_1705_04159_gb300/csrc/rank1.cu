// rank1.cu -- rows of small degree from chol(Lambda_s) and d rank-one terms.
//
// A row with d ratings has Lambda* = Lambda_s + sum_t x_t x_t^T, x_t =
// sqrt(alpha) v_t (t = 0 .. d-1).  L_s = chol(Lambda_s) is a by-product of the
// hyper draw and the same for every row of the side; with w_t = L_s^-1 x_t,
//   Lambda* = L_s (I + sum_t w_t w_t^T) L_s^T,
// and the lower Cholesky factor of I + sum_t w_t w_t^T is the product
// N = M_0 M_1 ... M_{d-1} of the factors M_s = chol(I + p_s p_s^T) with
// p_s = (M_0 ... M_{s-1})^-1 w_s: each factor adds one term, as
// N_s N_s^T = N_{s-1} (I + p_s p_s^T) N_{s-1}^T = N_{s-1} N_{s-1}^T + w_s w_s^T.
// Products of lower-triangular factors with positive diagonals are again
// such factors, so L* = L_s N is the unique factor a direct Cholesky
// factorisation of Lambda* gives: the draws are the same up to rounding.
//
// chol(I + p p^T) is diagonal plus semiseparable.  With the prefix sums
// B_i = 1 + sum_{k<i} p_k^2 and B'_i = B_i + p_i^2 (one step of the textbook
// rank-one update of the identity, unrolled),
//   M_ii = sqrt(B'_i / B_i),   M_ik = p_i p_k / sqrt(B_k B'_k)  (i > k),
// and with rho_i = sqrt(B_i / B'_i) and gamma_i = p_i / sqrt(B_i B'_i) its
// inverse and inverse transpose act on a vector through one prefix or one
// suffix sum:
//   (M^-1 y)_i = rho_i y_i - gamma_i sum_{k<i} p_k y_k,
//   (M^-T w)_i = rho_i w_i - p_i sum_{k>i} gamma_k w_k.
// So, with c = L_s^-1 b,
//   y = M_{d-1}^-1 ... M_0^-1 c = L*^-1 b,
//   u = L_s^-T M_0^-T ... M_{d-1}^-T (y + z) = L*^-T (y + z):
// products of L_s^-1 with the x_t and b, one of L_s^-T, and O(d^2)
// warp-wide scans -- instead of d K column steps, each a dependent square root
// and division, of successive rank-one updates of the factor.  This is the
// cheaper kernel for rows with few ratings of paper Sec. III (Fig. 2).  The
// factor's diagonal is L*_ii = (L_s)_ii prod_s M_s,ii, so the pivot rule of
// the other row kernels (L*_ii^2 against Lambda*_ii) still decides which rows
// go to the FP64 redo.
//
// The w_t do not depend on the row but through the neighbour j: w_t = L_s^-1
// sqrt(alpha) v_j, and c = L_s^-1 b0 + sqrt(alpha) sum_t r_t w_t.  Where the bin's
// ratings outnumber the other side's rows, lower_rows forms them for every j once
// per sweep (PRE), and a row is left with the scans and the product with L_s^-T.  The
// other form takes the same products row by row and then the same steps, so a
// row's draw is bitwise the same in both: which one runs depends on the other
// rows of the bin and on the memory at hand.
//
// Layout.  linv_columns writes T = (L_s^-1)^T, KP x LD floats (KP = K rounded
// up to 32, LD = KP + 4, zero outside the triangle), once per sweep, in FP64
// arithmetic from the packed FP32 factor.  Each CTA keeps T in shared memory;
// its warps take groups of kR1Rows rows in turn, one row after the other up to
// the last product, which they share (a value of T read once serves them all).
// Lane l owns elements l + 32 m.  T[k][i] at k LD + i: the forward product
// reads T[k][l + 32 m] (consecutive in l) one float at a time, and the
// transposed one reads T[l + 32 m][k .. k + 3] as one 16-byte load (rows
// 16-byte aligned, LD = 4 mod 32, so eight lanes of a load phase fall on eight
// different groups of four banks).  Per warp: d + 1 vectors (w_t and p_t; the
// last c, then y), the d prefix sums B'_s (the backward pass recomputes rho and
// gamma from them) and kR1Rows vectors of normals, then of right-hand sides.
//
// What bounds it: issue.  480,000 rows of 1.9 ratings on average, K = 64,
// 5,800 rows on the other side: 951 -> 515 us.
#include <cuda_runtime.h>
#include <float.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "rows.cuh"

namespace gb {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kR1MaxWarps = 8;
constexpr int kR1Rows = 4;  // rows of a group (they share the product with L_s^-T)
constexpr size_t kR1Smem = 200 * 1024;  // dynamic shared memory of a CTA, at most

__device__ __forceinline__ int tri(int i) { return (i * (i + 1)) >> 1; }

__device__ __forceinline__ float comp(const float4& v, int e) {
  return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w;
}

// T = (L_s^-1)^T from the packed factor (row i at i (i + 1) / 2), one warp per
// row k of T, i.e. column k of L_s^-1: L_s t = e_k by column-oriented forward
// substitution in FP64 -- lane l holds t_i for i = l + 32 m; at step j the
// owner of row j scales t_j by 1 / L_jj (computed before the loop) and
// broadcasts it, and every lane subtracts L_ij t_j from its rows, so a step is
// one shuffle and one multiply-add, with no reduction.  The block of L from
// row and column k on is first brought to shared memory in FP64, square with
// zeros above the diagonal (rows at or above the step then subtract nothing)
// and an odd row stride: no step waits for a global load, converts or branches.
int linv_smem(int K) { return (int)sizeof(double) * K * (K | 1); }

template <int NPL>
__global__ void __launch_bounds__(32) linv_columns(const float* __restrict__ lchol, int K,
                                                   float* __restrict__ T) {
  constexpr int KP = 32 * NPL, LD = KP + 4;
  extern __shared__ double s_l[];
  const int k = blockIdx.x, lane = threadIdx.x, n = K - k;
  float* out = T + (int64_t)k * LD;
  for (int i = lane; i < LD; i += 32)
    if (i < k || i >= K) out[i] = 0.f;
  if (n <= 0) return;
  const int ld = n | 1;
  for (int i = 0; i < n; ++i) {
    const float* row = lchol + tri(k + i) + k;
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      const int j = lane + 32 * m;
      if (j < n) s_l[i * ld + j] = j <= i ? (double)__ldg(row + j) : 0.0;
    }
  }
  __syncwarp();
  // local row q = i - k
  double t[NPL], rdiag[NPL];
#pragma unroll
  for (int m = 0; m < NPL; ++m) {
    const int q = lane + 32 * m;
    t[m] = q == 0 ? 1.0 : 0.0;
    rdiag[m] = q < n ? 1.0 / s_l[q * ld + q] : 0.0;
  }
#pragma unroll
  for (int mb = 0; mb < NPL; ++mb) {
    for (int jj = 0; jj < 32; ++jj) {
      const int j = 32 * mb + jj;
      if (j >= n) break;
      const double tj = __shfl_sync(kFull, t[mb] * rdiag[mb], jj);
      if (lane == jj) out[k + j] = (float)tj;
#pragma unroll
      for (int m = mb; m < NPL; ++m) {
        const int q = min(lane + 32 * m, n - 1);
        t[m] = fma(-s_l[q * ld + j], tj, t[m]);
      }
    }
  }
}

// Inclusive (v) and exclusive (ex) prefix sums over the elements l + 32 m of G
// vectors at once: a 32-lane scan per block, then the carries of the blocks
// before.  The exclusive sums are shifted inclusive ones, never inclusive
// minus the element (that subtraction would cancel when one term dominates).
template <int G, int NPL>
__device__ __forceinline__ void scan_prefix(float (&v)[G][NPL], float (&ex)[G][NPL], int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int m = 0; m < NPL; ++m) {
        const float t = __shfl_up_sync(kFull, v[g][m], o);
        if (lane >= o) v[g][m] += t;
      }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    float carry = 0.f;
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      const float tot = __shfl_sync(kFull, v[g][m], 31);
      const float up = __shfl_up_sync(kFull, v[g][m], 1);
      ex[g][m] = lane == 0 ? carry : up + carry;
      v[g][m] += carry;
      carry += tot;
    }
  }
}

// Exclusive suffix sums (sum over k > i) over the elements l + 32 m.
template <int NPL>
__device__ __forceinline__ void scan_suffix(float (&v)[NPL], float (&ex)[NPL], int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      const float t = __shfl_down_sync(kFull, v[m], o);
      if (lane + o < 32) v[m] += t;
    }
  }
  float carry = 0.f;
#pragma unroll
  for (int m = NPL - 1; m >= 0; --m) {
    const float tot = __shfl_sync(kFull, v[m], 0);
    const float dn = __shfl_down_sync(kFull, v[m], 1);
    ex[m] = lane == 31 ? carry : dn + carry;
    carry += tot;
  }
}

// v_g <- L_s^-1 v_g for G vectors of KP floats at v (in place): lane l sums
// T[k][l + 32 m] v_g[k] over k, the v_g[k] read four at a time as broadcasts.
// Rows of block m need k < 32 (m + 1) only (L_s^-1 is lower triangular).
template <int NPL, int G>
__device__ __forceinline__ void lower_times(const float* T, float* v, int K, int lane) {
  constexpr int KP = 32 * NPL, LD = KP + 4;
  float acc[G][NPL];
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int m = 0; m < NPL; ++m) acc[g][m] = 0.f;
#pragma unroll
  for (int kc = 0; kc < NPL; ++kc) {
#pragma unroll 2
    for (int k4 = 0; k4 < 32; k4 += 4) {
      const int k = 32 * kc + k4;
      if (k >= K) break;  // uniform; rows k .. k+3 of T exist and are zero past K
      float4 xv[G];
#pragma unroll
      for (int g = 0; g < G; ++g) xv[g] = *reinterpret_cast<const float4*>(v + g * KP + k);
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int m = kc; m < NPL; ++m) {
          const float t = T[(k + e) * LD + lane + 32 * m];
#pragma unroll
          for (int g = 0; g < G; ++g) acc[g][m] = fmaf(t, comp(xv[g], e), acc[g][m]);
        }
    }
  }
  __syncwarp();  // every lane has read the inputs
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int m = 0; m < NPL; ++m) v[g * KP + lane + 32 * m] = acc[g][m];
  __syncwarp();
}

// The factor of p = v_0 (its rho and B', the latter to Bp) and v_g <- M^-1 v_g
// for the G vectors v_1 .. v_G after it; the prefix sums of p^2 and of the
// p y_g do not depend on one another, so they are scanned together.  Each lane
// reads and writes its own elements.
template <int NPL, int G>
__device__ __forceinline__ void factor_step(float* v, float* Bp, float (&pr)[NPL], int lane) {
  constexpr int KP = 32 * NPL;
  float p[NPL], y[G][NPL], s[G + 1][NPL], ex[G + 1][NPL];
#pragma unroll
  for (int m = 0; m < NPL; ++m) {
    p[m] = v[lane + 32 * m];
    s[G][m] = p[m] * p[m];
  }
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      y[g][m] = v[(g + 1) * KP + lane + 32 * m];
      s[g][m] = p[m] * y[g][m];
    }
  scan_prefix<G + 1, NPL>(s, ex, lane);
#pragma unroll
  for (int m = 0; m < NPL; ++m) {
    const float Bi = 1.f + s[G][m], Be = 1.f + ex[G][m];
    const float r1 = rsqrtf(Be), r2 = rsqrtf(Bi);
    const float rho = Be * r1 * r2, gam = p[m] * r1 * r2;
    Bp[lane + 32 * m] = Bi;
    pr[m] *= rho * rho;
#pragma unroll
    for (int g = 0; g < G; ++g)
      v[(g + 1) * KP + lane + 32 * m] = fmaf(rho, y[g][m], -gam * ex[g][m]);
  }
}

// M^-1 on n vectors at v, given p and its rho and gamma (those past the first
// few of a row with many ratings)
template <int NPL>
__device__ __forceinline__ void factor_rest(float* v, int n, const float* p, const float* Bp, int lane) {
  constexpr int KP = 32 * NPL;
  float pv[NPL], rho[NPL], gam[NPL];
#pragma unroll
  for (int m = 0; m < NPL; ++m) {
    const int i = lane + 32 * m;
    pv[m] = p[i];
    const float Bi = Bp[i];
    const float Be = i == 0 ? 1.f : Bp[i - 1];
    const float r1 = rsqrtf(Be), r2 = rsqrtf(Bi);
    rho[m] = Be * r1 * r2;
    gam[m] = pv[m] * r1 * r2;
  }
  for (; n > 0; --n, v += KP) {
    float y[NPL], s[1][NPL], ex[1][NPL];
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      y[m] = v[lane + 32 * m];
      s[0][m] = pv[m] * y[m];
    }
    scan_prefix<1, NPL>(s, ex, lane);
#pragma unroll
    for (int m = 0; m < NPL; ++m) v[lane + 32 * m] = fmaf(rho[m], y[m], -gam[m] * ex[0][m]);
  }
}

template <int NPL>
__device__ __forceinline__ void lower_times_n(const float* T, float* v, int n, int K, int lane) {
  constexpr int KP = 32 * NPL;
  for (int g0 = 0; g0 < n; g0 += 4) {
    switch (min(4, n - g0)) {
      case 1: lower_times<NPL, 1>(T, v + g0 * KP, K, lane); break;
      case 2: lower_times<NPL, 2>(T, v + g0 * KP, K, lane); break;
      case 3: lower_times<NPL, 3>(T, v + g0 * KP, K, lane); break;
      default: lower_times<NPL, 4>(T, v + g0 * KP, K, lane); break;
    }
  }
}

// floats of shared memory per warp for rows of degree <= D
__host__ __device__ __forceinline__ int r1_warp_floats(int D, int KP) {
  return (2 * D + 1 + kR1Rows) * KP;
}

// W row j = L_s^-1 (sqrt(alpha) row j of V) for j < n, and row n = L_s^-1 b0: KP
// floats per row, zero past K.  A warp takes four rows at a time.
template <int NPL>
__global__ void __launch_bounds__(32 * kR1MaxWarps)
    lower_rows(const float* __restrict__ V, int64_t n, int K, float alpha, const float* __restrict__ b0,
               const float* __restrict__ Tg, float* __restrict__ W) {
  constexpr int KP = 32 * NPL, LD = KP + 4;
  extern __shared__ __align__(16) float r1s[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < KP * LD / 4; e += blockDim.x)
    reinterpret_cast<float4*>(r1s)[e] = __ldg(reinterpret_cast<const float4*>(Tg) + e);
  __syncthreads();
  float* vec = r1s + KP * LD + warp * 4 * KP;
  const float sa = sqrtf(alpha);
  const int64_t stride = (int64_t)gridDim.x * (blockDim.x >> 5) * 4;
  for (int64_t j0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 4; j0 <= n; j0 += stride) {
    __syncwarp();
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float* v = j0 + g < n ? V + (j0 + g) * K : b0;
#pragma unroll
      for (int m = 0; m < NPL; ++m) {
        const int i = lane + 32 * m;
        const float x = j0 + g <= n && i < K ? __ldg(v + i) : 0.f;
        vec[g * KP + i] = j0 + g < n ? sa * x : x;
      }
    }
    __syncwarp();
    lower_times<NPL, 4>(r1s, vec, K, lane);
#pragma unroll
    for (int g = 0; g < 4; ++g)
      if (j0 + g <= n) {
#pragma unroll
        for (int m = 0; m < NPL; ++m) W[(j0 + g) * KP + lane + 32 * m] = vec[g * KP + lane + 32 * m];
      }
  }
}

// PRE: W holds sqrt(alpha) L_s^-1 of the other side's rows and L_s^-1 b0 (lower_rows)
template <int NPL, bool PRE>
__global__ void __launch_bounds__(32 * kR1MaxWarps)
    row_rank1(const SweepArgs a, const float* __restrict__ lchol, const float* __restrict__ Tg,
              const float* __restrict__ W, int D, int warps) {
  constexpr int KP = 32 * NPL, LD = KP + 4;
  extern __shared__ __align__(16) float r1s[];
  const int K = a.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* T = r1s;
  {
    const float4* src = reinterpret_cast<const float4*>(Tg);
    float4* dst = reinterpret_cast<float4*>(T);
    for (int e = threadIdx.x; e < KP * LD / 4; e += blockDim.x) dst[e] = __ldg(src + e);
  }
  __syncthreads();  // the only block-wide barrier; warps go their own way after it
  float* vec = T + KP * LD + warp * r1_warp_floats(D, KP);
  float* Bp = vec + (D + 1) * KP;
  float* zb = Bp + D * KP;  // [kR1Rows][KP]
  // per-element constants: L_s^-1 b0 (b0 = Lambda_s mu_s, the bordered hyper
  // matrix's last row), the diagonal of Lambda_s and that of L_s squared
  float bs[NPL], ds[NPL], ls2[NPL];
  if (!PRE) {
#pragma unroll
    for (int m = 0; m < NPL; ++m) {
      const int i = lane + 32 * m;
      vec[i] = i < K ? __ldg(a.lamaug + (int64_t)K * (K + 1) + i) : 0.f;
    }
    __syncwarp();
    lower_times<NPL, 1>(T, vec, K, lane);
  }
#pragma unroll
  for (int m = 0; m < NPL; ++m) {
    const int i = lane + 32 * m;
    bs[m] = i < K ? (PRE ? __ldg(W + a.n_other * KP + i) : vec[i]) : 0.f;
    ds[m] = i < K ? __ldg(a.lamaug + (int64_t)i * (K + 1) + i) : 0.f;
    const float l = i < K ? __ldg(lchol + tri(i) + i) : 1.f;
    ls2[m] = l * l;
  }
  const float sa = sqrtf(a.alpha);
  const uint32_t tw = *a.tp;
  const int64_t stride = (int64_t)gridDim.x * warps * kR1Rows;
  for (int64_t s0 = a.row_begin + ((int64_t)blockIdx.x * warps + warp) * kR1Rows; s0 < a.row_end;
       s0 += stride) {
    __syncwarp();  // the previous group's reads of the warp's buffers are done
    const int nrow = (int)min((int64_t)kR1Rows, a.row_end - s0);
    // lane r: row r of the group, its first rating and its degree
    int grow = -1, gdeg = 0;
    int64_t gp0 = 0;
    if (lane < nrow) {
      grow = a.rows ? a.rows[s0 + lane] : (int)(s0 + lane);
      gp0 = a.ptr[grow];
      gdeg = (int)(a.ptr[grow + 1] - gp0);
    }
    // normals of the group's rows, a lane per four
    for (int e = lane; e < kR1Rows * KP / 4; e += 32) {
      const int r = e / (KP / 4), q = e - r * (KP / 4);
      const int row = __shfl_sync(kFull, grow, r);
      float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      if (4 * q < K && r < nrow) {
        z = normal4_f32(philox(make_uint4((uint32_t)row, tw, (uint32_t)q, a.sw), a.key));
        if (4 * q + 1 >= K) z.y = 0.f;
        if (4 * q + 2 >= K) z.z = 0.f;
        if (4 * q + 3 >= K) z.w = 0.f;
      }
      *reinterpret_cast<float4*>(zb + 4 * e) = z;
    }
    __syncwarp();
    unsigned drop = 0;  // rows of the group left to the FP64 redo
    for (int r = 0; r < nrow; ++r) {
      const int d = __shfl_sync(kFull, gdeg, r);
      const int64_t p0 = __shfl_sync(kFull, gp0, r);
      if (d > D) {  // not in this bin's degree range
        drop |= 1u << r;
        continue;
      }
      // Lambda*_ii, then w_t = L_s^-1 x_t and c = L_s^-1 b0 + sum_t sqrt(alpha)
      // r_t w_t: the same operations in the same order whether the w_t were
      // formed before or are formed here
      float b[NPL], d0[NPL];
#pragma unroll
      for (int m = 0; m < NPL; ++m) {
        b[m] = bs[m];
        d0[m] = ds[m];
      }
      // the ratings of the second pass, a lane each (d <= 32)
      const float rl = !PRE && lane < d ? sa * __ldg(a.val + p0 + lane) : 0.f;
      for (int t = 0; t < d; ++t) {
        const int32_t j = __ldg(a.idx + p0 + t);
        const float sr = PRE ? sa * __ldg(a.val + p0 + t) : 0.f;
        const float* vj = a.Vo + (int64_t)j * K;
        const float* wj = PRE ? W + (int64_t)j * KP : nullptr;
#pragma unroll
        for (int m = 0; m < NPL; ++m) {
          const int i = lane + 32 * m;
          const float v = i < K ? __ldg(vj + i) : 0.f;
          const float x = sa * v;
          d0[m] = fmaf(x, x, d0[m]);
          const float w = PRE ? __ldg(wj + i) : x;
          vec[t * KP + i] = w;
          if (PRE) b[m] = fmaf(sr, w, b[m]);
        }
      }
      if (!PRE) {
        __syncwarp();
        lower_times_n<NPL>(T, vec, d, K, lane);
        for (int t = 0; t < d; ++t) {
          const float sr = __shfl_sync(kFull, rl, t);
#pragma unroll
          for (int m = 0; m < NPL; ++m) b[m] = fmaf(sr, vec[t * KP + lane + 32 * m], b[m]);
        }
      }
#pragma unroll
      for (int m = 0; m < NPL; ++m) vec[d * KP + lane + 32 * m] = b[m];
      // the factors: p_s, then M_s^-1 applied to w_{s+1} .. w_{d-1} and to c
      float pr[NPL];  // prod_s rho_s^2 = (L_s)_ii^2 / L*_ii^2
#pragma unroll
      for (int m = 0; m < NPL; ++m) pr[m] = 1.f;
      for (int s = 0; s < d; ++s) {
        float* v = vec + s * KP;
        float* B = Bp + s * KP;
        const int n = d - s;
        switch (n) {
          case 1: factor_step<NPL, 1>(v, B, pr, lane); break;
          case 2: factor_step<NPL, 2>(v, B, pr, lane); break;
          default: factor_step<NPL, 3>(v, B, pr, lane); break;
        }
        if (n > 3) {
          __syncwarp();  // B' of the lanes before
          factor_rest<NPL>(v + 4 * KP, n - 3, v, B, lane);
        }
      }
      __syncwarp();  // B' of other lanes is read below
      // w = y + z, then M_{d-1}^-T .. M_0^-T
      float* zr = zb + r * KP;
      float w[NPL];
#pragma unroll
      for (int m = 0; m < NPL; ++m) w[m] = vec[d * KP + lane + 32 * m] + zr[lane + 32 * m];
      for (int s = d - 1; s >= 0; --s) {
        float t[NPL], ex[NPL], p[NPL], rho[NPL];
#pragma unroll
        for (int m = 0; m < NPL; ++m) {
          const int i = lane + 32 * m;
          p[m] = vec[s * KP + i];
          const float Bi = Bp[s * KP + i];
          const float Be = i == 0 ? 1.f : Bp[s * KP + i - 1];
          const float r1 = rsqrtf(Be), r2 = rsqrtf(Bi);
          rho[m] = Be * r1 * r2;
          t[m] = p[m] * r1 * r2 * w[m];  // gamma_i w_i
        }
        scan_suffix<NPL>(t, ex, lane);
#pragma unroll
        for (int m = 0; m < NPL; ++m) w[m] = fmaf(rho[m], w[m], -p[m] * ex[m]);
      }
#pragma unroll
      for (int m = 0; m < NPL; ++m) zr[lane + 32 * m] = w[m];
      // pivot rule: L*_ii^2 = (L_s)_ii^2 / pr_i against pivot_rel Lambda*_ii
      bool bad = false;
#pragma unroll
      for (int m = 0; m < NPL; ++m) {
        const int i = lane + 32 * m;
        if (i < K && !(ls2[m] > pr[m] * fmaxf(a.pivot_rel * d0[m], FLT_MIN))) bad = true;
      }
      if (__any_sync(kFull, bad)) drop |= 1u << r;
      __syncwarp();  // the row's buffers are rewritten by the next row
    }
    // u = L_s^-T w: lane l sums T[l + 32 m][k] w_k over k >= 32 m, for all rows
    float u[kR1Rows][NPL];
#pragma unroll
    for (int r = 0; r < kR1Rows; ++r)
#pragma unroll
      for (int m = 0; m < NPL; ++m) u[r][m] = 0.f;
#pragma unroll
    for (int kc = 0; kc < NPL; ++kc) {
#pragma unroll 2
      for (int k4 = 0; k4 < 32; k4 += 4) {
        const int k = 32 * kc + k4;
        if (k >= K) break;
        float4 wv[kR1Rows];
#pragma unroll
        for (int r = 0; r < kR1Rows; ++r) wv[r] = *reinterpret_cast<const float4*>(zb + r * KP + k);
#pragma unroll
        for (int m = 0; m <= kc; ++m) {
          const float4 t4 = *reinterpret_cast<const float4*>(T + (lane + 32 * m) * LD + k);
#pragma unroll
          for (int r = 0; r < kR1Rows; ++r) {
            u[r][m] = fmaf(t4.x, wv[r].x, u[r][m]);
            u[r][m] = fmaf(t4.y, wv[r].y, u[r][m]);
            u[r][m] = fmaf(t4.z, wv[r].z, u[r][m]);
            u[r][m] = fmaf(t4.w, wv[r].w, u[r][m]);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kR1Rows; ++r) {
      const int row = __shfl_sync(kFull, grow, r);
      if (r < nrow && !(drop >> r & 1u)) {
        float* out = a.X + (int64_t)row * K;
#pragma unroll
        for (int m = 0; m < NPL; ++m) {
          const int i = lane + 32 * m;
          if (i < K) {
            out[i] = u[r][m];
            write_shadow(a, row, i, u[r][m]);
          }
        }
      }
    }
    if (lane < nrow && (drop >> lane & 1u)) a.flag_rows[atomicAdd(a.flag_count, 1)] = grow;
  }
}

// CTAs of `kern` that fill the device, at most `need`
template <typename F>
int r1_grid(F kern, int threads, size_t smem, int64_t need, unsigned* grid) {
  BPMF_TRY(allow_smem(kern, kR1Smem));
  int dev = 0, sms = 1, occ = 1;
  BPMF_CUDA_CHECK(cudaGetDevice(&dev));
  BPMF_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  BPMF_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem));
  *grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sms * std::max(occ, 1)));
  return BPMF_OK;
}

template <int NPL>
int launch_r1(const SweepArgs& a, const float* lchol, float* T, float* W, int D, cudaStream_t st) {
  constexpr int KP = 32 * NPL, LD = KP + 4;
  BPMF_TRY(allow_smem(linv_columns<NPL>, linv_smem(KP)));
  linv_columns<NPL><<<KP, 32, linv_smem(a.K), st>>>(lchol, a.K, T);
  BPMF_CUDA_CHECK(cudaGetLastError());
  const size_t tbytes = sizeof(float) * KP * LD;
  unsigned grid = 1;
  if (W != nullptr) {
    const size_t smem = tbytes + sizeof(float) * kR1MaxWarps * 4 * KP;
    BPMF_TRY(r1_grid(lower_rows<NPL>, 32 * kR1MaxWarps, smem,
                     (a.n_other + 4 * kR1MaxWarps) / (4 * kR1MaxWarps), &grid));
    lower_rows<NPL><<<grid, 32 * kR1MaxWarps, smem, st>>>(a.Vo, a.n_other, a.K, a.alpha,
                                                          a.lamaug + (int64_t)a.K * (a.K + 1), T, W);
    BPMF_CUDA_CHECK(cudaGetLastError());
  }
  const size_t per = sizeof(float) * (size_t)r1_warp_floats(D, KP);
  int w = kR1MaxWarps;
  while (w > 1 && tbytes + w * per > kR1Smem) --w;
  const size_t smem = tbytes + w * per;
  const int64_t n = a.row_end - a.row_begin, per_cta = (int64_t)w * kR1Rows;
  auto kern = W != nullptr ? row_rank1<NPL, true> : row_rank1<NPL, false>;
  BPMF_TRY(r1_grid(kern, 32 * w, smem, (n + per_cta - 1) / per_cta, &grid));
  kern<<<grid, 32 * w, smem, st>>>(a, lchol, T, W, D, w);
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

}  // namespace

int64_t rank1_pre_floats(int K, int64_t n_other, int64_t rows, int64_t ratings) {
  // one product of L_s^-1 per row of the other side against one per row and
  // rating of the bin, the former in batches of four.  100,000 rows, K = 64, the
  // products formed once against row by row: two ratings a row, 6, 3, 2 and 1
  // times as many rows and ratings as rows on the other side: 343 / 417,
  // 367 / 423, 382 / 426, 439 / 440 us; six ratings a row, 3.5 and 2 times:
  // 936 / 956, 1014 / 975 us (K = 100: ahead from 1 times on; K = 16: even at 3).
  if (ratings == 0 || rows + ratings < 3 * n_other) return 0;
  return (n_other + 1) * ((K + 31) & ~31);
}

int launch_rows_rank1(const SweepArgs& a, const float* lchol, float* linvT, float* pre,
                      int max_degree, cudaStream_t st, int64_t* launches) {
  if (a.row_end <= a.row_begin) return BPMF_OK;
  if (max_degree < 0 || max_degree > kTinyDegreeMax) return BPMF_EINVAL;
  *launches += pre != nullptr ? 3 : 2;
  if (a.K <= 32) return launch_r1<1>(a, lchol, linvT, pre, max_degree, st);
  if (a.K <= 64) return launch_r1<2>(a, lchol, linvT, pre, max_degree, st);
  if (a.K <= 96) return launch_r1<3>(a, lchol, linvT, pre, max_degree, st);
  return launch_r1<4>(a, lchol, linvT, pre, max_degree, st);
}

}  // namespace gb
