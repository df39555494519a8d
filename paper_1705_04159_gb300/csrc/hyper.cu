// hyper.cu -- hyperparameter draw of one side (Algorithm 1, "sample
// hyper-parameters movies based on V" / "users based on U").
//
// BPMF's hyperprior (paper Sec. II) is Normal-Wishart: Lambda ~ W(W0, nu0),
// mu | Lambda ~ N(mu0, (beta0 Lambda)^-1).  Given the n factor rows x_i of a
// side, with mean xbar and centred scatter S = sum (x_i - xbar)(x_i - xbar)^T,
// the posterior is Normal-Wishart with
//   beta* = beta0 + n, nu* = nu0 + n, mu* = (beta0 mu0 + n xbar) / (beta0 + n),
//   W*^-1 = W0^-1 + S + beta0 n / (beta0 + n) (mu0 - xbar)(mu0 - xbar)^T.
// Lambda is drawn by Bartlett's decomposition (C = chol(W*), A lower with
// A_kk^2 ~ chi^2(nu* - k), A_kl ~ N(0,1); Lambda = (C A)(C A)^T) and
// mu = mu* + chol(beta* Lambda)^-T z.
//
// Device work: (1) column sums of the factor rows with FP32 partials per block
// combined in FP64; (2) the centred scatter, a K x K Gram over all rows with
// FP32 register tiles per block, combined in FP64 in a fixed block order;
// (3) the FP64 draw, O(K^3) and independent of the row count (wishart.cu).
#include <cuda_runtime.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "hyper.cuh"

namespace gb {
namespace {

constexpr int kRedThreads = 256;

// ---- (1) column sums: part[b * K + k] = sum over block b's rows of x[., k].
// Thread t takes column group c = t % NC (four columns when K % 4 == 0, read
// as one 16-byte load, else one column) and rows g, g + G, .. of the block's
// range (g = t / NC, G = kRedThreads / NC row groups), eight loads in flight,
// summed in FP32 over up to 64 rows and then in FP64; the row groups are
// added in shared memory in the order g = 0, 1, ..
template <bool VEC>
__global__ void __launch_bounds__(kRedThreads) colsum_partial(const float* __restrict__ X, int64_t R,
                                                               int K, double* __restrict__ part) {
  constexpr int W = VEC ? 4 : 1;  // columns per thread
  __shared__ double grp_sum[kRedThreads * 4];  // [G][K]: G K <= 4 kRedThreads
  const int NC = K / W, G = kRedThreads / NC;
  const int t = threadIdx.x, c = t % NC, g = t / NC;
  const int64_t per = (R + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per;
  const int64_t r1 = min(R, r0 + per);
  double acc[W];
#pragma unroll
  for (int w = 0; w < W; ++w) acc[w] = 0.0;
  auto load = [&](int64_t r, float (&x)[W]) {
    if constexpr (VEC) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(X + r * K) + c);
      x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
      x[0] = __ldg(X + r * K + c);
    }
  };
  if (g < G) {
    // batches of eight rows per thread (eight loads in flight), eight
    // batches summed in FP32 before the FP64 sum
    int64_t r = r0 + g;
    while (r < r1) {
      float s[W];
#pragma unroll
      for (int w = 0; w < W; ++w) s[w] = 0.f;
      for (int b8 = 0; b8 < 8 && r < r1; ++b8, r += (int64_t)G * 8) {
        float x[8][W];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (r + (int64_t)G * u < r1) {
            load(r + (int64_t)G * u, x[u]);
          } else {
#pragma unroll
            for (int w = 0; w < W; ++w) x[u][w] = 0.f;
          }
        }
#pragma unroll
        for (int w = 0; w < W; ++w)
          s[w] += ((x[0][w] + x[1][w]) + (x[2][w] + x[3][w])) + ((x[4][w] + x[5][w]) + (x[6][w] + x[7][w]));
      }
#pragma unroll
      for (int w = 0; w < W; ++w) acc[w] += (double)s[w];
    }
#pragma unroll
    for (int w = 0; w < W; ++w) grp_sum[g * K + c * W + w] = acc[w];
  }
  __syncthreads();
  for (int k = t; k < K; k += kRedThreads) {
    double tot = 0.0;
    for (int q = 0; q < G; ++q) tot += grp_sum[q * K + k];
    part[(int64_t)blockIdx.x * K + k] = tot;
  }
}

// Sum over the blocks' partials of one entry by one warp: lane l adds blocks
// l, l + 32, .. in order, then a fixed shuffle tree; lane 0's total is the
// same in every run.
__device__ __forceinline__ double warp_sum_partials(const double* __restrict__ part, int blocks,
                                                    int64_t stride, int64_t e, int lane) {
  double s = 0.0;
#pragma unroll 4
  for (int b = lane; b < blocks; b += 32) s += part[(int64_t)b * stride + e];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

constexpr int kFinalWarps = 8;

// a warp per column k
__global__ void __launch_bounds__(32 * kFinalWarps) colsum_final(
    const double* __restrict__ part, int blocks, int K, int64_t R, double* __restrict__ xbar,
    float* __restrict__ xbarf) {
  const int lane = threadIdx.x & 31;
  const int k = blockIdx.x * kFinalWarps + (threadIdx.x >> 5);
  if (k >= K) return;  // the whole warp
  const double s = warp_sum_partials(part, blocks, K, k, lane) / (double)R;
  if (lane == 0) {
    xbar[k] = s;
    xbarf[k] = (float)s;
  }
}

// ---- (2) centred scatter S = sum (x - xbar)(x - xbar)^T.  With g = ceil(K / 8)
// and the features in two halves of 4 g, group I is features 4 I .. 4 I + 3 of
// both halves, and the lower triangle is cut into T = g (g + 1) / 2 tiles, the
// 8 x 8 products of group I with group J <= I; a block's threads are (tile,
// subset) pairs: thread t takes tile t % T and, if r = t / T < S, rows r, r + S,
// .. of every chunk.  Neighbouring groups then lie 16 bytes apart and a
// warp's 16-byte loads fall on different banks.  Chunks are copied by cp.async
// into a ring of kScatStages stages; a thread centres what it copied itself
// (always the same columns, so it keeps their means) before the one barrier of
// the chunk.  The S subsets' FP32 sums are added in FP32 in shared memory, in a
// fixed order of four chains (one chain of the 17 subsets of K = 33 .. 40 put S up
// to 1.2 times as far from FP64 as the six subsets of 4 x 4 tiles), and go to the
// block's FP64 partial: at the end, and often enough that no FP32 accumulator sums
// more than kScatFlushRows rows.
// What bounds it: the FP32 multiply-adds, with their shared-memory loads close
// behind.  480,189 rows by 64 blocks, K = 64: 552 us with 4 x 4 tiles, a
// centring pass with a division an element and two barriers a chunk, 287 now
// (chunks of 32 rows 330, and 361 with 288 threads in 96 registers);
// by 26 blocks, K = 100: 2,078 (8 x 8 tiles) -> 1,528 (64 and 26 blocks are the
// allocation-free entry point's, at most one an SM; an iteration's up to 304: both
// sides' reductions of a 480,189 x 17,770 one, K = 100, 800 -> 520).  Two CTAs share an
// SM up to K = 112; past it the ring takes 120 KB and more, and the registers are
// cut for two all the same.  TF32 tensor-core products,
// split in two and summed in FP32 every eight rows, took 205 us at K = 64 but
// their truncated sums doubled the error (2.8e-8 rms of the scale, here 1.5e-8).
constexpr int kScatStages = 4;
constexpr int kScatFlushRows = 512;
constexpr int kScatRows = 64;  // rows per chunk

struct ScatGeom {
  int g, KP, T, S;
  __host__ __device__ ScatGeom(int K, int threads) {
    g = (K + 7) / 8;
    KP = 8 * g;
    T = g * (g + 1) / 2;
    S = threads / T;
  }
  __host__ __device__ int floats() const {
    const int ring = kScatStages * kScatRows * KP, sums = S * T * 64;
    return ring > sums ? ring : sums;
  }
  // the most that any K up to max_k takes (S T <= threads)
  static constexpr int max_floats(int max_k, int threads) {
    return kScatStages * kScatRows * max_k > threads * 64 ? kScatStages * kScatRows * max_k : threads * 64;
  }
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// VEC: K % 4 == 0 and X 16-byte aligned (16-byte copies), else 4-byte copies
template <int NT, bool VEC>
__global__ void __launch_bounds__(NT, 2) scatter_partial(const float* __restrict__ X, int64_t R, int K,
                                                                   const float* __restrict__ xbarf,
                                                                   double* __restrict__ part) {
  constexpr int W = VEC ? 4 : 1;
  extern __shared__ __align__(16) float xs[];  // [kScatStages][kScatRows][KP]; sums [S][16][T][4]
  const ScatGeom G(K, NT);
  const int KP = G.KP, T = G.T, S = G.S, H = 4 * G.g, stage_f = kScatRows * KP;
  const int tid = threadIdx.x;
  const int q = tid % T, r = tid / T;
  const bool active = r < S;
  int I = 0;
  while ((I + 1) * (I + 2) / 2 <= q) ++I;
  const int J = q - I * (I + 1) / 2;
  const int64_t per = (R + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(R, (int64_t)blockIdx.x * per);
  const int64_t r1 = min(R, r0 + per);
  const int64_t nchunks = (r1 - r0 + kScatRows - 1) / kScatRows;
  // this thread's pieces of a chunk: columns W cc .. of rows cr, cr + cstep, ..
  const int P = K / W, cstep = NT / P, cc = tid % P, cr = tid / P < cstep ? tid / P : kScatRows;
  float mean[W];
#pragma unroll
  for (int w = 0; w < W; ++w) mean[w] = xbarf[W * cc + w];
  // the padding columns K .. KP - 1 are never copied: zeroed here, and after the sums have met
  auto zero_padding = [&]() {
    for (int e = tid; e < kScatStages * kScatRows; e += NT)
      for (int k = K; k < KP; ++k) xs[e * KP + k] = 0.f;
  };
  zero_padding();
  auto issue = [&](int64_t c) {
    if (c < nchunks) {
      const int64_t c0 = r0 + c * kScatRows;
      const int cnt = (int)min((int64_t)kScatRows, r1 - c0);
      float* dst = xs + (int)(c % kScatStages) * stage_f + W * cc;
      const float* src = X + c0 * K + W * cc;
      for (int rr = cr; rr < cnt; rr += cstep) {
        if (VEC) cp_async16(dst + rr * KP, src + (int64_t)rr * K);
        else cp_async4(dst + rr * KP, src + (int64_t)rr * K);
      }
    }
    cp_async_commit();  // one group per chunk index, empty past the end
  };
  float acc[8][8];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
  double* out = part + (int64_t)blockIdx.x * K * K;
  bool first = true;
  // the block's sums so far to its partial; acc back to zero
  auto flush = [&]() {
    float4* sums = reinterpret_cast<float4*>(xs);
    if (active) {
#pragma unroll
      for (int v = 0; v < 16; ++v)
        sums[(r * 16 + v) * T + q] = make_float4(acc[v >> 1][4 * (v & 1)], acc[v >> 1][4 * (v & 1) + 1],
                                                 acc[v >> 1][4 * (v & 1) + 2], acc[v >> 1][4 * (v & 1) + 3]);
    }
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
    __syncthreads();
    for (int e = tid; e < 16 * T; e += NT) {
      float4 s4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) s4[u] = u < S ? sums[u * 16 * T + e] : make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k = 4; k < S; k += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (k + u < S) {
            const float4 x = sums[(k + u) * 16 * T + e];
            s4[u].x += x.x; s4[u].y += x.y; s4[u].z += x.z; s4[u].w += x.w;
          }
        }
      }
      const float4 s = make_float4((s4[0].x + s4[1].x) + (s4[2].x + s4[3].x), (s4[0].y + s4[1].y) + (s4[2].y + s4[3].y),
                                   (s4[0].z + s4[1].z) + (s4[2].z + s4[3].z), (s4[0].w + s4[1].w) + (s4[2].w + s4[3].w));
      const int v = e / T, p = v >> 1, t = e - v * T;
      int ti = 0;
      while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
      const int tj = t - ti * (ti + 1) / 2;
      const int i = (p < 4 ? 4 * ti + p : H + 4 * ti + p - 4), j0 = 4 * tj + (v & 1 ? H : 0);
      const float x[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        // past the diagonal: the mirrored entry, which no other tile holds
        // unless the groups are the same
        const int j = j0 + w, hi = max(i, j), lo = min(i, j);
        if (hi < K && (j <= i || ti != tj))
          out[hi * K + lo] = first ? (double)x[w] : out[hi * K + lo] + (double)x[w];
      }
    }
    first = false;
  };
  const int64_t flush_chunks = max(1, kScatFlushRows / ((kScatRows + S - 1) / S));  // rows of a subset a chunk
  for (int c = 0; c < kScatStages - 1; ++c) issue(c);
  for (int64_t c = 0; c < nchunks; ++c) {
    cp_async_wait<kScatStages - 2>();  // chunk c has landed (this thread's copies)
    const int cnt = (int)min((int64_t)kScatRows, r1 - r0 - c * kScatRows);
    float* xb = xs + (int)(c % kScatStages) * stage_f;
    for (int rr = cr; rr < cnt; rr += cstep) {
      float* x = xb + rr * KP + W * cc;
      if constexpr (VEC) {
        float4 v = *reinterpret_cast<float4*>(x);
        v.x -= mean[0]; v.y -= mean[1]; v.z -= mean[2]; v.w -= mean[3];
        *reinterpret_cast<float4*>(x) = v;
      } else {
        x[0] -= mean[0];
      }
    }
    __syncthreads();             // everyone's pieces; chunk c - 1 is no longer read
    issue(c + kScatStages - 1);  // into the stage chunk c - 1 used
    if (active) {
      const float *ai = xb + 4 * I, *bj = xb + 4 * J;
#pragma unroll 2
      for (int rr = r; rr < cnt; rr += S) {
        float a[8], b[8];
        *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(ai + rr * KP);
        *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(ai + rr * KP + H);
        *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(bj + rr * KP);
        *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(bj + rr * KP + H);
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
          for (int p2 = 0; p2 < 8; ++p2) acc[p][p2] = fmaf(a[p], b[p2], acc[p][p2]);
      }
    }
    if ((c + 1) % flush_chunks == 0 && c + 1 < nchunks) {
      // the sums meet in the ring's memory: the copies in flight land first
      // and are made again
      cp_async_wait<0>();
      __syncthreads();
      flush();
      __syncthreads();
      zero_padding();
      __syncthreads();
      for (int k = 1; k < kScatStages; ++k) issue(c + k);
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  flush();
}

// The same for K <= 32, where tiles of eight would leave few of them (K = 10, 8
// iterations of a job: 836 us instead of 807).  The lower triangle is cut into T = g (g + 1) / 2 tiles of TM x TM (g = ceil(K / TM)), and a
// block's threads are (tile, subset) pairs: thread t takes tile q = t % T
// and, if r = t / T < S, rows r, r + S, .. of every chunk of rows.  Chunks
// are copied by cp.async into a ring of kScatStages shared-memory stages
// (rows zero padded to g TM columns), so that three chunks are in flight
// while one is used; each landed chunk is centred in place before use.  The
// FP32 tile sums of the S subsets are added in shared memory in the order
// r = 1, 2, .. into subset 0, which moves them into the block's FP64 partial:
// at the end, and often enough that no FP32 accumulator sums more than
// kSmallFlushRows rows.
constexpr int kSmallThreads = 288;
constexpr int kSmallFlushRows = 1024;
// rows per chunk
constexpr int kSmallRows = 32;

constexpr int kSmallScatK = 32;
int scatter_tm(int K) { return K > 16 ? 4 : K > 4 ? 2 : 1; }
__host__ __device__ constexpr int scatter_tiles(int K, int TM) {
  const int g = (K + TM - 1) / TM;
  return g * (g + 1) / 2;
}
constexpr int scatter_smem(int K, int TM) {
  const int g = (K + TM - 1) / TM;
  return (int)sizeof(float) * (kScatStages * kSmallRows * g * TM + scatter_tiles(K, TM) * TM * TM);
}
static_assert(scatter_smem(kSmallScatK, 4) <= kSmemNoOptIn, "scatter_small takes no opt-in");

template <int TM>
__device__ __forceinline__ void ld_tm(const float* p, float (&x)[TM]) {
  if constexpr (TM == 4) {
    const float4 u = *reinterpret_cast<const float4*>(p);
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
  } else if constexpr (TM == 2) {
    const float2 u = *reinterpret_cast<const float2*>(p);
    x[0] = u.x; x[1] = u.y;
  } else {
    x[0] = p[0];
  }
}

// VEC: K % 4 == 0 and X 16-byte aligned (16-byte copies), else 4-byte copies
template <int TM, bool VEC>
__global__ void __launch_bounds__(kSmallThreads, 2) scatter_small(const float* __restrict__ X, int64_t R,
                                                                int K, const float* __restrict__ xbarf,
                                                                double* __restrict__ part) {
  constexpr int ROWS = kSmallRows;
  extern __shared__ float sbuf[];
  const int g = (K + TM - 1) / TM, KP = g * TM, T = g * (g + 1) / 2;
  const int S = kSmallThreads / T > 1 ? kSmallThreads / T : 1;
  const int stage_f = ROWS * KP;
  float* xs = sbuf;                            // [kScatStages][ROWS][KP]
  float* cmb = sbuf + kScatStages * stage_f;   // [T][TM * TM]
  const int tid = threadIdx.x;
  const int q = tid % T, r = tid / T;
  const bool active = r < S;
  int I = 0;
  while ((I + 1) * (I + 2) / 2 <= q) ++I;
  const int J = q - I * (I + 1) / 2;
  const int64_t per = (R + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = min(R, (int64_t)blockIdx.x * per);
  const int64_t r1 = min(R, r0 + per);
  const int64_t nchunks = (r1 - r0 + ROWS - 1) / ROWS;
  float acc[TM][TM];
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < TM; ++b) acc[a][b] = 0.f;
  // the padding columns K .. KP - 1 are never copied: zero them once
  for (int e = tid; e < kScatStages * stage_f; e += kSmallThreads) xs[e] = 0.f;
  __syncthreads();
  auto issue = [&](int64_t c) {
    if (c < nchunks) {
      const int64_t c0 = r0 + c * ROWS;
      const int cnt = (int)min((int64_t)ROWS, r1 - c0);
      float* dst = xs + (int)(c % kScatStages) * stage_f;
      const float* src = X + c0 * K;
      if (VEC) {
        const int q4 = K >> 2;  // 16-byte pieces per row
        for (int e = tid; e < cnt * q4; e += kSmallThreads) {
          const int rr = e / q4, cc = e - rr * q4;
          cp_async16(dst + rr * KP + 4 * cc, src + (int64_t)rr * K + 4 * cc);
        }
      } else {
        for (int e = tid; e < cnt * K; e += kSmallThreads) {
          const int rr = e / K, cc = e - rr * K;
          cp_async4(dst + rr * KP + cc, src + (int64_t)rr * K + cc);
        }
      }
    }
    cp_async_commit();  // one group per chunk index, empty past the end
  };
  double* out = part + (int64_t)blockIdx.x * K * K;
  int flushed = 0;  // 0: the partial is not written yet
  auto flush = [&]() {
    for (int r2 = 1; r2 < S; ++r2) {
      __syncthreads();
      if (active && r == r2) {
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
          for (int b = 0; b < TM; ++b) cmb[q * TM * TM + a * TM + b] = acc[a][b];
      }
      __syncthreads();
      if (active && r == 0) {
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
          for (int b = 0; b < TM; ++b) acc[a][b] += cmb[q * TM * TM + a * TM + b];
      }
    }
    if (active && r == 0) {
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TM; ++b) {
          const int i = I * TM + a, j = J * TM + b;
          if (i < K && j <= i) out[i * K + j] = flushed ? out[i * K + j] + (double)acc[a][b] : (double)acc[a][b];
        }
    }
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int b = 0; b < TM; ++b) acc[a][b] = 0.f;
  };
  const int flush_chunks = max(1, kSmallFlushRows / ((ROWS + S - 1) / S));  // rows of a subset a chunk
  for (int c = 0; c < kScatStages - 1; ++c) issue(c);
  int nchunk = 0;
  for (int64_t c = 0; c < nchunks; ++c) {
    cp_async_wait<kScatStages - 2>();  // chunk c has landed (this thread's copies)
    __syncthreads();                   // everyone's copies; chunk c - 1 is no longer read
    issue(c + kScatStages - 1);        // into the stage chunk c - 1 used
    const int64_t c0 = r0 + c * ROWS;
    const int cnt = (int)min((int64_t)ROWS, r1 - c0);
    float* xb = xs + (int)(c % kScatStages) * stage_f;
    for (int e = tid; e < cnt * K; e += kSmallThreads) {
      const int rr = e / K, k = e - rr * K;
      xb[rr * KP + k] -= xbarf[k];
    }
    __syncthreads();
    if (active) {
      for (int rr = r; rr < cnt; rr += S) {
        float a[TM], b[TM];
        ld_tm<TM>(xb + rr * KP + I * TM, a);
        ld_tm<TM>(xb + rr * KP + J * TM, b);
#pragma unroll
        for (int p = 0; p < TM; ++p)
#pragma unroll
          for (int p2 = 0; p2 < TM; ++p2) acc[p][p2] = fmaf(a[p], b[p2], acc[p][p2]);
      }
    }
    if (++nchunk == flush_chunks && c + 1 < nchunks) {
      flush();
      flushed = 1;
      nchunk = 0;
    }
  }
  cp_async_wait<0>();
  flush();
}

// a warp per entry (i, j) of the lower triangle, mirrored
__global__ void __launch_bounds__(32 * kFinalWarps) scatter_final(
    const double* __restrict__ part, int blocks, int K, double* __restrict__ S) {
  const int lane = threadIdx.x & 31;
  const int e = blockIdx.x * kFinalWarps + (threadIdx.x >> 5);
  if (e >= K * K) return;
  const int i = e / K, j = e % K;
  if (j > i) return;  // the whole warp
  const double s = warp_sum_partials(part, blocks, (int64_t)K * K, e, lane);
  if (lane == 0) {
    S[i * K + j] = s;
    S[j * K + i] = s;
  }
}

// FP32 copy of Lambda bordered by b0 = Lambda mu: the (K+1) x (K+1) matrix
// [[Lambda, b0], [b0^T, 0]] that the row kernels add alpha times the
// rating-augmented Gram to.
__device__ void write_bordered(const double* lam, const double* mu, int K, float* out) {
  const int KA = K + 1, nt = blockDim.x;
  // four loads in flight per thread and pass
  for (int e0 = threadIdx.x; e0 < K * K; e0 += 4 * nt) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = e0 + u * nt < K * K ? lam[e0 + u * nt] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * nt;
      if (e < K * K) out[(e / K) * KA + (e % K)] = (float)v[u];
    }
  }
  // b0 = Lambda mu, a warp per row (lane l takes k = l, l + 32, ..; a fixed
  // shuffle tree); blockDim.x is a multiple of 32
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  constexpr int kNpl = kMaxK / 32;
  double mk[kNpl];
#pragma unroll
  for (int m = 0; m < kNpl; ++m) mk[m] = lane + 32 * m < K ? mu[lane + 32 * m] : 0.0;
  for (int i = threadIdx.x >> 5; i < K; i += nw) {
    double li[kNpl];
#pragma unroll
    for (int m = 0; m < kNpl; ++m) li[m] = lane + 32 * m < K ? lam[i * K + lane + 32 * m] : 0.0;
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < kNpl; ++m)
      if (32 * m < K) s = fma(li[m], mk[m], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      out[K * KA + i] = (float)s;
      out[i * KA + K] = (float)s;
    }
  }
  if (threadIdx.x == 0) out[K * KA + K] = 0.f;
  __syncthreads();
}

// float copies of a side's hyperparameters (after bpmf_set_state)
__global__ void hyper_f32(const double* lam, const double* mu, int K, float* lamaug) {
  write_bordered(lam, mu, K, lamaug);
}

template <int TM, bool VEC>
int launch_scatter_tm(const float* X, int64_t R, int K, const float* xbarf, double* part, int blocks,
                      cudaStream_t st) {
  const int smem = scatter_smem(K, TM);
  scatter_small<TM, VEC><<<blocks, kSmallThreads, smem, st>>>(X, R, K, xbarf, part);
  return BPMF_OK;
}

// 16-byte loads and copies of the rows need K % 4 == 0 and an aligned X
bool rows_vec(const float* X, int K) { return (K & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0; }

int launch_scatter(const float* X, int64_t R, int K, const float* xbarf, double* part, int blocks,
                   cudaStream_t st) {
  const bool v = rows_vec(X, K);
  if (K <= kSmallScatK) {
    switch (scatter_tm(K)) {
      case 4: return v ? launch_scatter_tm<4, true>(X, R, K, xbarf, part, blocks, st)
                       : launch_scatter_tm<4, false>(X, R, K, xbarf, part, blocks, st);
      case 2: return v ? launch_scatter_tm<2, true>(X, R, K, xbarf, part, blocks, st)
                       : launch_scatter_tm<2, false>(X, R, K, xbarf, part, blocks, st);
      default: return v ? launch_scatter_tm<1, true>(X, R, K, xbarf, part, blocks, st)
                        : launch_scatter_tm<1, false>(X, R, K, xbarf, part, blocks, st);
    }
  }
  // up to 36 tiles leave 252 or more of 256 threads busy; 91 and 136 want 288
  constexpr int kNarrow = 64;
  const int threads = K <= kNarrow ? 256 : 288;
  auto kern = K <= kNarrow ? (v ? scatter_partial<256, true> : scatter_partial<256, false>)
                      : (v ? scatter_partial<288, true> : scatter_partial<288, false>);
  const int smem = (int)sizeof(float) * ScatGeom(K, threads).floats();
  BPMF_TRY(allow_smem(kern, sizeof(float) * ScatGeom::max_floats(K <= kNarrow ? kNarrow : kMaxK, threads)));
  kern<<<blocks, threads, smem, st>>>(X, R, K, xbarf, part);
  return BPMF_OK;
}

int launch_colsum(const float* X, int64_t R, int K, double* part, int blocks, cudaStream_t st) {
  if (rows_vec(X, K)) colsum_partial<true><<<blocks, kRedThreads, 0, st>>>(X, R, K, part);
  else colsum_partial<false><<<blocks, kRedThreads, 0, st>>>(X, R, K, part);
  return BPMF_OK;
}

}  // namespace

int launch_hyper(Handle* h, int s, cudaStream_t st, bool alt) {
  SideDev& sd = h->side[s];
  const int K = h->K;
  if (st == nullptr) st = h->stream;
  double* red = alt ? h->red2 : h->red;
  double* wscr = alt ? h->wscr2 : h->wscr;
  const int64_t R = sd.R;
  // blocks: up to 2 per SM, at least 64 rows each
  int blocks = 2 * h->num_sms;
  if ((int64_t)blocks * 64 > R) blocks = (int)std::max<int64_t>(1, (R + 63) / 64);
  double* part = red;  // holds blocks * K * K doubles (sized at init)
  float* xbarf = reinterpret_cast<float*>(wscr + 6 * K * K + 4 * K);
  {
    PhaseTimer timer(h, BPMF_T_HYPER_REDUCE, st);
    BPMF_TRY(launch_colsum(sd.X, R, K, part, blocks, st));
    colsum_final<<<(K + kFinalWarps - 1) / kFinalWarps, 32 * kFinalWarps, 0, st>>>(
        part, blocks, K, R, sd.xbar, xbarf);
    BPMF_TRY(launch_scatter(sd.X, R, K, xbarf, part, blocks, st));
    scatter_final<<<(K * K + kFinalWarps - 1) / kFinalWarps, 32 * kFinalWarps, 0, st>>>(
        part, blocks, K, sd.S);
    BPMF_CUDA_CHECK(cudaGetLastError());
    h->kernels += 5;
  }
  HyperArgs a;
  a.xbar = sd.xbar;
  a.S = sd.S;
  a.n = R;
  a.mu0 = h->mu0;
  a.beta0 = h->cfg.beta0;
  a.nu0 = h->cfg.nu0;
  a.wmean = a.beta0 * (double)R / (a.beta0 + (double)R);
  a.W0inv = h->W0inv;
  a.seed = h->cfg.seed;
  a.tp = h->d_iter;
  a.side = s;
  a.K = K;
  a.scr = wscr;
  a.lam = sd.lam;
  a.mu = sd.mu;
  a.lamaug = sd.lamaug;
  a.lchol = sd.lchol;
  a.status = h->status;
  a.gamma_cap = h->gamma_cap;
  {
    PhaseTimer timer(h, BPMF_T_HYPER_DRAW, st);
    BPMF_TRY(launch_wishart(a, h->wish_ctas, st, &h->kernels));
  }
  sd.have_hyper = true;
  sd.have_stats = true;
  return BPMF_OK;
}

// The row mean and centred scatter of X (R x K) into xbar and S, with the
// per-block partials in `part` (blocks * K * K doubles) and the FP32 mean in
// `xbarf` (K floats); both are caller-provided scratch.
int launch_stats_into(const float* X, int64_t R, int K, double* part, int blocks, double* xbar,
                      double* S, float* xbarf, cudaStream_t st) {
  BPMF_TRY(launch_colsum(X, R, K, part, blocks, st));
  colsum_final<<<(K + kFinalWarps - 1) / kFinalWarps, 32 * kFinalWarps, 0, st>>>(part, blocks, K, R,
                                                                                xbar, xbarf);
  BPMF_TRY(launch_scatter(X, R, K, xbarf, part, blocks, st));
  scatter_final<<<(K * K + kFinalWarps - 1) / kFinalWarps, 32 * kFinalWarps, 0, st>>>(part, blocks,
                                                                                     K, S);
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

int launch_hyper_to_f32(Handle* h, int s) {
  SideDev& sd = h->side[s];
  hyper_f32<<<1, 256, 0, h->stream>>>(sd.lam, sd.mu, h->K, sd.lamaug);
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

}  // namespace gb
