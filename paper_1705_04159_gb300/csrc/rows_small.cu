// rows_small.cu -- row draws of small latent dimension, one warp per row, FP32,
// and the pieces of split rows.
//
// The conditional is the one of rows.cu (Algorithm 1's row update): for row
// i with rated neighbours j,
//   Lambda* = Lambda_s + alpha sum_j v_j v_j^T,  b = Lambda_s mu_s + alpha sum_j r_ij v_j,
//   L = chol(Lambda*),  u_i = L^-T (L^-1 b + z).
// For K <= 55 the bordered matrix has at most 28 tiles of 8 x 8 (g <= 7 a side)
// and one warp holds the whole Gram of the rating-augmented neighbours
// x_j = [v_j, r_ij] in registers, so no block-wide barrier is needed (the
// light-row kernel of the degree bins, paper Sec. III):
//   Gram: neighbours are staged 16 or 32 at a time in the warp's shared memory with
//     cp.async (double-buffered) and multiplied eight at a time on the tensor
//     cores, mma.m16n8k8 over pairs of row tiles; FP32 operands are split into
//     two TF32 parts, x = h + l, and l h + h l + h h of one step of eight is
//     formed from zero and then added in FP32: the tensor core's accumulator
//     rounds towards zero, which over many steps would add up to a bias (over
//     1,024 neighbours 1e-5 of the sum; by the step 2.0e-7, FP32 multiply-adds
//     one after the other 5.1e-7).  The two parts keep 23 of an operand's 24 bits and
//     l l is left out, which a row of a few ratings and a small K shows: its draw was
//     up to 1.3 times as far from FP64 as with FP32 multiply-adds (rms; 1.0 times
//     at 12 ratings, 0.6 at 100, any number at K >= 24).  So for K <= 23 rows of up
//     to 16 ratings, and the pieces of a hub up to 64 for K <= 15 (they add up in
//     FP32), take multiply-adds (sm_few): 100,000 rows of 14 ratings, K = 16, 273 ->
//     292 us, of 6 ratings 268 -> 273.  The staged row stride is an odd multiple of
//     eight floats, so the fragments (features 8 I + lane / 4 of neighbours
//     lane % 4 and + 4) load without bank conflicts;
//   the factorisation and the draw: warp_chol.cuh.
// The base matrix (Lambda_s bordered by Lambda_s mu_s) is shared by the CTA's
// warps.  Pieces of split rows (hubs) take the same Gram and store it; one CTA
// per hub adds its pieces in order and draws.
// Where K is a multiple of eight the rating would make a tile row of its own;
// the Gram then covers the features alone, and sum_j r_ij v_j is formed by
// FP32 multiply-adds from the fragments at hand (K = 32: 18 tensor products a
// step instead of 33).
// What bounds it: issue and latency, more in the factorisation than in the Gram
// at 100 ratings a row (K = 50: 10.8k warp instructions a row, issue slots 49%
// busy, tensor pipe 28%; K = 32: 5.6k, 63%, 22%).  A sweep of 30,000 rows with
// 3M ratings, K = 50, took 1,450 us with one CTA per row and FP32
// multiply-adds, and takes 732; K = 32, 546 -> 331 us.  An iteration of
// 138,493 x 26,744 with 20M ratings, K = 32, took 3,560 us with one warp per
// row and FP32 multiply-adds (hub pieces: a CTA each), 2,816 with the rating as
// a tile row, and takes 2,208; stages of 16 neighbours instead of 32: 2,321.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "rows.cuh"
#include "tile_chol.cuh"
#include "warp_chol.cuh"

namespace gb {
namespace {

constexpr int kSmWarps = 4;   // warps (rows) per CTA
// CTAs per SM the registers are cut for: 80 to 128 a thread without spills, 168
// where the Gram takes up to 76
constexpr int sm_ctas(int g) { return g <= 3 ? 6 : g == 4 ? 5 : g == 5 ? 4 : 3; }
constexpr int kSmMaxG = 7;    // K <= 55

// g tile rows, the last of them row K alone if B (K = 8 (g - 1)): the Gram's
// tiles then cover the K features, and sum_j r_ij v_j is kept aside.
template <int g, bool B>
struct SmGeom {
  static constexpr int KP = 8 * g;
  static constexpr int G = B ? g - 1 : g;             // tile rows of the Gram
  static constexpr int LDT = G & 1 ? 8 * G : 8 * G + 8;  // staged row stride: an odd multiple of 8
  static constexpr int NP = (G + 1) / 2;              // pairs of row tiles
  static constexpr int NT = g * (g + 1) / 2;          // tiles
  // accumulators: pair k covers tile columns 0 .. min(2 k + 1, G - 1), from k (k + 1)
  static constexpr int NA = G & 1 ? (NP - 1) * NP + 2 * NP - 1 : NP * (NP + 1);
  __host__ __device__ static constexpr int cols(int k) { return 2 * k + 2 < G ? 2 * k + 2 : G; }
  // neighbours staged at a time; 32 of seven tile rows would leave the L1 32 KB
  // (K = 50: 744 us instead of 732, K = 32: 331 instead of 340)
  static constexpr int kChunk = G < 7 ? 32 : 16;
  // up to so many neighbours of a row, and of a piece, by FP32 multiply-adds (sm_few)
  static constexpr int kFew = g <= 3 ? 16 : 0, kFewPiece = g <= 2 ? 64 : kFew;
  static constexpr int kRows = 2 * kChunk * LDT;    // staged rows, then ratings if B
  static constexpr int kStage = kRows + (B ? 2 * kChunk : 0);
  // per warp: staging buffers, reused by the tiles; thresholds, 1 / diagonal, z
  static constexpr int kFloats = (kStage > NT * kTileF ? kStage : NT * kTileF) + 3 * KP;
};

template <int V>
__device__ __forceinline__ void cp_async(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (V == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  else if constexpr (V == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Stages neighbours whose ids and ratings lanes 0 .. cnt - 1 hold, V floats per
// copy, 8, 16 or 32 lanes (V = 4, 2, 1) a row and at most two copies each; the
// ratings go Rs floats apart to R; the rows up to the next multiple of eight
// are zeroed.
template <int LDT, int V>
__device__ __forceinline__ void sm_stage(const float* __restrict__ Vo, int K, float* T, float* R, int Rs,
                                         int j, float r, int cnt, int lane) {
  constexpr int kLanes = 32 / V, kStep = V;  // lanes a row, rows a step
  const int q = V * (lane % kLanes);
  int rr = lane / kLanes;
  float* dst = T + rr * LDT + q;
#pragma unroll 4
  for (int k = 0; k < cnt; k += kStep) {
    const int jr = __shfl_sync(0xffffffffu, j, rr);
    const float* src = Vo + (int64_t)jr * K + q;
    if (rr < cnt) {
      if (q < K) cp_async<V>(dst, src);
      if (q + 32 < K) cp_async<V>(dst + 32, src + 32);
    }
    rr += kStep;
    dst += kStep * LDT;
  }
  const int pad = -cnt & 7;
  if (pad) {
    for (int k = 0; k < pad; ++k)
      for (int c = lane; c < K; c += 32) T[(cnt + k) * LDT + c] = 0.f;
  }
  if (lane < cnt + pad) R[lane * Rs] = lane < cnt ? r : 0.f;
  cp_async_commit();
}

__device__ __forceinline__ void mma_tf32_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// o += x x^T of n staged neighbours by FP32 multiply-adds, neighbour by
// neighbour (X0: the first one's row, zeros past n up to a multiple of four); if
// B, s as sm_step forms it
template <int g, bool B>
__device__ __forceinline__ void sm_few(const float* X0, const float* R, int n, int lane,
                                       float (&o)[SmGeom<g, B>::NA][4], float (&s)[SmGeom<g, B>::G]) {
  using S = SmGeom<g, B>;
  const int t = lane & 3;
  const float *xr = X0 + (lane >> 2), *xc = X0 + 2 * t;
#pragma unroll 1
  for (int e0 = 0; e0 < n; e0 += 4, xr += 4 * S::LDT, xc += 4 * S::LDT) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float x[S::G];
#pragma unroll
      for (int I = 0; I < S::G; ++I) x[I] = xr[e * S::LDT + 8 * I];
#pragma unroll
      for (int J = 0; J < S::G; ++J) {
        const float2 y = ldf2(xc + e * S::LDT + 8 * J);
#pragma unroll
        for (int I = J; I < S::G; ++I) {
          float(&d)[4] = o[(I >> 1) * ((I >> 1) + 1) + J];
          d[2 * (I & 1)] = fmaf(x[I], y.x, d[2 * (I & 1)]);
          d[2 * (I & 1) + 1] = fmaf(x[I], y.y, d[2 * (I & 1) + 1]);
        }
      }
      if (B && e == t) {  // a lane in four keeps the sum of a neighbour
        const float r = R[e0];
#pragma unroll
        for (int I = 0; I < S::G; ++I) s[I] = fmaf(r, x[I], s[I]);
      }
    }
  }
}

// o += sum over eight staged neighbours of x x^T (lower tiles, in pairs); if
// B, s += their r x (R: their ratings; a lane's own two neighbours only)
template <int g, bool B>
__device__ __forceinline__ void sm_step(const float* X, const float* R, float (&o)[SmGeom<g, B>::NA][4],
                                        float (&s)[SmGeom<g, B>::G]) {
  using S = SmGeom<g, B>;
  uint32_t h0[S::G], h1[S::G], l0[S::G], l1[S::G];
  float r0 = 0.f, r1 = 0.f;
  if (B) {
    r0 = R[0];
    r1 = R[4];
  }
#pragma unroll
  for (int I = 0; I < S::G; ++I) {
    const float x0 = X[8 * I], x1 = X[4 * S::LDT + 8 * I];
    split_tf32(x0, h0[I], l0[I]);
    split_tf32(x1, h1[I], l1[I]);
    if (B) s[I] = fmaf(r1, x1, fmaf(r0, x0, s[I]));
  }
#pragma unroll
  for (int k = 0; k < S::NP; ++k) {
    const int u = 2 * k, v = 2 * k + 1 < S::G ? 2 * k + 1 : 2 * k;
#pragma unroll
    for (int J0 = 0; J0 < S::G; J0 += 4) {
      float d[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (J0 + c < S::cols(k))
          mma_tf32_zero(d[c], l0[u], l0[v], l1[u], l1[v], h0[J0 + c], h1[J0 + c]);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (J0 + c < S::cols(k)) mma_tf32(d[c], h0[u], h0[v], h1[u], h1[v], l0[J0 + c], l1[J0 + c]);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (J0 + c < S::cols(k)) mma_tf32(d[c], h0[u], h0[v], h1[u], h1[v], h0[J0 + c], h1[J0 + c]);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (J0 + c < S::cols(k)) {
#pragma unroll
          for (int q = 0; q < 4; ++q) o[k * (k + 1) + J0 + c][q] += d[c][q];
        }
    }
  }
}

// o (and s) = sums over ratings [e0, e1)
template <int g, bool B, int V>
__device__ __forceinline__ void sm_gram_v(const SweepArgs& a, float* T, int64_t e0, int64_t e1, int few, int lane,
                                          float (&o)[SmGeom<g, B>::NA][4], float (&s)[SmGeom<g, B>::G]) {
  using S = SmGeom<g, B>;
  constexpr int kBuf = S::kChunk * S::LDT;
  const int K = a.K;
  const int64_t n = e1 - e0;
  const float* X = T + (lane & 3) * S::LDT + (lane >> 2);
  const float* R = T + S::kRows + (lane & 3);
  // ids and ratings of the chunk after the one being staged, a lane each
  int j = 0;
  float r = 0.f;
  auto load = [&](int64_t c0) {
    j = 0;
    r = 0.f;
    if (lane < S::kChunk && c0 + lane < n) {
      j = __ldg(a.idx + e0 + c0 + lane);
      r = __ldg(a.val + e0 + c0 + lane);
    }
  };
  auto count = [&](int64_t c0) { return (int)min((int64_t)S::kChunk, n - c0); };
  auto stage = [&](int64_t c0, int buf) {
    float* row = T + buf * kBuf;
    sm_stage<S::LDT, V>(a.Vo, K, row, B ? T + S::kRows + buf * S::kChunk : row + K, B ? 1 : S::LDT, j, r,
                        count(c0), lane);
  };
  if (n <= 0) return;
  load(0);
  stage(0, 0);
  load(S::kChunk);
  int buf = 0;
  for (int64_t c0 = 0; c0 < n; c0 += S::kChunk, buf ^= 1) {
    if (c0 + S::kChunk < n) {
      stage(c0 + S::kChunk, buf ^ 1);
      load(c0 + 2 * S::kChunk);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    const float *Xb = X + buf * kBuf, *Rb = R + buf * S::kChunk;
    const int cnt = count(c0);
    if (n <= few) {
      sm_few<g, B>(T + buf * kBuf, Rb, cnt, lane, o, s);
    } else {
#pragma unroll 1
      for (int k = 0; k < cnt; k += 8) sm_step<g, B>(Xb + k * S::LDT, Rb + k, o, s);
    }
    __syncwarp();  // the buffer is refilled next
  }
}

template <int g, bool B>
__device__ __forceinline__ void sm_gram(const SweepArgs& a, float* T, int64_t e0, int64_t e1, int few, int lane,
                                        float (&o)[SmGeom<g, B>::NA][4], float (&s)[SmGeom<g, B>::G]) {
  using S = SmGeom<g, B>;
#pragma unroll
  for (int i = 0; i < S::NA; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) o[i][q] = 0.f;
#pragma unroll
  for (int i = 0; i < S::G; ++i) s[i] = 0.f;
  if constexpr (B) {
    sm_gram_v<g, B, 4>(a, T, e0, e1, few, lane, o, s);
    // over the four lanes that share a feature
#pragma unroll
    for (int i = 0; i < S::G; ++i) {
      s[i] += __shfl_xor_sync(0xffffffffu, s[i], 1);
      s[i] += __shfl_xor_sync(0xffffffffu, s[i], 2);
    }
  } else {
    // the columns past the rating stay zero in both buffers
    for (int e = lane; e < 2 * S::kChunk; e += 32) {
#pragma unroll
      for (int c = S::KP - 8; c < S::KP; ++c)
        if (c > a.K) T[e * S::LDT + c] = 0.f;
    }
    __syncwarp();
    if ((a.K & 3) == 0) sm_gram_v<g, B, 4>(a, T, e0, e1, few, lane, o, s);
    else if ((a.K & 1) == 0) sm_gram_v<g, B, 2>(a, T, e0, e1, few, lane, o, s);
    else sm_gram_v<g, B, 1>(a, T, e0, e1, few, lane, o, s);
  }
}

template <int g, bool B>
__global__ void __launch_bounds__(32 * kSmWarps, sm_ctas(g)) row_small(const SweepArgs a) {
  using S = SmGeom<g, B>;
  extern __shared__ __align__(16) float ssm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* base = ssm;
  for (int e = threadIdx.x; e < S::KP * S::KP; e += blockDim.x) {
    const int i = e / S::KP, j = e - i * S::KP;
    if ((j >> 3) <= (i >> 3)) base[tidx(i >> 3, j >> 3) * kTileF + trow(i & 7) + (j & 7)] = row_base(a, i, j);
  }
  __syncthreads();  // the only block-wide barrier
  const int64_t slot = a.row_begin + (int64_t)blockIdx.x * kSmWarps + warp;
  if (slot >= a.row_end) return;
  const int row = a.rows ? a.rows[slot] : (int)slot;
  float* T = ssm + S::NT * kTileF + warp * S::kFloats;
  float* thr = T + S::kFloats - 3 * S::KP;
  float* rinv = thr + S::KP;
  float* zv = rinv + S::KP;
  {
    float o[S::NA][4], s[S::G];
    sm_gram<g, B>(a, T, a.ptr[row], a.ptr[row + 1], S::kFew, lane, o, s);
    // A = base + alpha G as tiles, over the staging buffers
    const int gr = lane >> 2, t2 = 2 * (lane & 3), fo = trow(gr) + t2;
#pragma unroll
    for (int k = 0; k < S::NP; ++k)
#pragma unroll
      for (int J = 0; J < S::G; ++J)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int I = 2 * k + h;
          if (J <= I && I < S::G) {
            const int off = tidx(I, J) * kTileF + fo;
            const float2 b = ldf2(base + off);
            const float x = fmaf(a.alpha, o[k * (k + 1) + J][2 * h], b.x);
            const float y = fmaf(a.alpha, o[k * (k + 1) + J][2 * h + 1], b.y);
            *reinterpret_cast<float2*>(T + off) = make_float2(x, y);
            if (J == I && (gr & ~1) == t2)
              thr[8 * I + gr] = 8 * I + gr < a.K ? pivot_threshold(a.pivot_rel, gr & 1 ? y : x) : -INFINITY;
          }
        }
    if (B) {  // row K, and the padding after it
#pragma unroll
      for (int J = 0; J < g; ++J) {
        const int off = tidx(g - 1, J) * kTileF + fo;
        float2 b = ldf2(base + off);
        if (J < S::G) {
          const float sx = __shfl_sync(0xffffffffu, s[J < S::G ? J : 0], 4 * t2);
          const float sy = __shfl_sync(0xffffffffu, s[J < S::G ? J : 0], 4 * t2 + 4);
          if (gr == 0) b = make_float2(fmaf(a.alpha, sx, b.x), fmaf(a.alpha, sy, b.y));
        }
        *reinterpret_cast<float2*>(T + off) = b;
      }
      if (lane < 8) thr[8 * (g - 1) + lane] = -INFINITY;
    }
  }
  __syncwarp();
  row_draw(a, g, T, thr, rinv, zv, row, lane);
}

// Partial Gram of one piece of a split row by one warp, stored as raw tiles in
// the numbering of tile_chol.cuh.
template <int g, bool B>
__global__ void __launch_bounds__(32 * kSmWarps, sm_ctas(g)) piece_small(const SweepArgs a, int64_t npieces) {
  using S = SmGeom<g, B>;
  extern __shared__ __align__(16) float ssm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t pc = (int64_t)blockIdx.x * kSmWarps + warp;
  if (pc >= npieces) return;
  float o[S::NA][4], s[S::G];
  sm_gram<g, B>(a, ssm + warp * S::kStage, a.piece_e0[pc], a.piece_e1[pc], S::kFewPiece, lane, o, s);
  float* dst = a.part + pc * S::NT * 64 + 2 * lane;
#pragma unroll
  for (int k = 0; k < S::NP; ++k)
#pragma unroll
    for (int J = 0; J < S::G; ++J)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int I = 2 * k + h;
        if (J <= I && I < S::G)
          *reinterpret_cast<float2*>(dst + tile_id(I, J, g) * 64) =
              make_float2(o[k * (k + 1) + J][2 * h], o[k * (k + 1) + J][2 * h + 1]);
      }
  if (B && (lane & 3) == 0) {  // row K of the last tile row, all that the draw reads of it
#pragma unroll
    for (int J = 0; J < S::G; ++J) a.part[(pc * S::NT + tile_id(g - 1, J, g)) * 64 + (lane >> 2)] = s[J];
  }
}

// Hub rows from their partial Grams, any K: a CTA adds the pieces of its hub
// in order (each thread some groups of four elements, four pieces' loads in
// flight), forms the tiles, and one warp draws the row.
constexpr int kHubThreads = 256;
__global__ void __launch_bounds__(kHubThreads) hub_draw(const SweepArgs a) {
  extern __shared__ __align__(16) float ssm[];
  const int K = a.K, g = (K + 8) / 8, NT = g * (g + 1) / 2;
  float* T = ssm;
  float* thr = T + NT * kTileF;
  float* rinv = thr + 8 * g;
  float* zv = rinv + 8 * g;
  const int64_t slot = a.row_begin + blockIdx.x;
  const int32_t pb = a.hub_piece0[slot], pe = a.hub_piece0[slot + 1];
  for (int e = threadIdx.x; e < NT * 16; e += kHubThreads) {
    const int64_t stride = (int64_t)NT * 16;
    const float4* src = reinterpret_cast<const float4*>(a.part) + pb * stride + e;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    int32_t p = pb;
    for (; p + 4 <= pe; p += 4, src += 4 * stride) {
      float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = __ldcs(src + u * stride);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s.x += x[u].x; s.y += x[u].y; s.z += x[u].z; s.w += x[u].w;
      }
    }
    for (; p < pe; ++p, src += stride) {
      const float4 x = __ldcs(src);
      s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    int I, J;
    tri_tile(e >> 4, g, I, J);
    const int r = (e >> 1) & 7, c = (e & 1) * 4;
    const int i = 8 * I + r, j = 8 * J + c;
    const float4 v = make_float4(row_elem(a, i, j, s.x), row_elem(a, i, j + 1, s.y), row_elem(a, i, j + 2, s.z),
                                 row_elem(a, i, j + 3, s.w));
    *reinterpret_cast<float4*>(T + tidx(I, J) * kTileF + trow(r) + c) = v;
    if (I == J && (r & 4) == c) {
      const float d = (r & 3) == 0 ? v.x : (r & 3) == 1 ? v.y : (r & 3) == 2 ? v.z : v.w;
      thr[i] = i < K ? pivot_threshold(a.pivot_rel, d) : -INFINITY;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) row_draw<2>(a, g, T, thr, rinv, zv, a.rows ? a.rows[slot] : (int)slot, threadIdx.x);
}

template <int g, bool B>
int launch_small(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  using S = SmGeom<g, B>;
  const int smem = (S::NT * kTileF + kSmWarps * S::kFloats) * (int)sizeof(float);
  BPMF_TRY(allow_smem(row_small<g, B>, smem));
  const int64_t n = a.row_end - a.row_begin;
  for (int64_t off = 0; off < n; off += (int64_t)kSmWarps << 27) {
    SweepArgs b = a;
    b.row_begin = a.row_begin + off;
    b.row_end = b.row_begin + std::min<int64_t>(n - off, (int64_t)kSmWarps << 27);
    const int64_t blocks = (b.row_end - b.row_begin + kSmWarps - 1) / kSmWarps;
    row_small<g, B><<<(unsigned)blocks, 32 * kSmWarps, smem, st>>>(b);
    BPMF_CUDA_CHECK(cudaGetLastError());
    if (launches) *launches += 1;
  }
  return BPMF_OK;
}

template <int g, bool B>
int launch_small_pieces(const SweepArgs& a, int64_t npieces, cudaStream_t st, int64_t* launches) {
  using S = SmGeom<g, B>;
  const int smem = kSmWarps * S::kStage * (int)sizeof(float);
  BPMF_TRY(allow_smem(piece_small<g, B>, smem));
  piece_small<g, B><<<(unsigned)((npieces + kSmWarps - 1) / kSmWarps), 32 * kSmWarps, smem, st>>>(a, npieces);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

}  // namespace

bool small_supported(int K) { return K >= 1 && (K + 8) / 8 <= kSmMaxG; }

int launch_rows_small(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  if (a.row_end <= a.row_begin) return BPMF_OK;
#define GB_SMALL(fn, ...)                                                                      \
  if (a.K % 8 == 0) {                                                                          \
    switch (a.K / 8) {                                                                         \
      case 1: return fn<2, true>(__VA_ARGS__);                                                 \
      case 2: return fn<3, true>(__VA_ARGS__);                                                 \
      case 3: return fn<4, true>(__VA_ARGS__);                                                 \
      case 4: return fn<5, true>(__VA_ARGS__);                                                 \
      case 5: return fn<6, true>(__VA_ARGS__);                                                 \
      case 6: return fn<7, true>(__VA_ARGS__);                                                 \
    }                                                                                          \
  }                                                                                            \
  switch ((a.K + 8) / 8) {                                                                     \
    case 1: return fn<1, false>(__VA_ARGS__);                                                  \
    case 2: return fn<2, false>(__VA_ARGS__);                                                  \
    case 3: return fn<3, false>(__VA_ARGS__);                                                  \
    case 4: return fn<4, false>(__VA_ARGS__);                                                  \
    case 5: return fn<5, false>(__VA_ARGS__);                                                  \
    case 6: return fn<6, false>(__VA_ARGS__);                                                  \
    case 7: return fn<7, false>(__VA_ARGS__);                                                  \
    default: return BPMF_EINVAL;                                                               \
  }
  GB_SMALL(launch_small, a, st, launches)
}

int launch_pieces_small(const SweepArgs& a, int64_t npieces, cudaStream_t st, int64_t* launches) {
  if (npieces <= 0) return BPMF_OK;
  GB_SMALL(launch_small_pieces, a, npieces, st, launches)
}
#undef GB_SMALL

int64_t partial_floats_per_piece(int K) {
  const int g = (K + 8) / 8;
  return (int64_t)g * (g + 1) / 2 * 64;
}

int launch_hub_draw(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  const int64_t n = a.row_end - a.row_begin;
  if (n <= 0) return BPMF_OK;
  auto bytes = [](int g) { return (g * (g + 1) / 2 * kTileF + 3 * 8 * g) * sizeof(float); };
  static_assert(bytes((kMaxK + 8) / 8) <= kSmemNoOptIn, "hub_draw takes no opt-in");
  const size_t smem = bytes((a.K + 8) / 8);
  hub_draw<<<(unsigned)n, kHubThreads, smem, st>>>(a);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

}  // namespace gb
