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
//   Gram: neighbours are staged 16 at a time in the warp's shared memory with
//     cp.async (double-buffered) and multiplied eight at a time on the tensor
//     cores, mma.m16n8k8 over pairs of row tiles; FP32 operands are split into
//     two TF32 parts, x = h + l, and l h + h l + h h of one step of eight is
//     formed from zero and then added in FP32: the tensor core's accumulator
//     rounds towards zero, which over many steps would add up to a bias (over
//     1,024 neighbours 1e-5 of the sum; by the step 2.0e-7, FP32 multiply-adds
//     one after the other 5.1e-7).  The staged row stride is an odd multiple of
//     eight floats, so the fragments (features 8 I + lane / 4 of neighbours
//     lane % 4 and + 4) load without bank conflicts;
//   the factorisation and the draw: warp_chol.cuh.
// The base matrix (Lambda_s bordered by Lambda_s mu_s) is shared by the CTA's
// warps.  Pieces of split rows (hubs) take the same Gram and store it; one CTA
// per hub adds its pieces in order and draws.
// What bounds it: instruction issue.  A sweep of
// 30,000 rows with 3M ratings, K = 50, took 1,450 us with one CTA per row and
// FP32 multiply-adds, and takes 729; an iteration of 138,493 x 26,744 with 20M
// ratings, K = 32, 3,560 us with one warp per row and FP32 multiply-adds (hub
// pieces: a CTA each), and takes 2,816.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "rows.cuh"
#include "tile_chol.cuh"
#include "warp_chol.cuh"

namespace gb {
namespace {

constexpr int kSmChunk = 16;  // neighbours staged per step
constexpr int kSmWarps = 4;   // warps (rows) per CTA
// CTAs per SM the registers are cut for: 128 a thread, 168 where the Gram takes up to 76
constexpr int sm_ctas(int g) { return g <= 5 ? 4 : 3; }
constexpr int kSmMaxG = 7;    // K <= 55

template <int g>
struct SmGeom {
  static constexpr int KP = 8 * g;
  static constexpr int LDT = g & 1 ? KP : KP + 8;  // staged row stride: an odd multiple of 8
  static constexpr int NP = (g + 1) / 2;           // pairs of row tiles
  static constexpr int NT = g * (g + 1) / 2;       // tiles
  // accumulators: pair k covers tile columns 0 .. min(2 k + 1, g - 1), from k (k + 1)
  static constexpr int NA = g & 1 ? (NP - 1) * NP + 2 * NP - 1 : NP * (NP + 1);
  __host__ __device__ static constexpr int cols(int k) { return 2 * k + 2 < g ? 2 * k + 2 : g; }
  static constexpr int kStage = 2 * kSmChunk * LDT;
  // per warp: staging buffers, reused by the tiles; thresholds, 1 / diagonal, z
  static constexpr int kFloats = (kStage > NT * kTileF ? kStage : NT * kTileF) + 3 * KP;
};

// 16-, 8- and 4-byte copies, zero-filling when not live
__device__ __forceinline__ void cp_async_z(float* dst, const float* src, int bytes, bool live) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = live ? bytes : 0;
  if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
  else if (bytes == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Stages neighbours whose ids and ratings lanes 0 .. cnt - 1 hold, V floats per
// copy; the rows up to the next multiple of eight are zeroed.
template <int g, int V>
__device__ __forceinline__ void sm_stage(const float* __restrict__ Vo, int K, float* T, int j, float r,
                                         int cnt, int lane) {
  constexpr int LDT = SmGeom<g>::LDT;
  const int P = K / V, n = ((cnt + 7) & ~7) * P;
  // lane l copies pieces l, l + 32, ..: row rr, piece q, stepped without divisions
  int rr = lane / P, q = lane - rr * P;
  const int dr = 32 / P, dq = 32 - dr * P;
  for (int e0 = 0; e0 < n; e0 += 32) {
    const int jr = __shfl_sync(0xffffffffu, j, rr & 31);
    if (e0 + lane < n) cp_async_z(T + rr * LDT + V * q, Vo + (int64_t)jr * K + V * q, 4 * V, rr < cnt);
    rr += dr;
    q += dq;
    if (q >= P) {
      q -= P;
      ++rr;
    }
  }
  if (lane < ((cnt + 7) & ~7)) T[lane * LDT + K] = lane < cnt ? r : 0.f;
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

// o += sum over eight staged neighbours of x x^T (lower tiles, in pairs)
template <int g>
__device__ __forceinline__ void sm_step(const float* X, float (&o)[SmGeom<g>::NA][4]) {
  using S = SmGeom<g>;
  uint32_t h0[g], h1[g], l0[g], l1[g];
#pragma unroll
  for (int I = 0; I < g; ++I) {
    split_tf32(X[8 * I], h0[I], l0[I]);
    split_tf32(X[4 * S::LDT + 8 * I], h1[I], l1[I]);
  }
#pragma unroll
  for (int k = 0; k < S::NP; ++k) {
    const int u = 2 * k, v = 2 * k + 1 < g ? 2 * k + 1 : 2 * k;
#pragma unroll
    for (int J0 = 0; J0 < g; J0 += 4) {
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

// o = sum over ratings [e0, e1) of x x^T
template <int g, int V>
__device__ __forceinline__ void sm_gram_v(const SweepArgs& a, float* T, int64_t e0, int64_t e1, int lane,
                                          float (&o)[SmGeom<g>::NA][4]) {
  using S = SmGeom<g>;
  constexpr int kBuf = kSmChunk * S::LDT;
  const int K = a.K;
  const int64_t n = e1 - e0;
  const float* X = T + (lane & 3) * S::LDT + (lane >> 2);
  // ids and ratings of the chunk after the one being staged, a lane each
  int j = 0;
  float r = 0.f;
  auto load = [&](int64_t c0) {
    j = 0;
    r = 0.f;
    if (lane < kSmChunk && c0 + lane < n) {
      j = __ldg(a.idx + e0 + c0 + lane);
      r = __ldg(a.val + e0 + c0 + lane);
    }
  };
  auto count = [&](int64_t c0) { return (int)min((int64_t)kSmChunk, n - c0); };
  if (n <= 0) return;
  load(0);
  sm_stage<g, V>(a.Vo, K, T, j, r, count(0), lane);
  load(kSmChunk);
  int buf = 0;
  for (int64_t c0 = 0; c0 < n; c0 += kSmChunk, buf ^= 1) {
    if (c0 + kSmChunk < n) {
      sm_stage<g, V>(a.Vo, K, T + (buf ^ 1) * kBuf, j, r, count(c0 + kSmChunk), lane);
      load(c0 + 2 * kSmChunk);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncwarp();
    sm_step<g>(X + buf * kBuf, o);
    if (count(c0) > 8) sm_step<g>(X + buf * kBuf + 8 * S::LDT, o);
    __syncwarp();  // the buffer is refilled next
  }
}

template <int g>
__device__ __forceinline__ void sm_gram(const SweepArgs& a, float* T, int64_t e0, int64_t e1, int lane,
                                        float (&o)[SmGeom<g>::NA][4]) {
  using S = SmGeom<g>;
#pragma unroll
  for (int i = 0; i < S::NA; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) o[i][q] = 0.f;
  // the columns past the rating stay zero in both buffers
  for (int e = lane; e < 2 * kSmChunk; e += 32) {
#pragma unroll
    for (int c = S::KP - 8; c < S::KP; ++c)
      if (c > a.K) T[e * S::LDT + c] = 0.f;
  }
  __syncwarp();
  if ((a.K & 3) == 0) sm_gram_v<g, 4>(a, T, e0, e1, lane, o);
  else if ((a.K & 1) == 0) sm_gram_v<g, 2>(a, T, e0, e1, lane, o);
  else sm_gram_v<g, 1>(a, T, e0, e1, lane, o);
}

template <int g>
__global__ void __launch_bounds__(32 * kSmWarps, sm_ctas(g)) row_small(const SweepArgs a) {
  using S = SmGeom<g>;
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
    float o[S::NA][4];
    sm_gram<g>(a, T, a.ptr[row], a.ptr[row + 1], lane, o);
    // A = base + alpha G as tiles, over the staging buffers
    const int gr = lane >> 2, t2 = 2 * (lane & 3), fo = trow(gr) + t2;
#pragma unroll
    for (int k = 0; k < S::NP; ++k)
#pragma unroll
      for (int J = 0; J < g; ++J)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int I = 2 * k + h;
          if (J <= I && I < g) {
            const int off = tidx(I, J) * kTileF + fo;
            const float2 b = ldf2(base + off);
            const float x = fmaf(a.alpha, o[k * (k + 1) + J][2 * h], b.x);
            const float y = fmaf(a.alpha, o[k * (k + 1) + J][2 * h + 1], b.y);
            *reinterpret_cast<float2*>(T + off) = make_float2(x, y);
            if (J == I && (gr & ~1) == t2)
              thr[8 * I + gr] = 8 * I + gr < a.K ? pivot_threshold(a.pivot_rel, gr & 1 ? y : x) : -INFINITY;
          }
        }
  }
  __syncwarp();
  row_draw(a, g, T, thr, rinv, zv, row, lane);
}

// Partial Gram of one piece of a split row by one warp, stored as raw tiles in
// the numbering of tile_chol.cuh.
template <int g>
__global__ void __launch_bounds__(32 * kSmWarps, sm_ctas(g)) piece_small(const SweepArgs a, int64_t npieces) {
  using S = SmGeom<g>;
  extern __shared__ __align__(16) float ssm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t pc = (int64_t)blockIdx.x * kSmWarps + warp;
  if (pc >= npieces) return;
  float o[S::NA][4];
  sm_gram<g>(a, ssm + warp * S::kStage, a.piece_e0[pc], a.piece_e1[pc], lane, o);
  float* dst = a.part + pc * S::NT * 64 + 2 * lane;
#pragma unroll
  for (int k = 0; k < S::NP; ++k)
#pragma unroll
    for (int J = 0; J < g; ++J)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int I = 2 * k + h;
        if (J <= I && I < g)
          *reinterpret_cast<float2*>(dst + tile_id(I, J, g) * 64) =
              make_float2(o[k * (k + 1) + J][2 * h], o[k * (k + 1) + J][2 * h + 1]);
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
  if (threadIdx.x < 32) row_draw(a, g, T, thr, rinv, zv, a.rows ? a.rows[slot] : (int)slot, threadIdx.x);
}

template <int g>
int launch_small(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  using S = SmGeom<g>;
  const int smem = (S::NT * kTileF + kSmWarps * S::kFloats) * (int)sizeof(float);
  BPMF_CUDA_CHECK(cudaFuncSetAttribute(row_small<g>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  const int64_t n = a.row_end - a.row_begin;
  for (int64_t off = 0; off < n; off += (int64_t)kSmWarps << 27) {
    SweepArgs b = a;
    b.row_begin = a.row_begin + off;
    b.row_end = b.row_begin + std::min<int64_t>(n - off, (int64_t)kSmWarps << 27);
    const int64_t blocks = (b.row_end - b.row_begin + kSmWarps - 1) / kSmWarps;
    row_small<g><<<(unsigned)blocks, 32 * kSmWarps, smem, st>>>(b);
    BPMF_CUDA_CHECK(cudaGetLastError());
    if (launches) *launches += 1;
  }
  return BPMF_OK;
}

template <int g>
int launch_small_pieces(const SweepArgs& a, int64_t npieces, cudaStream_t st, int64_t* launches) {
  using S = SmGeom<g>;
  const int smem = kSmWarps * S::kStage * (int)sizeof(float);
  BPMF_CUDA_CHECK(cudaFuncSetAttribute(piece_small<g>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  piece_small<g><<<(unsigned)((npieces + kSmWarps - 1) / kSmWarps), 32 * kSmWarps, smem, st>>>(a, npieces);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

}  // namespace

bool small_supported(int K) { return K >= 1 && (K + 8) / 8 <= kSmMaxG; }

int launch_rows_small(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  if (a.row_end <= a.row_begin) return BPMF_OK;
  switch ((a.K + 8) / 8) {
    case 1: return launch_small<1>(a, st, launches);
    case 2: return launch_small<2>(a, st, launches);
    case 3: return launch_small<3>(a, st, launches);
    case 4: return launch_small<4>(a, st, launches);
    case 5: return launch_small<5>(a, st, launches);
    case 6: return launch_small<6>(a, st, launches);
    case 7: return launch_small<7>(a, st, launches);
    default: return BPMF_EINVAL;
  }
}

int launch_pieces_small(const SweepArgs& a, int64_t npieces, cudaStream_t st, int64_t* launches) {
  if (npieces <= 0) return BPMF_OK;
  switch ((a.K + 8) / 8) {
    case 1: return launch_small_pieces<1>(a, npieces, st, launches);
    case 2: return launch_small_pieces<2>(a, npieces, st, launches);
    case 3: return launch_small_pieces<3>(a, npieces, st, launches);
    case 4: return launch_small_pieces<4>(a, npieces, st, launches);
    case 5: return launch_small_pieces<5>(a, npieces, st, launches);
    case 6: return launch_small_pieces<6>(a, npieces, st, launches);
    case 7: return launch_small_pieces<7>(a, npieces, st, launches);
    default: return BPMF_EINVAL;
  }
}

int64_t partial_floats_per_piece(int K) {
  const int g = (K + 8) / 8;
  return (int64_t)g * (g + 1) / 2 * 64;
}

int launch_hub_draw(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  const int64_t n = a.row_end - a.row_begin;
  if (n <= 0) return BPMF_OK;
  const int g = (a.K + 8) / 8;
  const int smem = (g * (g + 1) / 2 * kTileF + 3 * 8 * g) * (int)sizeof(float);
  BPMF_CUDA_CHECK(cudaFuncSetAttribute(hub_draw, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  hub_draw<<<(unsigned)n, kHubThreads, smem, st>>>(a);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

}  // namespace gb
