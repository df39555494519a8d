// rows.cu -- per-row conditional draws of one side (Algorithm 1's "update
// movie m / user u based on the ratings for it and the model of the other
// side, plus randomly sampled noise") on the FP32 CUDA cores, the partial
// Grams of split rows, the FP64 redo of rows whose FP32 pivot fails, and the
// initial factors.
//
// For row i with rated neighbours j (rows of the other side, factors v_j)
// and centred ratings r_ij:
//   Lambda* = Lambda_s + alpha sum_j v_j v_j^T      (K x K, SPD)
//   b       = Lambda_s mu_s + alpha sum_j r_ij v_j
//   L = chol(Lambda*) (lower), y = L^-1 b, u_i = L^-T (y + z)
// with z the K Philox normals of (seed, iteration, side, i).  u_i has mean
// Lambda*^-1 b and covariance Lambda*^-1.  Rows of one side are independent
// given the other side (paper Sec. III), so every row is a unit of work.
//
// Gram: each staged neighbour row carries its rating as feature K, so one
// symmetric Gram of the (K+1)-vectors x_j = [v_j, r_ij] gives both
// sum v_j v_j^T and sum r_ij v_j (its last row).  Rows are staged 32 at a
// time in shared memory with cp.async, double-buffered, and accumulated in
// FP32 register tiles, a thread per tile (tile_chol.cuh numbers them); the
// bordered matrix is then factored from shared memory by one warp
// (warp_chol.cuh).  Latent dimensions up to 55 take rows_small.cu instead.
#include <cuda_runtime.h>

#include <algorithm>

#include "bpmf_impl.cuh"
#include "rows.cuh"
#include "tile_chol.cuh"
#include "warp_chol.cuh"

namespace gb {
namespace {

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Stages neighbour rows [e0, e0 + cnt) as (K+1)-vectors [v_j, r] at stride KPs;
// thread t copies pieces t, t + nt, .. of the rows, stepped without divisions.
__device__ __forceinline__ void stage_rows(const SweepArgs& a, int KPs, float* dst, int64_t e0,
                                           int cnt) {
  const int K = a.K, nt = blockDim.x, t = threadIdx.x;
  const bool vec = (K & 3) == 0;
  const int P = vec ? K >> 2 : K;
  const int dr = nt / P, dq = nt - dr * P;
  int rr = t / P, q = t - rr * P;
  while (rr < cnt) {
    const int64_t j = a.idx[e0 + rr];
    if (vec) cp_async16(dst + rr * KPs + 4 * q, a.Vo + j * K + 4 * q);
    else cp_async4(dst + rr * KPs + q, a.Vo + j * K + q);
    rr += dr;
    q += dq;
    if (q >= P) {
      q -= P;
      ++rr;
    }
  }
  for (int r2 = t; r2 < cnt; r2 += nt) cp_async4(dst + r2 * KPs + K, a.val + e0 + r2);
  cp_async_commit();
}

// Two FP32 fused multiply-adds in one instruction (d0 += a b0, d1 += a b1),
// each rounded as fmaf rounds it.
__device__ __forceinline__ void ffma2(float& d0, float& d1, float a, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rc;\n\t"
      "mov.b64 ra, {%2, %2};\n\t"
      "mov.b64 rb, {%3, %4};\n\t"
      "mov.b64 rc, {%0, %1};\n\t"
      "fma.rn.f32x2 rc, ra, rb, rc;\n\t"
      "mov.b64 {%0, %1}, rc;\n\t}"
      : "+f"(d0), "+f"(d1)
      : "f"(a), "f"(b0), "f"(b1));
}

// acc += sum over ratings [e0, e1) of x_j x_j^T (lower tiles, FP32).
__device__ __forceinline__ void gram_gather(const SweepArgs& a, const TileGeom& G, float* Vs,
                                            int64_t e0, int64_t e1, bool active, int ty, int tx,
                                            float (&acc)[8][8]) {
  constexpr int TM = 8;
  const int KPs = G.KPs;
  const int buf_floats = kChunk * KPs;
  // padding columns K+1 .. KPs-1 stay zero (cp.async writes columns 0..K only)
  const int pad = KPs - (a.K + 1);
  for (int e = threadIdx.x; e < 2 * kChunk * pad; e += blockDim.x) {
    const int rr = e / pad;
    Vs[rr * KPs + a.K + 1 + (e - rr * pad)] = 0.f;
  }
  const int64_t n = e1 - e0;
  const int64_t nch = (n + kChunk - 1) / kChunk;
  if (nch > 0) stage_rows(a, KPs, Vs, e0, (int)(n < kChunk ? n : kChunk));
  for (int64_t c = 0; c < nch; ++c) {
    if (c + 1 < nch) {
      const int64_t s0 = e0 + (c + 1) * kChunk;
      stage_rows(a, KPs, Vs + ((c + 1) & 1) * buf_floats, s0, (int)(e1 - s0 < kChunk ? e1 - s0 : kChunk));
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int cnt = (int)(n - c * kChunk < kChunk ? n - c * kChunk : kChunk);
    const float* B = Vs + (c & 1) * buf_floats;
    if (active) {
      for (int rr = 0; rr < cnt; ++rr) {
        float va[TM], vb[TM];
        ld8(B + rr * KPs + ty * TM, va);
        ld8(B + rr * KPs + tx * TM, vb);
#pragma unroll
        for (int p = 0; p < TM; ++p)
#pragma unroll
          for (int q = 0; q < TM; q += 2) ffma2(acc[p][q], acc[p][q + 1], va[p], vb[q], vb[q + 1]);
      }
    }
    __syncthreads();
  }
}

// the tiles reuse the staging buffers; thresholds, 1 / diagonal and z follow
int smem_bytes_fp32(const TileGeom& G) {
  return (int)sizeof(float) * (std::max(2 * kChunk * G.KPs, G.ntiles * kTileF) + 3 * G.KP);
}

}  // namespace

// A row of latent dimension past rows_small.cu's by one CTA: the Gram in
// register tiles, then the tiles go to shared memory and one warp factors them
// and draws.  30,000 rows of 100 ratings: K = 64 1,717 -> 1,050 us, K = 100
// 3,576 -> 1,756, K = 128 7,743 -> 3,391, the factorisation by the whole CTA
// with two barriers a panel before.
__global__ void __launch_bounds__(160) row_fp32(const SweepArgs a) {
  extern __shared__ __align__(16) float smem[];
  const TileGeom G(a.K, 8);
  const int64_t slot = a.row_begin + blockIdx.x;
  if (slot >= a.row_end) return;
  const int row = a.rows ? a.rows[slot] : (int)slot;
  const int tid = threadIdx.x;
  const bool active = tid < G.ntiles;
  int ty = 0, tx = 0;
  if (active) tri_tile(tid, G.g, ty, tx);
  float acc[8][8];
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[p][q] = 0.f;
  gram_gather(a, G, smem, a.ptr[row], a.ptr[row + 1], active, ty, tx, acc);
  __syncthreads();  // a row without ratings has met no barrier since it zeroed the padding
  float* T = smem;
  float* thr = smem + max(2 * kChunk * G.KPs, G.ntiles * kTileF);
  if (active) {
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      float x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = row_elem(a, 8 * ty + p, 8 * tx + q, acc[p][q]);
      st8(T + tidx(ty, tx) * kTileF + trow(p), x);
      if (ty == tx)
        thr[8 * ty + p] = 8 * ty + p < a.K ? pivot_threshold(a.pivot_rel, x[p]) : -INFINITY;
    }
  }
  __syncthreads();
  if (tid < 32) row_draw<2>(a, G.g, T, thr, thr + G.KP, thr + 2 * G.KP, row, tid);
}

// Partial Gram of one piece of a split row, stored as raw tiles.
__global__ void __launch_bounds__(160) piece_fp32(const SweepArgs a) {
  extern __shared__ __align__(16) float smem[];
  const TileGeom G(a.K, 8);
  const int64_t pc = blockIdx.x;
  const int tid = threadIdx.x;
  const bool active = tid < G.ntiles;
  int ty = 0, tx = 0;
  if (active) tri_tile(tid, G.g, ty, tx);
  float acc[8][8];
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[p][q] = 0.f;
  gram_gather(a, G, smem, a.piece_e0[pc], a.piece_e1[pc], active, ty, tx, acc);
  if (active) {
    float* dst = a.part + (pc * G.ntiles + tid) * 64;
#pragma unroll
    for (int p = 0; p < 8; ++p) st8(dst + 8 * p, acc[p]);
  }
}

// FP64 redo of flagged rows: one CTA per row, Lambda* and b rebuilt in FP64
// from the FP64 hyperparameters, Cholesky and solves in FP64 in shared
// memory, normals in FP64.  A failed FP64 pivot flags kStatusNotPD.
// The last block to have read the count publishes it and zeroes it and the
// persistent kernel's row counter for the next sweep.
__global__ void __launch_bounds__(256) row_fp64(const SweepArgs a, const double* __restrict__ lam,
                                                const double* __restrict__ mu, int* status,
                                                int32_t* redo_count, int* ticket, int* ws_counter) {
  extern __shared__ double dsm[];
  const int K = a.K;
  double* A = dsm;            // K*K
  double* b = A + K * K;      // K
  double* y = b + K;          // K
  __shared__ int bad;
  const int nflag = *a.flag_count;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ticket, 1) == (int)gridDim.x - 1) {
      *redo_count = nflag;
      *a.flag_count = 0;
      *ws_counter = 0;
      *ticket = 0;
    }
  }
  for (int f = blockIdx.x; f < nflag; f += gridDim.x) {
    const int row = a.flag_rows[f];
    const int64_t p0 = a.ptr[row], p1 = a.ptr[row + 1];
    __syncthreads();
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
      const int i = e / K, j = e % K;
      double s = 0.0;
      if (j <= i)
        for (int64_t q = p0; q < p1; ++q) {
          const float* v = a.Vo + (int64_t)a.idx[q] * K;
          s += (double)v[i] * (double)v[j];
        }
      A[e] = lam[e] + (double)a.alpha * s;
    }
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      double s = 0.0, t = 0.0;
      for (int64_t q = p0; q < p1; ++q)
        s += (double)a.val[q] * (double)a.Vo[(int64_t)a.idx[q] * K + i];
      for (int k = 0; k < K; ++k) t += lam[i * K + k] * mu[k];
      b[i] = t + (double)a.alpha * s;
    }
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    for (int k = 0; k < K; ++k) {
      const double piv = A[k * K + k];
      __syncthreads();
      if (!(piv > 0.0) && threadIdx.x == 0) bad = 1;
      const double d = piv > 0.0 ? sqrt(piv) : 1.0;
      for (int i = k + 1 + threadIdx.x; i < K; i += blockDim.x) A[i * K + k] /= d;
      if (threadIdx.x == 0) A[k * K + k] = d;
      __syncthreads();
      const int m = K - k - 1;
      for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = k + 1 + e / m, j = k + 1 + e % m;
        if (j <= i) A[i * K + j] -= A[i * K + k] * A[j * K + k];
      }
      __syncthreads();
    }
    if (bad) {
      if (threadIdx.x == 0) atomicOr(status, kStatusNotPD);
      continue;
    }
    if (threadIdx.x == 0) {
      for (int i = 0; i < K; ++i) {
        double t = b[i];
        for (int k = 0; k < i; ++k) t -= A[i * K + k] * y[k];
        y[i] = t / A[i * K + i];
      }
      for (int i = 0; i < K; ++i) y[i] += normal_at_f64(a.key, (uint32_t)row, *a.tp, a.sw, (uint32_t)i);
      for (int i = K - 1; i >= 0; --i) {
        double t = y[i];
        for (int k = i + 1; k < K; ++k) t -= A[k * K + i] * b[k];
        b[i] = t / A[i * K + i];
      }
      for (int i = 0; i < K; ++i) {
        a.X[(int64_t)row * K + i] = (float)b[i];
        write_shadow(a, row, i, (float)b[i]);
      }
    }
  }
}

__global__ void init_factors_kernel(float* X, int64_t R, int K, uint2 key, uint32_t sw) {
  const int Q = (K + 3) / 4;
  const int64_t total = R * Q;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / Q;
    const int q = (int)(e - i * Q);
    const float4 z = normal4_f32(philox(make_uint4((uint32_t)i, 0u, (uint32_t)q, sw), key));
    const float zz[4] = {z.x, z.y, z.z, z.w};
    for (int w = 0; w < 4; ++w)
      if (4 * q + w < K) X[i * K + 4 * q + w] = 0.1f * zz[w];
  }
}

int launch_rows_fp32(const SweepArgs& a, cudaStream_t st, int64_t* launches) {
  if (small_supported(a.K)) return launch_rows_small(a, st, launches);
  const int64_t nrows = a.row_end - a.row_begin;
  if (nrows <= 0) return BPMF_OK;
  const TileGeom G(a.K, 8);
  const int smem = smem_bytes_fp32(G);
  BPMF_TRY(allow_smem(row_fp32, smem_bytes_fp32(TileGeom(kMaxK, 8))));
  for (int64_t off = 0; off < nrows; off += 1LL << 30) {
    SweepArgs b = a;
    b.row_begin = a.row_begin + off;
    b.row_end = b.row_begin + std::min<int64_t>(nrows - off, 1LL << 30);
    row_fp32<<<(unsigned)(b.row_end - b.row_begin), G.nthreads, smem, st>>>(b);
    BPMF_CUDA_CHECK(cudaGetLastError());
    if (launches) *launches += 1;
  }
  return BPMF_OK;
}

int launch_pieces_fp32(const SweepArgs& a, int64_t npieces, cudaStream_t st, int64_t* launches) {
  if (small_supported(a.K)) return launch_pieces_small(a, npieces, st, launches);
  if (npieces <= 0) return BPMF_OK;
  const TileGeom G(a.K, 8);
  const int smem = (int)sizeof(float) * 2 * kChunk * G.KPs;
  BPMF_TRY(allow_smem(piece_fp32, sizeof(float) * 2 * kChunk * TileGeom(kMaxK, 8).KPs));
  piece_fp32<<<(unsigned)npieces, G.nthreads, smem, st>>>(a);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

SweepArgs make_sweep_args(Handle* h, int s) {
  SideDev& sd = h->side[s];
  SideDev& od = h->side[1 - s];
  SweepArgs a{};
  a.ptr = sd.ptr;
  a.idx = sd.idx;
  a.val = sd.val;
  a.Vo = od.X;
  a.X = sd.X;
  a.lamaug = sd.lamaug;
  a.rows = nullptr;
  a.row_begin = 0;
  a.row_end = sd.R;
  a.K = h->K;
  a.alpha = (float)h->cfg.alpha;
  a.key = seed_key(h->cfg.seed);
  a.tp = h->d_iter;
  a.sw = stream_word(kStreamRow, s);
  a.flag_rows = h->flag_rows;
  a.flag_count = h->flag_count;
  a.pivot_rel = (float)h->cfg.pivot_rel;
  a.wait_ns = h->wait_ns;
  a.hold_arrive = h->hold_arrive;
  a.piece_row = sd.piece_row;
  a.piece_e0 = sd.piece_e0;
  a.piece_e1 = sd.piece_e1;
  a.hub_piece0 = sd.hub_piece0;
  a.part = h->hub_part;
  a.work = sd.work;
  a.Vhi = od.Xhi;
  a.Vlo = od.Xlo;
  a.Xhi = sd.Xhi;
  a.Xlo = sd.Xlo;
  a.KS = od.KS;
  a.n_other = od.R;
  return a;
}

int launch_fp64_redo(Handle* h, int s, const SweepArgs& a) {
  const size_t smem = sizeof(double) * ((size_t)h->K * h->K + 2 * h->K);
  BPMF_TRY(allow_smem(row_fp64, sizeof(double) * (kMaxK * kMaxK + 2 * kMaxK)));
  row_fp64<<<h->num_sms, 256, smem, h->stream>>>(a, h->side[s].lam, h->side[s].mu, h->status,
                                                   h->redo_count, h->redo_ticket, h->ws_counter);
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

int clear_sweep_counts(Handle* h) {
  BPMF_CUDA_CHECK(cudaMemsetAsync(h->flag_count, 0, sizeof(int32_t), h->stream));
  BPMF_CUDA_CHECK(cudaMemsetAsync(h->ws_counter, 0, sizeof(int), h->stream));
  return BPMF_OK;
}

int launch_sweep(Handle* h, int s) {
  cudaStream_t st = h->stream;
  SweepArgs a = make_sweep_args(h, s);
  int rc = BPMF_OK;
  {
    PhaseTimer timer(h, s == BPMF_USERS ? BPMF_T_ROWS_USERS : BPMF_T_ROWS_MOVIES);
    if (h->cfg.path == BPMF_PATH_PLAIN) {
      rc = launch_rows_fp32(a, st, &h->kernels);
    } else {
      rc = launch_sweep_binned(h, s, a);
    }
  }
  if (rc != BPMF_OK) {  // the redo will not take these back
    clear_sweep_counts(h);
    return rc;
  }
  PhaseTimer timer(h, BPMF_T_FP64_REDO);
  BPMF_TRY(launch_fp64_redo(h, s, a));
  h->kernels += 1;
  return BPMF_OK;
}

int launch_init_factors(Handle* h, int s) {
  SideDev& sd = h->side[s];
  const int Q = (h->K + 3) / 4;
  const int64_t total = sd.R * Q;
  int64_t g = (total + 255) / 256;
  if (g > 8 * 1024) g = 8 * 1024;
  if (g < 1) g = 1;
  init_factors_kernel<<<(unsigned)g, 256, 0, h->stream>>>(sd.X, sd.R, h->K, seed_key(h->cfg.seed),
                                                          stream_word(kStreamInit, s));
  BPMF_CUDA_CHECK(cudaGetLastError());
  return BPMF_OK;
}

}  // namespace gb
