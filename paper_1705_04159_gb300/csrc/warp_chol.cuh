// warp_chol.cuh -- one row's factorisation and draw by one warp, on 8 x 8 FP32
// tiles in shared memory.
//
// The bordered matrix [[Lambda*, b], [b^T, inf]] ((K + 1) x (K + 1), padded with
// the identity to 8 g, lower triangle) lies as tiles (I, J), J <= I < g, at
// kTileF (I (I + 1) / 2 + J); its factor's row K is y = L^-1 b, and the draw is
// u = L^-T (y + z).
//
// The factorisation is left-looking by block columns J of eight columns:
//   update: A_IJ -= sum_{p<J} L_Ip L_Jp^T for all row tiles I >= J, on the
//     tensor cores by mma.m16n8k8 (two row tiles at a time) with FP32 operands
//     split into two TF32 parts, x = h + l: h h^T in one or two FP32 accumulators
//     and h l^T + l h^T in another (l l^T, at most 2^-22 relative, is dropped), so
//     only the p-sums of like size meet in an accumulator.  The tensor core's sums
//     round towards zero: over the 16 steps of K = 128 one accumulator's bias put a
//     draw up to 1.33 times as far from FP64 as FP32 multiply-adds (rms, K >= 88, 8 to
//     64 ratings under a well-conditioned prior), two in turn, each of half the
//     steps and half the size, at most 0.96 times.  K <= 55, where one stays within
//     1.0 times, and the persistent kernel, whose bf16 Gram sets its error (1.00 times;
//     rows without ratings 0.6 to 0.96), take one (W): with two there, 50,000 x 12,000
//     with 2.5M ratings, K = 64, 2,309 -> 2,397 us for two iterations;
//   diagonal tile: Cholesky in registers by every lane;
//   panel: the rows below by substitution, a lane per row.
// A tile is 8 rows of 8 floats (trow), and a lane's fragment of an operand or
// an accumulator is the same pair of neighbouring floats everywhere: column
// pair t of row g (lane 4 g + t), taking the operands' k index t for column 2t
// and t + 4 for column 2t + 1.  So tiles are loaded by 8-byte conflict-free
// loads and never rearranged.
// What bounds it: instruction issue and latency of one warp (at K = 100, about
// 14k warp instructions and 3.7k shared-memory wavefronts a row; the
// right-looking FP32 form before it needed 17.2k and 7.3k, and its wavefronts
// alone were 72% of what the SM can serve).  Six rows side by side on an SM,
// nothing else running: 5.43 -> 4.15 us per row at K = 100, 2.80 -> 2.10 at
// K = 64, 1.28 -> 0.96 at K = 32; error of the draws against FP64 2.8e-7 ->
// 2.4e-7, 2.1e-7 -> 1.7e-7 and 1.4e-7 -> 1.2e-7.  Two pairs of row tiles per
// step of the update measured as fast as three and faster than four (4.29 us
// at K = 100, 2.26 at K = 64), in fewer registers.
#pragma once

#include <math.h>
#include <stdint.h>

#include "bpmf_impl.cuh"
#include "rows.cuh"

namespace gb {

constexpr int kTileF = 68;  // floats per 8 x 8 tile (see trow)

// Offset of row r in a tile: rows 0-3 at 8 r, rows 4-7 four floats further, so
// that eight lanes' 16-byte accesses to the same half of a tile's eight rows
// (the drain's stores, the panel's loads and stores) fall on different banks.
// Tiles are 68 floats apart, so consecutive tile bases fall on eight
// different bank groups.
__host__ __device__ __forceinline__ int trow(int r) { return r * 8 + ((r >> 2) << 2); }

__device__ __forceinline__ void ld8(const float* p, float (&x)[8]) {
  const float4 u = reinterpret_cast<const float4*>(p)[0];
  const float4 v = reinterpret_cast<const float4*>(p)[1];
  x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
  x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
}
__device__ __forceinline__ void st8(float* p, const float (&x)[8]) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
}

__device__ __forceinline__ int tidx(int I, int J) { return I * (I + 1) / 2 + J; }

__device__ __forceinline__ float2 ldf2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// D += A B on 16 x 8 x 8 elements, TF32 operands, FP32 accumulator
__device__ __forceinline__ void mma_tf32(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// x = h + l: h to the nearest TF32 value (10 fraction bits), l the exact rest,
// whose own TF32 part the tensor core reads
__device__ __forceinline__ void split_tf32(float x, uint32_t& h, uint32_t& l) {
  h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  l = __float_as_uint(x - __uint_as_float(h));
}

__device__ __forceinline__ float rsqrt_normal(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// A_IJ -= sum_{p<J} L_Ip L_Jp^T for the 2 NPR row tiles I = I0 .. (those below
// g; pairs wholly past it compute on the last tile and store nothing), the
// steps p taking W accumulators in turn.  The next step's fragments are loaded as
// soon as the current ones are split, so after the last step they are those of
// column J itself.
template <int NPR, int W>
__device__ __forceinline__ void warp_update(float* T, int g, int J, int I0, int fo) {
  float acc[W][NPR][4], cross[NPR][4];
  float2 fu[NPR], fv[NPR];
  float *pu[NPR], *pv[NPR];
#pragma unroll
  for (int i = 0; i < NPR; ++i) {
    const int I = min(I0 + 2 * i, g - 1);
    pu[i] = T + tidx(I, 0) * kTileF + fo;
    pv[i] = I + 1 < g ? pu[i] + (I + 1) * kTileF : pu[i];
    fu[i] = ldf2(pu[i]);
    fv[i] = ldf2(pv[i]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cross[i][q] = 0.f;
#pragma unroll
      for (int w = 0; w < W; ++w) acc[w][i][q] = 0.f;
    }
  }
  const float* pb = T + tidx(J, 0) * kTileF + fo;
  float2 b = ldf2(pb);
  int off = 0;
#pragma unroll 1
  for (int p = 0; p < J; p += W) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w > 0 && p + w >= J) break;
      off += kTileF;
      uint32_t bh0, bl0, bh1, bl1;
      split_tf32(b.x, bh0, bl0);
      split_tf32(b.y, bh1, bl1);
      b = ldf2(pb + off);
      uint32_t l[NPR][4];
#pragma unroll
      for (int i = 0; i < NPR; ++i) {
        uint32_t h0, h1, h2, h3;
        split_tf32(fu[i].x, h0, l[i][0]);
        split_tf32(fv[i].x, h1, l[i][1]);
        split_tf32(fu[i].y, h2, l[i][2]);
        split_tf32(fv[i].y, h3, l[i][3]);
        fu[i] = ldf2(pu[i] + off);
        fv[i] = ldf2(pv[i] + off);
        mma_tf32(acc[w][i], h0, h1, h2, h3, bh0, bh1);
        mma_tf32(cross[i], h0, h1, h2, h3, bl0, bl1);
      }
#pragma unroll
      for (int i = 0; i < NPR; ++i)
        mma_tf32(cross[i], l[i][0], l[i][1], l[i][2], l[i][3], bh0, bh1);
    }
  }
#pragma unroll
  for (int i = 0; i < NPR; ++i) {
    const int I = I0 + 2 * i;
    float s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[q] = cross[i][q];
#pragma unroll
      for (int w = W - 1; w >= 0; --w) s[q] = acc[w][i][q] + s[q];
    }
    if (I < g) *reinterpret_cast<float2*>(pu[i] + off) = make_float2(fu[i].x - s[0], fu[i].y - s[1]);
    if (I + 1 < g) *reinterpret_cast<float2*>(pv[i] + off) = make_float2(fv[i].x - s[2], fv[i].y - s[3]);
  }
}

// x L_JJ^T = a for rows r0 .. nr - 1 (at most 32 N of them) of those below the
// diagonal tile, N rows per lane side by side
template <int N>
__device__ __forceinline__ void warp_panel(int r0, int nr, int J, float* T, const float (&d)[8][8],
                                         const float (&rdv)[8], int lane) {
  float x[N][8];
  float* row[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const int rr = r0 + lane + 32 * k, I = J + 1 + (rr >> 3);
    row[k] = T + tidx(I, J) * kTileF + trow(rr & 7);
    if (rr < nr) ld8(row[k], x[k]);
  }
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int k = 0; k < N; ++k) {
      x[k][c] *= rdv[c];
#pragma unroll
      for (int s = c + 1; s < 8; ++s) x[k][s] = fmaf(-x[k][c], d[s][c], x[k][s]);
    }
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (r0 + lane + 32 * k < nr) st8(row[k], x[k]);
}

// Left-looking Cholesky of g x g tiles (lower triangle) by one warp.  Returns false if a
// pivot met the pivot rule of tile_chol.cuh (at or below thr, formed from its
// starting diagonal; -inf on the bordered row K and on the padding: row K's
// starting diagonal is infinite, so its pivot is too, whatever y^T y it loses, with
// the reciprocal root 0, and the padding keeps its ones).  The diagonals
// themselves are not stored; rinv holds their reciprocals.
template <int W>
__device__ __forceinline__ bool warp_cholesky(int g, float* T, const float* thr_s, float* rinv,
                                              int lane) {
  bool fail = false;
  const int fo = trow(lane >> 2) + 2 * (lane & 3);
#pragma unroll 1
  for (int J = 0; J < g; ++J) {
    if (J > 0) {
      int I0 = J;
#pragma unroll 1
      for (; g - I0 > 2; I0 += 4) warp_update<2, W>(T, g, J, I0, fo);
      if (g - I0 > 0) warp_update<1, W>(T, g, J, I0, fo);
      __syncwarp();
    }
    float* D = T + tidx(J, J) * kTileF;
    float d[8][8], rdv[8], thr[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) ld8(D + trow(i), d[i]);
    ld8(thr_s + 8 * J, thr);
    __syncwarp();  // every lane has loaded the tile that every lane writes below
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      // A failed pivot leaves NaN or inf in the rest of the factorisation,
      // which is discarded with the row (the FP64 redo draws it).  A pivot
      // that passes is a normal number, where the flushing root is the same.
      const float piv = d[c][c];
      fail = fail || !(piv > thr[c]);
      const float rd = rsqrt_normal(piv);
      rdv[c] = rd;
#pragma unroll
      for (int i = c + 1; i < 8; ++i) d[i][c] *= rd;
#pragma unroll
      for (int j = c + 1; j < 8; ++j)
#pragma unroll
        for (int i = j; i < 8; ++i) d[i][j] = fmaf(-d[i][c], d[j][c], d[i][j]);
    }
    // every lane holds the same factor, so every lane writes it: same
    // address, same value, no divergent stores
#pragma unroll
    for (int i = 1; i < 8; ++i) {
      float4* dst = reinterpret_cast<float4*>(D + trow(i));
      dst[0] = make_float4(d[i][0], d[i][1], d[i][2], d[i][3]);
      if (i > 4) dst[1] = make_float4(d[i][4], d[i][5], d[i][6], d[i][7]);
    }
    st8(rinv + 8 * J, rdv);
    const int nr = 8 * (g - 1 - J);
#pragma unroll 1
    for (int r0 = 0; r0 < nr; r0 += 64) warp_panel<2>(r0, nr, J, T, d, rdv, lane);
    __syncwarp();
  }
  return !fail;
}

// u = L^-T (y + z), y row K of the factor, by 8-row blocks from the bottom:
// lane 2 J + h keeps columns 8 J + 4 h .. + 3 (so one pass covers all of a
// row), the block's eight values come to every lane by shuffles, every lane
// solves the 8 x 8 system, and each subtracts the block's part from its
// columns.  The next block's diagonal tile is loaded a step ahead; the other
// tiles are not, which would take 32 registers more.
__device__ __forceinline__ void warp_back(const SweepArgs& a, const float* T, const float* rinv,
                                          const float* zv, int row, int lane) {
  const int K = a.K;
  float* out = a.X + (int64_t)row * K;
  const int J = lane >> 1, h4 = (lane & 1) << 2;
  const int IK = K >> 3, pk = K & 7;
  float v[4];
  {
    const float4 y = *reinterpret_cast<const float4*>(
        T + (J <= IK ? tidx(IK, J) * kTileF + trow(pk) + h4 : 0));
    const float4 z = *reinterpret_cast<const float4*>(zv + (J <= IK ? 8 * J + h4 : 0));
    v[0] = y.x + z.x; v[1] = y.y + z.y; v[2] = y.z + z.z; v[3] = y.w + z.w;
  }
  float d[8][8], rd[8];  // the strict lower triangle of tile (I, I), 1 / diagonal
  auto load_diag = [&](int I) {
    const float* Dg = T + tidx(I, I) * kTileF;
#pragma unroll
    for (int r = 1; r < 8; ++r) {
      const float4 a = *reinterpret_cast<const float4*>(Dg + trow(r));
      d[r][0] = a.x; d[r][1] = a.y; d[r][2] = a.z; d[r][3] = a.w;
      if (r > 4) {
        const float4 b = *reinterpret_cast<const float4*>(Dg + trow(r) + 4);
        d[r][4] = b.x; d[r][5] = b.y; d[r][6] = b.z; d[r][7] = b.w;
      }
    }
    ld8(rinv + 8 * I, rd);
  };
  int I = (K - 1) >> 3;
  load_diag(I);
#pragma unroll 1
  for (; I >= 0; --I) {
    float u[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) u[q] = __shfl_sync(0xffffffffu, v[q & 3], 2 * I + (q >> 2));
    const int nI = K - 8 * I;  // rows of the block (row K and the padding are not solved for)
#pragma unroll
    for (int c = 7; c >= 0; --c) {
      u[c] = c < nI ? u[c] * rd[c] : 0.f;
#pragma unroll
      for (int r = 0; r < c; ++r) u[r] = fmaf(-d[c][r], u[c], u[r]);
    }
    if (J < I) {
      const float* L = T + tidx(I, J) * kTileF + h4;
      float4 lc[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) lc[q] = *reinterpret_cast<const float4*>(L + trow(q));
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        v[0] = fmaf(-lc[q].x, u[q], v[0]);
        v[1] = fmaf(-lc[q].y, u[q], v[1]);
        v[2] = fmaf(-lc[q].z, u[q], v[2]);
        v[3] = fmaf(-lc[q].w, u[q], v[3]);
      }
    } else if (J == I) {
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = h4 ? u[4 + k] : u[k];
    }
    load_diag(I > 0 ? I - 1 : 0);
  }
  const int c0 = 8 * J + h4;
  if ((K & 3) == 0) {  // the row of X starts on a 16-byte boundary
    if (c0 < K) {
      *reinterpret_cast<float4*>(out + c0) = make_float4(v[0], v[1], v[2], v[3]);
      if (a.Xhi != nullptr) {
        __nv_bfloat16 h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) split_bf16(v[k], h[k], l[k]);
        __nv_bfloat162* hi = reinterpret_cast<__nv_bfloat162*>(a.Xhi + (int64_t)row * a.KS + c0);
        __nv_bfloat162* lo = reinterpret_cast<__nv_bfloat162*>(a.Xlo + (int64_t)row * a.KS + c0);
        hi[0] = __nv_bfloat162(h[0], h[1]);
        hi[1] = __nv_bfloat162(h[2], h[3]);
        lo[0] = __nv_bfloat162(l[0], l[1]);
        lo[1] = __nv_bfloat162(l[2], l[3]);
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (c0 + k < K) {
        out[c0 + k] = v[k];
        write_shadow(a, row, c0 + k, v[k]);
      }
  }
}

// Element (i, j) of the base matrix: the lower triangle of the bordered
// [[Lambda_s, b0], [b0^T, inf]], identity on the padding past row K.  No draw reads
// the corner; a finite one, 1e30, sent rows with alpha sum r^2 past it to the FP64
// redo, by the NaN that the root of a negative pivot leaves in the padding.
__device__ __forceinline__ float row_base(const SweepArgs& a, int i, int j) {
  const int K = a.K, KA = K + 1;
  if (i >= KA || j >= KA) return i == j ? 1.f : 0.f;
  return j > i ? 0.f : i == K && j == K ? INFINITY : __ldg(a.lamaug + i * KA + j);
}

// Element (i, j) of base + alpha G from the Gram's; what the Gram holds in the
// corner (K, K) and outside the bordered lower triangle is not looked at.
__device__ __forceinline__ float row_elem(const SweepArgs& a, int i, int j, float s) {
  const float b = row_base(a, i, j);
  return i > a.K || j > i || j >= a.K ? b : fmaf(a.alpha, s, b);
}

// One warp factors the tiles and draws the row, or leaves it to the FP64 redo;
// zv has room for K rounded up to 4.
template <int W = 1>
__device__ __forceinline__ void row_draw(const SweepArgs& a, int g, float* T, const float* thr,
                                         float* rinv, float* zv, int row, int lane) {
  const uint32_t tw = *a.tp;
  for (int q = lane; 4 * q < a.K; q += 32)
    *reinterpret_cast<float4*>(zv + 4 * q) =
        normal4_f32(philox(make_uint4((uint32_t)row, tw, (uint32_t)q, a.sw), a.key));
  const bool ok = warp_cholesky<W>(g, T, thr, rinv, lane);
  if (ok) warp_back(a, T, rinv, zv, row, lane);
  else if (lane == 0) a.flag_rows[atomicAdd(a.flag_count, 1)] = row;
}

}  // namespace gb
