// tile_chol.cuh -- pivot rule, tile numbering and small helpers shared by the
// row kernels.
//
// The row draw (Algorithm 1's row update) needs L = chol(Lambda*), y = L^-1 b
// and u = L^-T (y + z).  The kernels factor the bordered matrix
//     [[Lambda*, b], [b^T, .]]   ((K+1) x (K+1))
// whose Cholesky factor is [[L, 0], [y^T, .]]: the forward solve comes out of
// the factorisation as its last row.  Only u = L^-T (y + z) is left, done by
// one warp.  The lower triangle is cut into 8 x 8 tiles on a g x g grid.
#pragma once

#include <float.h>

#include "bpmf_impl.cuh"

namespace gb {

// Pivot rule: a pivot at or below prel (SweepArgs::pivot_rel) times its
// column's starting diagonal means the FP32 factorisation may have lost too
// many digits there, and the row is redone in FP64.  The pivot ratio of
// column k is 1 / (A_kk (A_k^-1)_kk) for the leading block A_k, so a small
// ratio marks an ill-conditioned row; a non-positive pivot always fails.
// The threshold is formed from the starting diagonal alone, off the
// dependence chain of the factorisation: the pivot meets one comparison.
__device__ __forceinline__ float pivot_threshold(float prel, float d0) {
  return fmaxf(prel * d0, FLT_MIN);
}
// A failed pivot is replaced by this finite stand-in so that the rest of the
// factorisation stays finite (its output is discarded).
__device__ __forceinline__ float pivot_stand_in(float piv, float d0) {
  return fmaxf(fabsf(piv), fabsf(d0) * 1e-4f) + FLT_MIN;
}

struct TileGeom {
  int K, KA, TM, g, KP, KPs, LDS, ntiles, nthreads;
  __host__ __device__ TileGeom(int K_, int TM_) : K(K_), KA(K_ + 1), TM(TM_) {
    g = (KA + TM - 1) / TM;
    KP = g * TM;
    KPs = (KP + 3) & ~3;
    LDS = KP + 1;
    ntiles = g * (g + 1) / 2;
    nthreads = ((ntiles > 32 ? ntiles : 32) + 31) & ~31;
  }
};

// Tile numbering from the bottom-right corner: t = u (u + 1) / 2 + v with
// u = g - 1 - tx and v = ty - tx.  The trailing triangle of every panel
// (tx > c) is then the prefix t < (g-1-c)(g-c)/2, so the threads that still
// have work at panel c fill whole warps, and the panel's own column of tiles
// is one contiguous run of thread ids.
__device__ __forceinline__ void tri_tile(int t, int g, int& ty, int& tx) {
  int u = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((u + 1) * (u + 2) / 2 <= t) ++u;
  while (u * (u + 1) / 2 > t) --u;
  tx = g - 1 - u;
  ty = tx + (t - u * (u + 1) / 2);
}
__host__ __device__ __forceinline__ int tile_id(int ty, int tx, int g) {
  const int u = g - 1 - tx;
  return u * (u + 1) / 2 + (ty - tx);
}

// The K normals of the row (Box-Muller on Philox counter (row, t, q, sw)).
__device__ __forceinline__ void row_normals(float* zv, int K, int row, uint32_t t, uint32_t sw,
                                            uint2 key) {
  for (int q = threadIdx.x; 4 * q < K; q += blockDim.x) {
    const float4 z = normal4_f32(philox(make_uint4((uint32_t)row, t, (uint32_t)q, sw), key));
    zv[4 * q] = z.x;
    if (4 * q + 1 < K) zv[4 * q + 1] = z.y;
    if (4 * q + 2 < K) zv[4 * q + 2] = z.z;
    if (4 * q + 3 < K) zv[4 * q + 3] = z.w;
  }
}

}  // namespace gb
