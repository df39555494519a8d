// rows_ws.cu -- row draws by a persistent, warp-specialised kernel (mixed
// path, heavy rows).
//
// Same conditional as rows.cu and rows_tc.cu (Algorithm 1's row update): the
// Gram of the rating-augmented neighbour vectors x_j = [v_j, r_ij] gives
// Lambda* = Lambda_s + alpha sum v_j v_j^T and b = Lambda_s mu_s + alpha sum
// r_ij v_j as one bordered matrix; its Cholesky factor L holds y = L^-1 b in
// its last row; u = L^-T (y + z).
//
// One CTA per SM takes rows of the degree order from a global counter
// (largest first) and runs them through a pipeline of warp roles:
//   gather (warps 0-3): copies the bf16 hi/lo shadow rows of the neighbours,
//     NB per stage (32, or 64 on a side whose rows average 256 or more
//     ratings), by tensor-memory-accelerator gather4 copies (four neighbour
//     rows x 64 features each) straight into MN-major operand tiles with the
//     128-byte swizzle, into a ring of stages (64-neighbour stages copy the
//     features past 64 by 16-byte cp.async instead); the MMA warp patches
//     the rating in as feature K;
//   MMA (warp 8, one elected thread): per 16 neighbours hi.hi + hi.lo + lo.hi into
//     one of three FP32 accumulators in tensor memory (G = X^T X with X the
//     stage's neighbours x features; lo.lo, ~2^-16 relative, is dropped); on
//     sides whose rows average 2048 ratings or more, hi.[hi lo] as one wide
//     product into two accumulators instead, and the drain adds hi.lo and its
//     transpose;
//   drain (warps 4-7, thread m = tensor-memory lane m = matrix row m):
//     forms A = base + alpha G (base = bordered [[Lambda_s, b0], [b0^T, 0]],
//     kept in tensor memory, or in shared memory where the accumulators take
//     all of it) and writes its lower triangle as 8 x 8 FP32 tiles into a free
//     consumer slot, releasing the accumulator for the next row;
//   consumers (warps 9.., one row each): left-looking blocked Cholesky of the
//     slot (per 8-column block: the updates from the columns before by
//     mma.m16n8k8 on operands split into two TF32 parts, the diagonal tile in
//     registers by every lane, the panel by forward substitution), then
//     u = L^-T (y + z) by back substitution.
// So the tensor cores, the gathers and the FP32 factorisations of up to
// eleven rows per SM overlap, with no CTA-wide barrier on the way.
//
// Every mbarrier wait polls with a wall-clock bound; on a timeout the CTA
// records kStatusTimeout, every role leaves its loop, outstanding copies and
// MMAs are waited for (bounded) and the tensor memory is freed.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "bpmf_impl.cuh"
#include "rows.cuh"
#include "tc_ptx.cuh"
#include "tile_chol.cuh"
#include "warp_chol.cuh"

namespace gb {
namespace {

// Operand tiles (hi and lo, one each per stage) are MN-major with the
// 128-byte swizzle: neighbour k of the stage is a 128-byte row of 64 features
// (row k % 8 of the 1024-byte atom of 8-neighbour group k / 8), features
// 64 .. 127 in a second block of atoms NB * 128 bytes further; within each
// row the 16-byte chunk c sits at position c ^ (k % 8).  This is the layout
// the tensor memory accelerator writes for a box of 64 bf16 with the
// 128-byte swizzle, so one gather4 fills four neighbour rows of one block.
constexpr int kWsAtom = 1024;        // 8 neighbour rows x 128 bytes
constexpr int64_t kWsLongRow = 256;  // mean ratings per row from which stages hold 64 neighbours
// Neighbours per stage NB: 32 (two MMA K-steps) or 64 (four), chosen per side:
// bigger stages halve the hand-offs per neighbour where rows are long.
template <int NB>
struct WsNb {
  static constexpr int kBlk = NB * 128;             // bytes of one 64-feature block
  static constexpr int kOpBytes = 2 * kBlk;         // 128 features (the MMA reads M = 128 rows)
  static constexpr int kStageBytes = 2 * kOpBytes;  // hi + lo
  // Long-row stages split their copies: the first 64-feature block by TMA
  // gather4, the rest by 16-byte cp.async through another request path, as
  // the TMA issue rate (about 17 cycles per gather4 per SM) co-limits those
  // sides; short-row sides keep every copy on the TMA, where cp.async's
  // traffic through L1 would cost the consumers, which limit them.
  static constexpr bool kSplitCopy = NB >= 64;
};

// With XO ("cross once") the cross term h^T l + l^T h comes from one product:
// h^T h and h^T l go to two accumulators and the drain adds h^T l and its
// transpose (a second pass over the slot).  One wide product per step instead
// of three (92 cycles against 180 at K = 100), which pays where rows are long
// enough for the tensor pipe to set the pace (sides averaging kWsCrossRow
// ratings or more); where they are shorter the drain's second pass costs more
// than it saves.
constexpr int64_t kWsCrossRow = 2048;
template <bool XO>
__host__ __device__ constexpr uint32_t ws_acc_stride() { return XO ? 256u : 128u; }  // TMEM columns per buffer
// Tensor memory: the accumulators from column 0, three of 128 columns followed
// by the base matrix (columns 384 .. 511), or with XO two pairs that fill all
// 512 columns.
constexpr uint32_t kWsTmemCols = 512;
constexpr uint32_t kWsBaseCol = 384;
template <bool XO>
__host__ __device__ constexpr int ws_num_acc() { return XO ? 2 : 3; }
constexpr int kWsMaxAcc = 3;
__host__ __device__ constexpr int ws_stage_bytes(int nb) { return 2 * 2 * nb * 128; }
constexpr int kWsMaxStages = 16;
constexpr int kWsMaxCons = 7;
// The wide form: a ring of four stages instead of eight and as many consumers
// as fit, up to 11 (past seven, 640 threads of 95 registers instead of 113), for
// sides of K >= 64 without long rows, whose consumers set the pace: there
// eight stages of K = 64 leave seven consumers, of K = 72 five, of K >= 80 three.
// An iteration of 50,000 x 12,000 uniform cells with 2.5M ratings: K = 64 1,145
// -> 1,075 us, K = 80 1,772 -> 1,434, K = 100 2,837 -> 2,156; with 0.5M 999 -> 902,
// 1,705 -> 1,284 and 2,779 -> 2,079.  K = 56 gained 2% there and lost 4% with
// 60,000 x 17,770 and 5M (83 and 281 ratings a row), K <= 48 lost up to 7%.  Below
// K = 72 sides averaging kWsWideRow ratings or more lose (K = 64, 208 a row: 1%).  A
// row much longer than the others is copied by one SM at the pace of its ring:
// sides with one of more than kWsWideMax ratings keep eight stages
// (ChEMBL-shaped, K = 64: 1,320 us against 1,328; not measured with such rows at
// K >= 72, where eight stages leave far fewer consumers).
constexpr int kWsWideCons = 11, kWsWideK = 64, kWsWideAllK = 72;
constexpr int64_t kWsWideRow = 128, kWsWideMax = 1024;
constexpr int kWsRecs = 32;          // row records in flight: >= stages + accumulators + 1
constexpr int kWsGather = 128, kWsDrain = 128;
constexpr int kWsMmaWarp = 8, kWsConsWarp0 = 9;
// Warps are issued by the scheduler partition warp % 4.  Partition 0 holds
// a gather warp, a drain warp and the MMA warp; with six consumers, warp 12
// (partition 0) stays idle, so that the consumers spread evenly over
// partitions 1 .. 3 (two each) and take the same time per row: they take
// rows in turn, so an uneven spread leaves the faster ones waiting (with
// four, the plain order already puts one on each partition).
__host__ __device__ constexpr bool ws_skip_warp12(int C) { return C == 6; }
__host__ __device__ constexpr int ws_warps(int C) { return kWsConsWarp0 + C + (ws_skip_warp12(C) ? 1 : 0); }
// consumer index of warp w (-1: not a consumer)
__host__ __device__ constexpr int ws_consumer_of(int w, int C) {
  return w < kWsConsWarp0 ? -1
         : !ws_skip_warp12(C) ? (w - kWsConsWarp0 < C ? w - kWsConsWarp0 : -1)
         : w == 12 ? -1
         : (w < 12 ? w - kWsConsWarp0 : (w - kWsConsWarp0 - 1 < C ? w - kWsConsWarp0 - 1 : -1));
}
constexpr uint32_t kWsPolls = 100000;  // suspending polls of <= 20 us: a 2 s bound (final MMA wait)
constexpr uint32_t kWsAccCols = 128;

struct WsGeom {
  int K, KA, g, KP, NP, ntile;
  __host__ __device__ explicit WsGeom(int K_) : K(K_) {
    KA = K + 1;
    g = (KA + 7) / 8;
    KP = 8 * g;
    NP = (KA + 15) & ~15;
    ntile = g * (g + 1) / 2;
  }
  // consumer slot: header (4 ints), tiles, pivot thresholds, 1 / diagonal, z
  __host__ __device__ int slot_floats() const { return 4 + ntile * kTileF + 3 * KP; }
};

struct StageMeta {
  int cnt;    // neighbours in this stage (0 for a row without ratings)
  int flags;  // 1: first stage of the row, 2: last stage of the row, 4: no more rows
  int pad0, pad1;
};
struct RowRec {
  int row;  // -1: no more rows
  int nst;  // stages with ratings (0: the row has none)
  int pad0, pad1;
};

struct WsShared {
  uint8_t* stages;
  float* slots;
  float* base;  // base tiles (with XO only)
  uint64_t* empty;
  uint64_t* tma;  // the stage's copies have landed (and its metadata and ratings are written)
  uint64_t* acc_full;
  uint64_t* acc_empty;
  uint64_t* slot_full;
  uint64_t* slot_empty;
  uint64_t* fin;
  uint64_t* row_ready;  // the gather leader published the next row
  uint64_t* row_read;   // every gather thread has read it
  uint64_t* drain_sync;  // every drain thread has written its rows (cross-term pass)
  StageMeta* meta;
  RowRec* recs;
  float* rating;   // [stage][neighbour]: ratings waiting to be patched in
  int* next_row;   // [4]: row, first rating, last rating
  int* abort;
  uint32_t* taddr;
  uint64_t wait_ns;  // bound of every pipeline wait (SweepArgs::wait_ns)
};

// mbarriers: empty and tma per stage, full and empty per accumulator, full
// and empty per consumer slot, fin, row_ready, row_read, drain_sync (an even
// count, so that what follows stays 16-byte aligned)
__host__ __device__ inline int ws_nbar(int S, int C) { return 2 * S + 2 * kWsMaxAcc + 2 * C + 4; }
__host__ __device__ inline int ws_fixed_bytes(int nb, int S, int C) {
  // barriers, stage meta, row records, ratings, next_row, abort, taddr
  return 8 * ws_nbar(S, C) + 16 * S + 16 * kWsRecs + 4 * S * nb + 32;
}
// stages, consumer slots, base tiles (with XO), then the fixed part; one atom
// more, to start the stages on a 1024-byte boundary (the swizzle pattern
// follows address bits 7 .. 9)
__host__ __device__ inline int ws_smem_bytes(const WsGeom& G, int S, int C, int nb, bool cross) {
  return kWsAtom + S * ws_stage_bytes(nb) + C * G.slot_floats() * 4 +
         (cross ? G.ntile * kTileF * 4 : 0) + ws_fixed_bytes(nb, S, C);
}

__device__ __forceinline__ WsShared ws_carve(uint8_t* base, const WsGeom& G, int S, int C, int nb,
                                             bool cross) {
  WsShared w;
  w.stages = base;
  w.slots = reinterpret_cast<float*>(base + S * ws_stage_bytes(nb));
  w.base = w.slots + C * G.slot_floats();
  uint8_t* p = reinterpret_cast<uint8_t*>(w.base + (cross ? G.ntile * kTileF : 0));
  uint64_t* b = reinterpret_cast<uint64_t*>(p);
  w.empty = b;
  w.tma = b + S;
  w.acc_full = b + 2 * S;
  w.acc_empty = w.acc_full + kWsMaxAcc;
  w.slot_full = w.acc_empty + kWsMaxAcc;
  w.slot_empty = w.slot_full + C;
  w.fin = w.slot_empty + C;
  w.row_ready = w.fin + 1;
  w.row_read = w.fin + 2;
  w.drain_sync = w.fin + 3;
  p = reinterpret_cast<uint8_t*>(b + ws_nbar(S, C));
  w.meta = reinterpret_cast<StageMeta*>(p);
  w.recs = reinterpret_cast<RowRec*>(p + 16 * S);
  w.rating = reinterpret_cast<float*>(p + 16 * S + 16 * kWsRecs);
  int* q = reinterpret_cast<int*>(w.rating + S * nb);
  w.next_row = q;
  w.abort = q + 4;
  w.taddr = reinterpret_cast<uint32_t*>(q + 5);
  w.wait_ns = 0;
  return w;
}

__device__ __forceinline__ uint64_t ws_gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait by one thread: polls without a suspend hint (a suspended
// thread resumes late, and every hand-off of the pipeline pays for it), and
// gives up (setting abort) after `limit` ns of wall-clock time (2 s unless
// the caller set another bound), or as soon as another role has aborted.
__device__ __forceinline__ bool ws_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                        uint64_t limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = ws_gtimer();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 31u) == 0u) {
      if (*abort) return false;
      if (ws_gtimer() - t0 > limit) break;
    }
  }
  *abort = 1;
  return false;
}

// The same by a whole warp: every lane waits (and so acquires what the
// barrier publishes); the outcome is made uniform across the warp, so no
// lane leaves a loop that its neighbours stay in.
__device__ __forceinline__ bool ws_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort,
                                             uint64_t limit) {
  const bool ok = ws_wait(bar, parity, abort, limit);
  return __all_sync(0xffffffffu, ok) != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// Waits (bounded, whatever the abort flag and the pipeline bound say) until
// copies this warp issued have landed: shared memory must not be written
// after the block ends.  Copies land within microseconds; the 2 s bound only
// keeps the wait finite.
constexpr uint64_t kWsCopyDrainNs = 2000000000ull;
__device__ __forceinline__ void ws_wait_copies(uint64_t* bar, uint32_t parity, uint64_t limit) {
  const uint64_t t0 = ws_gtimer();
  while (!mbar_try_wait(bar, parity) && ws_gtimer() - t0 < limit) {
  }
}

// kind::f16 instruction descriptor, BF16 operands both MN-major (bits 15, 16).
__device__ __forceinline__ uint32_t idesc_bf16_mn(int M, int N) {
  return idesc_bf16_f32(M, N) | (1u << 15) | (1u << 16);
}

// ------------------------------------------------------------- gather --
// The four gather warps take the stages of the row sequence in turn (stage n
// by warp n % 4), so four stages are filled side by side.  In the warp that
// fills stage n, lane l holds neighbours l, l + 32, .. (NB / 32 of them); the
// rows of neighbours 4g .. 4g + 3, g < 4 ceil(cnt / 16), are copied into both
// operand tiles with one gather4 per 64-feature block and tile (with
// WsNb::kSplitCopy, the first block only: each lane copies the rest of its
// neighbours' rows by cp.async).  Rows past cnt (up to the MMA's
// 16-neighbour step) are read at an out-of-range row index, which the copy
// fills with zeros.  The rating (feature K) is patched in once the copies
// have landed (ws_patch_rating).
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap* map, int x, int y0,
                                            int y1, int y2, int y3, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y0), "r"(y1), "r"(y2), "r"(y3),
      "r"(smem_u32(bar))
      : "memory");
}
// 16-byte copy through L2 only, zero-filling past src_bytes (0: all zeros)
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes)
               : "memory");
}
// the barrier counts one arrival of this thread once its earlier cp.async
// copies have landed (the arrival is part of the barrier's initial count)
__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

template <int NB>
__device__ __forceinline__ void ws_issue_stage(const WsGeom& G, const SweepArgs& a,
                                               const CUtensorMap* map_hi, const CUtensorMap* map_lo,
                                               uint8_t* stage, uint64_t* bar, int cnt,
                                               const int32_t (&j)[NB / 32], int lane) {
  const int ngroups = 4 * ((cnt + 15) >> 4);
  const int nblk = G.KA > 64 ? 2 : 1;
  // row ids of this lane's neighbours, out of range past cnt
  int y[NB / 32];
#pragma unroll
  for (int u = 0; u < NB / 32; ++u) y[u] = lane + 32 * u < cnt ? (int)j[u] : (int)a.n_other;
  // the arrive (release) publishes the lanes' metadata and rating writes with
  // the copies: the MMA warp waits for this barrier alone
  const bool split = WsNb<NB>::kSplitCopy && nblk == 2;
  const int ntma = split ? 1 : nblk;  // feature blocks copied by TMA
  __syncwarp();
  if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)(ngroups * ntma * 2 * 512));
  __syncwarp();
  // One elected lane issues every copy, the ids coming to it by shuffles.
  // Issued by the lanes that hold the ids, each copy goes through a loop over
  // the lanes' operands: about 100 cycles per gather4, 2.3-3.4k per
  // 32-neighbour stage of K = 100 against 1.0-1.4k this way.
  const uint32_t hi0 = smem_u32(stage);
#pragma unroll
  for (int u = 0; u < NB / 32; ++u) {
    for (int g4 = 0; g4 < 8; g4 += 4) {  // 16 neighbours
      if (8 * u + g4 >= ngroups) break;
      int z[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) z[i] = __shfl_sync(0xffffffffu, y[u], 4 * g4 + i);
      if (elect_one()) {
        const uint32_t hi = hi0 + (uint32_t)((8 * u + g4) * 512);  // two groups per atom
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int* r = z + 4 * g;
          const uint32_t dst = hi + g * 512;
          tma_gather4(dst, map_hi, 0, r[0], r[1], r[2], r[3], bar);
          tma_gather4(dst + WsNb<NB>::kOpBytes, map_lo, 0, r[0], r[1], r[2], r[3], bar);
        }
        if (ntma == 2) {
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int* r = z + 4 * g;
            const uint32_t dst = hi + g * 512 + WsNb<NB>::kBlk;
            tma_gather4(dst, map_hi, 64, r[0], r[1], r[2], r[3], bar);
            tma_gather4(dst + WsNb<NB>::kOpBytes, map_lo, 64, r[0], r[1], r[2], r[3], bar);
          }
        }
      }
    }
  }
  if (split) {
    // features 64 .. KS - 1 (chunks 0 .. c1 - 1 of the second block) by
    // 16-byte cp.async into their swizzled places, rows past cnt (up to the
    // MMA's 16-neighbour step) zero-filled; the later chunks, among them the
    // rating's where K is a multiple of eight, stay zero from the start of
    // the kernel: a copy of them would read the next row, or past the last.
    // Every lane arrives on the stage's barrier once its copies have landed.
    const int c1 = (a.KS - 64) >> 3;
    const int kmax = 16 * ((cnt + 15) >> 4);
    const uint32_t base = smem_u32(stage) + (uint32_t)WsNb<NB>::kBlk;
#pragma unroll
    for (int u = 0; u < NB / 32; ++u) {
      const int k = lane + 32 * u;
      if (k < kmax) {
        const bool live = k < cnt;
        const int64_t jr = live ? (int64_t)j[u] : 0;
        const __nv_bfloat16* h = a.Vhi + jr * a.KS + 64;
        const __nv_bfloat16* l = a.Vlo + jr * a.KS + 64;
        const uint32_t row = base + (uint32_t)((k >> 3) * kWsAtom + (k & 7) * 128);
        for (int c = 0; c < c1; ++c) {
          const uint32_t off = (uint32_t)((c ^ (k & 7)) << 4);
          cp_async16_zfill(row + off, h + 8 * c, live ? 16u : 0u);
          cp_async16_zfill(row + WsNb<NB>::kOpBytes + off, l + 8 * c, live ? 16u : 0u);
        }
      }
    }
    cp_async_arrive_noinc(bar);
  }
}

// Feature K of neighbour k = the rating r, as bf16 hi and lo, at its
// swizzled place in the operand tiles.
template <int NB>
__device__ __forceinline__ void ws_patch_rating(const WsGeom& G, uint8_t* stage, float r, int k) {
  const int f = G.K, k0 = k & 7;
  const int off = (f >> 6) * WsNb<NB>::kBlk + (k >> 3) * kWsAtom + k0 * 128 +
                  ((((f >> 3) & 7) ^ k0) << 4) + 2 * (f & 7);
  const __nv_bfloat16 h = __float2bfloat16_rn(r);
  *reinterpret_cast<__nv_bfloat16*>(stage + off) = h;
  *reinterpret_cast<__nv_bfloat16*>(stage + WsNb<NB>::kOpBytes + off) =
      __float2bfloat16_rn(r - __bfloat162float(h));
}

// Stage n lives in ring slot (n % 4) + 4 ((n / 4) % (S / 4)) (S is a
// multiple of 4): every slot is filled by one gather warp only, in order, so
// no warp ever waits on a slot's barrier more than one phase ahead (an
// mbarrier wait tells phases apart by parity only).
__host__ __device__ __forceinline__ int ws_slot(uint32_t n, int S) {
  return (int)(n & 3u) + 4 * (int)((n >> 2) % (uint32_t)(S >> 2));
}

// A position in a ring of `size` entries and the parity of its passes,
// stepped instead of divided for: the roles take a step per stage or row.
struct RingPos {
  int i = 0;
  uint32_t parity = 0;  // of the number of times the ring has been passed
  __device__ __forceinline__ void next(int size) {
    if (++i == size) {
      i = 0;
      parity ^= 1u;
    }
  }
};

template <int NB>
__device__ __forceinline__ void ws_gather(const SweepArgs& a, const WsGeom& G, const WsShared& w,
                                          int S, int* counter, const CUtensorMap* map_hi,
                                          const CUtensorMap* map_lo) {
  constexpr int NL = NB / 32;  // neighbours per lane
  const int t = threadIdx.x;
  const int wg = t >> 5, lane = t & 31;
  const int nrows = (int)(a.row_end - a.row_begin);
  // a warp owns the S / 4 ring slots wg + 4 i; it only issues copies (the
  // MMA warp waits for them), and keeps the last stage issued into each slot
  // so that it can wait for those copies before the block ends
  uint32_t n = 0;             // stage sequence number (the same in every gather warp)
  int q = 0;                  // row sequence number
  int rec = 0;                // q % kWsRecs
  RingPos pos;                // of the warp's next stage among its S / 4 slots
  uint32_t last[4] = {~0u, ~0u, ~0u, ~0u};
  // thread 0 prefetches the next row's work entry (row, first, last rating)
  int4 wk = make_int4(-1, 0, 0, 0);
  int next_slot = 0;
  if (t == 0) {
    next_slot = atomicAdd(counter, 1);
    if (next_slot < nrows) wk = __ldg(a.work + a.row_begin + next_slot);
  }
  bool stop = false;
  for (;;) {
    if (t == 0) {
      // the slot is free once every gather thread has read the previous row
      const bool ok = q == 0 || ws_wait(w.row_read, (uint32_t)(q - 1) & 1u, w.abort, w.wait_ns);
      w.next_row[0] = ok ? wk.x : -1;
      w.next_row[1] = wk.y;
      w.next_row[2] = wk.z;
      mbar_arrive(w.row_ready);
      if (ok && wk.x >= 0) next_slot = atomicAdd(counter, 1);
    }
    if (!ws_wait_warp(w.row_ready, (uint32_t)q & 1u, w.abort, w.wait_ns)) break;
    const int row = w.next_row[0];
    const int e0 = w.next_row[1], e1 = row >= 0 ? w.next_row[2] : e0;
    mbar_arrive(w.row_read);
    if (t == 0)
      wk = next_slot < nrows && row >= 0 ? __ldg(a.work + a.row_begin + next_slot)
                                         : make_int4(-1, 0, 0, 0);
    const int nst_r = (e1 - e0 + NB - 1) / NB;
    const int nst = nst_r > 0 ? nst_r : 1;
    const int st_first = (int)((uint32_t)(wg - (int)(n & 3u)) & 3u);
    // neighbour ids and ratings of this lane for the warp's next stage (four
    // stages on), loaded while the current one is issued
    int32_t jn[NL];
    float rn[NL];
#pragma unroll
    for (int u = 0; u < NL; ++u) {
      const int k = lane + 32 * u;
      jn[u] = 0;
      rn[u] = 0.f;
      if (row >= 0 && st_first < nst && e0 + st_first * NB + k < e1) {
        jn[u] = __ldg(a.idx + e0 + st_first * NB + k);
        rn[u] = __ldg(a.val + e0 + st_first * NB + k);
      }
    }
    for (int st = st_first; st < nst; st += 4) {
      const uint32_t nn = n + (uint32_t)st;
      const int s = wg + 4 * pos.i;  // ws_slot(nn, S)
      const int e = e0 + st * NB;
      const int cnt = row < 0 ? 0 : (e1 - e < NB ? (e1 - e > 0 ? e1 - e : 0) : NB);
      int32_t j[NL];
      float r[NL];
#pragma unroll
      for (int u = 0; u < NL; ++u) {
        const int k = lane + 32 * u;
        j[u] = jn[u];
        r[u] = rn[u];
        if (row >= 0 && e + 4 * NB + k < e1) {
          jn[u] = __ldg(a.idx + e + 4 * NB + k);
          rn[u] = __ldg(a.val + e + 4 * NB + k);
        }
      }
      if (!ws_wait_warp(&w.empty[s], pos.parity ^ 1u, w.abort, w.wait_ns)) {
        stop = true;
        break;
      }
      if (lane == 0) {
        if (st == 0) {
          w.recs[rec].row = row;
          w.recs[rec].nst = row < 0 ? 0 : nst_r;
        }
        w.meta[s].cnt = cnt;
        w.meta[s].flags = (st == 0 ? 1 : 0) | (st == nst - 1 ? 2 : 0) | (row < 0 ? 4 : 0);
      }
#pragma unroll
      for (int u = 0; u < NL; ++u) {
        const int k = lane + 32 * u;
        w.rating[s * NB + k] = k < cnt ? r[u] : 0.f;
      }
      ws_issue_stage<NB>(G, a, map_hi, map_lo, w.stages + s * WsNb<NB>::kStageBytes, &w.tma[s], cnt,
                         j, lane);
      const int li = pos.i;
      pos.next(S >> 2);
      last[0] = li == 0 ? nn : last[0];
      last[1] = li == 1 ? nn : last[1];
      last[2] = li == 2 ? nn : last[2];
      last[3] = li == 3 ? nn : last[3];
    }
    n += (uint32_t)nst;
    if (stop || row < 0) break;
    ++q;
    rec = rec + 1 == kWsRecs ? 0 : rec + 1;
  }
  // whatever happened downstream, the copies this warp issued land before
  // the block ends (a slot's phases complete in order: its last one is enough)
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (last[i] != ~0u)
      ws_wait_copies(&w.tma[ws_slot(last[i], S)], (last[i] / (uint32_t)S) & 1u, kWsCopyDrainNs);
}

// ---------------------------------------------------------------- MMA --
// The whole MMA warp waits for each stage's copies (and with them its
// metadata and ratings), patches the ratings into their swizzled places,
// makes them visible to the tensor cores, and one elected lane issues the products.
// With `hold` (failure-path testing) the first row's accumulator is never
// handed to the drain, whose bounded wait then runs out.
template <int NB, bool XO>
__device__ __forceinline__ void ws_mma(const WsGeom& G, const WsShared& w, int S, uint32_t tmem,
                                       int hold) {
  const int lane = threadIdx.x & 31;
  // XO: the lo features follow the 128 hi features at the same block stride, so
  // [h | l] is one operand of 128 + NP columns and h^T [h | l] one product: 32 +
  // N / 4 cycles, 92 at K = 100 instead of 2 x 60.
  const uint32_t idesc = idesc_bf16_mn(128, XO ? 128 + G.NP : G.NP);
  // operand tile of the first stage: the leading byte offset steps between
  // 64-feature blocks, the stride one between atoms
  const uint64_t desc0 = smem_desc_sw128(smem_u32(w.stages), WsNb<NB>::kBlk, kWsAtom);
  uint32_t n = 0;
  RingPos acc_pos;   // the row's accumulator
  bool first_row = true;
  for (;;) {
    const int s = ws_slot(n, S);
    if (!ws_wait_warp(&w.tma[s], (n / (uint32_t)S) & 1u, w.abort, w.wait_ns)) break;
    uint8_t* stage = w.stages + s * WsNb<NB>::kStageBytes;
    const StageMeta m = w.meta[s];
#pragma unroll
    for (int t = 0; t < NB / 32; ++t)
      ws_patch_rating<NB>(G, stage, w.rating[s * NB + lane + 32 * t], lane + 32 * t);
    fence_proxy_async_smem();
    __syncwarp();
    const int b = acc_pos.i;
    if (m.flags & 1) {
      if (!ws_wait_warp(&w.acc_empty[b], acc_pos.parity ^ 1u, w.abort, w.wait_ns)) break;
    }
    tc_fence_after();
    if (elect_one()) {
      const uint32_t acc = tmem + (uint32_t)b * ws_acc_stride<XO>();
      // K-steps of 16 neighbours: two atoms apart (the descriptors count in
      // units of 16 bytes)
      const uint64_t dh = desc0 + (uint64_t)((s * WsNb<NB>::kStageBytes) >> 4);
      const int steps = (m.cnt + 15) >> 4;
#pragma unroll
      for (int kk = 0; kk < NB / 16; ++kk) {
        if (kk < steps) {
          const uint64_t h = dh + (uint64_t)((kk * 2 * kWsAtom) >> 4);
          const uint64_t l = h + (uint64_t)(WsNb<NB>::kOpBytes >> 4);
          const uint32_t more = kk == 0 ? (m.flags & 1) ^ 1u : 1u;
          if (XO) {
            tc_mma_bf16(acc, h, h, idesc, more);
          } else {
            tc_mma_bf16(acc, h, h, idesc, more);
            tc_mma_bf16(acc, h, l, idesc, 1u);
            tc_mma_bf16(acc, l, h, idesc, 1u);
          }
        }
      }
      tc_commit(&w.empty[s]);
      if ((m.flags & 2) && !(hold && first_row)) tc_commit(&w.acc_full[b]);
    }
    __syncwarp();
    ++n;
    if (m.flags & 2) {
      acc_pos.next(ws_num_acc<XO>());
      first_row = false;
      if (m.flags & 4) break;
    }
  }
  // every MMA issued has completed before the tensor memory is freed
  if (elect_one()) {
    tc_commit(w.fin);
    uint32_t polls = 0;
    while (!mbar_try_wait_sleep(w.fin, 0, 20000u) && ++polls < kWsPolls) {
    }
  }
  __syncwarp();
}

// -------------------------------------------------------------- drain --
// Thread m (0..127) owns tensor-memory lane m = row m of the accumulator.
//
// One row's drain stands between the MMA warp (which waits for the
// accumulator) and a consumer (which waits for the slot), so it is latency
// that counts.  The base matrix therefore sits on chip for the whole launch:
// in tensor memory beside the accumulators, read by the same kind of load in
// the same batch, or, with XO, in shared memory.  (Read from global memory
// tile by tile, as it was before, each 16 columns waited for a round trip to
// the L2: 8.5k cycles per row of K = 100, during which the consumers idled a
// quarter of their time.  60,000 rows of 188 ratings on average, K = 100:
// 3.06 -> 2.83 ms; K = 64, 50,000 rows of 45 and 12,000 of 188: 1.5 -> 1.3 ms
// for both sides.)
template <bool XO>
__device__ __forceinline__ void ws_drain(const SweepArgs& a, const WsGeom& G, const WsShared& w, int C,
                         uint32_t tmem) {
  const int m = threadIdx.x - kWsGather;
  const int wq = m >> 5, lane = m & 31;  // warp quarter: lanes 32 wq .. 32 wq + 31
  const int I = m >> 3, p = m & 7;
  const int slotf = G.slot_floats();
  const int row_tile = I * (I + 1) / 2;
  // columns 0 .. 32 wq + 31 cover the lower triangle of this warp's rows
  const int ncol = 32 * wq + 32 < G.NP ? 32 * wq + 32 : G.NP;
  const uint32_t quarter = (uint32_t)(32 * wq) << 16;
  if (XO) {
    if (m < G.KP) {
      for (int J = 0; J <= I; ++J) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = row_base(a, m, 8 * J + i);
        st8(w.base + (row_tile + J) * kTileF + trow(p), x);
      }
    }
  } else {
    for (int c0 = 0; c0 < ncol; c0 += 16) {
      float x[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = row_base(a, m, c0 + i);
      tmem_st16(tmem + kWsBaseCol + quarter + (uint32_t)c0, x);
    }
    tmem_wait_st();
  }
  RingPos acc_pos, slot_pos, rec_pos;
  uint32_t nsync = 0;  // completed phases of drain_sync
  for (;;) {
    const int b = acc_pos.i;
    if (!ws_wait_warp(&w.acc_full[b], acc_pos.parity, w.abort, w.wait_ns)) return;
    tc_fence_after();
    const RowRec r = w.recs[rec_pos.i];
    if (r.row < 0) {
      // one stop record per consumer, in slot order
      for (int i = 0; i < C; ++i, slot_pos.next(C)) {
        const int c = slot_pos.i;
        if (!ws_wait_warp(&w.slot_empty[c], slot_pos.parity ^ 1u, w.abort, w.wait_ns)) return;
        if (m == 0) reinterpret_cast<int*>(w.slots + c * slotf)[0] = -1;
        __syncwarp();
        if (lane == 0) mbar_arrive(&w.slot_full[c]);
      }
      return;
    }
    const int c = slot_pos.i;
    if (!ws_wait_warp(&w.slot_empty[c], slot_pos.parity ^ 1u, w.abort, w.wait_ns)) return;
    float* slot = w.slots + c * slotf;
    float* tiles = slot + 4;
    float* thr = tiles + G.ntile * kTileF;
    const uint32_t lane_base = tmem + (uint32_t)b * ws_acc_stride<XO>() + quarter;
    const bool gram = r.nst > 0;
    // A = base + alpha G, 16 columns at a time.  Entries past the diagonal in
    // the last tile are not read; G is zero in the padding rows and columns.
    for (int c0 = 0; c0 < ncol; c0 += 16) {
      float v[16], x[16];
      tmem_ld16(lane_base + (uint32_t)c0, v);
      if (XO) {
        float v2[16];
        tmem_ld16(lane_base + kWsAccCols + (uint32_t)c0, v2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int J = (c0 >> 3) + h;
          float y[8];
          ld8(w.base + (m < G.KP && J <= I ? (row_tile + J) * kTileF + trow(p) : 0), y);
#pragma unroll
          for (int i = 0; i < 8; ++i) x[8 * h + i] = y[i];
        }
        tmem_wait_ld(v);
        tmem_wait_ld(v2);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] += v2[i];
      } else {
        tmem_ld16(tmem + kWsBaseCol + quarter + (uint32_t)c0, x);
        tmem_wait_ld(v);
        tmem_wait_ld(x);
      }
      if (gram) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = fmaf(a.alpha, v[i], x[i]);
      }
      if (m < G.KP) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int J = (c0 >> 3) + h;
          if (J <= I) {
            float4* dst = reinterpret_cast<float4*>(tiles + (row_tile + J) * kTileF + trow(p));
            dst[0] = make_float4(x[8 * h], x[8 * h + 1], x[8 * h + 2], x[8 * h + 3]);
            dst[1] = make_float4(x[8 * h + 4], x[8 * h + 5], x[8 * h + 6], x[8 * h + 7]);
          }
        }
      }
    }
    if (XO && gram) {
      // the transposed cross term: thread n adds alpha (h^T l)[n][j] to the
      // slot's element (j, n) for j >= n (column n of the lower triangle,
      // which only this thread touches here), after every drain thread has
      // written its row above
      // a bounded barrier wait, so that a drain warp that has left on a
      // timeout cannot hold the others
      mbar_arrive(w.drain_sync);
      if (!ws_wait_warp(w.drain_sync, (uint32_t)nsync & 1u, w.abort, w.wait_ns)) return;
      ++nsync;
      const int n = m;
      for (int c0 = (32 * wq) & ~15; c0 < G.NP; c0 += 16) {
        float v[16], e[16];
        tmem_ld16(lane_base + kWsAccCols + (uint32_t)c0, v);
        // element (c0, n): the 16 rows are two tile rows of eight
        float* e0 = tiles + ((c0 >> 3) * ((c0 >> 3) + 1) / 2 + (n >> 3)) * kTileF + (n & 7);
        float* e1 = e0 + ((c0 >> 3) + 1) * kTileF;
        // all loads before the first store (the elements are distinct)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int j = c0 + i;
          e[i] = j >= n && j < G.KA ? (i < 8 ? e0 : e1)[trow(i & 7)] : 0.f;
        }
        tmem_wait_ld(v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int j = c0 + i;
          if (j >= n && j < G.KA) (i < 8 ? e0 : e1)[trow(i & 7)] = fmaf(a.alpha, v[i], e[i]);
        }
      }
    }
    // the pivot threshold from the row's own diagonal element, after any
    // transposed term (both are this thread's writes)
    if (m < G.KP)
      thr[m] = m < G.K ? pivot_threshold(a.pivot_rel, tiles[(row_tile + I) * kTileF + trow(p) + p])
                       : -INFINITY;
    if (m == 0) reinterpret_cast<int*>(slot)[0] = r.row;
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&w.acc_empty[b]);
      mbar_arrive(&w.slot_full[c]);
    }
    acc_pos.next(ws_num_acc<XO>());
    slot_pos.next(C);
    rec_pos.next(kWsRecs);
  }
}

// ----------------------------------------------------------- consumer --
// One warp factors a slot's tiles and solves for the row (warp_chol.cuh).
__device__ __forceinline__ void ws_consume(const SweepArgs& a, const WsGeom& G, const WsShared& w, int C) {
  const int c = ws_consumer_of(threadIdx.x >> 5, C);
  const int lane = threadIdx.x & 31;
  float* slot = w.slots + c * G.slot_floats();
  float* T = slot + 4;
  float* thr = T + G.ntile * kTileF;
  float* rinv = thr + G.KP;
  float* zv = rinv + G.KP;
  for (int qc = 0;; ++qc) {
    if (!ws_wait_warp(&w.slot_full[c], (uint32_t)qc & 1u, w.abort, w.wait_ns)) return;
    const int row = reinterpret_cast<const int*>(slot)[0];
    if (row < 0) return;
    row_draw(a, G.g, T, thr, rinv, zv, row, lane);
    __syncwarp();
    if (lane == 0) mbar_arrive(&w.slot_empty[c]);
  }
}

template <int NB, bool XO, int NT>
__global__ void __launch_bounds__(NT, 1) row_ws(const SweepArgs a,
                                                 const __grid_constant__ CUtensorMap map_hi,
                                                 const __grid_constant__ CUtensorMap map_lo, int S,
                                                 int C, int* counter, int* status) {
  extern __shared__ __align__(1024) uint8_t smem_ws[];
  const WsGeom G(a.K);
  uint8_t* base = smem_ws + ((kWsAtom - (smem_u32(smem_ws) & (kWsAtom - 1))) & (kWsAtom - 1));
  WsShared w = ws_carve(base, G, S, C, NB, XO);
  w.wait_ns = a.wait_ns;
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&w.empty[s], 1);
      // lane 0 of the filling warp arrives with the bytes to expect; with
      // split copies, every lane once more after its cp.async copies
      mbar_init(&w.tma[s], WsNb<NB>::kSplitCopy && G.KA > 64 ? 1 + 32 : 1);
    }
    for (int b = 0; b < ws_num_acc<XO>(); ++b) {
      mbar_init(&w.acc_full[b], 1);
      mbar_init(&w.acc_empty[b], kWsDrain / 32);  // lane 0 of each drain warp
    }
    for (int c = 0; c < C; ++c) {
      mbar_init(&w.slot_full[c], kWsDrain / 32);
      mbar_init(&w.slot_empty[c], 1);
    }
    mbar_init(w.fin, 1);
    mbar_init(w.row_ready, 1);
    mbar_init(w.row_read, kWsGather);
    mbar_init(w.drain_sync, kWsDrain);
    *w.abort = 0;
    mbar_fence_init();
  }
  // operand blocks no copy writes (features 64 .. 127 when K + 1 <= 64) stay zero
  for (int e = threadIdx.x; e < S * WsNb<NB>::kStageBytes / 16; e += blockDim.x)
    reinterpret_cast<uint4*>(w.stages)[e] = make_uint4(0, 0, 0, 0);
  if (warp == kWsMmaWarp) {
    tmem_alloc(w.taddr, kWsTmemCols);
    tmem_relinquish();
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *w.taddr;
  if (warp < 4) {
    ws_gather<NB>(a, G, w, S, counter, &map_hi, &map_lo);
  } else if (warp < 8) {
    ws_drain<XO>(a, G, w, C, tmem);
  } else if (warp == kWsMmaWarp) {
    ws_mma<NB, XO>(G, w, S, tmem, a.hold_arrive);
  } else if (ws_consumer_of(warp, C) >= 0) {
    ws_consume(a, G, w, C);
  }
  tc_fence_before();
  __syncthreads();
  if (*w.abort && threadIdx.x == 0) atomicOr(status, kStatusTimeout);
  if (warp == kWsMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kWsTmemCols);
  }
}

// bf16 hi/lo shadow of a factor matrix, rows padded to KS (a multiple of 8)
// for factors that are set or initialised (a draw writes its own); a thread
// converts eight columns, KS / 8 threads a row
constexpr int kShadowThreads = 256;
__global__ void __launch_bounds__(kShadowThreads) refresh_shadow_kernel(const float* __restrict__ X, int64_t R,
                                                                        int K, int KS,
                                                                        __nv_bfloat16* __restrict__ hi,
                                                                        __nv_bfloat16* __restrict__ lo) {
  const int Q = KS >> 3, per = kShadowThreads / Q;
  const int q = threadIdx.x % Q, rr = threadIdx.x / Q, c = 8 * q;
  if (rr >= per) return;
  for (int64_t r = (int64_t)blockIdx.x * per + rr; r < R; r += (int64_t)gridDim.x * per) {
    float x[8];
    if ((K & 3) == 0 && c + 8 <= K) {
      ld8(X + r * K + c, x);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = c + k < K ? X[r * K + c + k] : 0.f;
    }
    __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) split_bf16(x[k], h[k], l[k]);
    *reinterpret_cast<uint4*>(hi + r * KS + c) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + r * KS + c) = *reinterpret_cast<const uint4*>(l);
  }
}

}  // namespace

// Sides whose rows average 256 or more ratings (the movies of a
// Netflix-shaped set) take 64 neighbours per stage: half the stage hand-offs
// per neighbour; the others 32, which wastes less of the last stage of a
// short row.
int ws_stage_neighbours(int64_t nnz, int64_t R) {
  return R > 0 && nnz >= kWsLongRow * R ? 64 : 32;
}

bool ws_cross_once(int64_t nnz, int64_t R) { return R > 0 && nnz >= kWsCrossRow * R; }

bool ws_many_consumers(int K, int64_t nnz, int64_t R, int64_t max_degree) {
  return K >= kWsWideK && R > 0 && max_degree <= kWsWideMax && (K >= kWsWideAllK || nnz < kWsWideRow * R);
}

bool ws_supported(int K) { return K >= 8 && K + 1 <= 128; }

// Stages (a multiple of 4, one or more ring slots per gather warp) and
// consumer warps for latent dimension K and nb neighbours per stage (cross:
// with the base tiles in shared memory).  With
// `cons` > 0 that many consumers (as many as fit, if fewer) and the deepest
// ring up to kWsMaxStages that fits; otherwise 4 stages and as many consumers
// as fit, up to kWsWideCons, if wide; else 8 stages if at least 3 consumers fit
// beside them, or 4 stages and as many consumers as fit.
int ws_config(int K, int cons, int nb, bool cross, bool wide, int* S, int* C, int* most) {
  const WsGeom G(K);
  int dev = 0, max_smem = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return BPMF_ECUDA;
  }
  auto fit_cons = [&](int s, int most = kWsMaxCons) {
    int c = most;
    while (c > 0 && ws_smem_bytes(G, s, c, nb, cross) > max_smem) --c;
    return c;
  };
  int s = 8, c = 0;
  if (cons > 0) {
    c = std::min(cons, kWsMaxCons);
    s = kWsMaxStages;
    while (s > 4 && ws_smem_bytes(G, s, c, nb, cross) > max_smem) s -= 4;
    while (c > 1 && ws_smem_bytes(G, s, c, nb, cross) > max_smem) --c;  // more than fit: cut
  } else if (wide) {
    s = 4;
    c = fit_cons(s, kWsWideCons);
  } else {
    c = fit_cons(s);
    if (c < 3) {
      s = 4;
      c = fit_cons(s);
    }
  }
  if (c < 1 || ws_smem_bytes(G, s, c, nb, cross) > max_smem) return BPMF_EINVAL;
  *S = s;
  *C = c;
  *most = max_smem;
  return BPMF_OK;
}

namespace {

// cuTensorMapEncodeTiled of the driver, looked up once through the runtime
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// The other side's shadow (rows x KS bf16, rows 16-byte aligned) as a 2-D
// tensor read in boxes of 64 features x 1 row (gather4 boxes are one row
// high) with the 128-byte swizzle; rows and features past the end read as
// zeros.
int encode_shadow_map(const __nv_bfloat16* p, int64_t rows, int KS, CUtensorMap* map) {
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (enc == nullptr) {
    set_error("row_ws: cuTensorMapEncodeTiled is not available");
    return BPMF_ECUDA;
  }
  const cuuint64_t dim[2] = {(cuuint64_t)KS, (cuuint64_t)rows};
  const cuuint64_t stride[1] = {(cuuint64_t)KS * sizeof(__nv_bfloat16)};
  const cuuint32_t box[2] = {64, 1};
  const cuuint32_t step[2] = {1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(p),
                         dim, stride, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("row_ws: tensor map of the shadow rejected (%d)", (int)r);
    return BPMF_ECUDA;
  }
  return BPMF_OK;
}

}  // namespace

int launch_rows_ws(const SweepArgs& a, int num_sms, int cons, int nb, bool cross, bool wide,
                   int* counter, int* status, cudaStream_t st, int64_t* launches) {
  const int64_t nrows = a.row_end - a.row_begin;
  if (nrows <= 0) return BPMF_OK;
  if (nb != 32 && nb != 64) return BPMF_EINVAL;
  if (cross && nb != 64) return BPMF_EINVAL;
  int S = 0, C = 0, most = 0;
  BPMF_TRY(ws_config(a.K, cons, nb, cross, wide, &S, &C, &most));
  const WsGeom G(a.K);
  const int smem = ws_smem_bytes(G, S, C, nb, cross);
  auto kern = nb == 32 ? (C > kWsMaxCons ? row_ws<32, false, 640> : row_ws<32, false, 512>)
              : cross  ? row_ws<64, true, 512> : row_ws<64, false, 512>;
  BPMF_TRY(allow_smem(kern, most));
  const int grid = (int)std::min<int64_t>(num_sms, nrows);
  CUtensorMap map_hi, map_lo;
  BPMF_TRY(encode_shadow_map(a.Vhi, a.n_other, a.KS, &map_hi));
  BPMF_TRY(encode_shadow_map(a.Vlo, a.n_other, a.KS, &map_lo));
  kern<<<grid, 32 * ws_warps(C), smem, st>>>(a, map_hi, map_lo, S, C, counter, status);
  BPMF_CUDA_CHECK(cudaGetLastError());
  if (launches) *launches += 1;
  return BPMF_OK;
}

int launch_refresh_shadow(Handle* h, int s) {
  SideDev& sd = h->side[s];
  if (!sd.Xhi || sd.R == 0) return BPMF_OK;
  const int per = kShadowThreads / (sd.KS >> 3);
  const int64_t g = std::min<int64_t>((sd.R + per - 1) / per, 16LL * h->num_sms);
  refresh_shadow_kernel<<<(unsigned)g, kShadowThreads, 0, h->stream>>>(sd.X, sd.R, h->K, sd.KS, sd.Xhi, sd.Xlo);
  BPMF_CUDA_CHECK(cudaGetLastError());
  h->kernels += 1;
  return BPMF_OK;
}

}  // namespace gb
