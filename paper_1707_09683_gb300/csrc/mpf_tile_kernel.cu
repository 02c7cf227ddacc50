// mpf_tile_kernel.cu -- SSV (Alg. 7) and MSV (Alg. 2) for models longer
// than the striped shared-memory table holds, tiled along the model.
//
// SSV has no coupling across a row except its running maximum, so the model
// can be cut into tiles of kTileNodes nodes swept one after the other over
// the whole sequence: the cell at the first node of a tile reads, on the
// previous row, the last node of the tile before (Alg. 7's diagonal), and
// nothing else crosses the cut.  A block of warps takes a batch of
// consecutive length ranks (one sequence per warp, similar lengths) through
// all tiles of its query together: per tile the block stages the tile's
// scores into shared memory, and each warp sweeps its sequence with the
// tile's DP row in registers.  Lane l holds the kTileC consecutive nodes
// l*kTileC + c as kTileC/2 16-bit pairs, pair p = (node p, node p + kTileC/2)
// of the lane, so the diagonal of pair p is the previous row's pair p - 1 as
// it stands and only pair 0 is assembled (from the lane before's last node
// and this lane's node kTileC/2 - 1).  The previous tile's last node reaches
// lane 0 through the warp's boundary column in device memory: one int16 per
// row, written by lane 31 one row later than read (position i + 1 holds row
// i), two buffers by tile parity.
//
// Cells are the unsaturated form r = max(0, r'[k-1] + s) with s = bias -
// cost, one DPX add-then-max per pair of cells; R >= 255 is the overflow
// (the Sec. 2.1 reading of Alg. 7 the other kernels use).  Values above
// 32767 wrap to negative and restart at 0, which only happens after some
// cell has passed 255, so after R >= 255.  Nodes past M score -32768, which
// keeps them at 0.
//
// MSV couples the rows through xE -> xJ -> xB, which a tile cannot see.  As
// in the striped kernels' lazy form, v = max(0, dp - b) follows the same
// recurrence as SSV while the begin score b stays constant, and b moves
// only once xJ passes base.  So the tiles are swept with b held at its
// initial value.  What decides the sequence is the first row whose maximum
// over the whole model passes T = min(base + tec - b, 255 - bias - b - 1),
// and that maximum: a row's maximum passes T exactly when some lane of some
// tile has a cell above T in it, so each lane keeps the first such row of
// its own cells (over the tiles) and its largest cell there, and one warp
// reduction per sequence gives the row and the row maximum.  Then: no such
// row (raw from the largest cell, or, if no cell rose above b, from the
// best single-cell score of the residues); an overflow there (raw 255,
// flag); the last row (raw as if none); or a row after which xB would move
// -- the sequence's rank goes to the query's fallback list, which the exact
// lane-segment kernel scores next (Alg. 2 row by row).
//
// With b held the swept cells are the SSV cells, so the MSV kernel's largest
// cell is also SSV's R: the both-filter variant (MODE_TILE_MSV_SSV) writes
// the SSV outputs from it in the same sweep.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "mpf_internal.h"
#include "mpf_tmem.cuh"

namespace mpf {

namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr uint32_t kNone = 0xffffffffu;
constexpr int kChunks = kTileC / 8;   // 16-byte chunks (4 pairs) per lane and residue row
constexpr int kPairs = kTileC / 2;

// The larger of the two 16-bit halves.
__device__ __forceinline__ int half_max(uint32_t w) { return max((int)(int16_t)(w & 0xffffu), (int)(int16_t)(w >> 16)); }

// One row of the lane's tile segment: v holds the previous row and receives
// this row; `in` is the previous row's score of the node before the lane's
// segment.  rmax collects the row's cells (pair-wise maxima).
__device__ __forceinline__ void tile_row(uint32_t (&v)[kPairs], uint32_t in, const uint4 *srow,
                                         uint32_t &rmax) {
  // Pair 0's diagonal: (node before the segment, node kPairs - 1), previous row.
  const uint32_t d0 = __byte_perm(in, v[kPairs - 1], 0x5410);
#pragma unroll
  for (int q = kChunks - 1; q >= 0; --q) {
    const uint4 s = srow[q * 32];
    const uint32_t sq[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int e = 3; e >= 0; --e) {
      const int p = q * 4 + e;
      v[p] = __viaddmax_s16x2(p > 0 ? v[p - 1] : d0, sq[e], 0u);
    }
    rmax = __vimax3_s16x2(rmax, v[q * 4], v[q * 4 + 1]);
    rmax = __vimax3_s16x2(rmax, v[q * 4 + 2], v[q * 4 + 3]);
  }
}

// A pair of rows of the tensor-memory kernel (mpf_scan_kernel.cuh, row pairs:
// cells and scores in units of 2^kCellShift).

// Pair 0's diagonal: the node before the segment is in the high half of
// in_word (the lane before's last pair, or a boundary-column word).
template <int P>
__device__ __forceinline__ uint32_t first_cell(uint32_t in_word, const uint32_t (&v)[P]) {
  return __byte_perm(in_word, v[P - 1], 0x5432);
}
// First row: sums, not clamped.
template <int P>
__device__ __forceinline__ void pair_row_first(uint32_t (&v)[P], uint32_t in_word, const uint32_t (&sc)[P],
                                               uint32_t &rmax, uint32_t one) {
  const uint32_t d0 = first_cell(in_word, v);
#pragma unroll
  for (int p = P - 1; p >= 0; --p) {
    v[p] = add_imad(p > 0 ? v[p - 1] : d0, sc[p], one);
    if ((p & 1) == 0) rmax = __vimax3_s16x2(rmax, v[p + 1], v[p]);
  }
}
// Second row: both rows' clamps.
template <int P>
__device__ __forceinline__ void pair_row_second(uint32_t (&v)[P], uint32_t in_word, const uint32_t (&sc)[P],
                                                uint32_t &rmax) {
  const uint32_t d0 = first_cell(in_word, v);
#pragma unroll
  for (int p = P - 1; p >= 0; --p) {
    v[p] = __viaddmax_s16x2_relu(p > 0 ? v[p - 1] : d0, sc[p], sc[p]);
    if ((p & 1) == 0) rmax = __vimax3_s16x2(rmax, v[p + 1], v[p]);
  }
}

// MSV result of one sequence, by the whole warp: V, this lane's largest cell;
// outcome, what the sweep decided (warp-uniform).
enum Outcome { kExact, kOverflow, kRescore };
__device__ __noinline__ void msv_finish(const ScanParams &sp, const QueryDesc &qd, uint32_t r, uint32_t len,
                                        uint32_t orig, int lane, int b, int t, int V, Outcome outcome, bool both) {
  V = __reduce_max_sync(kAll, V);
  if (both && lane == 0) {   // SSV from the same largest cell
    const int raw = min(V, 255);
    const int flag = V >= 255 ? 1 : 0;
    qd.raw2[orig] = (uint8_t)raw;
    qd.flag2[orig] = (uint8_t)flag;
    if (qd.nat2)
      qd.nat2[orig] = flag ? __int_as_float(0x7f800000)
                           : __fsub_rn(__fdiv_rn(__int2float_rn(raw - qd.tbm - qd.tec - 2 * t), qd.scale), 3.0f);
  }
  // No cell rose above b: the best row maximum is the best single-cell
  // score of the residues (per-code maxima stored after the tiles).
  int g = -(1 << 20);
  if (V == 0 && len > 0 && outcome == kExact) {
    const int16_t *smax =
        reinterpret_cast<const int16_t *>(reinterpret_cast<const uint8_t *>(qd.table) + qd.smax_off);
    const int mine = (int)__ldg(smax + lane);
    const uint32_t w0 = __ldg(sp.seq_word + r);
    for (uint32_t j0 = 0; j0 < len; j0 += 32) {
      const uint32_t j = j0 + lane;
      uint32_t x = 0;
      if (j < len) x = (__ldg(sp.residues + w0 + (j >> 2)) >> (8 * (j & 3))) & 0xffu;
      if (!MPF_DCHECK(sp.status, x < 32u)) x = 0;
      const int sx = __shfl_sync(kAll, mine, (int)x);
      if (j < len) g = max(g, sx);
    }
    g = __reduce_max_sync(kAll, g);
  }
  if (lane != 0) return;
  int raw = 0, flag = 0;
  if (len > 0) {
    if (outcome == kOverflow) {
      raw = 255;
      flag = 1;
    } else if (outcome == kRescore) {
      // xB moves: score the sequence exactly.
      const uint32_t k = atomicAdd(qd.fallback_count, 1u);
      if (MPF_DCHECK(sp.status, k < sp.n_seqs)) qd.fallback_ranks[k] = r;
      return;
    } else {
      raw = max(0, b + (V > 0 ? V : g) - qd.tec);
    }
  }
  qd.raw[orig] = (uint8_t)raw;
  qd.flag[orig] = (uint8_t)flag;
  if (qd.nat)
    qd.nat[orig] = flag ? __int_as_float(0x7f800000)
                        : __fsub_rn(__fdiv_rn(__int2float_rn(raw - t - qd.base), qd.scale), 3.0f);
}

template <bool MSV, bool BOTH = false>
__global__ void __launch_bounds__(kTileWarps * 32) tile_kernel(ScanParams sp) {
  static_assert(MSV || !BOTH, "the both-filter sweep is the MSV sweep");
  // Shared memory: the tile's scores, [code][chunk][lane] x 4 pairs.
  extern __shared__ __align__(16) uint4 tsm[];
  __shared__ uint32_t s_item;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int W = blockDim.x >> 5;
  constexpr int kTileWords = 32 * kChunks * 32;   // uint4 per tile
  const uint64_t cw = (uint64_t)blockIdx.x * W + warp;
  // This warp's two boundary columns (int16 per row, position i + 1 = row i).
  int16_t *colbuf = reinterpret_cast<int16_t *>(sp.tile_col + cw * 2 * (uint64_t)sp.tile_col_stride);
  const uint32_t col_elems = sp.tile_col_stride / 2;
  // Debug builds: the table and this warp's columns within their buffers.
  if (!MPF_DCHECK(sp.status, (size_t)kTileWords * 16 <= dynamic_smem_bytes() &&
                                 (cw + 1) * 2 * sp.tile_col_stride <= sp.tile_col_bytes &&
                                 (sp.tile_col_stride & 15) == 0))
    return;

  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(sp.item_counter, 1u);
    __syncthreads();
    uint64_t rem = s_item;
    __syncthreads();   // read by all before the next item's write
    // Item: the rem-th batch of W consecutive selected ranks of a query.
    uint32_t qi = 0;
    uint64_t n_sel = 0;
    for (; qi < sp.n_queries; ++qi) {
      const QueryDesc &qd = sp.queries[qi];
      n_sel = qd.ranks ? (uint64_t)*qd.n_ranks : (uint64_t)sp.n_seqs;
      const uint64_t nb = (n_sel + W - 1) / W;
      if (rem < nb) break;
      rem -= nb;
    }
    if (qi == sp.n_queries) break;
    const QueryDesc &qd = sp.queries[qi];
    const uint64_t ri = rem * W + warp;
    bool active = ri < n_sel && MPF_DCHECK(sp.status, n_sel <= sp.n_seqs);
    uint32_t r = 0, w0 = 0, len = 0, orig = 0;
    if (active) {
      r = qd.ranks ? __ldg(qd.ranks + ri) : (uint32_t)ri;
      active = MPF_DCHECK(sp.status, r < sp.n_seqs);
    }
    if (active) {
      w0 = __ldg(sp.seq_word + r);
      len = __ldg(sp.seq_len + r);
      orig = __ldg(sp.seq_orig + r);
      // The columns hold positions 0..len, and the prefetch reads up to
      // position len + 10.
      active = MPF_DCHECK(sp.status, (uint64_t)w0 + ((len + 3u) >> 2) <= sp.n_words && orig < sp.n_seqs &&
                                         (uint64_t)len + 11 <= col_elems);
    }
    const int tj = qd.tjb ? (int)__ldg(qd.tjb + min(len, qd.n_tjb - 1u)) : qd.tjb_fixed;
    // MSV: the begin score held over the tiles, and the threshold T.
    const int b = min(min(255, max(0, qd.base - (tj + qd.tbm))), 255 - qd.bias);
    const int T = min(qd.base + qd.tec - b, 255 - qd.bias - b - 1);
    uint32_t frow = kNone;   // MSV: this lane's first row with a cell above T
    int fval = -1;
    const int nt = (int)((qd.M + kTileNodes - 1) / kTileNodes);
    uint32_t rmax = 0;   // running maximum, two 16-bit halves
    for (int t = 0; t < nt; ++t) {
      __syncthreads();   // every warp is done with the previous tile
      const uint4 *g = qd.table + (size_t)t * kTileWords;
      for (int i = threadIdx.x; i < kTileWords; i += blockDim.x) tsm[i] = __ldg(g + i);
      __syncthreads();
      if (!active) continue;
      const int16_t *cin = colbuf + (size_t)((t + 1) & 1) * col_elems;   // previous tile's column
      int16_t *cout = colbuf + (size_t)(t & 1) * col_elems;              // this tile's column
      const bool first = t == 0, write = t + 1 < nt;
      if (write && lane == 31) cout[0] = 0;   // row -1
      uint32_t v[kPairs];
#pragma unroll
      for (int p = 0; p < kPairs; ++p) v[p] = 0u;
      const uint4 *sbase = tsm + lane;
      // Rolling prefetch of the boundary column, four rows per 64-bit word.
      uint2 cur = make_uint2(0, 0), nxt = make_uint2(0, 0);
      if (lane == 0 && !first) {
        cur = __ldcg(reinterpret_cast<const uint2 *>(cin));
        nxt = __ldcg(reinterpret_cast<const uint2 *>(cin) + 1);
      }
      for (uint32_t i0 = 0; i0 < len; i0 += 4) {
        const uint32_t word = __ldg(sp.residues + w0 + (i0 >> 2));
        uint2 c = cur;
        if (lane == 0 && !first) {
          cur = nxt;
          nxt = __ldcg(reinterpret_cast<const uint2 *>(cin) + (i0 >> 2) + 2);
        }
        const uint32_t xs[4] = {__byte_perm(word, 0u, 0x4440), __byte_perm(word, 0u, 0x4441),
                                __byte_perm(word, 0u, 0x4442), __byte_perm(word, 0u, 0x4443)};
        const uint32_t cs[4] = {c.x & 0xffffu, c.x >> 16, c.y & 0xffffu, c.y >> 16};
        uint32_t rq[4] = {0u, 0u, 0u, 0u};   // MSV: this lane's maxima of the four rows
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (i0 + u < len) {
            uint32_t x = xs[u];
            if (!MPF_DCHECK(sp.status, x < 32u)) x = 0;
            // The node before the lane's segment, previous row: the lane
            // before's last node; for lane 0 the previous tile's last node.
            uint32_t in = __shfl_up_sync(kAll, v[kPairs - 1] >> 16, 1);
            if (lane == 0) in = cs[u];
            tile_row(v, in, sbase + x * (kChunks * 32), MSV ? rq[u] : rmax);
            if (write && lane == 31) cout[i0 + u + 1] = (int16_t)(v[kPairs - 1] >> 16);
          }
        }
        if (MSV) {
          // (Cells are >= 0 until an overflow, so the relu forms are exact.)
          const uint32_t r4 = __vimax3_s16x2(rq[0], rq[1], __vimax_s16x2_relu(rq[2], rq[3]));
          rmax = __vimax_s16x2_relu(rmax, r4);
          // The first of these rows with a cell above T, if not later than
          // this lane's first so far (rows after it cannot matter; the same
          // row in another tile keeps the larger cell).  Rows past the end
          // hold 0, which T = -1 would count: they are left out.
          if (i0 <= frow && half_max(r4) > T) {
#pragma unroll
            for (int u = 3; u >= 0; --u) {
              const int mu = half_max(rq[u]);
              const uint32_t row = i0 + u;
              if (mu > T && row < len) {
                if (row < frow) {
                  frow = row;
                  fval = mu;
                } else if (row == frow) {
                  fval = max(fval, mu);
                }
              }
            }
          }
        }
      }
    }
    if (MSV) {
      if (active) {
        // The first row with a cell above T, and its maximum.
        const uint32_t row = __reduce_min_sync(kAll, frow);
        const int m = __reduce_max_sync(kAll, frow == row ? fval : -1);
        const Outcome o = row == kNone ? kExact : b + m >= 255 - qd.bias ? kOverflow : row + 1 < len ? kRescore : kExact;
        msv_finish(sp, qd, r, len, orig, lane, b, tj, half_max(rmax), o, BOTH);
      }
      continue;
    }
    // R over the sequence: the largest half of any lane.
    int R = 0;
    if (active) R = half_max(rmax);
    R = __reduce_max_sync(kAll, R);
    if (active && lane == 0) {
      const int raw = min(R, 255);
      const int flag = R >= 255 ? 1 : 0;
      qd.raw[orig] = (uint8_t)raw;
      qd.flag[orig] = (uint8_t)flag;
      if (qd.nat)
        qd.nat[orig] = flag ? __int_as_float(0x7f800000)
                            : __fsub_rn(__fdiv_rn(__int2float_rn(raw - qd.tbm - qd.tec - 2 * tj), qd.scale), 3.0f);
    }
  }
}

// The tensor-memory variant: blocks of kTileWarpsTm warps, one block per SM
// (it allocates all of the SM's TMEM columns).  The tile's scores are not
// staged in shared memory: every lane quarter of TMEM holds the whole tile,
// code x's P words of lane l at columns x * P .. + P - 1 of the quarter's
// lane l (32 codes x 16 words = the 512 columns, or 25 x 20), and warp w
// reads quarter w mod 4.  Warp w fills codes 8 (w / 4) .. + 7 of its quarter
// from the tile in device memory.  One sequence per warp makes the residue
// code of a row warp-uniform, so a row's P words are one or two tcgen05.ld
// at one column address, issued a row ahead into the other of two register
// buffers.
//
// The sweep keeps the largest cell V only, which decides MSV as in the striped
// held pass: at or above 255 - bias - b some row overflowed, at most T the
// held rows are exact, in between the sequence goes to the fallback list.
// Rows go in pairs (16 ALU instructions for 16 words instead of 24).
// Eight rows per loop turn, the words ahead in two registers each loaded in
// place and lane 0's boundary word added instead of selected: a row of 16
// words has 24 instructions of cell work, and what surrounds it is what this
// saves.  Measured before / after with tiles of 16 words, 20,000 sequences
// (M = 5,000: SSV 1.79 / 1.71 ms, both filters 2.46 / 2.27; M = 3,500: SSV
// 1.43 / 1.37) and 5,000 (M = 10,000: SSV 2.99 / 2.64).  ncu, M = 5,000: 42
// instructions per row, 24 of them on the ALU pipe, which is 81% busy.
template <int P>
__device__ __forceinline__ void tile_ld(uint32_t (&r)[P], uint32_t a) {
  static_assert(P == 16 || P == 20, "words per lane");
  tm_ld_pow2<16>(r, a);
  if constexpr (P == 20) tm_ld_at<4, 16>(r + 16, a);
}

template <bool MSV, bool BOTH, int P>
__global__ void __launch_bounds__(kTileWarpsTm * 32, 1) tile_kernel_tm(ScanParams sp) {
  static_assert(MSV || !BOTH, "the both-filter sweep is the MSV sweep");
  constexpr int kCodes = P == kPairs ? 32 : kWideTileCodes;   // rows in TMEM
  static_assert(kCodes * P <= (int)kTmemColumns && kTileWarpsTm == 16, "a tile fits a lane quarter");
  __shared__ uint32_t s_item, s_tmem;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int W = blockDim.x >> 5;
  constexpr int kRowWords = P / 4 * 32, kTileWords = 32 * kRowWords;   // uint4 per code and per tile
  const uint64_t cw = (uint64_t)blockIdx.x * W + warp;
  // Boundary columns of 32-bit words: position i + 1 holds row i's last
  // pair of lane 31 (its last node in the high half), read by the next tile's lane 0.
  uint32_t *colbuf = reinterpret_cast<uint32_t *>(sp.tile_col + cw * 2 * (uint64_t)sp.tile_col_stride);
  const uint32_t col_elems = sp.tile_col_stride / 4;
  // Debug builds: the block shape and the block's columns within their
  // buffers (a block-uniform test, before the allocation).
  if (!MPF_DCHECK(sp.status, W == kTileWarpsTm &&
                                 ((uint64_t)blockIdx.x + 1) * W * 2 * sp.tile_col_stride <= sp.tile_col_bytes &&
                                 (sp.tile_col_stride & 15) == 0))
    return;
  if (warp == 0) tm_alloc(&s_tmem);
  tm_fence_before();
  __syncthreads();
  tm_fence_after();
  const uint32_t tm_lane = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const uint32_t not_first = lane != 0;

  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(sp.item_counter, 1u);
    __syncthreads();
    uint64_t rem = s_item;
    __syncthreads();
    uint32_t qi = 0;
    uint64_t n_sel = 0;
    for (; qi < sp.n_queries; ++qi) {
      const QueryDesc &qd = sp.queries[qi];
      n_sel = qd.ranks ? (uint64_t)*qd.n_ranks : (uint64_t)sp.n_seqs;
      const uint64_t nb = (n_sel + W - 1) / W;
      if (rem < nb) break;
      rem -= nb;
    }
    if (qi == sp.n_queries) break;   // block-uniform
    const QueryDesc &qd = sp.queries[qi];
    const uint64_t ri = rem * W + warp;
    bool active = ri < n_sel && MPF_DCHECK(sp.status, n_sel <= sp.n_seqs);
    uint32_t r = 0, w0 = 0, len = 0, orig = 0;
    if (active) {
      r = qd.ranks ? __ldg(qd.ranks + ri) : (uint32_t)ri;
      active = MPF_DCHECK(sp.status, r < sp.n_seqs);
    }
    if (active) {
      w0 = __ldg(sp.seq_word + r);
      len = __ldg(sp.seq_len + r);
      orig = __ldg(sp.seq_orig + r);
      active = MPF_DCHECK(sp.status, (uint64_t)w0 + ((len + 3u) >> 2) <= sp.n_words && orig < sp.n_seqs &&
                                         (uint64_t)len + 11 <= col_elems);
    }
    const int tj = qd.tjb ? (int)__ldg(qd.tjb + min(len, qd.n_tjb - 1u)) : qd.tjb_fixed;
    const int b = min(min(255, max(0, qd.base - (tj + qd.tbm))), 255 - qd.bias);
    const int T = min(qd.base + qd.tec - b, 255 - qd.bias - b - 1);
    const int nt = (int)tiles_of((int)qd.M, P);
    uint32_t rmax = 0, rmax2 = 0;   // running maxima over second and first rows of pairs
    for (int t = 0; t < nt; ++t) {
      // Every thread waited for its loads of the previous tile: order them
      // before this tile's TMEM writes.
      tm_fence_before();
      __syncthreads();
      tm_fence_after();
      {
        const uint4 *g = qd.table + (size_t)t * kTileWords + lane;
        const int x0 = 8 * (warp >> 2);
#pragma unroll 2
        for (int x = x0; x < min(x0 + 8, kCodes); ++x) {
          uint4 c[P / 4];
#pragma unroll
          for (int i = 0; i < P / 4; ++i) c[i] = __ldg(g + x * kRowWords + 32 * i);
          const uint32_t col = tm_lane + (uint32_t)(x * P);
#pragma unroll
          for (int i = 0; i < P / 4; ++i) tm_st4(col + 4 * i, c[i].x, c[i].y, c[i].z, c[i].w);
        }
        tm_wait_st();
      }
      tm_fence_before();
      __syncthreads();
      tm_fence_after();
      if (!active) continue;
      const uint32_t *cin = colbuf + (size_t)((t + 1) & 1) * col_elems;
      uint32_t *cout = colbuf + (size_t)(t & 1) * col_elems;
      const bool first = t == 0, write = t + 1 < nt;
      if (write && lane == 31) cout[0] = 0;
      uint32_t v[P];
#pragma unroll
      for (int p = 0; p < P; ++p) v[p] = 0u;
      // Residue words and boundary words (0 but in lane 0) of the rows ahead:
      // A, the next four rows, and B, the four after.  Each is loaded again as
      // soon as its rows are done, so a turn of eight rows moves no registers.
      auto word_at = [&](uint32_t i) {   // codes masked to 0..31, the tile's columns
        return (i < len ? __ldg(sp.residues + w0 + (i >> 2)) : 0u) & 0x1f1f1f1fu;
      };
      const bool bound_in = lane == 0 && !first, bound_out = write && lane == 31;
      uint4 cA = make_uint4(0, 0, 0, 0), cB = make_uint4(0, 0, 0, 0);
      if (bound_in) {
        cA = __ldcg(reinterpret_cast<const uint4 *>(cin));
        cB = __ldcg(reinterpret_cast<const uint4 *>(cin) + 1);
      }
      uint32_t wA = word_at(0), wB = word_at(4);
      // Score rows of the current and the next row.  Codes are < kCodes
      // in a sequence; the load issued for the row after the last one takes any
      // code (only waited for).
      uint32_t TA[P], TB[P];
      tile_ld<P>(TA, tm_lane + (wA & 255u) * (uint32_t)P);
      // One row: wait for its scores, issue the next row's load (code xn),
      // update.  The lane before's last node (high half) of the previous row
      // comes by shuffle; lane 0 takes the boundary word, by a multiply-add
      // on the FMA pipe.
      auto one_row = [&](const int u, uint32_t (&Tc)[P], uint32_t (&Tn)[P], uint32_t xn, uint32_t c,
                         uint32_t *out, bool last) {
        tm_wait_ld<P>(Tc);
        tile_ld<P>(Tn, tm_lane + xn * (uint32_t)P);
        const uint32_t in = __shfl_up_sync(kAll, v[P - 1], 1) * not_first + c;
        if (u & 1)
          pair_row_second(v, in, Tc, rmax);
        else
          pair_row_first(v, in, Tc, rmax2, sp.one);
        // The word handed on at the end of a turn carries no fraction past a
        // clearing row of the next tile.
        if (bound_out) out[u + 1] = last ? v[P - 1] & kCellMask2 : v[P - 1];
      };
      auto four_rows = [&](uint32_t w, const uint4 &c, uint32_t wn, uint32_t *out, bool turn_end) {
        one_row(0, TA, TB, __byte_perm(w, 0u, 0x4441), c.x, out, false);
        one_row(1, TB, TA, __byte_perm(w, 0u, 0x4442), c.y, out, false);
        one_row(2, TA, TB, __byte_perm(w, 0u, 0x4443), c.z, out, false);
        one_row(3, TB, TA, wn & 255u, c.w, out, turn_end);
      };
      uint32_t until_clear = 4 * kClearSteps;
      uint32_t i0 = 0;
      const uint4 *cnext = reinterpret_cast<const uint4 *>(cin) + 2;
      for (; i0 + 8 <= len; i0 += 8, cnext += 2) {   // warp-uniform: no row tests
        four_rows(wA, cA, wB, cout + i0, false);
        wA = word_at(i0 + 8);
        if (bound_in) cA = __ldcg(cnext);
        four_rows(wB, cB, wA, cout + i0 + 4, true);
        wB = word_at(i0 + 12);
        if (bound_in && i0 + 8 < len) cB = __ldcg(cnext + 1);
        until_clear -= 8;
        if (until_clear == 0) {   // drop the sums' carries
          until_clear = 4 * kClearSteps;
#pragma unroll
          for (int p = 0; p < P; ++p) v[p] &= kCellMask2;
        }
      }
      if (i0 + 4 <= len) {
        four_rows(wA, cA, wB, cout + i0, false);
        i0 += 4;
        wA = wB;
        cA = cB;
      }
      if (i0 < len) one_row(0, TA, TB, __byte_perm(wA, 0u, 0x4441), cA.x, cout + i0, false);
      if (i0 + 1 < len) one_row(1, TB, TA, __byte_perm(wA, 0u, 0x4442), cA.y, cout + i0, false);
      if (i0 + 2 < len) one_row(2, TA, TB, __byte_perm(wA, 0u, 0x4443), cA.z, cout + i0, false);
      tm_wait_ld<P>(TB);
      tm_wait_ld<P>(TA);   // the load issued after the last row
    }
    const int V = half_max(__vmaxs2(rmax, rmax2)) >> kCellShift;
    if (MSV) {
      if (active) {
        const int m = __reduce_max_sync(kAll, V);
        const Outcome o = b + m >= 255 - qd.bias ? kOverflow : m > T ? kRescore : kExact;
        msv_finish(sp, qd, r, len, orig, lane, b, tj, V, o, BOTH);
      }
      continue;
    }
    int R = 0;
    if (active) R = V;
    R = __reduce_max_sync(kAll, R);
    if (active && lane == 0) {
      const int raw = min(R, 255);
      const int flag = R >= 255 ? 1 : 0;
      qd.raw[orig] = (uint8_t)raw;
      qd.flag[orig] = (uint8_t)flag;
      if (qd.nat)
        qd.nat[orig] = flag ? __int_as_float(0x7f800000)
                            : __fsub_rn(__fdiv_rn(__int2float_rn(raw - qd.tbm - qd.tec - 2 * tj), qd.scale), 3.0f);
    }
  }
  tm_fence_before();
  __syncthreads();
  if (warp == 0) {
    tm_fence_after();
    tm_dealloc(s_tmem);
  }
}

}  // namespace

KernelFn tile_kernel_fn(int mode, bool tm, bool wide) {
  if (tm && wide)
    return mode == MODE_TILE_MSV_SSV ? tile_kernel_tm<true, true, kWideTileWords>
           : mode == MODE_TILE_MSV   ? tile_kernel_tm<true, false, kWideTileWords>
                                     : tile_kernel_tm<false, false, kWideTileWords>;
  if (tm)
    return mode == MODE_TILE_MSV_SSV ? tile_kernel_tm<true, true, kPairs>
           : mode == MODE_TILE_MSV   ? tile_kernel_tm<true, false, kPairs>
                                     : tile_kernel_tm<false, false, kPairs>;
  return mode == MODE_TILE_MSV_SSV ? tile_kernel<true, true> : mode == MODE_TILE_MSV ? tile_kernel<true> : tile_kernel<false>;
}

}  // namespace mpf
