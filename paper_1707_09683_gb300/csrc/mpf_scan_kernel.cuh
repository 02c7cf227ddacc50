// mpf_scan_kernel.cuh -- the MSV / SSV scan kernel for sm_103a.
//
// One kernel serves the single-query scan and the batched scan: resident
// thread blocks pull work items (query, database shard) from a counter,
// stage the query's striped cost table in shared memory, and stream the
// shard's sequences through their warps.
//
// Parallel decomposition (the five tiers of Sec. 3.1, re-mapped to GB300):
//   tier 1  thread blocks on the 152 SMs pull work items;
//   tier 2  warps pull batches of 32 / LG consecutive length ranks of their
//           item's shard from a shared-memory counter and run them in lock
//           step (sequences are length-sorted and shards interleave the
//           ranks, so the lengths of a batch nearly agree and a block's
//           batches shrink as it drains -- this replaces the pre-built warp
//           data blocks of Sec. 3.2 and Alg. 1);
//   tier 3  a group of LG lanes holds one sequence's DP row, striped over the
//           group (Farrar layout: cell k = (2*lane + half) * H + word);
//   tier 4  32 / LG groups per warp score different sequences at once;
//   tier 5  every 32-bit register holds two 16-bit cells updated by one
//           DPX instruction (byte SIMD -- vaddus4 etc. of Alg. 2 -- is not a
//           native instruction on sm_103, the 16x2 DPX forms are).
//
// Cell arithmetic.  With s = bias - cost (a signed score) and b = min(xB,
// 255 - bias), the byte update of Alg. 2 is exactly
//     dp = max(0, max(dp'[k-1], b) + s)
// because every dp' of a row that did not overflow is below 255 - bias, so
// clamping xB reproduces the saturating bias addition.  The SSV update of
// Alg. 7 is r = max(0, r'[k-1] + s) kept unsaturated in 16 bits; R >= 255 is
// the overflow and R is capped at the end.  MSV_FAST keeps v = max(0, dp - b),
// which follows the SSV recurrence while b is constant; b only changes when
// xJ passes base, so each lane keeps a running maximum and the group reduces
// it (Alg. 6) only on rows where some lane crosses the threshold at which xJ
// would pass base or the score would overflow.  Such a row updates xJ and b,
// rebases the cells and starts over with the threshold at which xJ would
// change again, so the rows in between stay reduction-free.  Before the first
// one a row can raise the running maximum by at most `bias`, so a warp runs
// four rows without any per-row test whenever no lane is within 4 * bias of T.
//
// Row pairs (SSV, held MSV and the two together, integer cells).  The kernels
// are bound by the integer ALU pipe, on which a DPX instruction takes two
// cycles per warp and scheduler: one add-then-max per word and row and half a
// 3-input max for the running maximum, 1.5 per word.  Two rows at a time need
// less, because the first row's clamp at zero can move into the second:
//     t = v + s1,   v'' = max(0, max(0, t) + s2) = max(0, s2, t + s2),
// one DPX instruction (__viaddmax_s16x2_relu(t, s2, s2)), with the running
// maximum over t and v''.  t is a plain 32-bit sum of the packed words, which
// the FMA pipe does (IMAD, add_imad).  That leaves 1.0 ALU instruction per
// word.  The sum carries from the low into the high half when the low sum is
// not negative and s1 is, so cells hold scores in units of 2^kCellShift: the
// carries (at most one per pair of rows along a diagonal) stay below a unit,
// where they change no comparison of scores, no clamp and no maximum (shifted
// back down at the end), and are cleared every kClearSteps steps.  Measured
// (GB300, clock64, 16 words per lane, table in registers): 52.7 words per
// clock and SM against 42.4 for two rows of add-then-max.
//
// Mixed sets (MIX).  A warp's lanes are dealt to several queries of any
// length, each with as many lanes as its nodes fill at H words per lane, and
// all score the warp's one sequence: the rows of every lane come from tensor
// memory at one residue's column, as for one query on 32 lanes.  A batch's
// shorter queries otherwise run kernels whose groups read different residues
// from shared memory, at half the rate (GCUPS alone, 100,000 sequences: M =
// 48 / 100 / 200 / 400 / 800 5,570 / 8,350 / 12,430 / 16,280 / 17,480; a set
// of 48, 200, 400 and 800 on 24 words 24,890).
//
// Segments.  A path of the SSV recurrence (and of held MSV, the same cells)
// visits at most M rows, so the largest cell of rows a .. b - 1 is known from
// a zero row M rows before a: a long sequence splits into segments of
// seg_rows rows that different groups score, each with seg_overlap >= M rows
// before it.  The units' maxima are combined by the last unit to finish
// (a counter per sequence), which writes the outputs.  Without this a launch
// ends with its longest sequences, one lane group each: 35,000 residues took
// milliseconds on a database that needs a tenth of one otherwise.  The host
// splits only sequences longer than the launch's rows per lane group
// (plan_split in mpf_api.cu), where the rows added by the overlap run on
// lanes that would idle.  MSV_FAST rescores such a sequence segment by
// segment, in order, and skips the segments whose largest cell is at most T:
// with b constant over a segment no row of it can change xJ.  A segment
// entered after a gap starts from a zero row seg_overlap <= seg_rows rows
// earlier, in the skipped segment, over which b did not change either.  One
// that follows the segment before it goes on with the group's cells.
//
// The F16 modes hold the same integers as IEEE half values and update a cell
// pair with one fused add-and-clamp-at-zero (HFMA2.RELU, v * 1 + s), which
// issues on the FMA pipe instead of the integer ALU pipe that the DPX
// instructions use.  Every value a scored cell takes before its sequence
// has reached the overflow threshold is an integer of magnitude below 2048,
// which half precision represents exactly; later values only need to stay
// above the threshold, and rounding is monotone.  Running maxima compare the
// half bit patterns of non-negative values as unsigned integers.
//
// Tensor-memory variant (TM, one sequence per warp, LG = 32).  The table is
// staged in shared memory as usual; then the first HT words of each lane's
// row are copied into the block's tensor memory (thread t of warp w owns TMEM
// lane 32 (w mod 4) + t: its row of code x is columns x * HT .. x * HT + HT -
// 1), for all 33 residue rows (TM_ALL: all H words up to 14, else 12) or, when
// every code of the database is below 20, for those codes and the padding
// code (TM_FEW: 24 words).  The kernel was held by shared memory's 128 B per
// clock for the words past HT: of a lane's 38 words (M = 2405) 26 came from
// there, 14 do with TM_FEW, and up to 24 words (M = 1536) none.  A row updates
// its words past HT from shared memory, then its TMEM words from the highest
// down; they come in two loads, each issued half a row ahead, so that a lane
// holds one row's TMEM words and not two (24 words in two buffers would not
// leave room for the cells).  Every row takes the same path, so the kernel
// has no per-row branch on the table source.  Measured (GB300, 60,000
// sequences, SSV, GCUPS): M = 2405 22,790 with TM_ALL, 25,140 with TM_FEW; 16
// queries of M = 100 packed 23,950.  ncu at M = 2405: ALU pipe 67% -> 75%.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include <type_traits>

#include "mpf_internal.h"
#include "mpf_tmem.cuh"

namespace mpf {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ int half_max(uint32_t w) {  // both halves are >= 0
  return max((int)(w & 0xffffu), (int)(w >> 16));
}

__device__ __forceinline__ uint32_t pack2(int v) {
  const uint32_t h = (uint32_t)(uint16_t)(int16_t)v;
  return (h << 16) | h;
}

__device__ __forceinline__ int sat8(int v) { return min(255, max(0, v)); }

// PTX prmt in its default mode: each selector nibble picks one of the eight
// bytes of (a, b) with its low three bits, and with its high bit set copies
// that byte's sign bit into all eight bits (the CUDA __byte_perm intrinsic
// uses only the low three bits).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

template <int LG>
__device__ __forceinline__ int group_max(int v) {
#pragma unroll
  for (int off = LG / 2; off >= 1; off >>= 1) v = max(v, __shfl_xor_sync(kFull, v, off, LG));
  return v;
}

__device__ __forceinline__ float nat_score(int num, float scale) {
  return __fsub_rn(__fdiv_rn(__int2float_rn(num), scale), 3.0f);
}

// Order-preserving key of a cell value: the integer in cell units, or the
// bit pattern of a non-negative half.
template <bool F16>
__device__ __forceinline__ int value_key(int v) {
  if (!F16) return v << kCellShift;
  return (int)__half_as_ushort(__int2half_rn(v));
}

template <bool F16>
__device__ __forceinline__ int key_value(int k) {
  if (!F16) return k >> kCellShift;
  if (k >= 0x7c00) return 1 << 20;   // +inf: far above every threshold
  return __half2int_rn(__ushort_as_half((unsigned short)k));
}

__device__ __forceinline__ uint32_t hfma2_relu_u32(uint32_t a, uint32_t b, uint32_t c) {
  const __half2 r = __hfma2_relu(*reinterpret_cast<const __half2 *>(&a),
                                 *reinterpret_cast<const __half2 *>(&b),
                                 *reinterpret_cast<const __half2 *>(&c));
  return *reinterpret_cast<const uint32_t *>(&r);
}

__device__ __forceinline__ uint32_t pack2_half(int v) {
  const uint32_t h = (uint32_t)__half_as_ushort(__int2half_rn(v));
  return (h << 16) | h;
}

// group_max for groups of any width side by side: this lane is lane gl of its
// group of `width` (every lane gets its group's maximum).
__device__ __forceinline__ int mixed_max(int v, int lane, int gl, int width) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_down_sync(kFull, v, off);
    if (gl + off < width) v = max(v, y);
  }
  return __shfl_sync(kFull, v, lane - gl);
}

template <int LG, int H, int MODE, int TM = TM_NONE, int QP = 1, bool MIX = false>
__global__ void __launch_bounds__(kBlockThreads, 1) scan_kernel(ScanParams p) {
  static_assert((H % 4 == 0 || H % 4 == 2) && H >= 4 && H <= kMaxWords, "words per lane");
  static_assert(!TM || ((LG == 32 || QP * LG == 32) && H >= kTmMinWords && MODE != MODE_MSV_DIRECT &&
                        MODE != MODE_MSV_FAST && MODE != MODE_MSV_FAST_F16),
                "tensor-memory variant");
  static_assert(QP == 1 || (TM && QP * LG == 32), "queries per warp");
  static_assert(!MIX || (TM == TM_FEW && LG == 32 && QP == 1 && tm_words(H, TM) == H), "mixed sets");
  constexpr int HT = tm_words(H, TM);   // words per lane from TMEM
  static_assert(HT == H || HT % 4 == 0, "shared-memory words start on a chunk");
  constexpr int Q = H / 4;               // full 4-word chunks per lane and row
  constexpr bool kTail = (H % 4) == 2;   // two more words from the tail region
  constexpr int NT = LG >= 16 ? 1 : 16 / LG;
  static_assert(LG == 1 || LG == 2 || LG == 4 || LG == 8 || LG == 16 || LG == 32, "lanes");
  constexpr int NC = LG >= 8 ? 1 : 8 / LG;
  constexpr int G = 32 / LG;
  constexpr bool kF16 = (MODE == MODE_SSV_F16 || MODE == MODE_MSV_FAST_F16 || MODE == MODE_MSV_HELD_F16);
  static_assert(QP == 1 || !kF16, "packed sets use integer cells");
  constexpr bool kSSV = (MODE == MODE_SSV || MODE == MODE_SSV_F16);
  constexpr bool kFast = (MODE == MODE_MSV_FAST || MODE == MODE_MSV_FAST_F16);
  constexpr bool kBoth = (MODE == MODE_MSV_SSV);   // held MSV and SSV outputs from one sweep
  constexpr bool kHeld = (MODE == MODE_MSV_HELD || MODE == MODE_MSV_HELD_F16 || kBoth);
  constexpr bool kDirect = (MODE == MODE_MSV_DIRECT);
  // Modes that may take a sequence in segments (see the file comment).
  constexpr bool kUnits = kSSV || kHeld;
  // SSV and held MSV with integer cells: rows in pairs (see the file comment).
  constexpr bool kPair = !kF16 && (kSSV || kHeld);
  // Where a pair's cells join the running maximum, in two chains: row by row,
  // two words per instruction, or both rows of a word with the second row,
  // words alternating.  The first spreads the ALU work over both rows; long
  // lanes are better off without its reads (GCUPS row by row / both rows,
  // SSV, 60,000 sequences: 20 words 25,300 / 25,150, 26 25,080 / 24,330, 28
  // 25,200 / 26,250, 38 25,420 / 26,140, 46 25,440 / 26,170; with one chain
  // 23,300, 24,850, 25,060, 25,130, 22,810).
  constexpr bool kFoldRows = H <= 26;
  const uint32_t one2 = 0x3c003c00u;   // (1.0, 1.0) as half2
  const uint32_t one = p.one;          // 1, opaque to the compiler (add_imad)
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_item, s_next;
  __shared__ uint32_t s_tmem;

  const int lane = threadIdx.x & 31;
  int gl = lane & (LG - 1), width = LG;   // lane of the group, its lanes (mixed sets: per item)
  const int grp = lane / LG;
  // Byte selector of the diagonal shift: bytes 2, 3 of the lane before's last
  // word, then bytes 0, 1 of this lane's.  With integer cells (0 .. 32767)
  // the group's first lane takes the sign copies of its own byte 1, which
  // are zero; fp16 cells zero it with a select instead.
  uint32_t shift_sel = (LG > 1 && gl != 0) ? 0x5432u : 0x54ddu;
  // QP > 1: the 32 / LG groups of a warp score one sequence against QP
  // queries (the QP consecutive queries of a work item), so every lane of
  // the warp reads the same residue and the TMEM column of a row is uniform.
  // Every lane of a warp follows the same sequence: a warp reduction (whose
  // result is uniform) hands each residue word to the rows.
  constexpr bool kUniform = TM != TM_NONE;
  constexpr bool kMapPad = TM == TM_FEW && HT == H;
  // Mixed sets: item i scores set i / n_shards, whose lanes belong to queries
  // as p.mix_lanes says (query, lane of its group, width; width 0: no query).
  const uint32_t n_items = (MIX ? p.n_sets : (p.n_queries + QP - 1) / QP) * p.n_shards;
  const int warp = (int)(threadIdx.x >> 5);
  uint32_t tm_lane = 0;   // TMEM address of this warp's lane quarter, column 0
  if constexpr (TM) {
    if (warp == 0) tm_alloc(&s_tmem);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    tm_lane = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
  }
  // TMEM rows: codes 0 .. tm_pad - 1, then the padding code.
  const uint32_t tm_pad = TM == TM_FEW ? p.tm_rows - 1u : (uint32_t)kTableRows - 1u;

  for (;;) {
    if (threadIdx.x == 0) {
      s_item = atomicAdd(p.item_counter, 1u);
      s_next = 0u;
    }
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= n_items) break;
    const uint32_t shard = item % p.n_shards;
    uint32_t qbase = item / p.n_shards * QP;
    uint32_t qi = qbase + (QP > 1 ? (uint32_t)grp : 0u);
    if constexpr (MIX) {
      const uint32_t m = __ldg(p.mix_lanes + qbase * 32 + lane);
      qbase = __ldg(p.mix_lanes + qbase * 32) & 0xffffu;   // lane 0 always has a query
      width = (int)(m >> 24);
      gl = (int)((m >> 16) & 0xffu);
      qi = width ? m & 0xffffu : p.n_queries;
      shift_sel = gl != 0 ? 0x5432u : 0x54ddu;
    }
    // QP > 1: a set may have empty slots (descriptors without a table, after
    // its queries), and the last item fewer queries.
    const bool qvalid = qi < p.n_queries && (QP == 1 || p.queries[qi].table != nullptr);
    const QueryDesc *qd = p.queries + (qvalid ? qi : qbase);
    const uint32_t tstride = QP > 1 ? p.qp_table_stride : 0u;   // shared-memory bytes per query's table
    // Debug builds: the table must fit the block's shared memory and the
    // selected ranks the database (the item is skipped otherwise).
    if (!MPF_DCHECK(p.status, (QP > 1 ? qd->table_bytes <= tstride && tstride % 16 == 0 &&
                                            QP * tstride <= dynamic_smem_bytes() && !qd->ranks
                                      : qd->table_bytes <= dynamic_smem_bytes()) &&
                                  p.pad_word < p.n_words && (!qd->ranks || *qd->n_ranks <= p.n_seqs))) {
      __syncthreads();
      continue;
    }
    // A shard without sequences (a short rank list, such as the few
    // sequences a held MSV pass leaves for rescoring) stages nothing.
    // So does a query whose list another launch takes.
    const uint64_t n_sel = qd->ranks ? (uint64_t)*qd->n_ranks : (uint64_t)p.n_units;
    if ((uint64_t)shard >= n_sel ||
        (qd->ranks && (n_sel <= qd->more_than || (qd->at_most && n_sel > qd->at_most)))) {
      __syncthreads();
      continue;
    }

    // Stage the striped table(s) (16-byte vector copies, coalesced); with
    // QP > 1 query g's table at g * tstride.
#pragma unroll 1
    for (int g = 0; g < (MIX ? 0 : QP); ++g) {
      if (qbase + (uint32_t)g >= p.n_queries) break;
      const QueryDesc *qg = p.queries + qbase + g;
      if (!qg->table) continue;
      const uint32_t nvec = qg->table_bytes >> 4;
      const uint4 *src = qg->table;
      uint4 *dst = reinterpret_cast<uint4 *>(smem + (uint32_t)g * tstride);
      for (uint32_t i = threadIdx.x; i < nvec; i += blockDim.x) dst[i] = __ldg(src + i);
    }
    __syncthreads();
    // A group past the last query computes on the first query's table and
    // writes nothing (its lanes must still follow the warp's sequence).
    const uint8_t *tbl_base = smem + (QP > 1 && qvalid ? (uint32_t)grp * tstride : 0u);
    const uint8_t *tbl_lane = tbl_base + (QP > 1 ? 0u : (grp % NC) * qd->copy_bytes) + gl * 16;
    // QP > 1: packed tables (one copy of each region; the table stride
    // spreads the groups of a phase over the banks).
    const uint8_t *tail_lane = tbl_base + qd->tail_off + ((QP > 1 ? 0 : grp % NT) * LG + gl) * 8;
    if constexpr (TM) {
      // Copy the first HT words of every lane's row of every code from the
      // staged table into tensor memory: warp q < 4 writes lane quarter q.
      tm_fence_after();
      if constexpr (MIX) {
        // Straight from device memory, rows dealt to the warps of a quarter.
        const uint2 *src = reinterpret_cast<const uint2 *>(qd->table) + (size_t)gl * (H / 2);
        for (uint32_t row = warp >> 2; row <= tm_pad; row += kBlockThreads / 128) {
          const uint32_t x = row == tm_pad ? (uint32_t)kPadCode : row;
          const uint2 *s2 = src + (size_t)x * (uint32_t)width * (H / 2);
          const uint32_t col = tm_lane + row * (uint32_t)HT;
          uint2 w[H / 2];
#pragma unroll
          for (int j = 0; j < H / 2; ++j) w[j] = width ? __ldg(s2 + j) : make_uint2(0xc000c000u, 0xc000c000u);
#pragma unroll
          for (int j = 0; j < H / 2; ++j) tm_st2(col + 2 * j, w[j].x, w[j].y);
        }
        tm_wait_st();
      } else if (warp < 4) {
        for (uint32_t row = 0; row <= tm_pad; ++row) {
          const uint32_t col = tm_lane + row * (uint32_t)HT;
          const uint32_t x = row == tm_pad ? (uint32_t)kPadCode : row;
#pragma unroll
          for (int j = 0; j < HT / 4; ++j) {
            const uint4 s4 = *reinterpret_cast<const uint4 *>(tbl_lane + x * qd->row_bytes + j * LG * 16);
            tm_st4(col + 4 * j, s4.x, s4.y, s4.z, s4.w);
          }
          if constexpr (HT % 4 == 2) {   // HT == H: the two tail words
            const uint2 t2 = *reinterpret_cast<const uint2 *>(tail_lane + x * qd->tail_row_bytes);
            tm_st2(col + 4 * (HT / 4), t2.x, t2.y);
          }
        }
        tm_wait_st();
      }
      tm_fence_before();
      __syncthreads();
      tm_fence_after();
    }

    const int bias = qd->bias, tbm = qd->tbm, tec = qd->tec, base = qd->base;
    const int cap = 255 - bias;
    const float scale = qd->scale;
    const uint8_t *tjb = qd->tjb;
    const uint32_t n_tjb = qd->n_tjb;
    const int tjb_fixed = qd->tjb_fixed;
    uint8_t *out_raw = qd->raw;
    uint8_t *out_flag = qd->flag;
    float *out_nat = qd->nat;
    const uint32_t row_bytes = qd->row_bytes;
    const uint32_t tail_row_bytes = qd->tail_row_bytes;
    const int16_t *smax = reinterpret_cast<const int16_t *>(
        (MIX ? reinterpret_cast<const uint8_t *>(qd->table) : tbl_base) + qd->smax_off);
    auto gmax = [&](int x) { return MIX ? mixed_max(x, lane, gl, width) : group_max<LG>(x); };
    const uint32_t *ranks = qd->ranks;

    for (;;) {
      // ---- take G consecutive length ranks of this shard (one per group;
      // QP > 1: one rank, the same sequence for every group) ----
      uint32_t k0 = 0;
      if (lane == 0) k0 = atomicAdd(&s_next, QP > 1 ? 1u : (uint32_t)G);
      k0 = __shfl_sync(kFull, k0, 0);
      const uint64_t kr = (uint64_t)shard + (uint64_t)(k0 + (QP > 1 ? 0 : grp)) * p.n_shards;
      bool active = kr < n_sel;
      if (!__any_sync(kFull, active)) break;
      // The first units are the segments of the longest sequences.
      uint64_t r = (ranks && active) ? (uint64_t)__ldg(ranks + kr) : kr - p.n_long_units + p.n_long;
      const bool split = kUnits && !ranks && active && kr < p.n_long_units;
      if (split) r = (uint64_t)__ldg(p.unit_rank + kr);
      if (active && !MPF_DCHECK(p.status, r < p.n_seqs)) active = false;

      // Group state (identical in every lane of a group).
      uint32_t wptr = p.pad_word, orig = 0;
      int len = 0, t = 0;
      if (active) {
        wptr = __ldg(p.seq_word + r);
        len = (int)__ldg(p.seq_len + r);
        orig = __ldg(p.seq_orig + r);
        t = tjb ? (int)__ldg(tjb + min((uint32_t)len, n_tjb - 1u)) : tjb_fixed;
        if (!MPF_DCHECK(p.status, (uint64_t)wptr + (uint64_t)((len + 3) >> 2) <= p.n_words &&
                                      orig < p.n_seqs)) {
          active = false;
          wptr = p.pad_word;
          len = 0;
        }
      }
      const uint32_t wstart = wptr;
      // Rows first_row .. first_row + rows - 1: the whole sequence, or this
      // unit's segment after the rows that its paths can come from.
      int first_row = 0, rows = len;
      if (split) {
        const int end = ((int)(kr - __ldg(p.unit_first + r)) + 1) * (int)p.seg_rows;
        first_row = max(end - (int)(p.seg_rows + p.seg_overlap), 0);
        rows = min(end, len) - first_row;
      }
      int xJ = 0;
      int b = min(sat8(base - (t + tbm)), cap);
      uint32_t b2 = pack2(b << kCellShift);
      int T = min(base + tec - b, cap - b - 1);
      int Tnear = 0;           // no trigger possible in 4 rows below it
      uint32_t Tk2 = 0u, Tnear2 = 0u;
      // "Some half of the running maximum is above the key K" as one add and
      // one mask: the halves (keys <= 0x7fff) plus 0x7fff - K reach bit 15
      // exactly when they exceed K, and no sum carries into the other half.
      auto arm = [&]() {
        Tnear = T - 4 * max(bias, 0);
        Tk2 = pack2(0x7fff - value_key<kF16>(max(T, 0)));
        Tnear2 = pack2(0x7fff - value_key<kF16>(max(Tnear, 0)));
      };
      if constexpr (kFast) arm();
      bool done = false, exact = false;

      // Lane state: H words of two 16-bit cells and a running maximum (key).
      uint32_t v[H];
#pragma unroll
      for (int q = 0; q < H; ++q) v[q] = 0u;
      uint32_t vacc = 0u, vacc2 = 0u;   // running maximum (vacc2: the other half of the row pairs' chain)
      int nsteps = 0;          // residue words of the rows
      bool busy = active;      // this group has rows to score
      uint32_t cur = 0u, ahead = 0u;   // the current residue word, and the next one as loaded

      // Tensor-memory words of a row come in two loads, the low words and the
      // high words (processed first, after the words in shared memory); each
      // load is issued while the row before its use is half done, so a lane
      // holds one row's words and not two.  Either load may bring columns of
      // the same row past those it is for; they are not used.
      constexpr int HI = TM == TM_NONE ? 0 : HT <= 12 ? 4 : 8;
      constexpr int LO = HT - HI;
      constexpr int LOW = TM == TM_NONE ? 1 : LO <= 4 ? 4 : LO <= 8 ? 8 : 16;
      static_assert(TM == TM_NONE || (LO >= 4 && LOW <= HT && LO <= 16), "load widths");
      uint32_t tlo[LOW], thi[HI > 0 ? HI : 1];
      auto tm_col = [&](uint32_t xc) -> uint32_t {
        if (!MPF_DCHECK(p.status, xc < (uint32_t)kTableRows)) xc = kPadCode;
        return tm_lane + (TM == TM_FEW && !kMapPad ? min(xc, tm_pad) : xc) * (uint32_t)HT;
      };
      uint32_t tcol = 0;       // TMEM column of the current row's words
      // Lanes held whole in TMEM: padding codes become their TMEM row a word
      // at a time (bit 5 marks them: the database's codes are below 20).
      auto map_pad = [&](uint32_t w) {
        return kMapPad ? w - ((w >> 5) & 0x01010101u) * ((uint32_t)kPadCode - tm_pad) : w;
      };
      // Four rows of one residue word (nxt: the next word).  CHECK: test every
      // row for the MSV threshold (only needed when some lane is near it, or
      // in exact mode).
      auto four_rows = [&](const int step, auto check_tag, const uint32_t nxt) {
        constexpr bool CHECK = decltype(check_tag)::value;
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
         {
          // Rows past the end of a sequence read padding codes: their cells
          // score kNegInf, and the special states must not see them.
          const bool real = busy && (4 * step + rr) < rows;
          uint32_t x = __byte_perm(cur, 0u, 0x4440u + rr);   // residue code of row rr
          if (!MPF_DCHECK(p.status, x < (uint32_t)kTableRows)) x = kPadCode;
          if constexpr (TM) {
            tm_wait_ld<HI>(thi);
            tm_ld_pow2<LOW>(tlo, tcol);
          }
          const uint8_t *rowp = tbl_lane + x * row_bytes;
          // Diagonal shift (Alg. 5): cell k-1 of the previous row feeds cell k.
          const uint32_t wl = v[H - 1];
          uint32_t up = 0u;
          if (LG > 1) {
            up = __shfl_up_sync(kFull, wl, 1, LG);
            if (kF16 && gl == 0) up = 0u;
          }
          // Cell k - 1 of the previous row: the lane before's last cell and
          // this lane's high-half cell of the last word.  The group's first
          // lane takes zero instead, as sign copies of a non-negative cell.
          const uint32_t mpv = prmt(up, wl, kF16 ? 0x5432u : shift_sel);
          uint32_t rmax = 0u;
          // Update word q from the previous row's word q - 1 and score word sc.
          auto cell = [&](const int q, const uint32_t sc) {
            const uint32_t prev = (q == 0) ? mpv : v[q - 1];
            if constexpr (kPair) {
              if ((rr & 1) == 0) {
                v[q] = add_imad(prev, sc, one);
              } else {
                const uint32_t u = __viaddmax_s16x2_relu(prev, sc, sc);
                if constexpr (!kFoldRows) {
                  uint32_t &acc = (q & 1) ? vacc2 : vacc;
                  acc = __vimax3_s16x2(acc, v[q], u);
                }
                v[q] = u;
              }
            } else if (kF16)
              v[q] = hfma2_relu_u32(prev, one2, sc);
            else if (kDirect)
              v[q] = __viaddmax_s16x2(__vimax_s16x2_relu(prev, b2), sc, 0u);
            else
              v[q] = __viaddmax_s16x2(prev, sc, 0u);
          };
          // Fold words q + 1 and q into the row / running maximum.
          auto fold = [&](const int q) {
            if constexpr (kPair) {
              uint32_t &acc = (rr & 1) == 0 ? vacc : vacc2;
              if constexpr (kFoldRows) acc = __vimax3_s16x2(acc, v[q + 1], v[q]);
            } else if (kDirect)
              rmax = __vimax3_u16x2(rmax, v[q + 1], v[q]);
            else
              vacc = __vimax3_u16x2(vacc, v[q + 1], v[q]);
          };
          // Words from shared memory, highest first (in-place update): the
          // two-word tail, then the 4-word chunks down to chunk j_lo.
          auto smem_words = [&](const int j_lo) {
            if (kTail) {   // words 4Q+1 and 4Q
              const uint2 t2 = *reinterpret_cast<const uint2 *>(tail_lane + x * tail_row_bytes);
              cell(4 * Q + 1, t2.y);
              cell(4 * Q, t2.x);
              fold(4 * Q);
            }
#pragma unroll
            for (int j = Q - 1; j >= j_lo; --j) {
              const uint4 s4 = *reinterpret_cast<const uint4 *>(rowp + j * LG * 16);
              cell(4 * j + 3, s4.w);
              cell(4 * j + 2, s4.z);
              cell(4 * j + 1, s4.y);
              cell(4 * j, s4.x);
              fold(4 * j + 2);
              fold(4 * j);
            }
          };
          if constexpr (TM) {
            if constexpr (HT < H) smem_words(HT / 4);
#pragma unroll
            for (int q = HI - 1; q >= 1; q -= 2) {
              cell(LO + q, thi[q]);
              cell(LO + q - 1, thi[q - 1]);
              fold(LO + q - 1);
            }
            tm_wait_ld<LOW>(tlo);
            tcol = tm_col(rr < 3 ? __byte_perm(cur, 0u, 0x4440u + rr + 1) : nxt & 0xffu);
            tm_ld_at<HI, LO>(thi, tcol);
#pragma unroll
            for (int q = LO - 1; q >= 1; q -= 2) {
              cell(q, tlo[q]);
              cell(q - 1, tlo[q - 1]);
              fold(q - 1);
            }
          } else {
            smem_words(0);
          }
          if (kDirect) {
            // xE of this row (Alg. 6), then the J and B special states.
            const int xE = group_max<LG>(half_max(rmax)) >> kCellShift;
            if (real && !done) {
              if (xE >= cap) {
                done = true;
              } else {
                xJ = max(xJ, xE - tec);
                b = min(sat8(max(base, xJ) - (t + tbm)), cap);
                b2 = pack2(b << kCellShift);
              }
            }
          } else if (kFast && CHECK) {
            const bool trig = real && !done && ((vacc + Tk2) & 0x80008000u) != 0u;
            if (__any_sync(kFull, trig)) {
              const int mm = key_value<kF16>(group_max<LG>(half_max(vacc)));
              if (real && !done && mm > T) {
                const int xE = b + mm;
                if (xE >= cap) {
                  done = true;
                } else {
                  xJ = max(xJ, xE - tec);
                  const int bn = min(sat8(max(base, xJ) - (t + tbm)), cap);
                  if (bn > b) {
#pragma unroll
                    for (int q = 0; q < H; ++q)
                      v[q] = kF16 ? hfma2_relu_u32(v[q], one2, pack2_half(b - bn))
                                  : __viaddmax_s16x2(v[q], pack2((b - bn) * (1 << kCellShift)), 0u);
                  }
                  b = bn;
                  exact = true;
                  // Lazy again: a later row changes xJ or overflows only with
                  // a cell above the new threshold (0 or more: b stays below
                  // cap).  From here on every row is tested.
                  T = min(xJ + tec - b, cap - b - 1);
                  arm();
                  vacc = 0u;
                }
              }
            }
          }
         }
        }
      };

      // A rescored sequence that was split takes its segments one by one and
      // leaves out those whose largest cell cannot move xJ (see kUnits).
      int seg = 0, left = 0;   // next segment, and words left of the current one
      bool follows = false;
      const int n_segs = kFast && active && r < p.n_long ? (int)(__ldg(p.unit_first + r + 1) - __ldg(p.unit_first + r)) : 1;
      for (;;) {
      if constexpr (kFast) {
        if (done) left = 0;
        if (left == 0) busy = false;
        if (left == 0 && active && !done) {
          while (n_segs > 1 && seg < n_segs && __ldcg(qd->unit_max + __ldg(p.unit_first + r) + seg) <= T) {
            ++seg;
            follows = false;
          }
          if (seg < n_segs) {
            busy = true;
            if (n_segs > 1) {
              const int end = (seg + 1) * (int)p.seg_rows;
              first_row = max(end - (int)(p.seg_rows + (follows ? 0u : p.seg_overlap)), 0);
              rows = min(end, len) - first_row;
            }
            if (!follows) {
#pragma unroll
              for (int q = 0; q < H; ++q) v[q] = 0u;
            }
            left = (rows + 3) >> 2;
            ++seg;
            follows = true;
          }
        }
        if (!__any_sync(kFull, busy)) break;
      }
      nsteps = kFast ? left : busy ? (rows + 3) >> 2 : 0;
      wptr = busy ? wstart + ((uint32_t)first_row >> 2) : p.pad_word;
      int wsteps = (int)__reduce_max_sync(kFull, (uint32_t)nsteps);
      // Past its segment's end a group would run padding rows, which clear the
      // cells that its next segment follows on: the warp stops where the first
      // such group ends, and the others go on with theirs in the next turn.
      if constexpr (kFast && G > 1)
        wsteps = min(wsteps, (int)__reduce_min_sync(kFull, busy && seg < n_segs ? (uint32_t)nsteps : (uint32_t)INT_MAX));
      cur = __ldg(p.residues + (nsteps > 0 ? wptr : p.pad_word));
      if constexpr (kUniform) cur = __reduce_max_sync(kFull, cur);
      ahead = __ldg(p.residues + (1 < nsteps ? wptr + 1u : p.pad_word));
      if constexpr (TM) {   // first row
        cur = map_pad(cur);
        tcol = tm_col(cur & 0xffu);
        tm_ld_at<HI, LO>(thi, tcol);
      }

      int since_clear = 0;
      if constexpr (kUniform) {
        // Two words per turn, loaded a turn ahead (unguarded: at most four
        // words past the rows' last, three past its chunk; they lie in the
        // database, whose last chunk is spare, and are not scored).
        const uint32_t *wp = p.residues + wptr;
        uint32_t a1 = ahead, a2 = __ldg(wp + 2);
        for (int step = 0; step < wsteps; step += 2) {
          const uint32_t n1 = map_pad(__reduce_max_sync(kFull, a1)), n2 = map_pad(__reduce_max_sync(kFull, a2));
          a1 = __ldg(wp + step + 3);
          a2 = __ldg(wp + step + 4);
          four_rows(step, std::false_type{}, n1);
          cur = n1;
          if (step + 1 < wsteps) {
            four_rows(step + 1, std::false_type{}, n2);
            cur = n2;
          }
          if constexpr (kPair) {
            since_clear += 2;
            if (since_clear == kClearSteps) {
              since_clear = 0;
#pragma unroll
              for (int q = 0; q < H; ++q) v[q] &= kCellMask2;
            }
          }
        }
      } else
      for (int step = 0; step < wsteps; ++step) {
        // Prefetch the residue words; past the end a group reads padding.
        const uint32_t nxt = ahead;
        ahead = __ldg(p.residues + (step + 2 < nsteps ? wptr + (uint32_t)step + 2u : p.pad_word));
        if (kFast) {
          const bool near = busy && !done && (exact || Tnear < 0 || ((vacc + Tnear2) & 0x80008000u) != 0u);
          if (__any_sync(kFull, near))
            four_rows(step, std::true_type{}, nxt);
          else
            four_rows(step, std::false_type{}, nxt);
        } else {
          four_rows(step, std::false_type{}, nxt);
        }
        cur = nxt;
        if constexpr (kPair) {
          // Drop the sums' carries (at most one per pair of rows) while they
          // are below one score unit.
          if (++since_clear == kClearSteps) {
            since_clear = 0;
#pragma unroll
            for (int q = 0; q < H; ++q) v[q] &= kCellMask2;
          }
        }
      }

      if constexpr (TM) tm_wait_ld<HI>(thi);   // the load issued after the last row
      if constexpr (!kFast) break;
      left = max(left - wsteps, 0);
      first_row += 4 * wsteps;
      rows -= 4 * wsteps;
      }

      // ---- finalise the G sequences -------------------------------------
      bool own = active && qvalid;   // this group writes its sequence's outputs
      if constexpr (kPair) vacc = __vmaxs2(vacc, vacc2);
      int V = key_value<kF16>(gmax(half_max(vacc)));
      if (kUnits && __any_sync(kFull, split)) {
        // Of a split sequence's units the last one to finish goes on, with
        // the largest cell of all of them.
        uint32_t first = 0, n = 0, last = 1;
        if (split && own) {
          first = __ldg(p.unit_first + r);
          n = __ldg(p.unit_first + r + 1) - first;
          if (gl == 0) {
            __stcg(qd->unit_max + kr, V);
            __threadfence();
            last = atomicAdd(qd->unit_done + r, 1u) == n - 1u ? 1u : 0u;
            __threadfence();
          }
        }
        last = __shfl_sync(kFull, last, lane - gl);
        own = own && last;
        if (split && own)
          for (uint32_t u = gl; u < n; u += (uint32_t)width) V = max(V, __ldcg(qd->unit_max + first + u));
        V = gmax(V);
      }
      if (kFast || kHeld) {
        // A sequence whose cells never rose above the begin score: its best
        // row maximum is the best single-cell score of its residues.
        const bool rescue = own && !done && !exact && V == 0 && len > 0;
        int g = INT_MIN / 2;
        if (rescue) {
          for (int w = gl; w < (len + 3) >> 2; w += width) {
            const uint32_t word = __ldg(p.residues + wstart + (uint32_t)w);
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (4 * w + i < len && MPF_DCHECK(p.status, ((word >> (8 * i)) & 0xffu) < (uint32_t)kTableRows))
                g = max(g, (int)smax[(word >> (8 * i)) & 0xffu]);
          }
        }
        g = gmax(g);
        if (kBoth && own && gl == 0) {
          // SSV (Alg. 7) from the same largest cell: with b held the MSV
          // cells minus b are exactly the SSV cells.
          const bool ovf = V >= 255;
          const int raw = ovf ? 255 : V;
          qd->raw2[orig] = (uint8_t)raw;
          qd->flag2[orig] = ovf ? 1 : 0;
          if (qd->nat2) qd->nat2[orig] = ovf ? __int_as_float(0x7f800000) : nat_score(raw - tbm - tec - 2 * t, scale);
        }
        if (kHeld && own && gl == 0) {
          // The begin score b was held for every row.  V, the largest cell
          // of any row, decides: at or above 255 - bias - b some row
          // overflowed (with b held or after it rose, cells only grow);
          // at most T no row could move xJ past base, so the held rows are
          // exact; in between xB would have moved: an exact kernel rescores
          // the sequence.
          if (V >= cap - b) {
            out_raw[orig] = 255;
            out_flag[orig] = 1;
            if (out_nat) out_nat[orig] = __int_as_float(0x7f800000);
          } else if (V > T) {
            const uint32_t slot = atomicAdd(qd->fallback_count, 1u);
            if (MPF_DCHECK(p.status, slot < p.n_seqs)) qd->fallback_ranks[slot] = (uint32_t)r;
          } else {
            const int G2 = V > 0 ? V : g;
            const int raw = len > 0 ? max(0, b + G2 - tec) : 0;
            out_raw[orig] = (uint8_t)raw;
            out_flag[orig] = 0;
            if (out_nat) out_nat[orig] = nat_score(raw - t - base, scale);
          }
        }
        if (kFast && own && gl == 0) {
          int raw;
          uint8_t flag = 0;
          if (done) {
            raw = 255;
            flag = 1;
          } else if (exact) {
            raw = xJ;
          } else {
            const int G2 = V > 0 ? V : g;
            raw = len > 0 ? max(0, b + G2 - tec) : 0;
          }
          out_raw[orig] = (uint8_t)raw;
          out_flag[orig] = flag;
          if (out_nat) out_nat[orig] = flag ? __int_as_float(0x7f800000) : nat_score(raw - t - base, scale);
        }
      } else if (kDirect) {
        if (own && gl == 0) {
          const int raw = done ? 255 : xJ;
          out_raw[orig] = (uint8_t)raw;
          out_flag[orig] = done ? 1 : 0;
          if (out_nat) out_nat[orig] = done ? __int_as_float(0x7f800000) : nat_score(raw - t - base, scale);
        }
      } else {  // SSV
        if (own && gl == 0) {
          const bool ovf = V >= 255;
          const int raw = ovf ? 255 : V;
          out_raw[orig] = (uint8_t)raw;
          out_flag[orig] = ovf ? 1 : 0;
          if (out_nat) out_nat[orig] = ovf ? __int_as_float(0x7f800000) : nat_score(raw - tbm - tec - 2 * t, scale);
        }
      }
    }
    if constexpr (TM) tm_fence_before();   // this item's TMEM reads before the next item's writes
    __syncthreads();
  }
  if constexpr (TM) {
    if (warp == 0) {
      tm_fence_after();
      tm_dealloc(s_tmem);
    }
  }
}

}  // namespace mpf
