// mpf_internal.h -- structures shared by the host API and the scan kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mpf {

// Debug builds (compiled with -DMPF_DEBUG_CHECKS, libmpf_debug.so): kernels
// test their indexes against the buffers they were given; a failed test
// records kStatusBadIndex in the status word and the access is skipped, so
// nothing traps.  Release builds compile the tests away.
constexpr int kStatusBadIndex = 2;
#ifdef __CUDACC__
__device__ __forceinline__ void report_bad_index(int *status) {
  if (status) atomicCAS(status, 0, kStatusBadIndex);
}
// a + b as one 32-bit multiply-add (a * one + b, one = 1 in a register the
// compiler does not see through): it issues on the FMA pipe, beside the
// integer ALU pipe of the DPX instructions.
__device__ __forceinline__ uint32_t add_imad(uint32_t a, uint32_t b, uint32_t one) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(one), "r"(b));
  return r;
}

// Dynamic shared memory of the running block, in bytes.
__device__ __forceinline__ uint32_t dynamic_smem_bytes() {
  uint32_t r;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
  return r;
}
#endif
#ifdef MPF_DEBUG_CHECKS
#define MPF_DCHECK(status, cond) ((cond) || (mpf::report_bad_index(status), false))
#else
#define MPF_DCHECK(status, cond) true
#endif

// Residue code of padding rows.  Database sequences are padded with it to a
// 16-byte boundary; its table row scores kNegInf at every node, so a padding
// row leaves every score unchanged (the paper's '#' residue, Sec. 3.2).
constexpr int kPadCode = 32;
constexpr int kTableRows = 33;           // codes 0..31 plus padding
constexpr int kNegInf = -16384;          // table entry of padding rows and nodes > M
// Integer cells and table entries of the striped kernels hold scores in units
// of 2^kCellShift (every score and cell that counts is below 510 in
// magnitude, so 16 bits hold it).  The low bits take the carries that 32-bit
// sums of packed cells leave in the upper half: at most one per pair of
// rows, cleared every kClearSteps steps of four rows, before they reach a
// unit.
constexpr int kCellShift = 6;
constexpr int kClearSteps = 30;
constexpr uint32_t kCellMask2 = 0xffc0ffc0u;
static_assert(2 * kClearSteps < (1 << kCellShift), "carries stay below one score unit");
constexpr int kBlockThreads = 512;
constexpr int kMaxWords = 48;
constexpr int kStripedMaxM = 2 * 32 * kMaxWords;   // longest model of the striped kernels
constexpr int kMaxLongM = 100000;                  // longest model of the long-model kernel
constexpr int kLongThreads = 256;

enum Mode : int {
  MODE_SSV = 0,           // Alg. 7, 16-bit integer cells (DPX)
  MODE_MSV_FAST = 1,      // Alg. 2, begin score held constant between J changes
  MODE_MSV_DIRECT = 2,    // Alg. 2, J/B update after every row
  MODE_SSV_F16 = 3,       // MODE_SSV with cells as fp16 integers (FMA pipe)
  MODE_MSV_FAST_F16 = 4,  // MODE_MSV_FAST with cells as fp16 integers
  MODE_LONG_MSV = 5,      // models beyond kStripedMaxM, MSV: long_kernel
  MODE_TILE_SSV = 7,      // models beyond kStripedMaxM, SSV: tile_kernel<SSV>
  MODE_TILE_MSV = 8,      // models beyond kStripedMaxM, MSV when b may be held: tile_kernel<MSV>
                          //   (with MODE_LONG_MSV over the sequences it leaves)
  MODE_MSV_HELD = 9,      // Alg. 2 with the begin score held for the whole sequence: no per-row
                          //   tests; sequences whose running maximum passes T are listed and
                          //   rescored by MODE_MSV_FAST
  MODE_MSV_HELD_F16 = 10, // MODE_MSV_HELD with cells as fp16 integers
  MODE_MSV_SSV = 11,      // MODE_MSV_HELD and MODE_SSV from one sweep: with b held the MSV
                          //   cells minus b follow the SSV recurrence, so the largest cell
                          //   gives both filters' scores
  MODE_TILE_MSV_SSV = 12, // MODE_TILE_MSV and MODE_TILE_SSV from one sweep (the same reason)
};

// Striped kernels that read their table from tensor memory (one sequence per
// warp): the first words of each lane's row of every residue code come from
// TMEM, the rest from shared memory.  A database whose codes are all below
// kTmFewCodes needs few rows (its codes and the padding code), so 24 words of
// each fit the 512 columns (21 x 24 = 504); otherwise all 33 rows are held,
// with 12 words, or all of up to 14 (33 x 14 = 462).
constexpr uint32_t kTmemColumns = 512;   // 32-bit columns of an SM's tensor memory
constexpr int kTmMinWords = 8;      // fewer words per lane: the shared-memory kernels
constexpr int kTmFewCodes = 20;
enum TmTable : int { TM_NONE = 0, TM_ALL = 1, TM_FEW = 2 };   // table in shared memory; TMEM, all codes; TMEM, few codes
// Words per lane read from TMEM for a lane of `words` words.
__host__ __device__ constexpr int tm_words(int words, int tm) {
  return tm == TM_NONE ? 0 : tm == TM_FEW ? (words <= 24 ? words : 24) : (words <= 14 ? words : 12);
}

// Score-table formats: signed 16-bit integers, or the same integers as fp16.
// TABLE_I16_PACKED: integer scores in the packed geometry (one copy of each
// region; the tables of the queries that share a warp's sequence).
enum TableFormat : int { TABLE_I16 = 0, TABLE_F16 = 1, TABLE_I16_PACKED = 16, TABLE_I16_MIX = 17 };
inline int table_format(int mode) {
  return (mode == MODE_SSV_F16 || mode == MODE_MSV_FAST_F16 || mode == MODE_MSV_HELD_F16) ? TABLE_F16
                                                                                           : TABLE_I16;
}

// One profile in one kernel layout (lives in device memory).
struct QueryDesc {
  const uint4 *table;     // shared-memory image: copies x 33 rows x quads x lanes
  uint32_t table_bytes;   // bytes to stage, multiple of 16 (includes smax)
  uint32_t row_bytes;     // stride between residue rows
  uint32_t copy_bytes;    // stride between bank-offset copies
  uint32_t smax_off;      // byte offset of 33 int16 per-code maximum scores
  uint32_t tail_off;      // byte offset of the two-word tail region (words % 4 == 2)
  uint32_t tail_row_bytes;
  int bias, tbm, tec, base, tjb_fixed;
  float scale;
  const uint8_t *tjb;     // per-length tjb (nullable)
  uint32_t n_tjb;
  uint32_t M;             // model length (long-model kernel)
  uint32_t seg_words;     // long-model kernel: cost words (4 nodes) per lane segment
  uint8_t *raw;           // outputs indexed by original sequence number
  uint8_t *flag;
  float *nat;             // nullable
  uint8_t *raw2;          // MODE_MSV_SSV: the SSV outputs (raw, flag above: MSV)
  uint8_t *flag2;
  float *nat2;            // nullable
  // Nullable: score only these length ranks (ascending), *n_ranks of them
  // (a device count written by an earlier kernel on the same stream).
  const uint32_t *ranks;
  const uint32_t *n_ranks;
  uint32_t more_than, at_most;   // of rank lists: score only more than, and (not 0) at most so many ranks
  // Tiled MSV kernel and MSV_HELD: sequences left to an exact kernel (their
  // length ranks, and the count, zero before the launch).
  uint32_t *fallback_ranks;
  uint32_t *fallback_count;
  // Split sequences (striped kernels): each unit's largest cell, and per rank
  // the units that have finished (zero before the launch).
  int *unit_max;
  uint32_t *unit_done;
};

struct ScanParams {
  const uint32_t *residues;   // residue words (4 codes each)
  uint32_t n_words;           // words in residues (debug index checks)
  const uint32_t *seq_word;   // per length rank: first word of the sequence
  const uint32_t *seq_len;    // per length rank: length
  const uint32_t *seq_orig;   // per length rank: original sequence number
  uint32_t n_seqs;
  uint32_t pad_word;          // a word of four padding codes
  const QueryDesc *queries;
  uint32_t n_queries;
  uint32_t n_shards;          // work item i = (query i / n_shards, shard i % n_shards)
  uint32_t *item_counter;     // zero before the launch
  int *status;                // nonzero: error reported by a kernel
  uint32_t long_words;        // long-model kernel: largest seg_words of its queries
  uint8_t *tile_col;          // tiled kernel: per resident warp two columns of
  uint32_t tile_col_stride;   //   tile_col_stride bytes (an int16 per row)
  uint64_t tile_col_bytes;
  // Work units of the striped kernels without rank lists: first the segments
  // of ranks 0 .. n_long - 1 (unit u belongs to rank unit_rank[u], whose
  // units start at unit_first[rank]; seg_rows rows each, read from
  // seg_overlap rows before), then the other ranks whole.
  uint32_t n_units, n_long, n_long_units, seg_rows, seg_overlap;
  const uint32_t *unit_rank, *unit_first;
  uint32_t n_sets;            // mixed sets: their number, and 32 words per set (query | lane of its
  const uint32_t *mix_lanes;  //   group << 16 | lanes of the group << 24; 0 lanes: none)
  uint32_t tm_rows;           // TM_FEW kernels: TMEM rows, the database's codes and the padding code
  uint32_t one;               // 1 (striped kernels: see add_imad)
  uint32_t qp_table_stride;   // striped kernels with several queries per warp: bytes per staged table
};

typedef void (*KernelFn)(ScanParams);

// Long-model MSV kernel (mpf_long_kernel.cu, MODE_LONG_MSV), DP row as
// 16-bit pairs or (bytes) as bytes.
KernelFn long_kernel_for(int mode, bool bytes, int seg_words);
size_t long_smem_per_warp(int seg_words, bool bytes);

// Tiled kernel for long models (mpf_tile_kernel.cu, MODE_TILE_SSV and
// MODE_TILE_MSV): tiles of kTileNodes nodes, kTileC per lane, blocks of
// kTileWarps warps; per resident warp two columns of tile_col_stride bytes.
// Table: per tile [code 0..31][chunk 0..kTileC/8-1][lane] x 4 int16 pairs,
// pair p of lane l = nodes (l*kTileC + p, l*kTileC + p + kTileC/2), scores
// s = bias - cost (codes >= K: bias - 255; nodes past M: -32768); after the
// tiles (QueryDesc::smax_off) 32 int16 per-code maxima of s over the model.
constexpr int kTileC = 32;
constexpr int kTileNodes = 32 * kTileC;
constexpr int kTileWarps = 8;
constexpr int kTileWarpsTm = 16;
constexpr size_t kTileTableBytes = (size_t)32 * kTileNodes * 2;   // per tile
// Words (pairs) per lane of a tile: kTileC / 2, or kWideTileWords for the
// tensor-memory variant with wide tiles, whose 512 columns hold the rows of
// codes below kWideTileCodes.
constexpr int kWideTileWords = 20;
constexpr int kWideTileCodes = (int)(kTmemColumns / kWideTileWords);
__host__ __device__ constexpr size_t tiles_of(int M, int words) { return ((size_t)M + 64 * words - 1) / (64 * words); }
constexpr size_t tile_bytes(int words) { return (size_t)32 * 32 * words * 4; }
// The tiled kernel for a mode (MODE_TILE_*); tm: the tensor-memory variant
// (blocks of kTileWarpsTm warps, one per SM, the tile's scores in TMEM); wide:
// its tiles of kWideTileWords words per lane.
KernelFn tile_kernel_fn(int mode, bool tm, bool wide);

// Stage-to-stage hand-off (mpf_pipeline.cu): SSV -> MSV (raw_bytes 1) and
// MSV -> Viterbi (raw_bytes 2).
constexpr int kSelectChunk = 4096;   // length ranks per selection block
int launch_select(const uint32_t *seq_orig, uint64_t n, int n_q, const uint8_t *in_flag,
                  const float *in_nat, float min_nat, void *out_raw, int raw_bytes,
                  uint8_t *out_flag, float *out_nat, uint32_t *chunk_count,
                  uint32_t *chunk_offset, uint32_t *ranks, uint32_t *n_ranks, cudaStream_t st);
int launch_pvalues(const float *nat, uint64_t n, float mu, float lambda, float *p, int num_sms,
                   cudaStream_t st);

// P7Viterbi filter (mpf_viterbi.cu).  Tables are int16 in device memory,
// striped (node l*Q + j in slot j*32 + l); -32768 is minus infinity.
constexpr int kVitFastMaxThreads = 512;
// Viterbi launch keys: kind * kVitKeyKind + the launch shape; queries with
// equal keys share a launch.
constexpr int kVitKeyKind = 1000000;
enum VitKind {
  kVitFastShared = 0,      // fast kernel, DP rows in shared memory
  kVitFastSharedNoD = 1,   // the same without the stored D row
  kVitGeneralShared = 2,   // general kernel, rows in shared memory
  kVitFastDevice = 3,      // fast kernel, rows in device memory (key + 1: without the stored D row)
  kVitGeneralDevice = 4,   // general kernel, rows in device memory
  kVitFastTeam = 5,        // fast kernel, a team of warps per sequence
  kVitFastDual = 6,        // both kinds 0/1 and 5, each taking the queries on its side of team_max
};
inline int vit_key_kind(int key) { return key / kVitKeyKind; }
inline bool vit_key_device_rows(int key) {
  return vit_key_kind(key) == kVitFastDevice || vit_key_kind(key) == kVitGeneralDevice;
}
constexpr int kVitRows = 32;         // msc rows: residue codes 0..31
constexpr int kVitTrans = 8;         // BM, MM, IM, DM, MI, II, MD, DD
constexpr int kVitSpecial = 8;       // NN, NB, EC, CC, CT, EJ, JJ, JB

// Tables of the packed Viterbi kernel: kVitPackPlanes transition planes (MD,
// DD, MM, IM, DM, MI, II) of `words` x 32 words, then kVitRows rows of match
// scores and as many for the second step.
constexpr int kVitPackPlanes = 7;
struct VitPackTables {
  const uint32_t *trans;
  int words;                  // 64 nodes each
};

// One query of a Viterbi launch (lives in device memory).
struct VitQuery {
  const int16_t *msc;         // kVitRows x Mpad match scores (codes >= K: -32768)
  const int16_t *trans;       // kVitTrans x Mpad
  int sp[kVitSpecial];
  int M, Mpad;                // nodes; row length, a multiple of 32
  int base;
  float scale;
  int16_t *score;             // outputs indexed by original sequence number
  uint8_t *flag;
  float *nat;                 // nullable
  const uint32_t *ranks;      // nullable: score only these length ranks (ascending),
  const uint32_t *n_ranks;    //   *n_ranks of them
  // Packed kernel (mpf_vit_packed.cu), if the query qualifies: tables for one
  // warp per sequence and for teams (words 0: none); teams score the query
  // when it selects at most pk_team_max sequences.
  VitPackTables pk_solo, pk_team;
  int64_t pk_team_max;
  int pk_bm, pk_emax, pk_off; // entry move; largest match score, at least 1; first offset
  uint32_t pk_split;          // residue codes whose match scores are added in two steps
  int pk_rebase;              // the offset may be lowered
  uint32_t *fb_ranks;         // sequences left to the 32-bit kernels, and their count
  uint32_t *fb_count;
  int64_t team_max;           // the team kernel scores the query when it selects at most
                              //   this many sequences, the one-warp kernels otherwise
};

struct VitParams {
  const uint32_t *residues;   // database words (4 codes each)
  uint32_t n_words;           // words in residues (debug index checks)
  int *status;                // debug index checks (nullable)
  const uint32_t *seq_word;   // per length rank
  const uint32_t *seq_len;
  const uint32_t *seq_orig;
  uint32_t n_seqs;
  uint32_t n_queries;
  int max_Mpad;               // largest Mpad of the queries (sets shared memory)
  const VitQuery *queries;
  uint32_t *counters;         // one per query, zero before the launch
  int team_warps;             // packed kernel: warps per sequence
  uint2 *state;               // models past the shared-memory rows: per-warp DP rows, else null
  uint64_t state_bytes;
};
// key: from viterbi_shape_key for the group's longest model (the kernel
// and launch shape; kinds with device rows need p.state).  Tables in the
// striped layout (msc [32][Q][32] int16, trans [Q][32] x 8 int16 with Q =
// Mpad / 32).  n_codes: distinct residue codes in the database (sizes the
// L1 share).  Returns 0, 1 on a CUDA error, 2 if the rows do not fit.
int launch_viterbi(const VitParams &p, int key, int n_codes, int max_smem, int num_sms, cudaStream_t st);
// Shared memory of a block of `warps` warps that store the D row.
size_t viterbi_fast_smem_bytes(int Mpad, int warps);
// Device scratch of a launch over models of up to Mpad nodes that keeps its
// rows in device memory.
size_t viterbi_state_bytes(bool fast, int Mpad, int num_sms);
// The VitQuery::team_max of a query with this key and length.
int64_t viterbi_team_max(int key, int Mpad, int n_codes, int max_smem, int num_sms);
// Launch key (kernel and launch shape) for one model length, or -1 if no
// shape fits.  fast: every transition and special score <= 0 (else the
// general kernel).  n_seqs: sequences each query of the launch scores, 0
// when the host does not know (a rank list counted on the device).
int viterbi_shape_key(bool fast, int Mpad, int n_codes, int max_smem, int num_sms, uint64_t n_seqs);

// Packed Viterbi kernel (mpf_vit_packed.cu): two nodes per register, one warp
// or a team of `warps` warps per sequence with qh words per lane each.
constexpr int kVitPackReach = 16384;   // largest decline of one move or match step
constexpr int kVitPackStep = 8192;     // offset change when the entry score nears the floor
constexpr int kVitPackShortQH = 8;     // segments up to this many nodes: passing costs in 16 bits
constexpr int kVitPackRegQH = 8;       // words per lane up to which the transitions stay in registers
constexpr int kVitPack512QH = 28;      // words per lane up to which blocks have 512 threads
constexpr int kVitPackMaxSolo = 48;    // words per lane of the longest model one warp takes
constexpr int kVitPackTeamQH = 5, kVitPackMaxTeamQH = 8;   // words per lane of teams: wanted, at most
struct VitPackShape {
  int warps = 0, qh = 0;
};
// The shape for a model of M nodes (warps 0: none).
VitPackShape vit_pack_solo(int M);
VitPackShape vit_pack_team(int M);
// Scores the queries of p (all of shape s); returns as launch_viterbi.
int launch_viterbi_packed(const VitParams &p, VitPackShape s, int max_smem, int num_sms, cudaStream_t st);

// Kernel instantiation for (lanes, words, mode), or nullptr if not built.
KernelFn kernel_for(int lanes, int words, int mode);
// The tensor-memory variants (lanes = 32) for databases of any codes and of
// few (TM_FEW: the integer SSV, held MSV and one-sweep modes, from the word
// counts on where it differs), or nullptr if not built.
KernelFn kernel_lg32_tm(int words, int mode);
KernelFn kernel_lg32_tmfew(int words, int mode);
// Mixed sets (few codes, every word in tensor memory).
KernelFn kernel_mix(int words, int mode);
constexpr int kMixWordsMin = 14, kMixWordsMax = 24;
// Tensor-memory variants that score one sequence against 32 / lanes queries
// per warp (lanes 1 to 16), or nullptr if not built.
KernelFn kernel_qp_tm(int lanes, int words, int mode);
KernelFn kernel_qp_tmfew(int lanes, int words, int mode);
KernelFn kernel_qp_tmfew_lg1(int words, int mode);
KernelFn kernel_qp_tmfew_lg2(int words, int mode);
KernelFn kernel_qp_tmfew_lg4(int words, int mode);
KernelFn kernel_qp_tmfew_lg8(int words, int mode);
KernelFn kernel_qp_tmfew_lg16(int words, int mode);
KernelFn kernel_qp_tm_lg1(int words, int mode);
KernelFn kernel_qp_tm_lg2(int words, int mode);
KernelFn kernel_qp_tm_lg4(int words, int mode);
KernelFn kernel_qp_tm_lg8(int words, int mode);
KernelFn kernel_qp_tm_lg16(int words, int mode);
KernelFn kernel_lg1(int words, int mode);
KernelFn kernel_lg2(int words, int mode);
KernelFn kernel_lg4(int words, int mode);
KernelFn kernel_lg8(int words, int mode);
KernelFn kernel_lg16(int words, int mode);
KernelFn kernel_lg32(int words, int mode);

// Shared-memory table geometry of a (lanes, words) layout.  Words 4q..4q+3
// of a lane are one 16-byte chunk of the quad region; when words % 4 == 2 the
// last two words of every lane are 8-byte chunks of a separate tail region.
//
// Quad region: for each residue row, the quads of the group's lanes are
// adjacent 16-byte chunks, so 8 lanes of one group (one phase of a 128-bit
// shared load) hit 8 distinct 16-byte bank groups.  Groups of fewer than 8
// lanes share a phase with other groups (other residues): the region then
// holds 8 / lanes copies with 128-byte aligned rows and bases offset by
// lanes * 16 bytes, and group g reads copy g mod copies.
// Tail region: a 64-bit load runs in phases of 16 lanes; each residue row is
// 128 bytes (256 for 32-lane groups) holding 16 / lanes copies of the
// group's 8-byte chunks side by side, and group g reads copy g mod copies.
// Packed geometry (the tables of queries that share a warp's sequence, each
// staged at its own offset): one copy of each region, tail rows of lanes x 8
// bytes.
struct TableGeom {
  int lanes, words, copies, quads, tail_words, tail_copies;
  uint32_t row_bytes, copy_bytes, tail_off, tail_row_bytes, smax_off, table_bytes;
};

inline TableGeom table_geom(int lanes, int words, bool packed = false) {
  TableGeom g;
  g.lanes = lanes;
  g.words = words;
  g.quads = words / 4;
  g.tail_words = words % 4;
  g.copies = (packed || lanes >= 8) ? 1 : 8 / lanes;
  uint32_t row = (uint32_t)g.quads * (uint32_t)lanes * 16u;
  if (g.copies > 1) row = (row + 127u) & ~127u;
  g.row_bytes = row;
  g.copy_bytes = (uint32_t)kTableRows * row + (g.copies > 1 ? (uint32_t)lanes * 16u : 0u);
  g.tail_off = (uint32_t)g.copies * g.copy_bytes;
  g.tail_off = (g.tail_off + 127u) & ~127u;
  g.tail_copies = (packed || lanes >= 16) ? 1 : 16 / lanes;
  g.tail_row_bytes = g.tail_words ? (uint32_t)(g.tail_copies * lanes * 8) : 0u;
  g.smax_off = g.tail_off + (uint32_t)kTableRows * g.tail_row_bytes;
  g.table_bytes = (g.smax_off + 80u + 15u) & ~15u;   // 33 int16, whole 16-byte chunks
  return g;
}

// Shared-memory bytes between the staged tables of a packed warp set
// (32 / lanes queries).  Rows of a phase's groups sit at the same table
// offset, so the stride spreads them over the banks: it is a multiple of
// 128 bytes plus lanes * 16 (at most 64; 0 for 16 lanes), which puts the
// 8 / lanes groups of a 128-bit phase on distinct 16-byte bank groups and
// the two 8-lane groups of a 64-bit tail phase on distinct halves.
inline uint32_t packed_table_stride(int lanes, int words) {
  const uint32_t tb = table_geom(lanes, words, true).table_bytes;
  const uint32_t off = lanes >= 16 ? 0u : (uint32_t)(lanes * 16 < 64 ? lanes * 16 : 64);
  return ((tb + 127u) & ~127u) + off;
}

}  // namespace mpf
