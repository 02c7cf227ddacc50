// mpf_vit_packed.cu -- the P7Viterbi filter (Eq. 1 of Sec. 2.1) with two
// nodes per register, for profiles whose moves are all <= 0 and whose local
// entry is uniform (any log-probability profile in local mode).
//
// The 32-bit kernels of mpf_viterbi.cu spend about 60 issue slots per cell:
// one DPX instruction per term and node, the unpacking of eight 16-bit
// transitions, and three row arrays read and written in shared memory.  Here
// a 16x2 DPX instruction handles a term of two nodes and the DP row stays in
// registers, as do the profile's transitions up to 8 words per lane (512
// nodes; longer models: tensor memory), so a row reads its residue's match
// scores (one 32-bit word per two nodes, L1) and nothing of its own.  What
// bounds it: the ALU pipe, 77-85% busy at M = 400-2405 (a DPX instruction
// takes two cycles per warp and scheduler); launches with few sequences are
// bound by a row's chain of dependent steps.  Measured (GB300, one query, calls
// back to back, random sequences of mean 355, ms, the 32-bit kernels before /
// now): M = 400 on 20,000 sequences 4.47 / 1.70, M = 2405 27.4 / 6.89 (2,457
// GCUPS), M = 150 on 1,003 1.68 / 0.68.
//
// Layout.  A warp, or a team of W warps, scores one sequence.  In node order
// the team's warps, their lanes and the two halves of a lane's words form one chain of
// segments of QH nodes: word j of lane l of warp w holds nodes
// ((w*32 + l)*2 + h)*QH + j, h = 0 in the low half.  A row sweeps the words
// once: M (3 transitions, entry, match score), I, the true delete scores of
// the row before (its chain recomputed from the entering score, cheaper than
// a third row) and this row's segment-local delete chain, 10.5 DPX
// instructions per word.  Then the segments' maps d -> max(A, d + B) of the
// delete score entering them compose: the two halves of a lane, a warp scan
// over lanes, and across the team's warps through shared memory, with one
// named barrier per row.
//
// Exactness.  The filter's scores are 16-bit words (every sum saturates to
// [-32768, 32767]); a register half holds v' = v - off.
//   * DPX sums wrap, so every operand pair must stay in range.  No move and
//     no match score is below -kVitPackReach (match scores below it are added
//     in two steps, on the residue codes that have any), states are floored
//     at F' = -32768 + kVitPackReach, and so no sum falls below -32768.
//   * With moves <= 0 a state at or below the entry score xB + tBM of the
//     next row can never win a maximum there, so a state that is stored as
//     max(v, F) gives the same results while F <= xB + tBM.  As xB sinks with
//     long sequences, off is lowered (at least one row's decline early).
//     States floored before that stay without effect when every tMI and tII
//     is at or below the largest decline of xB per row (can_rebase, checked
//     per profile): they sink at least as fast as the entry score.  At off =
//     -kVitPackReach the floor is the true -32768 and nothing is conditional.
//   * M is at most 32766 - off + (largest match score) before the row's
//     overflow test (the first entry score is at most 32766, checked per
//     profile; a later one comes from a state of a row without overflow): off
//     starts at that score - 1, so M fits, and M >= 32767 is seen exactly.  After off was lowered a row near the top of the range
//     cannot be told from an overflow; such sequences, and rows whose best
//     score is at the floor while it would matter, are left to the 32-bit
//     kernels: their length ranks are appended to the query's list, which a
//     later launch on the stream scores.
//   * The scan over lanes may stop early: a delete score at most E (the row's
//     largest M) that has crossed segments whose moves sum to B is at most E
//     + B, and without effect once that is at or below the next entry score.
//   * Nodes past M have moves and match scores of -kVitPackReach (-32768 on
//     the codes added in two steps), and feed only one another: their M is at
//     most the entry score plus the row's smallest possible match score, so
//     at most E, or at least 2 * kVitPackReach below an earlier row's E, which
//     xC and xJ already hold.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "mpf_internal.h"
#include "mpf_tmem.cuh"

namespace mpf {

namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr int kNeg = -32768;
constexpr int kFloor = -32768 + kVitPackReach;   // F'
constexpr int kMinusInf = -(1 << 29);
constexpr int kThreads = 512, kWarps = kThreads / 32;
// Transition planes of the tables, the order in which registers hold them.
enum Plane { kMD, kDD, kMM, kIM, kDM, kMI, kII };
constexpr int kPlanes = kVitPackPlanes;

__device__ __forceinline__ int lo16(uint32_t w) { return (int)(int16_t)(w & 0xffffu); }
__device__ __forceinline__ int hi16(uint32_t w) { return ((int)w) >> 16; }
__device__ __forceinline__ uint32_t pack16(int lo, int hi) { return __byte_perm((uint32_t)lo, (uint32_t)hi, 0x5410); }
__device__ __forceinline__ uint32_t addmax2(uint32_t a, uint32_t b, uint32_t c) { return __viaddmax_s16x2(a, b, c); }
__device__ __forceinline__ int addmax(int a, int b, int c) { return __viaddmax_s32(a, b, c); }

// A load that stays where it is written among the others and the TMEM loads
// (hoisted together, a row's match scores would take QH registers).
__device__ __forceinline__ uint32_t ld_ordered(const uint32_t *a) {
  uint32_t r;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(r) : "l"(a));
  return r;
}
constexpr int kWindow = 6;   // match-score words in flight per lane

// What a team's warps tell one another after a row (two buffers, by row
// parity), and per query what passing through a whole warp costs.
struct RowEnd {
  int A;        // delete score at the warp's last node, nothing entering
  uint32_t M;   // its last words (the high half is the last node)
  uint32_t I;
  int pad;
};
struct WarpPass {
  int tMD0, tDD0, rest;   // moves into its first node's D; sum of tDD over the other nodes
};

// Long lanes (one warp per sequence) keep the transitions in tensor memory,
// eight columns per word: every lane of a warp reads the same column, so a
// word's seven planes are one tcgen05.ld.  In shared memory they took seven of
// the eight L1 wavefronts per word (M = 2405: 82% of the pipe, 1,990 GCUPS).
__host__ __device__ constexpr bool in_tmem(int qh, bool team) { return !team && qh > kVitPackRegQH; }
// Threads per block at most (registers: 2 QH words of the row), and blocks
// per SM that the registers must leave room for.  Without TMEM blocks are
// small (a team, or four one-warp sequences), so that an SM whose sequences
// of one launch have run out takes blocks of another, and a launch with few
// sequences spreads them over the SMs (ms, 512-thread blocks / now: M = 100
// on 10,000 sequences 1.06 / 0.91, M = 2405 on 2,000 1.83 / 1.65).
__host__ __device__ constexpr int block_threads(int qh, bool team) {
  return team ? kThreads : !in_tmem(qh, team) ? 128 : qh <= kVitPack512QH ? kThreads : 384;
}
__host__ __device__ constexpr int block_min(int qh, bool team) {
  return team || in_tmem(qh, team) ? 1 : qh <= 1 ? 8 : qh <= 2 ? 6 : qh <= 3 ? 5 : 4;
}

template <int QH, bool TEAM>
__global__ void __launch_bounds__(block_threads(QH, TEAM), block_min(QH, TEAM))
    viterbi_packed_kernel(VitParams p) {
  constexpr bool TM = in_tmem(QH, TEAM);
  __shared__ uint32_t s_tmem;
  __shared__ RowEnd s_row[2][kWarps];
  __shared__ int s_max[4][kWarps];     // per team: largest M of a row (rows modulo 4)
  __shared__ WarpPass s_pass[kWarps];
  __shared__ uint32_t s_next[kWarps];
  __shared__ int s_wn[3][block_threads(QH, TEAM)];   // window sums of the later scan steps
  __shared__ int s_top[kWarps];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int W = TEAM ? p.team_warps : 1;
  const int team = TEAM ? warp / W : warp, w = TEAM ? warp - team * W : 0;
  const int base_w = team * W;   // first warp of the team in the block
  auto team_barrier = [&]() {
    if constexpr (TEAM) asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(W * 32) : "memory");
  };
  if (!MPF_DCHECK(p.status, (blockDim.x >> 5) <= kWarps && (blockDim.x >> 5) % W == 0)) return;
  const uint32_t F2 = pack16(kFloor, kFloor);
  uint32_t tm_lane = 0;   // TMEM address of this warp's lane quarter, column 0
  if constexpr (TM) {
    if (warp == 0) tm_alloc(&s_tmem);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    tm_lane = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
  }

  for (uint32_t qi = 0; qi < p.n_queries; ++qi) {
    const VitQuery &Q = p.queries[qi];
    const uint64_t n_sel = Q.ranks ? (uint64_t)*Q.n_ranks : (uint64_t)p.n_seqs;
    // A query with both layouts is scored by teams up to pk_team_max sequences.
    if (TEAM ? (int64_t)n_sel > Q.pk_team_max : (int64_t)n_sel <= Q.pk_team_max) continue;
    const VitPackTables &tb = TEAM ? Q.pk_team : Q.pk_solo;
    if (!MPF_DCHECK(p.status, n_sel <= p.n_seqs && tb.words == W * QH)) continue;

    // Lanes of few words add every match score in two steps, which costs no
    // more than the test and the branch on the residue's code.
    constexpr bool kAlways = !TEAM && QH <= 2;

    // ---- this lane's transitions and the query's constants ----
    const uint32_t *tp = tb.trans + ((size_t)w * QH) * 32 + lane;
    const size_t plane = (size_t)W * QH * 32;
    uint32_t tr[TM ? 1 : QH][8];
    if constexpr (TM) {
      tm_fence_before();   // every warp is done with the previous query's planes
      __syncthreads();
      tm_fence_after();
      if (warp < 4) {
        for (int j = 0; j < QH; ++j) {
          uint32_t t[kPlanes];
#pragma unroll
          for (int n = 0; n < kPlanes; ++n) t[n] = __ldg(tp + n * plane + j * 32);
          tm_st4(tm_lane + 8 * j, t[0], t[1], t[2], t[3]);
          tm_st4(tm_lane + 8 * j + 4, t[4], t[5], t[6], 0u);
        }
        tm_wait_st();
      }
      tm_fence_before();
      __syncthreads();
      tm_fence_after();
    } else {
#pragma unroll
      for (int j = 0; j < QH; ++j)
#pragma unroll
        for (int n = 0; n < kPlanes; ++n) tr[j][n] = __ldg(tp + n * plane + j * 32);
    }
    int Blo = 0, Bhi = 0;
    uint32_t first[kPlanes];
#pragma unroll
    for (int n = 0; n < kPlanes; ++n) first[n] = __ldg(tp + n * plane);
#pragma unroll
    for (int j = 0; j < QH; ++j) {
      const uint32_t t = __ldg(tp + kDD * plane + j * 32);
      Blo += lo16(t);
      Bhi += hi16(t);
    }
    // M of the node before a segment reaches its end through D at this cost.
    // Short segments: in 16 bits, at least -kVitPackReach (checked per
    // profile) where the end has a node after it, and of no effect elsewhere.
    constexpr bool kShort = QH <= kVitPackShortQH;
    const int clo = lo16(first[kMD]) + Blo - lo16(first[kDD]), chi = hi16(first[kMD]) + Bhi - hi16(first[kDD]);
    const uint32_t cMD = pack16(max(clo, -kVitPackReach), max(chi, -kVitPackReach));
    int P = Blo + Bhi;   // inclusive prefix over lanes
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(kAll, P, off);
      if (lane >= off) P += y;
    }
    // Sum of B over lanes (lane - 2^r, lane], and the largest over the warp.
    // (of the first step that is not always taken).
    int Wn0, Wn1, Wmaxf = 0;
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      const int y = __shfl_up_sync(kAll, P, 1 << r);
      const int Wn = lane >= (1 << r) ? P - y : kMinusInf;
      const int m = __reduce_max_sync(kAll, Wn);
      if (r == 0) Wn0 = Wn;
      if (r == 1) Wn1 = Wn;
      if (r == (QH <= 4 ? 2 : QH <= 8 ? 1 : 0)) Wmaxf = m;
      if (r >= 2) s_wn[r - 2][threadIdx.x] = Wn;   // read by this thread only
    }
    int pre = 0, tMD0 = 0, tDD0 = 0, pass = 0;
    if constexpr (TEAM) {
      tMD0 = __shfl_sync(kAll, lo16(first[kMD]), 0);
      tDD0 = __shfl_sync(kAll, lo16(first[kDD]), 0);
      // From the warp's first node to the node before this lane's segment.
      pre = __shfl_up_sync(kAll, P, 1) - tDD0;
      team_barrier();   // every warp is done with the previous query's constants
      if (lane == 31) s_pass[warp] = WarpPass{tMD0, tDD0, P - tDD0};
      if (lane < 4) s_max[lane][team] = kFloor;
      team_barrier();
      pass = kMinusInf;   // cheapest way through a warp that another warp follows
      for (int v = 1; v + 1 < W; ++v)
        pass = max(pass, max(s_pass[base_w + v].tMD0, s_pass[base_w + v].tDD0) + s_pass[base_w + v].rest);
    }
    const int tNN = Q.sp[0], tNB = Q.sp[1], tEC = Q.sp[2], tCC = Q.sp[3];
    const int tEJ = Q.sp[5], tJJ = Q.sp[6], tJB = Q.sp[7];
    const int bm = Q.pk_bm, high = 32768 - Q.pk_emax;   // rows from `high` on may not be followed by another
    const int sink = max(-tNN, -tJJ) + 1;   // xB falls by less than this per row
    const uint32_t split = Q.pk_split;
    const uint32_t erow = (uint32_t)(W * QH * 32);   // words of a residue row
    const uint32_t *emis = tb.trans + kPlanes * plane + ((size_t)w * QH) * 32 + lane;

    for (;;) {
      uint32_t q = 0;
      if constexpr (TEAM) {
        if (w == 0 && lane == 0) s_next[team] = atomicAdd(p.counters + qi, 1u);
        team_barrier();
        q = s_next[team];
        team_barrier();   // read by all before the next sequence's write
      } else {
        if (lane == 0) q = atomicAdd(p.counters + qi, 1u);
        q = __shfl_sync(kAll, q, 0);
      }
      if ((uint64_t)q >= n_sel) break;
      const uint32_t r = Q.ranks ? __ldg(Q.ranks + q) : q;
      if (!MPF_DCHECK(p.status, r < p.n_seqs)) continue;
      const uint32_t w0 = __ldg(p.seq_word + r);
      const int len = (int)__ldg(p.seq_len + r);
      if (!MPF_DCHECK(p.status, (uint64_t)w0 + (uint64_t)((len + 3) >> 2) + 2 <= p.n_words)) continue;

      // Short lanes load a row's match scores while the row before ends, long
      // ones a few words ahead.
      uint32_t M[QH], I[QH], e[TM ? 1 : QH], f[kAlways ? QH : 1];
#pragma unroll
      for (int j = 0; j < QH; ++j) M[j] = I[j] = F2;
      uint32_t pM = F2, pI = F2, pD = F2;   // previous row: M, I, true D of the node before each half
      int off = Q.pk_off;
      int xN = Q.base, xJ = kNeg, xC = kNeg;
      int lo = addmax(xN, tNB, kNeg) + bm - off;   // next row's entry score, in offset units
      uint32_t xbm = pack16(max(lo, kFloor), max(lo, kFloor));
      int result = 0;     // 1 overflow, 2 left to the 32-bit kernel
      // Residues: the current word, shifted as its rows are used, and the
      // next one (loads reach two words past the sequence, inside the
      // database's spare words).  Match scores are loaded a row ahead; the load after the
      // last row takes whatever code follows (at most the padding code 32,
      // whose row is the second half's first, or row 31 where both halves are
      // read) and is not used.
      const uint32_t *res = p.residues + w0;
      uint32_t word = __ldg(res), wnext = __ldg(res + 1);
      uint32_t x = word & 0xffu;
      auto load_scores = [&]() {
        const uint32_t *er = emis + (kAlways ? min(x, kVitRows - 1u) : x) * erow;
        if constexpr (!TM) {
#pragma unroll
          for (int j = 0; j < QH; ++j) {
            e[j] = __ldg(er + j * 32);
            if constexpr (kAlways) f[j] = __ldg(er + kVitRows * erow + j * 32);
          }
        }
      };
      load_scores();
      for (int i = 0; i < len; ++i) {
        // ---- sweep ----
        uint32_t d = F2, mx = F2;
        auto sweep = [&](auto split_tag) {
          [[maybe_unused]] const uint32_t *e1 = emis + x * erow, *e2 = emis + (kVitRows + x) * erow;
          uint32_t dM = pM, dI = pI, dD = pD, mprev = F2;
          uint32_t tm[2][8];   // a word's transitions from TMEM, loaded a word ahead
          [[maybe_unused]] uint32_t ew[kWindow];
          if constexpr (TM) {
            tm_ld_pow2<8>(tm[0], tm_lane);
#pragma unroll
            for (int j = 0; j < kWindow; ++j) ew[j] = ld_ordered(e1 + j * 32);
          }
#pragma unroll
          for (int j = 0; j < QH; ++j) {
            uint32_t *t = TM ? tm[j & 1] : tr[TM ? 0 : j];
            if constexpr (TM) {
              tm_wait_ld<8>(t);
              if (j + 1 < QH) tm_ld_pow2<8>(tm[(j + 1) & 1], tm_lane + 8 * (j + 1));
            }
            uint32_t ej;
            if constexpr (TM) {
              ej = ew[j % kWindow];
              if (j + kWindow < QH) ew[j % kWindow] = ld_ordered(e1 + (j + kWindow) * 32);
            } else {
              ej = e[TM ? 0 : j];
            }
            const uint32_t Do = addmax2(dD, t[kDD], addmax2(dM, t[kMD], F2));
            uint32_t best = addmax2(dM, t[kMM], xbm);
            best = addmax2(dI, t[kIM], best);
            best = addmax2(dD, t[kDM], best);
            uint32_t Mn = addmax2(best, ej, F2);
            if constexpr (kAlways)
              Mn = addmax2(Mn, f[j], F2);
            else if constexpr (decltype(split_tag)::value)
              Mn = addmax2(Mn, ld_ordered(e2 + j * 32), F2);
            const uint32_t In = addmax2(I[j], t[kII], addmax2(M[j], t[kMI], F2));
            if (j > 0) d = addmax2(d, t[kDD], addmax2(mprev, t[kMD], F2));
            if (j & 1)
              mx = __vimax3_s16x2(mx, mprev, Mn);
            else if (j == QH - 1)
              mx = __vmaxs2(mx, Mn);
            dM = M[j];
            dI = I[j];
            dD = Do;
            M[j] = Mn;
            I[j] = In;
            mprev = Mn;
          }
        };
        if constexpr (kAlways)
          sweep(std::true_type{});
        else if ((split >> x) & 1u)
          sweep(std::true_type{});
        else
          sweep(std::false_type{});

        // The next row's residue and match scores.
        const bool turn = (i & 3) == 3;
        word = turn ? wnext : word >> 8;
        if (turn) wnext = __ldg(res + ((i >> 2) + 2));
        x = word & 0xffu;
        if (!MPF_DCHECK(p.status, x <= (uint32_t)kVitRows)) x = 0;
        load_scores();

        // ---- row end: E, the delete scores entering the segments ----
        int xe = __reduce_max_sync(kAll, max(lo16(mx), hi16(mx)));
        const uint32_t wl = M[QH - 1], il = I[QH - 1];
        uint32_t um = __shfl_up_sync(kAll, wl, 1), ui = __shfl_up_sync(kAll, il, 1);
        if (lane == 0) um = ui = F2;
        pM = __byte_perm(um, wl, 0x5432);   // M of the node before each half
        int Alo, A;
        if constexpr (kShort) {
          const uint32_t A2 = addmax2(pM, cMD, d);
          Alo = lo16(A2);
          A = addmax(Alo, Bhi, hi16(A2));
        } else {
          Alo = addmax(lo16(pM), clo, lo16(d));
          A = addmax(Alo, Bhi, addmax(hi16(pM), chi, hi16(d)));
        }
        // The next row's entry score is at least thr (lo: this row's).
        const int thr = max(lo - sink, kFloor);
        // Scan steps: the first kFree always (at usual moves and scores a
        // delete score crosses 2 kFree QH nodes or more in many rows), the
        // others where they can matter, behind one branch.
        constexpr int kFree = QH <= 4 ? 2 : QH <= 8 ? 1 : 0;
        if constexpr (kFree > 0) A = addmax(__shfl_up_sync(kAll, A, 1), Wn0, A);
        if constexpr (kFree > 1) A = addmax(__shfl_up_sync(kAll, A, 2), Wn1, A);
        if (xe + Wmaxf > thr) {
          if constexpr (kFree < 1) A = addmax(__shfl_up_sync(kAll, A, 1), Wn0, A);
          if constexpr (kFree < 2) A = addmax(__shfl_up_sync(kAll, A, 2), Wn1, A);
          A = addmax(__shfl_up_sync(kAll, A, 4), s_wn[0][threadIdx.x], A);
          A = addmax(__shfl_up_sync(kAll, A, 8), s_wn[1][threadIdx.x], A);
          A = addmax(__shfl_up_sync(kAll, A, 16), s_wn[2][threadIdx.x], A);
        }
        int din = __shfl_up_sync(kAll, A, 1);
        if (lane == 0) din = kFloor;
        if constexpr (TEAM) {
          RowEnd *row = s_row[i & 1];
          int *best = &s_max[i & 3][team];
          if (lane == 31) row[warp] = RowEnd{A, wl, il, 0};
          if (lane == 0) atomicMax(best, xe);
          // The next row's slot: last read three rows ago.
          if (threadIdx.x == base_w * 32 + 1) s_max[(i + 1) & 3][team] = kFloor;
          team_barrier();
          xe = *reinterpret_cast<volatile int *>(best);
          if (w > 0) {
            const RowEnd before = row[warp - 1];
            int D = before.A;
            if (xe + pass > thr) {   // a delete score may matter past a whole warp
              D = row[base_w].A;
              for (int v = 1; v < w; ++v) {
                const WarpPass c = s_pass[base_w + v];
                const int x0 = addmax(D, c.tDD0, hi16(row[base_w + v - 1].M) + c.tMD0);
                D = addmax(x0, c.rest, row[base_w + v].A);
              }
            }
            const int Mb = hi16(before.M);
            const int x0 = addmax(D, tDD0, Mb + tMD0);   // delete score of the warp's first node
            din = addmax(x0, pre, din);
            if (lane == 0) {
              din = D;
              ui = before.I;
              pM = __byte_perm(before.M, wl, 0x5432);
              Alo = addmax(Mb, clo, Alo);
            }
          }
        }
        const int hin = addmax(din, Blo, Alo);
        pD = pack16(din, hin);   // both at or above the floor
        pI = __byte_perm(ui, il, 0x5432);

        // ---- special states ----
        const int xE = xe + off;
        xN = addmax(xN, tNN, kNeg);
        xC = addmax(xC, tCC, addmax(xE, tEC, kNeg));
        xJ = addmax(xJ, tJJ, addmax(xE, tEJ, kNeg));
        lo = addmax(xN, tNB, addmax(xJ, tJB, kNeg)) + bm - off;
        // Rare: E out of the range that leaves the row exact, or the entry
        // score close to the floor.
        if ((uint32_t)(xe - kFloor - 1) >= (uint32_t)(high - kFloor - 1) || lo < kFloor + sink) {
          if (xe >= high) {
            result = xE >= 32767 ? 1 : 2;
            break;
          }
          // E at the floor: harmless unless it counts in a special state.
          if (xe <= kFloor && off > -kVitPackReach && (xE + tEC >= xC || xE + tEJ >= xJ)) {
            result = 2;
            break;
          }
          // Lower the offset: every state above the floor moves up.
          const int D = min(kVitPackStep, off + kVitPackReach);
          if (lo >= kFloor + sink || D == 0) {
            // nothing to do
          } else if (!Q.pk_rebase) {
            if (lo < kFloor) {
              result = 2;
              break;
            }
          } else {
            uint32_t m2 = __vmaxs2(pD, __vmaxs2(pM, pI));
#pragma unroll
            for (int j = 0; j < QH; ++j) m2 = __vimax3_s16x2(m2, M[j], I[j]);
            int top = __reduce_max_sync(kAll, max(lo16(m2), hi16(m2)));
            if constexpr (TEAM) {   // the same verdict in every warp of the team
              team_barrier();
              if (lane == 0) s_top[warp] = top;
              team_barrier();
              for (int v = 0; v < W; ++v) top = max(top, s_top[base_w + v]);
            }
            if (top + D >= high) {
              result = 2;
              break;
            }
            auto up = [&](uint32_t v) {
              const int a = lo16(v), b = hi16(v);
              return pack16(a > kFloor ? a + D : a, b > kFloor ? b + D : b);
            };
#pragma unroll
            for (int j = 0; j < QH; ++j) {
              M[j] = up(M[j]);
              I[j] = up(I[j]);
            }
            pM = up(pM);
            pI = up(pI);
            pD = up(pD);
            off -= D;
            lo += D;
          }
        }
        const uint32_t l = (uint32_t)max(lo, kFloor);
        xbm = __byte_perm(l, l, 0x1010);
      }
      if (w == 0 && lane == 0) {
        const uint32_t orig = __ldg(p.seq_orig + r);
        if (!MPF_DCHECK(p.status, orig < p.n_seqs)) {
        } else if (result == 2) {
          const uint32_t slot = atomicAdd(Q.fb_count, 1u);
          if (MPF_DCHECK(p.status, slot < p.n_seqs)) Q.fb_ranks[slot] = r;
        } else if (result == 1) {
          Q.score[orig] = 32767;
          Q.flag[orig] = 1;
          if (Q.nat) Q.nat[orig] = __int_as_float(0x7f800000);
        } else {
          const int sc = addmax(xC, Q.sp[4], kNeg);
          Q.score[orig] = (int16_t)sc;
          Q.flag[orig] = 0;
          if (Q.nat) Q.nat[orig] = __fsub_rn(__fdiv_rn(__int2float_rn(sc - Q.base), Q.scale), 3.0f);
        }
      }
      if constexpr (TEAM) {
        // The row maxima of the next sequence start at the floor.
        team_barrier();
        if (w == 0 && lane < 4) s_max[lane][team] = kFloor;
      } else {
        __syncwarp();
      }
    }
  }
  if constexpr (TM) {
    tm_fence_before();
    __syncthreads();
    if (warp == 0) {
      tm_fence_after();
      tm_dealloc(s_tmem);
    }
  }
}

typedef void (*PackedFn)(VitParams);

PackedFn packed_for(VitPackShape s) {
#define MPF_TEAM(Q) \
  case Q: return viterbi_packed_kernel<Q, true>;
#define MPF_SOLO(Q) \
  case Q: return viterbi_packed_kernel<Q, false>;
  if (s.warps > 1) switch (s.qh) {
      MPF_TEAM(1) MPF_TEAM(2) MPF_TEAM(3) MPF_TEAM(4) MPF_TEAM(5) MPF_TEAM(6) MPF_TEAM(7) MPF_TEAM(8)
      default: return nullptr;
    }
  switch (s.qh) {
    MPF_SOLO(1) MPF_SOLO(2) MPF_SOLO(3) MPF_SOLO(4) MPF_SOLO(5) MPF_SOLO(6) MPF_SOLO(7) MPF_SOLO(8)
    MPF_SOLO(10) MPF_SOLO(12) MPF_SOLO(14) MPF_SOLO(16) MPF_SOLO(18) MPF_SOLO(20) MPF_SOLO(22) MPF_SOLO(24)
    MPF_SOLO(26) MPF_SOLO(28) MPF_SOLO(30) MPF_SOLO(32) MPF_SOLO(34) MPF_SOLO(36) MPF_SOLO(38) MPF_SOLO(40)
    MPF_SOLO(42) MPF_SOLO(44) MPF_SOLO(46) MPF_SOLO(48)
    default: return nullptr;
  }
#undef MPF_TEAM
#undef MPF_SOLO
}

}  // namespace

VitPackShape vit_pack_solo(int M) {
  VitPackShape s;
  const int words = (M + 63) / 64;   // 64 nodes per word of a warp
  if (words > kVitPackMaxSolo) return s;
  s.warps = 1;
  s.qh = words <= 8 ? words : (words + 1) / 2 * 2;
  return s;
}

VitPackShape vit_pack_team(int M) {
  VitPackShape s;
  const int words = (M + 63) / 64;
  if (words <= 8 || words > kWarps * kVitPackMaxTeamQH) return s;
  s.warps = std::min(kWarps, (words + kVitPackTeamQH - 1) / kVitPackTeamQH);
  s.qh = (words + s.warps - 1) / s.warps;
  return s;
}

int launch_viterbi_packed(const VitParams &p, VitPackShape s, int max_smem, int num_sms, cudaStream_t st) {
  if (p.n_queries == 0) return 0;
  const PackedFn fn = s.warps > 0 && s.warps <= kWarps ? packed_for(s) : nullptr;
  if (!fn) return 2;
  const int threads = s.warps > 1 ? 32 * s.warps : block_threads(s.qh, false);
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, (const void *)fn) != cudaSuccess) return 1;
  // A block with its transitions in tensor memory takes all of the SM's
  // columns: with its own shared memory it asks for more than half of what an
  // SM has, so that no second block that does so is placed on the SM.  The
  // match scores come through the L1, which is left the rest.
  const bool tm = in_tmem(s.qh, s.warps > 1);
  const size_t smem = tm ? (size_t)max_smem / 2 + 1024 - a.sharedSizeBytes : 0;
  int per_sm = 0;
  if (cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)fn, threads, smem) != cudaSuccess ||
      per_sm < 1 || (tm && per_sm != 1))
    return 1;
  const int carve = (int)((size_t)per_sm * (smem + a.sharedSizeBytes + 1024) * 100 / (228 * 1024)) + 1;
  if (cudaFuncSetAttribute((const void *)fn, cudaFuncAttributePreferredSharedMemoryCarveout, carve) != cudaSuccess)
    return 1;
  VitParams q = p;
  q.team_warps = s.warps;
  fn<<<num_sms * per_sm, threads, smem, st>>>(q);
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace mpf
