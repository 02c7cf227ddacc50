// mpf_inst.cu -- scan-kernel instantiations for one lane-group size.
//
// Compiled once per size (-DMPF_LG=1, 2, 4, 8, 16, 32; see build.py) into
// kernel_lg<MPF_LG>(): every mode of the striped scan kernel (eight) for each
// built word count -- multiples of four, and the counts with a two-word tail.
// With -DMPF_LG=32 -DMPF_TM=1 it builds kernel_lg32_tm() instead: the
// tensor-memory variants (SSV, held MSV and both in one sweep, at least
// kTmMinWords words).  With -DMPF_QP=1 (lanes 1 to 16) it builds kernel_qp_tm_lg<lanes>():
// the tensor-memory variants that score one sequence against 32 / lanes
// queries per warp (integer SSV, the held MSV pass and the two together).
// Either with -DMPF_FEW=1 builds the variants for databases of few residue
// codes (kernel_lg32_tmfew(), kernel_qp_tmfew_lg<lanes>(): those three modes,
// from 16 words on; shorter lanes fit tensor memory whole with every code).
// -DMPF_LG=32 -DMPF_MIX=1 builds kernel_mix(): the same modes for mixed sets.
#include "mpf_scan_kernel.cuh"

#ifndef MPF_LG
#error "compile with -DMPF_LG=<lanes per sequence>"
#endif
#define MPF_CAT2(a, b) a##b
#define MPF_CAT(a, b) MPF_CAT2(a, b)

// C(words) for each word count of a range.
#define MPF_WORDS_4_6(C) C(4) C(6)
#define MPF_WORDS_8_14(C) C(8) C(10) C(12) C(14)
#define MPF_WORDS_16_48(C)                                                                \
  C(16) C(18) C(20) C(22) C(24) C(26) C(28) C(30) C(32) C(34) C(36) C(38) C(40) C(42)     \
  C(44) C(46) C(48)

namespace mpf {

#if defined(MPF_MIX)

#define MPF_CASE(W)                                                                              \
  case W:                                                                                        \
    if (mode == MODE_SSV) return scan_kernel<32, W, MODE_SSV, TM_FEW, 1, true>;                  \
    if (mode == MODE_MSV_HELD) return scan_kernel<32, W, MODE_MSV_HELD, TM_FEW, 1, true>;        \
    if (mode == MODE_MSV_SSV) return scan_kernel<32, W, MODE_MSV_SSV, TM_FEW, 1, true>;          \
    return nullptr;

KernelFn kernel_mix(int words, int mode) {
  switch (words) {
    MPF_CASE(14) MPF_CASE(16) MPF_CASE(18) MPF_CASE(20) MPF_CASE(22) MPF_CASE(24)
    default:
      return nullptr;
  }
}

#elif defined(MPF_QP) || (defined(MPF_TM) && defined(MPF_FEW))

#ifdef MPF_QP
constexpr int kQueries = 32 / MPF_LG;
#else
constexpr int kQueries = 1;
#endif
#ifdef MPF_FEW
constexpr int kTable = TM_FEW;
#else
constexpr int kTable = TM_ALL;
#endif

#define MPF_CASE(W)                                                                           \
  case W:                                                                                     \
    if (mode == MODE_SSV) return scan_kernel<MPF_LG, W, MODE_SSV, kTable, kQueries>;          \
    if (mode == MODE_MSV_HELD) return scan_kernel<MPF_LG, W, MODE_MSV_HELD, kTable, kQueries>; \
    if (mode == MODE_MSV_SSV) return scan_kernel<MPF_LG, W, MODE_MSV_SSV, kTable, kQueries>;  \
    return nullptr;

#if defined(MPF_QP) && defined(MPF_FEW)
KernelFn MPF_CAT(kernel_qp_tmfew_lg, MPF_LG)(int words, int mode) {
#elif defined(MPF_QP)
KernelFn MPF_CAT(kernel_qp_tm_lg, MPF_LG)(int words, int mode) {
#else
KernelFn kernel_lg32_tmfew(int words, int mode) {
#endif
  switch (words) {
#ifndef MPF_FEW
    MPF_WORDS_8_14(MPF_CASE)
#endif
    MPF_WORDS_16_48(MPF_CASE)
    default:
      return nullptr;
  }
}

#elif defined(MPF_TM) && MPF_LG == 32

#define MPF_CASE(W)                                                                      \
  case W:                                                                                \
    if (mode == MODE_SSV) return scan_kernel<32, W, MODE_SSV, TM_ALL>;                   \
    if (mode == MODE_SSV_F16) return scan_kernel<32, W, MODE_SSV_F16, TM_ALL>;           \
    if (mode == MODE_MSV_HELD) return scan_kernel<32, W, MODE_MSV_HELD, TM_ALL>;         \
    if (mode == MODE_MSV_HELD_F16) return scan_kernel<32, W, MODE_MSV_HELD_F16, TM_ALL>; \
    if (mode == MODE_MSV_SSV) return scan_kernel<32, W, MODE_MSV_SSV, TM_ALL>;           \
    return nullptr;

KernelFn kernel_lg32_tm(int words, int mode) {
  switch (words) {
    MPF_WORDS_8_14(MPF_CASE)
    MPF_WORDS_16_48(MPF_CASE)
    default:
      return nullptr;
  }
}

#else

#define MPF_CASE(W)                                                                  \
  case W:                                                                            \
    if (mode == MODE_SSV) return scan_kernel<MPF_LG, W, MODE_SSV>;                   \
    if (mode == MODE_MSV_FAST) return scan_kernel<MPF_LG, W, MODE_MSV_FAST>;         \
    if (mode == MODE_MSV_DIRECT) return scan_kernel<MPF_LG, W, MODE_MSV_DIRECT>;     \
    if (mode == MODE_SSV_F16) return scan_kernel<MPF_LG, W, MODE_SSV_F16>;           \
    if (mode == MODE_MSV_FAST_F16) return scan_kernel<MPF_LG, W, MODE_MSV_FAST_F16>; \
    if (mode == MODE_MSV_HELD) return scan_kernel<MPF_LG, W, MODE_MSV_HELD>;         \
    if (mode == MODE_MSV_HELD_F16) return scan_kernel<MPF_LG, W, MODE_MSV_HELD_F16>; \
    if (mode == MODE_MSV_SSV) return scan_kernel<MPF_LG, W, MODE_MSV_SSV>;           \
    return nullptr;

KernelFn MPF_CAT(kernel_lg, MPF_LG)(int words, int mode) {
  switch (words) {
    MPF_WORDS_4_6(MPF_CASE)
    MPF_WORDS_8_14(MPF_CASE)
    MPF_WORDS_16_48(MPF_CASE)
    default:
      return nullptr;
  }
}

#endif

}  // namespace mpf
