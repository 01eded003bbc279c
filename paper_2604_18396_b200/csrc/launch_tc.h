// Launch functions of the tensor-core projection kernels (internal).
#pragma once
#include "river_ctx.h"
#include "gemm_tc.cuh"
#include "gemm_tc_wide.cuh"

namespace river {

// box: operand rows per copy (0: all np)
const river_ctx::BMap *tc_bmap(river_ctx *c, int K, int np, bool w4 = false, bool alt = false, int box = 0);
// operand rows per CTA of a projection's tensor-core kernels when the step has np
int row_tile(const river_ctx *c, int np);

// Both kernels of a projection (backbone rows, exit-layer rows) are in flight together: `phase` says which part of a
// launch function runs - the operand kernel, the GEMM, or both in a row.
enum : int { kTcPrep = 1, kTcGemm = 2, kTcBoth = 3 };

// launch_tc.cu: backbone rows, 5 <= rows <= 256
template <class Epi>
cudaError_t launch_tc(river_ctx *c, const ProjIn &in, const CUtensorMap &a0, const CUtensorMap &a1, const CUtensorMap &a2,
                      int K, int tiles, int n, int gateup, int q_tiles, int k_tiles, const int32_t *rows,
                      const int32_t *cnt, const Epi &epi, bool allow_split, const int32_t *hint, int phase = kTcBoth,
                      bool late_release = false, bool alt_operand = false);
#define RIVER_TC_DECL(E) \
    extern template cudaError_t launch_tc<E>(river_ctx *, const ProjIn &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, \
                                             int, int, int, int, int, int, const int32_t *, const int32_t *, const E &, bool, const int32_t *, \
                                             int, bool, bool);
RIVER_TC_DECL(TcQkvEpi) RIVER_TC_DECL(TcResidEpi) RIVER_TC_DECL(TcGateUpEpi) RIVER_TC_DECL(TcHeadEpi)
#undef RIVER_TC_DECL

// launch_tc_w4.cu: the operand kernels of both lists as one launch (then launch_tc / launch_tc_w4 with kTcGemm)
cudaError_t launch_tc_prep_pair(river_ctx *c, const ProjIn &in, int K, int n, const int32_t *rows_a, const int32_t *cnt_a,
                                const int32_t *rows_r, const int32_t *cnt_r);

// launch_tc_w4.cu: exit-layer rows through the dequantising kernel: m[0..2] are the code maps, w[0..2] the matching
// scale / zero arrays (one matrix, gate + up, or q + k + v)
template <class Epi>
cudaError_t launch_tc_w4(river_ctx *c, const ProjIn &in, const CUtensorMap *const (&m)[3], const river_w4 *const (&w)[3],
                         int K, int tiles, int n, int gateup, int q_tiles, int k_tiles, const int32_t *rows,
                         const int32_t *cnt, const int32_t *hint, const Epi &epi, int phase = kTcBoth, bool overlap = false,
                         bool alt_operand = false);
#define RIVER_TCW4_DECL(E) \
    extern template cudaError_t launch_tc_w4<E>(river_ctx *, const ProjIn &, const CUtensorMap *const (&)[3], const river_w4 *const (&)[3], \
                                                int, int, int, int, int, int, const int32_t *, const int32_t *, const int32_t *, const E &, \
                                                int, bool, bool);
RIVER_TCW4_DECL(TcQkvEpi) RIVER_TCW4_DECL(TcResidEpi) RIVER_TCW4_DECL(TcGateUpEpi)
#undef RIVER_TCW4_DECL

// launch_tc_wide.cu: the projections of a long prefill pass (up to wide_rows rows) on CTA pairs.  The row lists' lengths
// are known on the host there (n_list >= the device's count).  launch_wide_operand writes the operand rows (bf16 or f16
// high and low parts); launch_w4_expand the f16 form of up to three exit-layer matrices, one after the other, in wide_w.
inline uint16_t *wide_operand(const river_ctx *c, bool alt) { return alt ? c->wide_xalt : c->wide_x; }
cudaError_t launch_wide_operand(river_ctx *c, const ProjIn &in, int K, int n_list, const int32_t *rows, const int32_t *cnt, bool f16);
cudaError_t launch_w4_expand(river_ctx *c, const river_w4 *const (&w)[3], const int (&rows)[3], int K);
// map `hi` / `lo` of the wide operand rows in boxes of bn / 2 rows
const river_ctx::WMap *wide_map(river_ctx *c, int K, int bn, bool alt);
// launch_tc.cu: O and down of a long pass on tc_gemm_kernel (tc_pass_splits)
cudaError_t launch_tc_pass(river_ctx *c, const CUtensorMap &a0, int K, int tiles, int n_list, int splits, const int32_t *rows,
                           const int32_t *cnt, const TcResidEpi &epi, bool f16, bool alt_operand);
template <class Epi>
cudaError_t launch_tc_wide(river_ctx *c, const CUtensorMap &a0, const CUtensorMap &a1, const CUtensorMap &a2, int K, int tiles,
                           int n_list, int q_tiles, int k_tiles, int run_step, int head_step, const int32_t *rows, const int32_t *cnt,
                           const Epi &epi, bool f16, bool alt_operand);
#define RIVER_TCWIDE_DECL(E) \
    extern template cudaError_t launch_tc_wide<E>(river_ctx *, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, int, int, \
                                                  int, int, int, int, int, const int32_t *, const int32_t *, const E &, bool, bool);
RIVER_TCWIDE_DECL(WdQkvEpi) RIVER_TCWIDE_DECL(WdResidEpi) RIVER_TCWIDE_DECL(WdGateUpEpi)
#undef RIVER_TCWIDE_DECL

}  // namespace river
