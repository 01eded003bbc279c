// Launches of the tensor-core projection kernel for backbone rows (5 <= rows <= 256) and its operand kernel.
#include <algorithm>

#include "launch_tc.h"
#include "tensor_maps.h"

namespace river {

const river_ctx::BMap *tc_bmap(river_ctx *c, int K, int np, bool w4, bool alt, int box) {
    if (!box) box = np;
    for (auto &b : c->tc_bmaps)
        if (b.K == K && b.np == np && b.w4 == w4 && b.alt == alt && b.box == box) return &b;
    const bool behind = 2 * np <= 256;  // the lo rows follow the hi rows in use
    river_ctx::BMap b{K, np, box, w4, alt, behind && box == np, nullptr, nullptr, {}, {}};
    __nv_bfloat16 *base = alt ? (w4 ? c->tc_x4alt : c->tc_xalt) : (w4 ? c->tc_x4 : c->tc_xhi);
    b.base = base;
    b.lo_ptr = behind ? base + (size_t)np * K : base + (size_t)c->tc_max_pad * c->tc_kmax;
    const int hi_rows = b.one ? 2 * np : np;  // a box holds at most 256 rows; rows past the last are filled with zeros
    if (!make_map_bf16(&b.hi, base, K, hi_rows, b.one ? hi_rows : box) || !make_map_bf16(&b.lo, b.lo_ptr, K, np, box)) return nullptr;
    c->tc_bmaps.push_back(b);
    return &c->tc_bmaps.back();
}

int row_tile(const river_ctx *c, int np) {
    const river_config &g = c->cfg;
    return tc_row_tile(c->num_sms, np, std::max((g.Hq + 2 * g.Hkv) * g.dh / kTcBM, g.F / 64), g.d, c->rows_distinct);
}

template <class Epi>
cudaError_t launch_tc(river_ctx *c, const ProjIn &in, const CUtensorMap &a0, const CUtensorMap &a1, const CUtensorMap &a2,
                      int K, int tiles, int n, int gateup, int q_tiles, int k_tiles, const int32_t *rows,
                      const int32_t *cnt, const Epi &epi, bool allow_split, const int32_t *hint, int phase,
                      bool late_release, bool alt_operand) {
    // (the LM head's row tiles would each stream its weights: only where these leave SMs idle)
    const int np = (n + 15) / 16 * 16, nt = allow_split || tiles < c->num_sms ? row_tile(c, np) : np;
    const river_ctx::BMap *bm = tc_bmap(c, K, np, false, alt_operand, nt);
    if (alt_operand) phase &= ~kTcPrep;  // the operand rows are there already (the previous projection's epilogues)
    if (!bm) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    if (phase & kTcPrep) {
        e = launch_k(tc_prep_kernel, dim3(np, (K + kPrepChunk - 1) / kPrepChunk), dim3(256), 0, c->stream, true, in, rows, cnt, K,
                     c->tc_xhi, bm->lo_ptr);
        if (e != cudaSuccess) return e;
    }
    if (!(phase & kTcGemm)) return e;
    TcArgs a{};
    a.K = K; a.n_pad = nt; a.one_box = bm->one ? 1 : 0; a.late_release = late_release ? 1 : 0;
    const size_t stage = tc_stage_bytes(nt);
    const int most = c->short_sums ? tc_wide_segment(c->num_sms, c->cfg.max_batch, tiles, K, false) : 0;
    const TcPlan plan = tc_plan(c->num_sms, np, tiles, K, allow_split, c->rows_distinct, most);
    if (!plan.splits) return cudaErrorInvalidValue;
    const int occ = nt < np ? 2 : plan.occ, row_tiles = (np + nt - 1) / nt;  // (a row tile sums what all rows together would)
    a.splits = plan.splits; a.halves = plan.halves;
    a.n_stages = tc_stages_at(nt, occ);
    tc_cols(nt, occ, &a.wide);
    // the finished tile lives in the pipeline memory
    if (sizeof(float) * (size_t)nt * kTcLd > (size_t)a.n_stages * stage) return cudaErrorInvalidValue;
    a.gateup = gateup; a.qkv_q_tiles = q_tiles; a.qkv_k_tiles = k_tiles;
    a.rows = rows; a.cnt = cnt; a.dev_err = c->dev_err;
    a.hint = hint ? hint : cnt;
    const bool head_of_tiled = nt == np && row_tile(c, np) < np;  // (beside CTAs of a row tile: tc_footprints)
    const size_t smem = std::max<size_t>(tc_smem_bytes(nt, a.n_stages), a.halves || head_of_tiled ? kTcTwoSmem : 0);
    e = ensure_smem(c, tc_gemm_kernel<Epi>, smem);
    if (e != cudaSuccess) return e;
    return launch_kc(tc_gemm_kernel<Epi>, dim3(tiles * a.splits, row_tiles), dim3(kTcThreads), smem, c->stream, true, a.splits, a0,
                     a1, a2, bm->hi, bm->lo, a, epi);
}
cudaError_t launch_tc_pass(river_ctx *c, const CUtensorMap &a0, int K, int tiles, int n_list, int splits, const int32_t *rows,
                           const int32_t *cnt, const TcResidEpi &epi, bool f16, bool alt_operand) {
    const river_ctx::WMap *bm = wide_map(c, K, 2 * kTcPassRows, alt_operand);
    if (!bm) return cudaErrorInvalidValue;
    TcArgs a{};
    a.K = K; a.n_pad = kTcPassRows; a.splits = splits; a.halves = 1; a.wide = 1; a.f16 = f16 ? 1 : 0;
    a.n_stages = tc_stages_at(kTcPassRows, 2);
    a.rows = rows; a.cnt = cnt; a.dev_err = c->dev_err;
    a.hint = c->meta_dev;  // StepMeta::n_rows (the host launches nothing for an empty list)
    const size_t smem = std::max<size_t>(tc_smem_bytes(kTcPassRows, a.n_stages), kTcTwoSmem);
    const cudaError_t e = ensure_smem(c, tc_gemm_kernel<TcResidEpi>, smem);
    if (e != cudaSuccess) return e;
    return launch_kc(tc_gemm_kernel<TcResidEpi>, dim3(tiles * splits, (n_list + kTcPassRows - 1) / kTcPassRows), dim3(kTcThreads), smem, c->stream,
                     true, splits, a0, a0, a0, bm->hi, bm->lo, a, epi);
}
#define RIVER_TC_INST(E) \
    template cudaError_t launch_tc<E>(river_ctx *, const ProjIn &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, \
                                      int, int, int, int, int, int, const int32_t *, const int32_t *, const E &, bool, const int32_t *, \
                                      int, bool, bool);
RIVER_TC_INST(TcQkvEpi) RIVER_TC_INST(TcResidEpi) RIVER_TC_INST(TcGateUpEpi) RIVER_TC_INST(TcHeadEpi)
#undef RIVER_TC_INST

}  // namespace river
