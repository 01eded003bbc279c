// Launches of the tensor-core projection kernel for backbone rows (5 <= rows <= 256) and its operand kernel.
#include <algorithm>

#include "launch_tc.h"
#include "tensor_maps.h"

namespace river {

const river_ctx::BMap *tc_bmap(river_ctx *c, int K, int np, bool w4, bool alt) {
    for (auto &b : c->tc_bmaps)
        if (b.K == K && b.np == np && b.w4 == w4 && b.alt == alt) return &b;
    river_ctx::BMap b{K, np, w4, alt, 2 * np <= 256, nullptr, nullptr, {}, {}};
    __nv_bfloat16 *base = alt ? (w4 ? c->tc_x4alt : c->tc_xalt) : (w4 ? c->tc_x4 : c->tc_xhi);
    b.base = base;
    b.lo_ptr = b.one ? base + (size_t)np * K : base + (size_t)c->tc_max_pad * c->tc_kmax;
    const int hi_rows = b.one ? 2 * np : np;  // a box holds at most 256 rows
    if (!make_map_bf16(&b.hi, base, K, hi_rows, hi_rows) || !make_map_bf16(&b.lo, b.lo_ptr, K, np, np)) return nullptr;
    c->tc_bmaps.push_back(b);
    return &c->tc_bmaps.back();
}

int tc_footprints(int np, TcFootprint (&out)[2]) {
    int n = 0;
    for (int occ = tc_stages_at(np, 2) ? 2 : 1; occ <= 3; ++occ) {
        const int st = tc_stages_at(np, occ);
        if (!st) break;
        int wide;
        out[n].cols = tc_cols(np, occ, &wide);
        if (occ == 2 && np <= kTcHalvesRows) out[n].cols *= 2;  // (a.halves)
        out[n].smem = tc_smem_bytes(np, st);
        if (++n == 2 || occ == 1) break;
    }
    return n;
}

template <class Epi>
cudaError_t launch_tc(river_ctx *c, const ProjIn &in, const CUtensorMap &a0, const CUtensorMap &a1, const CUtensorMap &a2,
                      int K, int tiles, int n, int gateup, int q_tiles, int k_tiles, const int32_t *rows,
                      const int32_t *cnt, const Epi &epi, bool allow_split, const int32_t *hint, int phase,
                      bool late_release, bool alt_operand) {
    const int np = (n + 15) / 16 * 16;
    const river_ctx::BMap *bm = tc_bmap(c, K, np, false, alt_operand);
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
    a.K = K; a.n_pad = np; a.one_box = bm->one ? 1 : 0; a.late_release = late_release ? 1 : 0;
    const size_t stage = tc_stage_bytes(np);
    const int most = c->short_sums ? tc_wide_segment(c->num_sms, c->cfg.max_batch, tiles, K, false) : 0;
    const TcPlan plan = tc_plan(c->num_sms, np, tiles, K, allow_split, c->rows_distinct, most);
    if (!plan.splits) return cudaErrorInvalidValue;
    const int occ = plan.occ;
    a.splits = plan.splits; a.halves = plan.halves;
    a.n_stages = tc_stages_at(np, occ);
    tc_cols(np, occ, &a.wide);
    // the finished tile lives in the pipeline memory
    if (sizeof(float) * (size_t)np * kTcLd > (size_t)a.n_stages * stage) return cudaErrorInvalidValue;
    a.gateup = gateup; a.qkv_q_tiles = q_tiles; a.qkv_k_tiles = k_tiles;
    a.rows = rows; a.cnt = cnt; a.dev_err = c->dev_err;
    a.hint = hint ? hint : cnt;
    // (two CTAs with double accumulators and a third one of another launch never share an SM: 256 + 256 columns are all)
    const size_t smem = std::max<size_t>(tc_smem_bytes(np, a.n_stages), a.halves ? 90 * 1024 : 0);
    e = ensure_smem(c, tc_gemm_kernel<Epi>, smem);
    if (e != cudaSuccess) return e;
    return launch_kc(tc_gemm_kernel<Epi>, dim3(tiles * a.splits), dim3(kTcThreads), smem, c->stream, true, a.splits, a0,
                     a1, a2, bm->hi, bm->lo, a, epi);
}
#define RIVER_TC_INST(E) \
    template cudaError_t launch_tc<E>(river_ctx *, const ProjIn &, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, \
                                      int, int, int, int, int, int, const int32_t *, const int32_t *, const E &, bool, const int32_t *, \
                                      int, bool, bool);
RIVER_TC_INST(TcQkvEpi) RIVER_TC_INST(TcResidEpi) RIVER_TC_INST(TcGateUpEpi) RIVER_TC_INST(TcHeadEpi)
#undef RIVER_TC_INST

}  // namespace river
