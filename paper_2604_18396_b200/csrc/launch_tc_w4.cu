// Launches of the dequantising tensor-core kernel for exit-layer rows (5 <= rows <= 256) and its operand kernel.
#include <algorithm>

#include "launch_tc.h"
#include "gemm_tc_w4.cuh"

namespace river {

cudaError_t launch_tc_prep_pair(river_ctx *c, const ProjIn &in, int K, int n, const int32_t *rows_a, const int32_t *cnt_a,
                                const int32_t *rows_r, const int32_t *cnt_r) {
    const int np = (n + 15) / 16 * 16;
    const river_ctx::BMap *ba = tc_bmap(c, K, np, false);
    if (!ba) return cudaErrorInvalidValue;
    __nv_bfloat16 *alo = ba->lo_ptr;  // (the next call may move the map table)
    const river_ctx::BMap *br = tc_bmap(c, K, np, true);
    if (!br) return cudaErrorInvalidValue;
    PrepPair p{rows_a, cnt_a, rows_r, cnt_r, c->tc_xhi, alo, reinterpret_cast<__half *>(c->tc_x4),
               reinterpret_cast<__half *>(br->lo_ptr), (K + kPrepChunk - 1) / kPrepChunk};
    const int yr = (K + 2 * kPrepChunk - 1) / (2 * kPrepChunk);
    return launch_k(tc_prep_pair_kernel, dim3(np, p.ya + yr), dim3(256), 0, c->stream, true, in, p, K);
}

template <class Epi>
cudaError_t launch_tc_w4(river_ctx *c, const ProjIn &in, const CUtensorMap *const (&m)[3], const river_w4 *const (&w)[3],
                         int K, int tiles, int n, int gateup, int q_tiles, int k_tiles, const int32_t *rows,
                         const int32_t *cnt, const int32_t *hint, const Epi &epi, int phase, bool overlap, bool alt_operand) {
    const int np = (n + 15) / 16 * 16, nt = row_tile(c, np);
    const river_ctx::BMap *bm = tc_bmap(c, K, np, true, alt_operand, nt);
    if (alt_operand) phase &= ~kTcPrep;  // the operand rows are there already (the previous projection's epilogues)
    if (!bm) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    if (phase & kTcPrep) {
        e = launch_k(tc_prep_w4_kernel, dim3(np, (K + 2 * kPrepChunk - 1) / (2 * kPrepChunk)), dim3(256), 0, c->stream, true, in,
                     rows, cnt, K, reinterpret_cast<__half *>(c->tc_x4), reinterpret_cast<__half *>(bm->lo_ptr));
        if (e != cudaSuccess) return e;
    }
    if (!(phase & kTcGemm)) return e;
    TcW4Args a{};
    a.K = K; a.n_pad = nt; a.one_box = bm->one ? 1 : 0;
    const size_t stage = 2 * (size_t)nt * kTcBK * 2, raw = (size_t)kW4RawBufs * kW4RawBytes;
    const int most = c->short_sums ? tc_wide_segment(c->num_sms, c->cfg.max_batch, tiles, K, true) : 0;
    const W4Plan plan = w4_row_plan(w4_plan(c->num_sms, np, tiles, K, c->rows_distinct, most), np, nt);
    if (!plan.splits) return cudaErrorInvalidValue;
    a.n_stages = plan.n_stages; a.splits = plan.splits; a.wide = plan.wide; a.sets = plan.sets;
    if (sizeof(float) * (size_t)nt * kTcLd > (size_t)a.n_stages * stage + raw) return cudaErrorInvalidValue;
    const size_t smem = w4_smem_request(plan, np, nt);
    if (!smem) return cudaErrorInvalidValue;
    a.overlap = overlap ? 1 : 0;
    a.gateup = gateup; a.qkv_q_tiles = q_tiles; a.qkv_k_tiles = k_tiles;
    for (int i = 0; i < 3; ++i) { a.scale[i] = (const uint16_t *)w[i]->scale; a.zero[i] = (const uint16_t *)w[i]->zero; }
    a.rows = rows; a.cnt = cnt; a.hint = hint; a.dev_err = c->dev_err;
    e = ensure_smem(c, tc_gemm_w4_kernel<Epi>, smem);
    if (e != cudaSuccess) return e;
    return launch_kc(tc_gemm_w4_kernel<Epi>, dim3(tiles * a.splits, (np + nt - 1) / nt), dim3(kW4Threads), smem, c->stream, true, a.splits,
                     *m[0], *m[1], *m[2], bm->hi, bm->lo, a, epi);
}
#define RIVER_TCW4_INST(E) \
    template cudaError_t launch_tc_w4<E>(river_ctx *, const ProjIn &, const CUtensorMap *const (&)[3], const river_w4 *const (&)[3], \
                                         int, int, int, int, int, int, const int32_t *, const int32_t *, const int32_t *, const E &, \
                                         int, bool, bool);
RIVER_TCW4_INST(TcQkvEpi) RIVER_TCW4_INST(TcResidEpi) RIVER_TCW4_INST(TcGateUpEpi)
#undef RIVER_TCW4_INST

}  // namespace river
