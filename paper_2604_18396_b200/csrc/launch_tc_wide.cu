// Launches of the pair kernel that carries the projections of long prefill passes, and of the kernels that make its operands.
#include <algorithm>

#include "launch_tc.h"
#include "gemm_tc_wide.cuh"
#include "tensor_maps.h"

namespace river {

namespace {

// ---------------------------------------------------------------- exit-layer weights in f16, for the same kernel
// With hundreds of rows a 4-bit matrix is worth expanding once per pass: row r of the (up to three) matrices laid one after
// the other becomes K f16 values (q - z) * s - one rounding, as in tc_gemm_w4_kernel - with the inputs of every group of
// eight in the order (0,4,1,5,2,6,3,7) that the f16 operand rows have too.  A thread expands 32 codes.  Bound by HBM:
// 0.56 bytes read and 2 written per weight.
struct W4Expand { W4 m[3]; int rows[3]; };
__global__ void __launch_bounds__(256) w4_expand_kernel(const W4Expand e, int K, __half *out) {
    pdl_launch();
    pdl_wait();  // the GEMM before may still read the previous projection's expansion
    const int per_row = K >> 5;
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    int r = (int)(i / per_row), m = 0;
    const int c = (int)(i % per_row);  // 32-input run of the row
    if (r >= e.rows[0] + e.rows[1] + e.rows[2]) return;
    uint4 *dst = reinterpret_cast<uint4 *>(out + (size_t)r * K + 32 * c);
    while (r >= e.rows[m]) { r -= e.rows[m]; ++m; }
    const W4 w = e.m[m];
    const size_t g = (size_t)r * (K >> 6) + (c >> 1);
    const __half2 s2 = __float2half2_rn(bf16f(w.scale[g])), z2 = __float2half2_rn(bf16f(w.zero[g]));
    const uint4 v = ldg_stream16(w.codes + (size_t)r * (K >> 1) + 16 * c);
    dst[0] = w4_word_to_f16(v.x, z2, s2);
    dst[1] = w4_word_to_f16(v.y, z2, s2);
    dst[2] = w4_word_to_f16(v.z, z2, s2);
    dst[3] = w4_word_to_f16(v.w, z2, s2);
}

// Rows per tile: the tiles go to `pairs` CTA pairs in whole rounds, so a size that leaves the last round nearly full can win
// over a larger one that does not; a round takes about as long as its rows and 128 more (with the operand kernel, by itself: 8B-class gate/up, 1024 rows, 7 rounds of 256 rows 297 us, 10 of 192 338, 13 of 128 388; QKV: 2 of 256 112, 2 of
// 192 102, 3 of 128 122).
int wide_bn(int feature_pairs, int n, int pairs) {
    int best = 256;
    double best_t = 1e30;
    for (int bn = 256; bn >= 64; bn -= 32) {
        const int total = feature_pairs * ((n + bn - 1) / bn), rounds = (total + pairs - 1) / pairs;
        const double t = rounds * (bn + 128.0);
        if (t < best_t * 0.995) { best_t = t; best = bn; }
    }
    return best;
}

const river_ctx::WMap *wide_map(river_ctx *c, int K, int bn, bool alt) {
    for (auto &b : c->wide_maps)
        if (b.K == K && b.bn == bn && b.alt == alt) return &b;
    river_ctx::WMap b{K, bn, alt, {}, {}};
    uint16_t *hi = wide_operand(c, alt), *lo = hi + (size_t)c->wide_rows * K;
    if (!make_map_bf16(&b.hi, hi, K, c->wide_rows, bn / 2) || !make_map_bf16(&b.lo, lo, K, c->wide_rows, bn / 2)) return nullptr;
    c->wide_maps.push_back(b);
    return &c->wide_maps.back();
}

}  // namespace

cudaError_t launch_wide_operand(river_ctx *c, const ProjIn &in, int K, int n_list, const int32_t *rows, const int32_t *cnt, bool f16) {
    uint16_t *hi = wide_operand(c, false), *lo = hi + (size_t)c->wide_rows * K;
    if (f16)
        return launch_k(tc_prep_w4_kernel, dim3(n_list, (K + 2 * kPrepChunk - 1) / (2 * kPrepChunk)), dim3(256), 0, c->stream, true,
                        in, rows, cnt, K, reinterpret_cast<__half *>(hi), reinterpret_cast<__half *>(lo));
    return launch_k(tc_prep_kernel, dim3(n_list, (K + kPrepChunk - 1) / kPrepChunk), dim3(256), 0, c->stream, true, in, rows, cnt, K,
                    reinterpret_cast<__nv_bfloat16 *>(hi), reinterpret_cast<__nv_bfloat16 *>(lo));
}

cudaError_t launch_w4_expand(river_ctx *c, const river_w4 *const (&w)[3], const int (&rows)[3], int K) {
    W4Expand e{};
    long long threads = 0;
    for (int i = 0; i < 3; ++i) {
        e.rows[i] = rows[i];
        if (rows[i]) e.m[i] = w4_of(*w[i]);
        threads += (long long)rows[i] * (K / 32);
    }
    return launch_k(w4_expand_kernel, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, c->stream, true, e, K, c->wide_w);
}

template <class Epi>
cudaError_t launch_tc_wide(river_ctx *c, const CUtensorMap &a0, const CUtensorMap &a1, const CUtensorMap &a2, int K, int tiles,
                           int n_list, int q_tiles, int k_tiles, int run_step, int head_step, const int32_t *rows, const int32_t *cnt,
                           const Epi &epi, bool f16, bool alt_operand) {
    TcWideArgs a{};
    const int feature_pairs = tiles / 2, pairs = c->num_sms / 2;
    if (tiles & 1) return cudaErrorInvalidValue;  // (every shape of the exit layers' tensor-core kernels has whole pairs of tiles)
    a.K = K; a.tiles = tiles; a.f16 = f16 ? 1 : 0; a.q_tiles = q_tiles; a.k_tiles = k_tiles;
    a.run_step = run_step; a.head_step = head_step;
    a.rows = rows; a.cnt = cnt; a.dev_err = c->dev_err;
    a.seg = tc_wide_segment(c->num_sms, c->cfg.max_batch, tiles, K, f16);
    a.bn = wide_bn(feature_pairs, n_list, pairs);
    const river_ctx::WMap *bm = wide_map(c, K, a.bn, alt_operand);
    if (!bm) return cudaErrorInvalidValue;
    a.n_stages = 8;
    while (a.n_stages > 2 && tc_wide_smem_bytes(a.bn, a.n_stages) > 227 * 1024 - 64) --a.n_stages;
    const size_t smem = tc_wide_smem_bytes(a.bn, a.n_stages);
    const cudaError_t e = ensure_smem(c, tc_gemm_wide_kernel<Epi>, smem);
    if (e != cudaSuccess) return e;
    const int total = feature_pairs * ((n_list + a.bn - 1) / a.bn);
    return launch_kc(tc_gemm_wide_kernel<Epi>, dim3(2 * std::min(pairs, total)), dim3(kWdThreads), smem, c->stream, true, 2, a0, a1,
                     a2, bm->hi, bm->lo, a, epi);
}
#define RIVER_TCWIDE_INST(E) \
    template cudaError_t launch_tc_wide<E>(river_ctx *, const CUtensorMap &, const CUtensorMap &, const CUtensorMap &, int, int, int, \
                                           int, int, int, int, const int32_t *, const int32_t *, const E &, bool, bool);
RIVER_TCWIDE_INST(WdQkvEpi) RIVER_TCWIDE_INST(WdResidEpi) RIVER_TCWIDE_INST(WdGateUpEpi)
#undef RIVER_TCWIDE_INST

}  // namespace river
