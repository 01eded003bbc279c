// Launches of the pair kernel that carries the projections of long prefill passes, and of the kernels that make its operands.
#include <algorithm>

#include "launch_tc.h"
#include "gemm_tc_wide.cuh"
#include "tensor_maps.h"

namespace river {

namespace {

// ---------------------------------------------------------------- exit-layer weights in f16, for the same kernel
// With hundreds of rows a 4-bit matrix is worth expanding once per pass: the (up to three) matrices laid one after the other
// become f16 values (q - z) * s - one rounding, as in tc_gemm_w4_kernel - with the inputs of every group of eight in the order
// (0,4,1,5,2,6,3,7) that the f16 operand rows have too.  A warp takes a run of 1024 codes, 16 bytes per lane; four lanes trade their
// words, so that they store 64 bytes side by side.  Bound by HBM: 0.56 bytes read and 2 written per weight.
// 1B-class gate / up 29 -> 15 us (a thread stored its own 32 codes' 64 bytes 16 at a time before, half a sector each).  What did not
// help: the operand rows' kernel as part of this launch (its CTAs in front: mini shape, 1100 positions 622 -> 658 us), and an
// expansion beside the GEMM before it, in two buffers and CTAs without shared memory: they are not put next to that kernel's
// on an SM, find room on the idle ones only and finish late elsewhere (1B-class, 829 positions 1164 -> 1254).
struct W4Expand { W4 m[3]; int runs[3]; };
constexpr int kExpandRuns = 2;  // of a warp, under way at a time
__global__ void __launch_bounds__(256) w4_expand_kernel(const W4Expand e, __half *out) {
    pdl_launch();
    const int lane = threadIdx.x & 31, r0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * kExpandRuns, runs = e.runs[0] + e.runs[1] + e.runs[2];
    uint4 v[kExpandRuns];
    uint32_t sz[kExpandRuns];  // scale | zero
#pragma unroll
    for (int u = 0; u < kExpandRuns; ++u) {  // (weights depend on nothing)
        int r = min(r0 + u, runs - 1), m = 0;
        while (r >= e.runs[m]) { r -= e.runs[m]; ++m; }
        const W4 w = m == 0 ? e.m[0] : m == 1 ? e.m[1] : e.m[2];
        v[u] = ldg_stream16(w.codes + (size_t)r * 512 + 16 * lane);
        const size_t g = (size_t)r * 16 + (lane >> 1);
        sz[u] = (uint32_t)ldg_u16(w.scale + g) | (uint32_t)ldg_u16(w.zero + g) << 16;
    }
    pdl_wait();  // the GEMM before may still read the previous projection's expansion
#pragma unroll
    for (int u = 0; u < kExpandRuns; ++u) {
        if (r0 + u >= runs) break;  // (uniform over the warp)
        uint4 *dst = reinterpret_cast<uint4 *>(out) + (size_t)(r0 + u) * 128 + 4 * (lane & ~3) + (lane & 3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {  // lane (group, i) stores word i of lane (group, j)
            const int from = (lane & ~3) | j;
            const uint32_t a = __shfl_sync(0xffffffffu, v[u].x, from), b = __shfl_sync(0xffffffffu, v[u].y, from),
                           c = __shfl_sync(0xffffffffu, v[u].z, from), d = __shfl_sync(0xffffffffu, v[u].w, from),
                           t = __shfl_sync(0xffffffffu, sz[u], from);
            const uint32_t word = lane & 2 ? (lane & 1 ? d : c) : (lane & 1 ? b : a);
            dst[4 * j] = w4_word_to_f16(word, __float2half2_rn(bf16hi(t)), __float2half2_rn(bf16lo(t)));
        }
    }
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

}  // namespace

const river_ctx::WMap *wide_map(river_ctx *c, int K, int bn, bool alt) {
    for (auto &b : c->wide_maps)
        if (b.K == K && b.bn == bn && b.alt == alt) return &b;
    river_ctx::WMap b{K, bn, alt, {}, {}};
    uint16_t *hi = wide_operand(c, alt), *lo = hi + (size_t)c->wide_rows * K;
    if (!make_map_bf16(&b.hi, hi, K, c->wide_rows, bn / 2) || !make_map_bf16(&b.lo, lo, K, c->wide_rows, bn / 2)) return nullptr;
    c->wide_maps.push_back(b);
    return &c->wide_maps.back();
}

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
    long long runs = 0;
    for (int i = 0; i < 3; ++i) {
        if (rows[i]) e.m[i] = w4_of(*w[i]);
        e.runs[i] = (int)((long long)rows[i] * K / 1024);  // (whole: rows and inputs are multiples of 64 and 256)
        runs += e.runs[i];
    }
    return launch_k(w4_expand_kernel, dim3((unsigned)((runs + 8 * kExpandRuns - 1) / (8 * kExpandRuns))), dim3(256), 0, c->stream, true, e, c->wide_w);
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
