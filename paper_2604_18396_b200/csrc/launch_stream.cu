// Launches of the CUDA-core streaming kernels: projections of steps of up to four rows per pass, the LM head, and the merge of
// argmax partials (the tensor-core LM head's, and those of more rows than this one merges itself).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "launch.h"
#include "stream_plan.h"

namespace river {

namespace {

// Launch geometry: stream_small_share's where it applies; else warps per CTA and CTAs per SM such that every warp gets the same
// number of tasks (a task is R weight rows) and at least 16 warps per SM have loads in flight.  Chosen once per (kernel, task count, K, whether
// the rows are few).
template <class Kern>
StreamGeom pick_geometry(river_ctx *c, Kern kern, int rows, int tasks, size_t smem, int R, int K) {
    StreamGeom small;
    if (stream_small_share(c->num_sms, rows, tasks, K, R, small)) return small;
    StreamGeom best{256, c->num_sms};
    double best_cost = 1e30;
    int best_w = 0;
    for (int w = 4; w <= 16; ++w) {
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, w * 32, smem) != cudaSuccess || occ < 1) continue;
        occ = std::min(occ, 64 / w);
        for (int o = 1; o <= occ; ++o) {
            const int ctas = c->num_sms * o;
            const int per_cta = (tasks + ctas - 1) / ctas;
            const int rounds = (per_cta + w - 1) / w;
            const int W = w * o;
            const double cost = rounds * (W < 16 ? 16.0 / W : 1.0) * (1.0 + 0.002 * o);  // few large CTAs share x loads
            if (cost < best_cost - 1e-9 || (std::fabs(cost - best_cost) < 1e-9 && W > best_w)) {
                best_cost = cost; best_w = W; best = StreamGeom{w * 32, ctas};
            }
        }
    }
    return best;
}

template <class P, int N, int R>
cudaError_t launch_stream_t(river_ctx *c, const P &p, const ProjIn &in, const RowLists &rl, int K, int tasks, int n,
                            int has_river, bool pdl, int skip_backbone, const DecideArgs &dec) {
    const size_t smem = stream_smem_bytes(N, K);
    auto kern = stream_proj_kernel<P, N, R>;
    const void *fn = reinterpret_cast<const void *>(kern);
    const river_ctx::Geom *geom = nullptr;
    const bool few = n <= kStreamFewRows;
    for (auto &e : c->geoms)
        if (e.fn == fn && e.tasks == tasks && e.K == K && e.few == few) geom = &e;
    if (!geom) {
        const cudaError_t e = ensure_smem(c, kern, smem);
        if (e != cudaSuccess) return e;
        const StreamGeom g = pick_geometry(c, kern, n, tasks, smem, R, K);
        c->geoms.push_back({fn, tasks, K, few, g.threads, g.grid});
        geom = &c->geoms.back();
    }
    return launch_k(kern, dim3(geom->grid), dim3(geom->threads), smem, c->stream, pdl, p, in, rl, has_river,
                    xs_stride(K, 32), skip_backbone, dec);
}

}  // namespace

template <class P>
cudaError_t launch_stream(river_ctx *c, const P &p, const ProjIn &in, const RowLists &rl, int K, int tasks_r2, int n,
                          int has_river, bool pdl, int skip_backbone, const DecideArgs &dec) {
    if constexpr (std::is_same_v<P, ResidProblem>) {
        // Three and more rows of a long K do not fit into shared memory together, and a pass for each pair would stream the
        // weights twice: two launches of half the inputs instead, the second adding to the first one's output (8B-class
        // blocks, three rows: 1424 us a step, so 1319, the row count's own instance included).
        if (n >= 3 && !in.gain && !p.ld && K % (2 * p.group) == 0 && K % 128 == 0 && stream_smem_bytes(3, K) > 200 * 1024) {
            ResidProblem a = p, b = p;
            ProjIn ia = in, ib = in;
            const int half = K / 2;
            a.K = b.K = half; a.ld = b.ld = ia.ld = ib.ld = K;
            b.w += half; b.rw.codes += half / 2; b.rw.scale += half / p.group; b.rw.zero += half / p.group;
            b.resid = p.out; ib.src += half;
            const cudaError_t e = launch_stream(c, a, ia, rl, half, tasks_r2, n, has_river, pdl, skip_backbone, dec);
            return e != cudaSuccess ? e : launch_stream(c, b, ib, rl, half, tasks_r2, n, has_river, pdl, skip_backbone, dec);
        }
    }
    // rows per pass: as many as the step has (up to four: every row costs its shared-memory reads and FMAs for every weight,
    // a row of padding too), if they fit
    int n_sel = 1;
    while (n_sel < n && n_sel < 4 && stream_smem_bytes(n_sel + 1, K) <= 200 * 1024) ++n_sel;
    const int r = K >= 4096 ? 2 : 4;  // weight rows per task
    const int tasks = tasks_r2 * 2 / r;
#define STREAM_CASE(N_, R_) if (n_sel == N_ && r == R_) return launch_stream_t<P, N_, R_>(c, p, in, rl, K, tasks, n, has_river, pdl, skip_backbone, dec);
    STREAM_CASE(1, 2) STREAM_CASE(2, 2) STREAM_CASE(3, 2) STREAM_CASE(4, 2)
    STREAM_CASE(1, 4) STREAM_CASE(2, 4) STREAM_CASE(3, 4) STREAM_CASE(4, 4)
#undef STREAM_CASE
    return cudaErrorInvalidValue;
}
template cudaError_t launch_stream<QkvProblem>(river_ctx *, const QkvProblem &, const ProjIn &, const RowLists &, int, int, int, int, bool, int, const DecideArgs &);
template cudaError_t launch_stream<ResidProblem>(river_ctx *, const ResidProblem &, const ProjIn &, const RowLists &, int, int, int, int, bool, int, const DecideArgs &);
template cudaError_t launch_stream<GateUpProblem>(river_ctx *, const GateUpProblem &, const ProjIn &, const RowLists &, int, int, int, int, bool, int, const DecideArgs &);

cudaError_t launch_head_stream(river_ctx *c, const HeadArgs &a, int n_head) {
    const int n_sel = std::min(n_head, 4);
    const int xstride = xs_stride(a.d, 8);
    const size_t smem = sizeof(float) * (64 + (size_t)n_sel * xstride);
    const int share = (a.V / (n_sel == 1 ? 2 : 4) + c->head_grid - 1) / c->head_grid;
    const int few = n_head <= kStreamFewRows ? std::max(4, share) : 16;  // (as stream_small_share)
    const int threads = std::min(head_threads(n_sel), 32 * few);
#define HEAD_CASE(N_, R_)                                                                                          \
    if (n_sel == N_) {                                                                                             \
        const cudaError_t e = ensure_smem(c, lm_head_kernel<N_, R_>, smem);                                        \
        if (e != cudaSuccess) return e;                                                                            \
        return launch_k(lm_head_kernel<N_, R_>, dim3(c->head_grid), dim3(threads), smem, c->stream, true, a, xstride); \
    }
    HEAD_CASE(1, 2) HEAD_CASE(2, 4) HEAD_CASE(3, 4) HEAD_CASE(4, 4)
#undef HEAD_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_argmax_final(river_ctx *c, int n_head, int n_parts) {
    return launch_k(argmax_final_kernel, dim3(n_head), dim3(128), 0, c->stream, true, c->meta(),
                    (const float *)c->part_val, (const int32_t *)c->part_idx, n_parts,
                    c->rows_distinct ? c->exit_hist : (unsigned long long *)nullptr);  // (not for prefill chunks)
}

}  // namespace river
