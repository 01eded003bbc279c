// Host-side state of one decode context and the launch helpers shared by the translation units of the library.
// (Internal: the public interface is include/river.h.)
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "../../include/river.h"
#include "river_common.cuh"

constexpr int kStaging = 4;  // pinned metadata buffers in flight
enum KernelClass { K_BEGIN, K_QKV, K_ATTN, K_OPROJ, K_GATEUP, K_DOWN, K_SCORE, K_HEAD, K_ARGMAX, K_PREFILL_ATTN, kNumClasses };

struct river_ctx {
    river_config cfg;        // as given, except max_batch = max(max_batch, prefill_chunk): rows per launch sequence
    int user_max_batch = 0;  // rows per decode step the caller asked for
    std::vector<river_layer_weights> layers;
    const uint16_t *embed, *lm_head, *final_norm;
    cudaStream_t stream;
    int device = 0, num_sms = 0;
    __nv_bfloat16 *pool = nullptr;

    // workspace
    float *h[3], *qbuf, *obuf, *act, *part_val, *tau_i, *logits_i, *scores_i;
    float2 *rope_cs, *part_ml;
    float *part_o;
    CUtensorMap kv_tmap;
    int attn_splits_now = 1;
    bool attn_small_now = false;  // this step's attention runs on the small-step kernel (short contexts, 1-4 rows)
    unsigned *attn_tickets, *tickets;  // [max_batch*Hkv], [4]
    // tensor-core path: operand buffers, tensor maps of every weight matrix
    __nv_bfloat16 *tc_xhi = nullptr, *tc_xlo = nullptr;
    __nv_bfloat16 *tc_x4 = nullptr;  // the same pair for the exit-layer rows (f16 bits): both kernels of a projection run at once
    __nv_bfloat16 *tc_xalt = nullptr, *tc_x4alt = nullptr;  // second set: operand rows written by the PREVIOUS projection's
                                                            // epilogues (gate/up -> down) while that projection still reads its own
    int tc_max_pad = 0, tc_kmax = 0;
    bool tc_ok = false;
    struct LayerMaps { CUtensorMap q, k, v, o, g, u, d; };
    std::vector<LayerMaps> tc_maps;
    std::vector<LayerMaps> w4_maps;  // code matrices of the exit layers (u8 [rows][K/2], 128-byte boxes)
    bool w4tc_ok = false;
    CUtensorMap tc_map_head;
    // operand maps of the tensor-core projections for (K, padded rows): up to 128 rows the lo rows follow the hi rows
    // in one buffer (`lo_ptr` = tc_xhi + np K) and `hi` covers both (one copy per k-block); beyond, two buffers
    // (box: rows of a copy, np or a row tile's; `one`: one copy takes the hi and the lo rows)
    struct BMap { int K, np, box; bool w4, alt, one; __nv_bfloat16 *base, *lo_ptr; CUtensorMap hi, lo; };
    std::vector<BMap> tc_bmaps;
    // long prefill passes (launch_tc_wide.cu): rows per pass (0: not for this context), operand rows (high parts, low parts
    // behind them) of the projections that read h / the attention output, and of the down projection; f16 exit-layer weights
    int wide_rows = 0;
    uint16_t *wide_x = nullptr, *wide_xalt = nullptr;
    __half *wide_w = nullptr;
    std::vector<LayerMaps> wide_bmaps, wide_wmaps;  // the pair kernel's maps of the backbone and (one entry) over wide_w
    struct WMap { int K, bn; bool alt; CUtensorMap hi, lo; };
    std::vector<WMap> wide_maps;
    int32_t *hint_act;
    const uint8_t *attn_skip = nullptr;  // exit flags of the block whose attention is being launched (strategies that run nothing for rows that left), else null
    uint8_t *pos_depth = nullptr;  // [max_seqs][max_pages_per_seq * 16] KV Mask: backbone blocks the token at each position ran
    int attn_layer1 = 0;           // block (1-based) whose attention is being launched (KV Mask: the visibility test)
    unsigned long long *exit_hist = nullptr;  // [L + 1] exit layers of all decoded tokens so far (river_exit_histogram)
    int32_t *slot_cap = nullptr;  // [max_seqs] Mono-Decreasing Exit: the depth the sequence's last token reached
    bool prefill_attn_now = false;  // this chunk's attention runs on the tensor-core prefill kernel
    bool rows_distinct = true;  // every row of the current step is a different sequence (decode), not a prefill chunk
    bool short_sums = false;    // the batch kernels' projections under way sum no more inputs at a time than a long pass's (tc_wide_segment)
    struct GraphEntry { int n; bool small_attn; int attn_splits; cudaGraphExec_t exec; int launches; };
    std::vector<GraphEntry> graphs;
    double *inv_freq;
    int32_t *act_idx, *riv_idx, *n_act, *n_riv, *page_tbl_dev, *part_idx, *tok_i, *forced_i, *exit_i, *next_i;
    int32_t *meta_dev;  // [kMetaHdr + 11*meta_rows]: StepMeta, row_slot, row_pos, upd[3], head_rows, row_page, row_forced,
                        // tile_row0, tile_rows (query tiles of a prefill chunk), attn_order
    int32_t *prefill_fail;  // [max_seqs][L+1]: 1 where some prompt position of the sequence failed Eq. 1 after block l
    uint8_t *state;     // [(L+1)][state_stride]: sticky exit flags of the rows entering block l + 1 (entry L: at the LM head)
    int state_stride = 0;
    uint8_t *pass;
    int *dev_err;
    size_t ws_bytes = 0;

    // host state
    std::vector<int32_t> page_tbl, seq_len, free_pages;
    int32_t *meta_host[kStaging] = {nullptr, nullptr, nullptr, nullptr};
    int meta_host_rows[kStaging] = {0};  // the meta_rows each was last laid out for
    cudaEvent_t meta_ev[kStaging];
    int meta_next = 0;
    void *pin_io = nullptr;  // pinned staging for the *_host entry point
    size_t pin_io_bytes = 0;
    int32_t *pin_full_depth() const { return reinterpret_cast<int32_t *>(static_cast<char *>(pin_io) + pin_io_bytes) - 1; }  // holds L, for copies that nobody waits for
    std::vector<int32_t> last_pos;  // positions of the rows of the last decode step
    int head_grid = 0;

    river_stats_t st{};
    std::string err;

    // backbone offloading: blocks >= off_first keep their bf16 matrices in pinned host memory and are staged, on
    // demand, into the two device slots their layer entries alias
    int off_first = 0;  // 0 = off
    std::vector<river_layer_weights> off_host;
    cudaStream_t off_copy = nullptr;
    cudaEvent_t off_ready[2] = {nullptr, nullptr}, off_freed[2] = {nullptr, nullptr};
    int off_slot_layer[2] = {-1, -1};

    // per-context launch bookkeeping: the dynamic shared memory limit of every kernel that was set up, and the launch geometry
    // of the streaming kernels per (kernel, task count, K, up to four rows or more)
    struct SmemAttr { const void *fn; size_t bytes; };
    std::vector<SmemAttr> smem_attr;
    struct Geom { const void *fn; int tasks, K; bool few; int threads, grid; };
    std::vector<Geom> geoms;

    // optional per-kernel timing (river_profile): events around every launch of a step
    bool profiling = false;
    std::vector<cudaEvent_t> prof_ev;
    struct ProfRec { int cls; double bytes_act, bytes_riv; int list_idx; };
    std::vector<ProfRec> prof_rec;
    double prof_ms[kNumClasses] = {0}, prof_bytes[kNumClasses] = {0};
    int64_t prof_launches[kNumClasses] = {0};

    // The metadata block holds 11 arrays of meta_rows entries behind its header: cfg.max_batch for decode steps and short
    // prefill passes, wide_rows for a long pass.
    int meta_rows = 0;
    int list_rows = 0;  // entries per block of the row lists: max(cfg.max_batch, wide_rows)
    int meta_ints() const { return river::kMetaHdr + 11 * meta_rows; }
    river::StepMeta *meta() const { return reinterpret_cast<river::StepMeta *>(meta_dev); }
    int32_t *row_slot() const { return meta_dev + river::kMetaHdr; }
    int32_t *row_pos() const { return meta_dev + river::kMetaHdr + meta_rows; }
    int32_t *upd() const { return meta_dev + river::kMetaHdr + 2 * meta_rows; }
    int32_t *head_rows() const { return meta_dev + river::kMetaHdr + 5 * meta_rows; }
    int32_t *row_page() const { return meta_dev + river::kMetaHdr + 6 * meta_rows; }  // page of each row's new position
    int32_t *row_forced() const { return meta_dev + river::kMetaHdr + 7 * meta_rows; }  // prefill: forced exit per row
    int32_t *tile_row0() const { return meta_dev + river::kMetaHdr + 8 * meta_rows; }
    int32_t *tile_rows() const { return meta_dev + river::kMetaHdr + 9 * meta_rows; }
    int32_t *attn_order() const { return meta_dev + river::kMetaHdr + 10 * meta_rows; }  // rows, longest context first
    uint8_t *state_at(int l) const { return state + (size_t)l * state_stride; }
};

namespace river {

// Launch with the programmatic-dependent-launch attribute: the kernel may start while its predecessor in the
// stream is still running and orders itself with griddepcontrol.wait.  Every kernel launched this way calls
// griddepcontrol.wait before it touches anything a predecessor writes.
inline thread_local int64_t t_launches = 0;  // kernels this thread has launched: a step's count is what it adds
template <class... KArgs, class... Args>
cudaError_t launch_kc(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                      int cluster_x, Args &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int na = 0;
    if (pdl) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    if (cluster_x > 1) {  // consecutive CTAs along x form a thread-block cluster
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = cluster_x;
        at[na].val.clusterDim.y = 1;
        at[na].val.clusterDim.z = 1;
        ++na;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    ++t_launches;
    return cudaLaunchKernelEx(&cfg, kern, KArgs(std::forward<Args>(args))...);
}
template <class... KArgs, class... Args>
cudaError_t launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                     Args &&...args) {
    return launch_kc(kern, grid, block, smem, st, pdl, 1, std::forward<Args>(args)...);
}

// cudaFuncAttributeMaxDynamicSharedMemorySize belongs to the device, not to a context: a context that set it to what its
// own launches need would lower it under another context's larger launches (which then fail as invalid).  So every kernel's
// limit goes straight to the most the device allows beside its static shared memory - the same value whoever sets it - and
// a context only remembers that it has done so.
template <class Kern>
cudaError_t ensure_smem(river_ctx *c, Kern kern, size_t bytes) {
    const void *fn = reinterpret_cast<const void *>(kern);
    for (auto &a : c->smem_attr)
        if (a.fn == fn) return bytes <= a.bytes ? cudaSuccess : cudaErrorInvalidValue;
    cudaFuncAttributes fa;
    int most = 0;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
    if (e != cudaSuccess) return e;
    most -= (int)fa.sharedSizeBytes;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) != cudaSuccess) return e;
    c->smem_attr.push_back({fn, (size_t)most});
    return bytes <= (size_t)most ? cudaSuccess : cudaErrorInvalidValue;
}

inline KvAddr kv_addr(const river_ctx *c, int layer0) {
    KvAddr k;
    k.pool = c->pool;
    k.page_tbl = c->page_tbl_dev;
    k.row_slot = c->row_slot();
    k.row_pos = c->row_pos();
    k.row_page = c->row_page();
    k.n_pages = c->cfg.n_pages;
    k.max_pages_per_seq = c->cfg.max_pages_per_seq;
    k.Hkv = c->cfg.Hkv;
    k.dh = c->cfg.dh;
    k.layer0 = layer0;
    return k;
}

inline W4 w4_of(const river_w4 &r) {
    return W4{(const uint8_t *)r.codes, (const uint16_t *)r.scale, (const uint16_t *)r.zero};
}

}  // namespace river
