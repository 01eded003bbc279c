// Causal paged GQA attention of long prefill passes on tcgen05 (sm_100a).
//
// A CTA owns 128 query rows - 128 / GQ consecutive positions of one sequence x the GQ query heads of one KV head, head by head
// - and walks the cached keys 64 at a time:
//   S [128 x 64]  = (Q_hi + Q_lo) K^T   Q (scaled, split x = hi + lo: 16 mantissa bits) and the K pages in shared memory
//   O [128 x DH] += (P_hi + P_lo) V     P in tensor memory over the place of S, the V pages in shared memory as they lie
//                                       in the cache (keys as rows: the N-major operand), O in tensor memory
//   warp 0     TMA: K and V pages, one 16 x 64 box per lane; K of the next tile travels under the softmax, V under S
//   warp 1     TMEM allocation; one lane issues the MMAs
//   warps 2..5 softmax: thread = query row = TMEM lane; online, base 2, fp32; O is rescaled only when a row's maximum has grown
//              by more than 2^8 since it last was (the probabilities then reach 256 instead of 1: nothing in fp32)
// Two CTAs per SM (96 KB, 256 TMEM columns each): one's softmax runs under the other's MMAs.
//
// What bounds it: the tensor pipe - 24 MMAs of 85 cycles per 64 keys (an MMA of M = 128 takes that whatever its N up to 128), and
// beside it the softmax's issue slots.  8B-class shape, per block: 1024 positions 104 -> 61 us, the passes of a 4001-position
// prompt 306 -> 145 us on average, against the warp-level kernel (attn_prefill.cuh), which stays for short passes and prompts
// and for tiles of a single row.
#pragma once
#include "gemm_tc_w4.cuh"
#include "attn_prefill.cuh"

namespace river {

constexpr int kPtRows = 128;    // query rows per CTA
constexpr int kPtKeys = 64;     // keys per tile (four pages)
constexpr int kPtThreads = 192;
constexpr float kPtLazy = 8.f;  // growth of a row's maximum (log2) that O waits for before it is rescaled

struct PrefillTcArgs {
    const int32_t *tile_row0, *tile_rows;  // query tiles of up to 128 / GQ positions
    const float *q;
    float *out;
    KvAddr kv;
    int Hq;
    float qscale;
    int *dev_err;
};

// N-major operand (the V tile: rows = keys of 128 bytes, 64 dims per block), 128-byte swizzle: 8-key groups 1024 bytes apart,
// blocks of 64 dims `block` bytes apart.
__device__ __forceinline__ uint64_t pt_desc_n(uint32_t saddr, uint32_t block) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(block >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void pt_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,"
        "%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
          "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
          "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int DH, int GQ>
__global__ void __launch_bounds__(kPtThreads, 2) attn_prefill_tc_kernel(const __grid_constant__ CUtensorMap tmap, const PrefillTcArgs a) {
    constexpr int NB = DH / 64;                          // blocks of 64 dims
    constexpr int POS = kPtRows / GQ;                    // positions per tile
    constexpr uint32_t QB = kPtRows * 128, KB = kPtKeys * 128;  // bytes of one block of Q / of K or V
    constexpr uint32_t kO = 128, kCols = 256;            // TMEM: S / P in columns 0..63, O from 128 on
    extern __shared__ uint8_t pt_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(pt_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sq = smem;                                  // [hi | lo][NB][128 rows][128 bytes]
    uint8_t *sk = sq + 2 * NB * QB, *sv = sk + NB * KB;  // [NB][64 keys][128 bytes] each
    __shared__ uint64_t bars[6];                         // K landed, K free, V landed, S done, P written, PV done
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t b_k = smem_u32(&bars[0]), b_kfree = smem_u32(&bars[1]), b_v = smem_u32(&bars[2]), b_s = smem_u32(&bars[3]),
                   b_p = smem_u32(&bars[4]), b_pv = smem_u32(&bars[5]);
    volatile int *abortp = &s_abort;
    pdl_launch();
    if (tid == 0) {
        s_abort = 0;
        mbar_init(b_k, 1); mbar_init(b_kfree, 1); mbar_init(b_v, 1); mbar_init(b_s, 1); mbar_init(b_p, 4); mbar_init(b_pv, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
        tc_fence_before();
    }
    pdl_wait();  // q and the chunk's own K / V come from the kernel before this one
    // tiles in descending order: the longest prefixes first
    const int tile = gridDim.x - 1 - blockIdx.x, kvh = blockIdx.y;
    const int row0 = a.tile_row0[tile], n_rows = a.tile_rows[tile];
    const int slot = a.kv.row_slot[row0], pos0 = a.kv.row_pos[row0], last_pos = pos0 + n_rows - 1;
    const int n_kt = last_pos / kPtKeys + 1;

    // ---- Q rows, hi and lo parts, in the operand's swizzled order (row r = head g, position p: r = g POS + p)
    for (int u = tid; u < kPtRows * (DH / 8); u += kPtThreads) {
        const int r = u / (DH / 8), c8 = u % (DH / 8), g = r / POS, p = r % POS;  // eight dims
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = 0.f;
        if (p < n_rows) {
            const float4 *src = reinterpret_cast<const float4 *>(a.q + (size_t)(row0 + p) * a.Hq * DH + (size_t)(kvh * GQ + g) * DH + 8 * c8);
            const float4 v0 = __ldcg(src), v1 = __ldcg(src + 1);
            x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w; x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
        }
        uint32_t h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float y0 = x[2 * e] * a.qscale, y1 = x[2 * e + 1] * a.qscale;
            const __nv_bfloat16 h0 = __float2bfloat16_rn(y0), h1 = __float2bfloat16_rn(y1);
            h[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
            l[e] = pack_bf16x2(y0 - __bfloat162float(h0), y1 - __bfloat162float(h1));
        }
        uint8_t *dst = sq + (c8 >> 3) * QB + r * 128 + (((c8 & 7) ^ (r & 7)) * 16);
        *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4 *>(dst + NB * QB) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        // lane = (page, block): 16 x 64 boxes of K, then of V
        const int pg = lane / NB, blk = lane % NB;
        const int32_t *pt = a.kv.page_tbl + (size_t)slot * a.kv.max_pages_per_seq;
        bool ok = true;
        for (int t = 0; t < n_kt && ok; ++t) {
            const int n_pg = min(4, (last_pos - t * kPtKeys) / kPage + 1);
            int row_k = 0;
            const bool mine = lane < 4 * NB && pg < n_pg;
            if (mine) {
                int page = pt[4 * t + pg];
                if (page < 0 || page >= a.kv.n_pages) { atomicExch(a.dev_err, DEV_BAD_PAGE); page = 0; }
                row_k = (((a.kv.layer0 * a.kv.n_pages + page) * 2) * a.kv.Hkv + kvh) * kPage;
            }
            const uint32_t bytes = (uint32_t)n_pg * NB * kPage * 128, off = (uint32_t)blk * KB + (uint32_t)pg * (kPage * 128);
            int good = 1;
            if (lane == 0 && t > 0) good = mbar_wait(b_kfree, (t - 1) & 1, abortp, a.dev_err) ? 1 : 0;
            if (lane == 0 && good) mbar_expect_tx(b_k, bytes);
            if (!__shfl_sync(0xffffffffu, good, 0)) break;
            if (mine) tma_load_2d(smem_u32(sk) + off, &tmap, 64 * blk, row_k, b_k);
            if (lane == 0 && t > 0) good = mbar_wait(b_pv, (t - 1) & 1, abortp, a.dev_err) ? 1 : 0;
            if (lane == 0 && good) mbar_expect_tx(b_v, bytes);
            if (!__shfl_sync(0xffffffffu, good, 0)) { ok = false; break; }
            if (mine) tma_load_2d(smem_u32(sv) + off, &tmap, 64 * blk, row_k + a.kv.Hkv * kPage, b_v);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t id_s = tc_idesc(kPtKeys), id_o = tc_idesc(DH) | (1u << 16);  // (B of the second product: N-major)
            const uint64_t dq = tc_smem_desc(smem_u32(sq)), dk = tc_smem_desc(smem_u32(sk)), dv = pt_desc_n(smem_u32(sv), KB);
            for (int t = 0; t < n_kt; ++t) {
                const uint32_t par = t & 1;
                if (!mbar_wait(b_k, par, abortp, a.dev_err)) break;
                if (t > 0 && !mbar_wait(b_pv, par ^ 1, abortp, a.dev_err)) break;  // P of the tile before has been read
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < DH / 16; ++k) {
                    const uint64_t q = dq + (k >> 2) * (QB >> 4) + 2 * (k & 3), kk = dk + (k >> 2) * (KB >> 4) + 2 * (k & 3);
                    tc_mma(tmem, q, kk, id_s, k ? 1u : 0u);
                    tc_mma(tmem, q + NB * (QB >> 4), kk, id_s, 1u);
                }
                tc_commit(b_s);
                tc_commit(b_kfree);
                if (!mbar_wait(b_p, par, abortp, a.dev_err)) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < kPtKeys / 16; ++k) {  // P: 16 keys = 8 columns; V: 16 keys = 2048 bytes
                    tc_mma_ts(tmem + kO, tmem + 8 * k, dv + k * (2048 >> 4), id_o, (t | k) ? 1u : 0u);
                    tc_mma_ts(tmem + kO, tmem + 32 + 8 * k, dv + k * (2048 >> 4), id_o, 1u);
                }
                tc_commit(b_pv);
            }
        }
    } else {
        const int r = 32 * (warp & 3) + lane, p = r % POS, g = r / POS, pos = pos0 + p;
        const uint32_t lane0 = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        float m = -1e30f, l = 0.f;
        bool ok = true;
        for (int t = 0; t < n_kt; ++t) {
            ok = __all_sync(0xffffffffu, mbar_wait(b_s, t & 1, abortp, a.dev_err));
            if (!ok) break;
            tc_fence_after();
            float s[2][32];
            pt_ld32(lane0, s[0]);
            pt_ld32(lane0 + 32, s[1]);
            const int seen = pos - t * kPtKeys;  // keys 0 .. seen of the tile are visible (negative: none)
            float mx = m;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    if (32 * h + e > seen) s[h][e] = -1e30f;
                    mx = fmaxf(mx, s[h][e]);
                }
            // (m starts at -1e30: the first visible key always sets it; key 0 of tile 0 is visible to every row)
            const bool grow = mx > m + kPtLazy;
            if (__any_sync(0xffffffffu, grow)) {
                const float corr = grow ? ex2(m - mx) : 1.f;
                if (grow) m = mx;
                l *= corr;
                if (t > 0) {  // (the MMAs that wrote O are complete: S of this tile was issued behind them)
#pragma unroll 1
                    for (int c = 0; c < DH; c += 32) {
                        float o[32];
                        uint32_t w[32];
                        pt_ld32(lane0 + kO + c, o);
#pragma unroll
                        for (int e = 0; e < 32; ++e) w[e] = __float_as_uint(o[e] * corr);
                        tc_st32(lane0 + kO + c, w);
                    }
                }
            }
            uint32_t hi[32], lo[32];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    const float p0 = s[h][e] <= -1e29f ? 0.f : ex2(s[h][e] - m), p1 = s[h][e + 1] <= -1e29f ? 0.f : ex2(s[h][e + 1] - m);
                    l += p0 + p1;
                    const __nv_bfloat162 hh = __floats2bfloat162_rn(p0, p1);
                    hi[16 * h + e / 2] = *reinterpret_cast<const uint32_t *>(&hh);
                    const __nv_bfloat162 ll = __floats2bfloat162_rn(p0 - __low2float(hh), p1 - __high2float(hh));
                    lo[16 * h + e / 2] = *reinterpret_cast<const uint32_t *>(&ll);
                }
            tc_st32(lane0, hi);
            tc_st32(lane0 + 32, lo);
            ok = __all_sync(0xffffffffu, mbar_wait(b_v, t & 1, abortp, a.dev_err));  // V rows past the last position hold whatever
            if (!ok) break;                                                           // was there: zero them (0 x NaN is NaN)
            if (t == n_kt - 1) {
                const int from = last_pos + 1 - t * kPtKeys;  // first dead row
                for (int u = tid - 64; u < (kPtKeys - from) * 8 * NB; u += 128) {
                    const int key = from + u / (8 * NB), c = u % (8 * NB);
                    *reinterpret_cast<uint4 *>(sv + (c >> 3) * KB + key * 128 + (c & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_p);
        }
        if (ok && (ok = __all_sync(0xffffffffu, mbar_wait(b_pv, (n_kt - 1) & 1, abortp, a.dev_err)))) {
            tc_fence_after();
            const float inv = 1.f / l;
            float *dst = a.out + (size_t)(row0 + p) * a.Hq * DH + (size_t)(kvh * GQ + g) * DH;
#pragma unroll 1
            for (int c = 0; c < DH; c += 32) {
                float o[32];
                pt_ld32(lane0 + kO + c, o);
                if (p < n_rows)
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<float4 *>(dst + c + e) = make_float4(o[e] * inv, o[e + 1] * inv, o[e + 2] * inv, o[e + 3] * inv);
            }
            tc_fence_before();
        }
    }
    __syncwarp();
    if (*abortp) {  // a wait ran out: what this CTA has asked for lands within microseconds; do not leave before
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
    }
}

inline size_t attn_prefill_tc_smem_bytes(int DH) { return 1024 + (size_t)(DH / 64) * (2 * kPtRows * 128 + 2 * kPtKeys * 128); }

}  // namespace river
