// Causal paged GQA attention of long prefill passes on tcgen05 (sm_100a).
//
// A CTA owns 128 query rows - 128 / GQ consecutive positions of one sequence x the GQ query heads of one KV head, head by head
// - and walks the cached keys 128 at a time, in two streams that take every other tile: each has its own K and V buffers, its own
// S and O in tensor memory and its own running maximum and sum, and the two meet when the keys are through.
//   S [128 x 128] = (Q_hi + Q_lo) K^T   Q (scaled, split x = hi + lo: 16 mantissa bits) and the K pages in shared memory
//   O [128 x DH] += (P_hi + P_lo) V     P in tensor memory over the place of S, the V pages in shared memory as they lie
//                                       in the cache (keys as rows: the N-major operand), O in tensor memory
//   warps 0, 1    TMA, one per stream: K and V pages, one 16 x 64 box per lane; K of the stream's next tile travels under the
//                 softmax, V under S, the first ones under the preparation of Q
//   warp 2        tensor memory; one lane issues the MMAs, S of one stream, O of the other, so that each stream's softmax runs under
//                 the other's MMAs (left to themselves, a lane each, the two fell into step: both softmaxes, then both products)
//   warps 4..11   softmax, four per stream: thread = query row = TMEM lane; online, base 2, fp32; O is rescaled only when a row's
//                 maximum has grown by more than 2^8 since it last was (the probabilities then reach 256 instead of 1: nothing in
//                 fp32).  P goes to the tensor cores in two halves, the first while the second is still being made.
//
// What bounds it: the tensor pipe (64 MMAs of 79 cycles per 128 keys of each stream, 6300 cycles of which 5100 are theirs) once a CTA
// is under way, and before that its start: 4 us until Q, K and V of the first tiles are there, as many again for the first pass over
// the code on every SM.  128 keys per tile because an MMA of M = 128 takes 75-85 cycles whatever its N up to 128; two streams because S
// and O of one are half of tensor memory, and a serial walk (S, softmax, P V) leaves the pipe idle for more than half of it.  (ncu, 8B
// class, 1024 positions: 46.5 us cold, pipe active 24 % of the SMs' time - it counts the 32 cycles of mathematics in an MMA's 79 -, DRAM 21
// MB.)  us per
// block and pass, one stream of 64-key tiles in each of two CTAs per SM against this: 8B-class, passes of 1024 positions of one
// prompt 64 / 114 / 171 -> 43 / 71 / 100; two prompts of the 1B class 26 -> 24; tiny shape, up to 1245 positions 45 -> 21.  The
// warp-level kernel (attn_prefill.cuh) stays for short passes and prompts.
#pragma once
#include "gemm_tc_w4.cuh"
#include "attn_prefill.cuh"

namespace river {

constexpr int kPtRows = 128;    // query rows per CTA
constexpr int kPtKeys = 128;    // keys per tile (eight pages)
constexpr int kPtStreams = 2;
constexpr int kPtThreads = 32 * 6 * kPtStreams;
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
__device__ __forceinline__ void pt_ld32(uint32_t taddr, float (&v)[32]) {  // 32 consecutive columns of this thread's lane
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,"
        "%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
          "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
          "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 consecutive columns, left under way (pt_st_wait).
__device__ __forceinline__ void pt_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void pt_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <int DH, int GQ>
__global__ void __launch_bounds__(kPtThreads, 1) attn_prefill_tc_kernel(const __grid_constant__ CUtensorMap tmap, const PrefillTcArgs a) {
    constexpr int NB = DH / 64;                          // blocks of 64 dims
    constexpr int POS = kPtRows / GQ;                    // positions per tile
    constexpr uint32_t QB = kPtRows * 128, KB = kPtKeys * 128;  // bytes of one block of Q / of K or V
    constexpr uint32_t kO = 256;                         // TMEM: stream i has S / P in columns 128 i .., O in columns 256 + DH i ..
    extern __shared__ uint8_t pt_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(pt_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sq = smem;                                  // [hi | lo][NB][128 rows][128 bytes]
    uint8_t *skv = sq + 2 * NB * QB;                     // [stream][K | V][NB][128 keys][128 bytes]
    __shared__ uint64_t bars[6 * kPtStreams];            // per stream: K landed, V landed, S done, P written (2), PV done
    __shared__ float2 s_ml[kPtStreams][kPtRows];         // a row's maximum and sum in each stream
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abortp = &s_abort;
    if (tid == 0) {
        s_abort = 0;
        for (int i = 0; i < 6 * kPtStreams; ++i) mbar_init(smem_u32(&bars[i]), i % 6 == 3 || i % 6 == 4 ? 4 : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
        tc_fence_before();
        pdl_launch();  // (behind the allocation: see tc_gemm_kernel)
    }
    // (the pass's own layout was on the device before its first kernel started)
    // tiles in descending order, the KV heads of a tile side by side: the longest prefixes first
    const int n_qt = gridDim.x / a.kv.Hkv, tile = n_qt - 1 - (int)blockIdx.x / a.kv.Hkv, kvh = blockIdx.x % a.kv.Hkv;
    const int row0 = a.tile_row0[tile], n_rows = a.tile_rows[tile];
    const int slot = a.kv.row_slot[row0], pos0 = a.kv.row_pos[row0], last_pos = pos0 + n_rows - 1;
    const int n_kt = last_pos / kPtKeys + 1, n_of[kPtStreams] = {(n_kt + 1) / 2, n_kt / 2};  // tiles of the streams
    // role: the stream, its tiles st, st + 2, .., its barriers and buffers
    const int st = warp < 4 ? warp & 1 : (warp - 4) >> 2, n_mine = st ? n_of[1] : n_of[0];
    const uint32_t bar0 = smem_u32(&bars[6 * st]), b_k = bar0, b_v = bar0 + 8, b_s = bar0 + 16, b_p = bar0 + 24, b_pv = bar0 + 40;
    uint8_t *const sk = skv + (size_t)st * 2 * NB * KB, *const sv = sk + NB * KB;

    __syncthreads();  // (the barriers, for the copies)
    pdl_wait();       // q and the chunk's own K / V come from the kernel before this one
    int n_copied = 0;
    // lane = (page, block): 16 x 64 boxes of K, then of V
    auto copy_tile = [&](int i) {
        const int pg = lane / NB, blk = lane % NB, t = st + kPtStreams * i, n_pg = min(kPtKeys / kPage, (last_pos - t * kPtKeys) / kPage + 1);
        int row_k = 0;
        const bool mine = pg < n_pg;
        if (mine) {
            int page = a.kv.page_tbl[(size_t)slot * a.kv.max_pages_per_seq + (kPtKeys / kPage) * t + pg];
            if (page < 0 || page >= a.kv.n_pages) { atomicExch(a.dev_err, DEV_BAD_PAGE); page = 0; }
            row_k = (((a.kv.layer0 * a.kv.n_pages + page) * 2) * a.kv.Hkv + kvh) * kPage;
        }
        const uint32_t bytes = (uint32_t)n_pg * NB * kPage * 128, off = (uint32_t)blk * KB + (uint32_t)pg * (kPage * 128);
        int good = 1;
        if (lane == 0 && i > 0) good = mbar_wait(b_s, (i - 1) & 1, abortp, a.dev_err) ? 1 : 0;  // (S done: K has been read)
        if (lane == 0 && good) mbar_expect_tx(b_k, bytes);
        if (!__shfl_sync(0xffffffffu, good, 0)) return false;
        if (mine) tma_load_2d(smem_u32(sk) + off, &tmap, 64 * blk, row_k, b_k);
        if (lane == 0 && i > 0) good = mbar_wait(b_pv, (i - 1) & 1, abortp, a.dev_err) ? 1 : 0;
        if (lane == 0 && good) mbar_expect_tx(b_v, bytes);
        if (!__shfl_sync(0xffffffffu, good, 0)) return false;
        if (mine) tma_load_2d(smem_u32(sv) + off, &tmap, 64 * blk, row_k + a.kv.Hkv * kPage, b_v);
        return true;
    };
    if (warp < 2) {
        if (n_mine > 0 && copy_tile(0)) n_copied = 1;
    } else {
        // ---- Q rows, hi and lo parts, in the operand's swizzled order (row r = head g, position p: r = g POS + p): all of a
        // thread's loads are under way before the first is split
        constexpr int QT = kPtThreads - 64, UNITS = kPtRows * (DH / 8), PER = (UNITS + QT - 1) / QT;  // units of eight dims
        float4 x[PER][2];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int u = tid - 64 + k * QT, r = u / (DH / 8), c8 = u % (DH / 8), g = r / POS, p = r % POS;
            x[k][0] = x[k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (u < UNITS && p < n_rows) {
                const float4 *src = reinterpret_cast<const float4 *>(a.q + (size_t)(row0 + p) * a.Hq * DH + (size_t)(kvh * GQ + g) * DH + 8 * c8);
                x[k][0] = __ldcg(src);
                x[k][1] = __ldcg(src + 1);
            }
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int u = tid - 64 + k * QT, r = u / (DH / 8), c8 = u % (DH / 8);
            if (u >= UNITS) break;
            const float y[8] = {x[k][0].x, x[k][0].y, x[k][0].z, x[k][0].w, x[k][1].x, x[k][1].y, x[k][1].z, x[k][1].w};
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float y0 = y[2 * e] * a.qscale, y1 = y[2 * e + 1] * a.qscale;
                const __nv_bfloat16 h0 = __float2bfloat16_rn(y0), h1 = __float2bfloat16_rn(y1);
                h[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                l[e] = pack_bf16x2(y0 - __bfloat162float(h0), y1 - __bfloat162float(h1));
            }
            uint8_t *dst = sq + (c8 >> 3) * QB + r * 128 + (((c8 & 7) ^ (r & 7)) * 16);
            *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4 *>(dst + NB * QB) = make_uint4(l[0], l[1], l[2], l[3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem, t_s = tmem + 128u * st, t_o = tmem + kO + (uint32_t)DH * st;

    if (warp < 2) {
        for (int i = 1; i < n_mine && n_copied == i; ++i)
            if (copy_tile(i)) ++n_copied;
    } else if (warp < 4) {
        if (warp == 2 && lane == 0) {
            const uint32_t id_s = tc_idesc(kPtKeys), id_o = tc_idesc(DH) | (1u << 16);  // (B of the second product: N-major)
            const uint64_t dq = tc_smem_desc(smem_u32(sq)), dk0 = tc_smem_desc(smem_u32(skv)), dv0 = pt_desc_n(smem_u32(skv + NB * KB), KB);
            auto scores = [&](int j, int i) {  // S of stream j's tile i
                const uint32_t bar = smem_u32(&bars[6 * j]);
                if (!mbar_wait(bar, i & 1, abortp, a.dev_err)) return false;
                if (i > 0 && !mbar_wait(bar + 40, (i - 1) & 1, abortp, a.dev_err)) return false;  // P of the tile before has been read
                tc_fence_after();
                const uint64_t dk = dk0 + (uint32_t)j * ((2 * NB * KB) >> 4);
#pragma unroll
                for (int k = 0; k < DH / 16; ++k) {
                    const uint64_t q = dq + (k >> 2) * (QB >> 4) + 2 * (k & 3), kk = dk + (k >> 2) * (KB >> 4) + 2 * (k & 3);
                    tc_mma(tmem + 128u * j, q, kk, id_s, k ? 1u : 0u);
                    tc_mma(tmem + 128u * j, q + NB * (QB >> 4), kk, id_s, 1u);
                }
                tc_commit(bar + 16);
                return true;
            };
            auto values = [&](int j, int i) {  // O += P V
                const uint32_t bar = smem_u32(&bars[6 * j]), o = tmem + kO + (uint32_t)DH * j;
                const uint64_t dv = dv0 + (uint32_t)j * ((2 * NB * KB) >> 4);
#pragma unroll
                for (int h = 0; h < 2; ++h) {  // half of the keys
                    if (!mbar_wait(bar + 24 + 8 * h, i & 1, abortp, a.dev_err)) return false;
                    tc_fence_after();
#pragma unroll
                    for (int k = 0; k < 4; ++k) {  // P: 16 keys = 8 columns, the high parts of 32 keys, their low parts; V: 16 keys = 2048 bytes
                        const uint32_t p = tmem + 128u * j + 64 * h + 32 * (k >> 1) + 8 * (k & 1);
                        const uint64_t v = dv + (4 * h + k) * (2048 >> 4);
                        tc_mma_ts(o, p, v, id_o, (i | h | k) ? 1u : 0u);
                        tc_mma_ts(o, p + 16, v, id_o, 1u);
                    }
                }
                tc_commit(bar + 40);
                return true;
            };
            bool ok = true;
            for (int i = 0; i < n_of[0] && ok; ++i)
                ok = scores(0, i) && (i == 0 || values(1, i - 1)) && (i >= n_of[1] || scores(1, i)) && values(0, i);
            if (ok && n_of[1] == n_of[0]) values(1, n_of[1] - 1);
        }
    } else {
        const int r = 32 * (warp & 3) + lane, p = r % POS, pos = pos0 + p;
        const uint32_t quarter = (uint32_t)(32 * (warp & 3)) << 16, l_s = t_s + quarter, l_o = t_o + quarter;
        float m = -1e30f, l = 0.f;
        bool ok = true;
        for (int i = 0; i < n_mine; ++i) {
            const int t = st + kPtStreams * i;
            ok = __all_sync(0xffffffffu, mbar_wait(b_s, i & 1, abortp, a.dev_err));
            if (!ok) break;
            tc_fence_after();
            // keys 0 .. seen of the tile are visible to this row (negative: none)
            const int seen = pos - t * kPtKeys;
            const bool whole = t * kPtKeys + kPtKeys - 1 <= pos0;  // every row sees the whole tile
            // 32 scores are held at a time, and read twice: for the maximum, for the probabilities.  (Loops as short as this: all of a
            // launch's CTAs start together, and a kernel's first pass over its code waits for every line of it.)
            float s[32], mx = m;
            auto take = [&](int c) {  // keys 32 c .. of the tile
                pt_ld32(l_s + 32 * c, s);
                if (!whole)
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (e > seen - 32 * c) s[e] = -1e30f;
            };
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                take(c);
                float x[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                for (int e = 4; e < 32; ++e) x[e & 3] = fmaxf(x[e & 3], s[e]);
                mx = fmaxf(mx, fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])));
            }
            const bool grow = mx > m + kPtLazy;
            if (__any_sync(0xffffffffu, grow)) {
                const float corr = grow ? ex2(m - mx) : 1.f;
                if (grow) m = mx;
                l *= corr;
                if (i > 0) {  // (the MMAs that wrote O are complete: S of this tile was issued behind them)
#pragma unroll 1
                    for (int c = 0; c < DH; c += 32) {
                        float o[32];
                        uint32_t w[32];
                        pt_ld32(l_o + c, o);
#pragma unroll
                        for (int e = 0; e < 32; ++e) w[e] = __float_as_uint(o[e] * corr);
                        tc_st32(l_o + c, w);
                    }
                }
            }
            const float me = m == -1e30f ? 0.f : m;  // (a row that has not seen a key yet: its scores are -1e30, its probabilities 0)
            ok = __all_sync(0xffffffffu, mbar_wait(b_v, i & 1, abortp, a.dev_err));  // V rows past the last position hold whatever
            if (!ok) break;                                                           // was there: zero them (0 x NaN is NaN)
            if (t == n_kt - 1) {
                const int from = last_pos + 1 - t * kPtKeys;  // first dead row
                for (int u = (tid - 128) & 127; u < (kPtKeys - from) * 8 * NB; u += 128) {
                    const int key = from + u / (8 * NB), c = u % (8 * NB);
                    *reinterpret_cast<uint4 *>(sv + (c >> 3) * KB + key * 128 + (c & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                take(c);
                uint32_t hi[16], lo[16];
                float sum[2] = {0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float p0 = ex2(s[2 * e] - me), p1 = ex2(s[2 * e + 1] - me);
                    sum[0] += p0;
                    sum[1] += p1;
                    const __nv_bfloat162 hh = __floats2bfloat162_rn(p0, p1);
                    hi[e] = *reinterpret_cast<const uint32_t *>(&hh);
                    const __nv_bfloat162 ll = __floats2bfloat162_rn(p0 - __low2float(hh), p1 - __high2float(hh));
                    lo[e] = *reinterpret_cast<const uint32_t *>(&ll);
                }
                l += sum[0] + sum[1];
                pt_st16(l_s + 32 * c, hi);
                pt_st16(l_s + 32 * c + 16, lo);
                if (c & 1) {
                    pt_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(b_p + 4 * (c & 2));
                }
            }
        }
        if (ok && n_mine > 0) ok = __all_sync(0xffffffffu, mbar_wait(b_pv, (n_mine - 1) & 1, abortp, a.dev_err));
        s_ml[st][r] = make_float2(m, l);
        asm volatile("bar.sync 1, %0;" ::"n"(128 * kPtStreams) : "memory");  // (softmax threads; those that gave up come here as well)
        // ---- both streams' parts of a row, half of the dims per thread
        if (ok && !*abortp) {
            const int n_other = st ? n_of[0] : n_of[1];
            if (n_other > 0) mbar_wait(smem_u32(&bars[6 * (1 - st) + 5]), (n_other - 1) & 1, abortp, a.dev_err);  // (done: its threads have been there)
            tc_fence_after();
            const float2 m0 = s_ml[0][r], m1 = s_ml[1][r];
            const float mm = fmaxf(m0.x, m1.x), w0 = ex2(m0.x - mm), w1 = ex2(m1.x - mm), inv = 1.f / (m0.y * w0 + m1.y * w1);
            const float f0 = w0 * inv, f1 = w1 * inv;
            // 32 rows x 32 dims at a time through shared memory (the K and V tiles are done with): whole 128-byte lines of a row go out
            float *const stage = reinterpret_cast<float *>(skv) + (warp - 4) * 32 * 36;
#pragma unroll 1
            for (int c = DH / 2 * st; c < DH / 2 * (st + 1); c += 32) {
                float o[32];
                pt_ld32(tmem + kO + quarter + c, o);
#pragma unroll
                for (int e = 0; e < 32; ++e) o[e] *= f0;
                if (n_kt > 1) {  // (else the second stream had no tile and its O was never written)
                    float o1[32];
                    pt_ld32(tmem + kO + DH + quarter + c, o1);
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[e] += o1[e] * f1;
                }
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 32; e += 4) *reinterpret_cast<float4 *>(stage + lane * 36 + e) = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
                __syncwarp();
#pragma unroll
                for (int e = 0; e < 32; e += 4) {
                    const int rr = 32 * (warp & 3) + e + (lane >> 3), pp = rr % POS, gg = rr / POS;
                    if (pp < n_rows)
                        *reinterpret_cast<float4 *>(a.out + (size_t)(row0 + pp) * a.Hq * DH + (size_t)(kvh * GQ + gg) * DH + c + 4 * (lane & 7)) =
                            *reinterpret_cast<const float4 *>(stage + (e + (lane >> 3)) * 36 + 4 * (lane & 7));
                }
            }
            tc_fence_before();
        }
    }
    __syncwarp();
    if (*abortp) {  // a wait ran out: what this CTA has asked for lands within microseconds; do not leave before
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
    }
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

// (the head dim of 64 asks for as much as 128 does: a CTA takes all of an SM's tensor memory, so that no CTA that wants some - they
// all hold 50 KB and more - shares its SM and waits there)
inline size_t attn_prefill_tc_smem_bytes() { return 1024 + 2 * (2 * kPtRows * 128 + 2 * kPtStreams * kPtKeys * 128); }

}  // namespace river
