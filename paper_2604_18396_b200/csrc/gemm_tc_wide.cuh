// Projections of long prefill passes (hundreds of rows) on CTA PAIRS (sm_100a): tcgen05.mma.cta_group::2, persistent.
//
// D[256 output features x BN rows] per pair and tile: each CTA holds 128 of the features (its own A tile and its own 128
// TMEM lanes) and HALF of the activation rows' tile; the tensor cores of both read both halves.  A k-block (64 inputs) of
// a CTA is 16 KB of weights and BN / 2 rows of the activations' high and low parts (2 x 16 KB at BN = 256), consumed by
// eight MMAs: 4 hi + 4 lo (x = hi + lo keeps 16 mantissa bits, as in tc_gemm_kernel).
//   warp 0      one lane: 2-D TMA copies; both CTAs' copies count on the LEADER's full barrier (CTA 0 of the pair)
//   warp 1      TMEM allocation; in the leader one lane issues the MMAs; tcgen05.commit reports to both CTAs
//   warps 2..17 epilogue: four groups of four warps take 32-row chunks out of TMEM in turn, add a tile's segments up in
//               registers and run the projection's epilogue from there
// K is accumulated in segments of at most 1024 inputs, each from zero in one of two accumulators (2 x 256 columns), and the
// segments are added up in round-to-nearest fp32: the error of one long sum in the tensor cores grows with its length
// (logits of one 8B-class block against 64 bits: one sum 5.2e-4, segments of 2048 / 1024 / 512 inputs 3.9e-4 / 3.4e-4 / 2.3e-4;
// the K-split batch kernels 3.5e-4).  Segments of 1024 cost nothing measurable, of 512 about 3 %.  The same double buffering runs a tile's
// epilogue under the next tile's MMAs.  Tiles go to the pairs in the order (features outer, rows inner), so that the pairs
// working at one time share weight tiles in L2.
//
// What bounds it: the tensor pipe for gate/up and down (81 and 76 % of the kernel's time busy under ncu), and the power cap
// when passes follow each other; QKV and O (65 and 63 %) have too few tiles for whole rounds.  8B-class shape, 1024 rows, inside
// passes that follow each other, operand kernel included: QKV 94 us, O 59, gate/up 321, down 154 - 1.10, 1.16, 1.50 and 1.56 PFLOP/s of
// bf16 MMAs, half of them for the low parts - against 4 x (108, 42, 191, 81) us in passes of 256 rows on tc_gemm_kernel.
#pragma once
#include "gemm_tc.cuh"
#include "gemm_tc_w4.cuh"

namespace river {

constexpr int kWdEpiWarps = 16, kWdGroups = kWdEpiWarps / 4;
constexpr int kWdThreads = 64 + 32 * kWdEpiWarps;
constexpr int kWdChunk = 32;                                       // rows of an epilogue chunk
constexpr int kWdOwn = 256 / (kWdChunk * kWdGroups);               // chunks of a tile that one epilogue warp holds, at most
constexpr uint32_t kWdABytes = kTcBM * kTcBK * 2;

// ---------------------------------------------------------------- epilogues, straight from registers
// A thread holds tile row r = 32 quarter + lane of a 32-row chunk, v[e] = the value for list row n0 + e (e < live); `row` is the
// step row id of list row n0 + lane.  begin() runs before the tile's first segment is there: it sets the sums' start and
// requests what run() will need (run() gets its return value back), so that no load waits behind the last MMA (residual
// and cache slots read in run() instead: 8B-class O 68 us against 56, down 157 against 148, 1024 rows).  Nothing is staged: the copies lay a tile's weight rows down so that
// what belongs together (gate and up feature, the two halves of a rotary pair) sits 16 lanes apart in one warp - ONE copy
// per tile and k-block does that, through a five-dimensional map (make_map_paired); eight copies of 16 rows each kept the
// issuing lane from keeping up (8B-class gate/up, 1024 rows: 490 us against 433) - and lanes 0-15 finish the even
// rows of the chunk, lanes 16-31 the odd ones.
// out[row][f] = resid[row][f] + value; tile rows in the matrix's own order.  The sums start from the residual: every segment is
// rounded at its magnitude (14 times for K = 14336).  Added once, before the last segment, it moved no distance from 64-bit
// arithmetic (mini, 1B-class and 8B-class blocks, 300 and 1000 positions: the third digit) and cost 2-7 % of a prompt.
struct WdResidEpi {
    const float *resid;
    float *out;
    int out_dim;
    static constexpr bool kPaired = false;
    __device__ int begin(float (&v)[32], int ft, int quarter, int lane, int live, int row) const {  // the sums start from the residual
        const int f = ft * kTcBM + 32 * quarter + lane;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const int o = __shfl_sync(0xffffffffu, row, e) * out_dim + f;  // (a pass holds at most 1024 rows: 32-bit offsets)
            v[e] = e < live ? __ldcg(resid + o) : 0.f;
        }
        return 0;
    }
    __device__ void run(float (&v)[32], int ft, int quarter, int lane, int live, int row, int, int) const {
        const int f = ft * kTcBM + 32 * quarter + lane;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
            const int o = __shfl_sync(0xffffffffu, row, e) * out_dim + f;
            if (e < live) out[o] = v[e];
        }
    }
};
// Lane pairs (l, l + 16) trade so that lanes 0-15 hold (a, b) of chunk row e and lanes 16-31 (a, b) of row e + 1, where a
// is the value of the lower tile row and b of the upper one.
__device__ __forceinline__ void wd_trade(float v0, float v1, int lane, float &a, float &b) {
    const float got = __shfl_xor_sync(0xffffffffu, lane < 16 ? v1 : v0, 16);
    a = lane < 16 ? v0 : got;
    b = lane < 16 ? got : v1;
}
__device__ __forceinline__ int wd_zero(float (&v)[32]) {
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = 0.f;
    return 0;
}
struct WdGateUpEpi {  // 64 features per tile -> the down projection's operand rows, as TcGateUpEpi writes them
    int F;
    uint16_t *ohi, *olo;
    int f16, up_first;  // up_first: the lower row of a pair is the up feature
    static constexpr bool kPaired = true;
    __device__ int begin(float (&v)[32], int, int, int, int, int) const { return wd_zero(v); }
    __device__ void run(float (&v)[32], int ft, int quarter, int lane, int live, int, int, int n0) const {
        const int f = ft * 64 + 16 * quarter + (lane & 15), j = f & 7;
        const int at = f16 ? (f & ~7) + (j < 4 ? 2 * j : 2 * (j - 4) + 1) : f;
        const int odd = lane >> 4;
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
            float g, u;
            wd_trade(v[e], v[e + 1], lane, g, u);
            if (up_first) { const float s = g; g = u; u = s; }
            const float y = g / (1.f + __expf(-g)) * u;
            if (e + odd >= live) continue;
            const int o = (n0 + e + odd) * F + at;
            if (f16) {
                const __half h = __float2half_rn(y);
                ohi[o] = __half_as_ushort(h);
                olo[o] = __half_as_ushort(__float2half_rn(y - __half2float(h)));
            } else {
                const __nv_bfloat16 h = __float2bfloat16_rn(y);
                ohi[o] = __bfloat16_as_ushort(h);
                olo[o] = __bfloat16_as_ushort(__float2bfloat16_rn(y - __bfloat162float(h)));
            }
        }
    }
};
struct WdQkvEpi {  // tiles walk the concatenated [q heads | k heads | v heads] features; rotary + cache write
    int Hq, Hkv, dh;
    const float2 *rope_cs;
    float *q_out;
    KvAddr kv;
    int *dev_err;
    static constexpr bool kPaired = true;
    __device__ void locate(int ft, int quarter, int &which, int &head, int &i0) const {
        const int per = dh >> 5, feat0 = ft * kTcBM, qdim = Hq * dh, kvdim = Hkv * dh;
        which = feat0 < qdim ? 0 : (feat0 < qdim + kvdim ? 1 : 2);
        const int base = which == 0 ? feat0 : (which == 1 ? feat0 - qdim : feat0 - qdim - kvdim);
        head = base / dh + quarter / per;
        i0 = 16 * (quarter % per);
    }
    // the cache row (of dh values) of list row n0 + lane, -1: none
    __device__ int begin(float (&v)[32], int ft, int quarter, int lane, int live, int row) const {
        int which, head, i0, slot = -1;
        locate(ft, quarter, which, head, i0);
        if (which != 0 && lane < live) {
            const int page = kv.row_page[row];
            if (page < 0 || page >= kv.n_pages) atomicExch(dev_err, DEV_BAD_PAGE);
            else slot = (int)(kv.base(page, which - 1, head, kv.row_pos[row] % kPage) / dh);
        }
        wd_zero(v);
        return slot;
    }
    __device__ void run(float (&v)[32], int ft, int quarter, int lane, int live, int row, int slot, int) const {
        int which, head, i0;
        locate(ft, quarter, which, head, i0);
        const int half = dh >> 1, qdim = Hq * dh, i = i0 + (lane & 15), odd = lane >> 4;
#pragma unroll
        for (int e0 = 0; e0 < 32; e0 += 8) {
            float2 cs[4];
            int rw[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // the rotations of eight rows requested together
                rw[e] = __shfl_sync(0xffffffffu, row, e0 + 2 * e + odd);
                cs[e] = make_float2(1.f, 0.f);
                if (which != 2 && e0 + 2 * e + odd < live) cs[e] = rope_cs[rw[e] * half + i];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float lo, hi;
                wd_trade(v[e0 + 2 * e], v[e0 + 2 * e + 1], lane, lo, hi);
                const int at = __shfl_sync(0xffffffffu, slot, e0 + 2 * e + odd);
                if (e0 + 2 * e + odd >= live) continue;
                if (which != 2) {
                    const float a = lo * cs[e].x - hi * cs[e].y, b = hi * cs[e].x + lo * cs[e].y;
                    lo = a; hi = b;
                }
                if (which == 0) {
                    float *q = q_out + rw[e] * qdim + head * dh + i;
                    q[0] = lo;
                    q[half] = hi;
                } else if (at >= 0) {
                    __nv_bfloat16 *k = kv.pool + (size_t)at * dh + i;
                    k[0] = __float2bfloat16_rn(lo);
                    k[half] = __float2bfloat16_rn(hi);
                }
            }
        }
    }
};

struct TcWideArgs {
    int K;              // inner dimension (multiple of 64)
    int bn;             // rows per tile (multiple of 32, <= 256)
    int tiles;          // 128-feature tiles (an even number)
    int n_stages;
    int seg;            // k-blocks per accumulation segment
    int f16;            // operands are f16 (dequantised exit-layer weights), else bf16
    int q_tiles, k_tiles;     // QKV: tiles per matrix (0 otherwise)
    int run_step, head_step;  // paired maps (make_map_paired): how far a tile advances their outer coordinates
    const int32_t *rows;   // step row id of operand row n
    const int32_t *cnt;    // live operand rows (device)
    int *dev_err;
};

__device__ __forceinline__ uint32_t wd_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t wd_leader_addr(uint32_t saddr) {  // the same shared-memory offset in CTA 0 of the pair
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(saddr));
    return r;
}
// Copy into this CTA's shared memory; the bytes are counted on a barrier of the pair's leader.
__device__ __forceinline__ void wd_tma_load(uint32_t dst, const CUtensorMap *tmap, int x, int y, uint32_t leader_bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(leader_bar)
        : "memory");
}
__device__ __forceinline__ void wd_tma_load_5d(uint32_t dst, const CUtensorMap *tmap, int x, int run, int head, uint32_t leader_bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(tmap), "r"(x), "r"(0), "r"(run), "r"(head), "r"(leader_bar)
        : "memory");
}
__device__ __forceinline__ void wd_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void wd_commit(uint32_t bar) {  // one arrival on the barrier at this offset in BOTH CTAs
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void wd_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void wd_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <class Epi>
__global__ void __launch_bounds__(kWdThreads, 1) tc_gemm_wide_kernel(const __grid_constant__ CUtensorMap map_a0,
                                                                  const __grid_constant__ CUtensorMap map_a1,
                                                                  const __grid_constant__ CUtensorMap map_a2,
                                                                  const __grid_constant__ CUtensorMap map_bhi,
                                                                  const __grid_constant__ CUtensorMap map_blo,
                                                                  const TcWideArgs a, const Epi epi) {
    extern __shared__ uint8_t tc_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
    const int S = a.n_stages, bn = a.bn;
    const uint32_t b_bytes = (uint32_t)(bn / 2) * kTcBK * 2;       // a multiple of 2048
    const uint32_t stage_bytes = kWdABytes + 2 * b_bytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)S * stage_bytes);
    // full[S] (the leader's count), empty[S], acc_full[2], acc_empty[2] (the leader's count)
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * (uint32_t)S, accf0 = empty0 + 8 * (uint32_t)S, acce0 = accf0 + 16;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = wd_rank();
    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < S; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(accf0 + 8 * i, 1); mbar_init(acce0 + 8 * i, 2 * kWdEpiWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::);
        tc_fence_before();
        pdl_launch();  // (behind the allocation: see tc_gemm_kernel)
    }
    __syncthreads();
    wd_cluster_sync();  // the leader's barriers are ready before the other CTA's copies count on them
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int *abortp = &s_abort;
    pdl_wait();
    const int n_live = *a.cnt;
    const int n_tiles = (n_live + bn - 1) / bn, total = n_live > 0 ? (a.tiles / 2) * n_tiles : 0;
    const int pair0 = blockIdx.x >> 1, pairs = gridDim.x >> 1, nkb = a.K / kTcBK;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t s = 0, par = 1;  // (a fresh barrier: the wait for parity 1 returns at once)
            const uint32_t stage0 = smem_u32(smem), leader_full0 = wd_leader_addr(full0);
            int used = 0;
            bool ok = true;
            for (int t = pair0; t < total && ok; t += pairs) {
                const int ft = 2 * (t / n_tiles) + (int)rank, by = (t % n_tiles) * bn + (int)rank * (bn / 2);
                // where this CTA's weight rows live
                const CUtensorMap *ma = &map_a0;
                int at = ft;  // tile inside its matrix
                if (a.q_tiles) {
                    if (ft >= a.q_tiles + a.k_tiles) { ma = &map_a2; at = ft - a.q_tiles - a.k_tiles; }
                    else if (ft >= a.q_tiles) { ma = &map_a1; at = ft - a.q_tiles; }
                }
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(empty0 + 8 * s, par, abortp, a.dev_err)) { ok = false; break; }
                    if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2 * stage_bytes);
                    const uint32_t dst = stage0 + s * stage_bytes, bar = leader_full0 + 8 * s;
                    const int x = kb * kTcBK;
                    if constexpr (Epi::kPaired) wd_tma_load_5d(dst, ma, x, at * a.run_step, at * a.head_step, bar);
                    else wd_tma_load(dst, ma, x, at * kTcBM, bar);
                    wd_tma_load(dst + kWdABytes, &map_bhi, x, by, bar);
                    wd_tma_load(dst + kWdABytes + b_bytes, &map_blo, x, by, bar);
                    if (used < S) ++used;
                    if (++s == (uint32_t)S) { s = 0; par ^= 1u; }
                }
            }
            // every stage handed back before the CTA may end: no copy and no commit is still under way to it
            if (used < S) { s = 0; par = 0; }
            for (int i = 0; i < used && ok; ++i) {
                if (!mbar_wait(empty0 + 8 * s, par, abortp, a.dev_err)) ok = false;
                if (++s == (uint32_t)S) { s = 0; par ^= 1u; }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // D fp32, A and B both bf16 or both f16, K-major, M = 256 over the pair, N = bn
            const uint32_t idesc = (1u << 4) | (a.f16 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(bn >> 3) << 17) | (16u << 24);
            const uint64_t dfix = tc_smem_desc(0);
            const uint32_t stage16 = stage_bytes >> 4, b16 = b_bytes >> 4, first16 = smem_u32(smem) >> 4;
            uint32_t s = 0, par = 0, addr16 = first16;
            int j = 0;  // segments so far: they alternate between the two accumulators
            bool ok = true;
            for (int t = pair0; t < total && ok; t += pairs)
                for (int kb0 = 0; kb0 < nkb && ok; kb0 += a.seg, ++j) {
                    const uint32_t buf = j & 1;
                    if (!mbar_wait(acce0 + 8 * buf, ((j >> 1) & 1) ^ 1, abortp, a.dev_err)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d = tmem + buf * 256;
                    const int kb1 = min(kb0 + a.seg, nkb);
                    for (int kb = kb0; kb < kb1; ++kb) {
                        if (!mbar_wait(full0 + 8 * s, par, abortp, a.dev_err)) { ok = false; break; }
                        tc_fence_after();
                        const uint64_t da = dfix | addr16, dhi = da + (kWdABytes >> 4), dlo = dhi + b16;
#pragma unroll
                        for (int k = 0; k < kTcBK / 16; ++k) {
                            wd_mma(d, da + 2 * k, dhi + 2 * k, idesc, (kb != kb0 || k) ? 1u : 0u);
                            wd_mma(d, da + 2 * k, dlo + 2 * k, idesc, 1u);
                        }
                        wd_commit(empty0 + 8 * s);
                        if (++s == (uint32_t)S) { s = 0; par ^= 1u; addr16 = first16; } else addr16 += stage16;
                    }
                    wd_commit(accf0 + 8 * buf);
                }
        }
    } else {
        const int q = warp & 3, group = (warp - 2) >> 2;
        const uint32_t leader_acce0 = wd_leader_addr(acce0), lane0 = tmem + ((uint32_t)(q * 32) << 16);
        int j = 0;
        bool quit = false;
        for (int t = pair0; t < total && !quit; t += pairs) {
            const int ft = 2 * (t / n_tiles) + (int)rank, n0 = (t % n_tiles) * bn, live = min(bn, n_live - n0);
            float acc[kWdOwn][kWdChunk];  // this warp's chunks: columns 32 (group + 4 i)
            int row[kWdOwn], note[kWdOwn];  // what the epilogue reads elsewhere is requested now, under the MMAs
#pragma unroll
            for (int i = 0; i < kWdOwn; ++i) {
                const int c = kWdChunk * (group + kWdGroups * i);
                row[i] = c + lane < live ? a.rows[n0 + c + lane] : 0;
                note[i] = epi.begin(acc[i], ft, q, lane, min(kWdChunk, live - c), row[i]);
            }
#pragma unroll 1
            for (int kb0 = 0; kb0 < nkb; kb0 += a.seg, ++j) {
                const uint32_t buf = j & 1;
                const bool ok = mbar_wait_sleepy(accf0 + 8 * buf, (j >> 1) & 1, abortp, a.dev_err);
                if (!__all_sync(0xffffffffu, ok)) { quit = true; break; }
                tc_fence_after();
#pragma unroll
                for (int i = 0; i < kWdOwn; ++i) {
                    const int c = kWdChunk * (group + kWdGroups * i);
                    if (c < live) {
#pragma unroll
                        for (int h = 0; h < kWdChunk; h += 8) {
                            float v[8];
                            wd_ld8(lane0 + buf * 256 + (uint32_t)(c + h), v);
#pragma unroll
                            for (int e = 0; e < 8; ++e) acc[i][h + e] += v[e];
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(leader_acce0 + 8 * buf) : "memory");
            }
            if (quit) break;
#pragma unroll
            for (int i = 0; i < kWdOwn; ++i) {
                const int c = kWdChunk * (group + kWdGroups * i);
                if (c < live) epi.run(acc[i], ft, q, lane, min(kWdChunk, live - c), row[i], note[i], n0 + c);
            }
        }
    }
    __syncwarp();
    if (*abortp) {  // a wait ran out: what this CTA has asked for lands within microseconds; do not leave before
        for (int i = 0; i < 64; ++i) __nanosleep(4000);
    }
    tc_fence_before();
    __syncthreads();
    wd_cluster_sync();  // both CTAs are done with each other's shared and tensor memory
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

inline size_t tc_wide_smem_bytes(int bn, int n_stages) {
    return 1024 + (size_t)n_stages * (kWdABytes + (size_t)bn * kTcBK * 2) + sizeof(uint64_t) * (2 * n_stages + 4);
}

}  // namespace river
