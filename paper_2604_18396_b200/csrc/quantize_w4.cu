// river_quantize_w4: the exit layers' weights from the backbone's, on the GPU (sm_100a).
//
// River-LLM builds an exit layer by copying a backbone block and quantising its Attention and FFN matrices with a
// training-free 4-bit weight-only method, HQQ (paper Section 4.1).  One thread owns one group of `group` inputs of a
// weight row: the scale comes from the group's range ((max - min) / 15, stored as bf16); the zero-point starts at
// -min / s and is refined by HQQ's half-quadratic iteration - quantise, shrink the residual with the generalised soft
// threshold of an l_p norm (p = 0.7), re-solve the zero-point in closed form as the group mean of W_q - (W - W_e) / s,
// beta growing by 1.01 per round - and is stored as bf16; the codes are then taken against the stored scale and zero,
// so that (q - z) s is the best the stored triple can give.  refine_iters = 0 leaves the plain min/max grid.
// Every arithmetic step is a single fp32 operation in a fixed order (no fused multiply-add, sums sequential over the
// group), because it decides integers: a reference that follows the same order reproduces the codes bit for bit.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "../../include/river.h"

namespace {

constexpr int kMaxGroup = 128;

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Two fp32 operations in one instruction, each rounded as the single ones are.
struct F2 { float x, y; };
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ F2 unpack2(unsigned long long v) {
    F2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long v;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}

// The residual below which the soft threshold leaves nothing, (1 / beta)^(1 / 1.3), less 1 %: beta is 10 in the first round and
// grows by 1.01.  (A thousand single products are off by less than 1e-4 of it.)
constexpr float kThreshold0 = 0.99f * 0.170125f, kThresholdStep = 0.9923751f;

// One refinement round over a thread's group: the sum of q - (x - w_e) / s in the group's order, d = x / s.
// The general form, with the soft threshold (which wants the weights themselves: read again, so that a group's registers need
// not hold them beside d through the rounds that do without).
template <int G>
__device__ __forceinline__ float refine_sum_general(const uint32_t *x2, const unsigned long long (&d)[G / 2], float s, float z, float inv_beta) {
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const F2 dd = unpack2(d[i / 2]);
        const uint32_t xw = x2[i / 2];
        const float x = __uint_as_float((i & 1) ? (xw & 0xffff0000u) : (xw << 16));
        const float q = fminf(fmaxf(rintf(__fadd_rn((i & 1) ? dd.y : dd.x, z)), 0.f), 15.f);
        const float e = __fsub_rn(x, __fmul_rn(__fsub_rn(q, z), s));
        const float ae = fabsf(e);
        float we = 0.f;
        if (ae > 0.f) {
            const float t = __fsub_rn(ae, __fmul_rn(inv_beta, powf(ae, 0.7f - 1.0f)));
            we = copysignf(fmaxf(t, 0.f), e);
        }
        sum = __fadd_rn(sum, __fsub_rn(q, __fdiv_rn(__fsub_rn(x, we), s)));
    }
    return sum;
}
// The same where the threshold is known to be zero everywhere; CLAMP: some code may need clamping to [0, 15].
template <int G, bool CLAMP>
__device__ __forceinline__ float refine_sum_plain(const unsigned long long (&d)[G / 2], float z) {
    // adding and subtracting 1.5 * 2^23 rounds a value of a few units to the nearest even integer, as rintf does
    const unsigned long long z2 = pack2(z, z), up = pack2(12582912.f, 12582912.f), down = pack2(-12582912.f, -12582912.f);
    const unsigned long long neg = pack2(-1.f, -1.f);
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < G / 2; ++i) {
        unsigned long long r = add2(d[i], z2);
        if constexpr (CLAMP) {
            const F2 c = unpack2(r);
            r = pack2(fminf(fmaxf(c.x, 0.f), 15.f), fminf(fmaxf(c.y, 0.f), 15.f));
        }
        const F2 t = unpack2(fma2(d[i], neg, add2(add2(r, up), down)));  // q - d, rounded once
        sum = __fadd_rn(__fadd_rn(sum, t.x), t.y);
    }
    return sum;
}

// What bounds it: arithmetic (2.56 bytes per weight cross HBM once, every round touches every weight in registers).  The
// general round costs a power, two divisions and a dozen other operations per weight; two facts, tested once per group and
// round, take nearly all of it away without changing a bit:
//   * the soft threshold max(|e| - |e|^(p - 1) / beta, 0) is zero wherever |e|^1.3 < 1 / beta, i.e. |e| < 0.15-0.17 in the
//     published 20 rounds, while |e| is at most half a step for every weight inside the grid - and a weight outside it is
//     off by how far the group's smallest or largest weight lies outside.  The bound below adds 1e-6 of the operands for
//     the roundings of the 32-bit operations (each is below 2^-23 of them) and keeps 1 % from the threshold.
//   * with w_e = 0 the second division is x / s, the same in every round: taken once.
//   * when the group's own range needs no clamp, neither does any of its weights (adding z is monotonic).
//   * a round that gives back the zero-point it started from, bit for bit, is what every round behind it would do too - as
//     long as the threshold, which only falls with the rounds, is zero for this group in the last one as well: done.  Of the
//     20 rounds on normally distributed weights a group of 64 takes 4.2 so, the slowest of a warp's 32 groups 11.2.
// What is left are four packed additions per pair and the sum, whose order the bits depend on.
// Measured on 4096 x 14336, 64 inputs per group, 20 rounds: 5488 us with the general round everywhere, 295 us
// with every round taken, 222 us with the rounds that change something - 8 us a round and 130 us around them, spent on the quotients
// x / s, a power per round for the threshold, and the codes' rounding and conversion (16 a clock each): 142 us with the quotients
// from the reciprocal, the threshold carried along and the codes rounded by an addition; 140 with the range taken over pairs of bf16
// values (128 inputs per group 207 -> 193).  The FMA pipe is 75 % busy then.  Dealing a CTA's groups that still move out over its
// threads, after 3 and 6 rounds or after 6, left 40 % of the rounds away and won nothing (140 and 137; 32 and 128 inputs slower): at 4
// CTAs per SM the warps that wait at its barriers are missing beside the others' chains of additions.
// Weights whose half step lies above the threshold (scales of 0.3 and more) go through general rounds only, and those read the
// weights again: 4096 x 4096, standard deviation 4, groups of 32, 64 and 128, 1.30, 1.56 and 3.3 ms (64: 1.84 before the
// range was taken over pairs, which left registers for a fifth CTA per SM).
template <int G>
__global__ void __launch_bounds__(128) quantize_w4_kernel(const __nv_bfloat16 *w, long long n_groups, int refine_iters, float last_threshold,
                                                          uint8_t *codes, __nv_bfloat16 *scale, __nv_bfloat16 *zero) {
    const long long gi = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= n_groups) return;
    uint32_t xp[G / 2];  // the group's bf16 weights, two per register
    const uint4 *src = reinterpret_cast<const uint4 *>(w + gi * G);
#pragma unroll
    for (int i = 0; i < G / 8; ++i) {
        const uint4 v = src[i];
        xp[4 * i] = v.x; xp[4 * i + 1] = v.y; xp[4 * i + 2] = v.z; xp[4 * i + 3] = v.w;
    }
    auto x_at = [&](int i) { return __uint_as_float((i & 1) ? (xp[i / 2] & 0xffff0000u) : (xp[i / 2] << 16)); };
    float mn, mx;
    if constexpr (G >= 64) {  // two at a time (at 32 the compiler then keeps more registers, and general rounds lose 4 %)
        auto pair_at = [&](int i) { return *reinterpret_cast<const __nv_bfloat162 *>(&xp[i]); };
        __nv_bfloat162 mn2 = pair_at(0), mx2 = mn2;
#pragma unroll
        for (int i = 1; i < G / 2; ++i) { mn2 = __hmin2(mn2, pair_at(i)); mx2 = __hmax2(mx2, pair_at(i)); }
        mn = fminf(__low2float(mn2), __high2float(mn2));
        mx = fmaxf(__low2float(mx2), __high2float(mx2));
    } else {
        mn = mx = x_at(0);
#pragma unroll
        for (int i = 1; i < G; ++i) { mn = fminf(mn, x_at(i)); mx = fmaxf(mx, x_at(i)); }
    }
    const bool constant = mx == mn;
    float s = bf16_round(__fdiv_rn(__fsub_rn(mx, mn), 15.0f));
    if (constant || s == 0.f) s = 1.f;
    float z = __fdiv_rn(-mn, s);
    unsigned long long d[G / 2];
    // x / s, correctly rounded: with the reciprocal r = 1 / s correctly rounded, q = x r and the exact remainder x - q s, the sum
    // q + (x - q s) r is (Markstein, IBM J. Res. Dev. 34, 1990; true of every pair of 8-bit mantissas) - as long as the remainder
    // does not underflow: every weight of the group zero or at least 2^-60 in magnitude, s and the weights at most 2^60.
    uint32_t tiny = 0u;  // bit 15 of a half: a weight that is neither
#pragma unroll
    for (int i = 0; i < G / 2; ++i) {
        const uint32_t u = xp[i] & 0x7fff7fffu;
        tiny |= (u + 0x7fff7fffu) & ~(u + 0x5e805e80u);  // (0x8000 - 0x2180, the exponent of 2^-60)
    }
    if ((tiny & 0x80008000u) == 0u && s >= 0x1p-60f && s <= 0x1p60f && fmaxf(fabsf(mn), fabsf(mx)) <= 0x1p60f) {
        const float r = __frcp_rn(s);
        const unsigned long long r2 = pack2(r, r), s2 = pack2(-s, -s);
#pragma unroll
        for (int i = 0; i < G / 2; ++i) {
            const unsigned long long x = pack2(x_at(2 * i), x_at(2 * i + 1)), q = mul2(x, r2);
            d[i] = fma2(fma2(q, s2, x), r2, q);
        }
    } else {
#pragma unroll
        for (int i = 0; i < G / 2; ++i) d[i] = pack2(__fdiv_rn(x_at(2 * i), s), __fdiv_rn(x_at(2 * i + 1), s));
    }
    const float dmin = __fdiv_rn(mn, s), dmax = __fdiv_rn(mx, s);  // rounding is monotonic: every d lies between them
    const float xabs = fmaxf(fabsf(mn), fabsf(mx));
    float beta = 10.0f, threshold = kThreshold0;
    for (int it = 0; it < refine_iters; ++it) {
        const float lo = dmin + z, hi = dmax + z;  // the group's range on the code grid
        const float off = fmaxf(0.5f, fmaxf(-lo, hi - 15.f));
        const float bound = s * off + 1e-6f * (xabs + (15.f + fabsf(z)) * s);
        float sum;
        if (!(bound < threshold)) sum = refine_sum_general<G>(reinterpret_cast<const uint32_t *>(src), d, s, z, __fdiv_rn(1.0f, beta));  // (NaN too)
        else if (lo >= -0.5f && hi < 15.5f) sum = refine_sum_plain<G, false>(d, z);
        else sum = refine_sum_plain<G, true>(d, z);
        const float before = z;
        z = __fmul_rn(sum, 1.0f / (float)G);  // (a power of two)
        if (__float_as_uint(z) == __float_as_uint(before) && bound < last_threshold) break;
        beta = __fmul_rn(beta, 1.01f);
        threshold *= kThresholdStep;
    }
    float zb = bf16_round(z);
    if (constant) zb = bf16_round(-mn);
    const unsigned long long zb2 = pack2(zb, zb), up = pack2(12582912.f, 12582912.f);
    uint32_t packed[G / 8];
#pragma unroll
    for (int i = 0; i < G / 8; ++i) {
        uint32_t p = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // clamped, then rounded to the nearest even integer by adding 1.5 * 2^23, whose last bits are the code then
            const F2 v = unpack2(add2(d[4 * i + j], zb2));
            const F2 q = unpack2(add2(pack2(fminf(fmaxf(v.x, 0.f), 15.f), fminf(fmaxf(v.y, 0.f), 15.f)), up));
            p |= (__float_as_uint(q.x) & 15u) << (8 * j) | (__float_as_uint(q.y) & 15u) << (8 * j + 4);  // low nibble = even input
        }
        packed[i] = constant ? 0u : p;
    }
    uint4 *dst = reinterpret_cast<uint4 *>(codes + gi * (G / 2));
#pragma unroll
    for (int i = 0; i < G / 32; ++i) dst[i] = make_uint4(packed[4 * i], packed[4 * i + 1], packed[4 * i + 2], packed[4 * i + 3]);
    scale[gi] = __float2bfloat16_rn(s);
    zero[gi] = __float2bfloat16_rn(zb);
}

}  // namespace

extern "C" int river_quantize_w4(const void *w, int out, int in, int group, int refine_iters, void *codes, void *scale,
                                 void *zero, void *cuda_stream) {
    if (!w || !codes || !scale || !zero || out <= 0 || in <= 0 || refine_iters < 0 || refine_iters > 1000) return RIVER_E_BADARG;
    if (!(group == 32 || group == 64 || group == kMaxGroup) || in % group) return RIVER_E_SHAPE;
    if (((uintptr_t)w | (uintptr_t)codes) & 15) return RIVER_E_BADARG;  // whole groups in 16-byte loads and stores
    const long long n_groups = (long long)out * (in / group);
    const unsigned grid = (unsigned)((n_groups + 127) / 128);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    float last_threshold = kThreshold0;  // of the last round
    for (int i = 1; i < refine_iters; ++i) last_threshold *= kThresholdStep;
    const __nv_bfloat16 *wp = static_cast<const __nv_bfloat16 *>(w);
    uint8_t *cp = static_cast<uint8_t *>(codes);
    __nv_bfloat16 *sp = static_cast<__nv_bfloat16 *>(scale), *zp = static_cast<__nv_bfloat16 *>(zero);
    if (group == 32) quantize_w4_kernel<32><<<grid, 128, 0, st>>>(wp, n_groups, refine_iters, last_threshold, cp, sp, zp);
    else if (group == 64) quantize_w4_kernel<64><<<grid, 128, 0, st>>>(wp, n_groups, refine_iters, last_threshold, cp, sp, zp);
    else quantize_w4_kernel<128><<<grid, 128, 0, st>>>(wp, n_groups, refine_iters, last_threshold, cp, sp, zp);
    return cudaGetLastError() == cudaSuccess ? RIVER_OK : RIVER_E_DEVICE;
}
