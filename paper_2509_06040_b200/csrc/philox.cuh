// Counter-based Gaussian noise on the device: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11)
// and a float32 Box-Muller transform.  The stream definition (key, counter words, tags, uniform
// map, pairing) is the one stated at the top of bgrpo.h.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"

namespace bgrpo {

__device__ __forceinline__ void mulhilo(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
    uint64_t p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(p));
}

// Ten rounds; one round sends (c0,c1,c2,c3) to (hi(M1*c2)^c1^k0, lo(M1*c2), hi(M0*c0)^c3^k1, lo(M0*c0))
// and the key advances by the Weyl constants between rounds (the host has tabulated the ten keys).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const PhiloxKeys& keys) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0, lo0, hi1, lo1;
        mulhilo(kPhiloxM0, c.x, hi0, lo0);
        mulhilo(kPhiloxM1, c.z, hi1, lo1);
        c = make_uint4(hi1 ^ c.y ^ keys.k[r][0], lo1, hi0 ^ c.w ^ keys.k[r][1], lo0);
    }
    return c;
}

// Hardware special-function approximations (flush-to-zero forms: one MUFU each, no denormal fix-up code).
__device__ __forceinline__ float fast_sqrt(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_log2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_sin(float x) {
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float fast_cos(float x) {
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two float32 operations in one instruction (the same rounding as the two single ones).
__device__ __forceinline__ float2 mul2(float a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %2};\n\tmov.b64 y, {%3, %4};\n\tmul.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %2};\n\tmov.b64 y, {%3, %4};\n\tmov.b64 z, {%5, %6};\n\tfma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float4 mul4(float a, const float4& b) {
    const float2 lo = mul2(a, make_float2(b.x, b.y)), hi = mul2(a, make_float2(b.z, b.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float4 fma4(float a, const float4& b, const float4& c) {
    const float2 lo = fma2(a, make_float2(b.x, b.y), make_float2(c.x, c.y)), hi = fma2(a, make_float2(b.z, b.w), make_float2(c.z, c.w));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The float in [1, 2) whose mantissa is the word's top 23 bits: one funnel shift, (0x7f : x) >> 9 = 0x3f800000 | x >> 9.
__device__ __forceinline__ float one_to_two(uint32_t x) { return __uint_as_float(__funnelshift_r(x, 0x7fu, 9)); }

// One Box-Muller pair from two words: (r cos 2 pi u_b, r sin 2 pi u_b), r = sqrt(-2 ln u_a).  r2 receives r^2, the pair's
// sum of squares.
//
// Accuracy (the result must stay within ~1e-4 of the exact value so that g * xi, g ~ 0.1, moves a
// latent by well under 1e-5):
//  * -2 ln u_a comes from the hardware log2 (absolute error 2^-22 for arguments in (0.5, 2), relative
//    2^-22 elsewhere).  An absolute error in r^2 becomes a large relative error in r only when r is tiny,
//    i.e. u_a within 2^-9 of 1; there w = 1 - u_a is exact in float32 and the series
//    -2 ln(1 - w) = 2w + w^2 + ... (truncation below 1.3e-6 relative) replaces the log.
//  * the angle is folded to (-pi, pi), where the hardware sine/cosine are good to about 4e-7 absolute,
//    and the sign change is absorbed into r.
__device__ __forceinline__ float2 box_muller(uint32_t wa, uint32_t wb, float& r2) {
    const float ua = one_to_two(wa) - 0.99999994f;             // ((x >> 9) + 0.5) * 2^-23, exact
    const float w = 1.0f - ua;
    const float series = fmaf(w, w, w + w);
    const float viaLog = -1.3862944f * fast_log2(ua);          // -2 ln 2 * log2(u)
    r2 = (w < 0.001953125f) ? series : viaLog;
    const float nr = -fast_sqrt(r2);
    // 2 pi u_b - pi with u_b = m - (1 - 2^-24), m in [1, 2) the float built from the word's top 23 bits: the constant
    // term takes the subtraction in (its float32 rounding moves the angle by < 5e-7, i.e. xi by < 3e-6)
    const float th = fmaf(one_to_two(wb), 6.2831855f, -9.4247776f);
    return mul2(nr, make_float2(fast_cos(th), fast_sin(th)));
}

// Four normals and their sum of squares.
__device__ __forceinline__ float4 normal4(uint4 w, float& squares) {
    float ra, rb;
    const float2 a = box_muller(w.x, w.y, ra);
    const float2 b = box_muller(w.z, w.w, rb);
    squares = ra + rb;
    return make_float4(a.x, a.y, b.x, b.y);
}

// The first two Philox rounds split into what depends on (element block, tag) only and on (node, step) only: the first
// part is kept by a thread that draws the same elements for many nodes, the second is the same for a whole warp (uniform
// registers).  philox_from() goes on with round 3; the words are those of philox4x32_10.
struct NoiseElement { uint32_t x, y, z; };
struct NoiseNode { uint32_t x, z, w; };
__device__ __forceinline__ NoiseElement noise_element(uint32_t block, uint32_t tag, const PhiloxKeys& keys) {
    uint32_t hi0, lo0, hi1, lo1;
    mulhilo(kPhiloxM0, block, hi0, lo0);
    mulhilo(kPhiloxM1, hi0 ^ tag ^ keys.k[0][1], hi1, lo1);
    return {hi1, lo1, lo0};
}
__device__ __forceinline__ NoiseNode noise_node(uint32_t node, uint32_t step, const PhiloxKeys& keys) {
    uint32_t hi1, lo1, hi0, lo0;
    mulhilo(kPhiloxM1, step, hi1, lo1);
    mulhilo(kPhiloxM0, hi1 ^ node ^ keys.k[0][0], hi0, lo0);
    return {lo1 ^ keys.k[1][0], hi0 ^ keys.k[1][1], lo0};
}
// The part of a NoiseNode that all nodes of a step share, for the host to tabulate: px = lo(M1 step) ^ k[1][0],
// ph = hi(M1 step) ^ k[0][0].
inline void noise_step(uint32_t step, const PhiloxKeys& keys, uint32_t& px, uint32_t& ph) {
    const uint64_t prod = static_cast<uint64_t>(kPhiloxM1) * step;
    px = static_cast<uint32_t>(prod) ^ keys.k[1][0];
    ph = static_cast<uint32_t>(prod >> 32) ^ keys.k[0][0];
}
__device__ __forceinline__ NoiseNode noise_node_of(uint32_t node, uint32_t px, uint32_t ph, const PhiloxKeys& keys) {
    uint32_t hi0, lo0;
    mulhilo(kPhiloxM0, ph ^ node, hi0, lo0);
    return {px, hi0 ^ keys.k[1][1], lo0};
}
__device__ __forceinline__ uint4 philox_from(const NoiseElement& e, const NoiseNode& n, const PhiloxKeys& keys) {
    uint4 c = make_uint4(e.x ^ n.x, e.y, e.z ^ n.z, n.w);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        uint32_t hi0, lo0, hi1, lo1;
        mulhilo(kPhiloxM0, c.x, hi0, lo0);
        mulhilo(kPhiloxM1, c.z, hi1, lo1);
        c = make_uint4(hi1 ^ c.y ^ keys.k[r][0], lo1, hi0 ^ c.w ^ keys.k[r][1], lo0);
    }
    return c;
}

// Log-prob sums of the rollout kernels.  The squares of four normals (at most 2 * 33.3 with independent noise, twice that
// with a shared part) are rounded to a multiple of 2^-18 - 2e-6 of their mean, the rounding of a float32 log-prob of four
// elements - and added as integers: sums are exact from there on, so they do not depend on how a kernel cuts the row, and
// the level-by-level and the whole-tree kernel agree bit for bit.  A thread may add up to 30 of them in 32 bits; what a
// warp adds is bounded where it is added.
constexpr float kSquareScale = 262144.0f;
constexpr double kMostSquares = 66.6;          // of four normals: two r^2 = -2 ln u of u >= 2^-24; twice that with a shared part
__device__ __forceinline__ uint32_t quantized_squares(float squares) { return __float2uint_rn(squares * kSquareScale); }
__device__ __forceinline__ float squares_of(const float4& x) { return fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, x.w * x.w))); }
// the log-prob of an edge from its row's sum: -(1/D) sum (z' - mean)^2 / (2 g^2) + const with (z' - mean)^2 = g^2 xi^2
// (half_per: 0.5 / (kSquareScale D), from the host: a double division takes longer than the rest of the sum)
inline double logp_half_per(int64_t D) { return 0.5 / static_cast<double>(kSquareScale) / static_cast<double>(D); }
__device__ __forceinline__ float logp_from_squares(unsigned long long sum, double half_per, float g, float logp_const) {
    return g == 0.0f ? 0.0f : static_cast<float>(static_cast<double>(logp_const) - static_cast<double>(sum) * half_per);
}
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return x;
}

// Adds up a row of the pending level: THREADS threads of a CTA, `t` the thread's number among them; thread 0 writes.
// s_sum: the CTA's, when more than a warp works on the row (all of the CTA then gets here).
template <int THREADS>
__device__ __forceinline__ void finalize_row(const FinalizeDesc& f, int64_t row, double half_per, int t, unsigned long long* s_sum) {
    unsigned long long* q = f.sums + row * f.stride;
    unsigned long long s = 0;
#pragma unroll 8
    for (int c = t; c < f.per_row; c += THREADS) s += __ldcg(q + c);
    if (f.clear)
        for (int c = t; c < f.per_row; c += THREADS) q[c] = 0ull;
    s = warp_sum_u64(s);
    if (THREADS > 32) {
        if ((t & 31) == 0) s_sum[t >> 5] = s;
        __syncthreads();
        if (t == 0)
            for (int w = 1; w < THREADS / 32; ++w) s += s_sum[w];
    }
    if (t == 0) f.logp_out[row] = logp_from_squares(s, half_per, f.g, f.logp_const);
}

// All rows of the pending level: one warp per row, or one lane where a row's sum is one number (added with atomics, and cleared
// for the next who adds).
__device__ __forceinline__ void finalize_rows(const FinalizeDesc& f, int32_t n_trees, int32_t nodes_cap,
                                              double half_per, int warp_global, int warps_total, int32_t* status, int32_t per_row_cap) {
    const int n_rows = n_trees * f.W;
    if (f.clear) {
        for (int idx = warp_global + (threadIdx.x & 31) * warps_total; idx < n_rows; idx += 32 * warps_total) {      // spread over the warps first
            const int tree = idx / f.W;
            const int64_t row = static_cast<int64_t>(tree) * nodes_cap + f.off + (idx - tree * f.W);
            if (!BGRPO_IN_BOUNDS(status, f.off + f.W <= nodes_cap && f.per_row == 1 && f.stride == 1)) continue;
            f.logp_out[row] = logp_from_squares(__ldcg(f.sums + row), half_per, f.g, f.logp_const);
            f.sums[row] = 0ull;
        }
        return;
    }
    for (int idx = warp_global; idx < n_rows; idx += warps_total) {
        const int tree = idx / f.W;
        const int64_t row = static_cast<int64_t>(tree) * nodes_cap + f.off + (idx - tree * f.W);
        if (!BGRPO_IN_BOUNDS(status, f.off + f.W <= nodes_cap && 2 * f.per_row <= per_row_cap)) continue;
        finalize_row<32>(f, row, half_per, threadIdx.x & 31, nullptr);
    }
}

__device__ __forceinline__ float4 noise4(uint32_t block, uint32_t node, uint32_t step, uint32_t tag,
                                         const PhiloxKeys& keys) {
    float squares;
    return normal4(philox4x32_10(make_uint4(block, node, step, tag), keys), squares);
}

}  // namespace bgrpo
