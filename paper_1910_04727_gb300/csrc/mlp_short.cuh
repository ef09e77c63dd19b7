// GELU and the inverse normal of the surrogate network's BF16 activations and inputs by
// short approximations with the bits of the full functions.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace fm {

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
// bf16(gelu_f(z)) of two values, packed (z0 in the low half): the same bits as
// rounding gelu_f, at half its instructions.  1 + erf(z / sqrt 2) to about 2e-7
// by Hastings' rational form (Abramowitz & Stegun 7.1.26), g = max(z, 0) - |z| E
// / 2; where g - d and g + d, d = 4e-7 |z| (both sides' errors), round to the same
// BF16 number, gelu_f rounds to it too; else (a few pairs in ten thousand), and
// beyond |z| = 64 and for NaN, gelu_f itself.  tests/test_gpu_short_functions.py
// compares the two over all 2^32 FP32 numbers.
__device__ __forceinline__ float gelu_fast(float z, float az) {
    float t, e;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(az, 0.3275911f * 0.70710678f, 1.0f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z * z * (-0.5f * 1.44269504f)));
    float q = fmaf(t, 0.5f * 1.061405429f, 0.5f * -1.453152027f);
    q = fmaf(q, t, 0.5f * 1.421413741f);
    q = fmaf(q, t, 0.5f * -0.284496736f);
    q = fmaf(q, t, 0.5f * 0.254829592f);
    return fmaf(-az, q * t * e, fmaxf(z, -0.0f));   // -0.0f: keeps the sign of a zero
}
__device__ __forceinline__ uint32_t bf16x2_bits(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __noinline__ uint32_t gelu_bf16x2_slow(float z0, float z1) { return bf16x2_bits(gelu_f(z0), gelu_f(z1)); }
__device__ __forceinline__ uint32_t gelu_bf16x2(float z0, float z1) {
    const float a0 = fabsf(z0), a1 = fabsf(z1);
    const float g0 = gelu_fast(z0, a0), g1 = gelu_fast(z1, a1);
    constexpr float d = 4e-7f;
    const uint32_t up = bf16x2_bits(fmaf(a0, d, g0), fmaf(a1, d, g1));
    const uint32_t dn = bf16x2_bits(fmaf(a0, -d, g0), fmaf(a1, -d, g1));
    if (up == dn && a0 < 64.0f && a1 < 64.0f) return up;
    return gelu_bf16x2_slow(z0, z1);   // a call: inlined at every use, it made the epilogues outgrow the instruction cache
}

// bf16(Phi^-1(u)) of two MC input words, packed: u = (k + 1/2) 2^-23, k < 2^23 the
// top bits of a Philox word, the same bits as rounding normcdfinvf(u), at half
// its instructions.  Phi^-1(u) = (2u - 1) f(t), t = -log2(4 u (1 - u)), f a
// polynomial of degree 8 fitted for t <= 7 (2e-7 relative); u and 1 - u are exact.
// Where r (1 - d) and r (1 + d), d = 1e-6, round to the same BF16 number,
// normcdfinvf rounds to it too; else, and in the tails (0.4% of the words),
// normcdfinvf itself.  tests/test_gpu_short_functions.py compares the two over all 2^23
// words.
__device__ __forceinline__ float word_uniform(uint32_t k) { return ((float)k + 0.5f) * 0x1p-23f; }
__device__ __noinline__ uint32_t normal_bf16x2_slow(uint32_t k0, uint32_t k1) {
    return bf16x2_bits(normcdfinvf(word_uniform(k0)), normcdfinvf(word_uniform(k1)));
}
__device__ __forceinline__ float normal_fast(uint32_t k, float* t) {
    const float x = (float)k;
    const float u = fmaf(x, 0x1p-23f, 0x1p-24f), v = fmaf(x, -0x1p-23f, 1.0f - 0x1p-24f);
    float l;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(4.0f * u * v));
    *t = -l;
    const float s = -3.5f - l;
    float q = fmaf(s, 2.547130506513895e-09f, 3.641305568180542e-08f);
    q = fmaf(q, s, -5.891061505280959e-07f);
    q = fmaf(q, s, -6.486233132818597e-07f);
    q = fmaf(q, s, 7.1850219683256e-05f);
    q = fmaf(q, s, -0.0006209334242157638f);
    q = fmaf(q, s, -0.002644734922796488f);
    q = fmaf(q, s, 0.24235691130161285f);
    q = fmaf(q, s, 2.09747576713562f);
    return q * (u - v);
}
__device__ __forceinline__ uint32_t normal_bf16x2(uint32_t k0, uint32_t k1) {
    float t0, t1;
    const float r0 = normal_fast(k0, &t0), r1 = normal_fast(k1, &t1);
    constexpr float d = 1e-6f;
    const uint32_t up = bf16x2_bits(r0 * (1.0f + d), r1 * (1.0f + d));
    const uint32_t dn = bf16x2_bits(r0 * (1.0f - d), r1 * (1.0f - d));
    if (up == dn && t0 < 7.0f && t1 < 7.0f) return up;
    return normal_bf16x2_slow(k0, k1);
}
}  // namespace fm
