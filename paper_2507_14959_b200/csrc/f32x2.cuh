// Packed fp32 arithmetic and the GELU of the GEMM epilogues.
#pragma once

#include "common.cuh"

namespace {

// Exact-erf GELU x * Phi(x), evaluated in logistic form: Phi(x) = 1 / (1 + exp(-2 x p(x^2))) holds
// exactly for p = atanh(erf(x / sqrt 2)) / x, which a quadratic in x^2 fits well enough that
//   | x (1/2 + 1/2 tanh(x q(x^2))) - gelu(x) | < 2.6e-5   for all x     (q = p: 1 / (1 + e^-2u) = 1/2 + 1/2 tanh u),
// far below the bf16 rounding of the stored result except where the result itself is below 1e-2; the
// hardware tanh (tanh.approx.f32, relative error about 2^-11) adds less than a quarter of a bf16 step.
// The epilogue warps share their issue slots with the thread that issues the MMAs, so every
// instruction saved here counts: the arithmetic runs on pairs (packed fp32) and costs one special-function
// instruction per element (the form x / (1 + 2^(x q)) it replaces needed an exponential and a
// reciprocal: fused GEMMs 2.3 % slower in the bench step).

// Two fp32 values in one 64-bit register, for the packed fp32 arithmetic of sm_100 (one issue slot
// for two results; each half is the ordinary IEEE operation).
__device__ __forceinline__ uint64_t pk2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t r, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// the GELU described above, on a pair
__device__ __forceinline__ uint64_t gelu_erf2(uint64_t v) {
    // v^2 is capped where Phi has long saturated (the fitted q turns over beyond |v| = 7.2)
    float t0, t1;
    upk2(mul2(v, v), t0, t1);
    const uint64_t t = pk2(fminf(t0, 50.f), fminf(t1, 50.f));
    uint64_t q = fma2(t, pk2(-3.5151945e-04f, -3.5151945e-04f), pk2(3.7005664e-02f, 3.7005664e-02f));
    q = fma2(q, t, pk2(0.79750784f, 0.79750784f));
    float w0, w1, h0, h1;
    upk2(mul2(v, q), w0, w1);
    asm("tanh.approx.f32 %0, %1;" : "=f"(h0) : "f"(w0));
    asm("tanh.approx.f32 %0, %1;" : "=f"(h1) : "f"(w1));
    return mul2(v, fma2(pk2(h0, h1), pk2(0.5f, 0.5f), pk2(0.5f, 0.5f)));
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

}  // namespace
