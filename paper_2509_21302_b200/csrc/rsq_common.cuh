// Pieces of the exact rotate-smooth-quantize kernel (rsq.cu): butterflies, the statistics' summation tree, GELU, asynchronous copies.
#pragma once
#include "sm100_ptx.cuh"

namespace rsqc {

// (a0, a1) <- (a0 + b0, a1 + b1), (b0, b1) <- (a0 - b0, a1 - b1): two butterflies per instruction pair
__device__ __forceinline__ void bfly2(float &a0, float &a1, float &b0, float &b1)
{
    const uint64_t A = ptx::f32x2_pack(a0, a1), B = ptx::f32x2_pack(b0, b1);
    ptx::f32x2_unpack(ptx::f32x2_add(A, B), a0, a1);
    ptx::f32x2_unpack(ptx::f32x2_sub(A, B), b0, b1);
}

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_addr(smem_dst)), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Pairwise sum of N registers: adjacent pairs, recursively (the tree of the LayerNorm statistics).
template <int N>
__device__ __forceinline__ float tree_sum(const float (&a)[N])
{
    if constexpr (N == 1) {
        return a[0];
    } else {
        float b[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) b[i] = __fadd_rn(a[2 * i], a[2 * i + 1]);
        return tree_sum<N / 2>(b);
    }
}

// GELU x Phi(x) (the activation between the two linears of the MLP: the producer of fc2's input) of two bf16 values, rounded to
// bf16, evaluated so that the negative tail keeps its RELATIVE accuracy.  With t = |x|, z = t / sqrt(2):
//   Q(t) = 1 - Phi(t) = exp(-z^2) E(z) / 2,   E(z) = exp(z^2) erfc(z)  (smooth, from 1 down to ~1 / (z sqrt(pi))),
//   E(z) ~ s P(s),  s = 1 / (1 + 0.55 z),  P a degree-4 polynomial (own weighted least-squares fit on z in [0, 9.6]: relative
//   error below 6e-5), then gelu(x) = x - t Q for x >= 0 and -t Q for x < 0.
// At most one bf16 ulp wherever the result is a normal number above 2^-120; below that (x < -12.9) the exponential flushes to
// zero, with the sign of x.  NaN stays NaN, and an infinite x gives NaN (the product of infinity and a flushed tail).
// Everything but the two special-function operations of an element (reciprocal, exp2) runs on two elements per instruction; each of
// these operations rounds exactly like its scalar form, and no product feeds an addition that is not written as a fused one.  The fused
// kernel is bound by instruction issue and, through the four special-function operations of a pair, by that unit; scalar / paired, us back
// to back: K = 1024 15.9 / 15.3 at 10 992 rows, 158 / 154 at 137 400; K = 4096 62.2 / 59.9, 714 / 678.  (A polynomial for log2 Q, with the
// exponential alone on the special-function unit, took 14.4, 145, 54.1, 624, but gave other bits.)
__device__ __forceinline__ uint32_t gelu_bf16x2(uint32_t x)
{
    const uint32_t a = x | 0x80008000u;                    // -t
    uint32_t pos;                                          // x, or -0 for x < 0; x = -0 counts as +0
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(pos) : "r"(x), "r"(0x3F803F80u), "r"(0u));
    asm("max.bf16x2 %0, %0, %1;" : "+r"(pos) : "r"(0x80008000u));
    const uint64_t nt = ptx::f32x2_pack(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u));
    auto both = [](float v) { return ptx::f32x2_pack(v, v); };
    const uint64_t z = ptx::f32x2_mul(nt, both(-0.70710678f));
    float d0, d1, s0, s1, w0, w1, e0, e1, y0, y1;
    ptx::f32x2_unpack(ptx::f32x2_fma(both(0.55f), z, both(1.0f)), d0, d1);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s0) : "f"(d0));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s1) : "f"(d1));
    const uint64_t s = ptx::f32x2_pack(s0, s1);
    uint64_t p = both(-0.17450283f);
    p = ptx::f32x2_fma(p, s, both(0.33387650f));
    p = ptx::f32x2_fma(p, s, both(0.21415194f));
    p = ptx::f32x2_fma(p, s, both(0.31633197f));
    p = ptx::f32x2_fma(p, s, both(0.31008677f));
    ptx::f32x2_unpack(ptx::f32x2_mul(ptx::f32x2_mul(z, z), both(-1.44269504f)), w0, w1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(w0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(w1));
    const uint64_t q = ptx::f32x2_mul(ptx::f32x2_mul(both(0.5f), ptx::f32x2_pack(e0, e1)), ptx::f32x2_mul(s, p));
    ptx::f32x2_unpack(ptx::f32x2_fma(nt, q, ptx::f32x2_pack(__uint_as_float(pos << 16), __uint_as_float(pos & 0xFFFF0000u))), y0, y1);
    return ptx::pack_bf16x2(y0, y1);
}

// Parameters of the LayerNorm that may run in front of the rotation (gamma == nullptr: none).
struct LnArgs {
    const float *gamma, *beta;   // fp32 [K]
    float eps;
    uint16_t *out;               // LN == 2 / 4 only: bf16 [M, K], the normalized / activated rows (nothing else is computed)
};

}  // namespace rsqc
