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

// The same tree over the squares of N of the T registers, starting at O.
template <int N, int O = 0, int T>
__device__ __forceinline__ float tree_sum_squares(const float (&a)[T])
{
    if constexpr (N == 1) return __fmul_rn(a[O], a[O]);
    else return __fadd_rn(tree_sum_squares<N / 2, O>(a), tree_sum_squares<N / 2, O + N / 2>(a));
}

// GELU x Phi(x) (the activation between the two linears of the MLP: the producer of fc2's input) of two bf16 values, rounded to
// bf16.  With t = |x| the tail Q(t) = 1 - Phi(t) is taken as 2^P(t), P a polynomial of degree 9 (own minimax fit of log2 Q on
// [0, 13.25], by iteratively reweighted least squares), so that the negative tail keeps its RELATIVE accuracy; then
// gelu(x) = max(x, 0) - t Q(t).  Relative error of Q with the fp32 evaluation below 5e-5; beyond 13.25 the tail is below 2^-126 and
// flushes to zero.  The fused multiply-adds are written explicitly (the file is compiled without contraction).
// One special-function operation per element (8 cycles of that unit each) and everything else two elements per instruction: with a
// reciprocal beside the exponential and scalar arithmetic (37 instructions per pair instead of 19) the fused kernel was bound by both.
__device__ __forceinline__ uint32_t gelu_bf16x2(uint32_t x)
{
    uint32_t a = x | 0x80008000u, pos;                     // -t
    asm("max.bf16x2 %0, %1, %2;" : "=r"(a) : "r"(a), "r"(0xC154C154u));          // -13.25
    asm("max.bf16x2 %0, %1, %2;" : "=r"(pos) : "r"(x), "r"(0u));
    const uint64_t nt = ptx::f32x2_pack(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u));
    constexpr float c[10] = {-1.00003052f, 1.15097892f, -0.458792716f, 0.053958077f, 0.00866845064f,       // P(-(-t)): odd terms negated
                             0.00102148089f, 8.3747007e-05f, 4.47421826e-06f, 1.39110185e-07f, 1.90157845e-09f};
    uint64_t p = ptx::f32x2_pack(c[9], c[9]);
#pragma unroll
    for (int i = 8; i >= 0; --i) p = ptx::f32x2_fma(p, nt, ptx::f32x2_pack(c[i], c[i]));
    float p0, p1, q0, q1, y0, y1;
    ptx::f32x2_unpack(p, p0, p1);
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(q0) : "f"(p0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(q1) : "f"(p1));
    const uint64_t y = ptx::f32x2_fma(nt, ptx::f32x2_pack(q0, q1), ptx::f32x2_pack(__uint_as_float(pos << 16), __uint_as_float(pos & 0xFFFF0000u)));
    ptx::f32x2_unpack(y, y0, y1);
    return ptx::pack_bf16x2(y0, y1);
}

// Parameters of the LayerNorm that may run in front of the rotation (gamma == nullptr: none).
struct LnArgs {
    const float *gamma, *beta;   // fp32 [K]
    float eps;
    uint16_t *out;               // LN == 2 / 4 only: bf16 [M, K], the normalized / activated rows (nothing else is computed)
};

}  // namespace rsqc
