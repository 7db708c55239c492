// Integer GEMM + rescale + bias + bf16 for few token rows (Sec. 3.2, the same sums and the same epilogue as gemm_c8.cu / gemm.cu /
// gemm_grouped.cu, bit for bit).
//
// With a handful of rows nothing is bound by the tensor core: the layer is its N K bytes of weights (0.15 - 0.6 us of memory
// bandwidth) plus latency.  The persistent kernels give such a layer N / 256 CTA pairs, each of which walks all of K at the pace
// of full 256-row MMAs behind TMA and tensor-memory set-up.
// Here a CTA owns 16 channels and its warps share K, so that all weight bytes of the layer are in flight at once; they go from
// global memory straight into the fragments of mma.sync (whose rate does not matter here), a lane's 16 consecutive bytes of a
// row standing for whichever k the fragment asks for: the same permutation of K for both operands, which an integer sum does not
// see.  The warps' partial sums meet in shared memory.
#include <cuda_bf16.h>

#include "qvggt_internal.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"

namespace {

constexpr int CH = 16;          // channels per CTA: the rows of one MMA

__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 128 consecutive codes of a row are four lanes' pieces: 32 codes each.  One code per byte: 2 x 16 bytes, 64 codes apart.
// Two per byte: 16 bytes, expanded to the codes' values times 16 (products carry a factor of 256, taken out exactly).
template <bool PACKED>
struct Piece {
    uint4 v[PACKED ? 1 : 2];
    __device__ __forceinline__ void load(const unsigned char *row, int k128, int t)
    {
        if (PACKED) {
            v[0] = __ldcg(reinterpret_cast<const uint4 *>(row + 64 * k128) + t);
        } else {
            v[0] = __ldcg(reinterpret_cast<const uint4 *>(row + 128 * k128) + t);
            v[1] = __ldcg(reinterpret_cast<const uint4 *>(row + 128 * k128) + t + 4);
        }
    }
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < (PACKED ? 1 : 2); ++i) v[i] = make_uint4(0, 0, 0, 0);
    }
    __device__ __forceinline__ uint32_t word(int i) const      // 0 .. 7: four codes each
    {
        const uint4 &q = v[PACKED ? 0 : i >> 2];
        if (PACKED) {
            const int j = i >> 1;
            const uint32_t w = j == 0 ? q.x : j == 1 ? q.y : j == 2 ? q.z : q.w;
            return (i & 1) ? (w & 0xF0F0F0F0u) : ((w << 4) & 0xF0F0F0F0u);
        }
        const int j = i & 3;
        return j == 0 ? q.x : j == 1 ? q.y : j == 2 ? q.z : q.w;
    }
};

// NT: tiles of 8 token rows per CTA.  WARPS x BLOCKS x 128 = K: a warp takes the 128-code blocks warp, warp + WARPS, ...
template <bool PACKED, bool GROUPED, int NT, int WARPS, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32)
gemm_small_kernel(const unsigned char *__restrict__ Xq, const unsigned char *__restrict__ Wq, const float *__restrict__ a_scale,
                  const float *__restrict__ w_scale, const uint16_t *__restrict__ bias, uint16_t *__restrict__ Y, long long ldy, int M)
{
    constexpr int TOK = 8 * NT, KB = WARPS * BLOCKS, ROW = KB * (PACKED ? 64 : 128);    // bytes of a row of codes
    constexpr int PARTS = GROUPED ? KB : WARPS;             // partial sums per output
    constexpr int PITCH = CH + 4;
    __shared__ int part[PARTS * TOK * PITCH];               // [part][token][channel]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int n0 = blockIdx.x * CH, m0 = blockIdx.y * TOK;
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const unsigned char *w0 = Wq + (long long)(n0 + g) * ROW, *w1 = w0 + 8 * ROW;
    Piece<PACKED> wa[BLOCKS], wb[BLOCKS];
#pragma unroll
    for (int i = 0; i < BLOCKS; ++i) {
        wa[i].load(w0, warp + WARPS * i, t);
        wb[i].load(w1, warp + WARPS * i, t);
    }
    int acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0;
#pragma unroll
    for (int i = 0; i < BLOCKS; ++i) {
        Piece<PACKED> x[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int m = m0 + 8 * j + g;
            if (m < M) x[j].load(Xq + (long long)m * ROW, warp + WARPS * i, t);
            else x[j].clear();
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int s = 0; s < 4; ++s)
                mma_s8(acc[j], wa[i].word(2 * s), wb[i].word(2 * s), wa[i].word(2 * s + 1), wb[i].word(2 * s + 1), x[j].word(2 * s), x[j].word(2 * s + 1));
        if (GROUPED || i == BLOCKS - 1) {
            int *p = part + (GROUPED ? warp + WARPS * i : warp) * (TOK * PITCH);
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                // fragment: channels g and g + 8, tokens 2 t and 2 t + 1
                int *d = p + (8 * j + 2 * t) * PITCH + g;
                d[0] = acc[j][0]; d[PITCH] = acc[j][1]; d[8] = acc[j][2]; d[PITCH + 8] = acc[j][3];
                if (GROUPED) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0;
            }
        }
    }
    __syncthreads();
    // one thread per token and channel pair
    for (int o = threadIdx.x; o < TOK * (CH / 2); o += WARPS * 32) {
        const int tok = o / (CH / 2), c = 2 * (o % (CH / 2)), m = m0 + tok, n = n0 + c;
        if (m >= M) continue;
        const int *p = part + tok * PITCH + c;
        constexpr int SHIFT = PACKED ? 8 : 0;
        const float2 ws = __ldg(reinterpret_cast<const float2 *>(w_scale + n));
        const uint32_t bb = bias ? __ldg(reinterpret_cast<const uint32_t *>(bias + n)) : 0u;
        const float b0 = __uint_as_float(bb << 16), b1 = __uint_as_float(bb & 0xFFFF0000u);
        float z0, z1;
        if (GROUPED) {
            z0 = z1 = 0.0f;
            const float *as = a_scale + (long long)m * KB;
#pragma unroll
            for (int k = 0; k < KB; ++k) {                 // ascending groups, two roundings each
                const int2 s = *reinterpret_cast<const int2 *>(p + k * (TOK * PITCH));
                const float a = __ldg(as + k);
                z0 = __fadd_rn(z0, __fmul_rn(static_cast<float>(s.x >> SHIFT), a));
                z1 = __fadd_rn(z1, __fmul_rn(static_cast<float>(s.y >> SHIFT), a));
            }
            z0 = __fmul_rn(z0, ws.x);
            z1 = __fmul_rn(z1, ws.y);
        } else {
            int s0 = 0, s1 = 0;
#pragma unroll
            for (int k = 0; k < PARTS; ++k) {
                const int2 s = *reinterpret_cast<const int2 *>(p + k * (TOK * PITCH));
                s0 += s.x;
                s1 += s.y;
            }
            const float a = __ldg(a_scale + m);
            z0 = __fmul_rn(static_cast<float>(s0 >> SHIFT), __fmul_rn(a, ws.x));
            z1 = __fmul_rn(static_cast<float>(s1 >> SHIFT), __fmul_rn(a, ws.y));
        }
        *reinterpret_cast<uint32_t *>(Y + (long long)m * ldy + n) = ptx::pack_bf16x2(__fadd_rn(z0, b0), __fadd_rn(z1, b1));
    }
}

template <bool PACKED, bool GROUPED, int NT, int WARPS, int BLOCKS>
cudaError_t launch(const qvggt_weights *w, const void *Xq, const void *Wq, const float *a_scale, int M, void *Y, long long ldy, cudaStream_t st)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(w->N / CH, (M + 8 * NT - 1) / (8 * NT));
    cfg.blockDim = dim3(WARPS * 32);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_small_kernel<PACKED, GROUPED, NT, WARPS, BLOCKS>, static_cast<const unsigned char *>(Xq),
                              static_cast<const unsigned char *>(Wq), a_scale, (const float *)w->w_scale, (const uint16_t *)w->bias,
                              static_cast<uint16_t *>(Y), ldy, M);
}

template <bool PACKED, bool GROUPED>
cudaError_t dispatch(const qvggt_weights *w, const void *Xq, const void *Wq, const float *a_scale, int M, void *Y, long long ldy, cudaStream_t st)
{
    if (w->K == 1024) {
        if (M <= 8) return launch<PACKED, GROUPED, 1, 8, 1>(w, Xq, Wq, a_scale, M, Y, ldy, st);
        if (M <= 16) return launch<PACKED, GROUPED, 2, 8, 1>(w, Xq, Wq, a_scale, M, Y, ldy, st);
        return launch<PACKED, GROUPED, 4, 8, 1>(w, Xq, Wq, a_scale, M, Y, ldy, st);
    }
    if (M <= 8) return launch<PACKED, GROUPED, 1, 16, 2>(w, Xq, Wq, a_scale, M, Y, ldy, st);
    return launch<PACKED, GROUPED, 2, 16, 2>(w, Xq, Wq, a_scale, M, Y, ldy, st);
}

}  // namespace

// Where the lines lie: this kernel's time grows with M N K (its rate is that of mma.sync), the persistent kernels' hardly moves
// below one round of tiles.  What decides is the layer, the quantize launch and the GEMM behind it: the persistent kernels hide more of
// their start behind the quantize launch, so alone and back to back this kernel would win for longer than it does in a layer.
// Layers in a replayed graph (us, this kernel / the other one), each line between the first and the second M:
//   one code per byte   K = 1024: N = 256, M = 384 5.4 / 5.5, M = 576 6.4 / 5.9; N = 640, M = 128 5.0 / 5.4, M = 153 5.8 / 5.4;
//                                 N = 1024, M = 96 5.4 / 5.4, M = 192 6.0 / 5.5; N = 2048, M = 80 5.5 / 5.8, M = 96 5.7 / 5.6, M = 160 7.1 / 5.8;
//                                 N = 3072, M = 58 5.5 / 6.05, M = 69 6.4 / 5.8; N = 4096, M = 48 5.5 / 5.9, M = 56 6.4 / 5.9; N = 128 within
//                                 10 % either way from M = 512 to 2048.  Up to 96 rows the outputs decide at 3 * 2^16, beyond at half of that
//                       K = 4096: N = 128, M = 576 10.1 / 11.8, M = 640 11.9 / 11.8, M = 768 13.3 / 11.9; N = 384, M = 213 10.2 / 10.2, M = 256 11.1 / 10.2;
//                                 N = 640, M = 153 10.1 / 10.1, M = 166 10.8 / 10.1; N = 1024, M = 96 9.6 / 10.1, M = 112 10.3 / 10.15;
//                                 N = 4096, M = 24 9.3 / 11.1, M = 32 10.75 / 10.4
//   packed              K = 1024: N = 128, M = 6144 12.6 / 13.5, M = 8232 15.6 / 15.1; N = 3072, M = 256 9.1 / 9.3, M = 343 11.2 / 9.6
//                       K = 4096: N = 1024, M = 384 17.8 / 19.5, M = 514 21.4 / 21.6; N = 4096, M = 96 16.2 / 19.9, M = 128 20.3 / 18.8
//   group scales        K = 1024: N = 1024, M = 384 8.5 / 9.0, M = 514 9.6 / 8.9; N = 4096, M = 96 8.2 / 8.2, M = 128 9.1 / 8.3
//                       K = 4096: N = 128, M = 1152 19.4 / 21.5, M = 1536 24.2 / 22.8; N = 1024, M = 144 15.6 / 17.7, M = 192 19.4 / 17.5
// and the GEMM alone at 5 rows   K = 1024, N = 3072 2.3 / 4.5, packed 2.0 / 7.8, groups 2.4 / 6.3; K = 4096 2.5 / 8.0, 2.2 / 16.4, 3.1 / 14.8
bool qvggt_gemm_small_wins(const qvggt_weights *w, int M, bool packed, bool grouped)
{
    const long long outputs = (long long)M * w->N;
    if (w->K == 1024) return outputs <= (packed ? 3LL << 18 : grouped ? 3LL << 17 : M <= 96 ? 3LL << 16 : 3LL << 15);
    return outputs <= (packed ? 3LL << 17 : grouped ? 9LL << 14 : w->N < 640 ? 5LL << 14 : 3LL << 15);
}

cudaError_t qvggt_launch_gemm_small(const qvggt_weights *w, const void *Xq, const void *Wq, bool packed, const float *a_scale, bool grouped, int M,
                                    void *Y, long long ldy, cudaStream_t st)
{
    if (packed)
        return grouped ? dispatch<true, true>(w, Xq, Wq, a_scale, M, Y, ldy, st) : dispatch<true, false>(w, Xq, Wq, a_scale, M, Y, ldy, st);
    return grouped ? dispatch<false, true>(w, Xq, Wq, a_scale, M, Y, ldy, st) : dispatch<false, false>(w, Xq, Wq, a_scale, M, Y, ldy, st);
}
