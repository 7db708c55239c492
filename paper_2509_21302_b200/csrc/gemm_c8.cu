// W4A4 GEMM on codes held in 8-bit containers (Sec. 3.2: integer sum over the inner dimension, per-token and
// per-out-channel scales applied outside the sum), for sm_100a.
//
// tcgen05 has no 4-bit integer kind: whatever the storage format, the tensor core multiplies int8.  Here the
// producers already emit one code per byte (the quantize kernel for the activations, the offline weight
// preparation for the weights), so the tiles go from global memory straight into the 128-byte-swizzled operand
// stages by TMA and nothing in this kernel touches an operand byte with an ordinary instruction.  Per K-block
// a CTA's shared memory sees one TMA write and one tensor-core read of its 32 KB of operands, the minimum.
//
// Persistent and warp-specialised; a worker is a pair of CTAs on neighbouring SMs (tile 256 tokens x BN = 256 or 128
// channels, each CTA stages 128 token rows and BN / 2 weight rows; one thread of the leader CTA issues
// tcgen05.mma.cta_group::2.kind::i8 for both; accumulators int32 in tensor memory, two buffers of BN columns).
//   warps 0..7   epilogue: TMEM -> registers -> scale, bias, bf16 -> swizzled staging -> whole-line stores; no warp waits for another
//   warp  8      one elected thread issues tcgen05.mma and the commits that release stages / publish accumulators
//   warp  9      one thread per CTA issues the TMA loads of its half of every operand stage; both CTAs signal
//                the leader's "full" barrier (cta_group::2 form of the load)
// The tiles are dealt round-robin to the workers.
// Every wait is bounded; on expiry the kernel records a code in *status and all roles fall through to the
// common exit, where tensor memory is released.
#include <cuda.h>
#include <cuda_bf16.h>

#include "gemm_common.cuh"
#include "qvggt_internal.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"
#include "unpack_w4.cuh"

namespace {

using gemmc::Ring;
using gemmc::STG_BYTES;

constexpr int BM = 128;            // token rows per CTA (TMEM lanes)
constexpr int BK = 128;            // codes along K per stage = one 128-byte swizzled row
constexpr int ACC_BUFS = 2;        // TMEM accumulators: the epilogue of tile i overlaps the MMAs of tile i+1
constexpr int EPI_WARPS = 8;       // warp w: TMEM lane quarter w % 4, column part w / 4
constexpr int MMA_WARP = EPI_WARPS;
constexpr int TMA_WARP = EPI_WARPS + 1;
constexpr int THREADS = (EPI_WARPS + 2) * 32;

// BN = output channels per tile: 256, or 128 where that keeps more of the chip busy (see wide_tiles()).
template <int BN>
struct Lay {
    static constexpr int B_ROWS = BN / 2;                         // weight rows staged by one CTA
    static constexpr int STAGE = (BM + B_ROWS) * BK;              // 32 / 24 KB
    static constexpr int STAGES = BN == 256 ? 6 : 8;
    static constexpr int OFF_STG = STAGES * STAGE;                // operand stages first: they need 1024-byte alignment
    static constexpr int OFF_CH = OFF_STG + EPI_WARPS * STG_BYTES;          // per warp: scales and biases of its BN / 2 channels, fp32
    static constexpr int OFF_BAR = OFF_CH + EPI_WARPS * BN * 4;             // full[STAGES] empty[STAGES] tfull[2] tempty[2]
    static constexpr int NBARS = 2 * STAGES + 2 * ACC_BUFS;
    static constexpr int OFF_TMEM = OFF_BAR + NBARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 4;
    static constexpr int SMEM_BYTES = OFF_ABORT + 4;
    static constexpr int DYN_SMEM = SMEM_BYTES + 1024;            // slack to align the base to 1024 bytes
    static constexpr int TMEM_COLS = ACC_BUFS * BN;               // 512 / 256
    static_assert(DYN_SMEM <= 232448, "exceeds the 227 KB of shared memory a CTA may use");
    static_assert(2 * STAGE < (1 << 20), "transaction count of a stage must fit the barrier");
    static_assert(STAGE % 1024 == 0, "operand tiles must stay 1024-byte aligned");
};

// DUMP: also write the int32 sums to acc_debug (its own instantiation keeps that code out of the production kernel).
// wait_limit: bound of every device-side wait, in cycles.  skip_loads: the TMA producers issue nothing, so that the
// first wait for operands runs out (used only to exercise the timeout path; no asynchronous operation is in flight).
template <int BN, bool DUMP>
__global__ void __launch_bounds__(THREADS, 1)
gemm_c8_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
               uint16_t *__restrict__ Y, long long ldy,
               const float *__restrict__ a_scale, const float *__restrict__ w_scale, const uint16_t *__restrict__ bias,
               int *__restrict__ acc_debug, int M, int N, int K, int *status, long long wait_limit, int skip_loads)
{
    using L = Lay<BN>;
    constexpr int STAGES = L::STAGES, STAGE = L::STAGE, B_ROWS = L::B_ROWS, TMEM_COLS = L::TMEM_COLS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = ptx::smem_addr(smem);
    const uint32_t bar_full = sbase + L::OFF_BAR;
    const uint32_t bar_empty = bar_full + STAGES * 8;
    const uint32_t bar_tfull = bar_empty + STAGES * 8;
    const uint32_t bar_tempty = bar_tfull + ACC_BUFS * 8;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L::OFF_TMEM);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L::OFF_ABORT);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();                       // 0 = leader of the pair
    const int worker = blockIdx.x / 2, workers = gridDim.x / 2;
    const int KB = K / BK;
    const int n_tiles = (N + BN - 1) / BN;
    const int total_tiles = ((M + 2 * BM - 1) / (2 * BM)) * n_tiles;
    const int my_tiles = (total_tiles > worker) ? (total_tiles - 1 - worker) / workers + 1 : 0;

    if (threadIdx.x == 0) {
        gemmc::init_barriers(bar_full, STAGES, 1);                     // the leader's arrive.expect_tx (bytes of both CTAs)
        gemmc::init_barriers(bar_empty, STAGES, 1);                    // tcgen05.commit
        gemmc::init_barriers(bar_tfull, ACC_BUFS, 1);                  // tcgen05.commit
        gemmc::init_barriers(bar_tempty, ACC_BUFS, EPI_WARPS * 2);     // the epilogue warps of both CTAs
        *s_abort = 0;
        ptx::fence_mbar_init();
    }
    if (warp == MMA_WARP) { ptx::tmem_alloc_pair(ptx::smem_addr(s_tmem), TMEM_COLS); ptx::tmem_relinquish_pair(); }
    if (warp == TMA_WARP && lane == 0) {
        ptx::prefetch_tensormap(&map_x);
        ptx::prefetch_tensormap(&map_w);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();                     // the leader's barriers exist before the peer's loads signal them
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *s_tmem;
    // everything above touched only kernel parameters and on-chip state: it may overlap the tail of the previous
    // kernel in the stream; the operands (and the output buffer) may not be touched before that kernel is done
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    if (warp < EPI_WARPS) {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3, cpart = warp >> 2;   // TMEM lane quarter, column part
        unsigned char *stg = smem + L::OFF_STG + warp * STG_BYTES;
        const uint32_t stg_addr = sbase + L::OFF_STG + warp * STG_BYTES;
        float *wsb = reinterpret_cast<float *>(smem + L::OFF_CH) + warp * BN, *bsb = wsb + BN / 2;     // the warp's channel scales, biases
        const uint32_t leader_tempty = ptx::map_to_cta(bar_tempty, 0);
        const uint64_t one2 = ptx::f32x2_one(N & 127);                       // N is a multiple of 128
        bool alive = true;
        constexpr int CW = BN / 2, NCH = CW / 64;              // columns and 64-column chunks of one warp's part
        for (int t = 0; t < my_tiles; ++t) {
            const int tile = worker + t * workers;
            const int m0 = (tile / n_tiles) * (2 * BM) + (int)rank * BM + quarter * 32;
            const int n0 = (tile % n_tiles) * BN + cpart * CW; // first channel of this warp's part
            const int b = t & 1;
            const bool cols_ok = n0 < N;                       // N is a multiple of 128: a part is all in or all out
            // The scales and biases of the warp's channels: each warp keeps its own copy in shared memory, so that no warp ever
            // waits for another.
            float my_ws[CW / 32], my_bs[CW / 32];
#pragma unroll
            for (int e = 0; e < CW / 32; ++e) {
                const int n = n0 + 32 * e + lane;
                my_ws[e] = cols_ok ? __ldg(w_scale + n) : 0.0f;
                my_bs[e] = (cols_ok && bias) ? __uint_as_float(static_cast<uint32_t>(__ldg(bias + n)) << 16) : 0.0f;
            }
            uint64_t as2[2][2];                                // rows lane / 4 + 8 h of the warp's 16 u .. 16 u + 15
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int gm = m0 + 8 * u + (lane >> 2);
                const float as = gm < M ? __ldg(a_scale + gm) : 0.0f;
                as2[u >> 1][u & 1] = ptx::f32x2_pack(as, as);
            }
            __syncwarp();                                      // the previous tile's last reads
#pragma unroll
            for (int e = 0; e < CW / 32; ++e) {
                wsb[32 * e + lane] = my_ws[e];
                bsb[32 * e + lane] = my_bs[e];
            }
            __syncwarp();
            {
                int ok = 1;
                if (lane == 0) ok = (alive && ptx::mbar_wait(bar_tfull + 8 * b, (t >> 1) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_ACCUM, 32, wait_limit)) ? 1 : 0;
                alive = __shfl_sync(0xFFFFFFFFu, ok, 0) != 0;
            }
            ptx::tc_fence_after_sync();
            if (alive) {
#pragma unroll
                for (int c = 0; c < NCH; ++c) {
                    uint32_t raw[2][32];
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        ptx::tmem_ld_16x256b_x8(tmem_base + (static_cast<uint32_t>(quarter * 32 + 16 * u) << 16) + b * BN + cpart * CW + c * 64, raw[u]);
                    ptx::tmem_ld_wait();
                    if (c == NCH - 1) {                        // tensor memory goes back to the MMA thread
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        // (nobody waits for the last tiles' arrivals: none may be on its way when the leader CTA exits)
                        if (lane == 0 && t + ACC_BUFS < my_tiles) ptx::mbar_arrive_cluster(leader_tempty + 8 * b);
                    }
                    if (cols_ok) {
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int m = m0 + 16 * u, n = n0 + 64 * c;
                            gemmc::finish_16x64(raw[u], as2[u], wsb + 64 * c, bsb + 64 * c, stg, stg_addr, Y + (long long)m * ldy + n, ldy, M - m, lane, one2);
                            if (DUMP && acc_debug) gemmc::dump_16x64<0>(acc_debug + (long long)m * N + n, N, raw[u], M - m, lane);
                        }
                    }
                }
            }
        }
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------------------ MMA issuer (one thread of the leader CTA)
        // The thread is chosen by elect.sync, not by its lane number: the assembler then knows that one thread is active and keeps
        // the descriptors in uniform registers, where tcgen05 wants them (behind `lane == 0` every one is moved there anew, which
        // made this loop, at 545 cycles per K-block, the bound of the kernel).
        if (rank == 0 && ptx::elect_one()) {
            constexpr uint32_t idesc = ptx::idesc_i8(2 * BM, BN);
            bool alive = true;
            Ring r;
            int left = my_tiles * KB;                                      // K-blocks to come, this one included
            for (int t = 0; t < my_tiles && alive; ++t) {
                const int b = t & 1;
                if (t >= ACC_BUFS) {
                    alive = ptx::mbar_wait_cluster(bar_tempty + 8 * b, ((t >> 1) - 1) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_TMEM_FREE, wait_limit);
                    if (!alive) break;
                    ptx::tc_fence_after_sync();
                }
                const uint32_t d_tmem = tmem_base + b * BN;
                for (int kb = 0; kb < KB; ++kb) {
                    alive = ptx::mbar_wait_cluster(bar_full + 8 * r.s, r.ph, s_abort, status, QVGGT_DEV_TIMEOUT_FULL, wait_limit);
                    if (!alive) break;
                    ptx::tc_fence_after_sync();
                    const uint32_t a_addr = sbase + r.s * STAGE;
                    gemmc::mma_kblock_i8<true>(d_tmem, a_addr, a_addr + BM * BK, idesc, kb == 0);
                    if (left-- > STAGES) ptx::mma_commit_pair(bar_empty + 8 * r.s, 3);   // frees the stage in both CTAs, if a load waits for it
                    if (kb == KB - 1) ptx::mma_commit_pair(bar_tfull + 8 * b, 3);
                    r.advance(STAGES);
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ TMA producer (one thread per CTA)
        if (!skip_loads && ptx::elect_one()) {
            const uint32_t leader_full = ptx::map_to_cta(bar_full, 0);
            bool alive = true;
            Ring r;
            int it = 0;
            for (int t = 0; t < my_tiles && alive; ++t) {
                const int tile = worker + t * workers;
                const int m0 = (tile / n_tiles) * (2 * BM) + (int)rank * BM;
                const int n0 = (tile % n_tiles) * BN + (int)rank * B_ROWS;
                for (int kb = 0; kb < KB; ++kb, ++it) {
                    if (it >= STAGES) {
                        alive = ptx::mbar_wait(bar_empty + 8 * r.s, r.ph ^ 1, s_abort, status, QVGGT_DEV_TIMEOUT_EMPTY, 20, wait_limit);
                        if (!alive) break;
                    }
                    const uint32_t dst = sbase + r.s * STAGE;
                    // the leader's barrier expects the bytes of both CTAs; the peer's completions may arrive first
                    // (the count goes negative for a while), the phase cannot end before the leader has arrived
                    if (rank == 0) ptx::mbar_arrive_expect_tx(bar_full + 8 * r.s, 2 * STAGE);
                    ptx::tma_load_2d_pair(&map_x, leader_full + 8 * r.s, dst, kb * BK, m0);
                    ptx::tma_load_2d_pair(&map_w, leader_full + 8 * r.s, dst + BM * BK, kb * BK, n0);
                    r.advance(STAGES);
                }
            }
        }
        __syncwarp();
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync_relaxed();        // no remote arrival or multicast commit may target a CTA that has exited: each one is waited for
    if (warp == MMA_WARP) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

// ------------------------------------------------------------------------------------------------
// The same TMA-fed CTA-pair design for one activation scale per token per 128 rotated channels (an extension of the
// paper's token-wise granularity; the weights keep one scale per output channel).  A K-block of 128 codes is one scale
// group, so every K-block accumulates into its own tensor-memory buffer (four of 128 columns, handed over two at a
// time) and the epilogue warps rescale a pair while the next one runs:
//   s = fl(s + fl(float(acc_g) * a_scale[m][g])), g ascending;  Y = bf16(fl(fl(s * w_scale[n]) + bias[n])).
// Tile 256 tokens x 128 channels per pair; an epilogue thread keeps 32 running sums of its row in registers.  The epilogue
// sets the pace: per K-block ~280 cycles of MMA work against 725 (K = 4096) - 1000 (K = 1024), of which the arithmetic
// (conversion, packed multiply, packed uncontracted add) is ~250, the wait for the pair and its hand-over ~200 and, at
// K = 1024, the end of a tile ~250 (2050 cycles for eight K-blocks).  With the arithmetic taken out of a copy for timing the launch
// takes 58 instead of 82 us (10 992 rows, K = 1024, N = 4096), without the operand loads as well 52.  Measured and slower:
// the whole next K-block's sums in registers (they do not fit beside the running sums, not even with the issuing warps' registers
// moved to these), accumulators released one by one (84 us), ordinary stores instead of the TMA store (87 us: the
// warp then waits for its own lines), the next tile's first scales fetched ahead (84 us).
namespace grp {

constexpr int GN = 128;                                // channels per tile
constexpr int GEPI = 16;                               // epilogue warps: lane quarter w % 4, 32-column part w / 4 (four per scheduler: the
                                                       // epilogue is latency-bound, cf. 1400 against 2400 cycles per K-block with eight)
constexpr int G_MMA_WARP = GEPI, G_TMA_WARP = GEPI + 1;
constexpr int GTHREADS = (GEPI + 2) * 32;
constexpr int GB_ROWS = GN / 2;                        // weight rows staged by one CTA
constexpr int GSTAGE = (BM + GB_ROWS) * BK;            // 24 KB
constexpr int GACC = 4, GPAIRS = GACC / 2;             // accumulators of 128 columns; they are handed over two K-blocks at a time
constexpr int GSTAGES = 7;
constexpr int OFF_STG = GSTAGES * GSTAGE;
constexpr int OFF_CH = OFF_STG + GEPI * STG_BYTES;          // per warp: 32 channel scales, 32 biases, fp32
constexpr int OFF_BAR = OFF_CH + GEPI * 64 * 4;                 // full[GSTAGES] empty[GSTAGES] tfull[2] tempty[2]
constexpr int NBARS = 2 * GSTAGES + 2 * GPAIRS;
constexpr int OFF_TMEM = OFF_BAR + NBARS * 8;
constexpr int OFF_ABORT = OFF_TMEM + 4;
constexpr int DYN_SMEM = OFF_ABORT + 4 + 1024;                    // slack to align the base to 1024 bytes
constexpr int TMEM_COLS = GACC * GN;                              // 512
static_assert(DYN_SMEM <= 232448, "exceeds the 227 KB of shared memory a CTA may use");
static_assert(GSTAGE % 1024 == 0, "operand tiles must stay 1024-byte aligned");

// WIDE: the scales are read 16 bytes at a time (a row of them is 32 or 128 bytes).  The caller's pointer need only be aligned to 4
// bytes; off a 16-byte boundary the other instantiation runs (chosen inside one kernel, the second form of the loads cost the
// aligned call 1.1 %: 817.5 -> 826.3 us for an MLP of 43 968 rows).
template <bool DUMP, bool WIDE>
__global__ void __launch_bounds__(GTHREADS, 1)
gemm_c8_grouped_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                       const __grid_constant__ CUtensorMap map_y, const float *__restrict__ a_scale,
                       const float *__restrict__ w_scale, const uint16_t *__restrict__ bias, int *__restrict__ acc_debug,
                       int M, int N, int K, int *status)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = ptx::smem_addr(smem);
    const uint32_t bar_full = sbase + OFF_BAR;
    const uint32_t bar_empty = bar_full + GSTAGES * 8;
    const uint32_t bar_tfull = bar_empty + GSTAGES * 8;
    const uint32_t bar_tempty = bar_tfull + GPAIRS * 8;
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + OFF_TMEM);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + OFF_ABORT);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();
    const int worker = blockIdx.x / 2, workers = gridDim.x / 2;
    const int KB = K / BK;                                   // = number of scale groups
    const int n_tiles = N / GN;
    const int total_tiles = ((M + 2 * BM - 1) / (2 * BM)) * n_tiles;
    const int my_tiles = (total_tiles > worker) ? (total_tiles - 1 - worker) / workers + 1 : 0;

    if (threadIdx.x == 0) {
        gemmc::init_barriers(bar_full, GSTAGES, 1);
        gemmc::init_barriers(bar_empty, GSTAGES, 1);
        gemmc::init_barriers(bar_tfull, GPAIRS, 1);
        gemmc::init_barriers(bar_tempty, GPAIRS, GEPI * 2);
        *s_abort = 0;
        ptx::fence_mbar_init();
    }
    if (warp == G_MMA_WARP) { ptx::tmem_alloc_pair(ptx::smem_addr(s_tmem), TMEM_COLS); ptx::tmem_relinquish_pair(); }
    if (warp == G_TMA_WARP && lane == 0) {
        ptx::prefetch_tensormap(&map_x);
        ptx::prefetch_tensormap(&map_w);
        ptx::prefetch_tensormap(&map_y);
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *s_tmem;
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    if (warp < GEPI) {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3, cpart = warp >> 2;   // TMEM lane quarter, 32-column part
        unsigned char *stg = smem + OFF_STG + warp * STG_BYTES;
        const uint32_t stg_addr = sbase + OFF_STG + warp * STG_BYTES;
        float *wsb = reinterpret_cast<float *>(smem + OFF_CH) + warp * 64, *bsb = wsb + 32;   // the warp's channel scales, biases
        const uint32_t leader_tempty = ptx::map_to_cta(bar_tempty, 0);
        const uint64_t one2 = ptx::f32x2_one(N & 127);                       // N is a multiple of 128
        const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
        bool alive = true;
        int pair = 0;                                               // pairs of K-blocks seen so far (all tiles)
        for (int t = 0; t < my_tiles; ++t) {
            const int tile = worker + t * workers;
            const int m0 = (tile / n_tiles) * (2 * BM) + (int)rank * BM + quarter * 32;
            const int n0 = (tile % n_tiles) * GN + cpart * 32;
            const int gm = m0 + lane;
            const bool row_ok = gm < M;
            // The scales and biases of the warp's 32 channels, one channel per lane, fetched here and needed at the end of the tile: each
            // warp keeps its own copy, so that no warp ever waits for another.
            const float my_ws = __ldg(w_scale + n0 + lane);
            const float my_bs = bias ? __uint_as_float(static_cast<uint32_t>(__ldg(bias + n0 + lane)) << 16) : 0.0f;
            uint64_t sum2[16];                                      // running sums of 32 channels, two per register pair
#pragma unroll
            for (int j = 0; j < 16; ++j) sum2[j] = 0;
            // The row's scales come from L2, four groups per load, one load ahead (fetched one by one they set the pace: the latency
            // of one load per K-block).  Without WIDE the four groups are four loads, still one step ahead.
            const float *as_row = a_scale + (long long)(row_ok ? gm : 0) * KB;
            auto four_scales = [&](int kb) {
                const float *p = as_row + kb;
                return WIDE ? __ldg(reinterpret_cast<const float4 *>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
            };
            float4 as_next = four_scales(0);
            auto wait_full = [&](int p) {      // every warp polls for itself: no warp waits for a slower one between K-blocks
                const bool ok = alive && ptx::mbar_wait(bar_tfull + 8 * (p % GPAIRS), (p / GPAIRS) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_ACCUM, 20);
                alive = __all_sync(0xFFFFFFFFu, ok);
                ptx::tc_fence_after_sync();
            };
            auto add_group = [&](const uint32_t (&raw)[16], int half, float as) {
                const uint64_t as2 = ptx::f32x2_pack(as, as);
#pragma unroll
                for (int j = 0; j < 16; j += 2)
                    sum2[8 * half + j / 2] = ptx::f32x2_add_uncontracted(
                        ptx::f32x2_mul(ptx::f32x2_pack(static_cast<float>(static_cast<int>(raw[j])), static_cast<float>(static_cast<int>(raw[j + 1]))), as2),
                        sum2[8 * half + j / 2], one2);
            };
            // The accumulators come in halves of 16 columns, each in flight while the other is rescaled.
            uint32_t lo[16], hi[16];
            const uint32_t my_cols = tmem_base + lane_base + cpart * 32;
            wait_full(pair);
            if (alive) ptx::tmem_ld_32x16(my_cols + (pair % GPAIRS) * 2 * GN, lo);
#pragma unroll 1
            for (int kb = 0; kb < KB; kb += 4) {
                const float as4[4] = {as_next.x, as_next.y, as_next.z, as_next.w};
                if (kb + 4 < KB) as_next = four_scales(kb + 4);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    if (!alive) continue;
                    const int b = pair % GPAIRS;
                    const uint32_t acc = my_cols + (2 * b + (g & 1)) * GN;
                    ptx::tmem_ld_wait_for(lo);
                    ptx::tmem_ld_32x16(acc + 16, hi);
                    add_group(lo, 0, as4[g]);
                    if (DUMP && acc_debug && row_ok) gemmc::dump_acc_x16(acc_debug + ((long long)(kb + g) * M + gm) * N + n0, lo);
                    ptx::tmem_ld_wait_for(hi);
                    if (g & 1) {
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0 && pair + GPAIRS < my_tiles * KB / 2) ptx::mbar_arrive_cluster(leader_tempty + 8 * b);   // if an MMA will wait for it
                        ++pair;
                        if (g < 3 || kb + 4 < KB) {
                            wait_full(pair);
                            if (alive) ptx::tmem_ld_32x16(my_cols + (pair % GPAIRS) * 2 * GN, lo);
                        }
                    } else {
                        ptx::tmem_ld_32x16(acc + GN, lo);
                    }
                    add_group(hi, 1, as4[g]);
                    if (DUMP && acc_debug && row_ok) gemmc::dump_acc_x16(acc_debug + ((long long)(kb + g) * M + gm) * N + n0 + 16, hi);
                }
            }
            wsb[lane] = my_ws;
            bsb[lane] = my_bs;
            __syncwarp();
            if (alive) {
                uint32_t out[16];
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    float z0, z1;
                    ptx::f32x2_unpack(ptx::f32x2_add_uncontracted(ptx::f32x2_mul(sum2[j / 2], *reinterpret_cast<const uint64_t *>(wsb + j)),
                                                                  *reinterpret_cast<const uint64_t *>(bsb + j), one2), z0, z1);
                    out[j >> 1] = ptx::pack_bf16x2(z0, z1);
                }
                gemmc::stage_row_32(stg, out, lane);
                gemmc::store_staged_32x32(&map_y, stg_addr, n0, m0, m0 < M, lane);
            }
            __syncwarp();                                           // wsb and bsb are rewritten at the end of the next tile
        }
        if (lane == 0) ptx::tma_store_wait_read<0>();
    } else if (warp == G_MMA_WARP) {
        // ------------------------------------------------------------ MMA issuer: one accumulator per K-block
        if (rank == 0 && ptx::elect_one()) {      // see gemm_c8_kernel
            constexpr uint32_t idesc = ptx::idesc_i8(2 * BM, GN);
            bool alive = true;
            Ring r;
            const int total_kb = my_tiles * KB;
            for (int it = 0; it < total_kb && alive; ++it) {       // K / 128 is even: pairs never straddle a tile
                const int b = it % GACC, p = it / 2;
                if (it >= GACC && !(it & 1)) {
                    alive = ptx::mbar_wait_cluster(bar_tempty + 8 * (p % GPAIRS), ((p / GPAIRS) - 1) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_TMEM_FREE);
                    if (!alive) break;
                    ptx::tc_fence_after_sync();
                }
                alive = ptx::mbar_wait_cluster(bar_full + 8 * r.s, r.ph, s_abort, status, QVGGT_DEV_TIMEOUT_FULL);
                if (!alive) break;
                ptx::tc_fence_after_sync();
                const uint32_t a_addr = sbase + r.s * GSTAGE;
                gemmc::mma_kblock_i8<true>(tmem_base + b * GN, a_addr, a_addr + BM * BK, idesc, true);
                if (it + GSTAGES < total_kb) ptx::mma_commit_pair(bar_empty + 8 * r.s, 3);
                if (it & 1) ptx::mma_commit_pair(bar_tfull + 8 * (p % GPAIRS), 3);
                r.advance(GSTAGES);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ TMA producer (one thread per CTA)
        if (ptx::elect_one()) {
            const uint32_t leader_full = ptx::map_to_cta(bar_full, 0);
            bool alive = true;
            Ring r;
            int it = 0;
            for (int t = 0; t < my_tiles && alive; ++t) {
                const int tile = worker + t * workers;
                const int m0 = (tile / n_tiles) * (2 * BM) + (int)rank * BM;
                const int n0 = (tile % n_tiles) * GN + (int)rank * GB_ROWS;
                for (int kb = 0; kb < KB; ++kb, ++it) {
                    if (it >= GSTAGES) {
                        alive = ptx::mbar_wait(bar_empty + 8 * r.s, r.ph ^ 1, s_abort, status, QVGGT_DEV_TIMEOUT_EMPTY, 20);
                        if (!alive) break;
                    }
                    const uint32_t dst = sbase + r.s * GSTAGE;
                    if (rank == 0) ptx::mbar_arrive_expect_tx(bar_full + 8 * r.s, 2 * GSTAGE);
                    ptx::tma_load_2d_pair(&map_x, leader_full + 8 * r.s, dst, kb * BK, m0);
                    ptx::tma_load_2d_pair(&map_w, leader_full + 8 * r.s, dst + BM * BK, kb * BK, n0);
                    r.advance(GSTAGES);
                }
            }
        }
        __syncwarp();
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_sync_relaxed();        // every remote arrival was waited for
    if (warp == G_MMA_WARP) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

template <bool DUMP, bool WIDE>
cudaError_t launch(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y, long long ldy,
                   int *acc_debug, cudaStream_t st)
{
    static QvggtPerDevice cache;
    int max_workers = 0;
    cudaError_t e = qvggt_configure_kernel(gemm_c8_grouped_kernel<DUMP, WIDE>, GTHREADS, DYN_SMEM, 2, cache, &max_workers);
    if (e != cudaSuccess) return e;
    const int K = w->K, N = w->N;
    CUtensorMap map_x, map_w, map_y;
    if (!qvggt_make_map(&map_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, Xq8, K, M, K, BK, BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, w->Wq8, K, N, K, BK, GB_ROWS, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_y, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Y, N, M, (uint64_t)ldy * 2, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B))
        return cudaErrorInvalidValue;
    const int total_tiles = ((M + 2 * BM - 1) / (2 * BM)) * (N / GN);
    const int workers = total_tiles < max_workers ? total_tiles : max_workers;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(workers * 2);
    cfg.blockDim = dim3(GTHREADS);
    cfg.dynamicSmemBytes = DYN_SMEM;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_c8_grouped_kernel<DUMP, WIDE>, map_x, map_w, map_y, a_scale, (const float *)w->w_scale,
                              (const uint16_t *)w->bias, acc_debug, M, N, K, w->status);
}

}  // namespace grp

// Packed weight codes [N, K/2] (byte i = code 2i in bits 0-3, code 2i+1 in bits 4-7, two's complement) -> one code per
// byte [N, K], 16 packed bytes per thread.  Used when the handle keeps only the packed codes: the unpacked copy is a
// per-launch scratch of a few megabytes that the GEMM behind it reads back from L2.
__global__ void __launch_bounds__(256) unpack_w4_kernel(const uint4 *__restrict__ packed, uint4 *__restrict__ out, long long n16)
{
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();           // the scratch may still be read by the previous GEMM of the stream
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n16) return;
    qvggt_unpack_w4_item(packed, out, i);
}

template <int BN, bool DUMP>
cudaError_t launch_tiles(const qvggt_weights *w, const signed char *wq8, const signed char *Xq8, const float *a_scale, int M, void *Y, long long ldy,
                   int *acc_debug, cudaStream_t st, long long wait_limit, int skip_loads)
{
    using L = Lay<BN>;
    static QvggtPerDevice cache;
    int max_workers = 0;
    cudaError_t e = qvggt_configure_kernel(gemm_c8_kernel<BN, DUMP>, THREADS, L::DYN_SMEM, 2, cache, &max_workers);
    if (e != cudaSuccess) return e;
    const int K = w->K, N = w->N;
    CUtensorMap map_x, map_w;
    if (!qvggt_make_map(&map_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, Xq8, K, M, K, BK, BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, wq8, K, N, K, BK, L::B_ROWS, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    const int total_tiles = ((M + 2 * BM - 1) / (2 * BM)) * ((N + BN - 1) / BN);
    const int workers = total_tiles < max_workers ? total_tiles : max_workers;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // see grid_dependency_wait()
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(workers * 2);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = L::DYN_SMEM;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_c8_kernel<BN, DUMP>, map_x, map_w, static_cast<uint16_t *>(Y), ldy, a_scale, (const float *)w->w_scale,
                              (const uint16_t *)w->bias, acc_debug, M, N, K, w->status, wait_limit, skip_loads);
}

// Whether tiles of 256 channels are the faster ones for this shape.  A narrow tile takes 0.55 of a wide one's time per K-block
// (0.15 against 0.27 us) and half its epilogue, so the number of rounds decides: narrow tiles win while they need at most 1.5
// times as many (wide / narrow, us: K = 4096, N = 1024: 13.4 / 9.4 at 1374 rows, 22.9 / 20.1 at 5496, but 24.0 / 26.1 at 8244,
// 32.9 / 33.8 at 10 992), and with K = 1024, where the epilogue behind the last K-block weighs as much as the K-blocks, also when
// they turn a single round into two (N = 1024: 7.0 / 5.4 at 1374 rows, 7.5 / 7.0 at 2748; two rounds into four: N = 3072
// 10.7 / 11.5 at 2748 rows).
bool wide_tiles(int M, int N, int K, int workers)
{
    const long long row_tiles = (M + 2 * BM - 1) / (2 * BM);
    const long long wide = (row_tiles * ((N + 255) / 256) + workers - 1) / workers;
    const long long narrow = (row_tiles * ((N + 127) / 128) + workers - 1) / workers;
    return !(2 * narrow <= 3 * wide || (K == 1024 && wide == 1));
}

template <bool DUMP>
cudaError_t launch(const qvggt_weights *w, const signed char *wq8, const signed char *Xq8, const float *a_scale, int M, void *Y, long long ldy,
                   int *acc_debug, cudaStream_t st, long long wait_limit, int skip_loads)
{
    if (wide_tiles(M, w->N, w->K, qvggt_sm_count() / 2)) return launch_tiles<256, DUMP>(w, wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, wait_limit, skip_loads);
    return launch_tiles<128, DUMP>(w, wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, wait_limit, skip_loads);
}

}  // namespace

cudaError_t qvggt_launch_gemm_c8(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y,
                                 long long ldy, int *acc_debug, cudaStream_t st)
{
    if (M == 0) return cudaSuccess;
    if (!w->Wq8) return cudaErrorNotSupported;      // the handle was prepared without the 8-bit-container copy
    if (!acc_debug && qvggt_gemm_small_wins(w, M, false, false)) return qvggt_launch_gemm_small(w, Xq8, w->Wq8, false, a_scale, false, M, Y, ldy, st);
    return acc_debug ? launch<true>(w, w->Wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0)
                     : launch<false>(w, w->Wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0);
}

cudaError_t qvggt_launch_unpack_w4(const qvggt_weights *w, signed char *w_scratch, cudaStream_t st)
{
    if (!w->Wq) return cudaErrorNotSupported;       // the handle holds no packed codes
    const long long n16 = (long long)w->N * w->K / 32;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n16 + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, unpack_w4_kernel, reinterpret_cast<const uint4 *>(w->Wq), reinterpret_cast<uint4 *>(w_scratch), n16);
}

cudaError_t qvggt_launch_gemm_c8_packed_weights(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y,
                                                long long ldy, signed char *w_scratch, int *acc_debug, cudaStream_t st)
{
    if (M == 0) return cudaSuccess;
    cudaError_t e = qvggt_launch_unpack_w4(w, w_scratch, st);
    if (e != cudaSuccess) return e;
    if (!acc_debug && qvggt_gemm_small_wins(w, M, false, false)) return qvggt_launch_gemm_small(w, Xq8, w_scratch, false, a_scale, false, M, Y, ldy, st);
    return acc_debug ? launch<true>(w, w_scratch, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0)
                     : launch<false>(w, w_scratch, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0);
}

cudaError_t qvggt_launch_gemm_c8_expanded(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y,
                                          long long ldy, const signed char *w_expanded, int *acc_debug, cudaStream_t st)
{
    if (M == 0) return cudaSuccess;
    if (!acc_debug && qvggt_gemm_small_wins(w, M, false, false)) return qvggt_launch_gemm_small(w, Xq8, w_expanded, false, a_scale, false, M, Y, ldy, st);
    return acc_debug ? launch<true>(w, w_expanded, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0)
                     : launch<false>(w, w_expanded, Xq8, a_scale, M, Y, ldy, acc_debug, st, ptx::kWaitLimitCycles, 0);
}

cudaError_t qvggt_launch_gemm_c8_starved(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y,
                                         long long ldy, long long wait_limit_cycles, cudaStream_t st)
{
    if (M == 0) return cudaSuccess;
    if (!w->Wq8) return cudaErrorNotSupported;
    return launch<false>(w, w->Wq8, Xq8, a_scale, M, Y, ldy, nullptr, st, wait_limit_cycles, 1);
}

cudaError_t qvggt_launch_gemm_c8_grouped(const qvggt_weights *w, const signed char *Xq8, const float *a_scale, int M, void *Y,
                                         long long ldy, int *acc_debug, cudaStream_t st)
{
    if (M == 0) return cudaSuccess;
    if (!w->Wq8 || w->bits != 4) return cudaErrorNotSupported;
    if (!acc_debug && qvggt_gemm_small_wins(w, M, false, true)) return qvggt_launch_gemm_small(w, Xq8, w->Wq8, false, a_scale, true, M, Y, ldy, st);
    if (acc_debug) return grp::launch<true, false>(w, Xq8, a_scale, M, Y, ldy, acc_debug, st);
    return (reinterpret_cast<uintptr_t>(a_scale) & 15u) == 0 ? grp::launch<false, true>(w, Xq8, a_scale, M, Y, ldy, acc_debug, st)
                                                            : grp::launch<false, false>(w, Xq8, a_scale, M, Y, ldy, acc_debug, st);
}
