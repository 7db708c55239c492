// W4A4 GEMM on codes held in 8-bit containers (Sec. 3.2: integer sum over the inner dimension, per-token and
// per-out-channel scales applied outside the sum), for sm_100a.
//
// tcgen05 has no 4-bit integer kind: whatever the storage format, the tensor core multiplies int8.  Here the
// producers already emit one code per byte (the quantize kernel for the activations, the offline weight
// preparation for the weights), so the tiles go from global memory straight into the 128-byte-swizzled operand
// stages by TMA and nothing in this kernel touches an operand byte with an ordinary instruction.
//
// Persistent and warp-specialised; a worker is a pair of CTAs on neighbouring SMs (tile 256 tokens x up to 256 channels, each CTA stages
// 128 token rows and half of the tile's weight rows; one thread of the leader CTA issues tcgen05.mma.cta_group::2.kind::i8 for both;
// accumulators int32 in tensor memory, two buffers of 256 columns).
//   warps 0..7   epilogue: TMEM -> registers -> scale, bias, bf16 -> swizzled staging -> TMA stores; no warp waits for another
//   warp  8      one elected thread issues tcgen05.mma and the commits that release stages / publish accumulators
//   warp  9      one thread per CTA issues the TMA loads of its half of every operand stage; both CTAs signal
//                the leader's "full" barrier (cta_group::2 form of the load)
// What bounds it, and what follows from it (us back to back; the earlier form took A and B of every tile from L2, read the channel
// parameters from shared memory for every 16 rows and wrote 128-byte lines with ordinary stores):
//  - At 256 channels the MMAs of a K-block take 512 cycles and its 32 KB per CTA take as long from L2 (64 bytes per cycle and SM), so with
//    K = 1024, where a tile's outputs are another 8 KB per K-block, the traffic of the SM was the limit.  With K = 1024 the eight
//    K-blocks of the token rows (128 KB) stay in shared memory for as long as a worker's tiles share them, and only weights stream: in runs of
//    four tiles where every worker gets at least four (make_plan()).  Calls with fewer share nothing; what they gained is due to the next points.
//  - The epilogue shares the shared-memory pipe with the operands: parameters in registers, outputs through the TMA engine.
//  - The outputs are marked first to leave L2, see ptx::policy_evict_first().
//  - Tiles that do not fill a round of workers are cut into narrower ones (make_plan()).
//   K = 1024, N = 3072 / 1024 / 4096 and K = 4096, N = 1024 at 10 992 rows: 27.4 / 13.0 / 36.8 / 32.8 -> 24.8 / 11.3 / 31.9 / 29.9;
//   at 137 400 rows K = 1024, N = 4096: 432 -> 394 (at the power limit).
// Every wait is bounded; on expiry the kernel records a code in *status and all roles fall through to the
// common exit, where tensor memory is released.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "gemm_c8_plan.cuh"
#include "gemm_common.cuh"
#include "qvggt_internal.cuh"
#include "sm100_ptx.cuh"
#include "tensor_map.cuh"
#include "unpack_w4.cuh"

namespace {

using namespace gemm_c8;
using gemmc::Ring;
using gemmc::STG_BYTES;

constexpr int ACC_BUFS = 2;        // TMEM accumulators: the epilogue of tile i overlaps the MMAs of tile i+1
constexpr int ACC_COLS = MAX_UNITS * UNIT;
constexpr int EPI_WARPS = 8;       // warp w: TMEM lane quarter w % 4, part w / 4 of the tile
constexpr int MMA_WARP = EPI_WARPS;
constexpr int TMA_WARP = EPI_WARPS + 1;
constexpr int THREADS = (EPI_WARPS + 2) * 32;
constexpr int TMEM_COLS = ACC_BUFS * ACC_COLS;

constexpr int STG_WARP = 16 * 2 * UNIT;                // staging of one epilogue warp: 16 rows x 64 bf16, 128-byte swizzled
constexpr int OFF_OPS = EPI_WARPS * STG_WARP;          // operands: [resident token rows,] ring of stages (1024-byte aligned)
static_assert(EPI_WARPS * 4 * STG_WARP <= OPS_BYTES, "the last tile is staged where the operands were");
constexpr int OFF_BAR = OFF_OPS + OPS_BYTES;           // full[MAX_STAGES] empty[MAX_STAGES] tfull[2] tempty[2]
constexpr int NBARS = 2 * MAX_STAGES + 2 * ACC_BUFS;
constexpr int OFF_TMEM = OFF_BAR + NBARS * 8;
constexpr int OFF_ABORT = OFF_TMEM + 4;
constexpr int DYN_SMEM = OFF_ABORT + 4 + 1024;         // slack to align the base to 1024 bytes
static_assert(DYN_SMEM <= 232448, "exceeds the 227 KB of shared memory a CTA may use");
static_assert(2 * (A_BYTES + MAX_UNITS * UNIT_BYTES) < (1 << 20), "transaction count of a stage must fit the barrier");

// A position in the ring of operand stages together with the parity of the phase it is in.
struct StageRing {
    int s = 0;
    uint32_t ph = 0, stage;
    __device__ __forceinline__ explicit StageRing(uint32_t ring) : stage(ring) {}
    __device__ __forceinline__ void advance(const Plan &plan, uint32_t ring)
    {
        stage += plan.stage_bytes;
        if (++s == plan.stages) { s = 0; ph ^= 1; stage = ring; }
    }
};

// RESIDENT (K = 1024): all eight K-blocks of a tile's token rows stay in shared memory for as long as the worker's tiles share
// them, and only weight rows stream.
// DUMP: also write the int32 sums to acc_debug (its own instantiation keeps that code out of the production kernel).
// wait_limit: bound of every device-side wait, in cycles.  skip_loads: the TMA producers issue nothing, so that the
// first wait for operands runs out (used only to exercise the timeout path; no asynchronous operation is in flight).
template <bool RESIDENT, bool DUMP>
__global__ void __launch_bounds__(THREADS, 1)
gemm_c8_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_wu,
               const __grid_constant__ CUtensorMap map_y, const __grid_constant__ Plan plan, const float *__restrict__ a_scale, const float *__restrict__ w_scale, const uint16_t *__restrict__ bias,
               int *__restrict__ acc_debug, int M, int N, int K, int *status, long long wait_limit, int skip_loads)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = ptx::smem_addr(smem);
    const uint32_t bar_full = sbase + OFF_BAR;
    const uint32_t bar_empty = bar_full + MAX_STAGES * 8;
    const uint32_t bar_tfull = bar_empty + MAX_STAGES * 8;
    const uint32_t bar_tempty = bar_tfull + ACC_BUFS * 8;
    const uint32_t ops = sbase + OFF_OPS, ring = ops + (RESIDENT ? RES_KB * A_BYTES : 0);
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + OFF_TMEM);
    volatile int *s_abort = reinterpret_cast<volatile int *>(smem + OFF_ABORT);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();                       // 0 = leader of the pair
    const int KB = RESIDENT ? RES_KB : K / BK;

    // full: the leader's arrive.expect_tx (bytes of both CTAs); empty, tfull: tcgen05.commit; tempty: the epilogue warps of both CTAs
    if (threadIdx.x < NBARS) {
        ptx::mbar_init(bar_full + 8 * threadIdx.x, threadIdx.x < NBARS - ACC_BUFS ? 1 : EPI_WARPS * 2);
        ptx::fence_mbar_init();
        if (threadIdx.x == 0) *s_abort = 0;
    }
    if (warp == MMA_WARP) { ptx::tmem_alloc_pair(ptx::smem_addr(s_tmem), TMEM_COLS); ptx::tmem_relinquish_pair(); }
    if (warp == TMA_WARP && lane == 0) {
        ptx::prefetch_tensormap(&map_x);
        ptx::prefetch_tensormap(&map_w);
        ptx::prefetch_tensormap(&map_wu);
        ptx::prefetch_tensormap(&map_y);
    }
    // Both CTAs meet: the leader's barriers exist before the peer's loads signal them.  The first tile is worked out on the way.
    __syncwarp();
    ptx::tc_fence_before_sync();
    ptx::cluster_arrive();
    Tiles tile(plan, blockIdx.x / 2);
    const int my_tiles = tile.count;
    ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *s_tmem;
    // Everything up to grid_dependency_wait() touches only kernel parameters and on-chip state: it may overlap the tail of the previous
    // kernel in the stream; the operands, the output buffer and the status word may not be touched before that kernel is done.
    // Only then is the next kernel let in as well: let in at once, the blocks of a quantize launch were placed beside those of the one in
    // front that still ran, and unevenly (layers, us at once / here: K = 1024, N = 3072, 325 rows 6.90 / 6.54, N = 1024, 493 rows
    // 6.41 / 6.03; K = 4096, N = 1024, 257 rows 11.9 / 11.2; 400 shapes of 100 - 11 000 rows 0.5 % less in the mean).
    auto previous_kernel_done = [] {
        ptx::grid_dependency_wait();
        ptx::grid_launch_dependents();
    };

    if (warp < EPI_WARPS) {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3, part = warp >> 2;    // TMEM lane quarter; of the units, part 0 takes the first half
        const uint32_t stg_addr = sbase + warp * STG_WARP;
        const uint32_t leader_tempty = ptx::map_to_cta(bar_tempty, 0);
        const uint64_t one2 = ptx::f32x2_one(N & 127);                       // N is a multiple of 128
        const uint64_t policy = ptx::policy_evict_first();
        bool alive = true;
        previous_kernel_done();
        for (int t = 0; t < my_tiles; ++t, tile.next()) {
            const int m0 = tile.row * (2 * BM) + (int)rank * BM + quarter * 32;
            const int b = t & 1;
            // A tile of one unit is shared by rows: 16 of a warp's 32 each.
            const bool by_rows = tile.units == 1;
            const int first = by_rows ? 0 : part * ((tile.units + 1) / 2), units = by_rows ? 1 : part ? tile.units / 2 : (tile.units + 1) / 2;
            const int n0 = (tile.unit + first) * UNIT;         // first channel of this warp
            // Scales and biases of channels 8 e + 2 (lane mod 4) and + 1 of each unit, in the layout of the accumulator fragments and
            // straight into registers: read from shared memory for every 16 rows they took as much of its bandwidth as the outputs.
            uint64_t w2[2][8];
            uint32_t c2[2][8];
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int n = n0 + (k < units ? k * UNIT : 0) + 8 * e + 2 * (lane & 3);
                    w2[k][e] = __ldg(reinterpret_cast<const unsigned long long *>(w_scale + n));
                    c2[k][e] = bias ? __ldg(reinterpret_cast<const uint32_t *>(bias + n)) : 0u;
                }
            uint64_t as2[2][2];                                // rows lane / 4 + 8 h of the warp's 16 u .. 16 u + 15
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int gm = m0 + 8 * u + (lane >> 2);
                const float as = gm < M ? __ldg(a_scale + gm) : 0.0f;
                as2[u >> 1][u & 1] = ptx::f32x2_pack(as, as);
            }
            {
                int ok = 1;
                if (lane == 0) ok = (alive && ptx::mbar_wait(bar_tfull + 8 * b, (t >> 1) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_ACCUM, 0, wait_limit)) ? 1 : 0;
                alive = __shfl_sync(0xFFFFFFFFu, ok, 0) != 0;
            }
            ptx::tc_fence_after_sync();
            // Behind the last tile's MMAs nothing uses the operands' memory any more: each of its 16 x 64 pieces has a staging tile there,
            // where the others wait for the store of the piece before them (0.13 us of a launch of one tile per worker, us: K = 1024,
            // N = 4096, 600 rows 6.03 / 5.90; K = 4096, N = 1024, 4122 rows 13.54 / 13.40).
            const bool last = t == my_tiles - 1;
            const uint32_t stg = last ? ops + warp * (4 * STG_WARP) : stg_addr, stg_next = last ? STG_WARP : 0;
            if (alive) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (k < units) {
                        uint32_t raw[2][32];
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            ptx::tmem_ld_16x256b_x8(tmem_base + (static_cast<uint32_t>(quarter * 32 + 16 * u) << 16) + b * ACC_COLS + (first + k) * UNIT, raw[u]);
                        ptx::tmem_ld_wait();
                        if (k == units - 1) {                  // tensor memory goes back to the MMA thread
                            ptx::tc_fence_before_sync();
                            __syncwarp();
                            // (nobody waits for the last tiles' arrivals: none may be on its way when the leader CTA exits)
                            if (lane == 0 && t + ACC_BUFS < my_tiles) ptx::mbar_arrive_cluster(leader_tempty + 8 * b);
                        }
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int m = m0 + 16 * u, n = n0 + k * UNIT;
                            if (by_rows && u != part) continue;
                            gemmc::finish_16x64_tma(raw[u], as2[u], w2[k], c2[k], stg + (2 * k + u) * stg_next, !last, &map_y, n, m, m < M, lane, one2, policy);
                            if (DUMP && acc_debug) gemmc::dump_16x64<0>(acc_debug + (long long)m * N + n, N, raw[u], M - m, lane);
                        }
                    }
                }
            }
        }
        if (lane == 0) ptx::tma_store_wait_read<0>();
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------------------ MMA issuer (one thread of the leader CTA)
        // The thread is chosen by elect.sync, not by its lane number: the assembler then knows that one thread is active and keeps
        // the descriptors in uniform registers, where tcgen05 wants them (behind `lane == 0` every one is moved there anew, which
        // made this loop, at 545 cycles per K-block, the bound of the kernel).
        previous_kernel_done();                                            // the limit of the waits bounds this kernel's own work only
        if (rank == 0 && ptx::elect_one()) {
            bool alive = true;
            StageRing r(ring);
            int left = my_tiles * KB - plan.stages;                        // K-blocks for whose stage a load will wait
            for (int t = 0; t < my_tiles && alive; ++t, tile.next()) {
                const int b = t & 1;
                if (t >= ACC_BUFS) {
                    alive = ptx::mbar_wait_cluster(bar_tempty + 8 * b, ((t >> 1) - 1) & 1, s_abort, status, QVGGT_DEV_TIMEOUT_TMEM_FREE, wait_limit);
                    if (!alive) break;
                    ptx::tc_fence_after_sync();
                }
                const uint32_t d_tmem = tmem_base + b * ACC_COLS;
                auto k_blocks = [&](auto units) {                          // the width is a constant of the instruction descriptor
                    constexpr uint32_t idesc = ptx::idesc_i8(2 * BM, decltype(units)::value * UNIT);
                    for (int kb = 0; kb < KB; ++kb) {
                        alive = ptx::mbar_wait_cluster(bar_full + 8 * r.s, r.ph, s_abort, status, QVGGT_DEV_TIMEOUT_FULL, wait_limit);
                        if (!alive) break;
                        ptx::tc_fence_after_sync();
                        gemmc::mma_kblock_i8<true>(d_tmem, RESIDENT ? ops + kb * A_BYTES : r.stage, RESIDENT ? r.stage : r.stage + A_BYTES, idesc, kb == 0);
                        if (left-- > 0) ptx::mma_commit_pair(bar_empty + 8 * r.s, 3);   // frees the stage in both CTAs
                        if (kb == KB - 1) ptx::mma_commit_pair(bar_tfull + 8 * b, 3);
                        r.advance(plan, ring);
                    }
                };
                if (tile.units == 4) k_blocks(std::integral_constant<int, 4>());
                else if (tile.units == 3) k_blocks(std::integral_constant<int, 3>());
                else if (tile.units == 2) k_blocks(std::integral_constant<int, 2>());
                else k_blocks(std::integral_constant<int, 1>());
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ TMA producer (one thread per CTA)
        const uint32_t leader_full = ptx::map_to_cta(bar_full, 0);
        previous_kernel_done();
        if (!skip_loads && ptx::elect_one()) {
            bool alive = true;
            StageRing r(ring);
            int ahead = plan.stages, resident = -1;                        // K-blocks that need not wait for their stage; resident row tile
            for (int t = 0; t < my_tiles && alive; ++t, tile.next()) {
                const int m0 = tile.row * (2 * BM) + (int)rank * BM;
                const int n0 = tile.unit * UNIT + (int)rank * (tile.units * (UNIT / 2));
                // the box of weight rows may reach beyond a narrower tile: rows that nothing reads
                auto k_blocks = [&](const CUtensorMap *map, auto rows, int box_units) {
                    constexpr bool ROWS = decltype(rows)::value;
                    const uint32_t bytes = 2 * ((ROWS ? A_BYTES : 0) + box_units * UNIT_BYTES);
                    for (int kb = 0; kb < KB; ++kb) {
                        if (--ahead < 0) {
                            alive = ptx::mbar_wait(bar_empty + 8 * r.s, r.ph ^ 1, s_abort, status, QVGGT_DEV_TIMEOUT_EMPTY, 0, wait_limit);
                            if (!alive) break;
                        }
                        const uint32_t full = leader_full + 8 * r.s;
                        // the leader's barrier expects the bytes of both CTAs; the peer's completions may arrive first
                        // (the count goes negative for a while), the phase cannot end before the leader has arrived
                        if (rank == 0) ptx::mbar_arrive_expect_tx(bar_full + 8 * r.s, bytes);
                        // The K-block of the resident rows that this overwrites was last read RES_KB K-blocks ago, and the MMAs up to
                        // plan.stages <= RES_KB K-blocks ago are known to be done.
                        if (ROWS) ptx::tma_load_2d_pair(&map_x, full, RESIDENT ? ops + kb * A_BYTES : r.stage, kb * BK, m0);
                        ptx::tma_load_2d_pair(map, full, RESIDENT ? r.stage : r.stage + A_BYTES, kb * BK, n0);
                        r.advance(plan, ring);
                    }
                };
                const std::true_type yes;
                const std::false_type no;
                const bool load_rows = !RESIDENT || tile.row != resident, whole = t < plan.runs * plan.run + plan.rounds;
                resident = tile.row;
                if (load_rows) {
                    if (whole) k_blocks(&map_w, yes, plan.wide);
                    else k_blocks(&map_wu, yes, plan.cut);
                } else {
                    if (whole) k_blocks(&map_w, no, plan.wide);
                    else k_blocks(&map_wu, no, plan.cut);
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

template <bool RESIDENT, bool DUMP>
cudaError_t launch_plan(const qvggt_weights *w, const signed char *wq8, const signed char *Xq8, const float *a_scale, int M, void *Y, long long ldy,
                        int *acc_debug, cudaStream_t st, long long wait_limit, int skip_loads)
{
    static QvggtPerDevice cache;
    int workers = 0;
    cudaError_t e = qvggt_configure_kernel(gemm_c8_kernel<RESIDENT, DUMP>, THREADS, DYN_SMEM, 2, cache, &workers);
    if (e != cudaSuccess) return e;
    const int K = w->K, N = w->N;
    const Plan plan = make_plan(M, N, K, workers, &workers);
    CUtensorMap map_x, map_w, map_wu, map_y;
    if (!qvggt_make_map(&map_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, Xq8, K, M, K, BK, BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, wq8, K, N, K, BK, plan.wide * (UNIT / 2), CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_wu, CU_TENSOR_MAP_DATA_TYPE_UINT8, wq8, K, N, K, BK, plan.cut * (UNIT / 2), CU_TENSOR_MAP_SWIZZLE_128B) ||
        !qvggt_make_map(&map_y, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Y, N, M, (uint64_t)ldy * 2, UNIT, 16, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // see grid_dependency_wait()
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(workers * 2);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = DYN_SMEM;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_c8_kernel<RESIDENT, DUMP>, map_x, map_w, map_wu, map_y, plan, a_scale,
                              (const float *)w->w_scale, (const uint16_t *)w->bias, acc_debug, M, N, K, w->status, wait_limit, skip_loads);
}

template <bool DUMP>
cudaError_t launch(const qvggt_weights *w, const signed char *wq8, const signed char *Xq8, const float *a_scale, int M, void *Y, long long ldy,
                   int *acc_debug, cudaStream_t st, long long wait_limit, int skip_loads)
{
    if (w->K == RES_KB * BK) return launch_plan<true, DUMP>(w, wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, wait_limit, skip_loads);
    return launch_plan<false, DUMP>(w, wq8, Xq8, a_scale, M, Y, ldy, acc_debug, st, wait_limit, skip_loads);
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
