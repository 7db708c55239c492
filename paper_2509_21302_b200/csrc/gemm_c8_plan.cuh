// How the TMA-fed GEMM (gemm_c8.cu) cuts its output into tiles and deals them to its workers: plain arithmetic, the same on the host and
// in the kernel, with no CUDA header, so that it can be compiled and checked by itself.
#pragma once
#ifndef __CUDACC__
#include <algorithm>
#define __host__
#define __device__
#define __forceinline__ inline
using std::min;
#endif

namespace gemm_c8 {

constexpr int BM = 128;            // token rows per CTA (TMEM lanes)
constexpr int BK = 128;            // codes along K per stage = one 128-byte swizzled row
constexpr int UNIT = 64;           // channels per unit of work; a tile is 256 token rows x 1 .. 4 units
constexpr int MAX_UNITS = 4;

constexpr int A_BYTES = BM * BK;                       // one K-block of a CTA's token rows: 16 KB
constexpr int UNIT_BYTES = UNIT / 2 * BK;              // one K-block of a CTA's half of a unit's weight rows: 4 KB
constexpr int RES_KB = 8;                              // K-blocks of the token rows that stay resident (K = 1024)
constexpr int RUN = 4;                                 // consecutive tiles of a worker that share them, see make_plan()
constexpr int OPS_BYTES = 208 * 1024;                  // operands: [resident token rows,] ring of stages
constexpr int MAX_STAGES = 12;

// How the tiles are dealt to the workers; filled in by make_plan(), so that no thread of the kernel divides.  Work is counted in units of 256
// token rows x 64 channels; whole tiles are numbered along the channels, row tile by row tile.
struct Plan {
    int NU, NT;                  // units and whole tiles of a row tile: NT tiles of `narrow` units, the first `wider` of them one unit more
    int narrow, wider, wide;     // wide: most units of a whole tile
    int runs, run;               // each worker first takes `runs` times `run` consecutive tiles,
    int rounds;                  // then so many single tiles,
    int cut;                     // then at most one piece of `cut` units
    int workers, row_tiles;
    int behind_row, behind_unit, behind_first, behind_pieces;   // where the pieces begin, how many the begun row tile has, how many a row tile has
    unsigned long long div_nt, div_pieces;                      // see div()
    int stages, stage_bytes;
    // x / d for x d < 2^40, with m = ceil(2^40 / d)
    static __host__ __device__ unsigned long long reciprocal(int d) { return ((1ull << 40) + d - 1) / d; }
    static __host__ __device__ __forceinline__ int div(int x, unsigned long long m) { return (int)((x * m) >> 40); }
};

// The tiles of one worker, in order.
struct Tiles {
    int row, unit, units;                                 // the current tile: row tile, first unit, how many units
    int count;                                            // of tiles
    __device__ __forceinline__ Tiles(const Plan &plan, int worker_) : row(0), unit(0), units(0), worker(worker_), t(0), p(plan)
    {
        // behind the whole tiles: what is left of a row tile, then whole row tiles
        const int i = worker - p.behind_first, full = i < 0 ? 0 : Plan::div(i, p.div_pieces);
        behind_row = p.behind_row + (i < 0 ? 0 : 1 + full);
        behind_unit = i < 0 ? p.behind_unit + worker * p.cut : (i - full * p.behind_pieces) * p.cut;
        count = p.runs * p.run + p.rounds + (behind_row < p.row_tiles ? 1 : 0);
        at = worker * p.run;
        in_run = 0;
        next();
    }
    __device__ __forceinline__ void next()     // (one beyond the last is never used)
    {
        const int in_runs = p.runs * p.run;
        if (t < in_runs + p.rounds) {
            if (t >= in_runs) at = in_runs * p.workers + (t - in_runs) * p.workers + worker;
            row = Plan::div(at, p.div_nt);
            const int j = at - row * p.NT;
            unit = j * p.narrow + min(j, p.wider);
            units = p.narrow + (j < p.wider ? 1 : 0);
            ++at;
            if (++in_run == p.run) { in_run = 0; at += (p.workers - 1) * p.run; }
        } else {
            row = behind_row;
            unit = behind_unit;
            units = min(p.cut, p.NU - unit);
        }
        ++t;
    }

private:
    int worker, t, at, in_run, behind_row, behind_unit;
    const Plan &p;
};

// Whole tiles first, as many as every worker gets alike, and what remains (less than a round of them) cut into pieces as narrow as one more
// round allows: a launch of one round at K = 4096 takes 8.0 us with tiles of 64 channels, 8.2 - 8.7 with 128, 11.2 with 192 and 13.5 with 256
// (K = 4096, N = 1024: 32.8 -> 29.9 us at 10 992 rows, 13.7 -> 11.2 at 2748; cut in halves only, or not at all, before).
// A launch of nothing but pieces takes those of 64 channels only where they leave half of the chip free, at K = 4096 two thirds.  They gain
// 0.25 us over 128 channels at most, and the blocks of the quantize launch behind this one, let in while it runs, crowd on the SMs that it leaves.
// Layers in a replayed graph, us with 64 / 128 channels (n: pieces of 64 on 74 pairs of SMs):
//   K = 1024: N = 1024, 204 - 219 rows (n = 16) 5.5 / 5.8, 455 - 492 (32) 5.9 / 6.0 - 6.15, 666 - 759 (48) 7.0 / 6.4, 964 - 996 (64) 7.15 / 6.9;
//             N = 3072 (48), 141 - 195 rows 5.65 / 5.8, 222 - 256 6.04 / 5.9; N = 4096 (64), 174 - 230 rows 6.55 / 5.95
//   K = 4096: N = 1024, 192 - 209 rows (16) 10.26 / 10.52, 260 - 300 (32) 11.1 / 11.2, 369 - 458 (32) 11.95 / 11.4, 793 - 931 (64) 12.8 - 13.8 / 13.0 - 13.2;
//             N = 3072 (48) 12.1 / 11.3; N = 4096 (64) 12.3 / 11.4
// and the mean over 260 layers, 64 against 128 channels, K = 1024 / 4096: up to n = 24 0.972 / 0.986, 25 - 37 0.979 / 1.014, 38 - 49
// 1.026 / 1.020, 50 - 74 1.04 / 1.07.  Behind whole tiles, where the chip is busy anyway, the narrowest win at any number (K = 4096, N = 1024, 7975
// rows 50.8 / 52.4).
// With resident token rows the whole tiles are dealt in runs of four, as far as every worker gets as many: from 296 tiles on 74 pairs of SMs
// (N = 4096: 4609 rows, N = 3072: 6145, N = 1024: 18 689).  In smaller calls, and for the tiles left over, a worker's tiles lie a round apart
// and each loads its token rows anew.  Longer runs save more loads, but the chip's stores then
// scatter over more rows of the result, which costs DRAM more than the loads do; N = 4096, us at 10 992 / 43 968 / 137 400 rows, runs of
// 1: 37.9 / 135.7 / 412, 2: 37.6 / 138.5 / 418, 4: 35.1 / 129.5 / 397, 8: 36.5 / 140 / 437, 16: 38.0 / 142 / 439 (without the L2 policy
// of the stores).
inline Plan make_plan(int M, int N, int K, int max_workers, int *workers)
{
    const bool resident = K == RES_KB * BK;
    Plan p = {};
    p.row_tiles = (M - 1) / (2 * BM) + 1;
    p.NU = N / UNIT;
    p.NT = (p.NU + MAX_UNITS - 1) / MAX_UNITS;
    // Where N is no multiple of 256, tiles of 128 channels may fit two rounds although those of up to 256 are just more than one, and two such
    // rounds cost less than one of 256 and one of 64 (layers, us, 256 + 64 / 128 + 128: K = 4096, N = 1152, 3867 rows 34.2 / 31.1, N = 640, 6500 rows
    // 42.3 / 39.0; K = 1024 11.55 / 11.16 and 12.95 / 12.55; three or more rounds: K = 1024, N = 1152, 8100 rows 17.35 / 17.7).
    if (p.row_tiles * p.NT > max_workers && p.row_tiles * (p.NU / 2) <= 2 * max_workers) p.NT = p.NU / 2;
    p.narrow = p.NU / p.NT;
    p.wider = p.NU % p.NT;
    p.wide = p.narrow + (p.wider ? 1 : 0);
    p.div_nt = Plan::reciprocal(p.NT);
    const int tiles = p.row_tiles * p.NT;
    p.run = resident ? RUN : 1;
    p.runs = tiles / (p.run * max_workers);
    const int each = tiles / max_workers, first = each * max_workers, j = first % p.NT;
    p.rounds = each - p.runs * p.run;
    p.behind_row = first / p.NT;
    p.behind_unit = j * p.narrow + (j < p.wider ? j : p.wider);
    int pieces = 0;
    for (p.cut = 1;; ++p.cut) {
        p.behind_first = (p.NU - p.behind_unit + p.cut - 1) / p.cut;
        p.behind_pieces = (p.NU + p.cut - 1) / p.cut;
        pieces = p.behind_first + (p.row_tiles - 1 - p.behind_row) * p.behind_pieces;
        const bool crowding = p.cut == 1 && each == 0 && (resident ? 2 : 3) * pieces > max_workers;
        if ((pieces <= max_workers && !crowding) || p.cut == p.wide) break;
    }
    p.div_pieces = Plan::reciprocal(p.behind_pieces);
    *workers = p.workers = each == 0 ? pieces : max_workers;
    const int widest = each == 0 ? p.cut : p.wide;
    p.stage_bytes = (resident ? 0 : A_BYTES) + widest * UNIT_BYTES;
    const int fit = (OPS_BYTES - (resident ? RES_KB * A_BYTES : 0)) / p.stage_bytes, most = resident ? RES_KB : MAX_STAGES;
    p.stages = fit < most ? fit : most;
    return p;
}

}  // namespace gemm_c8
