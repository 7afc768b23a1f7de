// Host-side estimates that choose the multi-step kernel of a mid-size FP32
// lattice and its shape (lbm_capi.cu: plan_multi).
#include <algorithm>

#include "lbm_kernels.h"
#include "wave.cuh"

namespace plbm {

// The plan with the least estimated time per step.  The estimate is a fit
// (SM clocks) to sweeps over K, tile height and R on lattices of 128 x 32 to
// 2048 x 512 nodes, whose best plans it names within a few per cent: a launch
// costs 3900 plus 85 per row a block holds (the loads and stores of 64
// columns of 8 planes), a step 240 (barrier and the dependency chain of one
// row) plus 115 issue cycles per row of the busiest scheduler.  Blocks of one
// SM share its schedulers.  No sweep had sides along x and y, and the estimate
// has no term for their rules: 0.74 us a step for the 201 x 201 square, which
// takes 1.38; there it orders the plans as if the lattice were a channel.  The
// registers per thread that limit the blocks of an SM are rounded up over the
// boundary kinds: 56 to 78 at R = 1, 89 to 118 at R = 2, 123 to 128 above.
double tile_plan(int nx, int ny, int bc_x, int bc_y, int sms, TilePlan *out) {
    const bool open_x = bc_x == BC_SIDES, open_y = bc_y == BC_SIDES || bc_y == BC_WALLS;
    double best = 0.0;
    *out = TilePlan{};
    if ((long long)nx * ny > TILE_MAX_NODES) return best;
    for (int K = 4; K <= 12; K += 2) {
        for (int R = 1; R <= TILE_MAX_ROWS; ++R) {
            // m blocks per SM; m = 9: the tallest tiles R rows per warp allow
            for (int m = 1; m <= 9; ++m) {
                TilePlan p;
                p.steps = K;
                p.rows = R;
                const int cx = tile_columns(p, nx, open_x);
                const int cy = std::max(1, sms * m / cx);
                p.ty = m < 9 ? (ny + cy - 1) / cy : TILE_MAX_WARPS * R - 2 * K;
                if (p.ty < 1) continue;
                const int rows = tile_rows(p.ty, ny, open_y, K);
                if (rows > TILE_MAX_WARPS * R) continue;
                const long long blocks = (long long)cx * ((ny + p.ty - 1) / p.ty);
                const long long per_sm = (blocks + sms - 1) / sms;
                const int warps = (rows + R - 1) / R;
                const int fit = std::max(1, 65536 / (warps * 32 * (R == 1 ? 80 : 128)));
                const long long together = std::min<long long>(per_sm, fit);
                const long long waves = (per_sm + together - 1) / together;
                const bool whole = open_y && rows == ny;       // no rows go wrong
                double steps = 0.0;
                for (int s = 0; s < K; ++s) {
                    const int live = whole ? rows : std::max(p.ty, rows - 2 * s);
                    const int per_sched = ((live + R - 1) / R + 3) / 4;
                    steps += 240.0 + 115.0 * R * per_sched * together;
                }
                const double t = (3900.0 + waves * (steps + 85.0 * rows * together)) / K;
                if (out->steps == 0 || t < best) {
                    best = t;
                    *out = p;
                }
            }
        }
    }
    return best / 2000.0;      // us at about 2 GHz
}

// The plan with the least estimated time per step among 4 and 5 steps and
// segments of 16 to 128 rows: warps of one scheduler take 150 clocks per level
// and row each, 375 at least (a lone warp's dependency chain); 15 (12) of them
// are resident per SM with 4 (5) steps, so a lattice is marched in rounds of
// that many strip-segments per SM and the last round may be short; the reads
// and writes of a launch pass at 5.7 GB/ms, 9 when the state stays in L2.
// Against sweeps over both parameters the plan is within 5 % of the best at
// 2048^2 (5 steps, 48 rows: 13.0 us), 4096 x 2048 (5, 96: 23.5) and 4096 x 3900.
double wave_plan(int nx, int ny, int sms, WavePlan *out) {
    double best = 0.0;
    const double nodes = (double)nx * ny;
    for (int K = 4; K <= 5; ++K) {
        const int S = wave::stride_of(wave::halo(K)), slots = K == 4 ? 15 : 12;
        const long long tiles = (nx + S - 1) / S;
        for (int rows = 16; rows <= 128; rows += 8) {
            const int r = rows < ny ? rows : ny;
            const long long items = tiles * ((ny + r - 1) / r);
            const long long per_sm = (items + sms - 1) / sms;
            auto level = [](long long warps) {
                const double t = 150.0 * (double)((warps + 3) / 4);
                return t < 375.0 ? 375.0 : t;
            };
            const double pos = r + 2 * K;
            double us = pos * K * (double)(per_sm / slots) * level(slots);
            if (per_sm % slots) us += pos * K * level(per_sm % slots);
            us /= 2070.0;
            const double bytes = nodes * 32.0 * (0.9 * 64.0 / S * pos / r + 1.0);
            const double mem = bytes / (nodes * 64.0 > 1.1e8 ? 5.7e6 : 9e6);
            us = ((us > mem ? us : mem) + 2.0) / K;
            if (best == 0.0 || us < best) {
                best = us;
                out->steps = K;
                out->rows = rows;
            }
        }
    }
    return best;
}

// Rows per segment of a lattice that fills the GPU several times over: 12
// strip-segments are resident per SM, each marches its rows and 2 K more, and
// the last round should be full.  Fewest row positions over all rounds among
// segments of 64 to 256 rows (128 and 256 rows whatever the lattice, before:
// 4096^2 FP32 49.4 us a step, at 92 rows 44.4; FP16 56.4, at 171 rows 54.7;
// 8192^2 FP32 165.3, at 241 rows 164.0).
int wave_rows(int precision, int nx, int ny, int K, int sms) {
    const int stride = wave::stride_of(precision == PREC_FP32 ? wave::halo(K) : wave::HALO16);
    const long long tiles = (nx + stride - 1) / stride, slots = 12LL * sms;
    int best = ny < 256 ? ny : 256;
    long long best_cost = -1;
    for (long long segs = (ny + 255) / 256; segs <= (ny + 63) / 64; ++segs) {
        const int rows = (int)((ny + segs - 1) / segs);
        const long long rounds = (tiles * ((ny + rows - 1) / rows) + slots - 1) / slots;
        const long long cost = rounds * (rows + 2 * K);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = rows;
        }
    }
    return best;
}

}  // namespace plbm
