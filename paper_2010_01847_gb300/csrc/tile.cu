// Multi-step stream-collide for mid-size FP32 lattices: K time steps per
// launch on tiles held in registers.
//
// Between the lattices one cluster can hold (resident.cu) and those whose
// strips fill the GPU (wave.cu) a step is too short to be worth a launch of
// its own: one launch per step costs 2-4 us whatever it does.  Here the
// lattice is cut into about one tile per SM: 64 columns (two adjacent nodes
// per lane) by as many rows as the block's warps hold, R rows per warp, all
// 8 planes of every node in registers (at R = 4 the compiler keeps 32 to 60
// bytes of a thread's 128-register state in local memory).  A block loads its tile and a halo,
// advances it K steps and writes the tile's own nodes; the outermost ring of
// the halo goes wrong one node per step.  Within a warp the c_y neighbours
// are the thread's other rows and the c_x neighbours come from the lane's
// other node or by a shuffle; only the 6 planes that cross from one warp's
// rows to the next go through shared memory (two buffers, one barrier per
// step).  The rows of a step are independent, so the collision's dependency
// chain overlaps across them.
//
// The wrap, seam, walls and sides are worked out from each node's position,
// so any nx, ny and boundary kind runs here; beyond a wall or side the tile
// computes values that the treatments of Section 2.5 replace wherever a valid
// node would pull them.  The arithmetic is that of every FP32 kernel
// (collide_f32 node by node, the same operations in the same order), so the
// results are bit-identical to single steps.
//
// Launches are chained with programmatic dependent launch: the next launch
// works out its positions while the previous one ends, and waits for it
// before its first load.
#include "lbm_kernels.h"

namespace plbm {
namespace {

struct TileArgs {
    const float *src;
    float *dst;
    long long plane;
    int nx, ny, bc_x, bc_y;
    int tx, ty, tiles_x;    // own nodes of a tile, tiles per row of tiles
    int hx, hy;             // halo columns and rows (periodic axes and inner cuts)
    int steps;              // steps of this launch, <= hx and hy
};

__device__ __forceinline__ int wrap(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

__device__ __forceinline__ void seam_jump(float (&d)[8], float lo_axis, float lo_diag,
                                          float hi_axis, float hi_diag) {
    d[0] = d[0] + lo_axis;                                 // Eq. 59
    d[4] = d[4] + lo_diag;
    d[7] = d[7] + lo_diag;
    d[2] = d[2] - hi_axis;                                 // Eq. 60
    d[5] = d[5] - hi_diag;
    d[6] = d[6] - hi_diag;
}

// Section 2.5 on the lanes' nodes that lie on x side `side` (on_a, on_b) and
// on no y side: an isothermal side sets the node (Eq. 55), any other one its
// three unknown populations (Eqs. 57-58).
__device__ __forceinline__ void apply_x_side(float (&da)[8], float (&db)[8], const Coef<float> &k,
                                             bool on_a, bool on_b, int side) {
    if (k.side_kind[side] == SIDE_ISOTHERMAL) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float v = i < 4 ? k.side_axis[side] : k.side_diag[side];
            da[i] = on_a ? v : da[i];
            db[i] = on_b ? v : db[i];
        }
        return;
    }
    const int in0 = side ? 0 : 2, in1 = side ? 4 : 5, in2 = side ? 7 : 6;     // incident
    const int out0 = side ? 2 : 0, out1 = side ? 5 : 4, out2 = side ? 6 : 7;  // unknown
    const float ta = (da[in0] + da[in1] + da[in2]) + k.side_flux[side];
    const float tb = (db[in0] + db[in1] + db[in2]) + k.side_flux[side];
    da[out0] = on_a ? k.u_axis * ta : da[out0];
    da[out1] = on_a ? k.u_diag * ta : da[out1];
    da[out2] = on_a ? k.u_diag * ta : da[out2];
    db[out0] = on_b ? k.u_axis * tb : db[out0];
    db[out1] = on_b ? k.u_diag * tb : db[out1];
    db[out2] = on_b ? k.u_diag * tb : db[out2];
}

// Every warp of the block, from whichever loop it is in.
__device__ __forceinline__ void block_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// SEAM, WALLS, SIDES: which boundary rules the lattice has (the others are
// not compiled).
template <int R, bool SEAM, bool WALLS, bool SIDES>
__global__ void __launch_bounds__(TILE_MAX_WARPS * 32, 1)
tile_steps(const TileArgs a, const Coef<float> k) {
    // [buffer][warp][1, 4, 5 of its top row, 3, 6, 7 of its bottom row, each of
    // the lane's first and second column][lane]
    extern __shared__ float edges[];
    constexpr int EDGE = 12 * 32;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // uniform in the warp
    const int by = blockIdx.x / a.tiles_x, bx = blockIdx.x - by * a.tiles_x;
    const bool open_x = SIDES && a.bc_x == BC_SIDES, sides_y = SIDES && a.bc_y == BC_SIDES;
    const bool walls = WALLS && a.bc_y == BC_WALLS;
    const bool open_y = walls || sides_y;

    // the tile's own nodes and the first column and row the block holds
    // (a tile at an x side needs no halo there and owns that many more)
    const int x0 = open_x && bx ? a.hx + bx * a.tx : bx * a.tx, y0 = by * a.ty;
    const int x1 = open_x ? (bx == a.tiles_x - 1 ? a.nx : a.hx + (bx + 1) * a.tx)
                          : min(x0 + a.tx, a.nx);
    const int y1 = min(y0 + a.ty, a.ny);
    const int xs = open_x ? max(x0 - a.hx, 0) : x0 - a.hx;
    const int ys = open_y ? max(y0 - a.hy, 0) : y0 - a.hy;
    const int ye = open_y ? min(y1 + a.hy, a.ny) : y1 + a.hy;     // rows [ys, ye) are needed
    const int ca = xs + 2 * lane;                                 // the lane's columns ca, ca + 1
    const int xa = wrap(ca, a.nx), xb = wrap(ca + 1, a.nx);
    const bool xa_lo = xa == 0, xa_hi = xa == a.nx - 1, xb_lo = xb == 0, xb_hi = xb == a.nx - 1;
    // some lane of the warp pulls across the seam / lies on the low (1) or
    // high (2) x side
    const bool seam = SEAM && a.bc_x == BC_GRADIENT &&
                      __any_sync(0xffffffffu, xa_lo || xa_hi || xb_lo || xb_hi);
    const unsigned x_sides = !open_x ? 0u : (__any_sync(0xffffffffu, xa_lo || xb_lo) ? 1u : 0u) |
                                                (__any_sync(0xffffffffu, xa_hi || xb_hi) ? 2u : 0u);
    const float lo_axis_a = xa_lo ? k.jump_axis : 0.f, lo_diag_a = xa_lo ? k.jump_diag : 0.f;
    const float hi_axis_a = xa_hi ? k.jump_axis : 0.f, hi_diag_a = xa_hi ? k.jump_diag : 0.f;
    const float lo_axis_b = xb_lo ? k.jump_axis : 0.f, lo_diag_b = xb_lo ? k.jump_diag : 0.f;
    const float hi_axis_b = xb_hi ? k.jump_axis : 0.f, hi_diag_b = xb_hi ? k.jump_diag : 0.f;
    // 8-byte accesses where the lane's pair is adjacent and aligned
    const bool wide = a.nx % 2 == 0 && xs % 2 == 0;
    const int r0 = warp * R;                                      // the warp's rows ys + r0 ..
    int yr[R];
    // 4 bits per row: on the low / high y side, at the low / high wall
    unsigned y_rules = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        yr[r] = wrap(ys + r0 + r, a.ny);
        const unsigned at = (yr[r] == 0 ? 1u : 0u) | (yr[r] == a.ny - 1 ? 2u : 0u);
        y_rules |= (sides_y ? at : walls ? at << 2 : 0u) << (4 * r);
    }
    // the steps after which none of the warp's rows is valid any more
    int alive = 1 << 20;
    const int rows = ye - ys;
    if (!(open_y && ys == 0)) alive = min(alive, r0 + R - 1);
    if (!(open_y && ye == a.ny)) alive = min(alive, rows - 1 - r0);
    if (r0 >= rows) alive = -1;

    // the lane's nodes of each row: columns ca (fa) and ca + 1 (fb), as
    // scalars (a packed pair instruction takes two issue cycles like the two
    // scalar ones it replaces, and its operands would have to be moved into
    // register pairs)
    float fa[R][8], fb[R][8];
    // the previous launch's results (nothing above read them)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (alive >= 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float *p = a.src + (long long)yr[r] * a.nx;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float *q = p + (long long)i * a.plane;
                const float2 v = wide ? __ldcg(reinterpret_cast<const float2 *>(q + xa))
                                      : make_float2(__ldcg(q + xa), __ldcg(q + xb));
                fa[r][i] = v.x;
                fb[r][i] = v.y;
            }
        }
    }
    // (the outermost warps read their own edges: rows no valid node needs)
    const int w_lo = max(warp - 1, 0), w_hi = min(warp + 1, warps - 1);
    float *const mine = edges + warp * EDGE + lane, *const lower = edges + w_lo * EDGE + lane,
                 *const upper = edges + w_hi * EDGE + (6 * 32) + lane;
    auto put_edges = [&](int b) {
        float *m = mine + b * warps * EDGE;
        m[0 * 32] = fa[R - 1][1];
        m[1 * 32] = fb[R - 1][1];
        m[2 * 32] = fa[R - 1][4];
        m[3 * 32] = fb[R - 1][4];
        m[4 * 32] = fa[R - 1][5];
        m[5 * 32] = fb[R - 1][5];
        m[6 * 32] = fa[0][3];
        m[7 * 32] = fb[0][3];
        m[8 * 32] = fa[0][6];
        m[9 * 32] = fb[0][6];
        m[10 * 32] = fa[0][7];
        m[11 * 32] = fb[0][7];
    };
    // one step, reading the edges of buffer b
    auto advance = [&](int b) {
        const float *lo = lower + b * warps * EDGE, *hi = upper + b * warps * EDGE;
        const float lo1a = lo[0], lo1b = lo[32], lo4a = lo[64], lo4b = lo[96], lo5a = lo[128],
                    lo5b = lo[160];
        const float hi3a = hi[0], hi3b = hi[32], hi6a = hi[64], hi6b = hi[96], hi7a = hi[128],
                    hi7b = hi[160];
        // every row's pull first: the rows' collisions are independent
        float da[R][8], db[R][8];
        auto left = [](float v) { return __shfl_up_sync(0xffffffffu, v, 1); };
        auto right = [](float v) { return __shfl_down_sync(0xffffffffu, v, 1); };
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int rl = r > 0 ? r - 1 : 0, rh = r + 1 < R ? r + 1 : r;
            const bool first = r == 0, last = r + 1 == R;
            da[r][0] = left(fb[r][0]);
            db[r][0] = fa[r][0];
            da[r][2] = fb[r][2];
            db[r][2] = right(fa[r][2]);
            da[r][1] = first ? lo1a : fa[rl][1];
            db[r][1] = first ? lo1b : fb[rl][1];
            da[r][4] = left(first ? lo4b : fb[rl][4]);
            db[r][4] = first ? lo4a : fa[rl][4];
            da[r][5] = first ? lo5b : fb[rl][5];
            db[r][5] = right(first ? lo5a : fa[rl][5]);
            da[r][3] = last ? hi3a : fa[rh][3];
            db[r][3] = last ? hi3b : fb[rh][3];
            da[r][6] = last ? hi6b : fb[rh][6];
            db[r][6] = right(last ? hi6a : fa[rh][6]);
            da[r][7] = left(last ? hi7b : fb[rh][7]);
            db[r][7] = last ? hi7a : fa[rh][7];
        }
        // the boundary rules in the order and with the operations of
        // pull_node_with: seam jump, walls, sides.  Every branch is the same
        // for the whole warp; lanes are told apart by their values.
        if (SEAM && seam) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                seam_jump(da[r], lo_axis_a, lo_diag_a, hi_axis_a, hi_diag_a);
                seam_jump(db[r], lo_axis_b, lo_diag_b, hi_axis_b, hi_diag_b);
            }
        }
        if ((WALLS || SIDES) && y_rules) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (WALLS && (y_rules >> (4 * r) & 4u)) {
                    wall_bottom(da[r], k);
                    wall_bottom(db[r], k);
                }
                if (WALLS && (y_rules >> (4 * r) & 8u)) {
                    wall_top(da[r], k);
                    wall_top(db[r], k);
                }
                if (SIDES && (y_rules >> (4 * r) & 3u)) {      // a row on a y side
                    const bool lo = y_rules >> (4 * r) & 1u, hi = y_rules >> (4 * r) & 2u;
                    apply_sides(da[r], k, open_x && xa_lo, open_x && xa_hi, lo, hi);
                    apply_sides(db[r], k, open_x && xb_lo, open_x && xb_hi, lo, hi);
                }
            }
        }
        if (SIDES && x_sides) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (y_rules >> (4 * r) & 3u) continue;         // done above
                if (x_sides & 1u) apply_x_side(da[r], db[r], k, xa_lo, xb_lo, 0);
                if (x_sides & 2u) apply_x_side(da[r], db[r], k, xa_hi, xb_hi, 1);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            collide_f32<float>(da[r], k);
            collide_f32<float>(db[r], k);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                fa[r][i] = da[r][i];
                fb[r][i] = db[r][i];
            }
        }
    };
    if (alive >= 0) put_edges(0);
    block_barrier();
    // the steps this warp still has valid rows for (the loop's body holds no
    // branch around a step: the rows stay in their registers), then the
    // barriers of the other warps' steps
    const int mine_steps = min(alive, a.steps);
    int s = 1;
#pragma unroll 2
    for (; s <= mine_steps; ++s) {
        advance((s & 1) ^ 1);
        if (s < a.steps) {
            put_edges(s & 1);
            block_barrier();
        }
    }
    for (; s < a.steps; ++s) block_barrier();

    const bool own_a = ca >= x0 && ca < x1, own_b = ca + 1 >= x0 && ca + 1 < x1;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int y = ys + r0 + r;
        if (y < y0 || y >= y1) continue;
        float *p = a.dst + (long long)y * a.nx + ca;
        if (wide && own_a && own_b) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float2 *>(p + (long long)i * a.plane) =
                    make_float2(fa[r][i], fb[r][i]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (own_a) p[(long long)i * a.plane] = fa[r][i];
                if (own_b) p[(long long)i * a.plane + 1] = fb[r][i];
            }
        }
    }
}

template <int R>
cudaError_t launch_rows(const cudaLaunchConfig_t &cfg, const TileArgs &a, const Coef<float> &k) {
    const bool sides = a.bc_x == BC_SIDES || a.bc_y == BC_SIDES;
    const bool seam = a.bc_x == BC_GRADIENT, walls = a.bc_y == BC_WALLS;
    if (sides) return cudaLaunchKernelEx(&cfg, tile_steps<R, true, true, true>, a, k);
    if (seam && walls) return cudaLaunchKernelEx(&cfg, tile_steps<R, true, true, false>, a, k);
    if (seam) return cudaLaunchKernelEx(&cfg, tile_steps<R, true, false, false>, a, k);
    if (walls) return cudaLaunchKernelEx(&cfg, tile_steps<R, false, true, false>, a, k);
    return cudaLaunchKernelEx(&cfg, tile_steps<R, false, false, false>, a, k);
}

}  // namespace

cudaError_t launch_tile(const TilePlan &p, int steps, const float *src, float *dst, int nx, int ny,
                        int bc_x, int bc_y, const Coef<float> &k, cudaStream_t stream) {
    if (p.steps < 1 || steps < 1 || steps > p.steps || src == dst) return cudaErrorInvalidValue;
    const int hx = tile_halo(p.steps);
    TileArgs a{src, dst, (long long)nx * ny, nx, ny, bc_x, bc_y, 64 - 2 * hx, p.ty, 0, hx, steps,
               steps};
    if (a.tx < 2) return cudaErrorInvalidValue;
    a.tiles_x = tile_columns(p, nx, bc_x == BC_SIDES);
    const bool open_y = bc_y == BC_SIDES || bc_y == BC_WALLS;
    const int rows = tile_rows(p.ty, ny, open_y, steps);
    const int warps = (rows + p.rows - 1) / p.rows;
    if (warps > TILE_MAX_WARPS) return cudaErrorInvalidConfiguration;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.tiles_x * ((ny + p.ty - 1) / p.ty)), 1, 1);
    cfg.blockDim = dim3((unsigned)(32 * warps), 1, 1);
    cfg.dynamicSmemBytes = (size_t)2 * warps * 12 * 32 * sizeof(float);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    switch (p.rows) {
        case 1: return launch_rows<1>(cfg, a, k);
        case 2: return launch_rows<2>(cfg, a, k);
        case 3: return launch_rows<3>(cfg, a, k);
        default: return launch_rows<4>(cfg, a, k);
    }
}

}  // namespace plbm
