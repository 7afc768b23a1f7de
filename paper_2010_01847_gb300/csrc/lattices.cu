// The phonon lattice Boltzmann step on the one-dimensional D1Q2 and the
// three-dimensional D3Q14 lattices (Section 2.2 names both; their weights
// follow from the moment conditions of Section 2.3, see phonon_lbm.h), on
// periodic lattices, behind the lbm_nd_* entry points.
//
// Same design as the D2Q8 path: structure of arrays (Q planes of
// nx*ny*nz, x fastest), deviations d_i = s (e_i - w_i e_ref) with s = 1,
// pull streaming from the post-collision planes of the previous step, the
// collision in registers on deviations with exact-sum rounded weights, and
// captured CUDA graphs of 64 steps (FP32 D3Q14 lattices from half a million
// nodes: two steps per launch, step2_d3q14).  In a pull step every stored value is
// read by exactly one node, so one thread per node with x fastest reads each
// plane row once, coalesced (the +-1 shift along x costs one extra sector
// per warp, served from L2).
#include <unistd.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>

#include "../../include/phonon_lbm.h"
#include "lbm_kernels.h"

namespace plbm {
namespace {

// Velocity sets, with opposite velocities at adjacent indices (2j, 2j+1).
// D3Q14: i = 0..5 the axis velocities +x, -x, +y, -y, +z, -z; i = 6..13
// the corners +b_j, -b_j for b_j = (1,1,1), (1,1,-1), (1,-1,1), (1,-1,-1).
// D1Q2: +x, -x.
template <int LAT> struct Lat;
template <> struct Lat<LBM_LATTICE_D3Q14> {
    static constexpr int Q = 14, DIM = 3, AXIS = 6;
    __host__ __device__ static constexpr int sgn(int i) { return (i & 1) ? -1 : 1; }
    __host__ __device__ static constexpr int cx(int i) {
        return i < 6 ? (i < 2 ? sgn(i) : 0) : sgn(i);
    }
    __host__ __device__ static constexpr int cy(int i) {
        return i < 6 ? (i == 2 || i == 3 ? sgn(i) : 0) : sgn(i) * ((((i - 6) >> 2) & 1) ? -1 : 1);
    }
    __host__ __device__ static constexpr int cz(int i) {
        return i < 6 ? (i >= 4 ? sgn(i) : 0) : sgn(i) * ((((i - 6) >> 1) & 1) ? -1 : 1);
    }
};
template <> struct Lat<LBM_LATTICE_D1Q2> {
    static constexpr int Q = 2, DIM = 1, AXIS = 2;
    __host__ __device__ static constexpr int cx(int i) { return i == 0 ? 1 : -1; }
    __host__ __device__ static constexpr int cy(int) { return 0; }
    __host__ __device__ static constexpr int cz(int) { return 0; }
};

// Coefficients rounded once to the compute type C.  Eq. 13 on deviations:
// rho = sum d_i, m = sum c_i d_i, q = m - lambda m (Eq. 54), t_i = h_i c_i.q,
// eq_i = w_i rho + t_i (Eq. 15), d_i* = d_i - omega (d_i - eq_i) - sigma t_i
// (Eq. 16).  The rounded weights keep sum_i w_i = 1 and sum_i h_i c_ix^2 = 1
// exact (see exact_pair), so the collision conserves energy and, without
// resistive scattering, heat flux to rounding.
template <typename C> struct CoefN {
    C omega, sigma, lambda;
    C w_axis, w_corner;
    C h_axis, h_corner;
};

// The collision of one node, on Q pulled deviations.  Opposite velocities
// (2j, 2j + 1) share their difference, c_i.q and t_i, whose signs alone
// differ: 108 operations for D3Q14, where population by population they were
// about 160, with the same roundings.
template <int LAT, typename C>
__device__ __forceinline__ void collide_nd(C (&d)[Lat<LAT>::Q], const CoefN<C> &k) {
    using L = Lat<LAT>;
    C rho = d[0] + d[1], m[3];
    bool any[3] = {false, false, false};
#pragma unroll
    for (int i = 0; i < L::Q; i += 2) {       // opposite velocities are adjacent
        if (i) rho += d[i] + d[i + 1];
        const C s = d[i] - d[i + 1];
        const int c[3] = {L::cx(i), L::cy(i), L::cz(i)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!c[a]) continue;
            m[a] = !any[a] ? (c[a] > 0 ? s : -s) : c[a] > 0 ? m[a] + s : m[a] - s;
            any[a] = true;
        }
    }
    C q[3];
#pragma unroll
    for (int a = 0; a < L::DIM; ++a) q[a] = m[a] - k.lambda * m[a];
    const C wa = k.w_axis * rho, wc = k.w_corner * rho;
#pragma unroll
    for (int i = 0; i < L::Q; i += 2) {
        const int c[3] = {L::cx(i), L::cy(i), L::cz(i)};
        C cq = C(0);
        bool first = true;
#pragma unroll
        for (int a = 0; a < L::DIM; ++a) {
            if (!c[a]) continue;
            cq = first ? (c[a] > 0 ? q[a] : -q[a]) : c[a] > 0 ? cq + q[a] : cq - q[a];
            first = false;
        }
        const C t = (i < L::AXIS ? k.h_axis : k.h_corner) * cq;
        const C w = i < L::AXIS ? wa : wc;
        const C ep = w + t, em = w - t;
        d[i] = d[i] - k.omega * (d[i] - ep) - k.sigma * t;
        d[i + 1] = d[i + 1] - k.omega * (d[i + 1] - em) + k.sigma * t;
    }
}

struct Dims {
    int nx, ny, nz;
    long long plane;
};

// Pull of the Q populations arriving at node (x, y, z) from the
// post-collision planes `src` of a periodic lattice.  I: the type of an offset
// within a plane.
template <int LAT, typename T, typename I = long long>
__device__ __forceinline__ void pull_nd(const T *src, const Dims &g, int x, int y, int z,
                                        typename Store<T>::C (&d)[Lat<LAT>::Q]) {
    using L = Lat<LAT>;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        int sx = x - L::cx(i), sy = y - L::cy(i), sz = z - L::cz(i);
        sx = sx < 0 ? sx + g.nx : (sx >= g.nx ? sx - g.nx : sx);
        sy = sy < 0 ? sy + g.ny : (sy >= g.ny ? sy - g.ny : sy);
        sz = sz < 0 ? sz + g.nz : (sz >= g.nz ? sz - g.nz : sz);
        d[i] = Store<T>::load(src[(long long)i * g.plane + (((I)sz * g.ny + sy) * g.nx + sx)]);
    }
}

// One step, one thread per node, in chained launches (small lattices take less
// time per step than a launch does: D3Q14 32^3 2.25 -> 1.64 us, 64^3
// 5.86 -> 4.76).  I: unsigned for planes of less than 2^31 nodes (the
// position's four divisions and fourteen offsets in 64 bits were more
// instructions than the collision), else long long.
template <int LAT, typename T, typename I>
__global__ void __launch_bounds__(256)
step_nd(const T *src, T *dst, Dims g, CoefN<typename Store<T>::C> k) {
    using C = typename Store<T>::C;
    const I node = (I)blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= (I)g.plane) return;
    const I r = node / (I)g.nx;
    const int x = int(node - r * (I)g.nx);
    const int z = int(r / (I)g.ny), y = int(r - (I)z * (I)g.ny);
    C d[Lat<LAT>::Q];
    chain_wait();
    pull_nd<LAT, T, I>(src, g, x, y, z, d);
    chain_next();
    collide_nd<LAT>(d, k);
#pragma unroll
    for (int i = 0; i < Lat<LAT>::Q; ++i)
        __stcs(dst + (long long)i * g.plane + node, Store<T>::put(d[i]));
}

// Two time steps of an FP32 D3Q14 lattice per launch.  A single step is bound
// by memory (112 bytes per node); here a block owns a column of tiles, 32 x 10
// nodes of (x, y) and planes z0 .. z1 - 1, and marches up z: at position p
// every thread pulls its node of plane p from the source planes and collides
// it (step 1, kept in shared memory only), then the inner 30 x 8 threads pull
// plane p - 1 of step 1 from there, collide again and store step 2.  The outer
// ring and the planes z0 - 1 and z1 of step 1 are worked out by two blocks.
// The next plane's loads are issued before step 2 of this one.  The
// arithmetic is that of step_nd (pull_nd's values, collide_nd).
// 192^3: 118.0 -> 83.9 us a step; 96^3 15.7 -> 14.4; below PAIR_MIN_NODES
// chained single steps are faster (80^3 8.1 against 9.3 us, 64^3 4.8 against
// 7.2).  At 192^3 a launch reads 426 MB of DRAM, 8 % more than the state, and
// writes 352 MB before its end (the rest of the 396 MB is then in L2); DRAM is
// busy 61 % of the time and the issue slots 66 %.  What is left is each plane's
// barrier and loads, so several small blocks per SM do better than two large
// ones: 32 x 16 threads and 2 blocks 95.9 us, 32 x 12 and 3 (spilling) 101.4,
// 32 x 8 and 4 88.4, 32 x 10 and 3 83.9 (64 registers, 4 bytes spilled).
//
// Shared memory: the 5 populations with c_z = +1 are pulled two positions
// after they are written, those with c_z = 0 one, those with c_z = -1 in the
// same; with one barrier per position a slot may be written again two
// positions after its last read, so they keep 4, 3 and 2 planes.
constexpr long long PAIR_MIN_NODES = 1 << 19;
constexpr int P2_X = 32, P2_Y = 10, P2_THREADS = P2_X * P2_Y, P2_BLOCKS = 3;
constexpr int P2_SMEM = (5 * 4 + 4 * 3 + 5 * 2) * P2_THREADS * (int)sizeof(float);

__host__ __device__ constexpr int p2_ring(int cz) { return cz > 0 ? 4 : cz == 0 ? 3 : 2; }
// first element of population i's ring
__host__ __device__ constexpr int p2_base(int i) {
    using L = Lat<LBM_LATTICE_D3Q14>;
    int at = 0;
    for (int j = 0; j < i; ++j) at += p2_ring(L::cz(j));
    return at * P2_THREADS;
}

__global__ void __launch_bounds__(P2_THREADS, P2_BLOCKS)
step2_d3q14(const float *__restrict__ src, float *__restrict__ dst, Dims g, int tiles_x,
            int tiles_y, int seg, CoefN<float> k) {
    using L = Lat<LBM_LATTICE_D3Q14>;
    extern __shared__ float rings[];
    const int tx = threadIdx.x % P2_X, ty = threadIdx.x / P2_X;
    const int by = blockIdx.x / tiles_x % tiles_y, bx = blockIdx.x % tiles_x;
    const int z0 = int(blockIdx.x / tiles_x / tiles_y) * seg, z1 = min(z0 + seg, g.nz);
    const int ox = bx * (P2_X - 2) + tx - 1, oy = by * (P2_Y - 2) + ty - 1;
    const bool own = tx > 0 && tx < P2_X - 1 && ty > 0 && ty < P2_Y - 1 && ox < g.nx && oy < g.ny;
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    // byte offsets of the columns and rows the pull reads: [0] c = -1, [1] 0,
    // [2] +1 (a layer has less than 2^30 nodes; everything else of an address
    // is the same for the whole block)
    unsigned xo[3], yo[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        xo[c] = 4u * wrap(ox - (c - 1), g.nx);
        yo[c] = 4u * ((unsigned)wrap(oy - (c - 1), g.ny) * g.nx);
    }
    const long long layer = (long long)g.nx * g.ny;
    float d[L::Q];
    // the next plane of step 1 before its collision, from planes zl, zc, zh
    int zl = wrap(z0 - 2, g.nz), zc = wrap(z0 - 1, g.nz), zh = z0;
    auto load = [&]() {
        const float *const z[3] = {src + zh * layer, src + zc * layer, src + zl * layer};
        zl = zc;
        zc = zh;
        zh = zh + 1 == g.nz ? 0 : zh + 1;
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            d[i] = __ldg(reinterpret_cast<const float *>(
                reinterpret_cast<const char *>(z[L::cz(i) + 1] + (long long)i * g.plane) +
                (yo[L::cy(i) + 1] + xo[L::cx(i) + 1])));
    };
    load();
    float *out = dst + (long long)z0 * layer;
    const unsigned at = own ? 4u * ((unsigned)oy * g.nx + ox) : 0u;
    int s3 = 0;                            // position mod 3
    for (int p = z0 - 1, n = 0; p <= z1; ++p, ++n) {
        collide_nd<LBM_LATTICE_D3Q14>(d, k);
        float *const mine = rings + threadIdx.x;
        float *const w4 = mine + (n & 3) * P2_THREADS, *const w3 = mine + s3 * P2_THREADS,
                    *const w2 = mine + (n & 1) * P2_THREADS;
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            (L::cz(i) > 0 ? w4 : L::cz(i) == 0 ? w3 : w2)[p2_base(i)] = d[i];
        __syncthreads();
        if (p < z1) load();
        if (n >= 2 && own) {
            // step 2 of plane p - 1: c_z = +1 from plane p - 2, 0 from p - 1, -1 from p
            const float *const r4 = mine + ((n + 2) & 3) * P2_THREADS,
                        *const r3 = mine + (s3 == 0 ? 2 : s3 - 1) * P2_THREADS, *const r2 = w2;
            float f[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; ++i)
                f[i] = (L::cz(i) > 0 ? r4 : L::cz(i) == 0 ? r3 : r2)[p2_base(i) - L::cx(i) -
                                                                     L::cy(i) * P2_X];
            collide_nd<LBM_LATTICE_D3Q14>(f, k);
#pragma unroll
            for (int i = 0; i < L::Q; ++i)
                __stcs(reinterpret_cast<float *>(
                           reinterpret_cast<char *>(out + (long long)i * g.plane) + at),
                       f[i]);
        }
        if (n >= 2) out += layer;
        s3 = s3 == 2 ? 0 : s3 + 1;
    }
}

// Blocks' planes: the segments per column that take the fewest rounds of
// plane positions (P2_BLOCKS blocks per SM; a segment marches 2 planes more than it
// owns, and its prologue costs about one).
int p2_segment(const Dims &g, long long tiles, int sms) {
    int best = g.nz;
    long long best_cost = -1;
    for (int s = 1; s <= g.nz; ++s) {
        const int seg = (g.nz + s - 1) / s;
        const long long blocks = tiles * ((g.nz + seg - 1) / seg);
        const long long cost = (blocks + P2_BLOCKS * sms - 1) / (P2_BLOCKS * sms) * (seg + 3);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = seg;
        }
    }
    return best;
}

// e and q of the state at the current step (pulled when `pulled`, else the
// stored step-0 state), FP64 outputs e[n], q[dim][n].
template <int LAT, typename T>
__global__ void moments_nd(const T *__restrict__ src, Dims g, bool pulled, double e_ref,
                           double inv_s, CoefN<typename Store<T>::C> k, double *e, double *q) {
    using C = typename Store<T>::C;
    using L = Lat<LAT>;
    for (long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x; node < g.plane;
         node += (long long)gridDim.x * blockDim.x) {
        const int x = int(node % g.nx);
        const long long r = node / g.nx;
        const int y = int(r % g.ny), z = int(r / g.ny);
        C d[L::Q];
        if (pulled) pull_nd<LAT, T>(src, g, x, y, z, d);
        else
#pragma unroll
            for (int i = 0; i < L::Q; ++i) d[i] = Store<T>::load(src[(long long)i * g.plane + node]);
        C rho = C(0), m[3] = {C(0), C(0), C(0)};
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            rho += d[i];
            m[0] += C(L::cx(i)) * d[i];
            m[1] += C(L::cy(i)) * d[i];
            m[2] += C(L::cz(i)) * d[i];
        }
        if (e) e[node] = e_ref + (double)rho * inv_s;
        if (q)
            for (int a = 0; a < L::DIM; ++a)
                q[(long long)a * g.plane + node] = (double)(m[a] - k.lambda * m[a]) * inv_s;
    }
}

template <int LAT, typename T>
__global__ void populations_nd(const T *__restrict__ src, Dims g, bool pulled, double e_ref,
                               double inv_s, double w_axis, double w_corner, double *f) {
    using C = typename Store<T>::C;
    using L = Lat<LAT>;
    for (long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x; node < g.plane;
         node += (long long)gridDim.x * blockDim.x) {
        const int x = int(node % g.nx);
        const long long r = node / g.nx;
        const int y = int(r % g.ny), z = int(r / g.ny);
        C d[L::Q];
        if (pulled) pull_nd<LAT, T>(src, g, x, y, z, d);
        else
#pragma unroll
            for (int i = 0; i < L::Q; ++i) d[i] = Store<T>::load(src[(long long)i * g.plane + node]);
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            f[(long long)i * g.plane + node] =
                (double)d[i] * inv_s + (i < L::AXIS ? w_axis : w_corner) * e_ref;
    }
}

// Eq. 15 on deviations (compute type) as the step-0 state `pre`, and its
// collision as `post`.  e[n], q[dim][n] FP64 device arrays (q may be null).
template <int LAT, typename T>
__global__ void init_nd(const double *__restrict__ e, const double *__restrict__ q, Dims g,
                        double e_ref, CoefN<typename Store<T>::C> k, T *__restrict__ pre,
                        T *__restrict__ post) {
    using C = typename Store<T>::C;
    using L = Lat<LAT>;
    for (long long node = (long long)blockIdx.x * blockDim.x + threadIdx.x; node < g.plane;
         node += (long long)gridDim.x * blockDim.x) {
        const C de = (C)(e[node] - e_ref);
        C qa[3] = {C(0), C(0), C(0)};
        if (q)
            for (int a = 0; a < L::DIM; ++a) qa[a] = (C)q[(long long)a * g.plane + node];
        C d[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const C cq = C(L::cx(i)) * qa[0] + C(L::cy(i)) * qa[1] + C(L::cz(i)) * qa[2];
            const C v = (i < L::AXIS ? k.w_axis : k.w_corner) * de +
                        (i < L::AXIS ? k.h_axis : k.h_corner) * cq;
            const T s = Store<T>::put(v);
            pre[(long long)i * g.plane + node] = s;
            d[i] = Store<T>::load(s);
        }
        collide_nd<LAT>(d, k);
#pragma unroll
        for (int i = 0; i < L::Q; ++i) post[(long long)i * g.plane + node] = Store<T>::put(d[i]);
    }
}

// Per-block sums of (e - e_ref) and a non-finite count of the current state.
template <int LAT, typename T>
__global__ void __launch_bounds__(256)
energy_nd(const T *__restrict__ src, Dims g, bool pulled, double *__restrict__ partials) {
    using C = typename Store<T>::C;
    using L = Lat<LAT>;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < g.plane;
         base += stride) {
        const long long node = base + (threadIdx.x & 31);
        C loc[5] = {C(0), C(0), C(0), C(0), C(0)};
        if (node < g.plane) {
            const int x = int(node % g.nx);
            const long long r = node / g.nx;
            const int y = int(r % g.ny), z = int(r / g.ny);
            C d[L::Q];
            if (pulled) pull_nd<LAT, T>(src, g, x, y, z, d);
            else
#pragma unroll
                for (int i = 0; i < L::Q; ++i)
                    d[i] = Store<T>::load(src[(long long)i * g.plane + node]);
            C rho = C(0);
#pragma unroll
            for (int i = 0; i < L::Q; ++i) rho += d[i];
            loc[0] = rho;
            loc[4] = isfinite(rho) ? C(0) : C(1);
        }
        warp_flush_residual(loc, acc);
    }
    block_sum5_lane0(acc, partials + (size_t)blockIdx.x * 5);
}

// Sets bit 0 of *bad if one of the first n values of v is not finite, bit 1 if
// one of those up to `total` is not.
__global__ void nonfinite_nd(const double *__restrict__ v, long long n, long long total,
                             int *__restrict__ bad) {
    int mine = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x)
        if (!isfinite(v[i])) mine |= i < n ? 1 : 2;
    if (mine) atomicOr(bad, mine);
}

constexpr int ENERGY_BLOCKS = 1216;

unsigned grid_of(long long n) {
    long long b = (n + 255) / 256;
    if (b > 152LL * 32) b = 152LL * 32;
    return (unsigned)(b > 0 ? b : 1);
}

// Rounds w_a (count na) and w_c (count nc) to C so that na w_a + nc w_c == 1
// holds exactly in C's binary arithmetic: start from the nearest value of
// the exact w_a and step one unit in the last place at a time until the
// w_c it implies is exactly representable.  For double nothing is checked
// (rounding there moves the sum by ~1e-16 per step).
template <typename C> void exact_pair(double wa, int na, int nc, C &oa, C &oc);
template <> void exact_pair<double>(double wa, int na, int nc, double &oa, double &oc) {
    oa = wa;
    oc = (1.0 - na * wa) / nc;
}
template <> void exact_pair<float>(double wa, int na, int nc, float &oa, float &oc) {
    float a = (float)wa;
    for (int k = 0; k < 64; ++k) {
        for (int sgn = 0; sgn < 2; ++sgn) {
            float t = a;
            for (int s = 0; s < k; ++s) t = std::nextafter(t, sgn ? 1.0f : 0.0f);
            const double rest = 1.0 - na * (double)t;   // exact: float times small int
            const float c = (float)(rest / nc);
            if ((double)c * nc == rest) {                // exact in double for floats
                oa = t;
                oc = c;
                return;
            }
        }
    }
    oa = a;
    oc = (float)((1.0 - na * wa) / nc);
}

}  // namespace
}  // namespace plbm

using namespace plbm;

struct lbm_nd {
    int lattice = 0, dim = 0, Q = 0;
    int precision = 0;
    int device = 0;
    Dims g{};
    double tau_N = 0, tau_R = 0, tau = 0, tau_r = 0, kappa = 1, sigma = 0;
    double e_ref = 1.0;
    cudaStream_t stream = nullptr, cap_stream = nullptr;
    void *buf[2] = {nullptr, nullptr};
    size_t buf_bytes = 0;
    int cur = 0;
    long n = 0;
    long long launches = 0;         // stream-collide launches since lbm_nd_init
    bool initialised = false;
    double *fields = nullptr;       // (1 + dim) planes of doubles
    double *partials = nullptr;     // ENERGY_BLOCKS x 5
    double *sums = nullptr;         // 5
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    int graph_chunk = 64;
    int pair_seg = 0;               // planes per block of the two-step kernel; 0: single steps
    std::string err;
};

namespace {

thread_local std::string g_nd_error;

lbm_status nd_fail(lbm_nd *c, lbm_status s, const std::string &m) {
    if (c) c->err = m;
    else g_nd_error = m;
    return s;
}

lbm_status nd_cuda(lbm_nd *c, cudaError_t e, const char *where) {
    (void)cudaGetLastError();
    return nd_fail(c, e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA,
                   std::string(where) + ": " + cudaGetErrorString(e));
}

#define NDCK(c, call)                                          \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) return nd_cuda(c, e_, #call);   \
    } while (0)

template <typename C> CoefN<C> coef_nd(const lbm_nd *c) {
    CoefN<C> k{};
    k.omega = (C)(1.0 / c->tau);
    k.sigma = (C)c->sigma;
    k.lambda = (C)(std::isinf(c->tau_r) ? 0.0 : 1.0 / (2.0 * c->tau_r + 1.0));
    if (c->lattice == LBM_LATTICE_D3Q14) {
        exact_pair<C>(1.0 / 9.0, 6, 8, k.w_axis, k.w_corner);    // 6 w_a + 8 w_c = 1
        exact_pair<C>(1.0 / 3.0, 2, 8, k.h_axis, k.h_corner);    // 2 h_a + 8 h_c = 1
    } else {
        k.w_axis = k.w_corner = (C)0.5;
        k.h_axis = k.h_corner = (C)0.5;
    }
    return k;
}

// Writes one byte of every page of a host buffer that is about to be filled.
// A caller's fresh array has no pages yet, and the copy from the device would
// take their faults one by one; here they are taken while the device still
// works on the launches before the copy (192^3 D3Q14, 226 MB of fields, 300
// steps: the pass 40.0 -> 36.5 ms).
void touch_pages(void *p, size_t bytes) {
    const long page = sysconf(_SC_PAGESIZE);
    if (!p || page <= 0) return;
    volatile char *c = (volatile char *)p;
    for (size_t i = 0; i < bytes; i += (size_t)page) c[i] = 0;
}

// Calls F<LAT, T>::run(c, args...) for the context's lattice and storage.
template <template <int, typename> class F, typename... A>
cudaError_t nd_dispatch(const lbm_nd *c, A... a) {
    if (c->lattice == LBM_LATTICE_D3Q14) {
        if (c->precision == PREC_FP64) return F<LBM_LATTICE_D3Q14, double>::run(c, a...);
        return F<LBM_LATTICE_D3Q14, float>::run(c, a...);
    }
    if (c->precision == PREC_FP64) return F<LBM_LATTICE_D1Q2, double>::run(c, a...);
    return F<LBM_LATTICE_D1Q2, float>::run(c, a...);
}

template <int LAT, typename T> struct StepNd {
    static cudaError_t run(const lbm_nd *c, int src, cudaStream_t s) {
        using C = typename Store<T>::C;
        const unsigned blocks = (unsigned)((c->g.plane + 255) / 256);
        return launch_chained(c->g.plane < 1LL << 31 ? step_nd<LAT, T, unsigned>
                                                     : step_nd<LAT, T, long long>,
                              blocks, 256, 0, s, (const T *)c->buf[src], (T *)c->buf[1 - src],
                              c->g, coef_nd<C>(c));
    }
};
template <int LAT, typename T> struct InitNd {
    static cudaError_t run(const lbm_nd *c, const double *e, const double *q) {
        using C = typename Store<T>::C;
        init_nd<LAT, T><<<grid_of(c->g.plane), 256, 0, c->stream>>>(
            e, q, c->g, c->e_ref, coef_nd<C>(c), (T *)c->buf[1], (T *)c->buf[0]);
        return cudaGetLastError();
    }
};
template <int LAT, typename T> struct MomentsNd {
    static cudaError_t run(const lbm_nd *c, double *e, double *q) {
        using C = typename Store<T>::C;
        moments_nd<LAT, T><<<grid_of(c->g.plane), 256, 0, c->stream>>>(
            (const T *)c->buf[1 - c->cur], c->g, c->n > 0, c->e_ref, 1.0, coef_nd<C>(c), e, q);
        return cudaGetLastError();
    }
};
template <int LAT, typename T> struct PopulationsNd {
    static cudaError_t run(const lbm_nd *c, double *f) {
        const double wa = LAT == LBM_LATTICE_D3Q14 ? 1.0 / 9.0 : 0.5;
        const double wc = LAT == LBM_LATTICE_D3Q14 ? 1.0 / 24.0 : 0.5;
        populations_nd<LAT, T><<<grid_of(c->g.plane), 256, 0, c->stream>>>(
            (const T *)c->buf[1 - c->cur], c->g, c->n > 0, c->e_ref, 1.0, wa, wc, f);
        return cudaGetLastError();
    }
};
template <int LAT, typename T> struct EnergyNd {
    static cudaError_t run(const lbm_nd *c, int) {
        energy_nd<LAT, T><<<ENERGY_BLOCKS, 256, 0, c->stream>>>((const T *)c->buf[1 - c->cur], c->g,
                                                                c->n > 0, c->partials);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return launch_finalize(c->partials, ENERGY_BLOCKS, c->sums, c->stream);
    }
};

// Two steps from buffer src (FP32 D3Q14).
cudaError_t nd_launch_pair(const lbm_nd *c, int src, cudaStream_t s) {
    const int tx = (c->g.nx + P2_X - 3) / (P2_X - 2), ty = (c->g.ny + P2_Y - 3) / (P2_Y - 2);
    const int segs = (c->g.nz + c->pair_seg - 1) / c->pair_seg;
    step2_d3q14<<<(unsigned)((long long)tx * ty * segs), P2_THREADS, P2_SMEM, s>>>(
        (const float *)c->buf[src], (float *)c->buf[1 - src], c->g, tx, ty, c->pair_seg,
        coef_nd<float>(c));
    return cudaGetLastError();
}

// Chooses the two-step kernel where its launches are long enough to pay.
void nd_plan_pairs(lbm_nd *c) {
    c->pair_seg = 0;
    if (c->lattice != LBM_LATTICE_D3Q14 || c->precision != PREC_FP32 ||
        c->g.plane < PAIR_MIN_NODES || (long long)c->g.nx * c->g.ny >= 1LL << 30)
        return;
    const long long tiles = (long long)((c->g.nx + P2_X - 3) / (P2_X - 2)) *
                            ((c->g.ny + P2_Y - 3) / (P2_Y - 2));
    if (tiles * c->g.nz > 0x7fffffffLL) return;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess ||
        sms < 1 ||
        cudaFuncSetAttribute(step2_d3q14, cudaFuncAttributeMaxDynamicSharedMemorySize, P2_SMEM) !=
            cudaSuccess) {
        (void)cudaGetLastError();
        return;
    }
    c->pair_seg = p2_segment(c->g, tiles, sms);
}

void nd_drop_graphs(lbm_nd *c) {
    for (auto &g : c->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
}

lbm_status nd_build_graph(lbm_nd *c, int start) {
    NDCK(c, cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t le = cudaSuccess;
    int src = start;
    for (int s = 0; s < c->graph_chunk && le == cudaSuccess; ++s) {
        le = nd_dispatch<StepNd>(c, src, c->cap_stream);
        src = 1 - src;
    }
    cudaGraph_t g = nullptr;
    cudaError_t ee = cudaStreamEndCapture(c->cap_stream, &g);
    if (le != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return nd_cuda(c, le, "capture of stream-collide launches");
    }
    if (ee != cudaSuccess) return nd_cuda(c, ee, "cudaStreamEndCapture");
    cudaError_t ie = cudaGraphInstantiate(&c->graph[start], g, 0);
    cudaGraphDestroy(g);
    if (ie != cudaSuccess) {
        c->graph[start] = nullptr;
        return nd_cuda(c, ie, "cudaGraphInstantiate");
    }
    return LBM_OK;
}

struct NdDevice {
    int old = -1;
    explicit NdDevice(int dev) {
        if (cudaGetDevice(&old) == cudaSuccess && old != dev) cudaSetDevice(dev);
        else old = -1;
    }
    ~NdDevice() {
        if (old >= 0) cudaSetDevice(old);
    }
};

}  // namespace

extern "C" {

double lbm_nd_lattice_speed(int lattice) {
    if (lattice == LBM_LATTICE_D3Q14) return std::sqrt(3.0 / 5.0);
    if (lattice == LBM_LATTICE_D1Q2) return 1.0 / std::sqrt(3.0);
    return 0.0;
}

lbm_status lbm_nd_create(int lattice, int nx, int ny, int nz, double tau_N, double tau_R,
                         int precision, double e_ref, void *stream, lbm_nd **out) {
    if (!out) return nd_fail(nullptr, LBM_EINVAL, "out is NULL");
    *out = nullptr;
    if (lattice != LBM_LATTICE_D1Q2 && lattice != LBM_LATTICE_D3Q14)
        return nd_fail(nullptr, LBM_EINVAL, "unknown lattice");
    if (nx < 1 || ny < 1 || nz < 1) return nd_fail(nullptr, LBM_EINVAL, "sizes must be >= 1");
    if (lattice == LBM_LATTICE_D1Q2 && (ny != 1 || nz != 1))
        return nd_fail(nullptr, LBM_EINVAL, "a D1Q2 lattice has ny = nz = 1");
    if ((long long)nx * ny * nz > (1LL << 40)) return nd_fail(nullptr, LBM_EINVAL, "too large");
    if (precision == LBM_FP16_DEV || precision == LBM_BF16_DEV)
        return nd_fail(nullptr, LBM_EUNSUPPORTED, "D1Q2 / D3Q14 store FP32 or FP64");
    if (precision != LBM_FP32 && precision != LBM_FP64)
        return nd_fail(nullptr, LBM_EINVAL, "unknown precision");
    if (std::isnan(tau_N) || std::isnan(tau_R) || !(tau_N > 0.0) || !(tau_R > 0.0) ||
        (std::isinf(tau_N) && std::isinf(tau_R)))
        return nd_fail(nullptr, LBM_EINVAL, "tau_N and tau_R must be > 0, not both infinite");
    if (!std::isfinite(e_ref)) return nd_fail(nullptr, LBM_EINVAL, "e_ref is not finite");
    lbm_nd *c = new lbm_nd();
    if (cudaGetDevice(&c->device) != cudaSuccess) {
        delete c;
        return nd_fail(nullptr, LBM_ECUDA, "no CUDA device");
    }
    c->lattice = lattice;
    c->dim = lattice == LBM_LATTICE_D3Q14 ? 3 : 1;
    c->Q = lattice == LBM_LATTICE_D3Q14 ? 14 : 2;
    c->precision = precision == LBM_FP64 ? PREC_FP64 : PREC_FP32;
    c->g = Dims{nx, ny, nz, (long long)nx * ny * nz};
    c->tau_N = tau_N;
    c->tau_R = tau_R;
    const double inv_c = (std::isinf(tau_N) ? 0.0 : 1.0 / tau_N) +
                         (std::isinf(tau_R) ? 0.0 : 1.0 / tau_R);
    c->tau = 1.0 / inv_c + 0.5;                                  // Eq. 49
    c->tau_r = tau_R;
    c->kappa = std::isinf(tau_R) ? 1.0 : 2.0 * tau_R / (2.0 * tau_R + 1.0);   // Eq. 54
    c->sigma = std::isinf(tau_R) ? 0.0 : (1.0 - 1.0 / (2.0 * c->tau)) / tau_R;  // Eq. 16
    c->e_ref = e_ref;
    c->stream = (cudaStream_t)stream;
    c->buf_bytes = (size_t)c->Q * (size_t)c->g.plane * (c->precision == PREC_FP64 ? 8 : 4);
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaMalloc(&c->buf[i], c->buf_bytes);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        lbm_status s = nd_cuda(nullptr, e, "lbm_nd_create");
        lbm_nd_destroy(c);
        return s;
    }
    nd_plan_pairs(c);
    *out = c;
    return LBM_OK;
}

void lbm_nd_destroy(lbm_nd *c) {
    if (!c) return;
    NdDevice g(c->device);
    if (c->stream || c->buf[0]) cudaStreamSynchronize(c->stream);
    nd_drop_graphs(c);
    if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
    cudaFree(c->buf[0]);
    cudaFree(c->buf[1]);
    cudaFree(c->fields);
    cudaFree(c->partials);
    cudaFree(c->sums);
    delete c;
}

static lbm_status nd_scratch(lbm_nd *c) {
    if (!c->fields)
        NDCK(c, cudaMalloc(&c->fields, sizeof(double) * (1 + c->dim) * (size_t)c->g.plane));
    if (!c->partials) NDCK(c, cudaMalloc(&c->partials, sizeof(double) * 5 * ENERGY_BLOCKS));
    if (!c->sums) NDCK(c, cudaMalloc(&c->sums, sizeof(double) * 5));
    return LBM_OK;
}

lbm_status lbm_nd_init(lbm_nd *c, const double *e, const double *q) {
    NvtxRange nvtx_("lbm_nd_init");
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    if (!e) return nd_fail(c, LBM_EINVAL, "e is NULL");
    NdDevice g(c->device);
    if (lbm_status s = nd_scratch(c)) return s;
    const size_t n = (size_t)c->g.plane;
    NDCK(c, cudaMemcpyAsync(c->fields, e, sizeof(double) * n, cudaMemcpyHostToDevice, c->stream));
    if (q)
        NDCK(c, cudaMemcpyAsync(c->fields + n, q, sizeof(double) * n * c->dim,
                                cudaMemcpyHostToDevice, c->stream));
    // captured launches stay valid: nothing in them depends on the fields
    int *const bad = (int *)c->sums;
    NDCK(c, cudaMemsetAsync(bad, 0, sizeof(int), c->stream));
    nonfinite_nd<<<grid_of(c->g.plane), 256, 0, c->stream>>>(
        c->fields, c->g.plane, q ? c->g.plane * (1 + c->dim) : c->g.plane, bad);
    NDCK(c, cudaGetLastError());
    int found = 0;
    NDCK(c, cudaMemcpyAsync(&found, bad, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    NDCK(c, cudaStreamSynchronize(c->stream));
    if (found)
        return nd_fail(c, LBM_EINVAL, found & 1 ? "e is not finite" : "q is not finite");
    NDCK(c, nd_dispatch<InitNd>(c, (const double *)c->fields, q ? (const double *)(c->fields + n)
                                                                : (const double *)nullptr));
    NDCK(c, cudaStreamSynchronize(c->stream));
    c->cur = 0;
    c->n = 0;
    c->launches = 0;
    c->initialised = true;
    return LBM_OK;
}

lbm_status lbm_nd_step(lbm_nd *c, long n) {
    NvtxRange nvtx_("lbm_nd_step");
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    if (n < 0) return nd_fail(c, LBM_EINVAL, "n must be >= 0");
    if (!c->initialised) return nd_fail(c, LBM_EINVAL, "lbm_nd_init has not been called");
    NdDevice g(c->device);
    long left = n;
    // two steps per launch, then one or two single steps: the read-outs pull
    // from the state one step back
    for (; c->pair_seg > 0 && left > 2; left -= 2) {
        NDCK(c, nd_launch_pair(c, c->cur, c->stream));
        c->cur = 1 - c->cur;
        c->n += 2;
        c->launches += 1;
    }
    if (left >= c->graph_chunk) {
        if (!c->graph[c->cur])
            if (lbm_status s = nd_build_graph(c, c->cur)) return s;
        while (left >= c->graph_chunk) {
            NDCK(c, cudaGraphLaunch(c->graph[c->cur], c->stream));
            left -= c->graph_chunk;
            c->n += c->graph_chunk;
            c->launches += c->graph_chunk;
        }
    }
    for (; left > 0; --left) {
        NDCK(c, nd_dispatch<StepNd>(c, c->cur, c->stream));
        c->cur = 1 - c->cur;
        c->n += 1;
        c->launches += 1;
    }
    return LBM_OK;
}

lbm_status lbm_nd_sync(lbm_nd *c) {
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    NdDevice g(c->device);
    NDCK(c, cudaStreamSynchronize(c->stream));
    return LBM_OK;
}

lbm_status lbm_nd_moments(lbm_nd *c, double *e, double *q) {
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    if (!c->initialised) return nd_fail(c, LBM_EINVAL, "lbm_nd_init has not been called");
    NdDevice g(c->device);
    if (lbm_status s = nd_scratch(c)) return s;
    const size_t n = (size_t)c->g.plane;
    NDCK(c, nd_dispatch<MomentsNd>(c, c->fields, c->fields + n));
    touch_pages(e, sizeof(double) * n);
    touch_pages(q, sizeof(double) * n * c->dim);
    if (e)
        NDCK(c, cudaMemcpyAsync(e, c->fields, sizeof(double) * n, cudaMemcpyDeviceToHost,
                                c->stream));
    if (q)
        NDCK(c, cudaMemcpyAsync(q, c->fields + n, sizeof(double) * n * c->dim,
                                cudaMemcpyDeviceToHost, c->stream));
    NDCK(c, cudaStreamSynchronize(c->stream));
    return LBM_OK;
}

lbm_status lbm_nd_populations(lbm_nd *c, double *f) {
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    if (!f) return nd_fail(c, LBM_EINVAL, "f is NULL");
    if (!c->initialised) return nd_fail(c, LBM_EINVAL, "lbm_nd_init has not been called");
    NdDevice g(c->device);
    const size_t bytes = sizeof(double) * (size_t)c->Q * (size_t)c->g.plane;
    double *dev = nullptr;
    NDCK(c, cudaMallocAsync((void **)&dev, bytes, c->stream));
    cudaError_t e = nd_dispatch<PopulationsNd>(c, dev);
    if (e == cudaSuccess) e = cudaMemcpyAsync(f, dev, bytes, cudaMemcpyDeviceToHost, c->stream);
    cudaFreeAsync(dev, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return nd_cuda(c, e, "lbm_nd_populations");
    return LBM_OK;
}

lbm_status lbm_nd_energy(lbm_nd *c, double *total) {
    if (!c) return nd_fail(nullptr, LBM_EINVAL, "ctx is NULL");
    if (!c->initialised) return nd_fail(c, LBM_EINVAL, "lbm_nd_init has not been called");
    NdDevice g(c->device);
    if (lbm_status s = nd_scratch(c)) return s;
    NDCK(c, nd_dispatch<EnergyNd>(c, 0));
    double sums[5];
    NDCK(c, cudaMemcpyAsync(sums, c->sums, sizeof(sums), cudaMemcpyDeviceToHost, c->stream));
    NDCK(c, cudaStreamSynchronize(c->stream));
    if (total) *total = (double)c->g.plane * c->e_ref + sums[0];
    if (sums[4] > 0.0) return nd_fail(c, LBM_ENONFINITE, "state holds NaN or Inf");
    return LBM_OK;
}

long lbm_nd_step_count(const lbm_nd *c) { return c ? c->n : -1; }

long long lbm_nd_kernel_launches(const lbm_nd *c) { return c ? c->launches : -1; }

const char *lbm_nd_last_error(const lbm_nd *c) {
    return c ? c->err.c_str() : g_nd_error.c_str();
}

}  // extern "C"
