// Small multilayer perceptron for the learned warm start: inference and
// training kernels.  Layer l maps X_l [B x K_l] to Z_l = X_l W_l^T + b_l
// (W_l stored [N_l x K_l] row-major), hidden layers apply GELU
// (x Phi(x), Phi the normal CDF); the last layer is linear.  Loss: mean
// squared error over all outputs.  Training: backpropagation and Adam.
//
// Precision: matrix products take BF16 operands on the tensor cores
// (mma.sync m16n8k16, FP32 accumulation); weights, biases, pre-activations,
// gradients and Adam moments are FP32; BF16 copies of the weights and of the
// layer inputs feed the products.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/phonon_lbm.h"
#include "lbm_kernels.h"

namespace plbm {
namespace {

constexpr int TK = 64;                     // k depth of a pipeline stage
constexpr int GEMM_THREADS = 128;          // 4 warps

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4],
                                         const unsigned (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float gelu(float x) {
    return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad(float x) {
    const float cdf = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
    const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
    return cdf + x * pdf;
}

enum { EPI_NONE = 0, EPI_GELU = 1, EPI_GELU_BWD = 2 };

// Every BF16 matrix has rows of ld = width rounded up to 8 elements (16-byte
// aligned rows, zeros behind the width), so every tile is filled by 16-byte
// asynchronous copies whatever the widths.
__host__ __device__ constexpr long long ld8(long long n) { return (n + 7) & ~7LL; }

// C[m, n] = sum_k A(m, k) B(k, n) (+ bias[n]), FP32, [M x N].  Outputs (each
// optional): pre = the result, out = the result after the epilogue, outb = the
// same in BF16 (rows of ld8(N), zeros behind N).  Epilogues: GELU (forward),
// GELU backward (the result times GELU'(aux[m, n]), aux the pre-activation of
// the layer below: dZ = dX (.) GELU'(Z)).
struct Product {
    const __nv_bfloat16 *A, *B;
    long long lda, ldb;
    const float *bias, *aux;
    float *pre, *out;
    __nv_bfloat16 *outb;
    int M, N, K, epi;
};

// Tile shape of a block's product: T x T outputs, four warps of T/2 x T/2.
// What bounds these products is latency, not rate: a few hundred rows and
// columns are one wave of small blocks, and each block's chain is load, wait,
// multiply.  So a stage is 64 deep and STAGES of them are in flight at once:
// with T = 32 the whole depth of 512 is requested before the first multiply.
// With one launch per layer and direction, a training step of the
// 3-256-256-256-256-512 network at 512 rows takes 60 us; a 32-deep loop that
// loaded, waited and multiplied in turn, in 24 launches, took 207.
// A row of a tile is padded by 8 elements (an odd number of 16-byte units:
// ldmatrix reads 8 rows without bank conflicts).
template <int T> struct Tile {
    static constexpr int STAGES = T == 32 ? 8 : 4;
    static constexpr int K_ROW = TK + 8, M_ROW = T + 8;       // row lengths of the two layouts
    static constexpr int OPERAND = T * K_ROW > TK * M_ROW ? T * K_ROW : TK * M_ROW;   // elements
    static constexpr int SMEM = STAGES * 2 * OPERAND * 2;     // bytes
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool valid) {
    const int n = valid ? 16 : 0;                              // 0: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm4_t(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// Copies of one operand's tile for depth k0 .. k0 + TK - 1.  KMAJOR: the
// operand is stored [line][k] (rows of `lines`, ld >= its depth); else
// [k][line].  r0: the tile's first line.
template <int T, bool KMAJOR>
__device__ __forceinline__ void stage_operand(unsigned dst, const __nv_bfloat16 *src, long long ld,
                                              int lines, int depth, int r0, int k0) {
#pragma unroll
    for (int it = 0; it < T * TK / 8 / GEMM_THREADS; ++it) {
        const int idx = it * GEMM_THREADS + threadIdx.x;
        if (KMAJOR) {
            const int r = idx / (TK / 8), c = (idx % (TK / 8)) * 8;
            const bool ok = r0 + r < lines && k0 + c < depth;   // a chunk past depth: zeros
            const long long o = ok ? (long long)(r0 + r) * ld + k0 + c : 0;
            cp_async16(dst + 2 * (r * Tile<T>::K_ROW + c), src + o, ok);
        } else {
            const int k = idx / (T / 8), c = (idx % (T / 8)) * 8;
            const bool ok = k0 + k < depth && r0 + c < lines;
            const long long o = ok ? (long long)(k0 + k) * ld + r0 + c : 0;
            cp_async16(dst + 2 * (k * Tile<T>::M_ROW + c), src + o, ok);
        }
    }
}

// The T x T tile at (m0, n0) of one product; every thread of the block calls
// it.  The depth is summed in k order, 16 at a time, whatever the tile.
template <int T, bool A_KMAJOR, bool B_KMAJOR>
__device__ __forceinline__ void product_tile(const Product &g, int m0, int n0, unsigned smem) {
    constexpr int MI = T / 32, NJ = T / 16;       // m16 and n8 tiles per warp
    constexpr int STAGES = Tile<T>::STAGES;
    constexpr unsigned OP = Tile<T>::OPERAND * 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * (T / 2), wn = (warp & 1) * (T / 2);
    const int gr = lane >> 2, tg = lane & 3;
    const int chunks = (g.K + TK - 1) / TK;
    auto stage = [&](int c) {
        if (c < chunks) {
            const unsigned a = smem + (c % STAGES) * 2 * OP;
            stage_operand<T, A_KMAJOR>(a, g.A, g.lda, g.M, g.K, m0, c * TK);
            stage_operand<T, B_KMAJOR>(a + OP, g.B, g.ldb, g.N, g.K, n0, c * TK);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int c = 0; c < STAGES - 1; ++c) stage(c);
    // the lane's row address in each operand's tile (see ldmatrix)
    const int j = lane >> 3, r = lane & 7;
    const unsigned a_at = A_KMAJOR ? 2 * ((wm + (lane & 15)) * Tile<T>::K_ROW + (lane >> 4) * 8)
                                   : 2 * (((j >> 1) * 8 + r) * Tile<T>::M_ROW + wm + (j & 1) * 8);
    const unsigned b_at = B_KMAJOR ? 2 * ((wn + (j >> 1) * 8 + r) * Tile<T>::K_ROW + (j & 1) * 8)
                                   : 2 * (((j & 1) * 8 + r) * Tile<T>::M_ROW + wn + (j >> 1) * 8);
    constexpr unsigned A_I = 2 * 16 * (A_KMAJOR ? Tile<T>::K_ROW : 1);     // next 16 lines
    constexpr unsigned B_J = 2 * 16 * (B_KMAJOR ? Tile<T>::K_ROW : 1);
    constexpr unsigned A_K = 2 * 16 * (A_KMAJOR ? 1 : Tile<T>::M_ROW);     // next 16 of the depth
    constexpr unsigned B_K = 2 * 16 * (B_KMAJOR ? 1 : Tile<T>::M_ROW);
    // what the epilogue reads, asked for before the products (behind them each
    // load would wait for the one before: the stores between may alias)
    float bias[NJ][2], aux[MI][NJ][4];
#pragma unroll
    for (int q = 0; q < NJ; ++q)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int n = n0 + wn + 8 * q + 2 * tg + e;
            bias[q][e] = g.bias && n < g.N ? g.bias[n] : 0.f;
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int m = m0 + wm + 16 * i + gr + 8 * h;
                    aux[i][q][2 * h + e] = g.epi == EPI_GELU_BWD && m < g.M && n < g.N
                                               ? g.aux[(long long)m * g.N + n]
                                               : 0.f;
                }
        }
    float acc[MI][NJ][4] = {};
    for (int c = 0; c < chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();              // stage c is there, stage c - 1 is read by all
        stage(c + STAGES - 1);
        const unsigned sa = smem + (c % STAGES) * 2 * OP, sb = sa + OP;
#pragma unroll
        for (int kk = 0; kk < TK / 16; ++kk) {
            if (c * TK + kk * 16 >= g.K) break;
            unsigned a[MI][4], b[NJ / 2][4];
#pragma unroll
            for (int i = 0; i < MI; ++i) {
                const unsigned at = sa + a_at + i * A_I + kk * A_K;
                if (A_KMAJOR) ldsm4(a[i], at);
                else ldsm4_t(a[i], at);
            }
#pragma unroll
            for (int q = 0; q < NJ / 2; ++q) {
                const unsigned at = sb + b_at + q * B_J + kk * B_K;
                if (B_KMAJOR) ldsm4(b[q], at);
                else ldsm4_t(b[q], at);
            }
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int q = 0; q < NJ; ++q) {
                    const unsigned bq[2] = {b[q / 2][(q & 1) * 2], b[q / 2][(q & 1) * 2 + 1]};
                    mma_bf16(acc[i][q], a[i], bq);
                }
        }
    }
    const long long ldo = ld8(g.N);
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int q = 0; q < NJ; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) {         // rows g, g + 8: two adjacent columns each
                const int m = m0 + wm + 16 * i + gr + 8 * h;
                const int n = n0 + wn + 8 * q + 2 * tg;
                if (m >= g.M || n >= ldo) continue;
                float v[2] = {0.f, 0.f};
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (n + e >= g.N) continue;
                    const long long o = (long long)m * g.N + n + e;
                    v[e] = acc[i][q][2 * h + e] + bias[q][e];
                    if (g.pre) g.pre[o] = v[e];
                    if (g.epi == EPI_GELU) v[e] = gelu(v[e]);
                    if (g.epi == EPI_GELU_BWD) v[e] = v[e] * gelu_grad(aux[i][q][2 * h + e]);
                    if (g.out) g.out[o] = v[e];
                }
                if (g.outb)
                    *reinterpret_cast<__nv_bfloat162 *>(g.outb + (long long)m * ldo + n) =
                        __floats2bfloat162_rn(v[0], v[1]);
            }
}

__host__ __device__ constexpr long long tiles_of(long long n, int t) { return (n + t - 1) / t; }

// Forward product of a layer: A = X [M x K], B(k, n) = W[n][k].
template <int T>
__global__ void __launch_bounds__(GEMM_THREADS) forward_product(const Product g) {
    extern __shared__ __align__(16) unsigned char tiles[];
    const int tn = (int)tiles_of(g.N, T);
    const int bm = blockIdx.x / tn, bn = blockIdx.x - bm * tn;
    product_tile<T, true, true>(g, bm * T, bn * T, (unsigned)__cvta_generic_to_shared(tiles));
}

// db[n] = sum over the batch of dZ[b, n]: 8 rows' worth of partial sums, sum
// w over rows w, w + 8, ... in order, then the 8 sums in order: a fixed order,
// so the result does not vary between runs.  A block takes 16 columns (thread
// w * 16 + column); its loads do not depend on the running sums, 32 in flight.
constexpr int BIAS_SUMS = 8, BIAS_COLS = GEMM_THREADS / BIAS_SUMS;
__device__ __forceinline__ void bias_block(const float *__restrict__ dz, int B, int N, int n0,
                                           float *__restrict__ db, float *part) {
    const int col = threadIdx.x % BIAS_COLS, w = threadIdx.x / BIAS_COLS, n = n0 + col;
    float s = 0.f;
    if (n < N) {
#pragma unroll 32
        for (int b = w; b < B; b += BIAS_SUMS) s += dz[(long long)b * N + n];
    }
    part[threadIdx.x] = s;
    __syncthreads();
    if (w == 0 && n < N) {
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < BIAS_SUMS; ++i) t += part[i * BIAS_COLS + col];
        db[n] = t;
    }
}

// Everything of a layer's backward pass that needs its dZ, in one launch:
// blocks [0, nw): dW = dZ^T X (w); [nw, nw + nx): dZ of the layer below (x,
// dX (.) GELU'); the rest: the bias gradient.  One launch in place of three
// in turn: each is a fraction of a wave (64, 128 and 16 blocks for the hidden
// layers at 512 rows).
template <int T>
__global__ void __launch_bounds__(GEMM_THREADS)
backward_products(const Product w, const Product x, long long nw, long long nx,
                  const float *__restrict__ dz, int batch, int N, float *__restrict__ db) {
    extern __shared__ __align__(16) unsigned char tiles[];
    const unsigned smem = (unsigned)__cvta_generic_to_shared(tiles);
    const long long id = blockIdx.x;
    if (id < nw) {
        const int tn = (int)tiles_of(w.N, T);
        const int bm = int(id / tn), bn = int(id - (long long)bm * tn);
        product_tile<T, false, false>(w, bm * T, bn * T, smem);
    } else if (id < nw + nx) {
        const int tn = (int)tiles_of(x.N, T);
        const int bm = int((id - nw) / tn), bn = int((id - nw) - (long long)bm * tn);
        product_tile<T, true, false>(x, bm * T, bn * T, smem);
    } else {
        bias_block(dz, batch, N, int(id - nw - nx) * BIAS_COLS, db, (float *)tiles);
    }
}

// Rows of n FP32 values as rows of ld8(n) BF16 values.
__global__ void to_bf16_rows(const float *__restrict__ x, __nv_bfloat16 *__restrict__ y,
                             long long rows, int n) {
    const long long ld = ld8(n), total = rows * ld;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / ld;
        const int c = int(i - r * ld);
        y[i] = __float2bfloat16_rn(c < n ? x[r * n + c] : 0.f);
    }
}

// SplitMix64 (Steele, Lea and Flood's generator) of a 64-bit counter.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Per-step scalars of the device training loop (train_setup writes them).
struct TrainState {
    long long t;          // Adam steps taken so far (all calls)
    long long local;      // steps of this call so far: the step being run, until train_setup
    float lr, c1, c2;     // learning rate and bias corrections of the step
};

// The minibatch of a training step: row j is sample (batch >= n ? j mod n :
// SplitMix64(seed ^ (step batch + j)) mod n), drawn with replacement.  Writes
// the samples and their input rows in BF16.
__global__ void gather_rows(const float *__restrict__ x, int kx, const TrainState *st,
                            unsigned long long seed, int n, int batch, int *rows,
                            __nv_bfloat16 *y) {
    const long long ld = ld8(kx), total = batch * ld;
    const unsigned long long base = (unsigned long long)st->local * (unsigned long long)batch;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int j = int(i / ld), c = int(i - j * ld);
        const int sample = batch >= n ? j % n
                                      : (int)(splitmix64(seed ^ (base + (unsigned)j)) %
                                              (unsigned long long)n);
        if (c == 0) rows[j] = sample;
        y[i] = __float2bfloat16_rn(c < kx ? x[(long long)sample * kx + c] : 0.f);
    }
}

// dY = 2 (Y - T) / (B N) (mean squared error), FP32 [B x N] and BF16 (rows of
// ld8(N)), and the loss partial sums, one per block.  rows: the sample of each
// row (nullptr: row j is sample j).  An SM adds about one FP64 value per clock,
// which bounds this kernel: a thread sums MSE_EACH squares before the block's
// tree (one value per thread, and the tree over five sums of which four were
// zero, took 12.8 us at 512 x 512; with the samples drawn again for every
// element).
constexpr int MSE_EACH = 4;
constexpr int LOSS_BLOCKS = 4096;
unsigned mse_blocks(long long n) {
    const long long b = (n + 256 * MSE_EACH - 1) / (256 * MSE_EACH);
    return (unsigned)(b > LOSS_BLOCKS ? LOSS_BLOCKS : b);
}
__global__ void __launch_bounds__(256)
mse_grad(const float *y, const float *t, const int *rows, long long n, int N, float scale,
         float *dy, __nv_bfloat16 *dyb, double *loss_partials) {
    const int ld = (int)ld8(N);
    const bool small = n <= 0xffffffffLL;          // 32-bit division
    auto row_of = [&](long long i) -> long long {
        return small ? (long long)((unsigned)i / (unsigned)N) : i / N;
    };
    double s = 0.0;
    for (long long base = (long long)blockIdx.x * (256 * MSE_EACH); base < n;
         base += (long long)gridDim.x * (256 * MSE_EACH)) {
        float d[MSE_EACH];
#pragma unroll
        for (int e = 0; e < MSE_EACH; ++e) {
            const long long i = base + e * 256 + threadIdx.x;
            d[e] = 0.f;
            if (i < n) {
                const long long j = row_of(i);
                d[e] = y[i] - t[(rows ? (long long)rows[j] : j) * N + (i - j * N)];
            }
        }
#pragma unroll
        for (int e = 0; e < MSE_EACH; ++e) {
            const long long i = base + e * 256 + threadIdx.x;
            if (i >= n) continue;
            const long long j = row_of(i);
            const int c = int(i - j * N);
            s += (double)(d[e] * d[e]);
            const float gval = 2.0f * d[e] * scale;
            dy[i] = gval;
            dyb[j * ld + c] = __float2bfloat16_rn(gval);
            if (c == N - 1)
                for (int z = N; z < ld; ++z) dyb[j * ld + z] = __float2bfloat16_rn(0.f);
        }
    }
    __shared__ double part[8];
    const double w = warp_sum_f64(s);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = w;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int i = 0; i < 8; ++i) sum += part[i];
        loss_partials[blockIdx.x] = sum;
    }
}

// The total of the loss partial sums in a fixed order (one block).
__global__ void __launch_bounds__(256)
sum_loss(const double *partials, int blocks, double *total) {
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < blocks; b += 256) acc[0] += partials[b];
    __shared__ double out[5];
    block_sum5_store(acc, out);
    if (threadIdx.x == 0) *total = out[0];
}

// One Adam update of parameter i (refreshing its BF16 copy if it is a weight).
__device__ __forceinline__ void adam_update(long long i, float *__restrict__ p,
                                            const float *__restrict__ g, float *__restrict__ m,
                                            float *__restrict__ v, float lr, float b1, float b2,
                                            float eps, float c1, float c2,
                                            const long long *__restrict__ wmap,
                                            __nv_bfloat16 *__restrict__ pb) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    if (wmap[i] >= 0) pb[wmap[i]] = __float2bfloat16_rn(w);
}

// Adam on the flat FP32 parameters, refreshing the BF16 copy of every weight.
__global__ void adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                     float *__restrict__ v, long long n, float lr, float b1, float b2, float eps,
                     float c1, float c2, const long long *__restrict__ wmap,
                     __nv_bfloat16 *__restrict__ pb) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        adam_update(i, p, g, m, v, lr, b1, b2, eps, c1, c2, wmap, pb);
}

// One thread: the step's loss (mean of the squared errors) into the history,
// its learning rate (cosine from lr to lr_final over `steps`) and Adam's bias
// corrections 1 - beta^t, then the counters.
__global__ void train_setup(TrainState *st, long long steps, float lr, float lr_final,
                            float b1, float b2, const double *__restrict__ total, double inv_n,
                            float *__restrict__ hist) {
    const long long t = st->t + 1, s = st->local;
    hist[s] = (float)(*total * inv_n);
    st->lr = (float)((double)lr_final +
                     0.5 * ((double)lr - (double)lr_final) *
                         (1.0 + cos(3.14159265358979323846 * (double)s / (double)steps)));
    st->c1 = 1.f - (float)pow((double)b1, (double)t);     // as lbm_mlp_train_step forms them
    st->c2 = 1.f - (float)pow((double)b2, (double)t);
    st->t = t;
    st->local = s + 1;
}

// Adam with the step's scalars from the device (the training loop).
__global__ void adam_dev(float *__restrict__ p, const float *__restrict__ g,
                         float *__restrict__ m, float *__restrict__ v, long long n, float b1,
                         float b2, float eps, const TrainState *__restrict__ st,
                         const long long *__restrict__ wmap, __nv_bfloat16 *__restrict__ pb) {
    const float lr = st->lr, c1 = st->c1, c2 = st->c2;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        adam_update(i, p, g, m, v, lr, b1, b2, eps, c1, c2, wmap, pb);
}

unsigned grid1(long long n) {
    long long b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

}  // namespace
}  // namespace plbm

using namespace plbm;

struct lbm_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::vector<int> widths;             // K_0, N_0 = K_1, ..., N_{L-1}
    int layers = 0;
    int max_batch = 0;
    std::vector<long long> w_off, b_off;  // offsets in the flat FP32 parameters
    std::vector<long long> wb_off;        // offsets in the BF16 weight copy
    long long n_params = 0, n_wb = 0;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *wb = nullptr;          // BF16 weights
    long long *wmap = nullptr;            // flat index -> BF16 index (or -1)
    std::vector<float *> pre;             // pre-activations per hidden layer [B x N_l]
    float *act = nullptr;                 // FP32 output of the last layer
    std::vector<__nv_bfloat16 *> actb;    // BF16 layer inputs: actb[0] = X, actb[l+1] = out of l
    float *g0 = nullptr, *g1 = nullptr;   // gradient ping-pong [B x max width]
    __nv_bfloat16 *gb = nullptr, *gb1 = nullptr;   // BF16 copies of the two
    // device training loop: state, capture streams (the second takes the
    // step's loss and scalars beside the backward pass) and their events
    TrainState *tstate = nullptr;
    int *rows = nullptr;                  // the minibatch's samples
    cudaStream_t cap = nullptr, cap2 = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    double *loss_part = nullptr;
    long long steps = 0;
    std::string err;
};

namespace {

lbm_status mfail(lbm_mlp *m, lbm_status s, const std::string &msg) {
    if (m) m->err = msg;
    else set_global_error(msg.c_str());
    return s;
}

lbm_status mcuda(lbm_mlp *m, cudaError_t e, const char *where) {
    std::string msg = std::string(where) + ": " + cudaGetErrorName(e);
    (void)cudaGetLastError();
    return mfail(m, e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, msg);
}

#define MCK(m, call)                                           \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) return mcuda(m, e_, #call);     \
    } while (0)

// 64 x 64 tiles when they give at least two blocks per SM, else 32 x 32 (the
// network's products are small: a few hundred rows and columns).
constexpr long long BIG_TILES = 2 * 152;

template <int T> cudaError_t launch_forward(const Product &g, cudaStream_t s) {
    const long long blocks = tiles_of(g.M, T) * tiles_of(g.N, T);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(forward_product<T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Tile<T>::SMEM);
    if (e != cudaSuccess) return e;
    forward_product<T><<<(unsigned)blocks, GEMM_THREADS, Tile<T>::SMEM, s>>>(g);
    return cudaGetLastError();
}

template <int T>
cudaError_t launch_backward(const Product &w, const Product &x, const float *dz, int batch, int N,
                            float *db, cudaStream_t s) {
    const long long nw = tiles_of(w.M, T) * tiles_of(w.N, T);
    const long long nx = x.A ? tiles_of(x.M, T) * tiles_of(x.N, T) : 0;
    const long long blocks = nw + nx + tiles_of(N, BIAS_COLS);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(backward_products<T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Tile<T>::SMEM);
    if (e != cudaSuccess) return e;
    backward_products<T><<<(unsigned)blocks, GEMM_THREADS, Tile<T>::SMEM, s>>>(w, x, nw, nx, dz,
                                                                               batch, N, db);
    return cudaGetLastError();
}

// The layers on the `batch` BF16 rows in actb[0], on stream s; the output
// layer's FP32 result is act[L-1].
cudaError_t forward_layers(lbm_mlp *m, int batch, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    for (int l = 0; l < m->layers && e == cudaSuccess; ++l) {
        const int K = m->widths[l], N = m->widths[l + 1];
        const bool last = l == m->layers - 1;
        Product g{};
        g.A = m->actb[l];
        g.lda = ld8(K);
        g.B = m->wb + m->wb_off[l];
        g.ldb = ld8(K);
        g.bias = m->params + m->b_off[l];
        g.pre = last ? nullptr : m->pre[l];
        g.out = last ? m->act : nullptr;
        g.outb = last ? nullptr : m->actb[l + 1];
        g.M = batch;
        g.N = N;
        g.K = K;
        g.epi = last ? EPI_NONE : EPI_GELU;
        e = tiles_of(batch, 64) * tiles_of(N, 64) >= BIG_TILES ? launch_forward<64>(g, s)
                                                               : launch_forward<32>(g, s);
    }
    return e;
}

// Forward pass of `batch` rows of X (FP32 device [batch x K_0]) on stream s.
cudaError_t forward(lbm_mlp *m, const float *x, int batch, cudaStream_t s) {
    to_bf16_rows<<<grid1((long long)batch * m->widths[0]), 256, 0, s>>>(x, m->actb[0], batch,
                                                                        m->widths[0]);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? forward_layers(m, batch, s) : e;
}

// dY of the rows the forward pass last ran against targets t (row j's target
// is row rows[j] of t; nullptr: row j), and the loss partial sums.
cudaError_t output_grad(lbm_mlp *m, const float *t, const int *rows, int batch, cudaStream_t s) {
    const int N = m->widths[m->layers];
    const long long no = (long long)batch * N;
    mse_grad<<<mse_blocks(no), 256, 0, s>>>(m->act, t, rows, no, N, 1.0f / (float)no, m->g0,
                                            m->gb, m->loss_part);
    return cudaGetLastError();
}

// The total loss (sum of squares) into loss_part[LOSS_BLOCKS].
cudaError_t total_loss(lbm_mlp *m, int batch, cudaStream_t s) {
    sum_loss<<<1, 256, 0, s>>>(m->loss_part, (int)mse_blocks((long long)batch * m->widths[m->layers]),
                               m->loss_part + LOSS_BLOCKS);
    return cudaGetLastError();
}

// Every parameter's gradient (into m->grads) after output_grad, on stream s;
// no host copy, no synchronisation.
cudaError_t backward(lbm_mlp *m, int batch, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    float *g = m->g0, *gn = m->g1;
    __nv_bfloat16 *gbf = m->gb, *gbn = m->gb1;
    for (int l = m->layers - 1; l >= 0 && e == cudaSuccess; --l) {
        const int K = m->widths[l], N = m->widths[l + 1];
        // dW_l = dZ_l^T X_l   ([N x K], sum over the batch)
        Product w{}, x{};
        w.A = gbf;
        w.lda = ld8(N);
        w.B = m->actb[l];
        w.ldb = ld8(K);
        w.out = m->grads + m->w_off[l];
        w.M = N;
        w.N = K;
        w.K = batch;
        long long big = tiles_of(N, 64) * tiles_of(K, 64);
        if (l > 0) {
            // dZ_{l-1} = (dZ_l W_l) (.) GELU'(Z_{l-1})   ([B x K], the GELU of
            // layer l - 1 in the product's epilogue)
            x.A = gbf;
            x.lda = ld8(N);
            x.B = m->wb + m->wb_off[l];
            x.ldb = ld8(K);
            x.aux = m->pre[l - 1];
            x.out = gn;
            x.outb = gbn;
            x.M = batch;
            x.N = K;
            x.K = N;
            x.epi = EPI_GELU_BWD;
            big += tiles_of(batch, 64) * tiles_of(K, 64);
        }
        e = big >= BIG_TILES ? launch_backward<64>(w, x, g, batch, N, m->grads + m->b_off[l], s)
                             : launch_backward<32>(w, x, g, batch, N, m->grads + m->b_off[l], s);
        std::swap(g, gn);
        std::swap(gbf, gbn);
    }
    return e;
}

}  // namespace

extern "C" {

lbm_status lbm_mlp_create(const int *widths, int n_widths, int max_batch, void *stream,
                          lbm_mlp **out) {
    if (!out) return mfail(nullptr, LBM_EINVAL, "out is NULL");
    *out = nullptr;
    if (!widths || n_widths < 2) return mfail(nullptr, LBM_EINVAL, "need at least 2 widths");
    if (max_batch < 1) return mfail(nullptr, LBM_EINVAL, "max_batch must be >= 1");
    for (int i = 0; i < n_widths; ++i)
        if (widths[i] < 1 || widths[i] > 65536)
            return mfail(nullptr, LBM_EINVAL, "layer widths must be in [1, 65536]");
    lbm_mlp *m = new lbm_mlp();
    cudaGetDevice(&m->device);
    m->stream = (cudaStream_t)stream;
    m->widths.assign(widths, widths + n_widths);
    m->layers = n_widths - 1;
    m->max_batch = max_batch;
    int wmax = 0;
    for (int l = 0; l < m->layers; ++l) {
        const int K = widths[l], N = widths[l + 1];
        m->w_off.push_back(m->n_params);
        m->n_params += (long long)N * K;
        m->b_off.push_back(m->n_params);
        m->n_params += N;
        m->wb_off.push_back(m->n_wb);
        m->n_wb += (long long)N * ld8(K);
    }
    for (int i = 0; i < n_widths; ++i) wmax = std::max(wmax, widths[i]);
    cudaError_t e = cudaSuccess;
    auto al = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    al((void **)&m->params, sizeof(float) * m->n_params);
    al((void **)&m->grads, sizeof(float) * m->n_params);
    al((void **)&m->m, sizeof(float) * m->n_params);
    al((void **)&m->v, sizeof(float) * m->n_params);
    al((void **)&m->wb, sizeof(__nv_bfloat16) * m->n_wb);
    al((void **)&m->wmap, sizeof(long long) * m->n_params);
    m->pre.assign(m->layers, nullptr);
    m->actb.assign(m->layers, nullptr);
    for (int l = 0; l < m->layers; ++l) {
        float **o = l < m->layers - 1 ? &m->pre[l] : &m->act;
        al((void **)o, sizeof(float) * (size_t)max_batch * widths[l + 1]);
        al((void **)&m->actb[l], sizeof(__nv_bfloat16) * (size_t)max_batch * ld8(widths[l]));
    }
    al((void **)&m->g0, sizeof(float) * (size_t)max_batch * wmax);
    al((void **)&m->g1, sizeof(float) * (size_t)max_batch * wmax);
    al((void **)&m->gb, sizeof(__nv_bfloat16) * (size_t)max_batch * ld8(wmax));
    al((void **)&m->gb1, sizeof(__nv_bfloat16) * (size_t)max_batch * ld8(wmax));
    al((void **)&m->loss_part, sizeof(double) * (LOSS_BLOCKS + 1));   // partials + total
    al((void **)&m->rows, sizeof(int) * (size_t)max_batch);
    if (e == cudaSuccess) {
        std::vector<long long> map(m->n_params, -1);
        for (int l = 0; l < m->layers; ++l) {
            const long long K = widths[l], nw = K * widths[l + 1];
            for (long long i = 0; i < nw; ++i)
                map[m->w_off[l] + i] = m->wb_off[l] + i / K * ld8(K) + i % K;
        }
        e = cudaMemcpy(m->wmap, map.data(), sizeof(long long) * m->n_params,
                       cudaMemcpyHostToDevice);
    }
    if (e == cudaSuccess) e = cudaMemset(m->params, 0, sizeof(float) * m->n_params);
    if (e == cudaSuccess) e = cudaMemset(m->m, 0, sizeof(float) * m->n_params);
    if (e == cudaSuccess) e = cudaMemset(m->v, 0, sizeof(float) * m->n_params);
    if (e == cudaSuccess) e = cudaMemset(m->wb, 0, sizeof(__nv_bfloat16) * m->n_wb);
    if (e != cudaSuccess) {
        lbm_status s = mcuda(nullptr, e, "lbm_mlp_create");
        lbm_mlp_destroy(m);
        return s;
    }
    *out = m;
    return LBM_OK;
}

void lbm_mlp_destroy(lbm_mlp *m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->params);
    cudaFree(m->grads);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->wb);
    cudaFree(m->wmap);
    for (auto p : m->pre) cudaFree(p);
    cudaFree(m->act);
    for (auto p : m->actb) cudaFree(p);
    cudaFree(m->g0);
    cudaFree(m->g1);
    cudaFree(m->gb);
    cudaFree(m->gb1);
    cudaFree(m->loss_part);
    cudaFree(m->tstate);
    cudaFree(m->rows);
    if (m->fork) cudaEventDestroy(m->fork);
    if (m->join) cudaEventDestroy(m->join);
    if (m->cap2) cudaStreamDestroy(m->cap2);
    if (m->cap) cudaStreamDestroy(m->cap);
    delete m;
}

size_t lbm_mlp_param_count(const lbm_mlp *m) { return m ? (size_t)m->n_params : 0; }

lbm_status lbm_mlp_set_params(lbm_mlp *m, const float *host) {
    if (!m || !host) return mfail(m, LBM_EINVAL, "NULL argument");
    MCK(m, cudaMemcpyAsync(m->params, host, sizeof(float) * m->n_params, cudaMemcpyHostToDevice,
                           m->stream));
    MCK(m, cudaMemsetAsync(m->m, 0, sizeof(float) * m->n_params, m->stream));
    MCK(m, cudaMemsetAsync(m->v, 0, sizeof(float) * m->n_params, m->stream));
    for (int l = 0; l < m->layers; ++l) {
        const long long nw = (long long)m->widths[l] * m->widths[l + 1];
        to_bf16_rows<<<grid1(nw), 256, 0, m->stream>>>(
            m->params + m->w_off[l], m->wb + m->wb_off[l], m->widths[l + 1], m->widths[l]);
        MCK(m, cudaGetLastError());
    }
    m->steps = 0;
    MCK(m, cudaStreamSynchronize(m->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp *m, float *host) {
    if (!m || !host) return mfail(m, LBM_EINVAL, "NULL argument");
    MCK(m, cudaMemcpyAsync(host, m->params, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost,
                           m->stream));
    MCK(m, cudaStreamSynchronize(m->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp *m, const float *x, int batch, float *y) {
    NvtxRange nvtx_("lbm_mlp_forward");
    if (!m || !x || !y) return mfail(m, LBM_EINVAL, "NULL argument");
    if (batch < 1 || batch > m->max_batch) return mfail(m, LBM_EINVAL, "batch out of range");
    MCK(m, forward(m, x, batch, m->stream));
    MCK(m, cudaMemcpyAsync(y, m->act,
                           sizeof(float) * (size_t)batch * m->widths[m->layers],
                           cudaMemcpyDeviceToDevice, m->stream));
    return LBM_OK;
}

// Loss and its gradient with respect to every parameter (into m->grads; a
// host copy when grads_host is not NULL).
static lbm_status loss_and_grad(lbm_mlp *m, const float *x, const float *t, int batch,
                                double *loss, float *grads_host) {
    cudaStream_t s = m->stream;
    MCK(m, forward(m, x, batch, s));
    MCK(m, output_grad(m, t, nullptr, batch, s));
    MCK(m, total_loss(m, batch, s));
    MCK(m, backward(m, batch, s));
    const long long no = (long long)batch * m->widths[m->layers];
    double hl = 0.0;
    MCK(m, cudaMemcpyAsync(&hl, m->loss_part + LOSS_BLOCKS, sizeof(double), cudaMemcpyDeviceToHost,
                           s));
    if (grads_host)
        MCK(m, cudaMemcpyAsync(grads_host, m->grads, sizeof(float) * m->n_params,
                               cudaMemcpyDeviceToHost, s));
    MCK(m, cudaStreamSynchronize(s));
    if (loss) *loss = hl / (double)no;
    return LBM_OK;
}

lbm_status lbm_mlp_loss_grad(lbm_mlp *m, const float *x, const float *t, int batch,
                             double *loss, float *grads_host) {
    if (!m || !x || !t) return mfail(m, LBM_EINVAL, "NULL argument");
    if (batch < 1 || batch > m->max_batch) return mfail(m, LBM_EINVAL, "batch out of range");
    return loss_and_grad(m, x, t, batch, loss, grads_host);
}

lbm_status lbm_mlp_train_step(lbm_mlp *m, const float *x, const float *t, int batch, float lr,
                              double *loss) {
    NvtxRange nvtx_("lbm_mlp_train_step");
    if (!m || !x || !t) return mfail(m, LBM_EINVAL, "NULL argument");
    if (batch < 1 || batch > m->max_batch) return mfail(m, LBM_EINVAL, "batch out of range");
    if (!(lr > 0.f)) return mfail(m, LBM_EINVAL, "lr must be > 0");
    if (lbm_status s = loss_and_grad(m, x, t, batch, loss, nullptr)) return s;
    m->steps += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - (float)std::pow(b1, (double)m->steps);
    const float c2 = 1.f - (float)std::pow(b2, (double)m->steps);
    adam<<<grid1(m->n_params), 256, 0, m->stream>>>(m->params, m->grads, m->m, m->v, m->n_params,
                                                    lr, b1, b2, 1e-8f, c1, c2, m->wmap, m->wb);
    MCK(m, cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp *m, const float *x, const float *t, int n, int batch,
                         long steps, float lr, float lr_final, unsigned long long seed,
                         float *loss_host) {
    NvtxRange nvtx_("lbm_mlp_train");
    if (!m || !x || !t) return mfail(m, LBM_EINVAL, "NULL argument");
    if (n < 1) return mfail(m, LBM_EINVAL, "n must be >= 1");
    if (batch < 1 || batch > m->max_batch) return mfail(m, LBM_EINVAL, "batch out of range");
    if (steps < 0) return mfail(m, LBM_EINVAL, "steps must be >= 0");
    if (!(lr > 0.f) || !(lr_final > 0.f)) return mfail(m, LBM_EINVAL, "learning rates must be > 0");
    if (steps == 0) return LBM_OK;
    const int L = m->layers, kx = m->widths[0], kt = m->widths[L];
    if (!m->tstate) {
        MCK(m, cudaMalloc(&m->tstate, sizeof(TrainState)));
    }
    if (!m->cap) MCK(m, cudaStreamCreateWithFlags(&m->cap, cudaStreamNonBlocking));
    if (!m->cap2) MCK(m, cudaStreamCreateWithFlags(&m->cap2, cudaStreamNonBlocking));
    if (!m->fork) MCK(m, cudaEventCreateWithFlags(&m->fork, cudaEventDisableTiming));
    if (!m->join) MCK(m, cudaEventCreateWithFlags(&m->join, cudaEventDisableTiming));
    TrainState st0{m->steps, 0, 0.f, 0.f, 0.f};
    float *hist = nullptr;
    MCK(m, cudaMalloc(&hist, sizeof(float) * (size_t)steps));
    cudaError_t e = cudaMemcpyAsync(m->tstate, &st0, sizeof(st0), cudaMemcpyHostToDevice,
                                    m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    // one Adam step, captured once and replayed: every per-step value (the
    // minibatch, the learning rate, the bias corrections) comes from the
    // device state, so the graph is the same for every step
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    const float b1 = 0.9f, b2 = 0.999f;
    if (e == cudaSuccess) e = cudaStreamBeginCapture(m->cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaStream_t s = m->cap, s2 = m->cap2;
        gather_rows<<<grid1(batch * ld8(kx)), 256, 0, s>>>(x, kx, m->tstate, seed, n, batch,
                                                           m->rows, m->actb[0]);
        cudaError_t le = cudaGetLastError();
        if (le == cudaSuccess) le = forward_layers(m, batch, s);
        if (le == cudaSuccess) le = output_grad(m, t, m->rows, batch, s);
        // beside the backward pass: the step's loss, its scalars and the counters
        if (le == cudaSuccess) le = cudaEventRecord(m->fork, s);
        if (le == cudaSuccess) le = cudaStreamWaitEvent(s2, m->fork, 0);
        if (le == cudaSuccess) le = total_loss(m, batch, s2);
        if (le == cudaSuccess) {
            train_setup<<<1, 1, 0, s2>>>(m->tstate, (long long)steps, lr, lr_final, b1, b2,
                                         m->loss_part + LOSS_BLOCKS, 1.0 / ((double)batch * kt),
                                         hist);
            le = cudaGetLastError();
        }
        if (le == cudaSuccess) le = cudaEventRecord(m->join, s2);
        if (le == cudaSuccess) le = backward(m, batch, s);
        if (le == cudaSuccess) le = cudaStreamWaitEvent(s, m->join, 0);
        if (le == cudaSuccess) {
            adam_dev<<<grid1(m->n_params), 256, 0, s>>>(m->params, m->grads, m->m, m->v,
                                                        m->n_params, b1, b2, 1e-8f, m->tstate,
                                                        m->wmap, m->wb);
            le = cudaGetLastError();
        }
        e = cudaStreamEndCapture(s, &g);
        if (le != cudaSuccess) e = le;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
    for (long i = 0; i < steps && e == cudaSuccess; ++i) e = cudaGraphLaunch(ge, m->stream);
    if (e == cudaSuccess && loss_host)
        e = cudaMemcpyAsync(loss_host, hist, sizeof(float) * (size_t)steps,
                            cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (ge) cudaGraphExecDestroy(ge);
    if (g) cudaGraphDestroy(g);
    cudaFree(hist);
    if (e != cudaSuccess) return mcuda(m, e, "lbm_mlp_train");
    m->steps += steps;
    return LBM_OK;
}

const char *lbm_mlp_last_error(const lbm_mlp *m) { return m ? m->err.c_str() : "mlp is NULL"; }

}  // extern "C"
