// nb_mlp.cu -- the learned opening-angle network: forward, backward,
// weight gradients and Adam, as hand-written kernels on the tensor cores.
//
// Network: 12 features -> 64 -> 64 -> 64 -> 1 with GELU, theta = 0.3 +
// 0.9 sigmoid(z).  Matrix products run as mma.sync m16n8k16 with BF16
// operands (layer inputs and weights rounded to BF16) and FP32 accumulation;
// biases, GELU, the output layer and all gradients outside the products are
// FP32.  Master weights are FP32 and are rounded to BF16 when fragments are
// loaded.  In inference a warp owns 16 samples (one m-tile); training runs in
// one thread-block cluster (k_mlp_train).  The matrices are tiny (K, N <=
// 64), so the warp-level MMA is used rather than 128-row tcgen05 tiles.
//
// Flat FP32 parameters (offsets in floats): W1 0 (64x16), b1 1024,
// W2 1088 (64x64), b2 5184, W3 5248, b3 9344, w4 9408 (64), b4 9920,
// mu 9928 (16), sigma 9944 (16); 9960 in all.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>

#include <type_traits>

#include "nb_internal.cuh"

#define MH 64
#define MKIN 16
#define MNIN 12
enum {
    P_W1 = 0, P_B1 = 1024, P_W2 = 1088, P_B2 = 5184, P_W3 = 5248, P_B3 = 9344,
    P_W4 = 9408, P_B4 = 9920, P_MU = 9928, P_SG = 9944, P_N = 9960
};
#define LAMBDA 4.0f
#define MLP_T 256

typedef __nv_bfloat16 bf16;
namespace cg = cooperative_groups;

// inference workspace (per padded sample count Bp), all offsets 256-byte
// aligned: the layers' BF16 inputs
struct MlpWork {
    bf16 *a0, *a1, *a2;
};

static size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

static size_t work_layout(int64_t Bp, MlpWork *w, char *base)
{
    size_t o = 0;
#define PUT(f, T, cnt)                                          \
    do {                                                        \
        if (w) w->f = (T *)(base + o);                          \
        o += al(sizeof(T) * (size_t)(cnt));                     \
    } while (0)
    PUT(a0, bf16, Bp * MKIN);
    PUT(a1, bf16, Bp * MH);
    PUT(a2, bf16, Bp * MH);
#undef PUT
    return o;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], const uint32_t b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float gelu(float x)
{
    return x * 0.5f * (1.0f + erff(x * 0.70710678118654752f));
}

// gelu(x) and its derivative from one erff (the product in the derivative is
// rounded on its own)
__device__ __forceinline__ float gelu_both(float x, float *grad)
{
    const float Phi = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
    const float phi = expf(-0.5f * x * x) * 0.39894228040143268f;
    *grad = __fadd_rn(Phi, __fmul_rn(x, phi));
    return x * Phi;
}

// A fragment (16 x 16) of a row-major BF16 matrix X (rows r0.., cols k0..)
__device__ __forceinline__ void frag_a_rows(const bf16 *X, int ld, int r0, int k0, uint32_t a[4])
{
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    a[0] = *reinterpret_cast<const uint32_t *>(X + (int64_t)(r0 + g) * ld + k0 + 2 * t);
    a[1] = *reinterpret_cast<const uint32_t *>(X + (int64_t)(r0 + g + 8) * ld + k0 + 2 * t);
    a[2] = *reinterpret_cast<const uint32_t *>(X + (int64_t)(r0 + g) * ld + k0 + 8 + 2 * t);
    a[3] = *reinterpret_cast<const uint32_t *>(X + (int64_t)(r0 + g + 8) * ld + k0 + 8 + 2 * t);
}

// B fragment (16 x 8) with B(k, n) = W[n][k], W FP32 row-major with K columns
__device__ __forceinline__ void frag_b_wt(const float *W, int K, int k0, int n0, uint32_t b[2])
{
    const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
    const float *p = W + (int64_t)(n0 + g) * K + k0 + 2 * t;
    b[0] = pack2(p[0], p[1]);
    b[1] = pack2(p[8], p[9]);
}

// one hidden layer for a 16-row tile: acc = A (16 x K, BF16 rows) * W^T
template <int K>
__device__ __forceinline__ void mma_layer(const bf16 *A, int ldA, int r0, const float *W,
                                          float acc[8][4])
{
    uint32_t a[4], b[2];
#pragma unroll
    for (int nt = 0; nt < 8; nt++) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
    for (int kt = 0; kt < K / 16; kt++) {
        frag_a_rows(A, ldA, r0, kt * 16, a);
#pragma unroll
        for (int nt = 0; nt < 8; nt++) {
            frag_b_wt(W, K, kt * 16, nt * 8, b);
            mma16816(acc[nt], a, b);
        }
    }
}

// z = w4 . h3 + b4 for the two rows (g, g + 8) a lane holds, FP32
__device__ __forceinline__ void out_z(const float acc[8][4], const float *P, float z[2])
{
    const int t = threadIdx.x & 3;
    float zr[2] = {0.f, 0.f};
#pragma unroll
    for (int nt = 0; nt < 8; nt++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int col = nt * 8 + 2 * t;
            zr[h] = fmaf(acc[nt][2 * h], P[P_W4 + col], zr[h]);
            zr[h] = fmaf(acc[nt][2 * h + 1], P[P_W4 + col + 1], zr[h]);
        }
#pragma unroll
    for (int h = 0; h < 2; h++) {
        zr[h] += __shfl_xor_sync(0xffffffffu, zr[h], 1);
        zr[h] += __shfl_xor_sync(0xffffffffu, zr[h], 2);
        z[h] = zr[h] + P[P_B4];
    }
}

__device__ __forceinline__ float norm_feature(const float *x, const float *P, int k)
{
    return k < MNIN ? __fdiv_rn(__fsub_rn(x[k], P[P_MU + k]), P[P_SG + k]) : 0.0f;
}

// ------------------------------------------------------------ input
// z0 = (x - mu) / sigma in FP32, rounded to BF16, padded to 16 columns;
// rows >= B are zero.  x has 16-float rows.
__global__ void __launch_bounds__(256)
k_mlp_input(const float *__restrict__ x, int64_t B, int64_t Bp, const float *__restrict__ P,
            bf16 *__restrict__ a0)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= Bp * MKIN) return;
    const int64_t r = i / MKIN;
    const int k = (int)(i % MKIN);
    float v = 0.0f;
    if (r < B && k < MNIN) v = norm_feature(x + r * MKIN, P, k);
    a0[i] = __float2bfloat16_rn(v);
}

// ------------------------------------------------------------ forward
// one warp per 16-sample tile
__global__ void __launch_bounds__(MLP_T)
k_mlp_fwd(const float *__restrict__ P, int64_t Bp, MlpWork w, float *__restrict__ theta_out,
          int64_t B, float fallback)
{
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int64_t tile = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (tile * 16 >= Bp) return;
    const int r0 = (int)(tile * 16);
    float acc[8][4];
    const float *Ws[3] = {P + P_W1, P + P_W2, P + P_W3};
    const float *bs[3] = {P + P_B1, P + P_B2, P + P_B3};
    const bf16 *ins[3] = {w.a0, w.a1, w.a2};
    bf16 *outs[2] = {w.a1, w.a2};
    for (int L = 0; L < 3; L++) {
        if (L == 0) mma_layer<MKIN>(ins[0], MKIN, r0, Ws[0], acc);
        else mma_layer<MH>(ins[L], MH, r0, Ws[L], acc);
#pragma unroll
        for (int nt = 0; nt < 8; nt++)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = r0 + g + 8 * h, col = nt * 8 + 2 * t;
                const float z0 = acc[nt][2 * h] + bs[L][col];
                const float z1 = acc[nt][2 * h + 1] + bs[L][col + 1];
                const float g0 = gelu(z0), g1 = gelu(z1);
                acc[nt][2 * h] = g0;
                acc[nt][2 * h + 1] = g1;
                if (L < 2)
                    *reinterpret_cast<uint32_t *>(outs[L] + (int64_t)row * MH + col) = pack2(g0, g1);
            }
        __syncwarp();
    }
    float z[2];
    out_z(acc, P, z);
    if (t == 0)
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int row = r0 + g + 8 * h;
            const float s = 1.0f / (1.0f + expf(-z[h]));
            float th = 0.3f + 0.9f * s;
            if (row < B) {
                if (!isfinite(th)) th = fallback;
                theta_out[row] = th;
            }
        }
}

// Inference for every group of a context: the same arithmetic as k_mlp_fwd
// with the layer activations in shared memory; the group count is read on
// the device (no host synchronisation, no workspace).
__global__ void __launch_bounds__(MLP_T)
k_mlp_infer(const float *__restrict__ P, const float *__restrict__ feat,
            const long long *__restrict__ cnt, float *__restrict__ theta, float fallback)
{
    nb_grid_wait();
    __shared__ __align__(16) bf16 sbuf[MLP_T / 32][2][16 * MH];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int64_t G = cnt[CNT_GROUPS];
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    bf16 *b0 = sbuf[wl][0], *b1 = sbuf[wl][1];
    for (int64_t tile = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; tile * 16 < G;
         tile += nwarps) {
        const int64_t r0 = tile * 16;
        for (int e = lane; e < 16 * MKIN; e += 32) {
            const int r = e / MKIN, k = e % MKIN;
            const float v = r0 + r < G ? norm_feature(feat + (r0 + r) * MKIN, P, k) : 0.0f;
            b0[r * MKIN + k] = __float2bfloat16_rn(v);
        }
        __syncwarp();
        float acc[8][4];
        const float *Ws[3] = {P + P_W1, P + P_W2, P + P_W3};
        const float *bs[3] = {P + P_B1, P + P_B2, P + P_B3};
        for (int L = 0; L < 3; L++) {
            bf16 *src = (L == 1) ? b1 : b0;
            bf16 *dst = (L == 1) ? b0 : b1;
            if (L == 0) mma_layer<MKIN>(src, MKIN, 0, Ws[0], acc);
            else mma_layer<MH>(src, MH, 0, Ws[L], acc);
            __syncwarp();
#pragma unroll
            for (int nt = 0; nt < 8; nt++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int row = g + 8 * h, col = nt * 8 + 2 * t;
                    const float g0 = gelu(acc[nt][2 * h] + bs[L][col]);
                    const float g1 = gelu(acc[nt][2 * h + 1] + bs[L][col + 1]);
                    acc[nt][2 * h] = g0;
                    acc[nt][2 * h + 1] = g1;
                    if (L < 2) *reinterpret_cast<uint32_t *>(dst + row * MH + col) = pack2(g0, g1);
                }
            __syncwarp();
        }
        float z[2];
        out_z(acc, P, z);
        if (t == 0)
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int64_t row = r0 + g + 8 * h;
                if (row < G) {
                    float th = 0.3f + 0.9f * (1.0f / (1.0f + expf(-z[h])));
                    theta[row] = isfinite(th) ? th : fallback;
                }
            }
        __syncwarp();
    }
}

void nb_launch_mlp_infer(nb_ctx *c, const float *params, const float *feat, float *theta,
                         float fallback)
{
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_mlp_infer, MLP_T, 0);
    if (blocks < 1) blocks = 1;
    nb_launch(k_mlp_infer, c->num_sms * blocks, MLP_T, 0, nb_queue(c), params, feat, c->cnt, theta,
              fallback);
    nb_launched(c, "k_mlp_infer");
}

// ------------------------------------------------------------ training data
// Median relative force error of each sampled group: rows off[k] .. off[k+1]
// of ref (FP64 judge accelerations) belong to sampled group k, targets[]
// gives their caller index into acc.  One warp per group, bitonic sort of up
// to 1024 errors in shared memory; median = mean of the two middle values.
#define GE_MAX 1024
__global__ void __launch_bounds__(128)
k_group_errors(const float *__restrict__ acc, const double *__restrict__ ref,
               const int64_t *__restrict__ targets, const int64_t *__restrict__ off, int64_t S,
               float *__restrict__ err)
{
    __shared__ float buf[4][GE_MAX];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (k >= S) return;
    const int64_t a = off[k];
    int n = (int)(off[k + 1] - a);
    if (n > GE_MAX) n = GE_MAX;
    int np = 1;
    while (np < n) np <<= 1;
    float *e = buf[wl];
    for (int i = lane; i < np; i += 32) {
        float v = INFINITY;
        if (i < n) {
            const int64_t o = targets[a + i];
            const double rx = ref[3 * (a + i)], ry = ref[3 * (a + i) + 1], rz = ref[3 * (a + i) + 2];
            const double dx = (double)acc[3 * o] - rx, dy = (double)acc[3 * o + 1] - ry,
                         dz = (double)acc[3 * o + 2] - rz;
            const double r = sqrt(rx * rx + ry * ry + rz * rz);
            v = (float)(sqrt(dx * dx + dy * dy + dz * dz) / (r > 0.0 ? r : 1.0));
        }
        e[i] = v;
    }
    __syncwarp();
    for (int size = 2; size <= np; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = lane; i < np; i += 32) {
                const int j = i ^ stride;
                if (j > i) {
                    const bool up = (i & size) == 0;
                    const float x = e[i], y = e[j];
                    if ((x > y) == up) { e[i] = y; e[j] = x; }
                }
            }
            __syncwarp();
        }
    if (lane == 0) err[k] = n > 0 ? 0.5f * (e[(n - 1) / 2] + e[n / 2]) : 0.0f;
}

// Label of each sample from its error curve err[t][k] (T x S, grid
// ascending).  Without costs: the largest grid theta whose error meets the
// budget (the smallest grid theta when none does).  With costs (interactions
// of the group at each theta) and group sizes: the grid theta minimising
// cost / n + lambda * ln(error), the allocation that trades interactions
// against error at one exchange rate lambda for every group.
__global__ void k_theta_labels(const float *__restrict__ err, const float *__restrict__ cost,
                               const float *__restrict__ nsz, const float *__restrict__ grid,
                               int T, int64_t S, float budget, float lambda,
                               float *__restrict__ labels)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= S) return;
    float lab = grid[0];
    if (!cost) {
        for (int t = 0; t < T; t++)
            if (err[(int64_t)t * S + k] <= budget) lab = grid[t];
    } else {
        float best = INFINITY;
        for (int t = 0; t < T; t++) {
            const float o = cost[(int64_t)t * S + k] / nsz[k] +
                            lambda * logf(fmaxf(err[(int64_t)t * S + k], 1e-9f));
            if (o < best) { best = o; lab = grid[t]; }
        }
    }
    labels[k] = lab;
}

extern "C" int nb_group_errors(const float *acc_dev, const double *ref_dev,
                               const int64_t *targets_dev, const int64_t *off_dev, int64_t S,
                               float *err_dev, void *stream)
{
    if (S < 0 || (S > 0 && (!acc_dev || !ref_dev || !targets_dev || !off_dev || !err_dev)))
        return NB_ERR_INVALID_ARG;
    if (S == 0) return NB_OK;
    k_group_errors<<<(int)((S * 32 + 127) / 128), 128, 0, (cudaStream_t)stream>>>(
        acc_dev, ref_dev, targets_dev, off_dev, S, err_dev);
    return cudaGetLastError() == cudaSuccess ? NB_OK : NB_ERR_CUDA;
}

extern "C" int nb_theta_labels(const float *err_dev, const float *cost_dev,
                               const float *size_dev, const float *grid_dev, int T, int64_t S,
                               float budget, float lambda, float *labels_dev, void *stream)
{
    if (T < 1 || S < 0 || (S > 0 && (!err_dev || !grid_dev || !labels_dev)) ||
        (cost_dev && !size_dev))
        return NB_ERR_INVALID_ARG;
    if (S == 0) return NB_OK;
    k_theta_labels<<<nb_grid(S, 256), 256, 0, (cudaStream_t)stream>>>(
        err_dev, cost_dev, size_dev, grid_dev, T, S, budget, lambda, labels_dev);
    return cudaGetLastError() == cudaSuccess ? NB_OK : NB_ERR_CUDA;
}

// ------------------------------------------------------------ training
// Forward, backward, weight gradients and Adam of consecutive batches in one
// launch of one thread-block cluster, the parameters held in shared memory.
//
// A step is a chain of ten small dependent products and reductions, bound by
// their latency, not by arithmetic (256 samples: 14 MFLOP).  As four launches
// a step over device memory it took 94 us, most of it in weight and bias sums
// that walked the batch in 11 blocks; it takes 9.8 us so (256 samples, a
// cluster of 16 blocks; 10.2 before the bias sums took their tiles in two
// alternating register sets and the next tile was put down between the two
// halves of the step's last barrier).
//
// Phase A: a block takes one 16-sample tile (tile k of a round goes to block
// k) forward and back.  Its 8 warps split a layer's 64 outputs, 8 columns
// each, so a lane holds the same 4 elements (rows g, g + 8, columns 2t, 2t + 1
// of its 8) of every layer's output and of its gradient.  It leaves its
// activations and gradients in the workspace.  Phase B: a block owns a part
// of the parameters (two 16x8 tiles each of W2 and W3, half of the blocks one
// of W1, 16 of the 256 bias and w4 entries), fetches the columns it needs and
// sums their gradients over the whole batch in sample order: dZ^T X by
// chained MMAs over the tiles, the bias and w4 entries one column per lane.
// The sums therefore do not depend on timing or on the split.  Batches of
// more than 16 CL samples take several rounds.  The owner then applies Adam
// with m and v in registers, and every block fetches the new parameters.
//
// The blocks exchange through L2 (written, cluster barrier, read past L1)
// and not through each other's shared memory: with remote 16-byte stores
// the 55 KB a block sends and the 38 KB of parameters took 16,500 of a step's
// 23,000 cycles.  Blocks in a cluster run together by definition, so the
// cluster barriers need no bound.  A launch covers at most MT_STEPS steps.
#define MT_T 256
#define MT_STEPS 256
#define MT_LD 72    // row stride of the 16 x 64 BF16 tiles (conflict-free ldmatrix)
#define MT_LD0 24   // ... of 16-column BF16 tiles
#define MT_LDF 68   // ... of the 16 x 64 FP32 tiles
#define MT_WLD 68   // row stride of W2, W3 in shared memory
#define MT_WLD0 20  // ... of W1
// shared parameter copy: the flat layout with padded rows
enum {
    S_W1 = 0, S_B1 = S_W1 + MH * MT_WLD0, S_W2 = S_B1 + MH, S_B2 = S_W2 + MH * MT_WLD,
    S_W3 = S_B2 + MH, S_B3 = S_W3 + MH * MT_WLD, S_W4 = S_B3 + MH, S_B4 = S_W4 + MH, S_N = S_B4 + 4
};

// per-step bias corrections of Adam, 1 - 0.9^t and 1 - 0.999^t
struct AdamCorr {
    float c1[MT_STEPS], c2[MT_STEPS];
};

// what the blocks exchange (in the caller's workspace): per tile of a round
// the 16-column blocks of each BF16 tile (8-column halves of the input), the
// FP32 columns of f, dz and the losses; and the parameters
struct TrainShare {
    bf16 d1[16][4][256], d2[16][4][256], d3[16][4][256], a1[16][4][256], a2[16][4][256];
    bf16 a0[16][2][128];
    float f[16][4][4][256];   // tile, quantity, 16-column block
    float dz[16][16], ls[16][16];
    float P[P_W4 + MH + 4];   // b4 last
};

struct TrainSmem {
    float P[S_N];
    // this block's tile: layer inputs and gradients in BF16; FP32 gradients
    // of the three layers and the last layer's output
    bf16 a0[16 * MT_LD0], a1[16 * MT_LD], a2[16 * MT_LD];
    bf16 d1[16 * MT_LD], d2[16 * MT_LD], d3[16 * MT_LD];
    float f[4][16 * MT_LDF];
    float dz[16], ls[16], y[16], mu[MKIN], sg[MKIN];
    // what this block fetched, 16 (owner slot, tile) pairs: the columns of
    // the owned gradient tiles, the owned columns of f; dz and the losses
    bf16 rd1[16][16 * MT_LD0], rd2[16][16 * MT_LD0], rd3[16][16 * MT_LD0];
    bf16 ra1[16][16 * MT_LD0], ra2[16][16 * MT_LD0], ra0[16][16 * 8];
    float rf[16][16 * 16], rdz[16][16], rls[16][16];
};

// (callers' buffers may sit at any 4-byte offset)
__device__ __forceinline__ float4 load4(const float *p)
{
    return make_float4(p[0], p[1], p[2], p[3]);
}

// place of flat parameter i < P_W4 + MH in the shared copy
__device__ __forceinline__ int smem_place(int i)
{
    if (i < P_B1) return S_W1 + (i >> 4) * MT_WLD0 + (i & 15);
    if (i < P_W2) return S_B1 + i - P_B1;
    if (i < P_B2) return S_W2 + ((i - P_W2) >> 6) * MT_WLD + ((i - P_W2) & 63);
    if (i < P_W3) return S_B2 + i - P_B2;
    if (i < P_B3) return S_W3 + ((i - P_W3) >> 6) * MT_WLD + ((i - P_W3) & 63);
    if (i < P_W4) return S_B3 + i - P_B3;
    return S_W4 + i - P_W4;
}

// 16 bytes to shared memory, read past L1
__device__ __forceinline__ void fetch16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src) : "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldm4(uint32_t a[4], const bf16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(smem_addr(p)) : "memory");
}

__device__ __forceinline__ void ldm4t(uint32_t a[4], const bf16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(smem_addr(p)) : "memory");
}

__device__ __forceinline__ void ldm2t(uint32_t b[2], const bf16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(b[0]), "=r"(b[1]) : "r"(smem_addr(p)) : "memory");
}

// 16 rows x 16 KT of A (BF16, row stride ld) times a B whose fragments come
// from the FP32 matrix W (row stride wld): B(k, n) = W[n][k], or W[k][n] (TR)
template <int KT, bool TR>
__device__ __forceinline__ void tile_mma(float c[4], const bf16 *A, int ld, const float *W, int wld,
                                         int n0, int lane)
{
    const int g = lane >> 2, t = lane & 3;
    const bf16 *ap = A + ((lane & 7) + ((lane >> 3) & 1) * 8) * ld + (lane >> 4) * 8;
    c[0] = c[1] = c[2] = c[3] = 0.f;
#pragma unroll
    for (int kt = 0; kt < KT; kt++) {
        uint32_t a[4], b[2];
        ldm4(a, ap + kt * 16);
        if (TR) {
            const float *p = W + (kt * 16 + 2 * t) * wld + n0 + g;
            b[0] = pack2(p[0], p[wld]);
            b[1] = pack2(p[8 * wld], p[9 * wld]);
        } else {
            const float2 *p = reinterpret_cast<const float2 *>(W + (n0 + g) * wld + kt * 16 + 2 * t);
            b[0] = pack2(p[0].x, p[0].y);
            b[1] = pack2(p[4].x, p[4].y);
        }
        mma16816(c, a, b);
    }
}

__device__ __forceinline__ void put_tile(bf16 *X, int w, int g, int t, const float v[4])
{
    *reinterpret_cast<uint32_t *>(X + g * MT_LD + w * 8 + 2 * t) = pack2(v[0], v[1]);
    *reinterpret_cast<uint32_t *>(X + (g + 8) * MT_LD + w * 8 + 2 * t) = pack2(v[2], v[3]);
}

__device__ __forceinline__ void put_f32(float *X, int w, int g, int t, const float v[4])
{
    *reinterpret_cast<float2 *>(X + g * MT_LDF + w * 8 + 2 * t) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2 *>(X + (g + 8) * MT_LDF + w * 8 + 2 * t) = make_float2(v[2], v[3]);
}

__device__ __forceinline__ float adam_step(float p, float gi, float &m, float &v, float lr, float c1,
                                           float c2)
{
    const float mi = 0.9f * m + 0.1f * gi;
    const float vi = 0.999f * v + 0.001f * gi * gi;
    m = mi;
    v = vi;
    return p - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

// steps step0 .. step0 + nsteps - 1 (TRAIN), or the gradient of one batch.
// order (nullable: identity) holds n sample indices per epoch.  grad receives
// the gradient (TRAIN false), loss the summed loss (TRAIN: per epoch; added to
// what is there, nullable).
template <int CL, bool TRAIN>
__global__ void __launch_bounds__(MT_T, 1)
k_mlp_train(float *__restrict__ P, float *__restrict__ am, float *__restrict__ av,
            const float *__restrict__ feat, const float *__restrict__ labels,
            const int32_t *__restrict__ order, int64_t n, int64_t batch, int64_t steps_per_epoch,
            int64_t step0, int nsteps, float lr, const AdamCorr corr, TrainShare *share,
            float *__restrict__ grad, float *__restrict__ loss)
{
    extern __shared__ __align__(16) unsigned char mt_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(mt_smem);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, t = lane & 3;
    constexpr int VR = 16 / CL;   // owner slots per block: slots rank VR .. rank VR + VR - 1
    TrainShare &X = *share;
    const int64_t ntiles = (batch + 15) / 16, rounds = (ntiles + CL - 1) / CL;
    const float invB = 1.0f / (float)batch;

    // parameters into the shared copy (every block)
    for (int q = tid; q < (P_W4 + MH) / 4; q += MT_T)
        *reinterpret_cast<float4 *>(S.P + smem_place(4 * q)) = load4(P + 4 * q);
    if (tid == 0) S.P[S_B4] = P[P_B4];
    if (tid < MKIN) {
        S.mu[tid] = P[P_MU + tid];
        S.sg[tid] = P[P_SG + tid];
    }

    // what this lane owns in slot v (flat parameter index, -1: nothing).
    // Warps 0, 1: W3; 2, 3: W2 (two 16x8 tiles each); 4: W1; 5: bias and w4
    // entries, a lane per column; 6: b4
    int own[VR], og[VR][2];   // element (row g, column 2t); offsets of rows g, g + 8
    bool has[VR];
    float om[VR][4], ov[VR][4];
#pragma unroll
    for (int v = 0; v < VR; v++) {
        const int vr = rank * VR + v;
        has[v] = false;
        own[v] = 0;
        int ld = MH;
        if (w < 4) {
            has[v] = true;
            own[v] = (w < 2 ? P_W3 : P_W2) + ((vr >> 2) * 16 + g) * MH + (2 * (vr & 3) + (w & 1)) * 8 +
                     2 * t;
        } else if (w == 4) {
            has[v] = vr < 8;
            ld = MKIN;
            own[v] = P_W1 + ((vr >> 1) * 16 + g) * MKIN + (vr & 1) * 8 + 2 * t;
        } else if (w == 5) {
            has[v] = lane < 16;
            const int which = vr >> 2;
            own[v] = (which == 0 ? P_B1 : which == 1 ? P_B2 : which == 2 ? P_B3 : P_W4) +
                     (vr & 3) * 16 + (lane & 15);
        } else if (w == 6) {
            has[v] = vr == 0 && lane == 0;
            own[v] = P_B4;
        }
        og[v][0] = own[v];
        og[v][1] = own[v] + 8 * ld;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            om[v][e] = ov[v][e] = 0.f;
            if (TRAIN && has[v] && (w < 5 || e == 0)) {
                om[v][e] = am[og[v][e >> 1] + (e & 1)];
                ov[v][e] = av[og[v][e >> 1] + (e & 1)];
            }
        }
    }

    // this thread's input element of a tile: row tid / 16, feature tid % 16.
    // The sample index is fetched two tiles ahead and the feature (and label)
    // one tile ahead.
    const int row = tid >> 4, col = tid & 15;
    int64_t s2 = 0, j2 = 0;   // the (step, round) whose index is fetched next
    int64_t e2 = step0 / steps_per_epoch, k2 = step0 - e2 * steps_per_epoch;   // ... its batch
    auto next_sample = [&]() -> int64_t {
        if (s2 >= nsteps) return -1;
        const int64_t r = (rank + j2 * CL) * 16 + row;
        const int64_t i = r >= batch ? -1 : !order ? r : order[e2 * n + k2 * batch + r];
        if (++j2 == rounds) {
            j2 = 0;
            s2++;
            if (++k2 == steps_per_epoch) {
                k2 = 0;
                e2++;
            }
        }
        return i;
    };
    float x1 = 0.f, y1 = 0.f;
    bool ok1 = false;
    auto fetch = [&](int64_t i) {
        ok1 = i >= 0;
        x1 = ok1 && col < MNIN ? feat[i * MKIN + col] : 0.f;
        y1 = ok1 && col == 0 ? labels[i] : 0.f;
    };
    int64_t i1 = next_sample();
    fetch(i1);
    i1 = next_sample();
    // the tile's input rows and labels into shared memory; the next one's are
    // fetched
    auto put_input = [&](bool has_tile) {
        if (has_tile) {
            S.a0[row * MT_LD0 + col] = __float2bfloat16_rn(
                ok1 && col < MNIN ? __fdiv_rn(__fsub_rn(x1, S.mu[col]), S.sg[col]) : 0.f);
            if (col == 0) S.y[row] = y1;
        }
        fetch(i1);
        i1 = next_sample();
    };
    // the running loss of the current epoch (one lane of block 0)
    int64_t le = step0 / steps_per_epoch, lk = step0 - le * steps_per_epoch;
    float lrun = 0.f;
    if (rank == 0 && w == 6 && loss) lrun = loss[TRAIN ? le : 0];
    __syncthreads();   // mu and sigma
    put_input(rank < ntiles);
    cl.sync();

    for (int s = 0; s < nsteps; s++) {
        float acc[VR][4], lacc = 0.f;
#pragma unroll
        for (int v = 0; v < VR; v++)
#pragma unroll
            for (int e = 0; e < 4; e++) acc[v][e] = 0.f;
        for (int64_t j = 0; j < rounds; j++) {
            const int64_t base = j * CL;                 // first tile of the round
            const int nk = ntiles - base < CL ? (int)(ntiles - base) : CL;
            if (j > 0) put_input(rank < nk);
            __syncthreads();
            if (rank < nk) {
                const int c0 = w * 8 + 2 * t;
                float z[4], h[4], g1[4], g2[4], g3[4], d[4];
                tile_mma<1, false>(z, S.a0, MT_LD0, S.P + S_W1, MT_WLD0, w * 8, lane);
#pragma unroll
                for (int e = 0; e < 4; e++) h[e] = gelu_both(z[e] + S.P[S_B1 + c0 + (e & 1)], &g1[e]);
                put_tile(S.a1, w, g, t, h);
                __syncthreads();
                tile_mma<4, false>(z, S.a1, MT_LD, S.P + S_W2, MT_WLD, w * 8, lane);
#pragma unroll
                for (int e = 0; e < 4; e++) h[e] = gelu_both(z[e] + S.P[S_B2 + c0 + (e & 1)], &g2[e]);
                put_tile(S.a2, w, g, t, h);
                __syncthreads();
                tile_mma<4, false>(z, S.a2, MT_LD, S.P + S_W3, MT_WLD, w * 8, lane);
#pragma unroll
                for (int e = 0; e < 4; e++) h[e] = gelu_both(z[e] + S.P[S_B3 + c0 + (e & 1)], &g3[e]);
                put_f32(S.f[3], w, g, t, h);
                __syncthreads();
                // z = w4 . h3 + b4 of rows g and g + 8 (every warp alike, in
                // the order of out_z), theta and dL/dz
                float zr[2] = {0.f, 0.f}, dz[2];
#pragma unroll
                for (int nt = 0; nt < 8; nt++) {
                    const float2 u = *reinterpret_cast<const float2 *>(S.P + S_W4 + nt * 8 + 2 * t);
#pragma unroll
                    for (int r = 0; r < 2; r++) {
                        const float2 q = *reinterpret_cast<const float2 *>(
                            S.f[3] + (g + 8 * r) * MT_LDF + nt * 8 + 2 * t);
                        zr[r] = fmaf(q.x, u.x, zr[r]);
                        zr[r] = fmaf(q.y, u.y, zr[r]);
                    }
                }
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    zr[r] += __shfl_xor_sync(0xffffffffu, zr[r], 1);
                    zr[r] += __shfl_xor_sync(0xffffffffu, zr[r], 2);
                    const float zz = zr[r] + S.P[S_B4];
                    const float sg = 1.0f / (1.0f + expf(-zz));
                    const float th = 0.3f + 0.9f * sg;
                    const float dd = th - S.y[g + 8 * r];
                    const float dth = (2.0f * dd + 2.0f * LAMBDA * fmaxf(dd, 0.0f)) * invB;
                    const bool in = (base + rank) * 16 + g + 8 * r < batch;
                    dz[r] = in ? dth * 0.9f * sg * (1.0f - sg) : 0.f;
                    const float l = dd * dd + LAMBDA * fmaxf(dd, 0.0f) * fmaxf(dd, 0.0f);
                    if (w == 0 && t == 0) {
                        S.dz[g + 8 * r] = dz[r];
                        S.ls[g + 8 * r] = in ? l : 0.f;
                    }
                }
                // backward
                const float u0 = S.P[S_W4 + c0], u1 = S.P[S_W4 + c0 + 1];
#pragma unroll
                for (int e = 0; e < 4; e++) d[e] = dz[e >> 1] * ((e & 1) ? u1 : u0) * g3[e];
                put_tile(S.d3, w, g, t, d);
                put_f32(S.f[2], w, g, t, d);
                __syncthreads();
                tile_mma<4, true>(d, S.d3, MT_LD, S.P + S_W3, MT_WLD, w * 8, lane);
#pragma unroll
                for (int e = 0; e < 4; e++) d[e] *= g2[e];
                put_tile(S.d2, w, g, t, d);
                put_f32(S.f[1], w, g, t, d);
                __syncthreads();
                tile_mma<4, true>(d, S.d2, MT_LD, S.P + S_W2, MT_WLD, w * 8, lane);
#pragma unroll
                for (int e = 0; e < 4; e++) d[e] *= g1[e];
                put_tile(S.d1, w, g, t, d);
                put_f32(S.f[0], w, g, t, d);
                __syncthreads();
                // leave the tile for the owners, 16 bytes a store
                {
                    const int c = tid & 127, r = c >> 3, ch = c & 7;   // row, 8-column chunk
                    const int blk = ch >> 1, dst = r * 16 + (ch & 1) * 8, src = r * MT_LD + ch * 8;
                    auto put = [&](bf16 *to, const bf16 *from) {
                        *reinterpret_cast<uint4 *>(to + dst) =
                            *reinterpret_cast<const uint4 *>(from + src);
                    };
                    if (tid < 128) {
                        put(X.d3[rank][blk], S.d3);
                        put(X.d2[rank][blk], S.d2);
                        put(X.d1[rank][blk], S.d1);
                    } else {
                        put(X.a2[rank][blk], S.a2);
                        put(X.a1[rank][blk], S.a1);
                        if (c < 32)   // (row, half) of the input tile
                            *reinterpret_cast<uint4 *>(X.a0[rank][c & 1] + (c >> 1) * 8) =
                                *reinterpret_cast<const uint4 *>(S.a0 + (c >> 1) * MT_LD0 +
                                                                 (c & 1) * 8);
                        else if (c < 36)
                            *reinterpret_cast<float4 *>(X.dz[rank] + (c & 3) * 4) =
                                *reinterpret_cast<const float4 *>(S.dz + (c & 3) * 4);
                        else if (c < 40)
                            *reinterpret_cast<float4 *>(X.ls[rank] + (c & 3) * 4) =
                                *reinterpret_cast<const float4 *>(S.ls + (c & 3) * 4);
                    }
                    // FP32 columns: row tid / 16, 4-column chunk tid % 16
                    const int rr = tid >> 4, c4 = tid & 15;
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        *reinterpret_cast<float4 *>(X.f[rank][k][c4 >> 2] + rr * 16 + (c4 & 3) * 4) =
                            *reinterpret_cast<const float4 *>(S.f[k] + rr * MT_LDF + c4 * 4);
                }
            }
            cl.sync();
            // fetch the owners' columns of the round's tiles
#pragma unroll
            for (int v = 0; v < VR; v++) {
                const int vr = rank * VR + v, hi = vr >> 2, lo = vr & 3;
                for (int q = tid; q < nk * 32; q += MT_T) {
                    const int k = q >> 5, r = (q >> 1) & 15, hf = q & 1;
                    const int src = r * 16 + hf * 8, dst = r * MT_LD0 + hf * 8, at = v * CL + k;
                    fetch16(&S.rd3[at][dst], &X.d3[k][hi][src]);
                    fetch16(&S.rd2[at][dst], &X.d2[k][hi][src]);
                    fetch16(&S.ra2[at][dst], &X.a2[k][lo][src]);
                    fetch16(&S.ra1[at][dst], &X.a1[k][lo][src]);
                    if (vr < 8) {
                        fetch16(&S.rd1[at][dst], &X.d1[k][vr >> 1][src]);
                        if (hf == 0) fetch16(&S.ra0[at][r * 8], &X.a0[k][vr & 1][r * 8]);
                    }
                }
                for (int q = tid; q < nk * 64; q += MT_T)
                    fetch16(&S.rf[v * CL + (q >> 6)][(q & 63) * 4], &X.f[q >> 6][hi][lo][(q & 63) * 4]);
            }
            if (tid < nk * 4) fetch16(&S.rdz[tid >> 2][(tid & 3) * 4], &X.dz[tid >> 2][(tid & 3) * 4]);
            else if (tid >= 64 && tid - 64 < nk * 4)
                fetch16(&S.rls[(tid - 64) >> 2][(tid & 3) * 4], &X.ls[(tid - 64) >> 2][(tid & 3) * 4]);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            // ---- phase B: the owned gradients over the round's tiles
#pragma unroll
            for (int v = 0; v < VR; v++) {
                const int vr = rank * VR + v;
                if (w < 5) {
                    if (w == 4 && vr >= 8) continue;
                    const bf16(*A)[16 * MT_LD0] = w < 2 ? S.rd3 : w < 4 ? S.rd2 : S.rd1;
                    const int ao = ((lane & 7) + (lane >> 4) * 8) * MT_LD0 + ((lane >> 3) & 1) * 8;
                    const int br = (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll 4
                    for (int k = 0; k < nk; k++) {
                        uint32_t a[4], b[2];
                        ldm4t(a, A[v * CL + k] + ao);
                        ldm2t(b, w < 2   ? S.ra2[v * CL + k] + br * MT_LD0 + (w & 1) * 8
                                 : w < 4 ? S.ra1[v * CL + k] + br * MT_LD0 + (w & 1) * 8
                                         : S.ra0[v * CL + k] + br * 8);
                        mma16816(acc[v], a, b);
                    }
                } else if (w == 5) {
                    const bool prod = (vr >> 2) == 3;   // w4: dz h3; biases: dZ
                    const int c = lane & 15;
                    // the column's rows in order; two tiles' loads in turn, so
                    // that one is in flight while the other is added
                    float sum = acc[v][0];
                    auto chain = [&](auto product) {
                        float x[2][16];
                        auto load = [&](int k, float (&to)[16]) {
#pragma unroll
                            for (int r = 0; r < 16; r++) to[r] = S.rf[v * CL + k][r * 16 + c];
                            if constexpr (decltype(product)::value)
#pragma unroll
                                for (int r = 0; r < 16; r++) to[r] = __fmul_rn(S.rdz[k][r], to[r]);
                        };
                        auto add = [&](const float (&from)[16]) {
#pragma unroll
                            for (int r = 0; r < 16; r++) sum = __fadd_rn(sum, from[r]);
                        };
                        load(0, x[0]);
                        for (int k = 0; k < nk; k += 2) {
                            if (k + 1 < nk) load(k + 1, x[1]);
                            add(x[0]);
                            if (k + 2 < nk) load(k + 2, x[0]);
                            if (k + 1 < nk) add(x[1]);
                        }
                    };
                    if (prod) chain(std::true_type{});
                    else chain(std::false_type{});
                    acc[v][0] = sum;
                } else if (w == 6 && rank == 0 && v == 0) {
                    for (int r = lane; r < nk * 16; r += 32) {
                        acc[0][0] += S.rdz[r >> 4][r & 15];
                        lacc += S.rls[r >> 4][r & 15];
                    }
                }
            }
            if (j + 1 < rounds) cl.sync();   // the exchanged tiles are used up
        }
        if (w == 6 && rank == 0) {
            for (int o = 16; o > 0; o >>= 1) {
                acc[0][0] += __shfl_xor_sync(0xffffffffu, acc[0][0], o);
                lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
            }
            lrun += lacc;
            if (++lk == steps_per_epoch || s + 1 == nsteps) {
                if (loss && lane == 0) loss[TRAIN ? le : 0] = lrun;
                if (lk == steps_per_epoch) {
                    lk = 0;
                    le++;
                    lrun = 0.f;
                }
            }
        }
        const float c1 = corr.c1[s], c2 = corr.c2[s];
#pragma unroll
        for (int v = 0; v < VR; v++) {
            if (!has[v]) continue;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                if (w >= 5 && h) continue;
                if (!TRAIN) {
                    grad[og[v][h]] = acc[v][2 * h];
                    if (w < 5) grad[og[v][h] + 1] = acc[v][2 * h + 1];
                    continue;
                }
                const float *home = S.P + (w == 6 ? S_B4 : smem_place(og[v][h]));
                float *to = X.P + (w == 6 ? P_W4 + MH : og[v][h]);
                const float p0 = adam_step(home[0], acc[v][2 * h], om[v][2 * h], ov[v][2 * h], lr, c1, c2);
                if (w < 5)
                    *reinterpret_cast<float2 *>(to) =
                        make_float2(p0, adam_step(home[1], acc[v][2 * h + 1], om[v][2 * h + 1],
                                                  ov[v][2 * h + 1], lr, c1, c2));
                else
                    *to = p0;
            }
        }
        // the next step's first tile is put down while the blocks meet (the
        // local tile was read before the last barrier)
        cl.barrier_arrive();
        if (s + 1 < nsteps) put_input(rank < ntiles);
        cl.barrier_wait();
        if (TRAIN) {   // the new parameters
            for (int q = tid; q < (P_W4 + MH) / 4; q += MT_T)
                fetch16(S.P + smem_place(4 * q), X.P + 4 * q);
            if (tid == 0) S.P[S_B4] = __ldcg(X.P + P_W4 + MH);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
        }
    }
    if (TRAIN)
#pragma unroll
        for (int v = 0; v < VR; v++) {
            if (!has[v]) continue;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                if (w >= 5 && e) continue;
                const int i = og[v][e >> 1] + (e & 1);
                P[i] = S.P[(w == 6 ? S_B4 : smem_place(og[v][e >> 1])) + (e & 1)];
                am[i] = om[v][e];
                av[i] = ov[v][e];
            }
        }
}

// ------------------------------------------------------------ host side
static int64_t pad16(int64_t b) { return (b + 15) / 16 * 16; }

extern "C" size_t nb_mlp_workspace_size(int64_t batch)
{
    // inference and training do not run in one call: room for the larger
    const size_t infer = work_layout(pad16(batch), nullptr, nullptr);
    return (infer > sizeof(TrainShare) ? infer : sizeof(TrainShare)) + 256;
}

static MlpWork layout_at(void *ws, int64_t Bp)
{
    MlpWork w;
    char *base = (char *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    work_layout(Bp, &w, base);
    return w;
}

static int mlp_forward(const float *P, const float *x, int64_t B, float *theta, MlpWork w,
                       float fallback, cudaStream_t s)
{
    const int64_t Bp = pad16(B);
    k_mlp_input<<<nb_grid(Bp * MKIN, 256), 256, 0, s>>>(x, B, Bp, P, w.a0);
    const int64_t warps = Bp / 16;
    const int blocks = (int)((warps * 32 + MLP_T - 1) / MLP_T);
    k_mlp_fwd<<<blocks, MLP_T, 0, s>>>(P, Bp, w, theta, B, fallback);
    return cudaGetLastError() == cudaSuccess ? NB_OK : NB_ERR_CUDA;
}

// one launch of k_mlp_train: a cluster of 16 blocks where the device can run
// one (above the portable 8, so it is asked for), else 8
template <int CL, bool TRAIN>
static cudaError_t launch_train_cl(float *P, float *m, float *v, const float *feat,
                                   const float *labels, const int32_t *order, int64_t n,
                                   int64_t batch, int64_t spe, int64_t step0, int nsteps, float lr,
                                   TrainShare *share, float *grad, float *loss, cudaStream_t s,
                                   bool *runs)
{
    auto *kern = k_mlp_train<CL, TRAIN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TrainSmem));
    if (e != cudaSuccess) return e;
    if (CL > 8) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(MT_T);
    cfg.dynamicSmemBytes = sizeof(TrainSmem);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    *runs = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0;
    if (!*runs) {
        cudaGetLastError();
        return cudaSuccess;
    }
    AdamCorr corr;
    for (int k = 0; k < nsteps; k++) {
        const float tt = (float)(step0 + k + 1);
        corr.c1[k] = 1.0f - powf(0.9f, tt);
        corr.c2[k] = 1.0f - powf(0.999f, tt);
    }
    return cudaLaunchKernelEx(&cfg, kern, P, m, v, feat, labels, order, n, batch, spe, step0,
                              nsteps, lr, corr, share, grad, loss);
}

template <bool TRAIN>
static int launch_train(float *P, float *m, float *v, const float *feat, const float *labels,
                        const int32_t *order, int64_t n, int64_t batch, int64_t spe,
                        int64_t step0, int nsteps, float lr, void *work, float *grad, float *loss,
                        cudaStream_t s)
{
    TrainShare *share = (TrainShare *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
    bool runs = false;
    cudaError_t e = launch_train_cl<16, TRAIN>(P, m, v, feat, labels, order, n, batch, spe, step0,
                                               nsteps, lr, share, grad, loss, s, &runs);
    if (e == cudaSuccess && !runs)
        e = launch_train_cl<8, TRAIN>(P, m, v, feat, labels, order, n, batch, spe, step0, nsteps,
                                      lr, share, grad, loss, s, &runs);
    if (e != cudaSuccess || !runs) {
        cudaGetLastError();
        return NB_ERR_CUDA;
    }
    return NB_OK;
}

extern "C" int nb_mlp_forward(const float *params, const float *feat, int64_t n,
                              float *theta_out, float fallback, void *work, void *stream)
{
    if (!params || n < 0 || (n > 0 && (!feat || !theta_out || !work))) return NB_ERR_INVALID_ARG;
    if (n == 0) return NB_OK;
    MlpWork w = layout_at(work, pad16(n));
    return mlp_forward(params, feat, n, theta_out, w, fallback, (cudaStream_t)stream);
}

extern "C" int nb_mlp_grad(const float *params, const float *feat, const float *labels,
                           int64_t n, float *grad_out, float *loss_out, void *work,
                           void *stream)
{
    if (!params || n <= 0 || !feat || !labels || !grad_out || !work) return NB_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(grad_out, 0, sizeof(float) * P_N, s) != cudaSuccess) return NB_ERR_CUDA;
    if (loss_out && cudaMemsetAsync(loss_out, 0, sizeof(float), s) != cudaSuccess) return NB_ERR_CUDA;
    return launch_train<false>(const_cast<float *>(params), nullptr, nullptr, feat, labels, nullptr,
                               n, n, 1, 0, 1, 0.f, work, grad_out, loss_out, s);
}

extern "C" int nb_mlp_train(float *params, float *adam_m, float *adam_v, const float *feat,
                            const float *labels, int64_t n, const int32_t *order, int epochs,
                            int batch, float lr, float *grad_work, float *loss_per_epoch,
                            void *work, void *stream)
{
    if (!params || !adam_m || !adam_v || !feat || !labels || !order || n <= 0 || epochs < 1 ||
        batch < 16 || batch > n || !grad_work || !work)
        return NB_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t spe = n / batch, total = spe * epochs;
    if (loss_per_epoch && cudaMemsetAsync(loss_per_epoch, 0, sizeof(float) * epochs, s) != cudaSuccess)
        return NB_ERR_CUDA;
    for (int64_t k = 0; k < total; k += MT_STEPS) {
        const int steps = (int)(total - k < MT_STEPS ? total - k : MT_STEPS);
        const int rc = launch_train<true>(params, adam_m, adam_v, feat, labels, order, n, batch,
                                          spe, k, steps, lr, work, nullptr, loss_per_epoch, s);
        if (rc) return rc;
    }
    return NB_OK;
}
