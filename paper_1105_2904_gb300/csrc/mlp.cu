// Learned drag / torque closure: a small multilayer perceptron trained and evaluated on the
// GPU (the C-ABI lbm_mlp_* of include/lbmp.h). The paper has no network; this is an addition
// that corrects the force and torque a coarse-resolution particle feels.
//
// Precision: weights and activations in bfloat16, products accumulated in FP32 on the tensor
// cores (mma.sync m16n8k16 bf16 -> f32), FP32 master weights and Adam moments, FP32 loss.
// Each layer's output gradient is kept in bfloat16 (it is a tensor-core operand).
//
// Two forms. Networks whose weights stay below FUSED_WEIGHTS and whose activations of 16 rows fit
// in shared memory (the closure network by far) run fused: a minibatch is two launches,
//   k_rows        gather, every layer, the loss gradient and the backward pass through every layer,
//                 16 rows per block
//   k_update      weight and bias gradients, the loss, Adam
// Larger ones run layer by layer, where a layer fills the chip by itself and 16-row blocks would
// each stream all of the weights. Both forms add in the same order and give the same bits.
//
// Kernels of the second form:
//   k_gemm        C[M][N] = sum_k A(m,k) B(k,n) with arbitrary element strides for A and B
//                 (so X W^T, dY W and dY^T X are one kernel), fused epilogue: + bias, relu,
//                 relu' mask, bfloat16 and / or FP32 output; or FP32 split-K partials
//   k_sum_splits  fixed-order sum of split-K partials (weight gradients)
//   k_colsum      fixed-order column sums (bias gradients)
//   k_loss        mean-squared error, its output gradient (bfloat16) and per-block partial sums
//   k_gather      minibatch rows (by index) of the FP32 inputs as bfloat16, and their targets
//   k_adam        Adam on the FP32 masters, refreshing the bfloat16 copies
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "lbmp.h"

namespace {

constexpr int BM = 64, BN = 64, BK = 32, PADK = BK + 8;
constexpr int GEMM_THREADS = 128;

struct GemmArgs {
    int M, N, K;
    const __nv_bfloat16* A;
    long long sam, sak;  // A(m,k) = A[m*sam + k*sak]
    const __nv_bfloat16* B;
    long long sbk, sbn;  // B(k,n) = B[k*sbk + n*sbn]
    const float* bias;   // [N] or null
    int relu;            // 1: max(v, 0)
    const __nv_bfloat16* mask;  // relu' mask: v *= (mask(m,n) > 0), mask(m,n) = mask[m*ldo + n]
    __nv_bfloat16* out16;       // C as bfloat16, out16[m*ldo + n] (or null)
    float* out32;               // C as FP32 (or null)
    long long ldo;
    int ksplit;                 // > 1: blockIdx.z takes K range z; out32 = partials [ksplit][M][N]
};

__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// One 64 x 64 output tile per block, four warps of 32 x 32; K in steps of 32 staged in shared
// memory as As[m][k] and Bs[n][k] (zero outside the matrices).
__global__ void __launch_bounds__(GEMM_THREADS) k_gemm(const GemmArgs g)
{
    __shared__ __align__(16) __nv_bfloat16 As[BM][PADK];
    __shared__ __align__(16) __nv_bfloat16 Bs[BN][PADK];
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int gq = lane >> 2, tq = lane & 3;
    int k_begin = 0, k_end = g.K;
    if (g.ksplit > 1) {
        const int per = ((g.K + g.ksplit - 1) / g.ksplit + BK - 1) / BK * BK;
        k_begin = blockIdx.z * per;
        k_end = min(g.K, k_begin + per);
    }
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    const __nv_bfloat16 zero = __float2bfloat16(0.f);
    for (int k0 = k_begin; k0 < k_end; k0 += BK) {
        for (int e = threadIdx.x; e < BM * BK; e += GEMM_THREADS) {
            const int r = e / BK, c = e % BK;
            const int m = m0 + r, k = k0 + c, n = n0 + r;
            As[r][c] = (m < g.M && k < k_end) ? g.A[(long long)m * g.sam + (long long)k * g.sak] : zero;
            Bs[r][c] = (n < g.N && k < k_end) ? g.B[(long long)k * g.sbk + (long long)n * g.sbn] : zero;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t a[2][4], b[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm + i * 16 + gq;
                a[i][0] = ld_pair(&As[r][kk + 2 * tq]);
                a[i][1] = ld_pair(&As[r + 8][kk + 2 * tq]);
                a[i][2] = ld_pair(&As[r][kk + 2 * tq + 8]);
                a[i][3] = ld_pair(&As[r + 8][kk + 2 * tq + 8]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = wn + j * 8 + gq;
                b[j][0] = ld_pair(&Bs[n][kk + 2 * tq]);
                b[j][1] = ld_pair(&Bs[n][kk + 2 * tq + 8]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
        }
        __syncthreads();
    }
    // epilogue: c0, c1 at (row gq, cols 2tq, 2tq+1); c2, c3 at row gq + 8
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int m = m0 + wm + i * 16 + gq + (q >= 2 ? 8 : 0);
                const int n = n0 + wn + j * 8 + 2 * tq + (q & 1);
                if (m >= g.M || n >= g.N) continue;
                float v = acc[i][j][q];
                if (g.ksplit > 1) {
                    g.out32[((long long)blockIdx.z * g.M + m) * g.N + n] = v;
                    continue;
                }
                if (g.bias) v += g.bias[n];
                if (g.relu) v = fmaxf(v, 0.f);
                if (g.mask && !(__bfloat162float(g.mask[(long long)m * g.ldo + n]) > 0.f)) v = 0.f;
                if (g.out16) g.out16[(long long)m * g.ldo + n] = __float2bfloat16(v);
                if (g.out32) g.out32[(long long)m * g.ldo + n] = v;
            }
}

// out[i] = sum over s of part[s][i], s in order.
__global__ void k_sum_splits(const float* __restrict__ part, int splits, long long n, float* __restrict__ out)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int z = 0; z < splits; ++z) s += part[(long long)z * n + i];
        out[i] = s;
    }
}

// out[n] = sum over rows m of d[m][n] (bfloat16 values, FP32 sum): one block per column,
// a fixed-order tree over the block.
__global__ void k_colsum(const __nv_bfloat16* __restrict__ d, int M, int N, float* __restrict__ out)
{
    __shared__ float part[256];
    const int n = blockIdx.x;
    float s = 0.f;
    for (int m = threadIdx.x; m < M; m += blockDim.x) s += __bfloat162float(d[(long long)m * N + n]);
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) part[threadIdx.x] += part[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = part[0];
}

// Mean-squared error over the B x O outputs: d = 2 (y - t) / (B O) as bfloat16, and one FP32
// partial sum of (y - t)^2 per block (block b covers entries b*256 .. b*256 + 255).
__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ t, long long n, float scale,
                       __nv_bfloat16* __restrict__ d, float* __restrict__ partial)
{
    __shared__ float part[256];
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    float r2 = 0.f;
    if (i < n) {
        const float r = y[i] - t[i];
        d[i] = __float2bfloat16(2.f * r * scale);
        r2 = r * r;
    }
    part[threadIdx.x] = r2;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) part[threadIdx.x] += part[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = part[0];
}

// loss_out[slot] = scale * sum of the partials, in order (one thread).
__global__ void k_loss_total(const float* __restrict__ partial, int nparts, double scale, double* loss_out, int slot)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int i = 0; i < nparts; ++i) s += (double)partial[i];
    loss_out[slot] += s * scale;
}

// Rows idx[r] of X (FP32, [n][K]) as bfloat16 rows r of Xb, each input standardised as
// (x - shift[c]) * scale[c] when shift / scale are given, and of T ([n][O]) as rows of Tb.
__global__ void k_gather(const float* __restrict__ X, const float* __restrict__ T, const int* __restrict__ idx,
                         int rows, int K, int O, const float* __restrict__ shift, const float* __restrict__ scale,
                         __nv_bfloat16* __restrict__ Xb, float* __restrict__ Tb)
{
    const long long nx = (long long)rows * K, total = nx + (long long)rows * O;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        if (e < nx) {
            const long long r = e / K, c = e % K;
            const long long src = idx ? idx[r] : r;
            float v = X[src * K + c];
            if (shift) v = (v - shift[c]) * scale[c];
            Xb[e] = __float2bfloat16(v);
        } else if (T) {
            const long long f = e - nx, r = f / O, c = f % O;
            const long long src = idx ? idx[r] : r;
            Tb[f] = T[src * O + c];
        }
    }
}

// One Adam step (Kingma & Ba, 2015) of parameter p with moments m, v and gradient g; c1, c2 the
// bias corrections.
__device__ __forceinline__ void adam_step(float& p, float& m, float& v, float g, float lr, float b1, float b2, float eps,
                                          float c1, float c2)
{
    m = fmaf(1.f - b1, g, b1 * m);  // (explicit, so that every kernel rounds alike)
    v = fmaf((1.f - b2) * g, g, b2 * v);
    p = p - lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// Adam on FP32 masters p with moments m, v; t_dev holds the number of
// steps taken so far (this is step t_dev + 1; k_adam_tick advances it afterwards).
__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, const float* __restrict__ g,
                       long long n, const int* __restrict__ t_dev, float lr, float b1, float b2, float eps,
                       __nv_bfloat16* __restrict__ p16)
{
    const int t = *t_dev + 1;
    const float c1 = 1.f - powf(b1, (float)t);
    const float c2 = 1.f - powf(b2, (float)t);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float pi = p[i], mi = m[i], vi = v[i];
        adam_step(pi, mi, vi, g[i], lr, b1, b2, eps, c1, c2);
        p[i] = pi;
        m[i] = mi;
        v[i] = vi;
        if (p16) p16[i] = __float2bfloat16(pi);
    }
}

// ---- fused form ------------------------------------------------------------------------------
// A training step of the closure network (259-128-128-6, 128 rows) is 38 MFLOP on 700 kB that sit
// in L2: nothing bounds it but latency, so what counts is the number of dependent launches and
// round trips. Rows are independent through all layers forwards and backwards; only the weight
// gradients need all rows. That gives two kernels. Weights are kept as bfloat16 in the order of
// the tensor-core fragments (forward B(k, n) = W[n][k]; backward B(k = j, n = c) = W[j][c]), so a
// lane's operand is one 8-byte load and a warp's 256 consecutive bytes, whatever the width of the
// layer (the closure's 259 inputs leave W's rows unaligned); Adam writes its new weights there.
// Epoch of 24 minibatches of 128 rows, with the parameters read back: 4963 -> 527 us (a minibatch was
// ~20 launches); forward pass of 200 rows 113 -> 14 us.

constexpr int MAX_LAYERS = 8;
constexpr int ROWS = 16;             // rows per block: one m16n8k16 tile
constexpr int ROWS_THREADS = 256;
constexpr int UPD_THREADS = 128;
constexpr int KCHUNK = 9;            // k-steps of weights a warp loads at once (the closure's 17 in two)
constexpr int RCHUNK = 8;            // k-steps of rows a warp of k_update loads at once (128 rows)
constexpr int SPLITS = 16;           // fixed-order split of the rows in the weight gradients
constexpr int LOSS_TILES = 4;        // sums of 256 squared errors per warp of k_update
// Up to here a 16-row block's pass over all weights (512 kB from L2) stays a matter of a few us, and the
// fused form is the faster one at every number of rows: gradients through 256-512-256, 262144 weights,
// fused and layer by layer, 128 rows 68 and 261 us, 1024 156 and 369, 16384 1771 and 2504, 65536 6960
// and 9550; through 64-256-256-64 45 and 257, 67 and 291, 503 and 1216, 1932 and 4208.
constexpr long long FUSED_WEIGHTS = 262144;
constexpr size_t FUSED_SMEM = 160 * 1024;

__host__ __device__ constexpr int pad16(int n) { return (n + 15) / 16 * 16; }
// Row stride of a bfloat16 tile in shared memory, an odd multiple of four words: the eight rows of a
// fragment fall into different banks.
__host__ __device__ constexpr int tile_ld(int n) { return pad16(n) + 8; }
__host__ __device__ constexpr long long frag_elems(int k, int n) { return (long long)((n + 7) / 8) * ((k + 15) / 16) * 128; }
// Position of B(k, n) among the fragments of a K x N operand (m16n8k16, "col" B).
__device__ __forceinline__ long long frag_pos(int k, int n, int K)
{
    const int ks = (K + 15) / 16;
    const int lane = (n & 7) * 4 + ((k & 7) >> 1);
    return (((long long)(n >> 3) * ks + (k >> 4)) * 32 + lane) * 4 + ((k >> 3) & 1) * 2 + (k & 1);
}

struct NetArgs {
    int L;
    int size[MAX_LAYERS + 1];
    long long w_off[MAX_LAYERS], b_off[MAX_LAYERS];
    long long wf_off[MAX_LAYERS], wb_off[MAX_LAYERS];  // fragment-ordered copies (backward: l >= 1)
    const float* p;
    __nv_bfloat16* wf;
    __nv_bfloat16* wb;
    const float *shift, *scale;  // input standardisation or null
    // between the two kernels: values by feature, ld rows each (the update's operands)
    int ld;
    __nv_bfloat16* hT[MAX_LAYERS];  // inputs of layer l
    __nv_bfloat16* dT[MAX_LAYERS];  // output gradients of layer l
    float* r2;                   // squared errors [rows][O]
};

struct RowsArgs {
    NetArgs n;
    const float* X;      // [.][K]
    const float* T;      // [.][O], null: forward pass only
    const int* idx;      // rows of the minibatch, null: 0..rows-1
    int rows;
    float* y;            // forward pass: [rows][O]
    float grad_scale;    // 1 / (rows O)
    int* tick;           // Adam's step count, advanced here when given (k_update reads it)
};

struct UpdateArgs {
    NetArgs n;
    int rows;
    float* p;
    float* m;
    float* v;
    float* g;
    const int* t;        // Adam's step number, null: gradients only
    float lr, b1, b2, eps;
    double* loss;        // loss of the minibatch is added here
    double loss_scale;
    float* loss_part;    // sums of the squared errors of 256 outputs each (more than LOSS_TILES of them)
    int* loss_done;      // loss warps that are through, zero between launches
};

// C (16 rows of `in` times a K x N operand in fragment order, plus the bias if given) for this
// warp's n-tiles, two at a time; put(row, column, value) for the lane's elements.
template <class PUT>
__device__ __forceinline__ void rows_gemm(const __nv_bfloat16* __restrict__ in, int ld, int K, int N,
                                          const __nv_bfloat16* __restrict__ frag, const float* __restrict__ bias, PUT&& put)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gq = lane >> 2, tq = lane & 3;
    const int KS = (K + 15) / 16, NT = (N + 7) / 8;
    for (int nt = 2 * warp; nt < NT; nt += 2 * (ROWS_THREADS / 32)) {
        const bool two = nt + 1 < NT;
        const uint2* b0p = reinterpret_cast<const uint2*>(frag) + (long long)nt * KS * 32 + lane;
        const uint2* b1p = two ? b0p + (long long)KS * 32 : b0p;
        float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f}, bs[2][2] = {};
        if (bias) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int col = nt * 8 + 8 * (q >> 1) + 2 * tq + (q & 1);
                if (col < N) bs[q >> 1][q & 1] = bias[col];
            }
        }
        for (int k0 = 0; k0 < KS; k0 += KCHUNK) {
            // the chunk's operands first, all in flight together
            uint2 v0[KCHUNK], v1[KCHUNK];
#pragma unroll
            for (int j = 0; j < KCHUNK; ++j) {
                const bool in_k = k0 + j < KS;
                v0[j] = in_k ? b0p[(k0 + j) * 32] : make_uint2(0u, 0u);
                v1[j] = in_k ? b1p[(k0 + j) * 32] : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int j = 0; j < KCHUNK; ++j) {
                if (k0 + j >= KS) break;
                const __nv_bfloat16* ap = in + gq * ld + (k0 + j) * 16 + 2 * tq;
                const uint32_t a[4] = {ld_pair(ap), ld_pair(ap + 8 * ld), ld_pair(ap + 8), ld_pair(ap + 8 * ld + 8)};
                const uint32_t b0[2] = {v0[j].x, v0[j].y}, b1[2] = {v1[j].x, v1[j].y};
                mma_bf16(c0, a, b0);
                mma_bf16(c1, a, b1);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = gq + (q >= 2 ? 8 : 0), col = nt * 8 + 2 * tq + (q & 1);
            if (col < N) put(row, col, bias ? c0[q] + bs[0][q & 1] : c0[q]);
            if (two && col + 8 < N) put(row, col + 8, bias ? c1[q] + bs[1][q & 1] : c1[q]);
        }
    }
}

__device__ __forceinline__ void wait_for_previous_kernel()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void let_next_kernel_start()
{
    asm volatile("griddepcontrol.launch_dependents;");
}

__global__ void __launch_bounds__(ROWS_THREADS) k_rows(const RowsArgs a)
{
    extern __shared__ __align__(16) __nv_bfloat16 sm[];
    const NetArgs& n = a.n;
    const int L = n.L, K0 = n.size[0], O = n.size[L];
    const int row0 = blockIdx.x * ROWS;
    const bool train = a.T != nullptr;
    __nv_bfloat16* h[MAX_LAYERS + 1];  // inputs of layer l ([ROWS][tile_ld]); h[L] stays unused
    __nv_bfloat16* d[MAX_LAYERS + 1];  // output gradients of layer l - 1, beside h
    int total = 0;
    for (int l = 0; l < L; ++l) {
        h[l] = sm + total;
        total += ROWS * tile_ld(n.size[l]);
    }
    if (train)
        for (int l = 1; l <= L; ++l) {
            d[l] = sm + total;
            total += ROWS * tile_ld(n.size[l]);
        }
    float* tgt = reinterpret_cast<float*>(sm + total);  // targets [ROWS][O]
    // padding rows and columns are zero
    for (int e = threadIdx.x; e < total / 8; e += ROWS_THREADS) reinterpret_cast<uint4*>(sm)[e] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    // the minibatch's rows; nothing here depends on the kernel before
    // (a warp takes two rows, eight columns of each lane in flight)
    for (int r = threadIdx.x >> 5; r < ROWS && row0 + r < a.rows; r += ROWS_THREADS / 32) {
        const long long src = a.idx ? a.idx[row0 + r] : row0 + r;
        const float* x = a.X + src * K0;
        if (train)
            for (int c = threadIdx.x & 31; c < O; c += 32) tgt[r * O + c] = a.T[src * O + c];
        for (int c0 = threadIdx.x & 31; c0 < K0; c0 += 8 * 32) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = c0 + 32 * j < K0 ? x[c0 + 32 * j] : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = c0 + 32 * j;
                if (c >= K0) continue;
                if (n.shift) v[j] = (v[j] - n.shift[c]) * n.scale[c];
                h[0][r * tile_ld(K0) + c] = __float2bfloat16(v[j]);
            }
        }
    }
    wait_for_previous_kernel();
    let_next_kernel_start();
    if (a.tick && blockIdx.x == 0 && threadIdx.x == 0) *a.tick += 1;
    __syncthreads();
    for (int l = 0; l < L; ++l) {
        const int K = n.size[l], N = n.size[l + 1];
        const float* bias = n.p + n.b_off[l];
        if (l + 1 < L) {
            __nv_bfloat16* out = h[l + 1];
            const int ldo = tile_ld(N);
            rows_gemm(h[l], tile_ld(K), K, N, n.wf + n.wf_off[l], bias,
                      [&](int r, int c, float v) {
                          // (rows beyond the last stay zero: k_update multiplies them by zero gradients, and
                          // relu(bias ...) of a zero input can be infinite where no real row's is)
                          out[r * ldo + c] = __float2bfloat16(row0 + r < a.rows ? fmaxf(v, 0.f) : 0.f);
                      });
        } else {
            rows_gemm(h[l], tile_ld(K), K, N, n.wf + n.wf_off[l], bias, [&](int r, int c, float y) {
                if (row0 + r >= a.rows) return;
                if (!train) {
                    a.y[(long long)(row0 + r) * O + c] = y;
                    return;
                }
                // mean-squared error: d = 2 (y - t) / (rows O)
                const float res = y - tgt[r * O + c];
                n.r2[(long long)(row0 + r) * O + c] = res * res;
                d[L][r * tile_ld(O) + c] = __float2bfloat16(2.f * res * a.grad_scale);
            });
        }
        __syncthreads();
    }
    if (!train) return;
    // d_l = (d_{l+1} W_l) relu'(h_l)
    for (int l = L - 1; l >= 1; --l) {
        const int K = n.size[l], N = n.size[l + 1], ldk = tile_ld(K);
        rows_gemm(d[l + 1], tile_ld(N), N, K, n.wb + n.wb_off[l], nullptr, [&](int r, int c, float v) {
            const bool on = __bfloat162float(h[l][r * ldk + c]) > 0.f;
            d[l][r * ldk + c] = __float2bfloat16(on ? v : 0.f);
        });
        __syncthreads();
    }
    // by feature, this block's 16 rows as two 16-byte stores
    auto transpose = [&](const __nv_bfloat16* from, int N, __nv_bfloat16* to) {
        const int ld = tile_ld(N);
        for (int c = threadIdx.x; c < N; c += ROWS_THREADS) {
            __align__(16) __nv_bfloat16 col[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) col[r] = from[r * ld + c];
            uint4* dst = reinterpret_cast<uint4*>(to + (long long)c * n.ld + row0);
            dst[0] = reinterpret_cast<const uint4*>(col)[0];
            dst[1] = reinterpret_cast<const uint4*>(col)[1];
        }
    };
    for (int l = 0; l < L; ++l) {
        transpose(h[l], n.size[l], n.hT[l]);
        transpose(d[l + 1], n.size[l + 1], n.dT[l]);
    }
}

// Sum of 256 values in the order of a halving tree (value t + value t + 128, then + 64, ...): lane t
// holds values t + 32 j.
__device__ __forceinline__ float tree256(float x[8])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] += x[j + 4];
    x[0] += x[2];
    x[1] += x[3];
    float s = x[0] + x[1];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    return s;  // lane 0
}

// One warp per 16 x 8 tile of a weight gradient dW[n][k] = sum_r d[r][n] h[r][k] (rows in SPLITS
// ranges, each summed on the tensor cores, the ranges added in order), per bias gradient and for the loss; Adam
// on the elements just formed.
__global__ void __launch_bounds__(UPD_THREADS) k_update(const UpdateArgs a)
{
    const NetArgs& n = a.n;
    const int lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
    int task = blockIdx.x * (UPD_THREADS / 32) + (threadIdx.x >> 5);
    wait_for_previous_kernel();
    let_next_kernel_start();
    float c1 = 1.f, c2 = 1.f;
    if (a.t) {
        const int t = *a.t;
        c1 = 1.f - powf(a.b1, (float)t);
        c2 = 1.f - powf(a.b2, (float)t);
    }
    const int per = ((a.rows + SPLITS - 1) / SPLITS + 31) / 32 * 32;  // rows of a range
    const int rows16 = (a.rows + 15) / 16 * 16;
    for (int l = 0; l < n.L; ++l) {
        const int K = n.size[l], N = n.size[l + 1];
        const int MT = (N + 15) / 16, NT = (K + 7) / 8;
        if (task >= MT * NT) {
            task -= MT * NT;
            continue;
        }
        const int n0 = task / NT * 16, k0 = task % NT * 8;
        const __nv_bfloat16* d0 = n.dT[l] + (long long)(n0 + gq) * n.ld + 2 * tq;
        const __nv_bfloat16* d1 = d0 + 8LL * n.ld;
        const __nv_bfloat16* hb = n.hT[l] + (long long)(k0 + gq) * n.ld + 2 * tq;
        const bool ok0 = n0 + gq < N, ok1 = n0 + gq + 8 < N, okb = k0 + gq < K;
        // this lane's parameters, loaded beside the operands
        long long at[4];
        float pv[4], mv[4], vv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int nn = n0 + gq + (q >= 2 ? 8 : 0), k = k0 + 2 * tq + (q & 1);
            at[q] = nn < N && k < K ? n.w_off[l] + (long long)nn * K + k : -1;
            if (a.t && at[q] >= 0) {
                pv[q] = a.p[at[q]];
                mv[q] = a.m[at[q]];
                vv[q] = a.v[at[q]];
            }
        }
        float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
        int next = per;  // first row of the next range
        for (int r0 = 0; r0 < rows16; r0 += 16 * RCHUNK) {
            uint32_t A[RCHUNK][4], B[RCHUNK][2];
#pragma unroll
            for (int j = 0; j < RCHUNK; ++j) {
                const int r = r0 + 16 * j;
                const bool in = r < rows16;
                A[j][0] = in && ok0 ? ld_pair(d0 + r) : 0u;
                A[j][1] = in && ok1 ? ld_pair(d1 + r) : 0u;
                A[j][2] = in && ok0 ? ld_pair(d0 + r + 8) : 0u;
                A[j][3] = in && ok1 ? ld_pair(d1 + r + 8) : 0u;
                B[j][0] = in && okb ? ld_pair(hb + r) : 0u;
                B[j][1] = in && okb ? ld_pair(hb + r + 8) : 0u;
            }
#pragma unroll
            for (int j = 0; j < RCHUNK; ++j) {
                const int r = r0 + 16 * j;
                if (r >= rows16) break;
                if (r == next) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        s[q] += c[q];
                        c[q] = 0.f;
                    }
                    next += per;
                }
                mma_bf16(c, A[j], B[j]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (at[q] < 0) continue;
            s[q] += c[q];
            a.g[at[q]] = s[q];
            if (!a.t) continue;
            adam_step(pv[q], mv[q], vv[q], s[q], a.lr, a.b1, a.b2, a.eps, c1, c2);
            a.p[at[q]] = pv[q];
            a.m[at[q]] = mv[q];
            a.v[at[q]] = vv[q];
            const __nv_bfloat16 w = __float2bfloat16(pv[q]);
            const int nn = n0 + gq + (q >= 2 ? 8 : 0), k = k0 + 2 * tq + (q & 1);
            n.wf[n.wf_off[l] + frag_pos(k, nn, K)] = w;
            if (l > 0) n.wb[n.wb_off[l] + frag_pos(nn, k, N)] = w;
        }
        return;
    }
    for (int l = 0; l < n.L; ++l) {
        const int N = n.size[l + 1];
        if (task >= N) {
            task -= N;
            continue;
        }
        const __nv_bfloat16* dr = n.dT[l] + (long long)task * n.ld;
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = lane + 32 * j < a.rows ? __bfloat162float(dr[lane + 32 * j]) : 0.f;
        for (int r0 = 256; r0 < a.rows; r0 += 256)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (r0 + lane + 32 * j < a.rows) x[j] += __bfloat162float(dr[r0 + lane + 32 * j]);
        const float s = tree256(x);
        if (lane == 0) {
            const long long i = n.b_off[l] + task;
            a.g[i] = s;
            if (a.t) adam_step(a.p[i], a.m[i], a.v[i], s, a.lr, a.b1, a.b2, a.eps, c1, c2);
        }
        return;
    }
    // The loss: sums of 256 squared errors, LOSS_TILES of them to a warp, added in order by the warp
    // that is through last (by the only one where there is one). One warp for all of them took 0.8 us
    // for each sum: gradients of 16384 rows through 64-256-256-64 2.12 -> 0.50 ms (layer by layer 1.22 ms).
    const long long m = (long long)a.rows * n.size[n.L];
    const int tiles = (int)((m + 255) / 256), warps = (tiles + LOSS_TILES - 1) / LOSS_TILES;
    if (task >= warps) return;
    float s[LOSS_TILES];
#pragma unroll
    for (int k = 0; k < LOSS_TILES; ++k) {
        const long long b = ((long long)task * LOSS_TILES + k) * 256 + lane;
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = b + 32 * j < m ? n.r2[b + 32 * j] : 0.f;
        s[k] = tree256(x);
    }
    double tot = 0.0;
    if (warps == 1) {
#pragma unroll
        for (int k = 0; k < LOSS_TILES; ++k)
            if (k < tiles) tot += (double)s[k];
        if (lane == 0) *a.loss += tot * a.loss_scale;
        return;
    }
    int last = 0;
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < LOSS_TILES; ++k)
            if (task * LOSS_TILES + k < tiles) a.loss_part[task * LOSS_TILES + k] = s[k];
        __threadfence();
        last = atomicAdd(a.loss_done, 1) == warps - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    float next = lane < tiles ? __ldcg(&a.loss_part[lane]) : 0.f;
    for (int b = 0; b < tiles; b += 32) {
        const float v = next;
        next = b + 32 + lane < tiles ? __ldcg(&a.loss_part[b + 32 + lane]) : 0.f;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const float t = __shfl_sync(0xffffffffu, v, k);
            if (b + k < tiles) tot += (double)t;
        }
    }
    if (lane == 0) {
        *a.loss += tot * a.loss_scale;
        *a.loss_done = 0;
    }
}

// The fragment-ordered copies of the weights (after they were set, or after a separate Adam step).
__global__ void k_pack_weights(const NetArgs n)
{
    for (int l = 0; l < n.L; ++l) {
        const int K = n.size[l], N = n.size[l + 1];
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < N * K; e += gridDim.x * blockDim.x) {
            const int j = e / K, k = e - j * K;
            const __nv_bfloat16 w = __float2bfloat16(n.p[n.w_off[l] + e]);
            n.wf[n.wf_off[l] + frag_pos(k, j, K)] = w;
            if (l > 0) n.wb[n.wb_off[l] + frag_pos(j, k, N)] = w;
        }
    }
}

__global__ void k_adam_tick(int* t_dev)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *t_dev += 1;
}

__global__ void k_to_bf16(const float* __restrict__ a, long long n, __nv_bfloat16* __restrict__ b)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16(a[i]);
}

int blocks_for(long long n, int t = 256) { return (int)std::max<long long>(1, std::min<long long>(4096, (n + t - 1) / t)); }

}  // namespace

struct lbm_mlp {
    int L = 0;
    std::vector<int> sizes;
    cudaStream_t stream = nullptr;
    // parameters, layer-major: W[l] (sizes[l+1] x sizes[l], row-major) then b[l]
    std::vector<long long> w_off, b_off;
    long long nparam = 0;
    float* p = nullptr;   // FP32 masters
    float* m = nullptr;
    float* v = nullptr;
    float* g = nullptr;   // gradients
    __nv_bfloat16* p16 = nullptr;  // bfloat16 copies (W entries used; b entries unused)
    int* t = nullptr;
    // workspace for up to `cap` rows
    int cap = 0;
    __nv_bfloat16* xb = nullptr;
    float* tb = nullptr;
    std::vector<__nv_bfloat16*> h;   // activations of hidden layers
    std::vector<__nv_bfloat16*> d;   // output gradients of every layer
    float* y = nullptr;
    float* partial = nullptr;        // split-K partials and loss partial sums
    size_t partial_floats = 0;
    int* idx = nullptr;
    int idx_cap = 0;
    double* loss_dev = nullptr;
    int loss_cap = 0;
    float* in_shift = nullptr;       // input standardisation (null: none)
    float* in_scale = nullptr;
    // fused form (k_rows, k_update)
    bool fused = false;
    std::vector<long long> wf_off, wb_off;
    __nv_bfloat16* wf = nullptr;     // weights in fragment order, forwards
    __nv_bfloat16* wb = nullptr;     // and backwards
    std::vector<__nv_bfloat16*> hT, dT;
    float* r2 = nullptr;
    float* loss_part = nullptr;
    int* loss_done = nullptr;
    std::vector<void*> allocs;
    std::string err;
};

namespace {

lbm_status mfail(lbm_mlp* n, lbm_status s, const std::string& msg)
{
    if (n) n->err = msg;
    return s;
}

#define MK(call)                                                                                              \
    do {                                                                                                      \
        cudaError_t e_ = (call);                                                                              \
        if (e_ != cudaSuccess) return mfail(net, LBM_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

template <typename T>
lbm_status malloc_dev(lbm_mlp* net, T** p, size_t count)
{
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(16, count * sizeof(T)));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return mfail(net, LBM_E_OOM, "cudaMalloc failed");
    }
    net->allocs.push_back(q);
    *p = (T*)q;
    return LBM_OK;
}

void free_dev(lbm_mlp* net, void* p)
{
    if (!p) return;
    auto it = std::find(net->allocs.begin(), net->allocs.end(), p);
    if (it != net->allocs.end()) net->allocs.erase(it);
    cudaFree(p);
}

lbm_status ensure_rows(lbm_mlp* net, int rows)
{
    if (rows <= net->cap) return LBM_OK;
    int cap = 1;
    while (cap < rows) cap <<= 1;
    free_dev(net, net->xb);
    free_dev(net, net->tb);
    free_dev(net, net->y);
    free_dev(net, net->partial);
    for (auto* q : net->h) free_dev(net, q);
    for (auto* q : net->d) free_dev(net, q);
    net->h.assign(net->L - 1, nullptr);
    net->d.assign(net->L, nullptr);
    const int K = net->sizes[0], O = net->sizes[net->L];
    lbm_status s;
    if (net->fused) {
        cap = std::max(cap, ROWS);
        for (auto* q : net->hT) free_dev(net, q);
        for (auto* q : net->dT) free_dev(net, q);
        free_dev(net, net->r2);
        free_dev(net, net->loss_part);
        net->cap = 0;
        net->r2 = net->loss_part = nullptr;
        net->hT.assign(net->L, nullptr);
        net->dT.assign(net->L, nullptr);
        for (size_t l = 0; l < (size_t)net->L; ++l) {
            if ((s = malloc_dev(net, &net->hT[l], (size_t)cap * net->sizes[l])) != LBM_OK) return s;
            if ((s = malloc_dev(net, &net->dT[l], (size_t)cap * net->sizes[l + 1])) != LBM_OK) return s;
        }
        if ((s = malloc_dev(net, &net->r2, (size_t)cap * O)) != LBM_OK) return s;
        if ((s = malloc_dev(net, &net->loss_part, ((size_t)cap * O + 255) / 256)) != LBM_OK) return s;
        net->cap = cap;
        return LBM_OK;
    }
    if ((s = malloc_dev(net, &net->xb, (size_t)cap * K)) != LBM_OK) return s;
    if ((s = malloc_dev(net, &net->tb, (size_t)cap * O)) != LBM_OK) return s;
    if ((s = malloc_dev(net, &net->y, (size_t)cap * O)) != LBM_OK) return s;
    for (int l = 0; l + 1 < net->L; ++l)
        if ((s = malloc_dev(net, &net->h[(size_t)l], (size_t)cap * net->sizes[(size_t)l + 1])) != LBM_OK) return s;
    for (int l = 0; l < net->L; ++l)
        if ((s = malloc_dev(net, &net->d[(size_t)l], (size_t)cap * net->sizes[(size_t)l + 1])) != LBM_OK) return s;
    size_t pf = (size_t)(cap * (long long)O + 255) / 256 + 16;
    for (int l = 0; l < net->L; ++l)
        pf = std::max(pf, (size_t)SPLITS * net->sizes[(size_t)l] * net->sizes[(size_t)l + 1]);
    if ((s = malloc_dev(net, &net->partial, pf)) != LBM_OK) return s;
    net->partial_floats = pf;
    net->cap = cap;
    return LBM_OK;
}

void gemm(cudaStream_t s, int M, int N, int K, const __nv_bfloat16* A, long long sam, long long sak,
          const __nv_bfloat16* B, long long sbk, long long sbn, const float* bias, int relu,
          const __nv_bfloat16* mask, __nv_bfloat16* out16, float* out32, long long ldo, int ksplit = 1)
{
    GemmArgs g{M, N, K, A, sam, sak, B, sbk, sbn, bias, relu, mask, out16, out32, ldo, ksplit};
    const dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, ksplit);
    k_gemm<<<grid, GEMM_THREADS, 0, s>>>(g);
}

// Forward pass of `rows` rows already in net->xb; output in net->y (FP32).
void forward(lbm_mlp* net, int rows)
{
    const __nv_bfloat16* in = net->xb;
    for (int l = 0; l < net->L; ++l) {
        const int K = net->sizes[(size_t)l], N = net->sizes[(size_t)l + 1];
        const __nv_bfloat16* W = net->p16 + net->w_off[(size_t)l];
        const float* b = net->p + net->b_off[(size_t)l];
        const bool last = l == net->L - 1;
        gemm(net->stream, rows, N, K, in, K, 1, W, 1, K, b, last ? 0 : 1, nullptr, last ? nullptr : net->h[(size_t)l],
             last ? net->y : nullptr, N);
        if (!last) in = net->h[(size_t)l];
    }
}

// Loss and gradients of `rows` rows in net->xb / net->tb (forward included). The loss is
// added to net->loss_dev[slot] (FP64).
void backward(lbm_mlp* net, int rows, int slot)
{
    const int O = net->sizes[(size_t)net->L];
    const long long n = (long long)rows * O;
    const int lb = (int)((n + 255) / 256);
    forward(net, rows);
    k_loss<<<lb, 256, 0, net->stream>>>(net->y, net->tb, n, 1.f / (float)n, net->d[(size_t)net->L - 1], net->partial);
    k_loss_total<<<1, 32, 0, net->stream>>>(net->partial, lb, 1.0 / (double)n, net->loss_dev, slot);
    for (int l = net->L - 1; l >= 0; --l) {
        const int K = net->sizes[(size_t)l], N = net->sizes[(size_t)l + 1];
        const __nv_bfloat16* din = net->d[(size_t)l];
        const __nv_bfloat16* hin = l == 0 ? net->xb : net->h[(size_t)l - 1];
        // dW[N][K] = d^T h: A(m=j, k=r) = d[r][j], B(k=r, n=c) = h[r][c]; split over the rows
        gemm(net->stream, N, K, rows, din, 1, N, hin, K, 1, nullptr, 0, nullptr, nullptr, net->partial, K, SPLITS);
        k_sum_splits<<<blocks_for((long long)N * K), 256, 0, net->stream>>>(net->partial, SPLITS, (long long)N * K,
                                                                           net->g + net->w_off[(size_t)l]);
        k_colsum<<<N, 256, 0, net->stream>>>(din, rows, N, net->g + net->b_off[(size_t)l]);
        if (l > 0) {
            // d_{l-1} = (d_l W_l) * relu'(h_{l-1}): A = d (rows x N), B(k=j, n=c) = W[j][c]
            const __nv_bfloat16* W = net->p16 + net->w_off[(size_t)l];
            gemm(net->stream, rows, K, N, din, N, 1, W, K, 1, nullptr, 0, net->h[(size_t)l - 1], net->d[(size_t)l - 1],
                 nullptr, K);
        }
    }
}

// ---- fused form: launches ------------------------------------------------------------------

size_t rows_smem(const lbm_mlp* net, bool train)
{
    size_t e = 0;
    for (int l = 0; l < net->L; ++l) e += (size_t)ROWS * tile_ld(net->sizes[(size_t)l]);
    if (train)
        for (int l = 1; l <= net->L; ++l) e += (size_t)ROWS * tile_ld(net->sizes[(size_t)l]);
    return e * sizeof(__nv_bfloat16) + (train ? sizeof(float) * ROWS * (size_t)net->sizes[(size_t)net->L] : 0);
}

NetArgs net_args(const lbm_mlp* net)
{
    NetArgs n{};
    n.L = net->L;
    for (size_t l = 0; l <= (size_t)net->L; ++l) n.size[l] = net->sizes[l];
    for (size_t l = 0; l < (size_t)net->L; ++l) {
        n.w_off[l] = net->w_off[l];
        n.b_off[l] = net->b_off[l];
        n.wf_off[l] = net->wf_off[l];
        n.wb_off[l] = net->wb_off[l];
        if (l < net->hT.size()) {
            n.hT[l] = net->hT[l];
            n.dT[l] = net->dT[l];
        }
    }
    n.p = net->p;
    n.wf = net->wf;
    n.wb = net->wb;
    n.shift = net->in_shift;
    n.scale = net->in_scale;
    n.ld = net->cap;
    n.r2 = net->r2;
    return n;
}

// `overlap`: the kernel may be set up while the one before it in the stream, one of this file's
// own, still runs (programmatic dependent launch; it waits before it touches that one's data).
template <class A>
void launch(void (*k)(const A), int grid, int block, size_t smem, bool overlap, cudaStream_t s, const A& a)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    cudaLaunchKernelEx(&c, k, a);
}

// Forward pass (t null) or forward, loss and backward pass of `rows` rows. `tick` advances Adam's
// step count. `overlap` only where x, t and idx were not written by the kernel before.
void fused_rows(lbm_mlp* net, const float* x, const float* t, const int* idx, int rows, float* y, bool tick, bool overlap)
{
    RowsArgs a{};
    a.n = net_args(net);
    a.X = x;
    a.T = t;
    a.idx = idx;
    a.rows = rows;
    a.y = y;
    a.grad_scale = 1.f / (float)((long long)rows * net->sizes[(size_t)net->L]);
    a.tick = tick ? net->t : nullptr;
    launch(k_rows, (rows + ROWS - 1) / ROWS, ROWS_THREADS, rows_smem(net, t != nullptr), overlap, net->stream, a);
}

// The gradients of the rows of the last fused_rows, the loss into loss_dev[slot], and with `step`
// the Adam step.
void fused_update(lbm_mlp* net, int rows, int slot, bool step, float lr, float b1, float b2, float eps)
{
    UpdateArgs a{};
    a.n = net_args(net);
    a.rows = rows;
    a.p = net->p;
    a.m = net->m;
    a.v = net->v;
    a.g = net->g;
    a.t = step ? net->t : nullptr;
    a.lr = lr;
    a.b1 = b1;
    a.b2 = b2;
    a.eps = eps;
    a.loss = net->loss_dev + slot;
    const long long outputs = (long long)rows * net->sizes[(size_t)net->L];
    a.loss_scale = 1.0 / (double)outputs;
    a.loss_part = net->loss_part;
    a.loss_done = net->loss_done;
    int tasks = (int)((outputs + 256 * LOSS_TILES - 1) / (256 * LOSS_TILES));
    for (size_t l = 0; l < (size_t)net->L; ++l)
        tasks += (net->sizes[l + 1] + 15) / 16 * ((net->sizes[l] + 7) / 8) + net->sizes[l + 1];
    constexpr int W = UPD_THREADS / 32;
    launch(k_update, (tasks + W - 1) / W, UPD_THREADS, 0, true, net->stream, a);
}

void refresh_weights(lbm_mlp* net)
{
    if (net->fused) k_pack_weights<<<blocks_for(net->nparam), 256, 0, net->stream>>>(net_args(net));
    else k_to_bf16<<<blocks_for(net->nparam), 256, 0, net->stream>>>(net->p, net->nparam, net->p16);
}

void adam(lbm_mlp* net, float lr, float b1, float b2, float eps)
{
    k_adam<<<blocks_for(net->nparam), 256, 0, net->stream>>>(net->p, net->m, net->v, net->g, net->nparam, net->t, lr, b1,
                                                              b2, eps, net->fused ? nullptr : net->p16);
    k_adam_tick<<<1, 32, 0, net->stream>>>(net->t);
    if (net->fused) refresh_weights(net);
}

lbm_status ensure_loss_slots(lbm_mlp* net, int n)
{
    if (n <= net->loss_cap) return LBM_OK;
    free_dev(net, net->loss_dev);
    net->loss_dev = nullptr;
    lbm_status s = malloc_dev(net, &net->loss_dev, (size_t)n);
    if (s != LBM_OK) return s;
    net->loss_cap = n;
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_mlp_create(lbm_mlp** out, int nlayers, const int* sizes, void* cuda_stream)
{
    if (!out) return LBM_E_INVALID;
    *out = nullptr;
    if (nlayers < 1 || nlayers > 8 || !sizes) return LBM_E_INVALID;
    for (int l = 0; l <= nlayers; ++l)
        if (sizes[l] < 1 || sizes[l] > 4096) return LBM_E_INVALID;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        return LBM_E_CUDA;
    }
    lbm_mlp* net = new lbm_mlp();
    net->L = nlayers;
    net->sizes.assign(sizes, sizes + nlayers + 1);
    net->stream = (cudaStream_t)cuda_stream;
    long long off = 0;
    for (int l = 0; l < nlayers; ++l) {
        net->w_off.push_back(off);
        off += (long long)sizes[l] * sizes[l + 1];
        net->b_off.push_back(off);
        off += sizes[l + 1];
    }
    net->nparam = off;
    lbm_status s = LBM_OK;
    if ((s = malloc_dev(net, &net->p, (size_t)off)) != LBM_OK || (s = malloc_dev(net, &net->m, (size_t)off)) != LBM_OK ||
        (s = malloc_dev(net, &net->v, (size_t)off)) != LBM_OK || (s = malloc_dev(net, &net->g, (size_t)off)) != LBM_OK ||
        (s = malloc_dev(net, &net->t, 1)) != LBM_OK) {
        lbm_mlp_destroy(net);
        return s;
    }
    long long weights = 0, wf = 0, wb = 0;
    for (int l = 0; l < nlayers; ++l) {
        weights += (long long)sizes[l] * sizes[l + 1];
        net->wf_off.push_back(wf);
        net->wb_off.push_back(wb);
        wf += frag_elems(sizes[l], sizes[l + 1]);
        if (l > 0) wb += frag_elems(sizes[l + 1], sizes[l]);
    }
    net->fused = weights <= FUSED_WEIGHTS && rows_smem(net, true) <= FUSED_SMEM &&
                 cudaFuncSetAttribute(k_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM) == cudaSuccess;
    if (net->fused)
        s = (s = malloc_dev(net, &net->wf, (size_t)wf)) != LBM_OK || (s = malloc_dev(net, &net->wb, (size_t)wb)) != LBM_OK
                ? s
                : malloc_dev(net, &net->loss_done, 1);
    else
        s = malloc_dev(net, &net->p16, (size_t)off);
    if (s != LBM_OK) {
        lbm_mlp_destroy(net);
        return s;
    }
    if (net->fused) {  // the fragments' padding stays zero
        cudaMemsetAsync(net->wf, 0, sizeof(__nv_bfloat16) * wf, net->stream);
        cudaMemsetAsync(net->wb, 0, sizeof(__nv_bfloat16) * wb, net->stream);
        cudaMemsetAsync(net->loss_done, 0, sizeof(int), net->stream);
    } else {
        cudaMemsetAsync(net->p16, 0, sizeof(__nv_bfloat16) * off, net->stream);
    }
    cudaMemsetAsync(net->p, 0, sizeof(float) * off, net->stream);
    cudaMemsetAsync(net->m, 0, sizeof(float) * off, net->stream);
    cudaMemsetAsync(net->v, 0, sizeof(float) * off, net->stream);
    cudaMemsetAsync(net->g, 0, sizeof(float) * off, net->stream);
    cudaMemsetAsync(net->t, 0, sizeof(int), net->stream);
    if (cudaStreamSynchronize(net->stream) != cudaSuccess) {
        cudaGetLastError();
        lbm_mlp_destroy(net);
        return LBM_E_CUDA;
    }
    *out = net;
    return LBM_OK;
}

long long lbm_mlp_num_params(const lbm_mlp* net) { return net ? net->nparam : -1; }

lbm_status lbm_mlp_set_params(lbm_mlp* net, const double* params)
{
    if (!net || !params) return LBM_E_INVALID;
    std::vector<float> h((size_t)net->nparam);
    for (long long i = 0; i < net->nparam; ++i) h[(size_t)i] = (float)params[i];
    MK(cudaMemcpyAsync(net->p, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice, net->stream));
    refresh_weights(net);
    MK(cudaGetLastError());
    MK(cudaMemsetAsync(net->m, 0, sizeof(float) * net->nparam, net->stream));
    MK(cudaMemsetAsync(net->v, 0, sizeof(float) * net->nparam, net->stream));
    MK(cudaMemsetAsync(net->t, 0, sizeof(int), net->stream));
    MK(cudaStreamSynchronize(net->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_set_input_scaling(lbm_mlp* net, const double* shift, const double* scale)
{
    if (!net || (!shift) != (!scale)) return LBM_E_INVALID;
    const int K = net->sizes[0];
    if (!shift) {
        free_dev(net, net->in_shift);
        free_dev(net, net->in_scale);
        net->in_shift = net->in_scale = nullptr;
        return LBM_OK;
    }
    std::vector<float> h((size_t)2 * K);
    for (int c = 0; c < K; ++c) {
        if (!std::isfinite(shift[c]) || !std::isfinite(scale[c])) return mfail(net, LBM_E_INVALID, "non-finite scaling");
        h[(size_t)c] = (float)shift[c];
        h[(size_t)K + c] = (float)scale[c];
    }
    lbm_status s = LBM_OK;
    if (!net->in_shift && ((s = malloc_dev(net, &net->in_shift, (size_t)K)) != LBM_OK ||
                           (s = malloc_dev(net, &net->in_scale, (size_t)K)) != LBM_OK))
        return s;
    MK(cudaMemcpyAsync(net->in_shift, h.data(), sizeof(float) * K, cudaMemcpyHostToDevice, net->stream));
    MK(cudaMemcpyAsync(net->in_scale, h.data() + K, sizeof(float) * K, cudaMemcpyHostToDevice, net->stream));
    MK(cudaStreamSynchronize(net->stream));
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp* net, double* params, double* grads)
{
    if (!net || (!params && !grads)) return LBM_E_INVALID;
    std::vector<float> h((size_t)net->nparam);
    if (params) {
        MK(cudaMemcpyAsync(h.data(), net->p, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, net->stream));
        MK(cudaStreamSynchronize(net->stream));
        for (long long i = 0; i < net->nparam; ++i) params[i] = h[(size_t)i];
    }
    if (grads) {
        MK(cudaMemcpyAsync(h.data(), net->g, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, net->stream));
        MK(cudaStreamSynchronize(net->stream));
        for (long long i = 0; i < net->nparam; ++i) grads[i] = h[(size_t)i];
    }
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp* net, const float* x, int rows, float* y)
{
    if (!net || !x || !y || rows < 0) return LBM_E_INVALID;
    if (rows == 0) return LBM_OK;
    if (net->fused) {
        const size_t nx = (size_t)rows * net->sizes[0], ny = (size_t)rows * net->sizes[(size_t)net->L];
        const bool alias = (uintptr_t)y < (uintptr_t)(x + nx) && (uintptr_t)x < (uintptr_t)(y + ny);
        if (alias) {  // blocks read their rows while others write theirs
            lbm_status s = ensure_rows(net, rows);
            if (s != LBM_OK) return s;
        }
        fused_rows(net, x, nullptr, nullptr, rows, alias ? net->r2 : y, false, false);
        if (alias) MK(cudaMemcpyAsync(y, net->r2, sizeof(float) * ny, cudaMemcpyDeviceToDevice, net->stream));
        MK(cudaGetLastError());
        return LBM_OK;
    }
    lbm_status s = ensure_rows(net, rows);
    if (s != LBM_OK) return s;
    const int K = net->sizes[0], O = net->sizes[(size_t)net->L];
    k_gather<<<blocks_for((long long)rows * K), 256, 0, net->stream>>>(x, nullptr, nullptr, rows, K, O, net->in_shift,
                                                                         net->in_scale, net->xb, nullptr);
    forward(net, rows);
    MK(cudaMemcpyAsync(y, net->y, sizeof(float) * (size_t)rows * O, cudaMemcpyDeviceToDevice, net->stream));
    MK(cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_mlp_loss_grad(lbm_mlp* net, const float* x, const float* t, int rows, double* loss)
{
    if (!net || !x || !t || rows < 1) return LBM_E_INVALID;
    lbm_status s = ensure_rows(net, rows);
    if (s == LBM_OK) s = ensure_loss_slots(net, 1);
    if (s != LBM_OK) return s;
    const int K = net->sizes[0], O = net->sizes[(size_t)net->L];
    MK(cudaMemsetAsync(net->loss_dev, 0, sizeof(double), net->stream));
    if (net->fused) {
        fused_rows(net, x, t, nullptr, rows, nullptr, false, false);
        fused_update(net, rows, 0, false, 0.f, 0.f, 0.f, 0.f);
    } else {
        k_gather<<<blocks_for((long long)rows * (K + O)), 256, 0, net->stream>>>(x, t, nullptr, rows, K, O, net->in_shift,
                                                                                   net->in_scale, net->xb, net->tb);
        backward(net, rows, 0);
    }
    MK(cudaGetLastError());
    if (loss) {
        MK(cudaMemcpyAsync(loss, net->loss_dev, sizeof(double), cudaMemcpyDeviceToHost, net->stream));
        MK(cudaStreamSynchronize(net->stream));
    }
    return LBM_OK;
}

lbm_status lbm_mlp_adam_step(lbm_mlp* net, double lr, double beta1, double beta2, double eps)
{
    if (!net || !(lr > 0.0)) return LBM_E_INVALID;
    adam(net, (float)lr, (float)beta1, (float)beta2, (float)eps);
    MK(cudaGetLastError());
    return LBM_OK;
}

lbm_status lbm_mlp_train(lbm_mlp* net, const float* x, const float* t, int n, int batch, int epochs, double lr,
                         unsigned seed, double* epoch_loss)
{
    if (!net || !x || !t || n < 1 || batch < 1 || epochs < 1 || !(lr > 0.0)) return LBM_E_INVALID;
    batch = std::min(batch, n);
    lbm_status s = ensure_rows(net, batch);
    if (s == LBM_OK) s = ensure_loss_slots(net, epochs);
    if (s != LBM_OK) return s;
    if (net->idx_cap < n) {
        free_dev(net, net->idx);
        net->idx = nullptr;
        if ((s = malloc_dev(net, &net->idx, (size_t)n)) != LBM_OK) return s;
        net->idx_cap = n;
    }
    const int K = net->sizes[0], O = net->sizes[(size_t)net->L];
    MK(cudaMemsetAsync(net->loss_dev, 0, sizeof(double) * epochs, net->stream));
    std::mt19937 rng(seed);
    std::vector<int> perm((size_t)n);
    const int nb = n / batch;  // full minibatches per epoch
    for (int e = 0; e < epochs; ++e) {
        for (int i = 0; i < n; ++i) perm[(size_t)i] = i;
        std::shuffle(perm.begin(), perm.end(), rng);
        MK(cudaMemcpyAsync(net->idx, perm.data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice, net->stream));
        for (int bi = 0; bi < nb; ++bi) {
            if (net->fused) {
                // (the first minibatch follows the copy of the permutation, the others k_update)
                fused_rows(net, x, t, net->idx + (size_t)bi * batch, batch, nullptr, true, bi > 0);
                fused_update(net, batch, e, true, (float)lr, 0.9f, 0.999f, 1e-8f);
                continue;
            }
            k_gather<<<blocks_for((long long)batch * (K + O)), 256, 0, net->stream>>>(x, t, net->idx + (size_t)bi * batch,
                                                                                      batch, K, O, net->in_shift,
                                                                                      net->in_scale, net->xb, net->tb);
            backward(net, batch, e);
            adam(net, (float)lr, 0.9f, 0.999f, 1e-8f);
        }
        // the host permutation buffer is reused next epoch: wait for its copy
        MK(cudaStreamSynchronize(net->stream));
    }
    MK(cudaGetLastError());
    if (epoch_loss) {
        std::vector<double> h((size_t)epochs);
        MK(cudaMemcpy(h.data(), net->loss_dev, sizeof(double) * epochs, cudaMemcpyDeviceToHost));
        for (int e = 0; e < epochs; ++e) epoch_loss[e] = h[(size_t)e] / nb;
    }
    return LBM_OK;
}

const char* lbm_mlp_last_error(const lbm_mlp* net) { return net ? net->err.c_str() : "null network"; }

void lbm_mlp_destroy(lbm_mlp* net)
{
    if (!net) return;
    if (net->stream) cudaStreamSynchronize(net->stream);
    else cudaDeviceSynchronize();
    for (void* p : net->allocs) cudaFree(p);
    delete net;
}

}  // extern "C"
