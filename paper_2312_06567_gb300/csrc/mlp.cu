// Learned initial guess for the Q' Newton solve: a 9 -> 64 -> 64 -> 5 SiLU
// network trained on the GPU on (features, Delta) pairs that the solver's own
// converged Newton solves log.  The paper has the Newton solve only; the
// guess is this project's addition (features, target and network as in
// mlp_features / the header's MLP entry points).
//
// Precision: weights and layer inputs are rounded to BF16 (the operands of
// every product), all sums accumulate in FP32, the optimiser keeps FP32
// master weights (Adam).  With bf16 = 0 the same kernels run on FP32
// operands (used by the gradient check against the FP64 reference).
//
// Training kernel: a block of 256 threads takes chunks of 32 samples through the
// three layers and back as small GEMMs on register tiles from shared memory, and
// leaves its sums of the weight gradients in a row of its own (grid <= two
// blocks per multiprocessor); the optimiser kernel adds the rows up in order.
// One value per thread and 64 samples per block, gradients by atomics, took
// 77 us for a batch of 4096 (64 of 152 multiprocessors, bank conflicts on W2's
// columns, 328,000 atomics); this takes 17 us (22 before the weights, features
// and targets were requested together instead of one round trip each), the
// update 5 us as before.
// Each forward value and each backward value of a sample is the same chain of
// FMAs in the same order as before; only sums over samples are ordered anew.
#include "bgk_internal.cuh"
#include "bgk_mlp.cuh"

namespace {

constexpr int SB = 32;       // samples per chunk
constexpr int NT = 256;      // threads per block
constexpr int LD = MLP_H + 4;                            // row stride of the tiles (16-byte rows, no bank conflicts)
constexpr int NSMALL = MLP_IN * MLP_H + MLP_H + MLP_H + MLP_H * MLP_OUT + MLP_OUT;      // all gradients but W2's
constexpr int NSR = (NSMALL + NT - 1) / NT;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float rnd(float x, int bf16) { return bf16 ? bf16r(x) : x; }
__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
    const float s = 1.f / (1.f + __expf(-z));
    return s * (1.f + z * (1.f - s));
}

struct TrainSmem {
    float w2[MLP_H][LD], w2t[MLP_H][LD];                 // W2 and its transpose
    float w1[MLP_IN][MLP_H], w3[MLP_H][MLP_OUT];
    float b1[MLP_H], b2[MLP_H], b3[8];
    float h1[SB][LD], h2[SB][LD], d2[SB][LD], d1[SB][LD];
    float xn[SB][MLP_IN + 3], dy[SB][8], tn[SB][8];
    float red[NT / 32];
};

// acc[r][c] += sum_k A[s0 + r][k] B[k][4 j4 + c], k ascending
__device__ __forceinline__ void tile2x4(const float (*A)[LD], const float (*B)[LD], int s0, int j, float (&acc)[2][4]) {
#pragma unroll 4
    for (int k = 0; k < MLP_H; k += 4) {
        const float4 a0 = *reinterpret_cast<const float4 *>(&A[s0][k]), a1 = *reinterpret_cast<const float4 *>(&A[s0 + 1][k]);
        const float x0[4] = {a0.x, a0.y, a0.z, a0.w}, x1[4] = {a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 b = *reinterpret_cast<const float4 *>(&B[k + i][j]);
            const float y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                acc[0][c] = fmaf(x0[i], y[c], acc[0][c]);
                acc[1][c] = fmaf(x1[i], y[c], acc[1][c]);
            }
        }
    }
}

// x[n][9] raw features, t[n][5] raw targets; idx[b] sample indices of this
// batch; part[gridDim.x][MLP_NPARAM], loss_part[gridDim.x].
__global__ void __launch_bounds__(NT, 2) k_mlp_train(MlpParams prm, const float *x, const float *t, const int *idx, int nb,
                                                     float *part, double *loss_part, int bf16) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem &sm = *reinterpret_cast<TrainSmem *>(smem_raw);
    const int tid = threadIdx.x;
    const float *W1 = prm.w, *b1 = W1 + MLP_IN * MLP_H, *W2 = b1 + MLP_H, *b2 = W2 + MLP_H * MLP_H;
    const float *W3 = b2 + MLP_H, *b3 = W3 + MLP_H * MLP_OUT;
    // the weights, all requested before any is used (one round trip)
    {
        float v2[MLP_H * MLP_H / NT], v1[(MLP_IN * MLP_H + NT - 1) / NT], v3[(MLP_H * MLP_OUT + NT - 1) / NT], vb[3];
#pragma unroll
        for (int q = 0; q < MLP_H * MLP_H / NT; ++q) v2[q] = W2[tid + q * NT];
#pragma unroll
        for (int q = 0; q < (MLP_IN * MLP_H + NT - 1) / NT; ++q) v1[q] = tid + q * NT < MLP_IN * MLP_H ? W1[tid + q * NT] : 0.f;
#pragma unroll
        for (int q = 0; q < (MLP_H * MLP_OUT + NT - 1) / NT; ++q) v3[q] = tid + q * NT < MLP_H * MLP_OUT ? W3[tid + q * NT] : 0.f;
        vb[0] = b1[tid % MLP_H]; vb[1] = b2[tid % MLP_H]; vb[2] = b3[tid % MLP_OUT];
#pragma unroll
        for (int q = 0; q < MLP_H * MLP_H / NT; ++q) {
            const int i = tid + q * NT;
            const float v = rnd(v2[q], bf16);
            sm.w2[i / MLP_H][i % MLP_H] = v;
            sm.w2t[i % MLP_H][i / MLP_H] = v;
        }
#pragma unroll
        for (int q = 0; q < (MLP_IN * MLP_H + NT - 1) / NT; ++q) {
            const int i = tid + q * NT;
            if (i < MLP_IN * MLP_H) sm.w1[i / MLP_H][i % MLP_H] = rnd(v1[q], bf16);
        }
#pragma unroll
        for (int q = 0; q < (MLP_H * MLP_OUT + NT - 1) / NT; ++q) {
            const int i = tid + q * NT;
            if (i < MLP_H * MLP_OUT) sm.w3[i / MLP_OUT][i % MLP_OUT] = rnd(v3[q], bf16);
        }
        if (tid < MLP_H) { sm.b1[tid] = vb[0]; sm.b2[tid] = vb[1]; }
        if (tid < MLP_OUT) sm.b3[tid] = vb[2];
    }
    const int j = 4 * (tid % 16), s0 = 2 * (tid / 16);   // this thread's 2 x 4 tile of a [32][64] layer
    const int gk = 4 * (tid / 16);                       // and rows gk..gk+3 of its 4 x 4 tile of W2's gradient
    float g2[4][4] = {}, gs[NSR] = {};
    float lsum = 0.f;
    for (int c0 = blockIdx.x * SB; c0 < nb; c0 += gridDim.x * SB) {
        const int ns = min(SB, nb - c0);
        __syncthreads();
        // features and targets, normalised (both gathers in flight at once)
        {
            const int sa = tid / MLP_IN, sb = (tid + NT) / MLP_IN, st = tid / MLP_OUT;
            const int fa = tid % MLP_IN, fb = (tid + NT) % MLP_IN, fo = tid % MLP_OUT;
            const bool ha = sa < ns, hb = sb < ns, ht = st < ns;
            const int ia = ha ? idx[c0 + sa] : 0, ib = hb ? idx[c0 + sb] : 0, it = ht ? idx[c0 + st] : 0;
            const float xa = ha ? x[(size_t)ia * MLP_IN + fa] : 0.f, xb = hb ? x[(size_t)ib * MLP_IN + fb] : 0.f;
            const float xt = ht ? t[(size_t)it * MLP_OUT + fo] : 0.f;
            if (sa < SB) sm.xn[sa][fa] = ha ? rnd((xa - prm.norm[fa]) / prm.norm[MLP_IN + fa], bf16) : 0.f;
            if (sb < SB) sm.xn[sb][fb] = hb ? rnd((xb - prm.norm[fb]) / prm.norm[MLP_IN + fb], bf16) : 0.f;
            if (st < SB) sm.tn[st][fo] = ht ? (xt - prm.norm[2 * MLP_IN + fo]) / prm.norm[2 * MLP_IN + MLP_OUT + fo] : 0.f;
        }
        __syncthreads();
        // ---- layers 1 and 2: z stays in the registers of the tile's thread
        float z1[2][4], z2[2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float z = sm.b1[j + c];
#pragma unroll
                for (int f = 0; f < MLP_IN; ++f) z = fmaf(sm.xn[s0 + r][f], sm.w1[f][j + c], z);
                z1[r][c] = z;
                sm.h1[s0 + r][j + c] = rnd(silu(z), bf16);
                z2[r][c] = sm.b2[j + c];
            }
        __syncthreads();
        tile2x4(sm.h1, sm.w2, s0, j, z2);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) sm.h2[s0 + r][j + c] = rnd(silu(z2[r][c]), bf16);
        __syncthreads();
        // ---- layer 3, residual, loss, dL/dy = 2 (y - tn) / (nb * 5)
        if (tid < SB * MLP_OUT) {
            const int s = tid / MLP_OUT, o = tid % MLP_OUT;
            float d = 0.f;
            if (s < ns) {
                float y = sm.b3[o];
#pragma unroll 8
                for (int k = 0; k < MLP_H; ++k) y = fmaf(sm.h2[s][k], sm.w3[k][o], y);
                const float r = y - sm.tn[s][o];
                lsum = fmaf(r, r, lsum);
                d = 2.f * r / (float)(nb * MLP_OUT);
            }
            sm.dy[s][o] = d;
        }
        __syncthreads();
        // ---- dz2 = (dy W3^T) * s'(z2), dz1 = (dz2 W2^T) * s'(z1)
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float d = 0.f;
#pragma unroll
                for (int o = 0; o < MLP_OUT; ++o) d = fmaf(sm.dy[s0 + r][o], sm.w3[j + c][o], d);
                sm.d2[s0 + r][j + c] = d * silu_grad(z2[r][c]);
            }
        __syncthreads();
        float d1[2][4] = {};
        tile2x4(sm.d2, sm.w2t, s0, j, d1);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) sm.d1[s0 + r][j + c] = d1[r][c] * silu_grad(z1[r][c]);
        __syncthreads();
        // ---- gradients: W2 as 4 x 4 tiles over the samples (padded ones have
        // dz = 0), the rest one value per thread and round
#pragma unroll 4
        for (int s = 0; s < SB; ++s) {
            const float4 a = *reinterpret_cast<const float4 *>(&sm.h1[s][gk]), b = *reinterpret_cast<const float4 *>(&sm.d2[s][j]);
            const float x0[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) g2[r][c] = fmaf(x0[r], y[c], g2[r][c]);
        }
#pragma unroll
        for (int q = 0; q < NSR; ++q) {
            int i = tid + q * NT;
            float g = gs[q];
            if (i < MLP_IN * MLP_H) {
                _Pragma("unroll 8") for (int s = 0; s < SB; ++s) g = fmaf(sm.xn[s][i / MLP_H], sm.d1[s][i % MLP_H], g);
            } else if ((i -= MLP_IN * MLP_H) < MLP_H) {
                _Pragma("unroll 8") for (int s = 0; s < SB; ++s) g += sm.d1[s][i];
            } else if ((i -= MLP_H) < MLP_H) {
                _Pragma("unroll 8") for (int s = 0; s < SB; ++s) g += sm.d2[s][i];
            } else if ((i -= MLP_H) < MLP_H * MLP_OUT) {
                _Pragma("unroll 8") for (int s = 0; s < SB; ++s) g = fmaf(sm.h2[s][i / MLP_OUT], sm.dy[s][i % MLP_OUT], g);
            } else if ((i -= MLP_H * MLP_OUT) < MLP_OUT) {
                _Pragma("unroll 8") for (int s = 0; s < SB; ++s) g += sm.dy[s][i];
            }
            gs[q] = g;
        }
    }
    // ---- this block's row: parameters in their flat order W1 b1 W2 b2 W3 b3
    float *row = part + (size_t)blockIdx.x * MLP_NPARAM;
    constexpr int OW2 = MLP_IN * MLP_H + MLP_H;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) row[OW2 + (gk + r) * MLP_H + j + c] = g2[r][c];
#pragma unroll
    for (int q = 0; q < NSR; ++q) {
        const int i = tid + q * NT;
        if (i < NSMALL) row[i < OW2 ? i : i + MLP_H * MLP_H] = gs[q];
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if ((tid & 31) == 0) sm.red[tid >> 5] = lsum;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < NT / 32; ++w) s += sm.red[w];
        loss_part[blockIdx.x] = s / (double)(nb * MLP_OUT);
    }
}

// The gradient as the sum of the training blocks' rows (eight threads per
// parameter, rows in a fixed order), then Adam on the FP32 master weights, or
// (grad not null) the gradient itself; the loss joins *loss.
__global__ void __launch_bounds__(NT) k_mlp_adam(float *w, float *m, float *v, const float *part, const double *loss_part,
                                                 int rows, float *grad, double *loss, float lr, float b1, float b2, float eps,
                                                 float c1, float c2) {
    __shared__ float red[NT / 32][33];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float g = 0.f;
    if (i < MLP_NPARAM) {
#pragma unroll 8
        for (int r = wib; r < rows; r += NT / 32) g += part[(size_t)r * MLP_NPARAM + i];
    }
    red[wib][lane] = g;
    __syncthreads();
    if (wib == 0 && i < MLP_NPARAM) {
        g = 0.f;
#pragma unroll
        for (int r = 0; r < NT / 32; ++r) g += red[r][lane];
        if (grad) {
            grad[i] = g;
        } else {
            const float mi = b1 * m[i] + (1.f - b1) * g;
            const float vi = b2 * v[i] + (1.f - b2) * g * g;
            m[i] = mi;
            v[i] = vi;
            w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        }
    }
    if (blockIdx.x == 0 && wib == 1) {
        double s = 0.0;
        for (int r = lane; r < rows; r += 32) s += loss_part[r];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *loss += s;
    }
}

}  // namespace

// blocks (and gradient rows) of a batch of nb samples
static int mlp_rows(int nb) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    const int chunks = (nb + SB - 1) / SB;
    return chunks < 2 * sms ? chunks : 2 * sms;
}

size_t mlp_train_scratch(int nb) { return (size_t)mlp_rows(nb) * (MLP_NPARAM * sizeof(float) + sizeof(double)); }

cudaError_t launch_mlp_train(const MlpParams &p, const float *x, const float *t, const int *idx, int nb, void *scratch,
                             int bf16, cudaStream_t s) {
    const size_t smem = sizeof(TrainSmem);
    static SmemLimit lim;
    size_t *attr = lim.slot();
    if (!attr) return cudaErrorInvalidDevice;
    if (smem > *attr) {
        cudaError_t e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        *attr = smem;
    }
    const int rows = mlp_rows(nb);
    if (rows < 1) return cudaErrorInvalidDevice;
    double *lp = (double *)scratch;
    k_mlp_train<<<rows, NT, smem, s>>>(p, x, t, idx, nb, (float *)(lp + rows), lp, bf16);
    return cudaGetLastError();
}

__global__ void k_mlp_round(const float *w, float *w16, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) w16[i] = mlp_round(w[i], 1);
}

cudaError_t launch_mlp_round(const float *w, float *w16, int n, cudaStream_t s) {
    k_mlp_round<<<(n + 255) / 256, 256, 0, s>>>(w, w16, n);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(float *w, float *m, float *v, const void *scratch, int nb, double *loss, float lr, float b1,
                            float b2, float eps, int step, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    const int rows = mlp_rows(nb);
    const double *lp = (const double *)scratch;
    k_mlp_adam<<<(MLP_NPARAM + 31) / 32, NT, 0, s>>>(w, m, v, (const float *)(lp + rows), lp, rows, nullptr, loss, lr, b1, b2, eps,
                                                     c1, c2);
    return cudaGetLastError();
}

cudaError_t launch_mlp_grad_sum(const void *scratch, int nb, float *grad, double *loss, cudaStream_t s) {
    const int rows = mlp_rows(nb);
    const double *lp = (const double *)scratch;
    k_mlp_adam<<<(MLP_NPARAM + 31) / 32, NT, 0, s>>>(nullptr, nullptr, nullptr, (const float *)(lp + rows), lp, rows, grad, loss,
                                                     0.f, 0.f, 0.f, 0.f, 1.f, 1.f);
    return cudaGetLastError();
}
