// Training of the warm-start MLP (see lelbm_mlp.cuh for features, targets and the
// parameter layout): hand-written forward/backward with BF16 weights and FP32
// accumulation, FP32 master weights updated by Adam, mean-squared loss on the
// standardised targets.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>
#include <random>
#include <vector>

#include "../../include/lelbm.h"
#include "lelbm_mlp.cuh"

namespace lbm {
namespace {

constexpr int TB = 64;  // samples per tile of the gradient kernel

// Sum and sum of squares of every column of a row-major [n x cols] array.
__global__ void column_stats_kernel(const float* A, long long n, int cols, double* sums) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n * cols;
         i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % cols);
        const double v = A[i];
        atomicAdd(&sums[c], v);
        atomicAdd(&sums[cols + c], v * v);
    }
}

__global__ void to_bf16_kernel(const float* src, __nv_bfloat16* dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16(src[i]);
}

// Loss and gradient over a range of samples, TB at a time.  FP32 throughout, at the BF16-rounded
// weights.  The six products of a tile (three layers forward, two back, and the three weight
// gradients) are register-tiled: a thread holds 8 samples x 4 features of a layer's tile, so a step
// of the inner loop is 32 FMAs for three shared-memory loads, where one thread per sample had to load
// an operand for every FMA.  Activations lie transposed in shared memory ([feature][sample]); the
// derivatives of SiLU wait in registers.  Blocks are persistent: each keeps the whole gradient in
// registers (a tile's sums are formed on their own, then added) and adds it to grad once, instead of
// one atomic addition per parameter and 64 samples.  Two blocks share an SM, so one computes while the
// other waits at a barrier.  FP32 FMAs and
// the shared-memory loads between them bound it (35 kFLOP a sample): 2^20 pairs in 2D take 1.29 ms, 28 TFLOP/s,
// where one thread per sample took 9.17 ms.
constexpr int kGradThreads = 128;
constexpr int kLD = TB + 4;  // row stride of the transposed tiles: float4 rows that start 4 banks apart

template <int D>
struct GradTile {
    using Md = MlpDims<D>;
    using Ly = MlpLayout<D>;
    static constexpr int H = Md::H;
    static constexpr int NI = (Md::NIN + 7) & ~7, NO = (Md::NOUT + 7) & ~7;  // padded with zeros
    float W1t[NI][H], W2t[H][H], W2[H][H], W3t[H][NO], W3[NO][H];  // t: [input][output]
    float b1[H], b2[H], b3[NO];
    float xs[NI][kLD], h1[H][kLD], h2[H][kLD], dz2[H][kLD], dy[NO][kLD];  // h2's place takes dz1
};

// acc[r][c] += sum_k A[k][s0 + r] B[k][f0 + c]
template <int K, int LB>
__device__ __forceinline__ void tile_product(const float* A, const float* B, float (&acc)[8][4]) {
#pragma unroll 8
    for (int k = 0; k < K; k++) {
        const float4 a0 = *reinterpret_cast<const float4*>(A + k * kLD);
        const float4 a1 = *reinterpret_cast<const float4*>(A + k * kLD + 4);
        const float4 b = *reinterpret_cast<const float4*>(B + k * LB);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int r = 0; r < 8; r++)
#pragma unroll
            for (int c = 0; c < 4; c++) acc[r][c] = fmaf(av[r], bv[c], acc[r][c]);
    }
}

// column c of a thread's tile to row f0 + c of a transposed array
__device__ __forceinline__ void store_column(float* row, const float (&v)[8][4], int c) {
    *reinterpret_cast<float4*>(row) = make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
    *reinterpret_cast<float4*>(row + 4) = make_float4(v[4][c], v[5][c], v[6][c], v[7][c]);
}

// out[r] += sum_s a[s] B[r][s] over the samples s of a tile: one row a, R rows of B that lie
// ldb floats apart.
template <int R>
__device__ __forceinline__ void sample_sums(const float* a, const float* B, int ldb, float (&out)[R]) {
    float t[R];
#pragma unroll
    for (int r = 0; r < R; r++) t[r] = 0.f;
#pragma unroll 4
    for (int s = 0; s < TB; s += 4) {
        const float4 x = *reinterpret_cast<const float4*>(a + s);
#pragma unroll
        for (int r = 0; r < R; r++) {
            const float4 y = *reinterpret_cast<const float4*>(B + r * ldb + s);
            t[r] = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, t[r]))));
        }
    }
#pragma unroll
    for (int r = 0; r < R; r++) out[r] += t[r];
}

template <int D>
__global__ void __launch_bounds__(kGradThreads, 2) mlp_grad_kernel(const __nv_bfloat16* Wb, const float* nrm,
                                                                   const float* X, const float* Y,
                                                                   const long long* idx, long long b0, int bsize,
                                                                   float scale, float* grad, double* loss) {
    using G = GradTile<D>;
    using Md = MlpDims<D>;
    using Ly = MlpLayout<D>;
    constexpr int NIN = Md::NIN, NOUT = Md::NOUT, H = Md::H, NI = G::NI, NO = G::NO;
    static_assert(H == 64 && TB == 64 && kGradThreads == 128, "thread tiles");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    G& S = *reinterpret_cast<G*>(smem_raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < NI * H; i += kGradThreads) {
        const int m = i / H, j = i % H;
        S.W1t[m][j] = m < NIN ? __bfloat162float(Wb[Ly::W1 + j * NIN + m]) : 0.f;
    }
    for (int i = tid; i < H * H; i += kGradThreads) {
        const float w = __bfloat162float(Wb[Ly::W2 + i]);
        S.W2[i / H][i % H] = w;
        S.W2t[i % H][i / H] = w;
    }
    for (int i = tid; i < NO * H; i += kGradThreads) {
        const int k = i / H, j = i % H;
        const float w = k < NOUT ? __bfloat162float(Wb[Ly::W3 + k * H + j]) : 0.f;
        S.W3[k][j] = w;
        S.W3t[j][k] = w;
    }
    for (int i = tid; i < H; i += kGradThreads) {
        S.b1[i] = __bfloat162float(Wb[Ly::B1 + i]);
        S.b2[i] = __bfloat162float(Wb[Ly::B2 + i]);
        if (i < NO) S.b3[i] = i < NOUT ? __bfloat162float(Wb[Ly::B3 + i]) : 0.f;
    }
    const int s0 = (tid >> 4) * 8, f0 = (tid & 15) * 4;  // layer tiles: 8 samples x 4 features
    const int row = tid & 63, half = tid >> 6;           // one row (sample, feature) and half of the other side
    const int gi = tid >> 4, gj = tid & 15;              // gW2: rows gi + 8 r, columns gj + 16 c
    float g2[8][4], g1[NI / 2], g3[NO / 2], gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, myloss = 0.f;
    double loss_sum = 0.0;
#pragma unroll
    for (int r = 0; r < 8; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) g2[r][c] = 0.f;
#pragma unroll
    for (int k = 0; k < NI / 2; k++) g1[k] = 0.f;
#pragma unroll
    for (int k = 0; k < NO / 2; k++) g3[k] = 0.f;

    const int ntile = (bsize + TB - 1) / TB;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int r = tile * TB + row;
        const bool valid = r < bsize;
        const long long src = valid ? (idx ? idx[b0 + r] : b0 + r) : 0;
        float tgt[NO / 2];
#pragma unroll
        for (int k = 0; k < NI / 2; k++) {
            const int m = half * (NI / 2) + k;
            S.xs[m][row] = valid && m < NIN ? (X[src * NIN + m] - nrm[m]) / nrm[NIN + m] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < NO / 2; k++) {
            const int o = half * (NO / 2) + k;
            tgt[k] = valid && o < NOUT ? (Y[src * NOUT + o] - nrm[2 * NIN + o]) / nrm[2 * NIN + NOUT + o] : 0.f;
        }
        __syncthreads();  // xs written (and, from the second tile on, the last one's sums read)
        float d1[8][4], d2[8][4];  // SiLU'(z1), SiLU'(z2)
        {
            float z[8][4];
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] = S.b1[f0 + c];
            tile_product<NI, H>(&S.xs[0][s0], &S.W1t[0][f0], z);
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const float e = 1.f / (1.f + __expf(-z[q][c]));
                    d1[q][c] = e * (1.f + z[q][c] * (1.f - e));
                    z[q][c] *= e;
                }
#pragma unroll
            for (int c = 0; c < 4; c++) store_column(&S.h1[f0 + c][s0], z, c);
        }
        __syncthreads();
        {
            float z[8][4];
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] = S.b2[f0 + c];
            tile_product<H, H>(&S.h1[0][s0], &S.W2t[0][f0], z);
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) {
                    const float e = 1.f / (1.f + __expf(-z[q][c]));
                    d2[q][c] = e * (1.f + z[q][c] * (1.f - e));
                    z[q][c] *= e;
                }
#pragma unroll
            for (int c = 0; c < 4; c++) store_column(&S.h2[f0 + c][s0], z, c);
        }
        __syncthreads();
        {
            // outputs, loss and dy: sample `row`, half of the outputs
            float y[NO / 2];
#pragma unroll
            for (int k = 0; k < NO / 2; k++) y[k] = S.b3[half * (NO / 2) + k];
#pragma unroll 8
            for (int i = 0; i < H; i++) {
                const float h = S.h2[i][row];
#pragma unroll
                for (int k = 0; k < NO / 2; k++) y[k] = fmaf(S.W3t[i][half * (NO / 2) + k], h, y[k]);
            }
#pragma unroll
            for (int k = 0; k < NO / 2; k++) {
                const int o = half * (NO / 2) + k;
                const float e = valid && o < NOUT ? y[k] - tgt[k] : 0.f;
                myloss += e * e;
                S.dy[o][row] = scale * e;
            }
        }
        __syncthreads();
        {
            // dz2 = (W3^T dy) SiLU'(z2)
            float z[8][4];
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] = 0.f;
            tile_product<NO, H>(&S.dy[0][s0], &S.W3[0][f0], z);
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] *= d2[q][c];
#pragma unroll
            for (int c = 0; c < 4; c++) store_column(&S.dz2[f0 + c][s0], z, c);
        }
        __syncthreads();
        {
            // dz1 = (W2^T dz2) SiLU'(z1)
            float z[8][4];
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] = 0.f;
            tile_product<H, H>(&S.dz2[0][s0], &S.W2[0][f0], z);
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) z[q][c] *= d1[q][c];
            sample_sums<NO / 2>(&S.h2[row][0], &S.dy[half * (NO / 2)][0], kLD, g3);
            __syncthreads();  // h2 read
#pragma unroll
            for (int c = 0; c < 4; c++) store_column(&S.h2[f0 + c][s0], z, c);
        }
        {
            // gW2 += dz2^T h1
            float t[8][4];
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) t[q][c] = 0.f;
#pragma unroll 2
            for (int s = 0; s < TB; s += 4) {
                float4 b[4];
#pragma unroll
                for (int c = 0; c < 4; c++) b[c] = *reinterpret_cast<const float4*>(&S.h1[gj + 16 * c][s]);
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const float4 a = *reinterpret_cast<const float4*>(&S.dz2[gi + 8 * q][s]);
#pragma unroll
                    for (int c = 0; c < 4; c++)
                        t[q][c] = fmaf(a.x, b[c].x, fmaf(a.y, b[c].y, fmaf(a.z, b[c].z, fmaf(a.w, b[c].w, t[q][c]))));
                }
            }
#pragma unroll
            for (int q = 0; q < 8; q++)
#pragma unroll
                for (int c = 0; c < 4; c++) g2[q][c] += t[q][c];
        }
        __syncthreads();  // dz1 written
        sample_sums<NI / 2>(&S.h2[row][0], &S.xs[half * (NI / 2)][0], kLD, g1);
        {
            const float* a = half ? &S.dz2[row][0] : &S.h2[row][0];
            float t = 0.f;
#pragma unroll 4
            for (int s = 0; s < TB; s += 4) {
                const float4 v = *reinterpret_cast<const float4*>(a + s);
                t += (v.x + v.y) + (v.z + v.w);
            }
            if (half)
                gb2 += t;
            else
                gb1 += t;
            if (tid < NO) {
                float u = 0.f;
#pragma unroll 4
                for (int s = 0; s < TB; s += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(&S.dy[tid][s]);
                    u += (v.x + v.y) + (v.z + v.w);
                }
                gb3 += u;
            }
        }
        loss_sum += (double)myloss;
        myloss = 0.f;
        __syncthreads();  // the tile's arrays are free
    }
#pragma unroll
    for (int q = 0; q < 8; q++)
#pragma unroll
        for (int c = 0; c < 4; c++) atomicAdd(&grad[Ly::W2 + (gi + 8 * q) * H + gj + 16 * c], g2[q][c]);
#pragma unroll
    for (int k = 0; k < NI / 2; k++) {
        const int m = half * (NI / 2) + k;
        if (m < NIN) atomicAdd(&grad[Ly::W1 + row * NIN + m], g1[k]);
    }
#pragma unroll
    for (int k = 0; k < NO / 2; k++) {
        const int o = half * (NO / 2) + k;
        if (o < NOUT) atomicAdd(&grad[Ly::W3 + o * H + row], g3[k]);
    }
    atomicAdd(&grad[half ? Ly::B2 + row : Ly::B1 + row], half ? gb2 : gb1);
    if (tid < NOUT) atomicAdd(&grad[Ly::B3 + tid], gb3);
    for (int o = 16; o > 0; o >>= 1) loss_sum += __shfl_xor_sync(0xffffffffu, loss_sum, o);
    if ((tid & 31) == 0) atomicAdd(loss, loss_sum);
}

// Adam on the FP32 master weights; refreshes the BF16 copy and clears the gradient.
__global__ void adam_kernel(float* master, __nv_bfloat16* Wb, float* grad, float* m1, float* m2, int nw, float lr,
                            float b1, float b2, float eps, float bc1, float bc2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += gridDim.x * blockDim.x) {
        const float g = grad[i];
        const float a = b1 * m1[i] + (1.f - b1) * g;
        const float v = b2 * m2[i] + (1.f - b2) * g * g;
        m1[i] = a;
        m2[i] = v;
        const float w = master[i] - lr * (a / bc1) / (sqrtf(v / bc2) + eps);
        master[i] = w;
        Wb[i] = __float2bfloat16(w);
        grad[i] = 0.f;
    }
}

template <int D>
int launch_grad(const __nv_bfloat16* Wb, const float* nrm, const float* X, const float* Y, const long long* idx,
                long long b0, int bsize, float scale, float* grad, double* loss, cudaStream_t s) {
    const size_t sm = sizeof(GradTile<D>);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(mlp_grad_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        return LELBM_E_CUDA;
    const int blocks = std::min((bsize + TB - 1) / TB, 2 * sms);  // two to an SM
    mlp_grad_kernel<D><<<blocks, kGradThreads, sm, s>>>(Wb, nrm, X, Y, idx, b0, bsize, scale, grad, loss);
    return cudaGetLastError() == cudaSuccess ? LELBM_OK : LELBM_E_CUDA;
}

int sizes(int dims, int* nin, int* nout, long long* ntot, long long* nw) {
    if (dims == 1) {
        *nin = MlpDims<1>::NIN;
        *nout = MlpDims<1>::NOUT;
        *ntot = MlpLayout<1>::NTOT;
        *nw = MlpLayout<1>::NW;
    } else if (dims == 2) {
        *nin = MlpDims<2>::NIN;
        *nout = MlpDims<2>::NOUT;
        *ntot = MlpLayout<2>::NTOT;
        *nw = MlpLayout<2>::NW;
    } else {
        return LELBM_E_INVAL;
    }
    return LELBM_OK;
}

}  // namespace
}  // namespace lbm

using namespace lbm;

extern "C" int lelbm_mlp_size(int dims, int* n_in, int* n_out, long long* n_params, long long* n_weights) {
    int a, b;
    long long c, d;
    const int rc = sizes(dims, &a, &b, &c, &d);
    if (rc) return rc;
    if (n_in) *n_in = a;
    if (n_out) *n_out = b;
    if (n_params) *n_params = c;
    if (n_weights) *n_weights = d;
    return LELBM_OK;
}

extern "C" int lelbm_mlp_init(int dims, unsigned long long seed, const float* X, const float* Y, long long n,
                              float* params) {
    int nin, nout;
    long long ntot, nw;
    if (sizes(dims, &nin, &nout, &ntot, &nw) || !params || (n > 0 && (!X || !Y))) return LELBM_E_INVAL;
    std::vector<float> p(ntot, 0.f);
    std::mt19937_64 rng(seed);
    const int H = 64;
    auto fill = [&](int off, int rows, int cols, float gain) {
        const float lim = gain * std::sqrt(6.0f / (float)cols);
        std::uniform_real_distribution<float> U(-lim, lim);
        for (int i = 0; i < rows * cols; i++) p[off + i] = U(rng);
    };
    const int W1 = 0, B1 = W1 + H * nin, W2 = B1 + H, B2 = W2 + H * H, W3 = B2 + H;
    fill(W1, H, nin, 1.0f);
    fill(W2, H, H, 1.0f);
    fill(W3, nout, H, 0.1f);  // small output layer: training starts near the Maxwellian start
    std::vector<double> sx(2 * nin, 0.0), sy(2 * nout, 0.0);
    if (n > 0) {
        double* d = nullptr;
        if (cudaMalloc((void**)&d, sizeof(double) * 2 * (nin + nout)) != cudaSuccess) return LELBM_E_NOMEM;
        cudaMemset(d, 0, sizeof(double) * 2 * (nin + nout));
        column_stats_kernel<<<1024, 256>>>(X, n, nin, d);
        column_stats_kernel<<<1024, 256>>>(Y, n, nout, d + 2 * nin);
        cudaError_t e = cudaMemcpy(sx.data(), d, sizeof(double) * 2 * nin, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(sy.data(), d + 2 * nin, sizeof(double) * 2 * nout, cudaMemcpyDeviceToHost);
        cudaFree(d);
        if (e != cudaSuccess) return LELBM_E_CUDA;
    }
    auto stats = [&](const std::vector<double>& s, int cols, int mo, int so) {
        for (int c = 0; c < cols; c++) {
            const double mean = n > 0 ? s[c] / n : 0.0;
            const double var = n > 0 ? std::max(s[cols + c] / n - mean * mean, 0.0) : 1.0;
            const double sd = std::sqrt(var);
            p[mo + c] = (float)mean;
            p[so + c] = (float)(sd > 1e-6 * std::max(1.0, std::fabs(mean)) ? sd : 1.0);
        }
    };
    stats(sx, nin, (int)nw, (int)nw + nin);
    stats(sy, nout, (int)nw + 2 * nin, (int)nw + 2 * nin + nout);
    std::copy(p.begin(), p.end(), params);
    return LELBM_OK;
}

extern "C" int lelbm_mlp_loss_grad(int dims, const float* params, const float* X, const float* Y, long long n,
                                   float* grad, double* loss, void* stream) {
    int nin, nout;
    long long ntot, nw;
    if (sizes(dims, &nin, &nout, &ntot, &nw) || !params || !X || !Y || !grad || n < 1) return LELBM_E_INVAL;
    if (n > (1LL << 31) - TB) return LELBM_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16* Wb = nullptr;
    double* dl = nullptr;
    if (cudaMalloc((void**)&Wb, sizeof(__nv_bfloat16) * nw) != cudaSuccess) return LELBM_E_NOMEM;
    if (cudaMalloc((void**)&dl, sizeof(double)) != cudaSuccess) {
        cudaFree(Wb);
        return LELBM_E_NOMEM;
    }
    cudaMemsetAsync(dl, 0, sizeof(double), s);
    cudaMemsetAsync(grad, 0, sizeof(float) * nw, s);
    to_bf16_kernel<<<64, 256, 0, s>>>(params, Wb, (int)nw);
    const float scale = 2.0f / (float)((double)n * nout);
    int rc = dims == 1 ? launch_grad<1>(Wb, params + nw, X, Y, nullptr, 0, (int)n, scale, grad, dl, s)
                       : launch_grad<2>(Wb, params + nw, X, Y, nullptr, 0, (int)n, scale, grad, dl, s);
    double h = 0.0;
    if (!rc && cudaMemcpyAsync(&h, dl, sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess) rc = LELBM_E_CUDA;
    if (!rc && cudaStreamSynchronize(s) != cudaSuccess) rc = LELBM_E_CUDA;
    cudaFree(Wb);
    cudaFree(dl);
    if (loss) *loss = h / ((double)n * nout);
    return rc;
}

extern "C" int lelbm_mlp_train(int dims, float* params, const float* X, const float* Y, long long n, int epochs,
                               int batch, float lr, unsigned long long seed, double* epoch_loss, void* stream) {
    int nin, nout;
    long long ntot, nw;
    if (sizes(dims, &nin, &nout, &ntot, &nw) || !params || !X || !Y || n < 1 || epochs < 1 || batch < 1 ||
        batch > (1 << 24) || !(lr > 0.f))
        return LELBM_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16* Wb = nullptr;
    float *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
    long long* idx = nullptr;
    double* dl = nullptr;
    int rc = LELBM_OK;
    if (cudaMalloc((void**)&Wb, sizeof(__nv_bfloat16) * nw) != cudaSuccess ||
        cudaMalloc((void**)&grad, sizeof(float) * nw) != cudaSuccess ||
        cudaMalloc((void**)&m1, sizeof(float) * nw) != cudaSuccess ||
        cudaMalloc((void**)&m2, sizeof(float) * nw) != cudaSuccess ||
        cudaMalloc((void**)&idx, sizeof(long long) * n) != cudaSuccess ||
        cudaMalloc((void**)&dl, sizeof(double) * epochs) != cudaSuccess)
        rc = LELBM_E_NOMEM;
    if (!rc) {
        cudaMemsetAsync(grad, 0, sizeof(float) * nw, s);
        cudaMemsetAsync(m1, 0, sizeof(float) * nw, s);
        cudaMemsetAsync(m2, 0, sizeof(float) * nw, s);
        cudaMemsetAsync(dl, 0, sizeof(double) * epochs, s);
        to_bf16_kernel<<<64, 256, 0, s>>>(params, Wb, (int)nw);
    }
    std::vector<long long> perm(n);
    std::iota(perm.begin(), perm.end(), 0LL);
    std::mt19937_64 rng(seed);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    long long tstep = 0;
    for (int ep = 0; ep < epochs && !rc; ep++) {
        std::shuffle(perm.begin(), perm.end(), rng);
        if (cudaMemcpyAsync(idx, perm.data(), sizeof(long long) * n, cudaMemcpyHostToDevice, s) != cudaSuccess) {
            rc = LELBM_E_CUDA;
            break;
        }
        for (long long b0 = 0; b0 < n && !rc; b0 += batch) {
            const int bs = (int)std::min<long long>(batch, n - b0);
            const float scale = 2.0f / (float)((double)bs * nout);
            rc = dims == 1 ? launch_grad<1>(Wb, params + nw, X, Y, idx, b0, bs, scale, grad, dl + ep, s)
                           : launch_grad<2>(Wb, params + nw, X, Y, idx, b0, bs, scale, grad, dl + ep, s);
            tstep++;
            const float bc1 = 1.f - std::pow(b1, (float)tstep), bc2 = 1.f - std::pow(b2, (float)tstep);
            adam_kernel<<<(int)((nw + 255) / 256), 256, 0, s>>>(params, Wb, grad, m1, m2, (int)nw, lr, b1, b2, eps,
                                                              bc1, bc2);
            if (cudaGetLastError() != cudaSuccess) rc = LELBM_E_CUDA;
        }
        // the host permutation buffer is reused next epoch: wait for this epoch's copy
        if (!rc && cudaStreamSynchronize(s) != cudaSuccess) rc = LELBM_E_CUDA;
    }
    if (!rc && epoch_loss) {
        std::vector<double> h(epochs);
        if (cudaMemcpy(h.data(), dl, sizeof(double) * epochs, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = LELBM_E_CUDA;
        for (int ep = 0; ep < epochs; ep++) epoch_loss[ep] = h[ep] / ((double)n * nout);
    }
    cudaFree(Wb);
    cudaFree(grad);
    cudaFree(m1);
    cudaFree(m2);
    cudaFree(idx);
    cudaFree(dl);
    return rc;
}
