// Learned level below level 0 (not in the paper): feature projection of the
// level-0 noise, a direct sampler of the features' exact law, and the
// kernels that train and run a 64-256-256-256-1 ReLU perceptron with BF16
// tensor-core GEMMs (dk_umma.cu), FP32 accumulation and FP32 master weights.
//
// Features.  With e_j the 32 lowest real orthonormal grid modes (cosine and
// sine per wave vector k, ordered by |k|^2) and g_j the per-step factor of the
// noise-free scheme on e_j, a level-0 sample's features are
//     F_(j,r) = sum_m g_j^(M-1-m) <Z^m_(.,r), e_j>,   r = 1, 2,
// i.e. the noise that the heat semigroup carries to time T on each low mode.
// For i.i.d. standard normals they are independent N(0, sum_i g_j^(2i)); the
// network sees F / sigma, so the level below 0 draws its inputs as plain
// standard normals, the exact law of the features of the coupled correction
// level, which keeps the telescoping sum unbiased whatever the network.
#include <cuda_bf16.h>

#include <cstdint>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace dk {

namespace {
constexpr unsigned kFullMask = 0xffffffffu;
}

// ------------------------------------------------------------------ features
// One CTA of 128 threads per sample (grid-stride over samples); thread t
// handles the cell pairs t, t + 128, ...; shared memory holds the mode table.
__global__ void __launch_bounds__(128) feature_kernel(const FeatArgs a) {
    extern __shared__ float fsm[];
    const int cells = a.n * a.n;
    float* E = fsm;                         // [32][cells]
    float* red = fsm + kModes * cells;      // [4][64]
    for (int i = threadIdx.x; i < kModes * cells; i += 128) E[i] = a.E[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long s = blockIdx.x; s < a.count; s += gridDim.x) {
        const long long sid = a.first + s;
        const uint32_t c2 = static_cast<uint32_t>(sid);
        const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);
        float acc[kModes][2];
#pragma unroll
        for (int k = 0; k < kModes; ++k) acc[k][0] = acc[k][1] = 0.f;
        for (int m = 0; m < a.M; ++m) {
#pragma unroll
            for (int k = 0; k < kModes; ++k) {
                acc[k][0] *= a.g[k];
                acc[k][1] *= a.g[k];
            }
            for (int p = threadIdx.x; p < cells / 2; p += 128) {
                const uint4 x = philox10(make_uint4(static_cast<uint32_t>(p), static_cast<uint32_t>(m), c2, c3),
                                         a.key0, a.key1);
                float z1a, z2a, z1b, z2b;
                box_muller(x.x, x.y, z1a, z2a);
                box_muller(x.z, x.w, z1b, z2b);
#pragma unroll
                for (int k = 0; k < kModes; ++k) {
                    const float2 e = *reinterpret_cast<const float2*>(E + k * cells + 2 * p);
                    acc[k][0] = fmaf(e.x, z1a, fmaf(e.y, z1b, acc[k][0]));
                    acc[k][1] = fmaf(e.x, z2a, fmaf(e.y, z2b, acc[k][1]));
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kModes; ++k)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float v = acc[k][r];
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(kFullMask, v, off);
                if (lane == 0) red[warp * kFeat + 2 * k + r] = v;
            }
        __syncthreads();
        if (threadIdx.x < kFeat) {
            const int j = threadIdx.x;
            const float f = (red[j] + red[kFeat + j] + red[2 * kFeat + j] + red[3 * kFeat + j]) * a.inv_sigma[j];
            a.X[s * kFeat + j] = __float2bfloat16_rn(f);
            if (a.Xf) a.Xf[s * kFeat + j] = f;
        }
        __syncthreads();
    }
}

// Direct draw of the standardised features: 64 normals per sample from
// Philox counters (j, 0, id, tag), j = 0..15 giving 4 normals each.
__global__ void direct_feature_kernel(const FeatArgs a) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= a.count * (kFeat / 4)) return;
    const long long s = t / (kFeat / 4);
    const int j = static_cast<int>(t % (kFeat / 4));
    const long long sid = a.first + s;
    const uint32_t c3 = a.tag | ((static_cast<uint32_t>(static_cast<unsigned long long>(sid) >> 32) & 0xffffu) << 16);
    const uint4 x = philox10(make_uint4(static_cast<uint32_t>(j), 0u, static_cast<uint32_t>(sid), c3), a.key0, a.key1);
    float z0, z1, z2, z3;
    box_muller(x.x, x.y, z0, z1);
    box_muller(x.z, x.w, z2, z3);
    __nv_bfloat16* o = a.X + s * kFeat + 4 * j;
    o[0] = __float2bfloat16_rn(z0);
    o[1] = __float2bfloat16_rn(z1);
    o[2] = __float2bfloat16_rn(z2);
    o[3] = __float2bfloat16_rn(z3);
    if (a.Xf) {
        float* of = a.Xf + s * kFeat + 4 * j;
        of[0] = z0; of[1] = z1; of[2] = z2; of[3] = z3;
    }
}

// ------------------------------------------------------------- BF16 GEMM
// The dense layers' GEMMs run on the 5th-generation tensor cores (tcgen05,
// dk_umma.cu); this file holds the output layer (K outputs, too narrow for a
// tensor-core tile), the feature kernels, Adam and the moment kernels.

// -------------------------------------------------------- small MLP kernels
// Output layer forward: y[b][o] = H3[b] . w4[o] + b4[o], o < KO (one warp per row).
__global__ void out_forward_kernel(const __nv_bfloat16* H, const float* w, const float* b, int B, int K, int KO,
                                   float* y) {
    launch_dependents();
    wait_previous_grid();
    const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= B) return;
    for (int o = 0; o < KO; ++o) {
        float s = 0.f;
        for (int k = lane; k < K; k += 32) s = fmaf(__bfloat162float(H[(size_t)row * K + k]), w[(size_t)o * K + k], s);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(kFullMask, s, off);
        if (lane == 0) y[(size_t)row * KO + o] = s + b[o];
    }
}

// Squared error of a batch summed over its n values (rows x outputs) and
// divided by the rows B, FP64 accumulation, one block of 256 threads.
__device__ __forceinline__ void mse_block(const float* y, const float* t, int n, int B, double* out) {
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) {
        const double d = static_cast<double>(y[i]) - t[i];
        s += d * d;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0] / B;
}

__global__ void __launch_bounds__(256) mse_kernel(const float* y, const float* t, int n, int B, double* out) {
    mse_block(y, t, n, B, out);
}

// Sum over the 256 threads of a block of eight values each; valid in threads 0..7
// (value t in thread t).
__device__ __forceinline__ float block_sum8(float (&v)[8]) {
    __shared__ float sh[8][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1)
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] += __shfl_xor_sync(kFullMask, v[i], off);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 8; ++i) sh[warp][i] = v[i];
    __syncthreads();
    float s = 0.f;
    if (threadIdx.x < 8)
        for (int w = 0; w < 8; ++w) s += sh[w][threadIdx.x];
    return s;
}

__device__ __forceinline__ void unpack8(const uint4& u, float (&v)[8]) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(h[i]);
        v[2 * i] = f.x;
        v[2 * i + 1] = f.y;
    }
}

// Backward of the output layer, with d = 2 (y - t) / B, in one launch of blocks
// of 256 threads with four tasks:
//   * dH[b][k] = (sum_o d[b][o] w4[o][k]) (H[b][k] > 0) as BF16, eight columns a thread;
//   * dw[o][k..k+7] = sum_b d[b][o] H[b][k..k+7], one block per o and eight columns;
//   * db[o] = sum_b d[b][o], one block per o;
//   * the loss, if asked for: squared error summed over the B x KO values and
//     divided by B in FP64, one block (the sum of mse_kernel).
// A column's batch sum in one thread is a chain of B additions behind their loads
// on two or three blocks of the GPU; over 256 threads of a block per eight columns
// it is B / 256 loads and a tree (1024 rows: this launch 5.8 us, layer_prep_kernel
// 7 to 9; a gradient 520 us with a thread per column and a launch per task, 187
// with these).
__global__ void __launch_bounds__(256) out_backward_kernel(const float* y, const float* t, const __nv_bfloat16* H,
                                                           const float* w, int B, int K, int KO, __nv_bfloat16* dH,
                                                           float* dw, float* db, double* loss) {
    launch_dependents();
    wait_previous_grid();
    const int tid = threadIdx.x, groups = K / 8;
    const float scale = static_cast<float>(B);
    const int n_el = static_cast<int>(((long long)B * groups + 255) / 256);
    int blk = blockIdx.x;
    if (blk < n_el) {
        const long long i = blk * 256LL + tid;
        if (i >= (long long)B * groups) return;
        const int b = static_cast<int>(i / groups), k = static_cast<int>(i % groups) * 8;
        float h[8], v[8];
        unpack8(*reinterpret_cast<const uint4*>(H + (size_t)b * K + k), h);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = 0.f;
        for (int o = 0; o < KO; ++o) {
            const size_t bo = (size_t)b * KO + o;
            const float d = 2.f * (y[bo] - t[bo]) / scale;
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = fmaf(d, w[(size_t)o * K + k + j], v[j]);
        }
        uint4 u;
        __nv_bfloat162* r = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            r[j] = __floats2bfloat162_rn(h[2 * j] > 0.f ? v[2 * j] : 0.f, h[2 * j + 1] > 0.f ? v[2 * j + 1] : 0.f);
        *reinterpret_cast<uint4*>(dH + (size_t)b * K + k) = u;
        return;
    }
    blk -= n_el;
    if (blk < KO * groups) {
        const int o = blk / groups, k = blk % groups * 8;
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int b = tid; b < B; b += 256) {
            const size_t bo = (size_t)b * KO + o;
            const float d = 2.f * (y[bo] - t[bo]) / scale;
            float h[8];
            unpack8(*reinterpret_cast<const uint4*>(H + (size_t)b * K + k), h);
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j] = fmaf(d, h[j], s[j]);
        }
        const float r = block_sum8(s);
        if (tid < 8) dw[(size_t)o * K + k + tid] = r;
        return;
    }
    blk -= KO * groups;
    if (blk < KO) {
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int b = tid; b < B; b += 256) s[0] += 2.f * (y[(size_t)b * KO + blk] - t[(size_t)b * KO + blk]) / scale;
        const float r = block_sum8(s);
        if (tid == 0) db[blk] = r;
        return;
    }
    mse_block(y, t, B * KO, B, loss);
}

// A layer's operands for the backward products, in one launch of blocks of 256
// threads: transposes (out[c][r] = in[r][c] of an R x C matrix, output rows ldo
// elements apart, one block per 32 x 32 tile) and the bias gradient, the column
// sums of X [B][N] (one block per eight columns).
struct PrepArgs {
    struct Transpose {
        const __nv_bfloat16* in;
        __nv_bfloat16* out;
        int R, C, ldo, tiles;
    } t[3];
    const __nv_bfloat16* X;
    float* colsum;
    int B, N;
};
__global__ void __launch_bounds__(256) layer_prep_kernel(const PrepArgs a) {
    launch_dependents();
    wait_previous_grid();
    __shared__ __nv_bfloat16 sh[32][33];
    int blk = blockIdx.x;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const PrepArgs::Transpose& t = a.t[i];
        if (blk < t.tiles) {
            const int cols = (t.C + 31) / 32, tx = threadIdx.x & 31;
            const int bx = blk % cols * 32, by = blk / cols * 32;
#pragma unroll
            for (int ty = threadIdx.x >> 5; ty < 32; ty += 8) {
                const int r = by + ty, c = bx + tx;
                if (r < t.R && c < t.C) sh[ty][tx] = t.in[(size_t)r * t.C + c];
            }
            __syncthreads();
#pragma unroll
            for (int ty = threadIdx.x >> 5; ty < 32; ty += 8) {
                const int c = bx + ty, r = by + tx;
                if (r < t.R && c < t.C) t.out[(size_t)c * t.ldo + r] = sh[tx][ty];
            }
            return;
        }
        blk -= t.tiles;
    }
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int b = threadIdx.x; b < a.B; b += 256) {
        float v[8];
        unpack8(*reinterpret_cast<const uint4*>(a.X + (size_t)b * a.N + blk * 8), v);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] += v[j];
    }
    const float r = block_sum8(s);
    if (threadIdx.x < 8) a.colsum[blk * 8 + threadIdx.x] = r;
}

// FP32 to BF16, round to nearest even.
__global__ void to_bf16_kernel(const float* x, long long n, __nv_bfloat16* y) {
    launch_dependents();
    wait_previous_grid();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) y[i] = __float2bfloat16_rn(x[i]);
}

// Adam (Kingma & Ba, 2015) with bias correction; refreshes the BF16 weights.
__global__ void adam_kernel(float* theta, const float* grad, float* m1, float* m2, int P, float lr, float b1, float b2,
                            float eps, float c1, float c2, const int* bf_index, __nv_bfloat16* theta_bf) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    const float gi = grad[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float v = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = v;
    const float upd = lr * (a / c1) / (sqrtf(v / c2) + eps);
    const float w = theta[i] - upd;
    theta[i] = w;
    const int j = bf_index[i];
    if (j >= 0) theta_bf[j] = __float2bfloat16_rn(w);
}

__global__ void gather_kernel(const __nv_bfloat16* X, const float* T, const int* idx, int B, int KO,
                              __nv_bfloat16* Xb, float* Tb) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)B * kFeat) return;
    const int b = static_cast<int>(i / kFeat), j = static_cast<int>(i % kFeat);
    const int src = idx[b];
    Xb[i] = X[(size_t)src * kFeat + j];
    if (j < KO) Tb[(size_t)b * KO + j] = T[(size_t)src * KO + j];
}

// Per-sample quantities of a surrogate batch into per-block FP64 partials
// (entry-major [stride][blocks]) in the moment layout of the level kernels,
// quantity by quantity: q = (j, l), j <= l when `products` (else l = j).
// That_k = network output k (sqrt(N)(Y_k - Ybar_k)); S_jl = That_j That_l.
// part = -1: dP = S (level below 0); part = 0: dP = P_0 - S with
// P_0 = N D_j D_l, D the level-0 sample's fluctuations (correction level).
__global__ void __launch_bounds__(256) surrogate_moments_kernel(const float* that, const double* d0, int d0_stride,
                                                                int part, double N, long long count, int stride,
                                                                int KO, int products, double* partials) {
    __shared__ double sh[8][12];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double rsN = 1.0 / sqrt(N);
    int q = 0;
    for (int j = 0; j < KO; ++j) {
        const int lend = products ? KO : j + 1;
        for (int l = j; l < lend; ++l, ++q) {
            double v[12];
#pragma unroll
            for (int e = 0; e < 12; ++e) v[e] = 0.0;
            for (long long i = blockIdx.x * 256LL + threadIdx.x; i < count; i += 256LL * gridDim.x) {
                const double tj = that[i * KO + j], tl = that[i * KO + l];
                const double S = tj * tl;
                const double dj = part == 0 ? d0[i * d0_stride + j] : 0.0;
                const double dl = part == 0 ? d0[i * d0_stride + l] : 0.0;
                const double pf = part == 0 ? N * dj * dl : S;
                const double pc = part == 0 ? S : 0.0;
                const double dp = pf - pc, dp2 = dp * dp;
                v[0] += dp; v[1] += dp2; v[2] += dp2 * dp; v[3] += dp2 * dp2;
                v[4] += pf; v[5] += pf * pf; v[6] += pc; v[7] += pc * pc;
                const double yf = part == 0 ? dj : tj * rsN;
                const double yc = part == 0 ? tj * rsN : 0.0;
                v[8] += yf; v[9] += yf * yf; v[10] += yc; v[11] += yc * yc;
            }
#pragma unroll
            for (int e = 0; e < 12; ++e)
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) v[e] += __shfl_xor_sync(kFullMask, v[e], off);
            if (lane == 0)
#pragma unroll
                for (int e = 0; e < 12; ++e) sh[w][e] = v[e];
            __syncthreads();
            if (threadIdx.x < 12 && 2 + 12 * q + (int)threadIdx.x < stride) {
                double t = 0.0;
                for (int ww = 0; ww < 8; ++ww) t += sh[ww][threadIdx.x];
                partials[(size_t)(2 + 12 * q + threadIdx.x) * gridDim.x + blockIdx.x] = t;
            }
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) {
        // entry 0: samples of this block; entry 1: mass error (none here)
        long long c = 0;
        for (long long i = blockIdx.x * 256LL; i < count; i += 256LL * gridDim.x) c += min(256LL, count - i);
        partials[blockIdx.x] = (double)c;
        partials[(size_t)gridDim.x + blockIdx.x] = 0.0;
    }
}

// ------------------------------------------------------------------ launch
cudaError_t launch_features(const FeatArgs& a, int max_ctas, cudaStream_t st) {
    const size_t smem = sizeof(float) * (kModes * a.n * a.n + 4 * kFeat);
    cudaError_t e = cudaFuncSetAttribute(feature_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<long long>(a.count, max_ctas);
    feature_kernel<<<grid, 128, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_direct_features(const FeatArgs& a, cudaStream_t st) {
    const long long threads = a.count * (kFeat / 4);
    direct_feature_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_out_forward(const __nv_bfloat16* H, const float* w, const float* b, int B, int K, int KO, float* y,
                               cudaStream_t st) {
    return launch_chained(out_forward_kernel, (B + 7) / 8, 256, 0, st, H, w, b, B, K, KO, y);
}

cudaError_t launch_out_backward(const float* y, const float* t, const __nv_bfloat16* H, const float* w, int B, int K,
                                int KO, __nv_bfloat16* dH, float* dw, float* db, double* loss, cudaStream_t st) {
    if (K % 8) return cudaErrorInvalidValue;
    const long long blocks = ((long long)B * (K / 8) + 255) / 256 + KO * (K / 8) + KO + (loss ? 1 : 0);
    return launch_chained(out_backward_kernel, (unsigned)blocks, 256, 0, st, y, t, H, w, B, K, KO, dH, dw, db, loss);
}

cudaError_t launch_layer_prep(const __nv_bfloat16* dH, __nv_bfloat16* dHt, const __nv_bfloat16* Hin, __nv_bfloat16* Hint,
                              int B, int N, int K, int ldt, const __nv_bfloat16* W, __nv_bfloat16* Wt, float* colsum,
                              cudaStream_t st) {
    if (N % 8 || ldt < B) return cudaErrorInvalidValue;
    const auto tiles = [](int R, int C) { return ((R + 31) / 32) * ((C + 31) / 32); };
    PrepArgs a{};
    a.t[0] = {dH, dHt, B, N, ldt, tiles(B, N)};
    a.t[1] = {Hin, Hint, B, K, ldt, tiles(B, K)};
    if (W) a.t[2] = {W, Wt, N, K, N, tiles(N, K)};
    a.X = dH; a.colsum = colsum; a.B = B; a.N = N;
    return launch_chained(layer_prep_kernel, a.t[0].tiles + a.t[1].tiles + a.t[2].tiles + N / 8, 256, 0, st, a);
}

cudaError_t launch_to_bf16(const float* x, long long n, __nv_bfloat16* y, cudaStream_t st) {
    return launch_chained(to_bf16_kernel, (unsigned)((n + 255) / 256), 256, 0, st, x, n, y);
}

cudaError_t launch_adam(float* theta, const float* grad, float* m1, float* m2, int P, float lr, float b1, float b2,
                        float eps, float c1, float c2, const int* bf_index, __nv_bfloat16* theta_bf,
                        cudaStream_t st) {
    adam_kernel<<<(P + 255) / 256, 256, 0, st>>>(theta, grad, m1, m2, P, lr, b1, b2, eps, c1, c2, bf_index, theta_bf);
    return cudaGetLastError();
}

cudaError_t launch_gather(const __nv_bfloat16* X, const float* T, const int* idx, int B, int KO, __nv_bfloat16* Xb,
                          float* Tb, cudaStream_t st) {
    gather_kernel<<<(unsigned)(((long long)B * kFeat + 255) / 256), 256, 0, st>>>(X, T, idx, B, KO, Xb, Tb);
    return cudaGetLastError();
}

cudaError_t launch_mse(const float* y, const float* t, int n, int B, double* out, cudaStream_t st) {
    mse_kernel<<<1, 256, 0, st>>>(y, t, n, B, out);
    return cudaGetLastError();
}

cudaError_t launch_surrogate_moments(const float* that, const double* d0, int d0_stride, int part, double N,
                                     long long count, int stride, int KO, int products, int blocks, double* partials,
                                     cudaStream_t st) {
    surrogate_moments_kernel<<<blocks, 256, 0, st>>>(that, d0, d0_stride, part, N, count, stride, KO, products,
                                                      partials);
    return cudaGetLastError();
}

}  // namespace dk
