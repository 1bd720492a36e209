// Model-tail operators on bf16 NHWC tensors with padded channels: k x k max-pool, global
// average pool and fully-connected layers.  All are memory-bound; float32 arithmetic.
#include "common.cuh"
#include "plan.h"

namespace cprune {

__global__ void __launch_bounds__(256) maxpool_kernel(const bf16x8 *__restrict__ x, int N, int H, int W, int c8,
                                                      int P, int Q, int k, int stride, int pad,
                                                      bf16x8 *__restrict__ y) {
    pdl_trigger();
    pdl_wait();
    long long total = (long long)N * P * Q * c8;
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    int cg = (int)(e % c8);
    long long t = e / c8;
    int q = (int)(t % Q);
    t /= Q;
    int p = (int)(t % P);
    int n = (int)(t / P);
    float m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = -INFINITY;
    for (int r = 0; r < k; ++r) {
        int h = p * stride - pad + r;
        if (h < 0 || h >= H) continue;
        for (int s = 0; s < k; ++s) {
            int v = q * stride - pad + s;
            if (v < 0 || v >= W) continue;
            float f[8];
            unpack8(ldg8(x + (((size_t)n * H + h) * W + v) * c8 + cg), f);
#pragma unroll
            for (int i = 0; i < 8; ++i) m[i] = fmaxf(m[i], f[i]);
        }
    }
    y[e] = pack8(m);
}

// One block per (image, 32 channel groups): 8 pixel lanes x 32 channel groups; each thread sums every 8th pixel of
// its channel group in float32, the lanes are added through shared memory in a fixed order, mean stored as bf16.  Bound by the
// latency of its loads: eight go out together, all of a 7x7 image (one by one 64 images of 1280 channels took 4.8 us
// in MobileNetV2, now 2.5; 8 x 56x56 x 64 channels by themselves 57 and 33 us).
constexpr int GAP_AHEAD = 8;
__global__ void __launch_bounds__(256) gap_kernel(const bf16x8 *__restrict__ x, int N, int HW, int c8,
                                                  bf16x8 *__restrict__ y) {
    __shared__ float part[8][32][9];
    pdl_trigger();
    pdl_wait();
    const int blocks_per_img = (c8 + 31) / 32;
    const int n = blockIdx.x / blocks_per_img;
    const int cg = (blockIdx.x - n * blocks_per_img) * 32 + (threadIdx.x & 31);
    const int pl = threadIdx.x >> 5;
    float s[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = 0.f;
    if (cg < c8) {
        const bf16x8 *px = x + (size_t)n * HW * c8 + cg;
        for (int i0 = pl; i0 < HW; i0 += 8 * GAP_AHEAD) {
            bf16x8 v[GAP_AHEAD];
#pragma unroll
            for (int i = 0; i < GAP_AHEAD; ++i)
                if (i0 + 8 * i < HW) v[i] = ldg8(px + (size_t)(i0 + 8 * i) * c8);
#pragma unroll
            for (int i = 0; i < GAP_AHEAD; ++i) {
                if (i0 + 8 * i >= HW) break;
                float f[8];
                unpack8(v[i], f);
#pragma unroll
                for (int j = 0; j < 8; ++j) s[j] += f[j];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) part[pl][threadIdx.x & 31][j] = s[j];
    __syncthreads();
    if (pl == 0 && cg < c8) {
        float t[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] = 0.f;
        for (int l = 0; l < 8; ++l)
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] += part[l][threadIdx.x & 31][j];
        const float inv = 1.f / (float)HW;
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] *= inv;
        y[(size_t)n * c8 + cg] = pack8(t);
    }
}

// Fully connected layer.  A block computes 8 * NT output features of 16 images; its eight warps share out the input
// features, 32 at a time, and their sums meet in shared memory in a fixed order.  The work is tiny (a few MFLOP per SM) and
// what it costs is the latency of reading a few megabytes of weights once, so everything is arranged for loads in flight:
// eight output features per block give 125 blocks for 1000 classes and up to 16 images, operands go straight from global memory into MMA
// registers (a thread's 16-byte piece of 8 neighbouring features serves two MMA steps: the order of the contraction index is
// free as long as both operands use the same), and the first pieces of the weights, which no kernel of the chain writes, are
// requested before the preceding kernel has finished.
// The tensor core truncates where it adds to an accumulator, so that a chain of MMAs loses more than float32 additions do.  Two
// MMAs (32 features) start from zero and are added to the running sum with a rounded addition; the eight warps' sums meet in
// float64.  Relative error (2-norm, against 64 bits): 512 features 5.4e-8, 1280 6.5e-8, 4096 9.0e-8, 25088 1.9e-7; as one chain per
// warp 8.7e-8, 1.5e-7, 4.7e-7, 3.3e-6; float32 fused multiply-adds 6.7e-8, 7.7e-8, 9.8e-8, 2.2e-7.
// More images take 16 features per block: the reads of the images' rows, one line per row and 64 bytes, are halved and the sums of a
// block stay few.  (Two tiles of images and 8 features, as it was, read the weights half as often, but a block needed 6.3 us whether its
// grid was one wave or two.)  In the networks, before and now: 1280 -> 1000 at 64 images 6.6 and 3.7 us, at 20 images 6.3 and 3.0 us;
// 512 -> 1000 at 64 images 6.4 and 3.3 us.  By themselves: 25088 -> 4096 at 8 images 119 and 45 us, at 128 images 751 and 297 us.
// (64 images 14.3 us with one warp per 4 features x 8 images on the FMA pipe.)
// Five pieces of 16 features ahead take 116 registers and let two blocks onto an SM, which is what a latency asks for as long as the grid
// fits; a grid of more blocks than that is bound by how many are resident, and goes three pieces ahead with three blocks to an SM (80
// registers): where a warp has no more than three pieces, and up to 4096 features where that saves a round of blocks.  us, two blocks to an SM / three /
// the tiles of 8 features by 32 images that these replaced (in graphs): 64 -> 4096 at 1024 images 88.8 / 55.7 / 69.0, 512 -> 4096 at 1024 images
// 114 / 80 / 104, 4096 -> 1000 at 256 images (three rounds, or four of two blocks) 27.6 / 24.6 / 34.6; with as many rounds 1280 -> 1000 at 128 images
// 7.1 / 7.5 / 9.4; 25088 -> 1000 at 512 images, where a block's own stream of loads counts for more, 227 / 260 / 723.
constexpr int FC_WARPS = 8, FC_AHEAD = 5, FC_AHEAD_MANY = 3, FC_BLOCKS_MANY = 3, FC_FEATURES_MANY = 4096;
constexpr int FC_SMS = 148;

template <int NT, int AHEAD, int BLOCKS>
__global__ void __launch_bounds__(FC_WARPS * 32, BLOCKS) fc_kernel(const bf16x8 *__restrict__ x, int N, int in8,
                                                           const bf16x8 *__restrict__ w, const float *__restrict__ b, int out,
                                                           int out_pad, int act, int out_is_f32, void *__restrict__ y) {
    __shared__ float part[FC_WARPS][16][NT * 8 + 1];
    pdl_trigger();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    constexpr int SHIFT = NT == 1 ? 3 : 4;
    const int tiles_o = (out_pad + NT * 8 - 8) >> SHIFT;
    const int o0 = (blockIdx.x % tiles_o) * (NT * 8), n0 = (int)(blockIdx.x / tiles_o) * 16;
    const bf16x8 zero = {{0u, 0u, 0u, 0u}};
    const bf16x8 *wrow = w + (size_t)(o0 + g) * in8 + t;
    auto load_w = [&](int c, bf16x8 *v) {
#pragma unroll
        for (int f = 0; f < NT; ++f) v[f] = c * 4 + t < in8 && (f == 0 || o0 + f * 8 < out_pad) ? ldg8(wrow + f * 8 * (size_t)in8 + c * 4) : zero;
    };
    bf16x8 wq[AHEAD][NT];
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) load_w(warp + i * FC_WARPS, wq[i]);
    pdl_wait();
    float acc[NT][4];
#pragma unroll
    for (int f = 0; f < NT; ++f)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[f][j] = 0.f;
    const int chunks = (in8 + 3) >> 2;
    for (int c0 = warp; c0 < chunks; c0 += AHEAD * FC_WARPS) {
        bf16x8 xq[AHEAD][2];
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const int q = (c0 + i * FC_WARPS) * 4 + t;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int n = n0 + h * 8 + g;
                xq[i][h] = (n < N && q < in8) ? ldg8(x + (size_t)n * in8 + q) : zero;
            }
        }
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
#pragma unroll
            for (int f = 0; f < NT; ++f) {
                float s[4] = {0.f, 0.f, 0.f, 0.f};
                mma_16816(s, xq[i][0].w[0], xq[i][1].w[0], xq[i][0].w[1], xq[i][1].w[1], wq[i][f].w[0], wq[i][f].w[1]);
                mma_16816(s, xq[i][0].w[2], xq[i][1].w[2], xq[i][0].w[3], xq[i][1].w[3], wq[i][f].w[2], wq[i][f].w[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[f][j] += s[j];
            }
            load_w(c0 + (AHEAD + i) * FC_WARPS, wq[i]);
        }
    }
#pragma unroll
    for (int f = 0; f < NT; ++f)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[warp][(j >> 1) * 8 + g][f * 8 + t * 2 + (j & 1)] = acc[f][j];
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * NT * 8; e += FC_WARPS * 32) {
        const int r = e >> SHIFT, c = e & (NT * 8 - 1), n = n0 + r, o = o0 + c;
        if (n >= N || (NT > 1 && o >= out_pad)) continue;
        double s[FC_WARPS];
#pragma unroll
        for (int q = 0; q < FC_WARPS; ++q) s[q] = part[q][r][c];
#pragma unroll
        for (int h = FC_WARPS / 2; h > 0; h /= 2)
#pragma unroll
            for (int q = 0; q < h; ++q) s[q] += s[q + h];
        const float v = apply_act((float)(s[0] + b[o]), act);
        if (out_is_f32) {
            if (o < out) ((float *)y)[(size_t)n * out + o] = v;
        } else {
            ((__nv_bfloat16 *)y)[(size_t)n * out_pad + o] = __float2bfloat16_rn(o < out ? v : 0.f);
        }
    }
}

cprune_status launch_maxpool(const void *x, int N, int H, int W, int c_pad, int k, int stride, int pad, void *y,
                             cudaStream_t st) {
    int P = (H + 2 * pad - k) / stride + 1, Q = (W + 2 * pad - k) / stride + 1;
    long long total = (long long)N * P * Q * (c_pad / 8);
    if (total == 0) return CPRUNE_OK;
    long long blocks = ceil_div(total, 256);
    if (blocks > 0x7fffffffLL) return CPRUNE_ERR_UNSUPPORTED;
    CPRUNE_CUDA_CHECK(launch_chained(maxpool_kernel, dim3((unsigned)blocks), dim3(256), 0, st, (const bf16x8 *)x, N, H, W, c_pad / 8, P, Q, k,
                                     stride, pad, (bf16x8 *)y));
    return CPRUNE_OK;
}

}  // namespace cprune

using namespace cprune;

extern "C" {

cprune_status cprune_maxpool(const void *x, int N, int H, int W, int C, int k, int stride, int pad, void *y,
                             void *stream) {
    if (!x || !y || N <= 0 || H <= 0 || W <= 0 || C <= 0 || k <= 0 || stride <= 0 || pad < 0 || 2 * pad > k)
        return CPRUNE_ERR_INVALID_ARG;
    if (H + 2 * pad < k || W + 2 * pad < k) return CPRUNE_ERR_INVALID_ARG;
    return launch_maxpool(x, N, H, W, cprune_padded_channels(C), k, stride, pad, y, (cudaStream_t)stream);
}

cprune_status cprune_global_avgpool(const void *x, int N, int H, int W, int C, void *y, void *stream) {
    if (!x || !y || N <= 0 || H <= 0 || W <= 0 || C <= 0) return CPRUNE_ERR_INVALID_ARG;
    int c8 = cprune_padded_channels(C) / 8;
    CPRUNE_CUDA_CHECK(launch_chained(gap_kernel, dim3(N * ((c8 + 31) / 32)), dim3(256), 0, (cudaStream_t)stream, (const bf16x8 *)x, N, H * W, c8,
                                     (bf16x8 *)y));
    return CPRUNE_OK;
}

cprune_status cprune_fc(const void *x, int N, int in, const void *w_packed, const float *b_packed, int out, int act,
                        int out_is_f32, void *y, void *stream) {
    if (!x || !w_packed || !b_packed || !y || N <= 0 || in <= 0 || out <= 0) return CPRUNE_ERR_INVALID_ARG;
    int in8 = cprune_padded_channels(in) / 8, out_pad = cprune_padded_channels(out);
    if ((long long)(out_pad >> 3) * ((N + 15) / 16) > 0x7fffffffLL) return CPRUNE_ERR_UNSUPPORTED;
    // One tile of 8 features per SM as long as there are SMs for them: one image 2.4 us.  Beyond that 16 features: 20 images of 1280
    // features 5.0 us with 8 (252 blocks, two or three to an SM) and 3.0 us with 16 (126 blocks).
    const long long tiles_n = (N + 15) / 16, narrow = (out_pad >> 3) * tiles_n, wide = (out_pad + 15) / 16 * tiles_n;
    const bool saves_a_round = ceil_div(wide, FC_BLOCKS_MANY * FC_SMS) < ceil_div(wide, 2 * FC_SMS);
    const bool many = wide > 2 * FC_SMS && (in <= FC_AHEAD_MANY * FC_WARPS * 32 || (in <= FC_FEATURES_MANY && saves_a_round));
    auto launch = [&](auto kernel, long long blocks) {
        return launch_chained(kernel, dim3((unsigned)blocks), dim3(FC_WARPS * 32), 0, (cudaStream_t)stream, (const bf16x8 *)x, N, in8, (const bf16x8 *)w_packed, b_packed, out,
                              out_pad, act, out_is_f32, y);
    };
    if (narrow <= FC_SMS) CPRUNE_CUDA_CHECK(launch(fc_kernel<1, FC_AHEAD, 0>, narrow));
    else if (many) CPRUNE_CUDA_CHECK(launch(fc_kernel<2, FC_AHEAD_MANY, FC_BLOCKS_MANY>, wide));
    else CPRUNE_CUDA_CHECK(launch(fc_kernel<2, FC_AHEAD, 0>, wide));
    return CPRUNE_OK;
}

}  // extern "C"
