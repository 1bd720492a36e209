// Dense conv task of few pixels (small batches, small images): every thread block computes a small tile of the output over
// the WHOLE contraction, so that a task is one launch of many short blocks (paper Sec. 3.4: a task is Conv2d + folded
// BatchNorm + activation; Sec. 3.5: the filter count is whatever pruning left).
//
// Why a third dense kernel: at batch 1 the tcgen05 kernels have a handful of 128-row tiles, so that they either leave most
// SMs idle or split the contraction and need a second kernel, and each pays for tensor-memory allocation, barriers, tensor
// maps and a pipeline fill (4 to 8 us) around a microsecond of work.  What bounds such a task is latency: one round trip for
// the input and one for the filters, on all SMs at once.  Here eight warps form 8 / kw groups; a group covers 16 * MT pixels
// x 8 * NT filters and its kw warps share out the contraction, 32 values (8 channels x 4 threads) at a time; their sums meet
// in shared memory in a fixed order.  Operands go straight from global memory into the registers of warp-level MMAs: a
// thread's 16-byte piece of 8 channels of one tap serves two MMA steps, because the order of the contraction index is free
// as long as both operands use the same.  The first pieces of the filters, which no kernel of the chain writes, are requested
// before the preceding kernel has finished.  A table in shared memory turns a piece number into tap and offset.
#include <cmath>

#include "common.cuh"
#include "plan.h"

namespace cprune {

constexpr int CS_WARPS = 8;
constexpr int CS_MAX_PIECES = 1700;      // 8-channel pieces of a filter (R * S * c_pad / 8): the table shares 48 KB with the sums

struct SmallParams {
    const bf16x8 *x, *w;
    const float *bias;
    const __nv_bfloat16 *res;
    __nv_bfloat16 *y;
    int H, W, P, Q, S, stride, pad;
    int c8, pieces;          // pieces per pixel and per filter
    int M;                   // conv pixels
    int k_pad, tiles_n, act;
    int kw;                  // warps that share a contraction: 1, 2, 4 or 8
};

template <int MT, int NT, bool POOL>
__global__ void __launch_bounds__(CS_WARPS * 32, 2) conv_small_kernel(const SmallParams p) {
    // chunks of the contraction in flight per warp, limited by registers
    constexpr int AHEAD = 2 * MT + NT <= 4 ? 5 : (2 * MT + NT <= 6 ? 3 : 2);
    constexpr int ROWS = MT * 16, COLS = NT * 8;
    extern __shared__ __align__(16) unsigned char cs_smem[];
    __shared__ __align__(8) float part[CS_WARPS][ROWS][COLS + 2];
    __shared__ __align__(8) float bias_s[COLS];
    int2 *table = reinterpret_cast<int2 *>(cs_smem);     // piece -> offset within the image (pieces), tap row << 16 | tap column

    pdl_trigger();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int kw = p.kw, group = warp / kw, kpart = warp - group * kw;
    const int group_rows = CS_WARPS / kw * ROWS;         // rows of the block
    const int mt = blockIdx.x / p.tiles_n, nt = blockIdx.x - mt * p.tiles_n;
    const int b0 = mt * group_rows, m0 = b0 + group * ROWS, o0 = nt * COLS;
    const int chunks = (p.pieces + 3) >> 2;
    const bf16x8 zero = {{0u, 0u, 0u, 0u}};

    // filters: written when the task was packed, not by the preceding kernel
    auto load_w = [&](int c, bf16x8 *v) {
        const int q = c * 4 + t;
#pragma unroll
        for (int n = 0; n < NT; ++n) v[n] = q < p.pieces ? ldg8(p.w + (size_t)(o0 + n * 8 + g) * p.pieces + q) : zero;
    };
    bf16x8 wq[AHEAD][NT];
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) load_w(kpart + i * kw, wq[i]);
    if (tid < COLS) bias_s[tid] = __ldg(p.bias + o0 + tid);

    for (int q = tid; q < chunks * 4; q += CS_WARPS * 32) {
        const int tap = q / p.c8, c = q - tap * p.c8;
        const int r = tap / p.S, s = tap - r * p.S;
        table[q] = q < p.pieces ? make_int2((r * p.W + s) * p.c8 + c, (r << 16) | s) : make_int2(0, 0x7fff0000);
    }
    // the pixels of this thread's fragment rows.  With a pool, rows 4 i .. 4 i + 3 are the window of pooled pixel i.
    auto pixel = [&](int m, int &n, int &ph, int &pw) {
        if (POOL) {
            const int i = m >> 2, hq = p.Q >> 1, per = (p.P >> 1) * hq;
            n = i / per;
            const int rem = i - n * per;
            ph = rem / hq;
            pw = (rem - ph * hq) * 2 + (m & 1);
            ph = ph * 2 + ((m >> 1) & 1);
        } else {
            const int per = p.P * p.Q;
            n = m / per;
            const int rem = m - n * per;
            ph = rem / p.Q;
            pw = rem - ph * p.Q;
        }
    };
    int base[MT][2], hw[MT][2];          // offset of the window's corner (pieces), its row << 16 | column
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = m0 + m * 16 + h * 8 + g;
            int n = 0, ph = 0, pw = 0;
            pixel(min(row, p.M - 1), n, ph, pw);
            const int hh = ph * p.stride - p.pad, ww = pw * p.stride - p.pad;
            base[m][h] = ((n * p.H + hh) * p.W + ww) * p.c8;
            hw[m][h] = (int)(((unsigned)hh << 16) | ((unsigned)ww & 0xffffu));
        }
    float acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[m][n][j] = 0.f;
    __syncthreads();
    pdl_wait();
    // residual of this thread's first output pair: on its way while the sums are formed
    const int pairs = group_rows * (COLS / 2);           // (row, two filters) items of the block; without a pool one output pair each
    auto residual = [&](int e) {
        const int r = e / (COLS / 2), k = o0 + (e - r * (COLS / 2)) * 2;
        return (b0 + r < p.M && k < p.k_pad) ? *reinterpret_cast<const uint32_t *>(p.res + (size_t)(b0 + r) * p.k_pad + k) : 0u;
    };
    uint32_t res0 = 0;
    if (!POOL && p.res && tid < pairs) res0 = residual(tid);
    for (int c0 = kpart; c0 < chunks; c0 += AHEAD * kw) {
        bf16x8 xq[AHEAD][MT][2];
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const int c = c0 + i * kw;
            const int2 e = c < chunks ? table[c * 4 + t] : make_int2(0, 0x7fff0000);
            const int r = e.y >> 16, s = e.y & 0xffff;
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int hh = (hw[m][h] >> 16) + r, ww = (int)(short)(hw[m][h] & 0xffff) + s;
                    xq[i][m][h] = ((unsigned)hh < (unsigned)p.H && (unsigned)ww < (unsigned)p.W) ? ldg8(p.x + (base[m][h] + e.x)) : zero;
                }
        }
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    mma_16816(acc[m][n], xq[i][m][0].w[0], xq[i][m][1].w[0], xq[i][m][0].w[1], xq[i][m][1].w[1], wq[i][n].w[0], wq[i][n].w[1]);
                    mma_16816(acc[m][n], xq[i][m][0].w[2], xq[i][m][1].w[2], xq[i][m][0].w[3], xq[i][m][1].w[3], wq[i][n].w[2], wq[i][n].w[3]);
                }
            if (c0 + AHEAD * kw < chunks) load_w(c0 + (AHEAD + i) * kw, wq[i]);
        }
    }
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2 *>(&part[warp][m * 16 + h * 8 + g][n * 8 + t * 2]) = make_float2(acc[m][n][2 * h], acc[m][n][2 * h + 1]);
    __syncthreads();
    // epilogue, two filters per thread: sums in warp order, bias, residual, activation (then the maximum over a window)
    const int items = POOL ? pairs / 4 : pairs;
    for (int e = tid; e < items; e += CS_WARPS * 32) {
        const int r = e / (COLS / 2), c = (e - r * (COLS / 2)) * 2, k = o0 + c;
        const int m = (POOL ? b0 / 4 : b0) + r;
        if (k >= p.k_pad || m >= (POOL ? p.M / 4 : p.M)) continue;
        float2 best = make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < (POOL ? 4 : 1); ++u) {
            const int row = POOL ? r * 4 + u : r, grp = row / ROWS, lr = row - grp * ROWS;
            float2 v = make_float2(0.f, 0.f);
            for (int q = 0; q < kw; ++q) {
                const float2 a = *reinterpret_cast<const float2 *>(&part[grp * kw + q][lr][c]);
                v.x += a.x; v.y += a.y;
            }
            v.x += bias_s[c]; v.y += bias_s[c + 1];
            if (!POOL && p.res) {
                const uint32_t rv = e == tid ? res0 : residual(e);
                v.x += __uint_as_float(rv << 16);
                v.y += __uint_as_float(rv & 0xffff0000u);
            }
            v.x = apply_act(v.x, p.act); v.y = apply_act(v.y, p.act);
            // (the maximum starts from the window's first value: one with minus infinity would turn a NaN into it)
            best = u == 0 ? v : make_float2(fmaxf(best.x, v.x), fmaxf(best.y, v.y));
        }
        *reinterpret_cast<__nv_bfloat162 *>(p.y + (size_t)m * p.k_pad + k) = __floats2bfloat162_rn(best.x, best.y);
    }
}

struct SmallTile { int mt, nt; };
static const SmallTile kTiles[] = {{1, 1}, {1, 2}, {2, 2}, {2, 4}};

// Called with the plan of the kernel that the task would run on otherwise (its estimate in plan->est_us, a CUDA-core plan
// included); takes the task over when the estimate here is lower.  The estimate counts a launch, the waves of blocks (two to an
// SM) with a round trip to memory per refill of a warp's registers, and the load instructions, whose eight rows occupy the
// L1 for about five cycles each.  Fitted to 1800 timings (30 layers of the pruned networks, batch 1 to 16, every tile and
// split): the time of what it picks is 5 % off the best choice on average.  The other kernels run in 1.1 times their estimates
// (with a split reduction 1.0 to 1.8 times, staged as they lie in memory, variant 2, 0.6 to 0.9 times).
// Where the line lies (us, other kernel / here): 3x3 64 -> 44 56x56 at batch 1 7.3 / 4.2, 2 7.6 / 6.0, 4 6.9 / 8.4;
// 3x3 512 -> 358 7x7 at batch 1 9.8 / 7.1, 4 12.5 / 11.5, 8 13.1 / 15.8; 1x1 720 -> 160 7x7 at batch 1 8.8 / 3.2, 16 9.8 / 5.0;
// 1x1 64 -> 288 14x14 at batch 1 6.2 / 3.1, 8 5.0 / 4.6, 16 5.2 / 5.8.
bool plan_conv_small(cprune_plan *plan, bool other_is_direct) {
    cprune_plan_info &i = plan->info;
    if (i.groups != 1 || plan->opts.pool == CPRUNE_POOL_MAX3X3S2 || plan->opts.flags) return false;
    const bool pool = plan->opts.pool == CPRUNE_POOL_MAX2X2;
    if (pool && plan->opts.residual) return false;
    const long long M = (long long)i.N * i.P * i.Q;
    const int pieces = i.R * i.S * (i.c_pad / 8), chunks = (pieces + 3) / 4;
    if (pieces > CS_MAX_PIECES || i.H > 16000 || i.W > 16000 || i.pad > 16000 || M > 1000000 ||
        (long long)i.N * i.H * i.W * (i.c_pad / 8) > 0x3fffffffLL)
        return false;
    const auto estimate = [&](const SmallTile &s, int k, int filters) {
        const int rows = CS_WARPS / k * 16 * s.mt;
        const double on_sm = (double)(ceil_div(M, rows) * ceil_div(filters, 8 * s.nt)) / 148.0;
        const int ahead = 2 * s.mt + s.nt <= 4 ? 5 : (2 * s.mt + s.nt <= 6 ? 3 : 2);
        const double per_warp = (double)ceil_div(chunks, k), rounds = (double)ceil_div((long long)per_warp, ahead);
        const double latency = ceil(on_sm / 2.0) * (rounds * 1740.0 + chunks * 0.93 + 700.0);
        const double issue = (on_sm > 1.0 ? on_sm : 1.0) * (8.0 * per_warp * (2 * s.mt + s.nt) * 5.1 + rows * 8.0 * s.nt * k * 0.57);
        return 1.66 + (latency + issue) / 1900.0;
    };
    // The split of the contraction fixes the order of its sums.  It is chosen for a typical filter count and not for this
    // task's, so that within this kernel a filter's results do not depend on how many other filters were pruned (2 % slower on
    // average).  Whether the task runs here does depend on its filter count, and the other kernels add in another order.
    int kw = 1;
    double best = 1e30;
    for (const SmallTile &s : kTiles)
        for (int k = 1; k <= CS_WARPS && (k == 1 || k / 2 < chunks); k *= 2)
            if (const double us = estimate(s, k, 96); us < best) { best = us; kw = k; }
    best = 1e30;
    int mt = 0, nt = 0;
    for (const SmallTile &s : kTiles)
        if (const double us = estimate(s, kw, i.k_pad); us < best) { best = us; mt = s.mt; nt = s.nt; }
    const double other = other_is_direct ? i.flops / 15.0e6 + 4.0 : plan->est_us * (plan->patch && plan->pt.dense ? 0.62 : (plan->splits > 1 ? 1.25 : 1.12));
    // the timings behind the estimate had everything in the L2, where small tasks find it: what goes beyond 8 MB at 5 TB/s on top
    // (1x1 144 -> 32 28x28 with a residual, 64 images: 19.4 us here, 10.1 us on the other kernel)
    const double bytes = 2.0 * ((double)i.N * i.H * i.W * i.c_pad + (double)M * i.k_pad * (plan->opts.residual ? 2 : 1) + (double)i.k_pad * pieces * 8);
    if (bytes > 8.0e6) best += (bytes - 8.0e6) / 5.0e6;
    if (best >= other) return false;
    plan->small = 1;
    plan->small_mt = mt; plan->small_nt = nt; plan->small_kw = kw;
    plan->est_us = best;
    plan->patch = 0;
    plan->narrow = 0;
    plan->small_c = 0;
    plan->s_packed = i.S;
    plan->orient = 0;
    plan->splits = 1;
    plan->partial_bytes = 0;
    plan->pre_bytes = 0;
    plan->fused_pool = pool ? 1 : 0;
    plan->bias_align = 4;
    i.tile_m = CS_WARPS / kw * 16 * mt;
    i.tile_n = 8 * nt;
    i.tile_k = 32;
    i.stages = 2;
    i.tiles_m = (int)ceil_div(M, i.tile_m);
    i.tiles_n = (int)ceil_div(i.k_pad, i.tile_n);
    i.k_alloc = i.tiles_n * i.tile_n;
    i.padded_flops = 2.0 * i.tiles_m * i.tile_m * (double)i.k_alloc * chunks * 32.0;
    return true;
}

template <int MT, int NT>
static cprune_status launch_small(const SmallParams &p, unsigned blocks, bool pool, cudaStream_t st) {
    const size_t smem = (size_t)((p.pieces + 3) / 4 * 4) * sizeof(int2);
    if (pool) CPRUNE_CUDA_CHECK(launch_chained(conv_small_kernel<MT, NT, true>, dim3(blocks), dim3(CS_WARPS * 32), smem, st, p));
    else CPRUNE_CUDA_CHECK(launch_chained(conv_small_kernel<MT, NT, false>, dim3(blocks), dim3(CS_WARPS * 32), smem, st, p));
    return CPRUNE_OK;
}

cprune_status launch_conv_small(const cprune_plan *plan, const void *x, const void *w, const float *b, const void *res, void *y, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    SmallParams p;
    p.x = (const bf16x8 *)x;
    p.w = (const bf16x8 *)w;
    p.bias = b;
    p.res = (const __nv_bfloat16 *)res;
    p.y = (__nv_bfloat16 *)y;
    p.H = i.H; p.W = i.W; p.P = i.P; p.Q = i.Q; p.S = i.S; p.stride = i.stride; p.pad = i.pad;
    p.c8 = i.c_pad / 8;
    p.pieces = i.R * i.S * p.c8;
    p.M = i.N * i.P * i.Q;
    p.k_pad = i.k_pad; p.tiles_n = i.tiles_n; p.act = plan->opts.activation;
    p.kw = plan->small_kw;
    const unsigned blocks = (unsigned)((long long)i.tiles_m * i.tiles_n);
    const bool pool = plan->fused_pool != 0;
    if (plan->small_mt == 1 && plan->small_nt == 1) return launch_small<1, 1>(p, blocks, pool, st);
    if (plan->small_mt == 1) return launch_small<1, 2>(p, blocks, pool, st);
    if (plan->small_nt == 2) return launch_small<2, 2>(p, blocks, pool, st);
    return launch_small<2, 4>(p, blocks, pool, st);
}

}  // namespace cprune
