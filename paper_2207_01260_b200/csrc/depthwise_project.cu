// A depthwise task and the 1x1 conv task that reads its result in one kernel (the depthwise and projection layers of an
// inverted-residual block, paper Sec. 4.1): the depthwise result, the widest tensor of the block, never leaves the SM.
//
// The depthwise half is that of depthwise.cu: a tile's input patch comes in with one tiled TMA load, a thread owns CH channels of two
// neighbouring output columns and walks down TR rows, float32 sums, the result rounded to bf16 exactly where the separate task would
// store it.  It goes into shared memory as the row operand of tcgen05.mma (a tile is one or two blocks of 128 pixels, 64 channels to a
// 128-byte row, 128-byte swizzle); the filters of the 1x1 task are the column operand, and the accumulator stays in tensor memory while the tile
// goes through its channels, a chunk at a time.  Then the same warps add bias and residual, clamp and store.
//
// What bounds it: the depthwise half, as in depthwise.cu, with the R - 1 rows that a tile of at most 256 pixels reads twice (C 32, 112x112, batch 64: 37.3 us,
// 33.2 without the epilogue, 37.9 without the stores of the row operand); with few tiles, its latency.  In the network (us, two kernels / one):
// batch 64 C 32 -> 16 112x112 41.5 / 35.3, C 108 -> 24 56x56 37.7 / 31.6, C 288 -> 64 14x14 13.0 / 8.9; batch 1 C 32 -> 16 112x112 8.2 / 4.7.
// Taps kept in shared memory for tiles of several chunks cost 1 to 2 us, and diagonal filter matrices on the tensor core instead of the
// CUDA cores 26 us where depthwise.cu takes 25 (C 108, 56x56, batch 64).
//
//   last warp   patch and filter loads, MMA issue;   all others   depthwise half and epilogue.
#include <cuda.h>

#include <cstring>
#include <mutex>

#include "common.cuh"
#include "depthwise_rows.cuh"
#include "plan.h"
#include "sm100_ptx.cuh"

namespace cprune {

constexpr int DP_MAX_THREADS = 480;        // of the depthwise half
constexpr int DP_CTRL = 128;

struct DpParams {
    const uint32_t *w;     // taps, bf16 pairs [R][R][c2]
    const float *b, *b2;
    const __nv_bfloat16 *res;
    __nv_bfloat16 *y;
    int P, Q, pad, c2;     // c2: words (channel pairs) per pixel
    int G, chunks, lanes;  // channel groups (of 8) per chunk, chunks, threads per strip
    int strips, segs, TR, TH, TW, IH, IW;
    int tiles_h, tiles_w, tiles;
    int dn, dth, dtw;      // the grid's size as images, tile rows, tile columns
    int patch_bytes, panels, panel_bytes, w_bytes;      // panels of 64 channels per chunk; filters of one panel
    int MT;                // 128-pixel blocks of a tile
    int k16, k_part, k_pad2, act2, tmem_cols;              // k_part: columns of an MMA (at most 256)
    int *status;
};

// eight float32 values -> bf16, clamped; the clamps return the operand that is a number (see the patch kernel)
__device__ __forceinline__ bf16x8 dp_pack8(const float *v, uint32_t lo, uint32_t hi) {
    bf16x8 r;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.w[j]) : "f"(v[2 * j + 1]), "f"(v[2 * j]));
        asm("max.bf16x2 %0, %0, %1;" : "+r"(r.w[j]) : "r"(lo));
        asm("min.bf16x2 %0, %0, %1;" : "+r"(r.w[j]) : "r"(hi));
    }
    return r;
}

template <int R, int CH, int ACT>
__global__ void __launch_bounds__(DP_MAX_THREADS + 32, 1)
depthwise_project_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w, const DpParams p) {
    constexpr int COLS = 2, NW = CH / 2;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw);
    const uint32_t a_bytes = (uint32_t)p.panels * (uint32_t)p.panel_bytes;
    const uint32_t w0 = base + a_bytes;
    const uint32_t w_chunk = (uint32_t)(p.panels * p.w_bytes);
    const uint32_t patch0 = w0 + (uint32_t)p.chunks * w_chunk;
    const uint32_t ctrl0 = patch0 + 2u * (uint32_t)p.patch_bytes;
    uint8_t *ctrl = smem + (ctrl0 - base);
    auto pfull = [&](int s) { return ctrl0 + 8u * s; };
    auto wfull = [&](int s) { return ctrl0 + 16u + 8u * s; };           // the filters of a chunk: at most two, and they stay
    const uint32_t afull = ctrl0 + 32u, adone = ctrl0 + 40u;
    uint32_t *tmem_slot = (uint32_t *)(ctrl + 48);
    volatile int *abort_flag = (volatile int *)(ctrl + 52);
    float *bias2_s = (float *)(ctrl + DP_CTRL);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int warps = (int)(blockDim.x >> 5) - 1;          // of the depthwise half
    if (warp == warps) {
        tmem_alloc(smem_u32(tmem_slot), (uint32_t)p.tmem_cols);
        tmem_relinquish();
        pdl_trigger();
        if (lane == 0) {
            mbar_init(pfull(0), 1); mbar_init(pfull(1), 1);
            for (int s = 0; s < p.chunks; ++s) mbar_init(wfull(s), 1);
            mbar_init(afull, warps);
            mbar_init(adone, 1);
            *abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    } else {
        // channels that fill up the last 16 have to be numbers: zeros
        if (p.G & 1)
            for (uint32_t e = threadIdx.x; e < a_bytes / 16u; e += (uint32_t)warps * 32u) ((uint4 *)smem)[e] = make_uint4(0u, 0u, 0u, 0u);
        for (int e = threadIdx.x; e < p.k16; e += warps * 32) bias2_s[e] = e < p.k_pad2 ? __ldg(p.b2 + e) : 0.f;
    }
    int n, th, tw;
    {
        const int r = blockIdx.x / p.tiles_w;
        tw = blockIdx.x - r * p.tiles_w;
        n = r / p.tiles_h;
        th = r - n * p.tiles_h;
    }
    auto advance = [&](int &n_, int &th_, int &tw_) {
        tw_ += p.dtw;
        if (tw_ >= p.tiles_w) { tw_ -= p.tiles_w; ++th_; }
        th_ += p.dth;
        if (th_ >= p.tiles_h) { th_ -= p.tiles_h; ++n_; }
        n_ += p.dn;
    };
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int my_tiles = (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, steps = my_tiles * p.chunks;
    bool ok = true;

    if (warp == warps) {
        // ------------------------------------------------------------------ loads and MMAs
        int lchunk = 0;                                    // next patch to load
        auto load_patch = [&](int buf) {
            if (elect_one()) {
                mbar_expect_tx(pfull(buf), (uint32_t)(p.IH * p.IW * p.G * 16));
                tma_load_4d(patch0 + (uint32_t)(buf * p.patch_bytes), &tm_x, pfull(buf), lchunk * p.G * 8, tw * p.TW - p.pad, th * p.TH - p.pad, n);
            }
            __syncwarp();
            if (++lchunk == p.chunks) { lchunk = 0; advance(n, th, tw); }
        };
        for (int s = 0; s < p.chunks && s < steps; ++s) {
            if (elect_one()) {
                mbar_expect_tx(wfull(s), (uint32_t)(p.panels * p.k16) * 128u);
                for (int q = 0; q < p.panels; ++q)
                    for (int k = 0; k < p.k16; k += p.k_part)
                        tma_load_2d(w0 + (uint32_t)s * w_chunk + (uint32_t)(q * p.w_bytes + k * 128), &tm_w, wfull(s), s * p.G * 8 + q * 64, k);
            }
            __syncwarp();
        }
        pdl_wait();
        load_patch(0);
        if (steps > 1) load_patch(1);
        const int ksteps_last = (((p.c2 + 3) >> 2) - (p.chunks - 1) * p.G + 1) >> 1;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.k_part >> 3) << 17) | (8u << 24);
        int chunk = 0;
        for (int i = 0; i < steps && ok; ++i) {
            ok = __all_sync(0xffffffffu, mbar_wait(wfull(chunk), 0u, abort_flag, p.status));
            ok = ok && __all_sync(0xffffffffu, mbar_wait(afull, (uint32_t)(i & 1), abort_flag, p.status));
            if (!ok) break;
            tc_fence_after();
            if (i + 2 < steps) load_patch(i & 1);          // (its last patch has been read)
            const uint32_t a_lo = desc_lo(base), b_lo = desc_lo(w0 + (uint32_t)chunk * w_chunk);
            if (elect_one()) {
                const int ksteps = chunk + 1 == p.chunks ? ksteps_last : p.G >> 1;
                for (int k = 0; k < ksteps; ++k) {
                    const uint32_t a = a_lo + (uint32_t)((k >> 2) * (p.panel_bytes >> 4) + (k & 3) * 2), b = b_lo + (uint32_t)((k >> 2) * (p.w_bytes >> 4) + (k & 3) * 2);
                    for (int mb = 0; mb < p.MT; ++mb)
                        for (int f = 0; f < p.k16; f += p.k_part)
                            umma_bf16_words(tmem_base + (uint32_t)(mb * p.k16 + f), a + (uint32_t)mb * 1024u, b + (uint32_t)f * 8u, DESC_HI_SW128, idesc, (chunk | k) ? 1u : 0u);
                }
                umma_commit(adone);
            }
            __syncwarp();
            if (++chunk == p.chunks) chunk = 0;
        }
    } else {
        // ------------------------------------------------------------------ depthwise half and epilogue
        const int sc = threadIdx.x / p.lanes, cq = threadIdx.x - sc * p.lanes;
        const int seg = sc / p.strips, strip = sc - seg * p.strips;
        const uint32_t pix = (uint32_t)p.G * 4u, row_words = (uint32_t)p.IW * pix;
        const uint32_t in0 = (uint32_t)(seg * p.TR) * row_words + (uint32_t)(strip * COLS) * pix + (uint32_t)(cq * NW);
        // where this thread's results go: pixel (row) and channels (16-byte piece of a 128-byte row, words in it)
        const int ch0 = cq * CH, px0 = seg * p.TR * p.TW + strip * COLS;
        uint8_t *const a_dst = smem + (ch0 >> 6) * p.panel_bytes + (ch0 & 7) * 2;
        const int piece = (ch0 >> 3) & 7;
        const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f), six2 = __floats2bfloat162_rn(6.f, 6.f);
        const uint32_t lo2 = p.act2 == CPRUNE_ACT_NONE ? 0x7fff7fffu : 0u, hi2 = p.act2 == CPRUNE_ACT_RELU6 ? 0x40C040C0u : 0x7fff7fffu;
        // (more than 256 filters: the accumulator's two halves hold up to 16 columns more than a stored pixel has channels)
        const int quarter = warp & 3, of_quarter = (warps - quarter + 3) >> 2, block_units = (p.k_pad2 + 15) >> 4, units = block_units * p.MT;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int erow0 = (quarter * 32 + lane) / p.TW, ecol0 = quarter * 32 + lane - erow0 * p.TW;      // this lane's pixel in either block
        const int erow1 = (128 + quarter * 32 + lane) / p.TW, ecol1 = 128 + quarter * 32 + lane - erow1 * p.TW;
        unsigned long long wf[R][R][NW], bf[NW];
        int chunk = 0;
        bool waited = false;
        for (int i = 0; i < steps; ++i) {
            const int word = chunk * p.G * 4 + cq * NW;
            // (the channels that fill up the last 16 have zero taps and pixels)
            const bool work = seg < p.segs && word < ((p.c2 + 7) & ~7), real = word < p.c2;
            if (work && (i == 0 || p.chunks > 1)) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int s = 0; s < R; ++s) {
                        uint32_t t[NW];
                        if (real) load_words<NW>(p.w + (r * R + s) * p.c2 + word, t);
                        else
#pragma unroll
                            for (int k = 0; k < NW; ++k) t[k] = 0u;
#pragma unroll
                        for (int k = 0; k < NW; ++k) wf[r][s][k] = widen2(t[k]);
                    }
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    const float lo = real ? __ldg(p.b + 2 * (word + k)) : 0.f, hi = real ? __ldg(p.b + 2 * (word + k) + 1) : 0.f;      // (any float32 address)
                    asm("mov.b64 %0, {%1, %2};" : "=l"(bf[k]) : "f"(lo), "f"(hi));
                }
            }
            ok = mbar_wait(pfull(i & 1), (uint32_t)(i >> 1) & 1u, abort_flag, p.status);
            if (i > 0) ok = ok && mbar_wait(adone, (uint32_t)(i - 1) & 1u, abort_flag, p.status);        // the row operand has been read
            const int ps = th * p.TH + seg * p.TR, qs = tw * p.TW + strip * COLS;
            const int rows = min(p.TR, p.P - ps);
            if (ok && work && rows > 0 && qs < p.Q) {
                const uint32_t *in = reinterpret_cast<const uint32_t *>(smem + (patch0 - base) + (i & 1) * p.patch_bytes) + in0;
                int px = px0;
                depthwise_rows<R, 1, CH, COLS>(
                    in, pix, row_words, rows, wf, bf,
                    [&](int c, const unsigned long long (&sum)[NW]) {
                        uint32_t o[NW];
#pragma unroll
                        for (int q = 0; q < NW; ++q) {
                            const float2 f = split2(sum[q]);
                            // 0 and 6 are bf16 values, so the clamp commutes with the rounding
                            __nv_bfloat162 v = __floats2bfloat162_rn(f.x, f.y);
                            if (ACT != CPRUNE_ACT_NONE) v = __hmax2(v, zero2);
                            if (ACT == CPRUNE_ACT_RELU6) v = __hmin2(v, six2);
                            o[q] = *reinterpret_cast<const uint32_t *>(&v);
                        }
                        uint8_t *d = a_dst + sub_off(px + c, piece);
                        if constexpr (NW == 2) *reinterpret_cast<uint2 *>(d) = make_uint2(o[0], o[1]);
                        else *reinterpret_cast<uint32_t *>(d) = o[0];
                    },
                    [&]() { px += p.TW; });
            }
            fence_async_smem();                            // the tensor core reads what was written here
            tc_fence_before();                             // (and overwrites the accumulator that the last epilogue read)
            ok = __all_sync(0xffffffffu, ok);
            if (lane == 0) mbar_arrive(afull);
            if (!ok) break;
            if (++chunk < p.chunks) continue;
            chunk = 0;
            // ---------------------------------------------------------------- epilogue of the tile
            // a unit: 16 filters of a pixel block; a lane has one pixel
            size_t o0 = 0;
            bool pixel = false;
            uint32_t column = 0;
            bf16x8 rv[2] = {};
            auto locate = [&](int u, int &c) {
                const bool second = u >= block_units;
                const int erow = second ? erow1 : erow0, ph = th * p.TH + erow, pw = tw * p.TW + (second ? ecol1 : ecol0);
                c = (u - (second ? block_units : 0)) * 16;
                column = (uint32_t)(c + (second ? p.k16 : 0));
                pixel = erow < p.TH && ph < p.P && pw < p.Q;
                o0 = (((size_t)n * p.P + ph) * p.Q + pw) * p.k_pad2 + c;
                if (p.res && pixel) {
                    rv[0] = ldg8(reinterpret_cast<const bf16x8 *>(p.res + o0));
                    if (c + 8 < p.k_pad2) rv[1] = ldg8(reinterpret_cast<const bf16x8 *>(p.res + o0 + 8));
                }
            };
            int u = warp >> 2, c = 0;
            if (p.res && !waited) { pdl_wait(); waited = true; }       // the residual is the result of an earlier kernel of the chain
            if (u < units) locate(u, c);
            ok = __all_sync(0xffffffffu, mbar_wait(adone, (uint32_t)i & 1u, abort_flag, p.status));
            if (!ok) break;
            tc_fence_after();
            while (u < units) {
                uint32_t v[16];
                tmem_ld16(t_lane + column, v);
                float f[16];
                const float4 *src = reinterpret_cast<const float4 *>(bias2_s + c);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 bb = src[j];
                    f[4 * j] = __uint_as_float(v[4 * j]) + bb.x; f[4 * j + 1] = __uint_as_float(v[4 * j + 1]) + bb.y;
                    f[4 * j + 2] = __uint_as_float(v[4 * j + 2]) + bb.z; f[4 * j + 3] = __uint_as_float(v[4 * j + 3]) + bb.w;
                }
                if (p.res) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            f[8 * h + 2 * j] += __uint_as_float(rv[h].w[j] << 16);
                            f[8 * h + 2 * j + 1] += __uint_as_float(rv[h].w[j] & 0xffff0000u);
                        }
                }
                if (pixel) {
                    *reinterpret_cast<bf16x8 *>(p.y + o0) = dp_pack8(f, lo2, hi2);
                    if (c + 8 < p.k_pad2) *reinterpret_cast<bf16x8 *>(p.y + o0 + 8) = dp_pack8(f + 8, lo2, hi2);
                }
                u += of_quarter;
                if (u < units) locate(u, c);
            }
            advance(n, th, tw);
        }
    }

    // ---------------------------------------------------------------------- teardown
    __syncwarp();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land before the memory goes away
    }
    tc_fence_before();
    __syncthreads();
    if (warp == warps) {
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------ host

// Chooses the tile, the chunk of channels and the block size, and whether the two tasks run as one kernel at all.  The model of a tile's time
// is that of plan_depthwise with a step for the meeting of the warps and a chunk's taps; over 120 shapes (batch 1 to 64, 160 tilings each) what it picks
// is 4 to 8 % off the best.
// Where the line lies (255 pairs of MobileNetV2 and MnasNet, batch 1 to 64, 40 to 80 % of the filters kept, time in the network as two
// kernels less as one): all channels at once on 60 blocks or more -1.3 to 7.8 us, 2.7 on average; two chunks on 120 blocks or more -1.6 to 5.3, 1.8 on
// average; fewer blocks, or three chunks and more, which a block goes through one after the other, -12 to 3.5, -4 on average.  Stride 2, whose
// patches are four times the tile and leave room for one block to an SM, -3.7 to 3.7, 0 on average: not built.
bool plan_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, DwProjTiling *out) {
    const cprune_plan_info &i = dw->info, &q = proj->info;
    *out = DwProjTiling();
    if (i.groups == 1 || dw->opts.residual || dw->opts.pool || i.R != i.S || (i.R != 3 && i.R != 5) || i.stride != 1) return false;
    if (q.groups != 1 || q.R != 1 || q.S != 1 || q.stride != 1 || q.pad != 0 || proj->opts.pool || q.kernel != CPRUNE_KERNEL_TENSOR) return false;
    if (proj->narrow || proj->small_c || q.N != i.N || q.C != i.K || q.H != i.P || q.W != i.Q) return false;
    DwProjTiling t = {};
    t.k_part = q.K <= 256 ? round_up(q.K, 16) : round_up((q.K + 1) / 2, 16);
    t.k16 = q.K <= 256 ? t.k_part : 2 * t.k_part;
    if (t.k16 > 512) return false;
    t.w_bytes = round_up(t.k16 * 128, 1024);
    const int ch = i.R == 3 ? 4 : 2, cols = 2, c8 = i.c_pad / 8, all_strips = (i.Q + cols - 1) / cols;
    const double step_cycles = 0.37 * i.R * i.R + 34.3;
    double best = 1e30;
    for (t.MT = 1; t.MT <= 2; ++t.MT)
        for (t.chunks = 1; t.chunks <= 3; ++t.chunks) {     // (three, which are not run, only to see whether two are the better choice)
            t.G = (c8 + t.chunks - 1) / t.chunks;
            if (t.chunks > 1) t.G = (t.G + 1) & ~1;        // chunks begin at multiples of 16 channels
            if (t.chunks > 1 && (t.chunks - 1) * t.G >= c8) continue;
            for (t.tmem_cols = 32; t.tmem_cols < t.MT * t.k16;) t.tmem_cols *= 2;
            if (t.G > 32 || t.tmem_cols > 512) continue;   // (a box has at most 256 channels)
            t.lanes = t.G * 8 / ch;
            t.panels = (t.G + 7) / 8;
            t.panel_bytes = t.MT * 16384;
            for (t.strips = 1; t.strips <= all_strips && t.strips * t.lanes <= DP_MAX_THREADS; ++t.strips) {
                t.TW = t.strips * cols;
                if (t.TW > 128 * t.MT) break;
                t.tiles_w = (i.Q + t.TW - 1) / t.TW;
                if (t.strips > 1 && t.tiles_w == (i.Q + t.TW - cols - 1) / (t.TW - cols)) continue;      // narrower tiles, as many of them
                t.IW = t.TW - 1 + i.R;
                if (t.IW > 256) break;
                for (t.TR = 1; t.TR <= i.P && t.TR * t.TW <= 128 * t.MT; ++t.TR)
                    for (t.segs = 1; t.segs * t.strips * t.lanes <= DP_MAX_THREADS && t.segs * t.TR * t.TW <= 128 * t.MT; ++t.segs) {
                        if (t.segs > 1 && (t.segs - 1) * t.TR >= i.P) break;
                        t.TH = t.segs * t.TR;
                        if (t.MT == 2 && t.TH * t.TW <= 128) continue;
                        t.IH = t.TH - 1 + i.R;
                        if (t.IH > 256) break;
                        t.patch_bytes = round_up(t.IH * t.IW * t.G * 16, 128);
                        t.tiles_h = (i.P + t.TH - 1) / t.TH;
                        const long long tiles = (long long)i.N * t.tiles_w * t.tiles_h;
                        if (tiles > 0x3fffffffLL / t.chunks) continue;
                        int warps = (t.lanes * t.strips * t.segs + 31) / 32;
                        if (warps < 4) warps = 4;          // (the four quarters of the accumulator's lanes)
                        t.smem_bytes = 1024 + t.panels * (t.panel_bytes + t.chunks * t.w_bytes) + 2 * t.patch_bytes + DP_CTRL + t.k16 * 4;
                        // (three chunks, which are not run, are compared as if two of them could be kept)
                        if (t.chunks == 3 && t.smem_bytes > 227 * 1024) t.smem_bytes -= t.panels * t.w_bytes;
                        if (t.smem_bytes > 227 * 1024) continue;
                        int resident = 227 * 1024 / (t.smem_bytes + 1024);
                        if (resident > 16 / (warps + 1)) resident = 16 / (warps + 1);                // by registers
                        if (resident > 512 / t.tmem_cols) resident = 512 / t.tmem_cols;
                        if (resident < 1) resident = 1;
                        long long ctas = 148LL * resident;
                        if (ctas > tiles) ctas = tiles;
                        const double on_sm = (double)ceil_div(ctas, 148), active = on_sm * warps;
                        const double share = (double)ceil_div(tiles, ctas) * on_sm * 0.78 + (double)tiles / 148.0 * 0.22;
                        const double hide = active < 12.0 ? 12.0 / active : 1.0;
                        const double work = share * t.chunks * warps * (t.TR + i.R + 1.0 + (t.chunks > 1 ? 1.0 : 0.0)) * step_cycles * hide;
                        const double load = share * t.chunks * t.patch_bytes / 50.0;
                        const double tail = share / on_sm * (600.0 + t.chunks * 300.0 + t.k16 * 8.0) * (on_sm > 1 ? 0.6 : 1.0);
                        const double total = (work > load ? work + 0.3 * load : load + 0.3 * work) + tail + active * 200.0;
                        if (total < best) {
                            best = total;
                            *out = t;
                            out->tiles = (int)tiles;
                            out->ctas = (int)ctas;
                            out->threads = (warps + 1) * 32;
                        }
                    }
            }
        }
    out->ok = best < 1e30 && (out->chunks == 1 ? out->ctas >= 60 : out->chunks == 2 && out->ctas >= 120);
    return out->ok != 0;
}

template <int R, int CH, int ACT>
static cprune_status launch_dp(const CUtensorMap *tm, const DpParams &p, const DwProjTiling &t, cudaStream_t st) {
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};    // the shared-memory limit of a kernel is a per-device attribute
    {
        int dev = 0;
        CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(depthwise_project_kernel<R, CH, ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            attr_set[dev] = true;
        }
    }
    CPRUNE_CUDA_CHECK(launch_chained(depthwise_project_kernel<R, CH, ACT>, dim3((unsigned)t.ctas), dim3((unsigned)t.threads), (size_t)t.smem_bytes, st, tm[0], tm[1], p));
    return CPRUNE_OK;
}
template <int R, int CH>
static cprune_status launch_dp_act(int act, const CUtensorMap *tm, const DpParams &p, const DwProjTiling &t, cudaStream_t st) {
    if (act == CPRUNE_ACT_NONE) return launch_dp<R, CH, CPRUNE_ACT_NONE>(tm, p, t, st);
    if (act == CPRUNE_ACT_RELU) return launch_dp<R, CH, CPRUNE_ACT_RELU>(tm, p, t, st);
    return launch_dp<R, CH, CPRUNE_ACT_RELU6>(tm, p, t, st);
}

cprune_status encode_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, const DwProjTiling &t, const void *x, const void *w2, CUtensorMap *tm) {
    const cprune_plan_info &i = dw->info;
    {
        const unsigned long long dims[4] = {(unsigned long long)i.c_pad, (unsigned long long)i.W, (unsigned long long)i.H, (unsigned long long)i.N};
        const unsigned long long strides[3] = {(unsigned long long)i.c_pad * 2, (unsigned long long)i.W * i.c_pad * 2, (unsigned long long)i.H * i.W * i.c_pad * 2};
        const unsigned box[4] = {(unsigned)(t.G * 8), (unsigned)t.IW, (unsigned)t.IH, 1};
        cprune_status s = encode_tiled_bf16(&tm[0], x, 4, dims, strides, box);
        if (s != CPRUNE_OK) return s;
    }
    {
        const unsigned long long dims[2] = {(unsigned long long)i.c_pad, (unsigned long long)proj->info.k_alloc};
        const unsigned long long strides[1] = {(unsigned long long)i.c_pad * 2};
        const unsigned box[2] = {64, (unsigned)t.k_part};
        cprune_status s = encode_tiled_bf16_swz(&tm[1], w2, 2, dims, strides, box, 128, true);
        if (s != CPRUNE_OK) return s;
    }
    return CPRUNE_OK;
}

cprune_status launch_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, const DwProjTiling &t, const CUtensorMap *tm, const void *w, const float *b,
                                       const float *b2, const void *res, void *y, cudaStream_t st) {
    const cprune_plan_info &i = dw->info;
    DpParams p;
    p.w = (const uint32_t *)w;
    p.b = b; p.b2 = b2;
    p.res = (const __nv_bfloat16 *)res;
    p.y = (__nv_bfloat16 *)y;
    p.P = i.P; p.Q = i.Q; p.pad = i.pad; p.c2 = i.c_pad / 2;
    p.G = t.G; p.chunks = t.chunks; p.lanes = t.lanes;
    p.strips = t.strips; p.segs = t.segs; p.TR = t.TR; p.TH = t.TH; p.TW = t.TW; p.IH = t.IH; p.IW = t.IW;
    p.tiles_h = t.tiles_h; p.tiles_w = t.tiles_w; p.tiles = t.tiles;
    p.dn = t.ctas / (t.tiles_h * t.tiles_w);
    p.dth = (t.ctas - p.dn * t.tiles_h * t.tiles_w) / t.tiles_w;
    p.dtw = t.ctas - (p.dn * t.tiles_h + p.dth) * t.tiles_w;
    p.MT = t.MT;
    p.patch_bytes = t.patch_bytes; p.panels = t.panels; p.panel_bytes = t.panel_bytes; p.w_bytes = t.w_bytes;
    p.k16 = t.k16; p.k_part = t.k_part; p.k_pad2 = proj->info.k_pad; p.act2 = proj->opts.activation; p.tmem_cols = t.tmem_cols;
    p.status = device_status_word();
    if (!p.status) return cuda_fail(cudaGetLastError(), "status word");
    const int act = dw->opts.activation;
    return i.R == 3 ? launch_dp_act<3, 4>(act, tm, p, t, st) : launch_dp_act<5, 2>(act, tm, p, t, st);
}

}  // namespace cprune
