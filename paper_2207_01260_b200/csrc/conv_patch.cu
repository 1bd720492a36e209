// Stride-1 dense conv task (3x3 and other R x S > 1) on the sm_100a tensor cores with the input
// patch kept in shared memory (paper Sec. 3.4: a task is Conv2d + folded BatchNorm + activation;
// Sec. 3.5: the filter count is whatever pruning left).
//
// Why a second tensor-core kernel: the im2col kernel (conv_tc.cu) writes every activation element
// R*S times into shared memory, and on this GPU the shared-memory port (128 bytes per clock: TMA
// writes plus the operand reads of tcgen05.mma) is what bounds it, not the tensor pipe.  Here a
// tile is TH whole output rows of one image.  Its input patch, (TH + R - 1) x (W + 2 pad) pixels x
// 64 channels, is loaded ONCE per channel block by one tiled TMA load (out-of-range pixels and
// channels arrive as zeros, which is the padding).  The patch sits in shared memory as rows of
// 128 bytes, one per pixel, in row-major order of the padded image, 128-byte swizzled.  For filter
// tap (r, s) the pixel operand of the MMA is the same patch read from a start address
// (r * Wp + s) * 128 bytes further on (Wp = W + 2 pad): the swizzle is a function of the
// shared-memory address, so a descriptor may start at any 128-byte row (checked on B200).
//
// The accumulator row of a pixel is its "slot" i * Wp + j (i row in the tile, j column); slots with
// j >= Q are the S - 1 wrap-around columns: they are computed and thrown away.  A tile has MT
// blocks of 128 slots (MT = 1 or 2, one accumulator each, both fed by the same filter stage).  Of images that fit several times
// (4x4, 7x7, 8x8) a tile takes whole ones, with the zero borders shared between rows and between images (us, 7x7 at 64 images
// 512 -> 358 filters 23.9 as im2col, 18.2 here; 4x4 at 128 images 301 -> 250 14.7 and 11.0; 8x8 187 -> 171 13.6 and 11.9, there
// against one image per tile).
//
// What bounds it: the shared-memory port, which per tap of 64 channels carries 4 x (128 + filters) x 32 bytes of MMA operands per
// block and the filters' own arrival, and the issuing warps.  An MMA warp fetches its instructions alone, two MMAs are pending at
// most, and every wait, commit and counter between taps is exposed (60 to 220 cycles a tap).  Hence one wait per filter row where
// two rows of filters fit, and one instantiation per kind of ring and epilogue, which keeps the code between the loops short.
//
// Pairs.  Where filters are streamed that port carries them twice over: 16 KB of a tap of 64 channels and 128 filters arrive for every 128 or
// 256 pixels, and every MMA reads them again.  Two CTAs of a cluster therefore take neighbouring tiles of the same filters, each with its own
// patch, staging and accumulator, and each holds half of the filters: one tcgen05.mma of cta_group::2 multiplies both patches, the
// barriers of the first CTA count what arrives in both, and its commits free the stages of both.  Cold, alone (us, one CTA / pairs): 131 -> 203
// 28x28, 64 images 36.9 / 32.2; 70 -> 160 with a residual 35.8 / 28.4; 101 -> 96 16x16, 128 images 18.8 / 14.1 (all filters fit, halved); in the network
// 512 -> 358 7x7 18.4 / 15.7, 179 -> 256 14x14 16.3 / 14.8.  Filters that fit one CTA gain nothing (45 -> 58 32x32 14.7 / 17.4).  An expect_tx that the other
// CTA sends across (release at cluster scope) cost 700 cycles a tap; the first CTA expects the bytes of both instead.
//
//   warp 0       patch loads (one per channel block); with a residual, one more load per group of
//                64 filters brings the residual tile in through the same ring;
//   warps 1, 2   filter loads, one per (channel block, tap), taken in turn; small filter sets
//                stay resident in shared memory for the whole kernel;
//   warps 3, 12  tcgen05.mma issue (3 and 20 with sixteen epilogue warps), one warp per accumulator
//                block; the residual tile is added by
//                one more MMA against a 64 x 64 identity held in shared memory (bf16 x 1.0 into an
//                fp32 accumulator is exact), so the epilogue never touches global memory for it
//                (the 1x1 instantiation, whose tile is flat, still adds it in the epilogue);
//   warps 4..11  epilogue (4..19 for flat 1x1 tasks): tcgen05.ld, bias, activation, bf16 into a swizzled staging
//                buffer, then ONE TMA store per group of 64 filters whose box is the tile's rows x
//                Wp pixels (wrap-around columns, rows below the image and filters beyond k_pad lie
//                outside the tensor map and are not written).  With a fused max-pool the staged
//                tile is pooled and copied out by hand instead, eight threads per output pixel.
// Every wait is bounded (see sm100_ptx.cuh); on expiry the CTA raises STATUS_TIMEOUT and leaves.
#include <cuda.h>

#include <cstdlib>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "plan.h"
#include "sm100_ptx.cuh"

namespace cprune {

constexpr int PK_POOL_WARPS = 8;          // 3x3-pool kernel: these warps pool the staged tile while the epilogue warps stage the next one
// kernel instantiations: 3x3 and other R x S > 1 with resident filters or a ring of filter rows, 1x1 staged as in memory, fused
// 3x3 pool on its own warps, other 1x1, and R x S > 1 with a ring of taps
constexpr int PK_GENERAL = 0, PK_DENSE = 1, PK_POOL3 = 2, PK_FLAT = 3, PK_TAPS = 4;
// Epilogue warps.  A flat tile has little for the MMAs to do, so its epilogue bounds it: a warp spends about 300 cycles on 16
// filters of 128 pixels, mostly the latencies of a chain of 50 instructions, and sixteen warps hide twice as many of them as
// eight (64 images, 1x1 24 -> 108 of 56x56: 23.1 -> 19.9 us; 32 -> 16 of 112x112: 26.3 -> 19.1 us).  The other tasks are bound by
// their MMAs and lose with sixteen (3x3 131 -> 203 of 28x28: 37.8 -> 39.6 us); beside the pooling warps there is room for eight.
__host__ __device__ constexpr int pk_epi_warps(int mode) { return mode == PK_DENSE || mode == PK_FLAT ? 16 : 8; }
__host__ __device__ constexpr int pk_threads(int mode) { return (5 + pk_epi_warps(mode) + (mode == PK_POOL3 ? PK_POOL_WARPS : 0)) * 32; }
constexpr int PK_MMA_WARP = 3;
constexpr int PK_FIRST_EPI = 4;
// (the warp after the epilogue warps issues for the second accumulator block when MT = 2)
constexpr int PK_MAX_WSTAGES = 32;
constexpr int PK_MAX_PATCH_STAGES = 4;   // patch ring: 2 stages, more for tasks with small patches and several channel blocks
constexpr int PK_CTRL_BYTES = 5120;      // barriers (1 KB) + slot table (2 KB) + bias (2 KB)
constexpr int PK_BIAS_FLOATS = 512;      // the task's bias is kept in shared memory when it has at most this many filters
constexpr int PK_BLOCK_BYTES = 16384;    // staged block: 128 slots x 64 filters bf16
constexpr int PK_IDENT_BYTES = 8192;     // 64 x 64 identity (bf16, 128-byte rows): filter-side operand that adds a residual block

struct PatchParams {
    int P, Q, Wp, TH, tiles_per_img, tiles_m, tiles_n;
    int TW, tiles_w, step_h, step_w, org;   // tile (ty, tx) starts at output (ty * step_h + org, tx * step_w + org) and spans TH x TW
    int out_h, out_w;                       // stored extent (after a fused pool)
    int FT, MT, R, S, pad, pad_w, cblks, ksteps_last, k_pad;   // pad: rows above the image in a patch; pad_w: columns left of it
    int wgroup;            // taps that share a filter barrier: a filter row, or one
    int act, wstages, pstages, resident, acc_bufs, staging_bufs, pool;
    int patch_bytes;       // shared memory of one patch stage
    int patch_box_bytes;   // bytes one patch load delivers
    int w_stage_bytes;     // shared memory of one filter stage (FT rows, rounded up to 1024 bytes)
    int rb16;              // bytes per pixel row in shared memory / 16: 8 (64 channels) or 2 (16 channels, regrouped stems)
    int dense;             // the staged tile is [slot][k_pad] as in memory and leaves by one bulk copy (flat tasks, one filter tile)
    int dense_pitch;       // ... bytes per slot in the staging buffer: k_pad * 2, or 16 more (then the tile leaves by a tiled copy)
    int stage_bytes;       // shared memory of one staging buffer
    int ipt, imgs;         // whole images per tile (0: tiles of one image), images of the task
    uint32_t img_mul, row_mul;   // ceil(2^32 / tiles_per_img), ceil(2^32 / tiles_w), or 0
    int res_blocks;        // residual added on the tensor core: 64-filter blocks of the residual tile per item (0: none)
    const float *bias;
    const __nv_bfloat16 *res;
    __nv_bfloat16 *y;
    int *status;
};

// Maximum of 8 non-negative bf16 values (after ReLU / ReLU6; max.f32 never yields -0): their bit patterns order like
// unsigned integers, so one SIMD integer instruction handles two values.
__device__ __forceinline__ uint4 bf16x8_max_nonneg(uint4 a, uint4 b) {
    return make_uint4(__vmaxu2(a.x, b.x), __vmaxu2(a.y, b.y), __vmaxu2(a.z, b.z), __vmaxu2(a.w, b.w));
}

__device__ __forceinline__ uint4 bf16x8_max(uint4 a, uint4 b) {
    uint4 r;
    __nv_bfloat162 *pa = reinterpret_cast<__nv_bfloat162 *>(&a), *pb = reinterpret_cast<__nv_bfloat162 *>(&b);
    __nv_bfloat162 *pr = reinterpret_cast<__nv_bfloat162 *>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) pr[i] = __hmax2(pa[i], pb[i]);
    return r;
}

// Eight accumulator values of one pixel + bias -> activated bf16.  Two sums per instruction; 0 and 6 are bf16 values, so that
// the clamps commute with the rounding.  The activation is a pair of bounds without a branch: the maximum and the minimum return
// the operand that is a number, so that a NaN bound leaves everything as it is and a NaN result becomes 0 under ReLU and ReLU6, as
// in every other kernel.  (The conversion's own ReLU keeps a NaN, and the minimum with 6 would make it a 6.  That form, which
// branches on the activation, took 141.4 and 509 us for VGG-16 and MobileNetV2 at full batch, this one 139.9 and 503 us.)
__device__ __forceinline__ unsigned long long pair64(uint32_t lo, uint32_t hi) {
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}
struct Clamp { uint32_t lo, hi; };        // bf16 pairs
__device__ __forceinline__ bf16x8 bias_act8(const uint32_t *v, const unsigned long long *bias, const Clamp act) {
    bf16x8 r;
    float lo[4], hi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        unsigned long long t;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(pair64(v[2 * j], v[2 * j + 1])), "l"(bias[j]));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo[j]), "=f"(hi[j]) : "l"(t));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.w[j]) : "f"(hi[j]), "f"(lo[j]));
#pragma unroll
    for (int j = 0; j < 4; ++j) asm("max.bf16x2 %0, %0, %1;" : "+r"(r.w[j]) : "r"(act.lo));
#pragma unroll
    for (int j = 0; j < 4; ++j) asm("min.bf16x2 %0, %0, %1;" : "+r"(r.w[j]) : "r"(act.hi));
    return r;
}

// One MMA of 16 channels, and the arrival of those issued so far, for one CTA or for a pair.
template <bool PAIR>
__device__ __forceinline__ void mma_words(uint32_t d_tmem, uint32_t a_lo, uint32_t w_lo, uint32_t desc_hi, uint32_t idesc, uint32_t accumulate) {
    if (PAIR) umma_bf16_words_pair(d_tmem, a_lo, w_lo, desc_hi, idesc, accumulate);
    else umma_bf16_words(d_tmem, a_lo, w_lo, desc_hi, idesc, accumulate);
}
template <bool PAIR>
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    if (PAIR) umma_commit_pair(bar);
    else umma_commit(bar);
}
// All MMAs of one filter tap for one accumulator block: nk steps of 16 channels.  a_lo and w_lo are
// the low words of the operand descriptors (start address in 16-byte units).  Called by the whole warp: the
// operands are computed by all lanes (they stay in uniform registers) and one elected lane issues.
template <bool PAIR>
__device__ __forceinline__ void issue_tap(uint32_t d_tmem, uint32_t a_lo, uint32_t w_lo, uint32_t desc_hi, uint32_t idesc,
                                          uint32_t accumulate, int nk, uint32_t commit_w, uint32_t commit_p) {
    uint32_t al[4], wl[4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) { wl[kk] = w_lo + (uint32_t)(2 * kk); al[kk] = a_lo + (uint32_t)(2 * kk); }
    if (elect_one()) {
        if (nk == 4) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma_words<PAIR>(d_tmem, al[kk], wl[kk], desc_hi, idesc, kk ? 1u : accumulate);
        } else {
            mma_words<PAIR>(d_tmem, al[0], wl[0], desc_hi, idesc, accumulate);
#pragma unroll
            for (int kk = 1; kk < 3; ++kk)
                if (kk < nk) mma_words<PAIR>(d_tmem, al[kk], wl[kk], desc_hi, idesc, 1u);
        }
        if (commit_w) mma_commit<PAIR>(commit_w);
        if (commit_p) mma_commit<PAIR>(commit_p);
    }
    __syncwarp();
}

// A whole filter row (S taps) from one elected block: nothing has to be waited for between its taps.
template <bool PAIR>
__device__ __forceinline__ void issue_row(uint32_t d_tmem, uint32_t a_lo, uint32_t w_lo, uint32_t desc_hi, uint32_t idesc,
                                          uint32_t accumulate, int nk, int S, uint32_t slot_step, uint32_t w_step, uint32_t commit_w, uint32_t commit_p) {
    if (elect_one()) {
        for (int s = 0; s < S; ++s) {
            if (nk == 4) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    mma_words<PAIR>(d_tmem, a_lo + (uint32_t)(2 * kk), w_lo + (uint32_t)(2 * kk), desc_hi, idesc, kk ? 1u : accumulate);
            } else {
                mma_words<PAIR>(d_tmem, a_lo, w_lo, desc_hi, idesc, accumulate);
#pragma unroll
                for (int kk = 1; kk < 3; ++kk)
                    if (kk < nk) mma_words<PAIR>(d_tmem, a_lo + (uint32_t)(2 * kk), w_lo + (uint32_t)(2 * kk), desc_hi, idesc, 1u);
            }
            accumulate = 1;
            a_lo += slot_step;
            w_lo += w_step;
            if (commit_w) { mma_commit<PAIR>(commit_w); commit_w += 8u; }     // every tap frees its own stage
        }
        if (commit_p) mma_commit<PAIR>(commit_p);
    }
    __syncwarp();
}

// First output pixel (may be -1 with the 3x3 pool, whose windows reach one pixel outside the tile's own pooled
// pixels) and image of tile tm.  The divisions are multiplications with reciprocals that the host has checked for every
// tile number (mul == 0: by division); flat tasks (one image, one row of tiles) need none.
__device__ __forceinline__ int quotient(int v, int d, uint32_t mul) { return mul ? (int)__umulhi((uint32_t)v, mul) : v / d; }
template <bool FLAT>
__device__ __forceinline__ void tile_origin(const PatchParams &p, int tm, int &n, int &p0, int &q0) {
    if (FLAT) {
        n = 0; p0 = 0; q0 = tm * p.step_w;
        return;
    }
    if (p.ipt) {
        n = tm * p.ipt; p0 = 0; q0 = 0;
        return;
    }
    n = quotient(tm, p.tiles_per_img, p.img_mul);
    const int r = tm - n * p.tiles_per_img;
    int ty = r, tx = 0;
    if (p.tiles_w > 1) { ty = quotient(r, p.tiles_w, p.row_mul); tx = r - ty * p.tiles_w; }
    p0 = ty * p.step_h + p.org;
    q0 = tx * p.step_w + p.org;
}

template <int MODE, bool RESIDENT, bool POOLED = false, int WIDTH = 0, bool PAIR = false>
__global__ void __launch_bounds__(pk_threads(MODE), 1)
conv_patch_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                  const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_res, const PatchParams p) {
    extern __shared__ uint8_t smem_raw[];
    constexpr bool DENSE = MODE == PK_DENSE;
    constexpr bool SPLIT = MODE == PK_POOL3;      // staging by the epilogue warps, pooling by PK_POOL_WARPS further warps
    constexpr int EPI_WARPS = pk_epi_warps(MODE);
    constexpr int MMA_WARP2 = PK_FIRST_EPI + EPI_WARPS;
    if (threadIdx.x == 0) {
        // the descriptors are fetched on first use otherwise, which the first loads would wait for
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_x) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_w) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_y) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_res) : "memory");
    }
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw);
    const uint32_t w_bytes = (uint32_t)p.w_stage_bytes;                   // stage stride
    const uint32_t w_tx_bytes = (uint32_t)p.FT * (PAIR ? 8u : 16u) * (uint32_t)p.rb16;  // bytes one filter load delivers
    const uint32_t patch0 = base;
    const uint32_t w0 = patch0 + (uint32_t)p.pstages * (uint32_t)p.patch_bytes;
    const uint32_t staging0 = w0 + (uint32_t)p.wstages * w_bytes;
    const uint32_t stage_buf_bytes = (uint32_t)p.stage_bytes;
    const uint32_t ident0 = staging0 + (uint32_t)p.staging_bufs * stage_buf_bytes;   // present when res_blocks > 0
    const uint32_t ctrl0 = ident0 + (p.res_blocks ? (uint32_t)PK_IDENT_BYTES : 0u);
    uint8_t *ctrl = smem + (ctrl0 - base);
    auto pfull = [&](int s) { return ctrl0 + 8u * s; };
    auto pempty = [&](int s) { return ctrl0 + 32u + 8u * s; };
    auto tfull = [&](int a) { return ctrl0 + 64u + 8u * a; };
    auto tempty = [&](int a) { return ctrl0 + 80u + 8u * a; };
    const uint32_t epi_bar = ctrl0 + 96u;
    auto res_full = [&](int b) { return ctrl0 + 112u + 8u * b; };   // residual tile landed in staging buffer b
    uint32_t *tmem_slot = (uint32_t *)(ctrl + 104);
    volatile int *abort_flag = (volatile int *)(ctrl + 108);
    auto sfull = [&](int b) { return ctrl0 + 640u + 8u * b; };      // 3x3-pool kernel: staging buffer b holds a finished group
    auto sempty = [&](int b) { return ctrl0 + 656u + 8u * b; };     // ... has been pooled and may be overwritten
    auto wfull = [&](int s) { return ctrl0 + 128u + 8u * s; };
    auto wempty = [&](int s) { return ctrl0 + 384u + 8u * s; };
    int2 *lut = (int2 *)(ctrl + 1024);   // entry -> (source slot | tile row << 16, output offset in elements); x < 0: nothing to store

    // the shuffle tells the compiler that the warp number is the same in all lanes, so that the role code below
    // (loop counters, descriptors, TMA coordinates) can live in uniform registers
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    constexpr bool FLAT = MODE == PK_DENSE || MODE == PK_FLAT;      // 1x1 tasks: one image of one row
    const int FR = FLAT ? 1 : WIDTH ? WIDTH : p.R, FS = FLAT || SPLIT ? 1 : WIDTH ? WIDTH : p.S, RS = FR * FS;
    const int ipt = FLAT || SPLIT ? 0 : p.ipt;
    // Pairs: two CTAs take neighbouring tiles of the same filters, each with its own patch and half of the filters; the first one's
    // MMA warps issue for both, and its barriers count what arrives in both.
    const int rank = PAIR ? (int)(blockIdx.x & 1u) : 0, first_item = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int item_step = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x, total_items = PAIR ? ((p.tiles_m + 1) >> 1) * p.tiles_n : p.tiles_m * p.tiles_n;
    auto tile_of = [&](int item, int &tm, int &nt) {
        tm = item; nt = 0;
        if (p.tiles_n > 1) { tm = item / p.tiles_n; nt = item - tm * p.tiles_n; }
        if (PAIR) tm = tm * 2 + rank;
    };

    if (warp == PK_MMA_WARP) {
        if (PAIR) { tmem_alloc_pair(smem_u32(tmem_slot), 512); tmem_relinquish_pair(); }
        else { tmem_alloc(smem_u32(tmem_slot), 512); tmem_relinquish(); }
        pdl_trigger();
    }
    // barrier set-up, spread over the lanes of warp 0 (one thread doing up to 70 initialisations costs microseconds).
    // Every accumulator block has its own issuing warp: stages are free, and a tile is complete, once all have committed.
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        constexpr int CTAS = PAIR ? 2 : 1;
        if (l < p.pstages) { mbar_init(pfull(l), 1); mbar_init(pempty(l), p.MT); }
        if (l < 2) { mbar_init(tfull(l), p.MT); mbar_init(tempty(l), EPI_WARPS * CTAS); mbar_init(res_full(l), 1); }
        if (l == 2) { mbar_init(epi_bar, EPI_WARPS); *abort_flag = 0; }
        if (SPLIT && l >= 4 && l < 6) { mbar_init(sfull(l - 4), EPI_WARPS); mbar_init(sempty(l - 4), PK_POOL_WARPS); }
        if (l < p.wstages) { mbar_init(wfull(l), p.wgroup); mbar_init(wempty(l), p.MT); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the bias (written when the task was packed, not by the preceding kernel) in shared memory: a read costs the
    // epilogue a fraction of what the same read through L1 does
    // (the epilogue warps copy it while the first tile is being computed: see there)
    float *bias_s = (float *)(ctrl + 3072);
    const int k_all = p.tiles_n * p.FT;
    const bool bias_staged = k_all <= PK_BIAS_FLOATS;
    const float *bias_src = bias_staged ? bias_s : p.bias;
    // 64 x 64 identity in the layout of a filter stage (128-byte rows, 128-byte swizzle): row r holds 1.0 at channel r
    if (p.res_blocks) {
        uint8_t *ident = smem + (ident0 - base);
        for (int e = threadIdx.x; e < 64 * 8; e += blockDim.x) {
            // (pairs: this CTA's half of the rows, for blocks of 64 filters and, from row 32 on, for the last block)
            const int i = e >> 3, c = e & 7, last = (p.FT & 63) ? (p.FT & 63) >> 1 : 32;
            const int r = !PAIR ? i : i < 32 ? rank * 32 + i : i < 32 + last ? rank * last + i - 32 : 64;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (c == (r >> 3)) {
                const uint32_t one = (r & 1) ? 0x3F800000u : 0x00003F80u;      // bf16 1.0 in the odd or even half
                const int word = (r & 7) >> 1;
                if (word == 0) v.x = one; else if (word == 1) v.y = one; else if (word == 2) v.z = one; else v.w = one;
            }
            *(uint4 *)(ident + sub_off(i, c)) = v;
        }
        fence_async_smem();
    }
    // Stacked images: each one's bottom and right border is the top border of the next and the left border of the next row.
    // What the last one lacks follows its patch in the stage and is cleared once (no load writes there).
    if (ipt) {
        const uint32_t tail = (uint32_t)(p.pad * p.Wp + p.pad) * 8u;      // 16-byte pieces
        for (uint32_t e = threadIdx.x; e < (uint32_t)p.pstages * tail; e += blockDim.x) {
            const uint32_t st = e / tail, q = e - st * tail;
            *(uint4 *)(smem + (patch0 - base) + st * (uint32_t)p.patch_bytes + (uint32_t)p.patch_box_bytes + q * 16u) = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_async_smem();
    }
    // slot table: which accumulator rows hold real output pixels and where they go
    for (int e = threadIdx.x; POOLED && e < 256 && p.pool == 1; e += blockDim.x) {
        int2 v = make_int2(-1, 0);
        {
            const int hq = p.Q >> 1;
            const int i2 = e / hq, j2 = e - i2 * hq;
            if (ipt) {           // the "row" that decides whether the pixel is stored is the image
                const int hp = p.P >> 1, im = i2 / hp, ii = i2 - im * hp;
                if (im < ipt) v = make_int2(((im * (p.P + p.pad) + 2 * ii) * p.Wp + 2 * j2) | (im << 16), e * p.k_pad);
            } else if (i2 < (p.TH >> 1)) v = make_int2((2 * i2 * p.Wp + 2 * j2) | ((2 * i2) << 16), (i2 * hq + j2) * p.k_pad);
        }
        lut[e] = v;
    }
    tc_fence_before();
    if (PAIR) { __syncwarp(); cluster_sync(); }      // (.aligned: the loops above may have left a warp's threads apart)
    else __syncthreads();
    tc_fence_after();
    // Set-up done.  Only the patch (and residual) loads of warp 0 read what the preceding kernel wrote, and everything
    // else in this kernel follows from them, so warp 0 alone waits for the predecessor; filters and bias were written
    // when the task was packed and are fetched right away.
    const uint32_t tmem_base = *tmem_slot;

    auto expect = [&](uint32_t bar, uint32_t bytes) {
        // (pairs: the first CTA expects the bytes of both; what the other's loads deliver before that is counted all the same)
        if (rank == 0) mbar_expect_tx(bar, PAIR ? 2 * bytes : bytes);
    };
    auto load_4d = [&](uint32_t dst, const CUtensorMap *map, uint32_t bar, int c0, int c1, int c2, int c3) {
        if (PAIR) tma_load_4d_pair(dst, map, leader_addr(bar), c0, c1, c2, c3);
        else tma_load_4d(dst, map, bar, c0, c1, c2, c3);
    };
    if (warp == 0) {
        // ------------------------------------------------------------------ patch loads
        pdl_wait();
        int ps = 0;
        uint32_t pphase = 0;
        bool ok = true;
        for (int item = first_item; item < total_items && ok; item += item_step) {
            int tm, nt;
            tile_of(item, tm, nt);
            int n, p0, q0;
            tile_origin<FLAT>(p, tm, n, p0, q0);
            for (int cb = 0; cb < p.cblks; ++cb) {
                ok = __all_sync(0xffffffffu, mbar_wait(pempty(ps), pphase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                if (elect_one()) {
                    expect(pfull(ps), (uint32_t)p.patch_box_bytes);
                    load_4d(patch0 + (uint32_t)ps * p.patch_bytes, &tm_x, pfull(ps), cb * 64, q0 - p.pad_w, p0 - p.pad, n);
                }
                __syncwarp();
                if (++ps == p.pstages) { ps = 0; pphase ^= 1u; }
            }
            // The residual tile goes through the same ring, 64 filters at a time: its box is the tile's TH x Wp output
            // pixels, so pixel (i, j) lands in the row of slot i * Wp + j (wrap-around columns read as zero), and the MMA
            // warps add it to the accumulator by multiplying it with the identity.
            for (int j = 0; j < p.res_blocks && ok; ++j) {
                ok = __all_sync(0xffffffffu, mbar_wait(pempty(ps), pphase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                if (elect_one()) {
                    expect(pfull(ps), (uint32_t)(p.TH * p.Wp * 128));
                    load_4d(patch0 + (uint32_t)ps * p.patch_bytes, &tm_res, pfull(ps), nt * p.FT + j * 64, q0, p0, n);
                }
                __syncwarp();
                if (++ps == p.pstages) { ps = 0; pphase ^= 1u; }
            }
        }
    } else if (warp < PK_MMA_WARP) {
        // ------------------------------------------------------------------ filter loads
        int ws = 0, wsub = 0, turn = 0;
        uint32_t wphase = 0;
        bool ok = true;
        const int me = warp - 1;
        for (int item = first_item; item < total_items && ok; item += item_step) {
            if (RESIDENT && item != first_item) break;     // the filters of the first tile stay
            int nt = 0;
            if (p.tiles_n > 1) nt = item % p.tiles_n;
            const int k0 = nt * p.FT + (PAIR ? rank * (p.FT >> 1) : 0);
            for (int cb = 0; cb < p.cblks && ok; ++cb) {
                for (int tap = 0; tap < RS; ++tap) {
                    const bool mine = turn == me;
                    turn ^= 1;
                    if (mine) {
                        if (!RESIDENT) ok = __all_sync(0xffffffffu, mbar_wait(wempty(ws), wphase ^ 1u, abort_flag, p.status));
                        if (!ok) break;
                        if (elect_one()) {
                            const uint32_t wb = wfull(MODE == PK_GENERAL ? ws - wsub : ws);   // the taps of a row complete one barrier
                            expect(wb, w_tx_bytes);
                            if (PAIR) tma_load_3d_pair(w0 + (uint32_t)ws * w_bytes, &tm_w, leader_addr(wb), cb * 64, tap, k0);
                            else tma_load_3d(w0 + (uint32_t)ws * w_bytes, &tm_w, wb, cb * 64, tap, k0);
                        }
                        __syncwarp();
                    }
                    if (MODE == PK_GENERAL && ++wsub == p.wgroup) wsub = 0;
                    if (++ws == p.wstages) { ws = 0; wphase ^= 1u; }
                }
            }
        }
    } else if (warp == PK_MMA_WARP || warp == MMA_WARP2) {
        // ------------------------------------------------------------------ MMA issue
        // tcgen05.mma issue is close to synchronous (about two instructions may be pending, measured), so the
        // bookkeeping between taps would leave the tensor pipe idle if one warp issued everything: with MT = 2
        // each accumulator block gets its own issuing warp and the two interleave.
        const int mb = warp == PK_MMA_WARP ? 0 : 1;
        if (mb < p.MT && rank == 0) {
        constexpr uint32_t M_BITS = (uint32_t)((PAIR ? 256 : 128) >> 4) << 24;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.FT >> 3) << 17) | M_BITS;
        int ps = 0, ws = 0, acc = 0;
        uint32_t pphase = 0, wphase = 0, acc_phase = 0;
        bool ok = true;
        // A lone warp pays several cycles for every instruction, so the loop works on the low descriptor words
        // only (32-bit adds) and issues a tap's MMAs from fully unrolled code.
        const uint32_t patch_lo0 = desc_lo(patch0), w_lo0 = desc_lo(w0);
        const uint32_t desc_hi = p.rb16 == 8 ? DESC_HI_SW128 : DESC_HI_SW32;
        const uint32_t slot_step = (uint32_t)p.rb16;                    // descriptor units (16 bytes) per pixel row
        const uint32_t patch_step = (uint32_t)p.patch_bytes >> 4, w_step = w_bytes >> 4;
        const uint32_t row_step = (uint32_t)(p.Wp - FS + 1) * slot_step;   // from tap (r, S-1) to (r+1, 0)
        uint32_t patch_lo = patch_lo0, w_lo = w_lo0;
        for (int item = first_item; item < total_items && ok; item += item_step) {
            ok = __all_sync(0xffffffffu, mbar_wait(tempty(acc), acc_phase ^ 1u, abort_flag, p.status));
            if (!ok) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)((acc * p.MT + mb) * p.FT);
            uint32_t accumulate = 0;
            for (int cb = 0; cb < p.cblks && ok; ++cb) {
                ok = __all_sync(0xffffffffu, mbar_wait(pfull(ps), pphase, abort_flag, p.status));
                if (!ok) break;
                const int nk = cb == p.cblks - 1 ? p.ksteps_last : 4;
                uint32_t tap_lo = patch_lo + (uint32_t)(mb * 128) * slot_step;      // the second block's slots follow the first's
                if (RESIDENT && item != first_item) {
                    // resident filters, loaded during the first tile: nothing to wait for, a filter row per elected block
                    for (int r = 0; r < FR; ++r) {
                        issue_row<PAIR>(d_tmem, tap_lo, w_lo, desc_hi, idesc, accumulate, nk, FS, slot_step, w_step, 0u, r == FR - 1 ? pempty(ps) : 0u);
                        accumulate = 1;
                        tap_lo += (uint32_t)p.Wp * slot_step;
                        w_lo += (uint32_t)FS * w_step;
                        ws += FS;
                        if (ws == p.wstages) { ws = 0; w_lo = w_lo0; }
                    }
                } else if constexpr (MODE == PK_GENERAL) {
                    // one wait per filter row, then the row's MMAs from one elected block; every tap frees its own stage
                    for (int r = 0; r < FR; ++r) {
                        ok = __all_sync(0xffffffffu, mbar_wait(wfull(ws), RESIDENT ? 0u : wphase, abort_flag, p.status));
                        if (!ok) break;
                        issue_row<PAIR>(d_tmem, tap_lo, w_lo, desc_hi, idesc, accumulate, nk, FS, slot_step, w_step, RESIDENT ? 0u : wempty(ws),
                                  r == FR - 1 ? pempty(ps) : 0u);
                        accumulate = 1;
                        tap_lo += (uint32_t)p.Wp * slot_step;
                        w_lo += (uint32_t)FS * w_step;
                        ws += FS;
                        if (ws == p.wstages) { ws = 0; wphase ^= 1u; w_lo = w_lo0; }
                    }
                } else {
                    int s = 0;
                    for (int tap = 0; tap < RS; ++tap) {
                        ok = __all_sync(0xffffffffu, mbar_wait(wfull(ws), RESIDENT ? 0u : wphase, abort_flag, p.status));
                        if (!ok) break;
                        {
                            const uint32_t cw = RESIDENT ? 0u : wempty(ws), cp = tap == RS - 1 ? pempty(ps) : 0u;
                            issue_tap<PAIR>(d_tmem, tap_lo, w_lo, desc_hi, idesc, accumulate, nk, cw, cp);
                        }
                        accumulate = 1;
                        w_lo += w_step;
                        if (++ws == p.wstages) { ws = 0; wphase ^= 1u; w_lo = w_lo0; }
                        tap_lo += slot_step;
                        if (++s == FS) { s = 0; tap_lo += row_step - slot_step; }
                    }
                }
                patch_lo += patch_step;
                if (++ps == p.pstages) { ps = 0; pphase ^= 1u; patch_lo = patch_lo0; }
            }
            // residual blocks: accumulator columns 64 j .. += residual tile (slots x 64 filters) x identity (bf16 values
            // times 1.0, accumulated in float32: exact)
            for (int j = 0; j < p.res_blocks && ok; ++j) {
                ok = __all_sync(0xffffffffu, mbar_wait(pfull(ps), pphase, abort_flag, p.status));
                if (!ok) break;
                const int nres = min(64, p.FT - j * 64);
                const uint32_t idesc_r = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nres >> 3) << 17) | M_BITS;
                issue_tap<PAIR>(d_tmem + (uint32_t)(j * 64), patch_lo + (uint32_t)(mb * 128) * slot_step, desc_lo(ident0 + (PAIR && nres < 64 ? 4096u : 0u)), DESC_HI_SW128, idesc_r, 1u,
                          nres >> 4, 0u, pempty(ps));
                patch_lo += patch_step;
                if (++ps == p.pstages) { ps = 0; pphase ^= 1u; patch_lo = patch_lo0; }
            }
            if (ok && elect_one()) mma_commit<PAIR>(tfull(acc));
            __syncwarp();
            if (p.acc_bufs == 2) { if (++acc == 2) { acc = 0; acc_phase ^= 1u; } }
            else acc_phase ^= 1u;
        }
        }
    } else if (SPLIT && warp > MMA_WARP2) {
        // ------------------------------------------------------------------ 3x3 stride-2 pooling of staged groups
        // The tile computed conv rows p0 .. p0 + TH - 1 (p0 odd or -1) and holds the windows of (TH - 1) / 2 x (TW - 1) / 2
        // pooled pixels, all nine slots of each inside the staged tile.  A thread handles up to 512 / (32 * PK_POOL_WARPS) (pooled pixel,
        // 8 filters) items, the same ones in every tile: the shared-memory offsets of their window slots are worked out once.
        const int ctid = threadIdx.x - (MMA_WARP2 + 1) * 32;
        constexpr int ITEMS = 512 / (PK_POOL_WARPS * 32);
        const int groups = (p.FT + 63) / 64;
        const int tpc = (p.TW - 1) >> 1;
        const int n_entries = ((p.TH - 1) >> 1) * tpc;
        const bool clamp_lo = p.act != CPRUNE_ACT_NONE;
        uint32_t win_off[ITEMS][9];
        int win_pi[ITEMS], win_pj[ITEMS];
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int e = ctid + it * (PK_POOL_WARPS * 32);
            const int ent = e >> 3, chunk = e & 7;
            win_pi[it] = ent / tpc; win_pj[it] = ent - win_pi[it] * tpc;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int sl = (2 * win_pi[it] + k / 3) * p.Wp + 2 * win_pj[it] + k % 3;
                win_off[it][k] = (uint32_t)((sl >> 7) * PK_BLOCK_BYTES) + sub_off(sl & 127, chunk);
            }
        }
        uint32_t counter = 0;
        bool ok = true;
        // pixels outside the image never win: after ReLU / ReLU6 every value is >= 0 (and every window holds a real
        // pixel), so they can be replaced by 0 and the maximum taken on the bit patterns; else by -inf
        const uint4 fill = clamp_lo ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
        for (int item = first_item; item < total_items && ok; item += item_step) {
            int tm, nt;
            tile_of(item, tm, nt);
            int n, p0, q0;
            tile_origin<FLAT>(p, tm, n, p0, q0);
            const int pr0 = (p0 + 1) >> 1, pc0 = (q0 + 1) >> 1;
            for (int g = 0; g < groups && ok; ++g) {
                const uint32_t b = counter & 1u;
                ok = __all_sync(0xffffffffu, mbar_wait(sfull(b), (counter >> 1) & 1u, abort_flag, p.status));
                if (!ok) break;
                const uint8_t *buf = smem + (staging0 - base) + b * stage_buf_bytes;
                const int kg = nt * p.FT + g * 64;
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    const int e = ctid + it * (PK_POOL_WARPS * 32);
                    const int chunk = e & 7;
                    const int pr = pr0 + win_pi[it], pc = pc0 + win_pj[it];
                    if (e < n_entries * 8 && pr < p.out_h && pc < p.out_w && g * 64 + chunk * 8 < p.FT && kg + chunk * 8 < p.k_pad) {
                        const int r0 = p0 + 2 * win_pi[it], c0 = q0 + 2 * win_pj[it];
                        // bit d of a mask: window row / column d lies inside the image
                        const uint32_t rmask = (r0 >= 0 ? 1u : 0u) | 2u | (r0 + 2 < p.P ? 4u : 0u);
                        const uint32_t cmask = (c0 >= 0 ? 1u : 0u) | 2u | (c0 + 2 < p.Q ? 4u : 0u);
                        uint4 w[9];
#pragma unroll
                        for (int k = 0; k < 9; ++k) {
                            const uint4 t = *(const uint4 *)(buf + win_off[it][k]);
                            w[k] = ((rmask >> (k / 3)) & (cmask >> (k % 3)) & 1u) ? t : fill;
                        }
                        uint4 m;
                        if (clamp_lo) {
                            const uint4 a0 = bf16x8_max_nonneg(bf16x8_max_nonneg(w[0], w[1]), bf16x8_max_nonneg(w[2], w[3]));
                            const uint4 a1 = bf16x8_max_nonneg(bf16x8_max_nonneg(w[4], w[5]), bf16x8_max_nonneg(w[6], w[7]));
                            m = bf16x8_max_nonneg(bf16x8_max_nonneg(a0, a1), w[8]);
                        } else {
                            const uint4 a0 = bf16x8_max(bf16x8_max(w[0], w[1]), bf16x8_max(w[2], w[3]));
                            const uint4 a1 = bf16x8_max(bf16x8_max(w[4], w[5]), bf16x8_max(w[6], w[7]));
                            m = bf16x8_max(bf16x8_max(a0, a1), w[8]);
                        }
                        *(uint4 *)(p.y + (((size_t)n * p.out_h + pr) * p.out_w + pc) * p.k_pad + kg + chunk * 8) = m;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(sempty(b));
                ++counter;
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        constexpr int EPI_THREADS = EPI_WARPS * 32;
        constexpr int SUBS = EPI_WARPS / 4;            // warps that share a quarter of the accumulator lanes
        constexpr int WCOLS = 64 / SUBS;               // ... each takes this many filters of a 64-filter group
        constexpr int UNITS = WCOLS / 16;              // 16-filter units of a warp per accumulator block
        const int quarter = warp & 3;
        const int sub = (warp - PK_FIRST_EPI) >> 2;
        const int trow = quarter * 32 + lane;          // accumulator lane = slot within its 128-slot block
        const int etid = threadIdx.x - PK_FIRST_EPI * 32;
        int acc = 0;
        uint32_t acc_phase = 0, epi_phase = 0, group_counter = 0;
        bool ok = true;
        auto epi_sync = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(epi_bar);
            bool r = __all_sync(0xffffffffu, mbar_wait(epi_bar, epi_phase, abort_flag, p.status, false));
            epi_phase ^= 1u;
            return r;
        };
        // the task's bias into shared memory, while the first tile is being computed
        if (bias_staged) {
            for (int e = etid; e < k_all; e += EPI_THREADS) bias_s[e] = __ldg(p.bias + e);
            ok = epi_sync();
        }
        // bf16 pairs: NaN (no bound), 0 and 6
        const Clamp act_clamp = {p.act == CPRUNE_ACT_NONE ? 0x7fff7fffu : 0u, p.act == CPRUNE_ACT_RELU6 ? 0x40C040C0u : 0x7fff7fffu};
        const bool clamp_lo = p.act != CPRUNE_ACT_NONE;      // results are >= 0
        const bool store_thread = warp == PK_FIRST_EPI && lane == 0;
        const int groups = (p.FT + 63) / 64;
        // one group and one filter tile: a thread stages the same filters in every tile and keeps their bias in registers
        const bool bias_const = groups == 1 && p.tiles_n == 1;
        unsigned long long bias_r[WCOLS / 2];
        auto load_bias = [&](int c) {                  // filters c .. c + WCOLS - 1
#pragma unroll
            for (int j = 0; j < WCOLS / 2; ++j)
                bias_r[j] = c + j * 2 < k_all ? *reinterpret_cast<const unsigned long long *>(bias_src + c + j * 2) : 0ull;
        };
        if (bias_const) load_bias(sub * WCOLS);
        const int n_entries = ipt ? ipt * (p.P >> 1) * (p.Q >> 1) : p.pool == 1 ? (p.TH >> 1) * (p.Q >> 1) : ((p.TH - 1) >> 1) * ((p.TW - 1) >> 1);
        // Residuals.  Everywhere but with dense staging the MMA warps add the residual on the tensor core (see there) and
        // the epilogue has nothing to do with it.  Dense staging: the residual of tile item_ (tiles_n == 1, one row of
        // tiles) is one contiguous range of memory, arrives in the staging buffer the tile will use and is added in place.
        const bool with_res = DENSE && p.res != nullptr;
        const bool dense_tiled = DENSE && p.dense_pitch != p.k_pad * 2;
        const int dense_n16 = (p.k_pad + 15) >> 4, dense_units = dense_n16 * p.MT;
        const uint32_t dense_block = 128u * (uint32_t)p.dense_pitch;
        auto load_residual_dense = [&](int item_, uint32_t counter) {
            const int q0_ = item_ * p.step_w;
            const uint32_t bytes = (uint32_t)min(p.TW, p.Q - q0_) * (uint32_t)p.k_pad * 2u;
            const uint32_t b = counter & 1u;
            if (dense_tiled) {
                // the box is the whole tile, one piece wider than the tensor: what lies outside arrives as zeros
                mbar_expect_tx(res_full(b), (uint32_t)p.TW * (uint32_t)p.dense_pitch);
                tma_load_4d(staging0 + b * stage_buf_bytes, &tm_res, res_full(b), 0, q0_, 0, 0);
            } else {
                mbar_expect_tx(res_full(b), bytes);
                bulk_load(staging0 + b * stage_buf_bytes, p.res + (size_t)q0_ * p.k_pad, bytes, res_full(b));
            }
        };
        if (with_res && store_thread && (int)blockIdx.x < total_items) {
            pdl_wait();        // the residual is the result of an earlier kernel of the chain
            load_residual_dense(blockIdx.x, 0);
        }
        for (int item = first_item; item < total_items && ok; item += item_step) {
            int tm, nt;
            tile_of(item, tm, nt);
            int n, p0, q0;
            tile_origin<FLAT>(p, tm, n, p0, q0);
            const int k0 = nt * p.FT;
            const int rows_valid = PAIR && tm >= p.tiles_m ? 0 : ipt ? p.imgs - n : p.P - p0;    // tile rows (or images) below this are real ones
            // first pooled pixel of the tile (2x2 pool: full-width tiles from an even row)
            __nv_bfloat16 *ytile = p.pool == 1 ? p.y + ((size_t)n * (p.P >> 1) + (p0 >> 1)) * (p.Q >> 1) * p.k_pad : nullptr;
            ok = __all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, p.status, false));
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * p.MT * p.FT);
            if constexpr (DENSE) {
                // Flat task with one filter tile: the tile's output is ONE contiguous range of y (slot-major, k_pad filters
                // per slot).  With an odd number of 16-byte pieces per slot it is staged in exactly that layout (the pieces
                // of eight neighbouring slots fall in distinct banks) and leaves by a single bulk copy; a residual arrives
                // the same way.  With an even number the staged slots are one piece longer, and the tile moves by a tiled
                // copy whose box is that one piece wider than the tensor: the piece outside is not written (read as zeros).
                const uint32_t b = group_counter & 1u;
                uint8_t *buf = smem + (staging0 - base) + b * stage_buf_bytes;
                const uint32_t pitch = (uint32_t)p.dense_pitch;
                if (with_res) {
                    ok = __all_sync(0xffffffffu, mbar_wait(res_full(b), (group_counter >> 1) & 1u, abort_flag, p.status, false));
                    if (!ok) break;
                }
                // 16-filter units of both accumulator blocks, dealt to the warps of a quarter in turn
                uint8_t *row = buf + (uint32_t)trow * pitch;
                auto stage_half = [&](uint8_t *dst, uint32_t *v, int c) {
                    unsigned long long bb[4];
                    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(bias_src + c), b1 = *reinterpret_cast<const ulonglong2 *>(bias_src + c + 4);
                    bb[0] = b0.x; bb[1] = b0.y; bb[2] = b1.x; bb[3] = b1.y;
                    if (with_res) {
                        // (acc + bias) + residual, as everywhere
                        const bf16x8 rv = *(const bf16x8 *)dst;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            unsigned long long t;
                            asm("add.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(pair64(v[2 * j], v[2 * j + 1])), "l"(bb[j]));
                            asm("mov.b64 {%0, %1}, %2;" : "=r"(v[2 * j]), "=r"(v[2 * j + 1]) : "l"(t));
                            bb[j] = pair64(rv.w[j] << 16, rv.w[j] & 0xffff0000u);
                        }
                    }
                    *(bf16x8 *)dst = bias_act8(v, bb, act_clamp);
                };
                for (int u = sub; u < dense_units; u += SUBS) {
                    const bool second = u >= dense_n16;
                    const int ch = (second ? u - dense_n16 : u) * 16;
                    uint8_t *dst = row + (second ? dense_block : 0u) + ch * 2;
                    uint32_t v[16];
                    tmem_ld16(t_row + (uint32_t)((second ? p.FT : 0) + ch), v);
                    tmem_ld_wait();
                    stage_half(dst, v, ch);
                    if (ch + 8 < p.k_pad) stage_half(dst + 16, v + 8, ch + 8);
                }
                // every warp has read what it needs of the accumulator (a warp without filters in the last group too)
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty(acc));
                fence_async_smem();
                // the other buffer, written next, was last read by the previous tile's store
                if (store_thread) tma_store_wait_read<0>();
                ok = epi_sync();
                if (!ok) break;
                if (store_thread) {
                    const int rows = min(p.TW, p.Q - q0);
                    if (dense_tiled) tma_store_4d(&tm_y, staging0 + b * stage_buf_bytes, 0, q0, 0, 0);
                    else bulk_store(p.y + (size_t)q0 * p.k_pad, staging0 + b * stage_buf_bytes, (uint32_t)rows * pitch);
                    tma_store_commit();
                    if (with_res && item + (int)gridDim.x < total_items) load_residual_dense(item + gridDim.x, group_counter + 1);
                }
                ++group_counter;
            } else {
            for (int g = 0; g < groups && ok; ++g) {
                const uint32_t boff = (p.staging_bufs == 2 ? (group_counter & 1u) : 0u) * stage_buf_bytes;
                uint8_t *buf = smem + (staging0 - base) + boff;
                const int ch = g * 64 + sub * WCOLS;         // this warp's filters of the group
                if constexpr (SPLIT) {
                    // the buffer's previous contents (two groups ago) must have been pooled
                    ok = __all_sync(0xffffffffu, mbar_wait(sempty(group_counter & 1u), ((group_counter >> 1) & 1u) ^ 1u, abort_flag, p.status, false));
                    if (!ok) break;
                }
                // Units of 16 filters of one accumulator block; the tensor-memory loads of a pair of them are in flight together:
                // those of the two blocks, or (two units per warp) both of block 0, then both of block 1.
                if (!bias_const && ch < p.FT) load_bias(k0 + ch);
                uint32_t va[16], vb[16];
#pragma unroll
                for (int q = 0; q < UNITS; ++q) {
                    const int mb_a = UNITS == 1 ? 0 : q, mb_b = UNITS == 1 ? 1 : q, cu_b = UNITS == 1 ? 0 : 1;
                    const bool do_a = mb_a < p.MT && ch < p.FT, do_b = mb_b < p.MT && ch + cu_b * 16 < p.FT;
                    if (do_a) tmem_ld16(t_row + (uint32_t)(mb_a * p.FT + ch), va);
                    if (do_b) tmem_ld16(t_row + (uint32_t)(mb_b * p.FT + ch + cu_b * 16), vb);
                    tmem_ld_wait();
                    if (q == UNITS - 1 && g == groups - 1) {     // accumulator fully read: hand it back
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            if (PAIR) mbar_arrive_cluster(leader_addr(tempty(acc)));
                            else mbar_arrive(tempty(acc));
                        }
                    }
                    if (do_a) {
                        uint8_t *blk = buf + mb_a * PK_BLOCK_BYTES;
                        *(bf16x8 *)(blk + sub_off(trow, sub * (WCOLS / 8))) = bias_act8(va, bias_r, act_clamp);
                        *(bf16x8 *)(blk + sub_off(trow, sub * (WCOLS / 8) + 1)) = bias_act8(va + 8, bias_r + 4, act_clamp);
                    }
                    if (do_b) {
                        uint8_t *blk = buf + mb_b * PK_BLOCK_BYTES;
                        *(bf16x8 *)(blk + sub_off(trow, sub * (WCOLS / 8) + cu_b * 2)) = bias_act8(vb, bias_r + cu_b * 8, act_clamp);
                        *(bf16x8 *)(blk + sub_off(trow, sub * (WCOLS / 8) + cu_b * 2 + 1)) = bias_act8(vb + 8, bias_r + cu_b * 8 + 4, act_clamp);
                    }
                }
                if constexpr (SPLIT) {
                    // hand the staged group to the pooling warps and go on with the next one
                    __syncwarp();
                    if (lane == 0) mbar_arrive(sfull(group_counter & 1u));
                    ++group_counter;
                    continue;
                }
                if constexpr (!POOLED) {
                    // one TMA store per group: the staged slots are TH rows of Wp pixels; the tensor map's box has
                    // that shape, and the wrap-around columns (j >= Q), rows below the image and filters beyond
                    // k_pad fall outside the tensor, where a store writes nothing
                    fence_async_smem();
                    // the buffer written next (the other one) was last read by the previous group's store
                    if (p.staging_bufs == 2 && store_thread) tma_store_wait_read<0>();
                    ok = epi_sync();
                    if (!ok) break;
                    if (store_thread) {
                        if (k0 + g * 64 < p.k_pad) tma_store_4d(&tm_y, staging0 + boff, k0 + g * 64, q0, p0, n);
                        tma_store_commit();
                        if (p.staging_bufs == 1) tma_store_wait_read<0>();
                    }
                    if (p.staging_bufs == 1) {
                        ok = epi_sync();
                        if (!ok) break;
                    }
                    ++group_counter;
                } else {
                ok = epi_sync();
                if (!ok) break;
                // copy-out: eight threads per output pixel, 16 bytes each
                const int kg = k0 + g * 64;
                auto staged = [&](int sl, int chunk) { return *(const uint4 *)(buf + (sl >> 7) * PK_BLOCK_BYTES + sub_off(sl & 127, chunk)); };
                if (p.pool == 1) {
                    for (int e = etid; e < n_entries * 8; e += EPI_THREADS) {
                        const int2 l = lut[e >> 3];
                        const int chunk = e & 7;
                        if (l.x >= 0 && (l.x >> 16) < rows_valid && g * 64 + chunk * 8 < p.FT && kg + chunk * 8 < p.k_pad) {
                            const int slot = l.x & 0xffff;
                            uint4 val = bf16x8_max(staged(slot, chunk), staged(slot + 1, chunk));
                            val = bf16x8_max(val, bf16x8_max(staged(slot + p.Wp, chunk), staged(slot + p.Wp + 1, chunk)));
                            *(uint4 *)(ytile + l.y + kg + chunk * 8) = val;
                        }
                    }
                } else {
                    // 3x3 stride-2 windows: the tile computed conv rows p0 .. p0 + TH - 1 (p0 odd or -1) and holds the
                    // windows of (TH - 1) / 2 x (TW - 1) / 2 pooled pixels.  All nine slots of a window are inside the
                    // staged tile, so they are loaded unconditionally; conv pixels outside the image are replaced by
                    // -inf (they never win).
                    const int pr0 = (p0 + 1) >> 1, pc0 = (q0 + 1) >> 1;
                    const uint4 ninf = make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
                    // after ReLU / ReLU6 all values are >= 0: pixels outside the image can be replaced by 0 (every
                    // window holds a real pixel) and the maximum taken on the bit patterns
                    const uint4 fill = clamp_lo ? make_uint4(0u, 0u, 0u, 0u) : ninf;
                    const int tpc = (p.TW - 1) >> 1;
                    for (int e = etid; e < n_entries * 8; e += EPI_THREADS) {
                        const int chunk = e & 7, win_pi = (e >> 3) / tpc, win_pj = (e >> 3) - win_pi * tpc;
                        const int pr = pr0 + win_pi, pc = pc0 + win_pj;
                        if (pr < p.out_h && pc < p.out_w && g * 64 + chunk * 8 < p.FT && kg + chunk * 8 < p.k_pad) {
                            const int r0 = p0 + 2 * win_pi, c0 = q0 + 2 * win_pj;
                            // bit d of a mask: window row / column d lies inside the image
                            const uint32_t rmask = (r0 >= 0 ? 1u : 0u) | 2u | (r0 + 2 < p.P ? 4u : 0u);
                            const uint32_t cmask = (c0 >= 0 ? 1u : 0u) | 2u | (c0 + 2 < p.Q ? 4u : 0u);
                            uint4 w[9];
#pragma unroll
                            for (int k = 0; k < 9; ++k) {
                                const uint4 t = staged((2 * win_pi + k / 3) * p.Wp + 2 * win_pj + k % 3, chunk);
                                w[k] = ((rmask >> (k / 3)) & (cmask >> (k % 3)) & 1u) ? t : fill;
                            }
                            uint4 m;
                            if (clamp_lo) {
                                const uint4 a0 = bf16x8_max_nonneg(bf16x8_max_nonneg(w[0], w[1]), bf16x8_max_nonneg(w[2], w[3]));
                                const uint4 a1 = bf16x8_max_nonneg(bf16x8_max_nonneg(w[4], w[5]), bf16x8_max_nonneg(w[6], w[7]));
                                m = bf16x8_max_nonneg(bf16x8_max_nonneg(a0, a1), w[8]);
                            } else {
                                const uint4 a0 = bf16x8_max(bf16x8_max(w[0], w[1]), bf16x8_max(w[2], w[3]));
                                const uint4 a1 = bf16x8_max(bf16x8_max(w[4], w[5]), bf16x8_max(w[6], w[7]));
                                m = bf16x8_max(bf16x8_max(a0, a1), w[8]);
                            }
                            *(uint4 *)(p.y + (((size_t)n * p.out_h + pr) * p.out_w + pc) * p.k_pad + kg + chunk * 8) = m;
                        }
                    }
                }
                if (p.staging_bufs == 1) {
                    ok = epi_sync();
                    if (!ok) break;
                }
                ++group_counter;
                }
            }
            }
            if (p.acc_bufs == 2) { if (++acc == 2) { acc = 0; acc_phase ^= 1u; } }
            else acc_phase ^= 1u;
        }
        if (store_thread) tma_store_wait_all();      // staged data must be read before the CTA's memory goes away
    }

    // ---------------------------------------------------------------------- teardown
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land before the memory goes away
    }
    tc_fence_before();
    if (PAIR) {
        __syncwarp();
        cluster_sync();        // (the other CTA's MMAs read this one's memory and arrive on its barriers)
    } else {
        __syncthreads();
    }
    if (warp == PK_MMA_WARP) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------ host

// Estimated cycles of one tile.  Per tcgen05.mma (M = 128, N = FT, K = 16) the tensor pipe needs FT / 2 cycles
// and the operand reads (128 + FT) * 32 bytes of the 128 bytes per clock that shared memory delivers; the TMA
// writes of filters and patches share that port (measured on B200).
// Pairs: half of the filters in either CTA; an MMA costs max(N / 2, 35 + N / 8) cycles (measured: 39 / 43 / 50 / 64 at N = 32 / 64 / 96 / 128).
static double tile_cycles(int MT, int FT, int RS, int cblks, int ksteps_last, int row_bytes, int Wp, int TH, int R, bool resident,
                          int acc_bufs, int pair) {
    double total = 0;
    for (int cb = 0; cb < cblks; ++cb) {
        const int nk = cb == cblks - 1 ? ksteps_last : 4;
        const double tensor = MT * nk * (FT / 2.0);
        const double own = pair ? FT / 2.0 : FT;           // filters in this CTA's shared memory
        const double smem = (MT * nk * ((128.0 + own) * 32.0 + (pair ? 384.0 : 0.0)) + (resident ? 0.0 : own * row_bytes)) / 128.0;
        total += RS * (tensor > smem ? tensor : smem) + Wp * (TH + R - 1) * row_bytes / 128.0;
    }
    const double epilogue = MT * ((FT + 63) / 64) * 1200.0;
    return total + (acc_bufs == 2 ? (epilogue > total ? epilogue - total : 0.0) : epilogue) + 1500.0;
}

// What the kernel sees.  Wide tasks (c_pad >= 16, stride 1): the task itself, 64 channels per shared-memory row.
// Stems with C * stride^2 <= 16 (stride 1 or 2): the input is first regrouped into 16-channel pixels, one per
// stride x stride block of input pixels (channel (dy * stride + dx) * C + c), with the zero columns of the padding
// written out.  Up to four consecutive regrouped pixels (the Se filter columns, 32 bytes each) are then read as
// ONE 128-byte shared-memory row through a tensor map whose pixel stride is 32 bytes, so that the task becomes a
// stride-1 task with Re x 1 taps of Se * 16 channels and no wrap-around slots.  (Rows of 32 bytes would work too,
// but the MMA's operand reads then cost a full shared-memory cycle per row: measured four times slower.)
struct PatchGeometry {
    int stem, sf, Re, Se, pad_lo, He, We, WP, cblks, ksteps_last, Wp, kR, kS, pad_w;
    // the tensors as the kernel addresses them: images x rows x columns of the input (wide tasks) and of the conv output
    // and the stored output.  A 1x1 stride-1 task is a plain matrix product: its pixels are viewed as ONE row of
    // N*H*W columns, so that tiles are runs of 128 or 256 pixels with nothing wasted (flat = 1).
    int flat, vN, vH, vW, vP, vQ, vOH, vOW;
};

static bool patch_geometry(const cprune_plan_info &i, PatchGeometry *g) {
    if (i.groups != 1) return false;
    g->flat = 0; g->vN = i.N; g->vH = i.H; g->vW = i.W; g->vP = i.P; g->vQ = i.Q; g->vOH = i.out_h; g->vOW = i.out_w;
    if (i.c_pad >= 16 && i.stride == 1 && i.R == 1 && i.S == 1 && i.pad == 0) {
        const long long M = (long long)i.N * i.H * i.W;
        if (M > 0x7fffffffLL) return false;
        g->flat = 1; g->vN = 1; g->vH = 1; g->vW = (int)M; g->vP = 1; g->vQ = (int)M; g->vOH = 1; g->vOW = (int)M;
        g->stem = 0; g->sf = 1; g->Re = 1; g->Se = 1; g->pad_lo = 0; g->He = 1; g->We = (int)M; g->WP = (int)M;
        g->cblks = (i.c_pad + 63) / 64;
        g->ksteps_last = (i.c_pad - (g->cblks - 1) * 64 + 15) / 16;
        g->Wp = 128;                           // per tile: set by the planner (128 or 256 pixels)
        g->kR = 1; g->kS = 1; g->pad_w = 0;
        return true;
    } else if (i.c_pad >= 16 && i.stride == 1) {
        if (i.R * i.S <= 1 || i.R > 7 || i.S > 7) return false;
        g->stem = 0; g->sf = 1; g->Re = i.R; g->Se = i.S; g->pad_lo = i.pad; g->He = i.H; g->We = i.W; g->WP = i.W;
        g->cblks = (i.c_pad + 63) / 64;
        g->ksteps_last = (i.c_pad - (g->cblks - 1) * 64 + 15) / 16;
        g->Wp = i.Q + i.S - 1;
        g->kR = i.R; g->kS = i.S; g->pad_w = i.pad;
        if (g->Wp < g->We + g->pad_lo) return false;
    } else if (i.c_pad == 8 && i.stride <= 2 && i.C * i.stride * i.stride <= 16 && i.R * i.S > 1 && i.R <= 8 && i.S <= 8) {
        const int sf = i.stride;
        if ((i.H % sf) || (i.W % sf)) return false;
        if ((size_t)4 * sf * i.W * 16 > 48 * 1024) return false;   // the regrouping pass stages 4 * sf input rows in shared memory
        if (i.R - 1 - i.pad < 0 || i.S - 1 - i.pad < 0) return false;
        g->stem = 1; g->sf = sf;
        g->pad_lo = sf == 1 ? i.pad : (i.pad + 1) / 2;
        g->Re = sf == 1 ? i.R : (i.R - 1 - i.pad) / 2 + g->pad_lo + 1;
        g->Se = sf == 1 ? i.S : (i.S - 1 - i.pad) / 2 + g->pad_lo + 1;
        if (g->Se > 4) return false;
        g->He = i.H / sf; g->We = i.W / sf;
        g->WP = i.Q + 3;                       // a row starting at the last output column still reads four pixels
        if (g->WP < g->We + g->pad_lo) return false;
        g->cblks = 1; g->ksteps_last = g->Se;
        g->Wp = i.Q;
        g->kR = g->Re; g->kS = 1; g->pad_w = 0;
    } else {
        return false;
    }
    if (g->Wp > 128) return false;
    if (i.P + g->Re - 1 < g->He + g->pad_lo) return false;
    return true;
}

// Decides whether the task runs on the patch kernel and with which tiling; fills plan->info tile fields.
cprune_status plan_conv_patch(cprune_plan *plan) {
    cprune_plan_info &i = plan->info;
    plan->patch = 0;
    plan->pre_bytes = 0;
    PatchGeometry g;
    if (!patch_geometry(i, &g)) return CPRUNE_ERR_UNSUPPORTED;
    const bool pool = plan->opts.pool == CPRUNE_POOL_MAX2X2;
    const bool pool3 = plan->opts.pool == CPRUNE_POOL_MAX3X3S2;
    if (pool && (plan->opts.residual || (i.P & 1) || (i.Q & 1))) return CPRUNE_ERR_UNSUPPORTED;
    // the 3x3 pool needs tiles narrower than the image, which only tasks without wrap-around slots allow
    if (pool3 && (plan->opts.residual || g.kS != 1)) return CPRUNE_ERR_UNSUPPORTED;
    if (g.flat && (pool || pool3)) return CPRUNE_ERR_UNSUPPORTED;
    const int k16 = round_up(i.K, 16);
    const int cblks = g.cblks, ksteps_last = g.ksteps_last, RB = 128;
    const int RS = g.kR * g.kS;
    double best_of[2] = {1e30, 1e30};        // of single blocks, of pairs
    PatchTiling tiling_of[2] = {};
    double pair_rounds = 1.0;
    const int pairs_allowed = !g.flat && !g.stem && !pool3 && g.kR == 3 && g.kS == 3 ? 1 : 0;
    for (int MT = 1; MT <= 2; ++MT)
      for (int pair = 0; pair <= pairs_allowed; ++pair) {
      // candidate tile shapes: whole-width rows; for the 3x3 pool (2 tpr + 1) x (2 tpc + 1) conv pixels around tpr x tpc pooled ones
      // and whole images next to each other where several fit
      const int n_shapes = pool3 ? 32 * 32 : 2;
      for (int shape = 0; shape < n_shapes; ++shape) {
        int ipt = 0;
        int TH, TW = g.vQ, tiles_w = 1, step_h, step_w = g.vQ, org = 0, tiles_per_img, Wp = g.Wp;
        if (!pool3 && shape == 1) {
            // small images (7x7: four to 256 slots): a pixel row is W + pad slots, an image (H + pad) rows, and each border is
            // shared by the two rows or images that it lies between
            if (g.flat || g.stem || i.R != i.S || (i.R & 1) == 0 || i.pad != i.R / 2) continue;
            Wp = g.vQ + i.pad;
            ipt = 128 * MT / ((g.vP + i.pad) * Wp);
            if (ipt < 2) continue;
            TH = (g.vP + i.pad) * ipt;
            step_h = TH;
            tiles_per_img = 1;
        } else if (g.flat) {
            TH = 1; TW = 128 * MT; Wp = TW; step_h = 1; step_w = TW;
            tiles_w = (g.vQ + TW - 1) / TW;
            tiles_per_img = tiles_w;
        } else if (pool3) {
            const int tpr = shape / 32 + 1, tpc = shape % 32 + 1;
            if (tpr > i.out_h || tpc > i.out_w) continue;
            TH = 2 * tpr + 1; TW = 2 * tpc + 1;
            if (TH * TW > 128 * MT) continue;
            Wp = TW;
            step_h = 2 * tpr; step_w = 2 * tpc; org = -1;
            tiles_w = (i.out_w + tpc - 1) / tpc;
            tiles_per_img = ((i.out_h + tpr - 1) / tpr) * tiles_w;
        } else {
            TH = (128 * MT) / Wp;
            if (TH > i.P) TH = i.P;
            if (pool) TH &= ~1;
            if (TH < 1) continue;
            step_h = TH;
            tiles_per_img = (i.P + TH - 1) / TH;
        }
        for (int tiles_n = 1; tiles_n <= 8; ++tiles_n) {
            // with several filter tiles every tile ends on a 64-filter boundary: the stores are 64 filters wide and
            // only the tensor's own edge clips them
            const int FT = round_up((k16 + tiles_n - 1) / tiles_n, tiles_n > 1 ? 64 : pair ? 32 : 16);
            if (FT > 256 || MT * FT > 512) continue;
            if ((k16 + FT - 1) / FT != tiles_n) continue;
            const int acc_bufs = 2 * MT * FT <= 512 ? 2 : 1;
            const int patch_bytes = round_up((128 * MT + (g.kR - 1) * Wp + g.kS - 1) * RB, 1024);
            if (!ipt && patch_bytes < Wp * (TH + g.kR - 1) * RB) continue;
            // patch ring depth: two stages; up to four when the task has that many channel blocks and the patches are
            // small (1x1 tasks), because each load's latency is otherwise exposed
            // (flat tasks: a tile is little work, and a patch load's latency under a stream of output writes is several
            // tiles long, so the ring is as deep as fits)
            int ps_max = 2;
            if (cblks > 2 && patch_bytes <= 32 * 1024) ps_max = cblks < PK_MAX_PATCH_STAGES ? cblks : PK_MAX_PATCH_STAGES;
            if (g.flat || g.stem) ps_max = PK_MAX_PATCH_STAGES;     // (stems: a tile is a few MMAs, shorter than a load's latency)
            // A residual travels through the patch ring too (64 filters per stage).  A deeper ring, which would let the
            // next tile's first patch be fetched while the residual blocks are still in use, was measured against the
            // shallow one with the shared memory spent on resident filters / more filter stages instead: the shallow ring
            // won on every ResNet-18 shape (26.5 vs 27.8 us, 21.1 vs 22.5 us, 21.9 vs 21.7 us).
            const int res_blocks_plan = plan->opts.residual ? (FT + 63) / 64 : 0;
          for (int pstages = ps_max; pstages >= 2; --pstages) {
            const int dense_pitch = ((((i.k_pad >> 3) & 1) || i.k_pad == 16) ? i.k_pad : i.k_pad + 8) * 2;
            const int dense_bytes = round_up(128 * MT * dense_pitch, 1024);
            const int dense = g.flat && tiles_n == 1 && dense_pitch <= 512 && dense_bytes <= 48 * 1024 &&
                              (dense_pitch == i.k_pad * 2 || !plan->opts.residual);
            // a residual is added on the tensor core (identity operand in shared memory), except with dense staging,
            // where it arrives in the staging buffer
            const int ident_bytes = (plan->opts.residual && !dense) ? PK_IDENT_BYTES : 0;
            const int fixed = 1024 + pstages * patch_bytes + PK_CTRL_BYTES + ident_bytes;
            const int budget = 227 * 1024 - fixed;
            const int sb_max = 2, sb_min = 1;
            const int w_stage = round_up((pair ? FT / 2 : FT) * RB, 1024);
            // flat tasks with one filter tile stage the tile as it lies in memory (k_pad filters per pixel) when that fits,
            // with the pixel pitch made an odd number of 16-byte pieces (no bank conflicts between neighbouring pixels;
            // 32-byte pixels conflict two-way and still gain, measured)
            const int stage_bytes = dense ? dense_bytes : MT * PK_BLOCK_BYTES;
            int staging_bufs = sb_max, wstages = 0, resident = 0, wgroup = g.kS;
            // resident filters when the whole set of this filter tile fits
            if (tiles_n == 1 && RS * cblks <= PK_MAX_WSTAGES) {
                for (int sb = sb_max; sb >= sb_min && !resident; --sb)
                    if (RS * cblks * w_stage + sb * stage_bytes <= budget) { resident = 1; staging_bufs = sb; wstages = RS * cblks; }
            }
            if (!resident) {
                // Streamed filters: a ring of filter rows, at least two, with one barrier each (3x3 301 -> 250 4x4 at 128 images
                // 12.2 us, tap by tap 14.8; 128 -> 89 28x28 at 64 images 17.9 and 19.4).  Taps one by one only where two rows do
                // not fit (256 filters, for instance), or where the patch ring had to become shallower for it at no gain.
                for (staging_bufs = sb_max; staging_bufs > sb_min && (budget - staging_bufs * stage_bytes) / w_stage < 2 * wgroup;) --staging_bufs;
                if ((budget - staging_bufs * stage_bytes) / w_stage < 2 * wgroup) {
                    wgroup = 1;
                    for (staging_bufs = sb_max; staging_bufs > sb_min && (budget - staging_bufs * stage_bytes) / w_stage < 3;) --staging_bufs;
                }
                wstages = (budget - staging_bufs * stage_bytes) / w_stage;
                if (wstages < 3) continue;
                // (four rows for tiles of whole images, which pass a row in 700 cycles: VGG-16 143.0 -> 141.4 us)
                const int most = ipt || pair ? 12 : 8;
                if (wstages > most) wstages = 2 * wgroup > most ? 2 * wgroup : most;
                wstages -= wstages % wgroup;
            }
            if (dense && staging_bufs != 2) continue;
            // the fused 3x3 pool runs on its own warps only beside two staging buffers, which is worth more than a deeper ring
            if (pool3 && staging_bufs != 2 && pstages > 2) continue;
            const long long tiles = (ipt ? ceil_div(g.vN, ipt) : (long long)g.vN * tiles_per_img) * tiles_n;
            const long long tiles_of_pairs = ((ipt ? ceil_div(g.vN, ipt) : (long long)g.vN * tiles_per_img) + 1) / 2 * tiles_n;
            const double waves = (double)(pair ? ceil_div(tiles_of_pairs, 74) : ceil_div(tiles, 148));
            double tile = tile_cycles(MT, FT, RS, cblks, ksteps_last, RB, Wp, TH, g.kR, resident != 0, acc_bufs, pair);
            // between two filter barriers the tensor pipe idles for as long as its queue of two MMAs is shorter than a wait
            // (measured: 221 cycles with 64 filters, 117 with 128, 65 with 192; the second issuing warp hides most of it)
            if (!resident && !g.flat) tile += cblks * (RS / wgroup) * (MT == 2 ? 60.0 : FT < 200 ? 280.0 - 1.2 * FT : 40.0);
            // a stage's round trip through both CTAs is longer than two filter rows
            if (pair && !resident) tile += cblks * (RS / wgroup) * (wstages >= 3 * wgroup ? 0.0 : 200.0);
            if (ipt) tile -= cblks * Wp * (g.kR - 1) * RB / 128.0;     // (no border rows beside the TH counted)
            if (res_blocks_plan && !dense) tile += res_blocks_plan * (MT * 4 * 48.0 + TH * Wp);   // residual MMAs and their loads
            double t = waves * tile;
            if (resident) t += RS * cblks * FT;    // one-time filter load
            if (staging_bufs == 1 && !g.flat) t += ((FT + 63) / 64) * 900.0;     // the last tile's stores, one after the other
            // what the estimate leaves out, fitted to 25 shapes: waits across the pair, a cluster's start
            if (pair) t = 1.15 * t + 800.0;
            if (t < best_of[pair]) {
                best_of[pair] = t;
                if (pair) pair_rounds = waves;
                tiling_of[pair] = {MT, TH, FT, tiles_n, tiles_per_img, wstages, resident, acc_bufs, staging_bufs, patch_bytes, TW, tiles_w, step_h, step_w, org, pstages, dense, stage_bytes, dense_pitch, ipt, wgroup, pair};
            }
            if (!pair && (resident || wgroup == g.kS)) break;      // the deepest patch ring beside which the filters fit
          }
        }
      }
    }
    // Where pairs begin.  The estimate says by how much they gain to within 6 %, and what it leaves out weighs most where a block goes
    // through few channel blocks, all its rounds together: pairs that go through one or two have to promise 4 %, through three 5 %, and filters that could
    // stay, 97 of them and more, 3 %.  Not so where a single block would take its filters tap by tap (256 of them, for instance): by themselves
    // such tasks say the same, but in networks they are the slower ones, 102 -> 256 14x14 with a residual, batch 40, by 6 us a task.
    // By themselves, in graphs, both ways in turn, 734 shapes that the cheaper estimate alone gave to pairs (16 to 512 channels and filters, 4x4 to 56x56, batch 1
    // to 128): 60 took more than 5 % longer than as single blocks, of those that are left 28; none that gains 2 % is given up.  128 -> 179 12x12, batch 64,
    // 10.4 us single and 11.2 as pairs; 60 -> 152 56x56, batch 128, 70 and 83; 131 -> 203 28x28, batch 64, 35.1 and 29.6.  Networks (us, single blocks
    // everywhere / the estimate alone / this line): ResNet-18 with 50 % kept, batch 20, 182.9 / 189.6 / 183.2; with 60 %, batch 48, 289.5 / 279.0 / 276.7, block outputs
    // pruned too 258.3 / 258.1 / 254.3; with 70 %, batch 64, 324.1 / 313.8 / 314.6.  256 -> 179 14x14, batch 64, stays a pair: by itself 16.1 us instead of
    // 15.1, in that network 1.3 us less.
    const PatchTiling &single = tiling_of[0], &paired = tiling_of[1];
    const double blocks_through = pair_rounds * cblks;
    double promise = 1.0;
    if (single.wgroup == g.kS && paired.FT > 96) {      // (79 of 79 pairs of up to 96 filters gain)
        if (paired.resident) promise = 0.97;
        if (blocks_through <= 3) promise = blocks_through <= 2 ? 0.96 : 0.95;
    }
    const bool pairs = best_of[0] >= 1e30 || best_of[1] < best_of[0] * promise;
    const double best = best_of[pairs ? 1 : 0];
    const PatchTiling bt = tiling_of[pairs ? 1 : 0];
    if (best >= 1e30) return CPRUNE_ERR_UNSUPPORTED;
    // share of accumulator rows that hold real pixels; below one half the im2col kernel is the better choice
    const long long tiles_m = bt.ipt ? ceil_div(g.vN, bt.ipt) : (long long)g.vN * bt.tiles_per_img;
    const double fill = (double)g.vP * g.vQ * g.vN / ((double)tiles_m * 128 * bt.MT);
    if (fill < 0.5) return CPRUNE_ERR_UNSUPPORTED;
    // too few tiles for the SMs: the im2col kernel can split the reduction over more CTAs
    if (tiles_m * bt.tiles_n < 64) return CPRUNE_ERR_UNSUPPORTED;
    plan->patch = 1;
    plan->pt = bt;
    plan->narrow = g.stem;
    plan->orient = 0;
    plan->small_c = 0;
    plan->s_packed = i.S;
    plan->splits = 1;
    plan->ipp = 0;
    plan->partial_bytes = 0;
    plan->pre_bytes = g.stem ? ((size_t)i.N * g.He * g.WP * 32 + 255) / 256 * 256 : 0;
    plan->fused_pool = (pool || pool3) ? 1 : 0;
    plan->bias_align = bt.tiles_n * bt.FT <= PK_BIAS_FLOATS ? 4 : 8;      // (more filters: read in pairs from global memory)
    i.tile_m = 128 * bt.MT;
    i.tile_n = bt.FT;
    i.tile_k = 64;
    i.stages = bt.pair ? (bt.wstages + 1) / 2 : bt.wstages;      // (of whole filters)
    i.tiles_m = (int)tiles_m;
    i.tiles_n = bt.tiles_n;
    i.k_alloc = bt.tiles_n * bt.FT;
    const int ksteps = (cblks - 1) * 4 + ksteps_last;
    i.padded_flops = 2.0 * (double)i.tiles_m * i.tile_m * (double)i.k_alloc * RS * ksteps * 16.0;
    plan->smem_bytes = 1024 + bt.pstages * bt.patch_bytes + bt.wstages * round_up((bt.pair ? bt.FT / 2 : bt.FT) * RB, 1024) +
                       bt.staging_bufs * bt.stage_bytes + PK_CTRL_BYTES + ((plan->opts.residual && !bt.dense) ? PK_IDENT_BYTES : 0);
    plan->est_us = best / 1900.0 + 4.0;      // cycles at about 1.9 GHz plus launch, set-up and drain
    return CPRUNE_OK;
}

// Regroups an NHWC tensor with C channels per pixel (T = bf16 with 8 channel lanes in memory, or float32 with C) into
// 16-channel bf16 pixels, one per sf x sf block of input pixels, in rows of WP pixels of which the first pad_lo (and
// whatever follows the image) are zero:
//   out[n][h2][pad_lo + w2][(dy * sf + dx) * C + c] = x[n][sf * h2 + dy][sf * w2 + dx][c], other channels zero.
// Two threads per output pixel, eight channels (one 16-byte store) each.
constexpr int RG_ROWS = 4;     // regrouped rows per block

template <typename T>
__global__ void __launch_bounds__(256) regroup_kernel(const T *__restrict__ x, int H, int W, int C, int c_mem, int sf, int pad_lo, int WP,
                                                      uint4 *__restrict__ out) {
    pdl_wait();        // first kernel of a chain: before its successor may start
    pdl_trigger();
    // one block per RG_ROWS regrouped rows of one image: their sf * RG_ROWS input rows are contiguous in memory and are
    // brought into shared memory with 16-byte loads first
    extern __shared__ __align__(16) unsigned char rg_smem[];
    __shared__ int src_off[16];            // regrouped channel -> offset within an sf x sf input block, or -1 (zero)
    T *srow = reinterpret_cast<T *>(rg_smem);
    const int H2 = H / sf, W2 = W / sf;
    const int blocks_per_img = (H2 + RG_ROWS - 1) / RG_ROWS;
    const int n = blockIdx.x / blocks_per_img;
    const int h2_0 = (blockIdx.x - n * blocks_per_img) * RG_ROWS;
    const int nrows = min(RG_ROWS, H2 - h2_0);
    const T *rows = x + ((size_t)n * H + (size_t)sf * h2_0) * W * c_mem;
    const int row_elems = sf * W * c_mem;                // input elements behind one regrouped row
    const int n_elems = nrows * row_elems;
    const size_t n_bytes = (size_t)n_elems * sizeof(T);
    if (threadIdx.x < 16) {
        const int ch = threadIdx.x, blk = ch / C, c = ch - blk * C;
        const int dy = blk / sf, dx = blk - dy * sf;
        src_off[ch] = blk < sf * sf ? (dy * W + dx) * c_mem + c : -1;
    }
    if (((reinterpret_cast<uintptr_t>(rows) | n_bytes) & 15) == 0) {
        const uint4 *src = reinterpret_cast<const uint4 *>(rows);
        uint4 *dst = reinterpret_cast<uint4 *>(rg_smem);
        const int n16 = (int)(n_bytes >> 4);
        // four loads in flight per thread: the block's latency is one round trip to memory, not one per 4 KB
        for (int i0 = threadIdx.x; i0 < n16; i0 += 4 * 256) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + u * 256 < n16) v[u] = __ldg(src + i0 + u * 256);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + u * 256 < n16) dst[i0 + u * 256] = v[u];
        }
    } else {
        for (int i = threadIdx.x; i < n_elems; i += blockDim.x) srow[i] = rows[i];
    }
    __syncthreads();
    uint4 *orow = out + ((size_t)n * H2 + h2_0) * WP * 2;
    const int per_row = WP * 2;
    const int step = sf * c_mem;                         // input elements between neighbouring regrouped pixels
    for (int e = threadIdx.x; e < nrows * per_row; e += blockDim.x) {
        const int r = e / per_row, c = e - r * per_row;
        const int half = c & 1, w2 = (c >> 1) - pad_lo;
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = 0.f;
        if (w2 >= 0 && w2 < W2) {
            const T *in = srow + (size_t)r * row_elems + w2 * step;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int o = src_off[half * 8 + k];
                if (o >= 0) v[k] = (float)in[o];
            }
        }
        const bf16x8 q = pack8(v);
        orow[e] = *reinterpret_cast<const uint4 *>(&q);
    }
}

// Filters of a regrouped stem: out[k][re * Se + se][(dy * sf + dx) * C + c] = w[k][c][sf * re + dy - er][sf * se + dx - es]
// (zero where that tap does not exist), er = sf * pad_lo - pad.  Rows k >= K are zero.
__global__ void __launch_bounds__(256) pack_regrouped_kernel(const float *__restrict__ w, int K, int C, int R, int S, int sf, int Re,
                                                             int Se, int er, int es, int k_alloc, __nv_bfloat16 *__restrict__ out) {
    const size_t total = (size_t)k_alloc * Re * Se * 16;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int ch = (int)(e % 16);
        size_t t = e / 16;
        const int se = (int)(t % Se); t /= Se;
        const int re = (int)(t % Re);
        const int k = (int)(t / Re);
        float v = 0.f;
        const int blk = ch / C, c = ch - blk * C;
        if (k < K && blk < sf * sf) {
            const int dy = blk / sf, dx = blk - dy * sf;
            const int r = sf * re + dy - er, s2 = sf * se + dx - es;
            if (r >= 0 && r < R && s2 >= 0 && s2 < S) v = w[(((size_t)k * C + c) * R + r) * S + s2];
        }
        out[e] = __float2bfloat16_rn(v);
    }
}

cprune_status pack_conv_patch(const cprune_plan *plan, const float *w, void *w_packed, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    PatchGeometry g;
    if (!patch_geometry(i, &g) || !g.stem) return CPRUNE_ERR_INTERNAL;
    const size_t total = (size_t)i.k_alloc * g.Re * g.Se * 16;
    size_t blocks = (total + 255) / 256;
    if (blocks > 148 * 16) blocks = 148 * 16;
    pack_regrouped_kernel<<<(unsigned)blocks, 256, 0, st>>>(w, i.K, i.C, i.R, i.S, g.sf, g.Re, g.Se, g.sf * g.pad_lo - i.pad,
                                                           g.sf * g.pad_lo - i.pad, i.k_alloc, (__nv_bfloat16 *)w_packed);
    CPRUNE_LAUNCH_CHECK("pack_regrouped_kernel");
    return CPRUNE_OK;
}

size_t packed_weight_bytes_patch(const cprune_plan *plan) {
    const cprune_plan_info &i = plan->info;
    PatchGeometry g;
    if (!patch_geometry(i, &g) || !g.stem) return 0;
    return (size_t)i.k_alloc * g.Re * g.Se * 32;
}

cprune_status regroup_stem_input(const cprune_plan *plan, const void *x, int x_is_f32, void *scratch, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    PatchGeometry g;
    if (!patch_geometry(i, &g) || !g.stem || !x || !scratch) return CPRUNE_ERR_INVALID_ARG;
    const unsigned blocks = (unsigned)(i.N * ((g.He + RG_ROWS - 1) / RG_ROWS));
    const size_t row_bytes = (size_t)RG_ROWS * g.sf * i.W * (x_is_f32 ? (size_t)i.C * 4 : (size_t)i.c_pad * 2);
    if (row_bytes > 48 * 1024) return CPRUNE_ERR_UNSUPPORTED;     // planning keeps such images off this path
    if (x_is_f32)
        CPRUNE_CUDA_CHECK(launch_chained(regroup_kernel<float>, dim3(blocks), dim3(256), row_bytes, st, (const float *)x, i.H, i.W, i.C, i.C, g.sf, g.pad_lo,
                                         g.WP, (uint4 *)scratch));
    else
        CPRUNE_CUDA_CHECK(launch_chained(regroup_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), row_bytes, st, (const __nv_bfloat16 *)x, i.H, i.W, i.C,
                                         i.c_pad, g.sf, g.pad_lo, g.WP, (uint4 *)scratch));
    return CPRUNE_OK;
}

cprune_status launch_conv_patch(cprune_plan *plan, const void *x, const void *w, const float *b, const void *res, void *y,
                                void *scratch, cudaStream_t st, bool input_regrouped) {
    const cprune_plan_info &i = plan->info;
    const PatchTiling &t = plan->pt;
    PatchGeometry g;
    if (!patch_geometry(i, &g)) return CPRUNE_ERR_INTERNAL;
    // patch row pitch: the tile's width plus the filter's; with stacked images a border column is shared by two rows
    const int Wp = t.ipt ? t.TW + i.pad : t.TW + g.kS - 1;
    const unsigned box_rows = t.ipt ? (unsigned)(i.P + i.pad) : (unsigned)(t.TH + g.kR - 1), box_out = t.ipt ? box_rows : (unsigned)t.TH;
    const unsigned box_imgs = t.ipt ? (unsigned)t.ipt : 1u;
    const void *xe = x;        // the tensor the patch loads read
    if (g.stem) {
        if (!scratch) return CPRUNE_ERR_INVALID_ARG;
        if (!input_regrouped) {
            cprune_status rs = regroup_stem_input(plan, x, 0, scratch, st);
            if (rs != CPRUNE_OK) return rs;
        }
        xe = scratch;
    }
    CUtensorMap tm_x, tm_w, tm_y, tm_res;
    {
        std::lock_guard<std::mutex> lock(plan->mu);
        if (plan->map_x != xe) {
            if (g.stem) {
                // rows of 64 values = four consecutive regrouped pixels; start positions are one pixel (32 bytes) apart
                const unsigned long long dims[4] = {64, (unsigned long long)i.Q, (unsigned long long)g.He, (unsigned long long)i.N};
                const unsigned long long strides[3] = {32, (unsigned long long)g.WP * 32, (unsigned long long)g.He * g.WP * 32};
                const unsigned box[4] = {64, (unsigned)Wp, (unsigned)(t.TH + g.kR - 1), 1};
                cprune_status s = encode_tiled_bf16_swz(&plan->tm_a, xe, 4, dims, strides, box, 128, true);
                if (s != CPRUNE_OK) return s;
            } else {
                const unsigned long long dims[4] = {(unsigned long long)i.c_pad, (unsigned long long)g.vW, (unsigned long long)g.vH,
                                                    (unsigned long long)g.vN};
                const unsigned long long strides[3] = {(unsigned long long)i.c_pad * 2, (unsigned long long)g.vW * i.c_pad * 2,
                                                       (unsigned long long)g.vH * g.vW * i.c_pad * 2};
                const unsigned box[4] = {64, (unsigned)Wp, box_rows, box_imgs};
                cprune_status s = encode_tiled_bf16_swz(&plan->tm_a, xe, 4, dims, strides, box, 128, true);
                if (s != CPRUNE_OK) return s;
            }
            plan->map_x = xe;
        }
        if (plan->map_w != w) {
            // filters [k_alloc][taps][channels of a tap]; a stem's tap is a filter row: Se pixels of 16 channels
            const unsigned long long ctap = g.stem ? (unsigned long long)g.Se * 16 : (unsigned long long)i.c_pad;
            const unsigned long long taps = (unsigned long long)(g.kR * g.kS);
            const unsigned long long dims[3] = {ctap, taps, (unsigned long long)i.k_alloc};
            const unsigned long long strides[2] = {ctap * 2, taps * ctap * 2};
            const unsigned box[3] = {64, 1, (unsigned)(t.pair ? t.FT / 2 : t.FT)};
            cprune_status s = encode_tiled_bf16_swz(&plan->tm_b, w, 3, dims, strides, box, 128, true);
            if (s != CPRUNE_OK) return s;
            plan->map_w = w;
        }
        if (plan->map_y != y) {
            // output [N][P][Q][k_pad]; a store is 64 filters x Wp pixels x TH rows (see the epilogue).  With a fused
            // pool the kernel stores by hand and the map is not used.
            const unsigned long long dims[4] = {(unsigned long long)i.k_pad, (unsigned long long)g.vOW, (unsigned long long)g.vOH,
                                                (unsigned long long)g.vN};
            const unsigned long long strides[3] = {(unsigned long long)i.k_pad * 2, (unsigned long long)g.vOW * i.k_pad * 2,
                                                   (unsigned long long)g.vOH * g.vOW * i.k_pad * 2};
            const bool dense_tiled = t.dense && t.dense_pitch != i.k_pad * 2;      // the whole staged tile, unswizzled
            const unsigned box[4] = {dense_tiled ? (unsigned)(t.dense_pitch / 2) : 64u, dense_tiled ? (unsigned)t.TW : (unsigned)Wp,
                                     dense_tiled ? 1u : box_out, box_imgs};
            cprune_status s = encode_tiled_bf16_swz(&plan->tm_y, y, 4, dims, strides, box, dense_tiled ? 0 : 128, false);
            if (s != CPRUNE_OK) return s;
            plan->map_y = y;
        }
        if (res && plan->map_res != res) {
            const unsigned long long dims[4] = {(unsigned long long)i.k_pad, (unsigned long long)g.vQ, (unsigned long long)g.vP,
                                                (unsigned long long)g.vN};
            const unsigned long long strides[3] = {(unsigned long long)i.k_pad * 2, (unsigned long long)g.vQ * i.k_pad * 2,
                                                   (unsigned long long)g.vP * g.vQ * i.k_pad * 2};
            const bool dense_tiled = t.dense && t.dense_pitch != i.k_pad * 2;
            const unsigned box[4] = {dense_tiled ? (unsigned)(t.dense_pitch / 2) : 64u, dense_tiled ? (unsigned)t.TW : (unsigned)Wp,
                                     dense_tiled ? 1u : box_out, box_imgs};
            cprune_status s = encode_tiled_bf16_swz(&plan->tm_res, res, 4, dims, strides, box, dense_tiled ? 0 : 128, true);
            if (s != CPRUNE_OK) return s;
            plan->map_res = res;
        }
        std::memcpy(&tm_x, &plan->tm_a, sizeof(CUtensorMap));
        std::memcpy(&tm_w, &plan->tm_b, sizeof(CUtensorMap));
        std::memcpy(&tm_y, &plan->tm_y, sizeof(CUtensorMap));
        std::memcpy(&tm_res, res ? &plan->tm_res : &plan->tm_y, sizeof(CUtensorMap));
    }
    // the shared-memory limit of a kernel is a per-device attribute
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};
    {
        int dev = 0;
        CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            const void *kernels[] = {(const void *)conv_patch_kernel<PK_GENERAL, false>, (const void *)conv_patch_kernel<PK_GENERAL, false, false, 3>, (const void *)conv_patch_kernel<PK_GENERAL, false, true, 3>, (const void *)conv_patch_kernel<PK_GENERAL, false, true>,
                                     (const void *)conv_patch_kernel<PK_GENERAL, true>, (const void *)conv_patch_kernel<PK_GENERAL, true, false, 3>, (const void *)conv_patch_kernel<PK_GENERAL, true, true, 3>,  (const void *)conv_patch_kernel<PK_GENERAL, true, true>,
                                     (const void *)conv_patch_kernel<PK_TAPS, false>,    (const void *)conv_patch_kernel<PK_TAPS, false, true>,
                                     (const void *)conv_patch_kernel<PK_GENERAL, false, false, 3, true>, (const void *)conv_patch_kernel<PK_GENERAL, false, true, 3, true>,
                                     (const void *)conv_patch_kernel<PK_GENERAL, true, false, 3, true>, (const void *)conv_patch_kernel<PK_GENERAL, true, true, 3, true>,
                                     (const void *)conv_patch_kernel<PK_TAPS, false, false, 3, true>, (const void *)conv_patch_kernel<PK_TAPS, false, true, 3, true>,
                                     (const void *)conv_patch_kernel<PK_FLAT, false>,    (const void *)conv_patch_kernel<PK_FLAT, true>,
                                     (const void *)conv_patch_kernel<PK_DENSE, false>,   (const void *)conv_patch_kernel<PK_DENSE, true>,
                                     (const void *)conv_patch_kernel<PK_POOL3, false>,   (const void *)conv_patch_kernel<PK_POOL3, true>};
            for (const void *k : kernels) CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            attr_set[dev] = true;
        }
    }
    PatchParams p;
    p.P = g.vP; p.Q = g.vQ; p.Wp = Wp; p.TH = t.TH; p.tiles_per_img = t.tiles_per_img;
    p.TW = t.TW; p.tiles_w = t.tiles_w; p.step_h = t.step_h; p.step_w = t.step_w; p.org = t.org;
    p.out_h = g.vOH; p.out_w = g.vOW;
    p.ipt = t.ipt; p.imgs = g.vN;
    // v * ceil(2^32 / d) / 2^32 has the integer part v / d as long as v * d < 2^32 (the error of the reciprocal is below 1 / 2^32)
    const auto reciprocal = [](long long d, long long most) {
        return d > 1 && d * most < (1ll << 32) ? (uint32_t)(((1ull << 32) + d - 1) / d) : 0u;
    };
    p.img_mul = reciprocal(t.tiles_per_img, i.tiles_m);
    p.row_mul = reciprocal(t.tiles_w, t.tiles_per_img);
    p.tiles_m = i.tiles_m; p.tiles_n = i.tiles_n; p.FT = t.FT; p.MT = t.MT; p.R = g.kR; p.S = g.kS; p.pad = g.pad_lo; p.pad_w = g.pad_w;
    p.cblks = g.cblks;
    p.ksteps_last = g.ksteps_last;
    p.k_pad = i.k_pad;
    p.act = plan->opts.activation;
    p.wgroup = t.wgroup; p.wstages = t.wstages; p.pstages = t.pstages; p.resident = t.resident; p.acc_bufs = t.acc_bufs; p.staging_bufs = t.staging_bufs;
    p.pool = plan->fused_pool ? plan->opts.pool : 0;
    p.patch_bytes = t.patch_bytes;
    p.patch_box_bytes = Wp * (int)(box_rows * box_imgs) * 128;
    p.rb16 = 8;
    p.dense = t.dense; p.stage_bytes = t.stage_bytes; p.dense_pitch = t.dense_pitch;
    p.w_stage_bytes = t.FT * (t.pair ? 64 : 128);
    p.bias = b;
    // dense staging takes the residual through the staging buffer; everywhere else the MMA warps add it
    p.res = t.dense ? (const __nv_bfloat16 *)res : nullptr;
    p.res_blocks = (res && !t.dense) ? (t.FT + 63) / 64 : 0;
    p.y = (__nv_bfloat16 *)y;
    p.status = device_status_word();
    if (!p.status) return cuda_fail(cudaGetLastError(), "status word");
    const int total = i.tiles_m * i.tiles_n;
    if (total == 0) return CPRUNE_OK;
    int sms = 148, dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
    const int pair_items = (i.tiles_m + 1) / 2 * i.tiles_n;
    const int grid = t.pair ? 2 * (pair_items < sms / 2 ? pair_items : sms / 2) : total < sms ? total : sms;
    // a fused 3x3 pool with two staging buffers: the instantiation with separate pooling warps
    const bool split_pool = p.pool == CPRUNE_POOL_MAX3X3S2 && t.staging_bufs == 2 && !res && !(plan->opts.flags & CPRUNE_FLAG_POOL_ON_EPILOGUE_WARPS);
    // One instantiation per kind of epilogue and of filter set, and for 3x3 filters: a role is one warp that fetches its
    // instructions alone, and each is faster the less code lies between its loops.  One kernel for all / now (us, 64 images):
    // 1x1 24 -> 108 56x56 20.2 / 17.6, 96 -> 432 14x14 10.7 / 9.6, 32 -> 16 112x112 19.7 / 18.8, 3x3 512 -> 358 7x7 20.5 / 18.2,
    // 64 -> 44 56x56 20.8 / 19.9, 131 -> 203 28x28 37.0 / 36.2.
    const auto launch = [&](auto kernel, int mode) {
        return launch_chained_as(t.pair != 0, kernel, dim3(grid), dim3(pk_threads(mode)), (size_t)plan->smem_bytes, st, tm_x, tm_w, tm_y, tm_res, p);
    };
    const bool r = t.resident != 0, pooled = p.pool != 0;
    cudaError_t e;
    if (t.pair && r) e = pooled ? launch(conv_patch_kernel<PK_GENERAL, true, true, 3, true>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, true, false, 3, true>, PK_GENERAL);
    else if (t.pair && t.wgroup == 3) e = pooled ? launch(conv_patch_kernel<PK_GENERAL, false, true, 3, true>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, false, false, 3, true>, PK_GENERAL);
    else if (t.pair) e = pooled ? launch(conv_patch_kernel<PK_TAPS, false, true, 3, true>, PK_TAPS) : launch(conv_patch_kernel<PK_TAPS, false, false, 3, true>, PK_TAPS);
    else if (t.dense) e = r ? launch(conv_patch_kernel<PK_DENSE, true>, PK_DENSE) : launch(conv_patch_kernel<PK_DENSE, false>, PK_DENSE);
    else if (g.flat) e = r ? launch(conv_patch_kernel<PK_FLAT, true>, PK_FLAT) : launch(conv_patch_kernel<PK_FLAT, false>, PK_FLAT);
    else if (split_pool) e = r ? launch(conv_patch_kernel<PK_POOL3, true>, PK_POOL3) : launch(conv_patch_kernel<PK_POOL3, false>, PK_POOL3);
    else if (g.kR == 3 && g.kS == 3 && r) e = pooled ? launch(conv_patch_kernel<PK_GENERAL, true, true, 3>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, true, false, 3>, PK_GENERAL);
    else if (g.kR == 3 && g.kS == 3 && t.wgroup == 3) e = pooled ? launch(conv_patch_kernel<PK_GENERAL, false, true, 3>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, false, false, 3>, PK_GENERAL);
    else if (r) e = pooled ? launch(conv_patch_kernel<PK_GENERAL, true, true>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, true>, PK_GENERAL);
    else if (t.wgroup == 1) e = pooled ? launch(conv_patch_kernel<PK_TAPS, false, true>, PK_TAPS) : launch(conv_patch_kernel<PK_TAPS, false>, PK_TAPS);
    else e = pooled ? launch(conv_patch_kernel<PK_GENERAL, false, true>, PK_GENERAL) : launch(conv_patch_kernel<PK_GENERAL, false>, PK_GENERAL);
    CPRUNE_CUDA_CHECK(e);
    return CPRUNE_OK;
}

}  // namespace cprune
