// First conv task of a model (3-channel stem, stride 1 or 2) straight from the float32 image: cast, convolution, bias,
// activation and, if the task asks for it, the 3x3 stride-2 max-pool in one pass over the image (paper Sec. 3.4: a task is
// the fused subgraph).
//
// The pixels are on the column side of the MMA and the filters on its 128 rows: D = 128 / KF conv rows of KF (32, 64 or 128)
// filters each, so that the rows are full for the 16 to 64 filters of a pruned stem (fewer where the tiles of a large image would not
// fit; the rows left over go nowhere).  Those D conv rows read the same
// RH = stride * (D - 1) + R input rows; a filter of conv row dy is packed with zero taps where its window does not reach.
//   K order     per input row, the 3 S values of a window one after the other, filled up with zeros to one MMA step (16 values, S <= 5)
//               or two.  A 128-byte operand row holds the windows of one output column in `per` (1, 2 or 4) neighbouring input rows.
//   filters     are the A operand and stay in tensor memory, 8 columns per MMA step: the MMAs read 32 bytes a column of the
//               operand tile and nothing else from shared memory, whose port every other role needs too (from shared memory, 128 more
//               rows an MMA and 16 KB a tile: with the former epilogue 41.1 instead of 40.4 us, and 6 tiles in the ring instead of 11).
//   loads       (1 warp) float32 rows by bulk copies, a few tiles ahead.
//   converters  (8 warps) read every output column's window from them, as pairs of floats where windows begin at an odd pixel (stride 2, odd
//               padding) and one by one elsewhere, and store it as bf16 into a swizzled operand tile.  (Overlapping windows are converted
//               and stored once per column: the MMA fetches one row of its operand's swizzle width per cycle, and with rows read in
//               place through an unswizzled descriptor the 7x7 stem of 64 images took 55 us.  A row buffer of bf16 pixels between
//               rows and windows converts every pixel once, but its meeting of eight warps per tile made a chain of 1600 cycles a tile; now
//               they meet nowhere and a tile takes 800.  The loads have to be predicated by hand: as branches they took 580 cycles of
//               a tile, now 170.)  Tiles form a ring; rows and columns outside the image are zeros.  The converters also say of every
//               tile whether it holds a pixel that is no number (infinite or NaN as a bf16 value).
//   MMA         (2 warps, one per accumulator, taking turns) one step = D conv rows: N = Q columns, K = RH windows.  One warp alone
//               leaves the tensor pipe idle between the tiles it waits for and commits: 48.0 instead of 41.1 us.  A tile is freed by
//               both.  Conv rows meet the input rows outside their window with zero taps, which is nothing unless a pixel is no number: the
//               rows of such a tile go to the accumulator lanes that want them alone (always doing so cost the pooled stem 7 us of 46).
//   epilogue    (8 warps) reads accumulators as 8 x 8 matrices and stores them transposed with stmatrix.  Without a pool the output rows of
//               a step are contiguous and leave as one bulk copy (copied by the threads: 24.2 instead of 22.0 us).  With the pool every conv
//               row leaves pair maxima and its odd columns; after one meeting a thread takes the maxima over windows of 8 filters, keeping
//               the odd conv row for the next step in registers.  Its loops are not unrolled: the roles share the instruction cache (39.4
//               instead of 40.6 us).
// A block works through consecutive steps; with a pool it recomputes one step where it starts inside an image (the odd conv
// row above).
// What bounds it: the epilogue's chain, whose warps share the issue slots (45 % of them busy at 8 images, 33 % before) with the converters'.  A
// step of the pooled 7x7 stem of 224x224 images takes 2400 cycles, of which the epilogue works 1950, the converters 1500 and the MMAs 1010.
// The plain 3x3 stem is at 4.1 TB/s (of 90 MB, 51 written).
// Stem of 64 224x224 images inside the network: 7x7 stride 2, 64 filters, pooled 49.6 us before the changes above, 38.0 now;
// 3x3 stride 2, 32 filters 29.5 and 22.0; 20 images 13.6 and 10.6; one image, pooled 9.4 and 8.2.
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "plan.h"
#include "sm100_ptx.cuh"

namespace cprune {

constexpr int ST_EPI_WARPS = 8, ST_CONV_WARPS = 8;
constexpr int ST_MMA_WARP = ST_EPI_WARPS + ST_CONV_WARPS;
constexpr int ST_MMA_WARPS = 2;           // each has one of the two accumulators
constexpr int ST_LOAD_WARP = ST_MMA_WARP + ST_MMA_WARPS;
constexpr int ST_THREADS = (ST_LOAD_WARP + 1) * 32;
constexpr int ST_MAX_RING = 12;           // operand tiles
constexpr int ST_RAW = 4;                 // tiles of float32 rows in flight

struct StemParams {
    const float *x;
    const uint4 *w;
    const float *bias;
    __nv_bfloat16 *y;
    int H, W, P, Q, out_h, out_w;
    int stride, pad;
    int D, KF, RH, N;
    int ksteps, accs, acc_stride;         // MMA steps (16 values) of a step, accumulators, their distance in columns
    int per, tiles, adv;                  // input rows per operand tile, tiles a step reads, tiles from step to step
    int cps, used;                        // 16-byte pieces of an input row's window in an operand row; MMA steps (16 values) that hold any of it
    int tile_bytes, raw_bytes, ring, stage_bytes;
    int steps_per_img, total_steps;
    int k_pad, S;
    unsigned long long lanes_on, lanes_new;   // 4 bits per input row of a step: accumulator lanes (32 each) whose window holds it, and begins with it
    int *status;
};

// A block's steps, image by image: `first` is the first step to compute (one earlier than wanted when the pool needs the conv
// row above), `from` the first to store, `to` one past the last.
struct StemSegment {
    int n, first, from, to;
};
template <bool POOL>
__device__ __forceinline__ bool next_segment(const StemParams &p, int &t, int t1, StemSegment &s) {
    if (t >= t1) return false;
    s.n = t / p.steps_per_img;
    s.from = t - s.n * p.steps_per_img;
    s.to = min(p.steps_per_img, s.from + (t1 - t));
    s.first = POOL && s.from > 0 ? s.from - 1 : s.from;
    t += s.to - s.from;
    return true;
}

template <int ACT>
__device__ __forceinline__ uint32_t act_pack2(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);      // 0 and 6 are bf16 values: the clamp commutes with the rounding
    if (ACT != CPRUNE_ACT_NONE) v = __hmax2(v, __floats2bfloat162_rn(0.f, 0.f));
    if (ACT == CPRUNE_ACT_RELU6) v = __hmin2(v, __floats2bfloat162_rn(6.f, 6.f));
    return *reinterpret_cast<const uint32_t *>(&v);
}
__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 v = __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&a), *reinterpret_cast<const __nv_bfloat162 *>(&b));
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ uint4 max8(const uint4 &a, const uint4 &b) { return make_uint4(max2(a.x, b.x), max2(a.y, b.y), max2(a.z, b.z), max2(a.w, b.w)); }

// a + 0 * v for bf16 pairs: a zero stays a zero unless v is infinite or NaN
__device__ __forceinline__ uint32_t times_zero2(uint32_t v, uint32_t a) {
    asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(a) : "r"(v), "r"(0u));
    return a;
}

// loads without branches; zeros where `on` is
__device__ __forceinline__ void ld_shared_if(float &a, float &b, uint32_t addr, uint32_t on) {
    a = b = 0.f;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.shared.v2.f32 {%0, %1}, [%2];\n\t}" : "+f"(a), "+f"(b) : "r"(addr), "r"(on));
}
__device__ __forceinline__ void ld_shared_if(float &a, uint32_t addr, uint32_t on) {
    a = 0.f;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.shared.f32 %0, [%1];\n\t}" : "+f"(a) : "r"(addr), "r"(on));
}
__device__ __forceinline__ void epilogue_sync() { asm volatile("barrier.sync 1, %0;" ::"n"(ST_EPI_WARPS * 32) : "memory"); }

// SW: the filters' width where windows begin at an odd pixel (stride 2, odd padding and width: their pixels are read as pairs of
// floats, 8-byte aligned one float ahead of the window), else 0
template <int ACT, bool POOL, int SW>
__global__ void __launch_bounds__(ST_THREADS, 1) conv_stem_kernel(const StemParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_base = smem_u32(smem_raw);
    const uint32_t base = (raw_base + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_base);
    uint8_t *ring = smem;
    uint8_t *raw = ring + (uint32_t)(p.ring * p.tile_bytes);
    uint8_t *stage = raw + ST_RAW * p.raw_bytes;
    uint8_t *ctrl = stage + (POOL ? 4 : 2) * p.stage_bytes;
    const uint32_t ctrl0 = smem_u32(ctrl);
    auto full = [&](int s) { return ctrl0 + 8u * s; };
    auto empty = [&](int s) { return ctrl0 + 96u + 8u * s; };
    auto tfull = [&](int a) { return ctrl0 + 192u + 8u * a; };
    auto tempty = [&](int a) { return ctrl0 + 208u + 8u * a; };
    const uint32_t wbar = ctrl0 + 224u;
    auto rfull = [&](int s) { return ctrl0 + 256u + 8u * s; };
    auto rempty = [&](int s) { return ctrl0 + 288u + 8u * s; };
    uint32_t *tmem_slot = (uint32_t *)(ctrl + 248);
    volatile int *abort_flag = (volatile int *)(ctrl + 252);
    uint8_t *flags = ctrl + 320;           // 16 tiles (more than the ring) x converter warps

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int t0 = (int)((long long)p.total_steps * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)p.total_steps * (blockIdx.x + 1) / gridDim.x);
    // float32 rows of a tile that lie inside the image
    auto rows_of = [&](int tile, int &r0, int &r1) {
        r0 = max(0, tile * p.per - p.pad);
        r1 = min(p.H, (tile + 1) * p.per - p.pad);
    };
    // position of the bulk copies, up to ST_RAW tiles ahead of the conversion (first lane of the loading warp only)
    int lt = t0, ltile = 0, lslot = 0;
    StemSegment ls = {0, 0, 0, 0};
    bool lmore = false;
    auto load_next = [&]() {
        int r0, r1;
        rows_of(ltile, r0, r1);
        const uint32_t bytes = r1 > r0 ? (uint32_t)((r1 - r0) * p.W) * 12u : 0u;
        mbar_expect_tx(rfull(lslot), bytes);
        if (bytes)
            bulk_load(smem_u32(raw) + (uint32_t)(lslot * p.raw_bytes + (r0 - (ltile * p.per - p.pad)) * p.W * 12), p.x + ((size_t)ls.n * p.H + r0) * p.W * 3,
                      bytes, rfull(lslot));
        if (++lslot == ST_RAW) lslot = 0;
        if (++ltile == (ls.to - 1) * p.adv + p.tiles) {
            lmore = next_segment<POOL>(p, lt, t1, ls);
            ltile = ls.first * p.adv;
        }
    };
    if (warp == ST_LOAD_WARP && lane == 0) {
        for (int s = 0; s < p.ring; ++s) { mbar_init(full(s), ST_CONV_WARPS); mbar_init(empty(s), p.accs); }
        for (int s = 0; s < ST_RAW; ++s) { mbar_init(rfull(s), 1); mbar_init(rempty(s), ST_CONV_WARPS); }
        for (int a = 0; a < 2; ++a) { mbar_init(tfull(a), 1); mbar_init(tempty(a), ST_EPI_WARPS); }
        mbar_init(wbar, ST_EPI_WARPS);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        pdl_wait();                        // the image
        lmore = next_segment<POOL>(p, lt, t1, ls);
        ltile = ls.first * p.adv;
        for (int s = 0; s < ST_RAW && lmore; ++s) load_next();
    }
    // what the MMA reads and the converters do not write (columns beyond Q, the fourth piece of a window) has to be finite, or zero
    for (int b = 0; b < p.ring; ++b)
        for (int e = tid; e < p.tile_bytes / 16; e += ST_THREADS)
            if ((e >> 3) >= p.Q || (((e ^ (e >> 3)) & (p.cps - 1)) == 3)) ((uint4 *)(ring + (uint32_t)(b * p.tile_bytes)))[e] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == ST_MMA_WARP) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
        // first kernel of a chain: before its successor may start
        pdl_wait();
        pdl_trigger();
    }
    fence_async_smem();                    // the tensor core reads the zeros
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot, tmem_w = tmem_base + (uint32_t)(p.accs * p.acc_stride);
    if (warp >= ST_EPI_WARPS && warp < ST_MMA_WARP) {
        // ------------------------------------------------------------------ converters
        // what this thread converts of every tile: at most two windows
        constexpr int THREADS = ST_CONV_WARPS * 32;
        constexpr int LOADS = SW ? (3 * SW + 1) / 2 : 24;      // pairs of floats, or floats
        constexpr int WORDS = SW ? (3 * SW + 1) / 2 : 12, PIECES = (WORDS + 3) / 4;
        const int ctid = tid - ST_EPI_WARPS * 32, row_len = p.W * 12;
        const int pieces = SW ? PIECES : min(PIECES, 2 * p.used);
        const bool two = p.per * p.Q > THREADS;
        const uint32_t raw0 = smem_u32(raw);
        int win_r[2], src[2];
        uint32_t dst[2][PIECES], mask[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = ctid + u * THREADS;
            const int r = e / p.Q, q = e - r * p.Q;
            const int off = (q * p.stride - p.pad) * 12 - (SW ? 4 : 0);
            win_r[u] = r < p.per ? r : -1;
            src[u] = r * row_len + off;
            mask[u] = 0u;
#pragma unroll
            for (int i = 0; i < LOADS; ++i) {                  // those of the window that lie inside the row
                const int at = off + i * (SW ? 8 : 4);
                if (at >= 0 && at < row_len && (SW || i < 3 * p.S)) mask[u] |= 1u << i;
            }
#pragma unroll
            for (int c = 0; c < PIECES; ++c) dst[u][c] = sub_off(q, r * p.cps + c);
        }
        int t = t0, slot = 0, rslot = 0, seq = 0;
        uint32_t phase = 0, rphase = 0;
        bool ok = true;
        StemSegment sg;
        while (ok && next_segment<POOL>(p, t, t1, sg)) {
            for (int b = sg.first * p.adv; b < (sg.to - 1) * p.adv + p.tiles; ++b) {
                ok = __all_sync(0xffffffffu, mbar_wait(rfull(rslot), rphase, abort_flag, p.status));
                if (!ok) break;
                const uint32_t rows = raw0 + (uint32_t)(rslot * p.raw_bytes);
                const int row0 = b * p.per - p.pad;
                float f[2][SW ? 2 * LOADS + 1 : LOADS];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u == 1 && !two) break;
                    const int row = row0 + win_r[u];
                    const uint32_t on = win_r[u] >= 0 && row >= 0 && row < p.H ? mask[u] : 0u;
#pragma unroll
                    for (int i = 0; i < LOADS; ++i) {
                        if (SW) {
                            ld_shared_if(f[u][2 * i], f[u][2 * i + 1], rows + (uint32_t)(src[u] + i * 8), on & (1u << i));
                        } else {
                            ld_shared_if(f[u][i], rows + (uint32_t)(src[u] + i * 4), on & (1u << i));
                        }
                    }
                    if (SW) f[u][2 * LOADS] = 0.f;
                }
                uint32_t w[2][PIECES * 4], odd[2] = {0u, 0u};      // odd: zeros, or NaN where a pixel is no number
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u == 1 && !two) break;
#pragma unroll
                    for (int i = 0; i < PIECES * 4; ++i) {
                        w[u][i] = i < WORDS ? (SW ? act_pack2<CPRUNE_ACT_NONE>(f[u][2 * i + 1], f[u][2 * i + 2]) : act_pack2<CPRUNE_ACT_NONE>(f[u][2 * i], f[u][2 * i + 1])) : 0u;
                        if (i < WORDS) odd[i & 1] = times_zero2(w[u][i], odd[i & 1]);
                    }
                }
                const bool any_odd = __any_sync(0xffffffffu, ((odd[0] | odd[1]) & 0x7fff7fffu) != 0u);
                if (lane == 0) mbar_arrive(rempty(rslot));
                ok = __all_sync(0xffffffffu, mbar_wait(empty(slot), phase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                uint8_t *dst0 = ring + (uint32_t)(slot * p.tile_bytes);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u == 1 && !two) break;
                    if (win_r[u] < 0) continue;
#pragma unroll
                    for (int c = 0; c < PIECES; ++c)
                        if (SW || c < pieces) *(uint4 *)(dst0 + dst[u][c]) = make_uint4(w[u][4 * c], w[u][4 * c + 1], w[u][4 * c + 2], w[u][4 * c + 3]);
                }
                if (lane == 0) flags[(seq & 15) * ST_CONV_WARPS + (warp - ST_EPI_WARPS)] = any_odd;
                ++seq;
                fence_async_smem();                        // the tensor core reads what these stores wrote
                __syncwarp();
                if (lane == 0) mbar_arrive(full(slot));
                if (++slot == p.ring) { slot = 0; phase ^= 1u; }
                if (++rslot == ST_RAW) { rslot = 0; rphase ^= 1u; }
            }
        }
    } else if (warp == ST_LOAD_WARP) {
        // ------------------------------------------------------------------ float32 rows
        if (lane == 0) {
            uint32_t phase = 0;
            while (lmore) {                                    // (the first ST_RAW tiles were requested above: lslot is 0 again)
                if (!mbar_wait(rempty(lslot), phase, abort_flag, p.status)) break;
                if (lslot == ST_RAW - 1) phase ^= 1u;
                load_next();
            }
        }
        __syncwarp();
    } else if (warp >= ST_MMA_WARP && warp < ST_LOAD_WARP) {
        // ------------------------------------------------------------------ MMA issue
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t ring0 = smem_u32(ring);
        const int used = p.used;                           // MMA steps (16 values) per input row
        uint32_t step_at[4], step_row[4];                  // a tile's MMA steps: offset in its rows (16 bytes), input row
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            step_row[k] = (uint32_t)(used == 2 ? k >> 1 : k);
            step_at[k] = step_row[k] * (uint32_t)p.cps + (uint32_t)(used == 2 ? (k & 1) * 2 : 0);
        }
        const uint32_t ring_lo = desc_lo(ring0), tile_step = (uint32_t)p.tile_bytes >> 4;
        const int mine = warp - ST_MMA_WARP;
        const uint32_t d_tmem = tmem_base + (uint32_t)(mine * p.acc_stride);
        int t = t0, it = 0;                                // it: parity of the segment's first step
        int wslot = 0, seq = 0, fslot = 0;                 // ring slots of the next tile to wait for and to free
        uint32_t acc_phase = 0, wphase = 0, odd = 0;       // odd: ring slots whose tile holds a pixel that is no number
        StemSegment sg;
        // tiles whose slot is filled again; the others are not freed: the arrival of a commit that nobody waits for could come after
        // the block's end
        int refilled = -p.ring;
        for (int u = t0; next_segment<POOL>(p, u, t1, sg);) refilled += (sg.to - sg.first - 1) * p.adv + p.tiles;
        int base_seq = 0;                                  // of the segment's first tile
        bool ok = mine < p.accs && __all_sync(0xffffffffu, mbar_wait(wbar, 0u, abort_flag, p.status));
        tc_fence_after();
        while (ok && next_segment<POOL>(p, t, t1, sg)) {
            const int steps = sg.to - sg.first, total = (steps - 1) * p.adv + p.tiles;
            int have = 0, freed = 0;                       // tiles of the segment that have arrived, that this warp is done with
            auto next_tile = [&]() {
                ok = __all_sync(0xffffffffu, mbar_wait(full(wslot), wphase, abort_flag, p.status));
                if (!ok) return;
                tc_fence_after();
                const uint32_t bit = 1u << wslot;
                odd = *(const volatile unsigned long long *)(flags + (seq++ & 15) * ST_CONV_WARPS) ? odd | bit : odd & ~bit;
                if (++wslot == p.ring) { wslot = 0; wphase ^= 1u; }
                ++have;
            };
            // (a tile is freed by every warp, and by neither before it has arrived: an early arrival would count for its predecessor)
            auto free_up_to = [&](int tile) {
                while (ok && freed < tile) {
                    if (have <= freed) next_tile();
                    if (ok && base_seq + freed < refilled && elect_one()) umma_commit(empty(fslot));
                    __syncwarp();
                    ++freed;
                    if (++fslot == p.ring) fslot = 0;
                }
            };
            for (int r = p.accs == 2 ? (it ^ mine) & 1 : 0; r < steps && ok; r += p.accs) {
                free_up_to(r * p.adv);
                ok = ok && __all_sync(0xffffffffu, mbar_wait(tempty(mine), acc_phase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                const int head = fslot;
                int slot = head;
                for (int j = 0; j < p.tiles; ++j) {
                    if (have <= r * p.adv + j) next_tile();
                    if (!ok) break;
                    const int nk = min(p.per, p.RH - j * p.per) * used;
                    const uint32_t a = tmem_w + (uint32_t)(j * p.per * used * 8), b_lo = ring_lo + (uint32_t)slot * tile_step;
                    const bool done = j < p.accs * p.adv;       // this warp's next step begins behind it
                    if (elect_one()) {
                        if (__builtin_expect(odd != 0u, 0)) {
                            // zero times a pixel that is no number is NaN: only the accumulator lanes whose window holds the row.
                            // A conv row's sums begin with the first tile, which clears all lanes, or with its own first row.
                            const bool odd_first = (odd >> head) & 1u, masked = odd_first || ((odd >> slot) & 1u);
                            const uint32_t on16 = masked ? (uint32_t)(p.lanes_on >> (j * p.per * 4)) : 0xffffu;
                            const uint32_t new16 = odd_first ? (uint32_t)(p.lanes_new >> (j * p.per * 4)) : (j == 0 ? 15u : 0u);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if (k >= nk) break;
                                const uint32_t on = (on16 >> (step_row[k] * 4)) & 15u, fresh = used == 2 && (k & 1) ? 0u : (new16 >> (step_row[k] * 4)) & 15u;
                                const uint32_t b = b_lo + step_at[k];
                                if (on != fresh) umma_bf16_tmem_lanes(d_tmem, a + 8u * k, b, DESC_HI_SW128, idesc, 1u, on ^ fresh);
                                if (fresh) umma_bf16_tmem_lanes(d_tmem, a + 8u * k, b, DESC_HI_SW128, idesc, 0u, fresh);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (k < nk) umma_bf16_tmem(d_tmem, a + 8u * k, b_lo + step_at[k], DESC_HI_SW128, idesc, (j | k) ? 1u : 0u);
                        }
                        if (done && base_seq + r * p.adv + j < refilled) umma_commit(empty(slot));
                        if (j + 1 == p.tiles) umma_commit(tfull(mine));
                    }
                    __syncwarp();
                    if (++slot == p.ring) slot = 0;
                    if (done) { ++freed; fslot = slot; }
                }
                acc_phase ^= 1u;
            }
            free_up_to(total);
            it ^= steps & 1;
            base_seq += total;
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3, half = warp >> 2, m = quarter * 32 + lane;
        const int dy = quarter * 32 / p.KF, k0 = quarter * 32 - dy * p.KF;     // the warp's conv row, first of its 32 filters
        // (rows of filters that a halved D leaves over, D * KF < 128, have no place in the staging buffer; the pool's D is always 2)
        const int filters = POOL || dy < p.D ? p.k_pad - k0 : 0;
        pdl_wait();
        float bias[4];                                         // of filters k0 + lane / 4 + 8 i
#pragma unroll
        for (int i = 0; i < 4; ++i) bias[i] = i * 8 < filters ? __ldg(p.bias + k0 + i * 8 + (lane >> 2)) : 0.f;
        const int units = p.N >> 4;
        const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
        // filters into tensor memory, 8 columns per MMA step, while the first tiles are on their way
        for (int f0 = half; f0 < p.ksteps; f0 += 18) {
            uint4 v[9][2];
#pragma unroll
            for (int i = 0; i < 9; ++i)
                if (f0 + 2 * i < p.ksteps) {
                    const uint4 *src = p.w + ((size_t)(f0 + 2 * i) * 128 + m) * 2;
                    v[i][0] = __ldg(src);
                    v[i][1] = __ldg(src + 1);
                }
#pragma unroll
            for (int i = 0; i < 9; ++i)
                if (f0 + 2 * i < p.ksteps) tmem_st8(tmem_w + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((f0 + 2 * i) * 8), v[i][0], v[i][1]);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(wbar);
        // staged pixels are an odd number of 16-byte pieces apart: the 8 pixels of a matrix that stmatrix stores meet no bank twice
        const int kp8 = p.k_pad >> 3, pitch = (POOL ? kp8 | 1 : kp8) * 16;
        const uint32_t stage0 = smem_u32(stage), dump = ctrl0 + 448u;
        // pieces that this thread copies from there to the output: pixel and piece of the first, advance to the next one
        const int copy_px = tid / kp8, copy_piece = tid - copy_px * kp8;
        const int next_px = ST_EPI_WARPS * 32 / kp8, next_piece = ST_EPI_WARPS * 32 - next_px * kp8;
        int t = t0, acc = 0, buf = 0;
        uint4 above[2];                                        // of this thread's pieces: maxima of the conv row above
        uint32_t acc_phase = 0;
        bool ok = true;                                        // (after a wait that ran out the warp goes on to meet the others, without waiting)
        StemSegment sg;
        while (next_segment<POOL>(p, t, t1, sg)) {
            for (int s = sg.first; s < sg.to; ++s) {
                ok = ok && __all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, p.status, false));
                tc_fence_after();
                const uint32_t t_acc = t_row + (uint32_t)(acc * p.acc_stride);
                if (POOL) {
                    // The warp's conv row, 16 columns of 16 filters at a time, leaves the maxima of columns 2 c and 2 c + 1 and, behind them, the
                    // odd columns by themselves: a window is a pair and the odd column left of it.  Two buffers: one meeting of the warps per step is enough
                    const uint32_t st = stage0 + (uint32_t)((2 * buf + dy) * p.stage_bytes + (lane >> 4) * p.out_w * pitch);
                    const int mi = (lane >> 3) & 1, px0 = ((lane & 7) >> 1) + (lane & 1) * 4;
#pragma unroll 1
                    for (int u = half; u < units; u += 2) {
                        uint32_t c[2][8];
                        tmem_ld_rows16(t_acc + (uint32_t)(u * 16), c[0]);
                        tmem_ld_rows16(t_acc + (16u << 16) + (uint32_t)(u * 16), c[1]);
                        tmem_ld_wait();
                        const int px = u * 8 + px0;
                        const uint32_t at = st + (uint32_t)(px * pitch + (k0 + mi * 8) * 2);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t w[4];
#pragma unroll
                            for (int r = 0; r < 2; ++r) {          // filters of matrix r; columns c and c + 4 of the pooled eight
                                float f[2], o[2];
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    o[e] = __uint_as_float(c[h][4 * e + 2 * r + 1]) + bias[2 * h + r];
                                    f[e] = fmaxf(__uint_as_float(c[h][4 * e + 2 * r]), __uint_as_float(c[h][4 * e + 2 * r + 1])) + bias[2 * h + r];
                                }
                                w[r] = act_pack2<ACT>(f[0], f[1]);
                                w[2 + r] = act_pack2<ACT>(o[0], o[1]);
                            }
                            stmatrix4_trans(px < p.out_w && h * 16 + mi * 8 < filters ? at + (uint32_t)(h * 32) : dump, w);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty(acc));
                    epilogue_sync();                               // the rows are in place
                    // (at most two pieces a thread: 64 columns of 64 filters)
                    const uint8_t *rows = stage + 2 * buf * p.stage_bytes;
                    uint4 *out = (uint4 *)(p.y + ((size_t)sg.n * p.out_h + s) * p.out_w * p.k_pad) + tid;
                    const bool carry = copy_piece + next_piece >= kp8;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int px = copy_px + (i ? next_px + carry : 0), piece = copy_piece + (i ? next_piece - (carry ? kp8 : 0) : 0);
                        if (px >= p.out_w) break;
                        const int e = px * pitch + piece * 16, left = px > 0 ? e + (p.out_w - 1) * pitch : e;
                        const uint4 below = max8(*(const uint4 *)(rows + p.stage_bytes + e), *(const uint4 *)(rows + p.stage_bytes + left));
                        if (s >= sg.from && ok) {
                            uint4 v = max8(max8(*(const uint4 *)(rows + e), *(const uint4 *)(rows + left)), below);
                            if (s > 0) v = max8(v, above[i]);
                            out[i * ST_EPI_WARPS * 32] = v;
                        }
                        above[i] = below;
                    }
                    buf ^= 1;
                } else {
                    const uint32_t st = stage0 + (uint32_t)(buf * p.stage_bytes + dy * p.Q * pitch);
#pragma unroll 1
                    for (int u = half; u < units; u += 2) {
                        if (filters <= 0) break;
                        uint32_t c[2][8];
                        tmem_ld_rows16(t_acc + (uint32_t)(u * 16), c[0]);
                        if (filters > 16) tmem_ld_rows16(t_acc + (16u << 16) + (uint32_t)(u * 16), c[1]);
                        tmem_ld_wait();
                        // matrices: 8 filters (lane bit 3) x 8 columns (lane bit 4)
                        const int px = u * 16 + (lane & 7) + (lane >> 4) * 8;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h * 16 >= filters) continue;
                            uint32_t w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)            // columns 2 (lane % 4) and the next one of half i / 2 of the 16, filters of half i % 2
                                w[i] = act_pack2<ACT>(__uint_as_float(c[h][2 * i]) + bias[2 * h + (i & 1)], __uint_as_float(c[h][2 * i + 1]) + bias[2 * h + (i & 1)]);
                            const int k = h * 16 + ((lane >> 3) & 1) * 8;
                            stmatrix4_trans(px < p.Q && k < filters ? st + (uint32_t)(px * pitch + (k0 + k) * 2) : dump, w);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty(acc));
                    fence_async_smem();
                    // the buffer written next was last read by the previous step's copy
                    if (tid == 0) tma_store_wait_read<0>();
                    epilogue_sync();
                    if (tid == 0 && ok) {
                        const int row = s * p.D;
                        bulk_store(p.y + ((size_t)sg.n * p.out_h + row) * p.out_w * p.k_pad, stage0 + (uint32_t)(buf * p.stage_bytes),
                                   (uint32_t)(min(p.D, p.P - row) * p.out_w * p.k_pad) * 2u);
                        tma_store_commit();
                    }
                    buf ^= 1;
                }
                if (++acc == p.accs) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (!POOL && tid == 0) tma_store_wait_all();           // staged data must be read before the block's memory goes away
    }

    // ---------------------------------------------------------------------- teardown
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land before the memory goes away
    }
    tc_fence_before();
    __syncthreads();
    if (warp == ST_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// Filters: out[MMA step][dy * KF + k][16 values], a step's input row i = step / used (used steps per row), value pixel * 3 + c of it; zero
// where the tap does not exist.
__global__ void __launch_bounds__(256) pack_stem_kernel(const float *__restrict__ w, int K, int R, int S, int stride, int D, int KF, int used,
                                                        int total, __nv_bfloat16 *__restrict__ out) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int step = e >> 11, m = (e >> 4) & 127, j = step / used;
        const int dy = m / KF, k = m - dy * KF;
        const int v = (step - j * used) * 16 + (e & 15), px = v / 3, c = v - px * 3;
        const int r = j - stride * dy;
        float f = 0.f;
        if (dy < D && k < K && r >= 0 && r < R && px < S) f = w[(((size_t)k * 3 + c) * R + r) * S + px];
        out[e] = __float2bfloat16_rn(f);
    }
}

// Decides whether a model runs this first task straight from its float32 image; fills plan->stem.
void plan_conv_stem(cprune_plan *plan) {
    const cprune_plan_info &i = plan->info;
    StemTiling &s = plan->stem;
    s.ok = 0;
    const bool pool = plan->opts.pool == CPRUNE_POOL_MAX3X3S2;
    if (i.groups != 1 || i.C != 3 || i.stride > 2 || plan->opts.residual || plan->opts.pool == CPRUNE_POOL_MAX2X2) return;
    if (plan->opts.kernel != CPRUNE_KERNEL_AUTO || plan->opts.flags) return;
    if ((i.W & 3) || i.Q > 240 || i.k_pad > 128 || i.R > 8 || i.S > 8 || i.pad >= i.S || i.pad >= i.R) return;
    if (pool && (i.k_pad > 64 || (i.P & 1) || (i.Q & 1) || i.Q > 128)) return;
    // Where the other path is as fast or faster (us, with the cast or regrouping pass, before / here): rows of 32 pixels, whose MMAs have
    // few columns (3x3 3 -> 45, 128 images, inside VGG-16: 13.7 / 13.1, the whole network 131.7 / 131.8), and small tasks of the few-pixel
    // kernel (3x3 stride 2, one 224x224 image).
    if (i.Q < 64 || (plan->small && plan->est_us < 6.0)) return;
    s.KF = pool ? 64 : (i.k_pad <= 32 ? 32 : (i.k_pad <= 64 ? 64 : 128));
    s.steps_per_img = 0;
    // rows per step as the filters allow; half as many where the operand tiles or the staged output would not fit
    for (s.D = pool ? 2 : 128 / s.KF; s.D >= 1 && !s.steps_per_img; s.D >>= 1) {
        if (pool && s.D != 2) return;
        const int new_rows = i.stride * s.D;               // input rows from step to step: a power of two
        s.RH = i.stride * (s.D - 1) + i.R;
        s.used = i.S <= 5 ? 1 : 2;                         // 3 values a pixel
        s.slot = 32 * s.used;
        s.ksteps = s.RH * s.used;
        while (128 / s.slot > new_rows) s.slot *= 2;
        s.per = 128 / s.slot;
        s.tiles = (s.RH + s.per - 1) / s.per;
        s.adv = new_rows / s.per;
        if (s.tiles < s.adv) s.tiles = s.adv;              // (filters shorter than the step: the rows between are read, zero taps)
        s.N = round_up(i.Q, 16);
        s.tile_bytes = round_up(s.N * 128, 1024);
        // tensor memory: two accumulators, or one where wide rows and long filters leave no room
        s.acc_stride = round_up(s.N, 32);
        s.accs = 2 * s.acc_stride + s.ksteps * 8 <= 512 ? 2 : 1;
        if (s.accs * s.acc_stride + s.ksteps * 8 > 512) continue;
        s.raw_bytes = round_up(s.per * i.W * 12, 128);
        s.stage_bytes = round_up((pool ? 2 * ((i.k_pad / 8) | 1) : s.D * i.k_pad / 8) * i.out_w * 16, 128);
        if (s.per * i.Q > 2 * ST_CONV_WARPS * 32) continue;
        for (s.ring = ST_MAX_RING; s.ring > s.tiles; --s.ring) {
            s.smem_bytes = 1024 + s.ring * s.tile_bytes + ST_RAW * s.raw_bytes + (pool ? 4 : 2) * s.stage_bytes + 512;
            if (s.smem_bytes <= 227 * 1024) {
                s.steps_per_img = pool ? i.P / 2 : (i.P + s.D - 1) / s.D;
                break;
            }
        }
        if (s.steps_per_img) break;
    }
    if (!s.steps_per_img || (long long)i.N * s.steps_per_img > 0x3fffffffLL) return;
    s.weight_bytes = (size_t)s.ksteps * 4096;
    s.ok = 1;
}

cprune_status pack_conv_stem(const cprune_plan *plan, const float *w, void *w_stem, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    const StemTiling &s = plan->stem;
    const int total = s.ksteps * 2048;
    pack_stem_kernel<<<(unsigned)ceil_div(total, 256), 256, 0, st>>>(w, i.K, i.R, i.S, i.stride, s.D, s.KF, s.used, total, (__nv_bfloat16 *)w_stem);
    CPRUNE_LAUNCH_CHECK("pack_stem_kernel");
    return CPRUNE_OK;
}

template <int ACT, bool POOL, int SW>
static cprune_status launch_stem(const StemParams &p, unsigned grid, size_t smem, cudaStream_t st) {
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};    // the shared-memory limit of a kernel is a per-device attribute
    int dev = 0;
    CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(conv_stem_kernel<ACT, POOL, SW>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            attr_set[dev] = true;
        }
    }
    CPRUNE_CUDA_CHECK(launch_chained(conv_stem_kernel<ACT, POOL, SW>, dim3(grid), dim3(ST_THREADS), smem, st, p));
    return CPRUNE_OK;
}
template <int ACT, bool POOL>
static cprune_status launch_stem_width(const StemParams &p, unsigned grid, size_t smem, cudaStream_t st) {
    if (p.stride == 2 && (p.pad & 1)) {
        if (p.S == 3) return launch_stem<ACT, POOL, 3>(p, grid, smem, st);
        if (p.S == 5) return launch_stem<ACT, POOL, 5>(p, grid, smem, st);
        if (p.S == 7) return launch_stem<ACT, POOL, 7>(p, grid, smem, st);
    }
    return launch_stem<ACT, POOL, 0>(p, grid, smem, st);
}

cprune_status launch_conv_stem(const cprune_plan *plan, const float *x, const void *w_packed, const float *b, void *y, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    const StemTiling &s = plan->stem;
    if (!s.ok || (((uintptr_t)x | (uintptr_t)w_packed) & 15) || ((uintptr_t)b & 3)) return CPRUNE_ERR_INVALID_ARG;
    StemParams p;
    p.x = x; p.w = (const uint4 *)((const char *)w_packed + s.weight_offset); p.bias = b; p.y = (__nv_bfloat16 *)y;
    p.H = i.H; p.W = i.W; p.P = i.P; p.Q = i.Q; p.out_h = i.out_h; p.out_w = i.out_w;
    p.stride = i.stride; p.pad = i.pad;
    p.D = s.D; p.KF = s.KF; p.RH = s.RH; p.N = s.N;
    p.per = s.per; p.tiles = s.tiles; p.adv = s.adv;
    p.cps = s.slot / 16; p.used = s.used; p.ksteps = s.ksteps; p.accs = s.accs; p.acc_stride = s.acc_stride;
    p.tile_bytes = s.tile_bytes; p.raw_bytes = s.raw_bytes; p.ring = s.ring; p.stage_bytes = s.stage_bytes;
    p.steps_per_img = s.steps_per_img; p.total_steps = i.N * s.steps_per_img;
    p.k_pad = i.k_pad; p.S = i.S;
    p.lanes_on = p.lanes_new = 0;
    for (int dy = 0; dy < s.D; ++dy)
        for (int r = 0; r < i.R; ++r) {
            const unsigned long long lanes = (unsigned long long)((1 << s.KF / 32) - 1) << (dy * s.KF / 32 + 4 * (i.stride * dy + r));
            p.lanes_on |= lanes;
            if (r == 0) p.lanes_new |= lanes;
        }
    p.status = device_status_word();
    if (!p.status) return cuda_fail(cudaGetLastError(), "status word");
    int sms = 148, dev = 0;
    CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
    const unsigned grid = (unsigned)(p.total_steps < sms ? p.total_steps : sms);
    const bool pool = plan->opts.pool != CPRUNE_POOL_NONE;
    const size_t smem = (size_t)s.smem_bytes;
    switch (plan->opts.activation) {
        case CPRUNE_ACT_NONE:
            return pool ? launch_stem_width<CPRUNE_ACT_NONE, true>(p, grid, smem, st) : launch_stem_width<CPRUNE_ACT_NONE, false>(p, grid, smem, st);
        case CPRUNE_ACT_RELU:
            return pool ? launch_stem_width<CPRUNE_ACT_RELU, true>(p, grid, smem, st) : launch_stem_width<CPRUNE_ACT_RELU, false>(p, grid, smem, st);
        default:
            return pool ? launch_stem_width<CPRUNE_ACT_RELU6, true>(p, grid, smem, st) : launch_stem_width<CPRUNE_ACT_RELU6, false>(p, grid, smem, st);
    }
}

}  // namespace cprune
