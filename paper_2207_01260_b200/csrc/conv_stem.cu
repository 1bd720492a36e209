// First conv task of a model (3-channel stem, stride 1 or 2) straight from the float32 image: cast, convolution, bias,
// activation and, if the task asks for it, the 3x3 stride-2 max-pool in one pass over the image (paper Sec. 3.4: a task is
// the fused subgraph).
//
// The pixels are on the column side of the MMA and the filters on its 128 rows: D = 128 / KF conv rows of KF (32, 64 or 128)
// filters each, so that the rows are full for the 16 to 64 filters of a pruned stem (fewer where the tiles of a large image would not
// fit; the rows left over go nowhere).  Those D conv rows read the same
// RH = stride * (D - 1) + R input rows; a filter of conv row dy is packed with zero taps where its window does not reach.
//   K order     per input row, the S pixels of a window in 4 channel lanes each: 32 bytes (S <= 4) or 64.  A 128-byte operand
//               row holds the windows of one output column in `per` (1, 2 or 4) neighbouring input rows.
//   converters  (8 warps) turn float32 rows, fetched by bulk copies a few tiles ahead, into bf16 pixels of 4 lanes in a row
//               buffer, and copy every output column's window from there into a swizzled operand tile.  (Overlapping windows
//               are stored once per column because the MMA fetches one row of its operand's swizzle width per cycle: with
//               the rows read in place through an unswizzled descriptor the 7x7 stem of 64 images took 55 us.)  Tiles form a
//               ring; rows outside the image are zeros, as are the columns left and right of it.  They also say of every tile
//               whether it holds a pixel that is no number (infinite or NaN as a bf16 value).
//   MMA         (1 warp) one step = D conv rows: N = Q columns, K = RH windows; filters stay in shared memory.  Conv rows meet the
//               input rows outside their window with zero taps, which is nothing unless a pixel is no number: the rows of such a
//               tile go to the accumulator lanes that want them alone (always doing so cost the pooled stem 7 us of 46).
//   epilogue    (8 warps) a thread owns one filter of one conv row and walks along the pixels, so the pool's horizontal
//               maximum stays in registers; odd conv rows hand theirs to the even ones through shared memory.  Results are
//               transposed through shared memory (2-byte stores, neighbouring lanes = neighbouring filters) and leave as one
//               bulk copy: the output rows of a step are contiguous.
// A block works through consecutive steps; with a pool it recomputes one step where it starts inside an image (the odd conv
// row above).
// What bounds it: no role's work but the waits from one to the next.  64 more images take the pooled 7x7 stem 38.7 us (1.6 us a
// step); without the conversions and window copies 36.9, without the MMAs 36.9, without the pooling arithmetic 36.3 us.  (3x3: 20.7,
// 17.8, 21.1 and 17.9 us.)  At 8 images issue slots are 33 % busy, the tensor pipe 12 %, DRAM 3 %.
// Stem of 64 224x224 images, launched back to back: 7x7 stride 2, 64 filters, pooled 63.8 us with a regrouping pass and the patch
// kernel, 51.3 us here; 3x3 stride 2, 32 filters 49.3 and 32.7 us.
#include <cuda.h>

#include <cstring>
#include <mutex>

#include "common.cuh"
#include "plan.h"
#include "sm100_ptx.cuh"

namespace cprune {

constexpr int ST_EPI_WARPS = 8, ST_CONV_WARPS = 8;
constexpr int ST_MMA_WARP = ST_EPI_WARPS + ST_CONV_WARPS;
constexpr int ST_THREADS = (ST_MMA_WARP + 1) * 32;
constexpr int ST_MAX_RING = 12;           // operand tiles
constexpr int ST_RAW = 4;                 // tiles of float32 rows in flight
constexpr int ST_ACC_STRIDE = 256;        // column offset of the second accumulator

struct StemParams {
    const float *x;
    const float *bias;
    __nv_bfloat16 *y;
    int H, W, P, Q, out_h, out_w;
    int stride, pad;
    int D, KF, RH, N;
    int per, tiles, adv;                  // input rows per operand tile, tiles a step reads, tiles from step to step
    int row_bytes, tile_bytes, raw_bytes, ring, stage_bytes, xch_words;
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

__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t &v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(taddr) : "memory");
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

// a + 0 * v for bf16 pairs: a zero stays a zero unless v is infinite or NaN
__device__ __forceinline__ uint32_t times_zero2(uint32_t v, uint32_t a) {
    asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(a) : "r"(v), "r"(0u));
    return a;
}

// CPS: 16-byte pieces of a window
template <int ACT, bool POOL, int CPS>
__global__ void __launch_bounds__(ST_THREADS, 1) conv_stem_kernel(const __grid_constant__ CUtensorMap tm_w, const StemParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_base = smem_u32(smem_raw);
    const uint32_t base = (raw_base + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_base);
    const uint32_t w_bytes = (uint32_t)p.tiles * 16384u;
    uint8_t *ring = smem + w_bytes;
    uint8_t *raw = ring + (uint32_t)(p.ring * p.tile_bytes);
    uint8_t *rows = raw + ST_RAW * p.raw_bytes;
    const int row_buf = p.per * p.row_bytes;
    uint8_t *stage = rows + 2 * row_buf;
    uint32_t *xch = (uint32_t *)(stage + 2 * p.stage_bytes);
    uint8_t *ctrl = (uint8_t *)(xch + (POOL ? 2 * 64 * p.xch_words : 0));
    const uint32_t ctrl0 = smem_u32(ctrl);
    auto full = [&](int s) { return ctrl0 + 8u * s; };
    auto empty = [&](int s) { return ctrl0 + 96u + 8u * s; };
    auto tfull = [&](int a) { return ctrl0 + 192u + 8u * a; };
    auto tempty = [&](int a) { return ctrl0 + 208u + 8u * a; };
    const uint32_t wbar = ctrl0 + 224u, epi_bar = ctrl0 + 232u, conv_bar = ctrl0 + 240u;
    auto rfull = [&](int s) { return ctrl0 + 256u + 8u * s; };
    uint32_t *tmem_slot = (uint32_t *)(ctrl + 248);
    volatile int *abort_flag = (volatile int *)(ctrl + 252);
    uint8_t *flags = ctrl + 288;           // 16 tiles (more than the ring and the tiles being converted) x converter warps

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    if (tid == 0) {
        for (int s = 0; s < p.ring; ++s) { mbar_init(full(s), ST_CONV_WARPS); mbar_init(empty(s), 1); }
        for (int s = 0; s < ST_RAW; ++s) mbar_init(rfull(s), 1);
        for (int a = 0; a < 2; ++a) { mbar_init(tfull(a), 1); mbar_init(tempty(a), ST_EPI_WARPS); }
        mbar_init(wbar, 1);
        mbar_init(epi_bar, ST_EPI_WARPS);
        mbar_init(conv_bar, ST_CONV_WARPS);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // first kernel of a chain: before its successor may start, and before the parameters are read
        pdl_wait();
        pdl_trigger();
        mbar_expect_tx(wbar, w_bytes);
        for (int b = 0; b < p.tiles; ++b) tma_load_2d(base + (uint32_t)b * 16384u, &tm_w, wbar, b * 64, 0);
    }
    // what the converters do not write (columns beyond Q, pixels beside the image) has to be finite, or zero
    for (int e = tid; e < p.ring * p.tile_bytes / 16; e += ST_THREADS) ((uint4 *)ring)[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < 2 * row_buf / 16; e += ST_THREADS) ((uint4 *)rows)[e] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == ST_MMA_WARP) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    fence_async_smem();                    // the tensor core reads the zeros
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int t0 = (int)((long long)p.total_steps * blockIdx.x / gridDim.x);
    const int t1 = (int)((long long)p.total_steps * (blockIdx.x + 1) / gridDim.x);

    if (warp >= ST_EPI_WARPS && warp < ST_MMA_WARP) {
        // ------------------------------------------------------------------ converters
        constexpr int THREADS = ST_CONV_WARPS * 32;
        const int ctid = tid - ST_EPI_WARPS * 32;
        const bool leader = ctid == 0;
        // float32 rows of a tile that lie inside the image
        auto rows_of = [&](int tile, int &r0, int &r1) {
            r0 = max(0, tile * p.per - p.pad);
            r1 = min(p.H, (tile + 1) * p.per - p.pad);
        };
        // position of the bulk copies, ST_RAW tiles ahead of the conversion (leader only)
        int lt = t0;
        StemSegment ls = {0, 0, 0, 0};
        bool lmore = next_segment<POOL>(p, lt, t1, ls);
        int ltile = ls.first * p.adv, lslot = 0;
        auto load_next = [&]() {
            if (!lmore) return;
            int r0, r1;
            rows_of(ltile, r0, r1);
            const uint32_t bytes = r1 > r0 ? (uint32_t)((r1 - r0) * p.W) * 12u : 0u;
            mbar_expect_tx(rfull(lslot), bytes);
            if (bytes) bulk_load(smem_u32(raw) + (uint32_t)(lslot * p.raw_bytes), p.x + ((size_t)ls.n * p.H + r0) * p.W * 3, bytes, rfull(lslot));
            lslot = (lslot + 1) % ST_RAW;
            if (++ltile == (ls.to - 1) * p.adv + p.tiles) {
                lmore = next_segment<POOL>(p, lt, t1, ls);
                ltile = ls.first * p.adv;
            }
        };
        if (leader) {
            pdl_wait();
            for (int s = 0; s < ST_RAW; ++s) load_next();
        }
        // what this thread converts and copies of every tile (the plan keeps it to two items each; a division per item and
        // tile would cost as much as the work)
        const int quads = p.W >> 2;
        int conv_r[2], conv_src[2], conv_dst[2], copy_src[2], copy_q[2], copy_r[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = ctid + u * THREADS;
            const int r = e / quads, xq = e - r * quads;
            conv_r[u] = r < p.per ? r : -1;
            conv_src[u] = (r * p.W + xq * 4) * 12;
            conv_dst[u] = r * p.row_bytes + (p.pad + xq * 4) * 8;
            const int cr = e / p.Q, q = e - cr * p.Q;
            copy_r[u] = cr < p.per ? cr : -1;
            copy_q[u] = q;
            copy_src[u] = cr * p.row_bytes + q * p.stride * 8;
        }
        const uint32_t keep = p.S & 1 ? 0u : 0xffffffffu;      // the second pixel of a window's last piece
        int t = t0, slot = 0, rslot = 0, buf = 0, seq = 0;
        uint32_t phase = 0, rphase = 0, conv_phase = 0;
        bool ok = true;
        StemSegment sg;
        while (ok && next_segment<POOL>(p, t, t1, sg)) {
            for (int b = sg.first * p.adv; b < (sg.to - 1) * p.adv + p.tiles; ++b) {
                int r0, r1;
                rows_of(b, r0, r1);
                ok = __all_sync(0xffffffffu, mbar_wait(rfull(rslot), rphase, abort_flag, p.status));
                if (!ok) break;
                uint8_t *rb = rows + buf * row_buf;
                const uint8_t *src = raw + rslot * p.raw_bytes;
                const int row0 = b * p.per - p.pad;
                uint32_t odd[2] = {0u, 0u};                // zeros, or NaN where a pixel is no number
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (conv_r[u] < 0) break;
                    const int row = row0 + conv_r[u];
                    float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f), f1 = f0, f2 = f0;
                    if (row >= r0 && row < r1) {
                        const float4 *s4 = (const float4 *)(src + conv_src[u] + (row0 - r0) * p.W * 12);
                        f0 = s4[0]; f1 = s4[1]; f2 = s4[2];
                    }
                    const uint2 px[4] = {make_uint2(act_pack2<CPRUNE_ACT_NONE>(f0.x, f0.y), act_pack2<CPRUNE_ACT_NONE>(f0.z, 0.f)),
                                         make_uint2(act_pack2<CPRUNE_ACT_NONE>(f0.w, f1.x), act_pack2<CPRUNE_ACT_NONE>(f1.y, 0.f)),
                                         make_uint2(act_pack2<CPRUNE_ACT_NONE>(f1.z, f1.w), act_pack2<CPRUNE_ACT_NONE>(f2.x, 0.f)),
                                         make_uint2(act_pack2<CPRUNE_ACT_NONE>(f2.y, f2.z), act_pack2<CPRUNE_ACT_NONE>(f2.w, 0.f))};
                    uint2 *dst = (uint2 *)(rb + conv_dst[u]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        dst[q] = px[q];
                        odd[0] = times_zero2(px[q].x, odd[0]);
                        odd[1] = times_zero2(px[q].y, odd[1]);
                    }
                }
                const bool any_odd = __any_sync(0xffffffffu, ((odd[0] | odd[1]) & 0x7fff7fffu) != 0u);
                if (lane == 0) flags[(seq & 15) * ST_CONV_WARPS + (warp - ST_EPI_WARPS)] = any_odd;
                ++seq;
                // everyone has read the float32 rows and written its pixels; the row buffer is written again two tiles on,
                // behind the next meeting
                __syncwarp();
                if (lane == 0) mbar_arrive(conv_bar);
                ok = __all_sync(0xffffffffu, mbar_wait(conv_bar, conv_phase, abort_flag, p.status));
                conv_phase ^= 1u;
                ok = ok && __all_sync(0xffffffffu, mbar_wait(empty(slot), phase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                if (leader) load_next();
                uint8_t *dst0 = ring + (uint32_t)(slot * p.tile_bytes);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (copy_r[u] < 0) break;
                    const uint8_t *win = rb + copy_src[u];
                    uint4 v[CPS];
                    if (p.stride == 2) {
#pragma unroll
                        for (int c = 0; c < CPS; ++c) v[c] = *(const uint4 *)(win + c * 16);
                    } else {
#pragma unroll
                        for (int c = 0; c < CPS; ++c) {
                            const uint2 lo = *(const uint2 *)(win + c * 16), hi = *(const uint2 *)(win + c * 16 + 8);
                            v[c] = make_uint4(lo.x, lo.y, hi.x, hi.y);
                        }
                    }
                    // pixels behind the window's last meet zero taps and have to be numbers: zeros
                    v[CPS - 1].z &= keep; v[CPS - 1].w &= keep;
                    if (p.S <= 2 * CPS - 2) {
#pragma unroll
                        for (int c = 0; c < CPS; ++c) {
                            if (2 * c >= p.S) v[c].x = v[c].y = 0u;
                            if (2 * c + 1 >= p.S) v[c].z = v[c].w = 0u;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < CPS; ++c) *(uint4 *)(dst0 + sub_off(copy_q[u], copy_r[u] * CPS + c)) = v[c];
                }
                fence_async_smem();                        // the tensor core reads what these stores wrote
                __syncwarp();
                if (lane == 0) mbar_arrive(full(slot));
                if (++slot == p.ring) { slot = 0; phase ^= 1u; }
                if (++rslot == ST_RAW) { rslot = 0; rphase ^= 1u; }
                buf ^= 1;
            }
        }
    } else if (warp == ST_MMA_WARP) {
        // ------------------------------------------------------------------ MMA issue
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t ring0 = smem_u32(ring);
        constexpr int ROW_STEPS = CPS / 2;                 // MMA steps (16 values) per input row
        const uint32_t a_lo0 = desc_lo(base), ring_lo = desc_lo(ring0), tile_step = (uint32_t)p.tile_bytes >> 4;
        int t = t0, acc = 0;
        uint32_t acc_phase = 0;
        int head = 0;                                      // ring slot of the oldest tile in use
        int wslot = 0, seq = 0;                            // next tile to wait for
        uint32_t wphase = 0, odd = 0;                      // odd: ring slots whose tile holds a pixel that is no number
        StemSegment sg;
        bool ok = __all_sync(0xffffffffu, mbar_wait(wbar, 0u, abort_flag, p.status));
        while (ok && next_segment<POOL>(p, t, t1, sg)) {
            int have = 0;                                  // tiles of the segment that have arrived
            for (int s = sg.first; s < sg.to && ok; ++s) {
                ok = __all_sync(0xffffffffu, mbar_wait(tempty(acc), acc_phase ^ 1u, abort_flag, p.status));
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * ST_ACC_STRIDE);
                const bool last = s + 1 == sg.to;
                int slot = head;
                bool odd_first = false;                    // the step's first tile is such a one
                for (int j = 0; j < p.tiles && ok; ++j) {
                    if (have <= (s - sg.first) * p.adv + j) {
                        ok = __all_sync(0xffffffffu, mbar_wait(full(wslot), wphase, abort_flag, p.status));
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t bit = 1u << wslot;
                        odd = *(const volatile unsigned long long *)(flags + (seq++ & 15) * ST_CONV_WARPS) ? odd | bit : odd & ~bit;
                        if (++wslot == p.ring) { wslot = 0; wphase ^= 1u; }
                        ++have;
                    }
                    const int nk = min(p.per, p.RH - j * p.per) * ROW_STEPS;
                    const uint32_t a_lo = a_lo0 + (uint32_t)j * 1024u, b_lo = ring_lo + (uint32_t)slot * tile_step;
                    const bool odd_tile = (odd >> slot) & 1u;
                    if (j == 0) odd_first = odd_tile;
                    if (elect_one()) {
                        if (__builtin_expect(odd_tile || odd_first, 0)) {
                            // zero times a pixel that is no number is NaN: only the accumulator lanes whose window holds the row.
                            // A conv row's sums begin with the first tile, which clears all lanes, or with its own first row.
                            const uint32_t on16 = (uint32_t)(p.lanes_on >> (j * p.per * 4)), new16 = odd_first ? (uint32_t)(p.lanes_new >> (j * p.per * 4)) : 0u;
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t on = (on16 >> (k / ROW_STEPS * 4)) & 15u, fresh = k % ROW_STEPS ? 0u : (new16 >> (k / ROW_STEPS * 4)) & 15u;
                                const uint32_t a = a_lo + (uint32_t)(2 * k), b = b_lo + (uint32_t)(2 * k);
                                if (on != fresh) umma_bf16_words_lanes(d_tmem, a, b, DESC_HI_SW128, idesc, 1u, on ^ fresh);
                                if (fresh) umma_bf16_words_lanes(d_tmem, a, b, DESC_HI_SW128, idesc, 0u, fresh);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (k < nk) umma_bf16_words(d_tmem, a_lo + (uint32_t)(2 * k), b_lo + (uint32_t)(2 * k), DESC_HI_SW128, idesc, (j | k) ? 1u : 0u);
                        }
                        if (j < p.adv || last) umma_commit(empty(slot));      // not needed by the next step
                        if (j + 1 == p.tiles) umma_commit(tfull(acc));
                    }
                    __syncwarp();
                    if (++slot == p.ring) slot = 0;
                }
                head += last ? p.tiles : p.adv;
                if (head >= p.ring) head -= p.ring;
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3, half = warp >> 2;
        const int m = quarter * 32 + lane;
        const int dy = m / p.KF, k = m - dy * p.KF;
        // rows of filters that a halved D leaves over (D * KF < 128) have no place in the staging buffer; the pool's D is always 2
        const bool k_ok = k < p.k_pad && (POOL || dy < p.D);
        pdl_wait();
        const float bias = k_ok ? __ldg(p.bias + k) : 0.f;
        const int units = p.N >> 4;
        const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
        int t = t0, acc = 0, buf = 0;
        uint32_t acc_phase = 0, epi_phase = 0;
        bool ok = true;
        auto epi_sync = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(epi_bar);
            const bool r = __all_sync(0xffffffffu, mbar_wait(epi_bar, epi_phase, abort_flag, p.status, false));
            epi_phase ^= 1u;
            return r;
        };
        StemSegment sg;
        while (ok && next_segment<POOL>(p, t, t1, sg)) {
            for (int s = sg.first; s < sg.to && ok; ++s) {
                ok = __all_sync(0xffffffffu, mbar_wait(tfull(acc), acc_phase, abort_flag, p.status, false));
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_acc = t_row + (uint32_t)(acc * ST_ACC_STRIDE);
                __nv_bfloat16 *st = (__nv_bfloat16 *)(stage + buf * p.stage_bytes) + k;
                if (POOL) {
                    // horizontal maxima of this thread's conv row: 8 pooled columns per 16 accumulator columns; the next 16
                    // columns are on their way while these are worked on
                    uint32_t hm[4][4];
                    uint32_t *mine = xch + (uint32_t)(((s & 1) * 64 + k) * p.xch_words);
                    uint32_t c[2][17];
                    auto load = [&](int v) {
                        const int u = half + 2 * v;
                        if (u < units) {
                            tmem_ld16(t_acc + (uint32_t)(u * 16), c[v & 1] + 1);
                            if (u > 0) tmem_ld1(t_acc + (uint32_t)(u * 16 - 1), c[v & 1][0]);
                            else c[v & 1][0] = 0xff800000u;        // -inf: no column left of the image
                        }
                    };
                    load(0);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        tmem_ld_wait();
                        if (v < 3) load(v + 1);
                        const int u = half + 2 * v;
                        if (u < units) {
                            float h[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                h[j] = fmaxf(fmaxf(__uint_as_float(c[v & 1][2 * j]), __uint_as_float(c[v & 1][2 * j + 1])), __uint_as_float(c[v & 1][2 * j + 2])) + bias;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                hm[v][j] = act_pack2<ACT>(h[2 * j], h[2 * j + 1]);
                                if (dy == 1) mine[u * 4 + j] = hm[v][j];
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty(acc));
                    ok = epi_sync();                       // the odd rows' maxima are in place
                    if (!ok) break;
                    if (s >= sg.from && dy == 0 && k_ok) {
                        const uint32_t *above = xch + (uint32_t)((((s & 1) ^ 1) * 64 + k) * p.xch_words);
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int u = half + 2 * v;
                            if (u < units) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    uint32_t r = max2(hm[v][j], mine[u * 4 + j]);
                                    if (s > 0) r = max2(r, above[u * 4 + j]);
                                    const int px = u * 8 + 2 * j;
                                    if (px < p.out_w) st[(uint32_t)(px * p.k_pad)] = __ushort_as_bfloat16((unsigned short)(r & 0xffffu));
                                    if (px + 1 < p.out_w) st[(uint32_t)((px + 1) * p.k_pad)] = __ushort_as_bfloat16((unsigned short)(r >> 16));
                                }
                            }
                        }
                    }
                } else {
                    __nv_bfloat16 *srow = st + (uint32_t)(dy * p.Q * p.k_pad);
                    for (int u = half; u < units; u += 4) {
                        uint32_t c[2][16];
                        tmem_ld16(t_acc + (uint32_t)(u * 16), c[0]);
                        if (u + 2 < units) tmem_ld16(t_acc + (uint32_t)((u + 2) * 16), c[1]);
                        tmem_ld_wait();
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (k_ok && u + 2 * h < units) {
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const uint32_t r = act_pack2<ACT>(__uint_as_float(c[h][2 * j]) + bias, __uint_as_float(c[h][2 * j + 1]) + bias);
                                    const int px = (u + 2 * h) * 16 + 2 * j;
                                    if (px < p.Q) srow[(uint32_t)(px * p.k_pad)] = __ushort_as_bfloat16((unsigned short)(r & 0xffffu));
                                    if (px + 1 < p.Q) srow[(uint32_t)((px + 1) * p.k_pad)] = __ushort_as_bfloat16((unsigned short)(r >> 16));
                                }
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty(acc));
                }
                if (s >= sg.from) {
                    fence_async_smem();
                    // the buffer written next was last read by the previous step's copy
                    if (tid == 0) tma_store_wait_read<0>();
                    ok = epi_sync();
                    if (!ok) break;
                    if (tid == 0) {
                        const int row = POOL ? s : s * p.D, nrows = POOL ? 1 : min(p.D, p.P - row);
                        bulk_store(p.y + ((size_t)sg.n * p.out_h + row) * p.out_w * p.k_pad, smem_u32(stage) + (uint32_t)(buf * p.stage_bytes),
                                   (uint32_t)(nrows * p.out_w * p.k_pad) * 2u);
                        tma_store_commit();
                    }
                    buf ^= 1;
                }
                if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            }
        }
        if (tid == 0) tma_store_wait_all();                // staged data must be read before the block's memory goes away
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

// Filters: out[dy * KF + k][tile * 64 + row in tile * (slot / 2) + pixel * 4 + c], zero where the tap does not exist.
__global__ void __launch_bounds__(256) pack_stem_kernel(const float *__restrict__ w, int K, int C, int R, int S, int stride, int D, int KF,
                                                        int RH, int per, int slot, int ktot, __nv_bfloat16 *__restrict__ out) {
    const int total = 128 * ktot, half = slot / 2;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int m = e / ktot, kk = e - m * ktot;
        const int dy = m / KF, k = m - dy * KF;
        const int tile = kk >> 6, in_tile = kk & 63;
        const int j = tile * per + in_tile / half, px = in_tile % half / 4, c = in_tile & 3;
        const int r = j - stride * dy;
        float v = 0.f;
        if (dy < D && k < K && j < RH && c < C && r >= 0 && r < R && px < S) v = w[(((size_t)k * C + c) * R + r) * S + px];
        out[e] = __float2bfloat16_rn(v);
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
    // Where the other path is faster (us, with the cast or regrouping pass, before / here): rows of 32 pixels, whose MMAs have
    // few columns (3x3 3 -> 45, 128 images 21 / 36), and small tasks of the few-pixel kernel (3x3 stride 2, one 224x224 image).
    if (i.Q < 64 || (plan->small && plan->est_us < 6.0)) return;
    s.KF = pool ? 64 : (i.k_pad <= 32 ? 32 : (i.k_pad <= 64 ? 64 : 128));
    s.steps_per_img = 0;
    // rows per step as the filters allow; half as many where the operand tiles or the staged output would not fit
    for (s.D = pool ? 2 : 128 / s.KF; s.D >= 1 && !s.steps_per_img; s.D >>= 1) {
        if (pool && s.D != 2) return;
        const int new_rows = i.stride * s.D;               // input rows from step to step: a power of two
        s.RH = i.stride * (s.D - 1) + i.R;
        s.slot = i.S <= 4 ? 32 : 64;
        while (128 / s.slot > new_rows) s.slot *= 2;
        s.per = 128 / s.slot;
        s.tiles = (s.RH + s.per - 1) / s.per;
        s.adv = new_rows / s.per;
        if (s.tiles < s.adv) s.tiles = s.adv;              // (filters shorter than the step: the rows between are read, zero taps)
        s.N = round_up(i.Q, 16);
        const int data = i.pad + i.W, read = (i.Q - 1) * i.stride + s.slot / 8;
        s.row_bytes = round_up(8 * (data > read ? data : read), 16);
        s.tile_bytes = round_up(s.N * 128, 1024);
        s.raw_bytes = round_up(s.per * i.W * 12, 128);
        s.stage_bytes = round_up((pool ? 1 : s.D) * i.out_w * i.k_pad * 2, 128);
        s.xch_words = (s.N / 4) | 1;
        if (s.per * (i.W / 4) > 2 * ST_CONV_WARPS * 32 || s.per * i.Q > 2 * ST_CONV_WARPS * 32) continue;
        for (s.ring = ST_MAX_RING; s.ring > s.tiles; --s.ring) {
            s.smem_bytes = 1024 + s.tiles * 16384 + s.ring * s.tile_bytes + ST_RAW * s.raw_bytes + 2 * s.per * s.row_bytes + 2 * s.stage_bytes +
                           (pool ? 2 * 64 * s.xch_words * 4 : 0) + 512;
            if (s.smem_bytes <= 227 * 1024) {
                s.steps_per_img = pool ? i.P / 2 : (i.P + s.D - 1) / s.D;
                break;
            }
        }
        if (s.steps_per_img) break;
    }
    if (!s.steps_per_img || (long long)i.N * s.steps_per_img > 0x3fffffffLL) return;
    s.ktot = s.tiles * 64;
    s.weight_bytes = (size_t)128 * s.ktot * 2;
    s.ok = 1;
}

cprune_status pack_conv_stem(const cprune_plan *plan, const float *w, void *w_stem, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    const StemTiling &s = plan->stem;
    pack_stem_kernel<<<(unsigned)ceil_div(128LL * s.ktot, 256), 256, 0, st>>>(w, i.K, i.C, i.R, i.S, i.stride, s.D, s.KF, s.RH, s.per, s.slot, s.ktot,
                                                                             (__nv_bfloat16 *)w_stem);
    CPRUNE_LAUNCH_CHECK("pack_stem_kernel");
    return CPRUNE_OK;
}

template <int ACT, bool POOL, int CPS>
static cprune_status launch_stem(const CUtensorMap &tm, const StemParams &p, unsigned grid, size_t smem, cudaStream_t st) {
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};    // the shared-memory limit of a kernel is a per-device attribute
    int dev = 0;
    CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
    {
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(conv_stem_kernel<ACT, POOL, CPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            attr_set[dev] = true;
        }
    }
    CPRUNE_CUDA_CHECK(launch_chained(conv_stem_kernel<ACT, POOL, CPS>, dim3(grid), dim3(ST_THREADS), smem, st, tm, p));
    return CPRUNE_OK;
}
template <int ACT, bool POOL>
static cprune_status launch_stem_slot(int slot, const CUtensorMap &tm, const StemParams &p, unsigned grid, size_t smem, cudaStream_t st) {
    if (slot == 32) return launch_stem<ACT, POOL, 2>(tm, p, grid, smem, st);
    if (slot == 64) return launch_stem<ACT, POOL, 4>(tm, p, grid, smem, st);
    return launch_stem<ACT, POOL, 8>(tm, p, grid, smem, st);
}

cprune_status launch_conv_stem(const cprune_plan *plan, const float *x, const void *w_packed, const float *b, void *y, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    const StemTiling &s = plan->stem;
    if (!s.ok || ((uintptr_t)x & 15)) return CPRUNE_ERR_INVALID_ARG;
    CUtensorMap tm;
    const unsigned long long dims[2] = {(unsigned long long)s.ktot, 128};
    const unsigned long long strides[1] = {(unsigned long long)s.ktot * 2};
    const unsigned box[2] = {64, 128};
    cprune_status e = encode_tiled_bf16_swz(&tm, (const char *)w_packed + s.weight_offset, 2, dims, strides, box, 128, true);
    if (e != CPRUNE_OK) return e;
    StemParams p;
    p.x = x; p.bias = b; p.y = (__nv_bfloat16 *)y;
    p.H = i.H; p.W = i.W; p.P = i.P; p.Q = i.Q; p.out_h = i.out_h; p.out_w = i.out_w;
    p.stride = i.stride; p.pad = i.pad;
    p.D = s.D; p.KF = s.KF; p.RH = s.RH; p.N = s.N;
    p.per = s.per; p.tiles = s.tiles; p.adv = s.adv;
    p.row_bytes = s.row_bytes; p.tile_bytes = s.tile_bytes; p.raw_bytes = s.raw_bytes; p.ring = s.ring; p.stage_bytes = s.stage_bytes;
    p.xch_words = s.xch_words;
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
            return pool ? launch_stem_slot<CPRUNE_ACT_NONE, true>(s.slot, tm, p, grid, smem, st) : launch_stem_slot<CPRUNE_ACT_NONE, false>(s.slot, tm, p, grid, smem, st);
        case CPRUNE_ACT_RELU:
            return pool ? launch_stem_slot<CPRUNE_ACT_RELU, true>(s.slot, tm, p, grid, smem, st) : launch_stem_slot<CPRUNE_ACT_RELU, false>(s.slot, tm, p, grid, smem, st);
        default:
            return pool ? launch_stem_slot<CPRUNE_ACT_RELU6, true>(s.slot, tm, p, grid, smem, st) : launch_stem_slot<CPRUNE_ACT_RELU6, false>(s.slot, tm, p, grid, smem, st);
    }
}

}  // namespace cprune
