// Depthwise task (groups == C == K), 3x3 or 5x5, stride 1 or 2 (MobileNetV2 and MnasNet, paper Sec. 4.1), CUDA cores.
// bf16 NHWC in and out with padded channels, float32 arithmetic, fused bias + activation (+ residual).
//
// A CTA keeps one block of up to 72 channels (its taps stay in registers) and works through tiles of output pixels of
// that block: CTAs that fit the chip at once share the tiles out (persistent, two patch buffers: the next tile's patch is
// on its way while one is computed).  A tile's input patch comes in with a single tiled TMA load (out-of-bounds pixels and
// channels read as zero, which is the padding), so every input byte is fetched from L2/HBM once per tile and all taps are
// served from shared memory.  A thread owns CH channels of COLS neighbouring output columns and walks down TR output rows.
// It reads and widens every pixel of its window once: an input row feeds all the output rows it overlaps, so
// NACC = ceil(R / STRIDE) rows of accumulators are alive, and the row loop is unrolled NACC times so that their rotation
// costs no moves.  The waits on the loads are bounded like every other device-side wait.
//
// What bounds it: latency at three warps per scheduler.  C 108, 56x56, batch 64, stride 1: two patch buffers of 28 KB let three
// CTAs of four warps onto an SM (registers would let four); 12.6 M warp instructions keep the issue slots 51 % busy while an SM
// works and 40 % over the kernel, a fifth of which is start and drain; DRAM 21 %.  Between two instructions of a warp 1.4 cycles
// of 5.5 go to fixed-latency dependences, 0.5 each to the math pipe, the CTA barrier per tile and dispatch, 0.4 to memory.
// Cold: 23.4 us = 3.7 TB/s (a thread per column of 8 channels, one tile per CTA: 30.9 us); 5x5, C 288, 14x14, batch 20:
// 6.6 us (22.0 us with the taps in shared memory).  Packed FMAs: 23.4 against 26.4 us with scalar ones.  Streaming row
// chunks through a ring instead of whole patches: 29 us; loads straight from global memory: 35 us.

#include <cstring>

#include "common.cuh"
#include "depthwise_rows.cuh"
#include "plan.h"
#include "sm100_ptx.cuh"

namespace cprune {

struct DwParams {
    const uint32_t *w;     // bf16 pairs [R][R][c2]
    const float *b;
    const uint32_t *res;
    uint32_t *y;
    int P, Q, pad;
    int c2;                // c_pad / 2: words per pixel
    int G;                 // channel groups (of 8) per CTA
    int strips, segs, TR;  // per CTA: column strips (COLS columns each), row segments (TR output rows each)
    int IH, IW;            // input patch
    int tiles_h, tiles_w, cblocks;
    int tiles, ctas;       // tiles per channel block (all images), CTAs that share them
    int dn, dth, dtw;      // `ctas` as images, tile rows, tile columns: the distance between a CTA's tiles
    int patch_bytes;       // stride of the two patch buffers
    int *status;
};

template <int R, int STRIDE, int CH, int COLS, int ACT>
__global__ void __launch_bounds__(256, 2) depthwise_kernel(const __grid_constant__ CUtensorMap tm_x, const DwParams p) {
    extern __shared__ __align__(128) uint8_t dw_smem[];
    __shared__ __align__(8) unsigned long long bars[2];
    __shared__ int abort_word;
    constexpr int NW = CH / 2;                           // words (channel pairs) per pixel

    pdl_trigger();
    const int G = p.G;
    const int first = blockIdx.x / p.cblocks, cb = blockIdx.x - first * p.cblocks;
    int n, th, tw;
    {
        const int r = first / p.tiles_w;
        tw = first - r * p.tiles_w;
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
    int ln = n, lth = th, ltw = tw, ltile = first;       // next tile to load (thread 0)
    auto load_tile = [&](int buf) {
        const uint32_t bar = smem_u32(&bars[buf]);
        mbar_expect_tx(bar, (uint32_t)(p.IH * p.IW * G * 16));
        tma_load_4d(smem_u32(dw_smem) + (uint32_t)(buf * p.patch_bytes), &tm_x, bar, cb * G * 8,
                    ltw * p.strips * COLS * STRIDE - p.pad, lth * p.segs * p.TR * STRIDE - p.pad, ln);
        advance(ln, lth, ltw);
        ltile += p.ctas;
    };
    if (threadIdx.x == 0) {
        abort_word = 0;
        mbar_init(smem_u32(&bars[0]), 1);
        mbar_init(smem_u32(&bars[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        pdl_wait();
        load_tile(0);
        if (ltile < p.tiles) load_tile(1);
    }
    __syncthreads();   // the barriers are initialised before anyone polls them

    const int lanes = G * 8 / CH;                        // threads per strip: neighbouring channels
    const int sc = threadIdx.x / lanes;
    const int cq = threadIdx.x - sc * lanes;
    const int seg = sc / p.strips, strip = sc - seg * p.strips;
    const int word = cb * G * 4 + cq * NW;               // first channel pair of this thread
    const bool in_tile = seg < p.segs && word < p.c2;

    // taps and bias were written when the task was packed, not by the preceding kernel (overlaps the load)
    unsigned long long wf[R][R][NW], bf[NW];
    if (in_tile) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int s = 0; s < R; ++s) {
                uint32_t t[NW];
                load_words<NW>(p.w + (r * R + s) * p.c2 + word, t);
#pragma unroll
                for (int k = 0; k < NW; ++k) wf[r][s][k] = widen2(t[k]);
            }
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const float lo = __ldg(p.b + 2 * (word + k)), hi = __ldg(p.b + 2 * (word + k) + 1);      // (any float32 address)
            asm("mov.b64 %0, {%1, %2};" : "=l"(bf[k]) : "f"(lo), "f"(hi));
        }
    }

    const bool has_res = p.res != nullptr;
    if (has_res) pdl_wait();                             // the residual is the result of an earlier kernel of the chain

    const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f), six2 = __floats2bfloat162_rn(6.f, 6.f);
    const uint32_t pix = (uint32_t)G * 4u;               // words per pixel of the patch
    const uint32_t row_words = (uint32_t)p.IW * pix;
    const uint32_t in0 = (uint32_t)(seg * p.TR * STRIDE) * row_words + (uint32_t)(strip * COLS * STRIDE) * pix + cq * NW;
    const uint32_t out_step = (uint32_t)p.Q * (uint32_t)p.c2;
    uint32_t buf = 0, phase = 0;
    for (int tile = first; tile < p.tiles; tile += p.ctas) {
        const bool ok = mbar_wait(smem_u32(&bars[buf]), phase, &abort_word, p.status);
        const int ps = (th * p.segs + seg) * p.TR, qs = (tw * p.strips + strip) * COLS;
        const int rows = min(p.TR, p.P - ps);
        if (ok && in_tile && rows > 0 && qs < p.Q) {
            const uint32_t *in = reinterpret_cast<const uint32_t *>(dw_smem + buf * p.patch_bytes) + in0;
            const size_t o0 = (((size_t)n * p.P + ps) * p.Q + qs) * p.c2 + word;
            uint32_t *dst = p.y + o0;
            const uint32_t *rsrc = p.res + o0;
            depthwise_rows<R, STRIDE, CH, COLS>(
                in, pix, row_words, rows, wf, bf,
                [&](int c, const unsigned long long (&sum)[NW]) {
                    if (c == 0 || qs + c < p.Q) {
                        uint32_t o[NW];
#pragma unroll
                        for (int q = 0; q < NW; ++q) {
                            float2 f = split2(sum[q]);
                            if (has_res) {
                                const uint32_t rv = rsrc[(uint32_t)c * p.c2 + q];
                                f.x += __uint_as_float(rv << 16);
                                f.y += __uint_as_float(rv & 0xffff0000u);
                            }
                            // 0 and 6 are bf16 values, so the clamp commutes with the rounding
                            __nv_bfloat162 v = __floats2bfloat162_rn(f.x, f.y);
                            if (ACT != CPRUNE_ACT_NONE) v = __hmax2(v, zero2);
                            if (ACT == CPRUNE_ACT_RELU6) v = __hmin2(v, six2);
                            o[q] = *reinterpret_cast<const uint32_t *>(&v);
                        }
                        uint32_t *d = dst + (uint32_t)c * p.c2;
                        if constexpr (NW == 2) *reinterpret_cast<uint2 *>(d) = make_uint2(o[0], o[1]);
                        else *d = o[0];
                    }
                },
                [&]() { dst += out_step; rsrc += out_step; });
        }
        advance(n, th, tw);
        if (__syncthreads_or(ok ? 0 : 1)) break;         // the buffer has been read by everyone (or somebody gave up)
        if (threadIdx.x == 0 && ltile < p.tiles) load_tile(buf);
        buf ^= 1u;
        if (buf == 0) phase ^= 1u;
    }
    if (*(volatile int *)&abort_word) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let a late copy land before the CTA's memory goes away
    }
}

// Channel groups (of 8 channels) per CTA: between 4 and 9, whichever wastes the fewest lanes in the last channel block
// (c_pad/8 = 18 -> 9, 14 -> 7, 4 -> 4); larger wins ties.
int depthwise_groups(int c8) {
    if (c8 <= 9) return c8;
    int best = 8;
    double best_util = 0.0;
    for (int g = 9; g >= 4; --g) {
        const double util = (double)c8 / (double)(((c8 + g - 1) / g) * g);
        if (util > best_util + 1e-9) { best_util = util; best = g; }
    }
    return best;
}

constexpr int DW_MAX_PATCH = 64 * 1024;

// Channels and columns per thread.  3x3: the nine taps of four channels fit the registers beside the accumulators (two or
// eight channels, one or four columns measured 3 to 40 % slower); 5x5: those of two channels.
static void dw_config(int R, int *ch, int *cols) { *ch = R == 3 ? 4 : 2; *cols = 2; }

// Chooses the tile (column strips x row segments x rows per segment) and the number of CTAs.  The model prices an SM's share
// of the tiles: the row steps of its warps (dearer when few warps share the SM or few CTAs cover each other's loads) and the
// patch bytes, plus a start-up per resident warp.  Its constants were fitted to a sweep of 55 to 420 tilings of 35 layers
// (batch 1 to 64) on B200; the tiling it picks is within 3 % of the best of the sweep on average, 8 % at worst.
cprune_status plan_depthwise(cprune_plan *plan) {
    const cprune_plan_info &i = plan->info;
    DwTiling &d = plan->dw;
    int ch, cols;
    dw_config(i.R, &ch, &cols);
    const bool s1 = i.stride == 1;
    const double step_cycles = s1 ? 0.37 * i.R * i.R + 34.3 : 0.5 * i.R * i.R + 41.7;
    const double step_extra = s1 ? 1.0 : 0.54, warps_needed = s1 ? 12.0 : 15.7, load_rate = s1 ? 50.0 : 100.0;
    const double warp_start = s1 ? 268.0 : 130.0, average_share = s1 ? 0.217 : 0.31, cover = s1 ? 0.055 : 0.09;
    const int c8 = i.c_pad / 8;
    d.G = depthwise_groups(c8);
    d.cblocks = (c8 + d.G - 1) / d.G;
    const int lanes = d.G * 8 / ch;
    const int nacc = (i.R + i.stride - 1) / i.stride;
    const int all_strips = (i.Q + cols - 1) / cols;
    double best = 1e30;
    for (int ns = 1; ns <= all_strips && ns * lanes <= 256; ++ns) {
        const int tiles_w = (all_strips + ns - 1) / ns;
        if (ns > 1 && tiles_w == (all_strips + ns - 2) / (ns - 1)) continue;      // narrower tiles, as many of them
        const int IW = (ns * cols - 1) * i.stride + i.R;
        if (IW > 256) break;
        for (int tr = 1; tr <= i.P && tr <= 28; ++tr) {
            for (int ng = 1; ng * ns * lanes <= 256; ++ng) {
                if (ng > 1 && (ng - 1) * tr >= i.P) break;
                const int IH = (ng * tr - 1) * i.stride + i.R;
                const int patch = round_up(IH * IW * d.G * 16, 128);
                if (IH > 256 || patch > DW_MAX_PATCH) break;
                const int tiles_h = (i.P + ng * tr - 1) / (ng * tr);
                const long long tiles = (long long)i.N * tiles_w * tiles_h;
                const int warps = (ng * ns * lanes + 31) / 32;
                int resident = 220 * 1024 / (2 * patch + 1024);
                if (resident > 18 / warps) resident = 18 / warps;                // by registers
                if (resident < 1) continue;
                long long ctas = 148LL * resident / d.cblocks;
                if (ctas < 1) ctas = 1;
                if (ctas > tiles) ctas = tiles;
                const double on_sm = (double)ceil_div(ctas * d.cblocks, 148), active = on_sm * warps;
                const double share = (double)ceil_div(tiles, ctas) * on_sm * (1.0 - average_share) + (double)tiles * d.cblocks / 148.0 * average_share;
                const double hide = (active < warps_needed ? warps_needed / active : 1.0) * (1.0 + cover / on_sm);
                const double work = share * warps * (tr + nacc - 1 + step_extra) * step_cycles * (s1 ? 1.0 : 0.85) * hide;
                const double load = share * patch / load_rate;
                const double t = (work > load ? work + 0.3 * load : load + 0.3 * work) + active * warp_start;
                if (t < best) {
                    best = t;
                    d.strips = ns; d.segs = ng; d.TR = tr; d.IH = IH; d.IW = IW; d.tiles_w = tiles_w; d.tiles_h = tiles_h;
                    d.tiles = tiles; d.ctas = (int)ctas; d.patch_bytes = patch;
                }
            }
        }
    }
    return best < 1e30 ? CPRUNE_OK : CPRUNE_ERR_UNSUPPORTED;
}

template <int R, int STRIDE, int CH, int COLS, int ACT>
static cprune_status launch_dw_act(const CUtensorMap &tm, const DwParams &p, unsigned blocks, cudaStream_t st) {
    const int threads = (p.strips * p.segs * (p.G * 8 / CH) + 31) / 32 * 32;
    const size_t smem = (size_t)p.patch_bytes * (p.tiles > p.ctas ? 2 : 1);
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};    // the shared-memory limit of a kernel is a per-device attribute
    {
        int dev = 0;
        CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(depthwise_kernel<R, STRIDE, CH, COLS, ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * DW_MAX_PATCH));
            attr_set[dev] = true;
        }
    }
    CPRUNE_CUDA_CHECK(launch_chained(depthwise_kernel<R, STRIDE, CH, COLS, ACT>, dim3(blocks), dim3(threads), smem, st, tm, p));
    CPRUNE_LAUNCH_CHECK("depthwise kernel");
    return CPRUNE_OK;
}

template <int R, int STRIDE, int CH, int COLS>
static cprune_status launch_dw(int act, const CUtensorMap &tm, const DwParams &p, unsigned blocks, cudaStream_t st) {
    if (act == CPRUNE_ACT_NONE) return launch_dw_act<R, STRIDE, CH, COLS, CPRUNE_ACT_NONE>(tm, p, blocks, st);
    if (act == CPRUNE_ACT_RELU) return launch_dw_act<R, STRIDE, CH, COLS, CPRUNE_ACT_RELU>(tm, p, blocks, st);
    return launch_dw_act<R, STRIDE, CH, COLS, CPRUNE_ACT_RELU6>(tm, p, blocks, st);
}

cprune_status launch_depthwise(cprune_plan *plan, const void *x, const void *w, const float *b, const void *res,
                               void *y, cudaStream_t st) {
    const cprune_plan_info &i = plan->info;
    const DwTiling &d = plan->dw;
    DwParams p;
    p.w = (const uint32_t *)w;
    p.b = b;
    p.res = (const uint32_t *)res;
    p.y = (uint32_t *)y;
    p.P = i.P; p.Q = i.Q; p.pad = i.pad;
    const int act = plan->opts.activation;
    p.c2 = i.c_pad / 2;
    p.G = d.G; p.strips = d.strips; p.segs = d.segs; p.TR = d.TR; p.IH = d.IH; p.IW = d.IW;
    p.tiles_h = d.tiles_h; p.tiles_w = d.tiles_w; p.cblocks = d.cblocks;
    p.tiles = (int)d.tiles; p.ctas = d.ctas; p.patch_bytes = d.patch_bytes;
    p.dn = d.ctas / (d.tiles_h * d.tiles_w);
    p.dth = (d.ctas - p.dn * d.tiles_h * d.tiles_w) / d.tiles_w;
    p.dtw = d.ctas - (p.dn * d.tiles_h + p.dth) * d.tiles_w;
    p.status = device_status_word();
    if (!p.status) return cuda_fail(cudaGetLastError(), "status word");
    CUtensorMap tm;
    {
        std::lock_guard<std::mutex> lock(plan->mu);
        if (plan->map_x != x) {
            unsigned long long dims[4] = {(unsigned long long)i.c_pad, (unsigned long long)i.W, (unsigned long long)i.H,
                                          (unsigned long long)i.N};
            unsigned long long strides[3] = {(unsigned long long)i.c_pad * 2, (unsigned long long)i.W * i.c_pad * 2,
                                             (unsigned long long)i.H * i.W * i.c_pad * 2};
            unsigned box[4] = {(unsigned)(p.G * 8), (unsigned)p.IW, (unsigned)p.IH, 1};
            cprune_status s = encode_tiled_bf16(&plan->tm_a, x, 4, dims, strides, box);
            if (s != CPRUNE_OK) return s;
            plan->map_x = x;
        }
        std::memcpy(&tm, &plan->tm_a, sizeof(CUtensorMap));
    }
    if (d.tiles > 0x3fffffffLL) return CPRUNE_ERR_UNSUPPORTED;
    const long long blocks = (long long)d.ctas * d.cblocks;
    if (i.R == 3) return i.stride == 1 ? launch_dw<3, 1, 4, 2>(act, tm, p, (unsigned)blocks, st) : launch_dw<3, 2, 4, 2>(act, tm, p, (unsigned)blocks, st);
    return i.stride == 1 ? launch_dw<5, 1, 2, 2>(act, tm, p, (unsigned)blocks, st) : launch_dw<5, 2, 2, 2>(act, tm, p, (unsigned)blocks, st);
}

}  // namespace cprune
