// Internal definition of a task plan and the launchers of the kernel families.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "cprune.h"

// Tiling of the patch kernel (conv_patch.cu): a tile is TH output rows of one image, MT blocks of 128 accumulator
// rows, FT filters.
struct PatchTiling {
    int MT, TH, FT, tiles_n, tiles_per_img, wstages, resident, acc_bufs, staging_bufs, patch_bytes;
    int TW, tiles_w, step_h, step_w, org;   // tile width, tiles per image row, distance between tiles, origin offset
    int pstages;                            // depth of the patch ring
    int dense;                              // flat tasks: a tile's output is staged as it lies in memory and stored by one bulk copy
    int stage_bytes;                        // shared memory of one staging buffer
    int dense_pitch;                        // dense staging: bytes between neighbouring pixels in the staging buffer
    int ipt;                                // whole images per tile where several fit (0: tiles are rows of one image)
    int wgroup;                             // filter taps under one barrier of the filter ring
    int pair;                               // two CTAs share the filters of a tile each (cta_group::2)
};

// Tiling of the depthwise kernel (depthwise.cu)
struct DwTiling {
    int G, cblocks;              // channel groups (of 8) per CTA, CTAs along the channels
    int strips, segs, TR;        // tile: column strips x row segments of TR output rows
    int IH, IW;                  // input patch
    int tiles_h, tiles_w;
    long long tiles;             // tiles of one channel block, all images
    int ctas;                    // CTAs that share them
    int patch_bytes;
};

// Tiling of the depthwise kernel with the 1x1 task behind it (depthwise_project.cu)
struct DwProjTiling {
    int ok;
    int MT, G, chunks, lanes, panels;        // 128-pixel blocks of a tile, channel groups (of 8) per chunk, chunks, threads per strip, 64-channel panels of a chunk
    int strips, segs, TR, TH, TW, IH, IW;    // tile: column strips x row segments of TR rows; its input patch
    int tiles_h, tiles_w, tiles, ctas, threads;
    int patch_bytes, panel_bytes, w_bytes, k16, k_part, tmem_cols, smem_bytes;
};

// Tiling of the stem kernel that reads a model's float32 image (conv_stem.cu): a step is D conv rows of KF filters each
struct StemTiling {
    int ok;
    int D, KF, RH, N;                        // conv rows of KF filters per step, input rows per step, MMA columns
    int used, ksteps, accs, acc_stride;      // MMA steps (16 values) per input row and per step; accumulators, their distance in columns
    int per, slot, tiles, adv;               // input rows per operand tile, bytes of a window, tiles a step reads, tiles from step to step
    int tile_bytes, raw_bytes, ring, stage_bytes, smem_bytes, steps_per_img;
    size_t weight_offset, weight_bytes;      // its filters behind the task's own in the packed weights
};

struct cprune_plan {
    cprune_plan_info info;
    cprune_task_opts opts;
    int refs;
    // tensor-core family: tensor maps are encoded for a given (x, w) pointer pair and reused
    // while the pointers stay the same
    std::mutex mu;
    const void *map_x = nullptr;
    const void *map_w = nullptr;
    const void *map_y = nullptr;
    const void *map_res = nullptr;
    alignas(64) CUtensorMap tm_a;   // activations (im2col mode)
    alignas(64) CUtensorMap tm_b;   // packed filters
    alignas(64) CUtensorMap tm_y;   // output, for the staged TMA stores
    alignas(64) CUtensorMap tm_res; // residual as an MMA operand (filter-major orientation)
    alignas(64) CUtensorMap tm_id;  // identity matrix
    int smem_bytes = 0;
    int orient = 0;                 // which side of the MMA the pixels are on
    int staging_bufs = 2;
    int fused_pool = 0;             // the 2x2 max-pool runs inside the conv kernel / the split-K finalize kernel
    int splits = 1;                 // split-K slices per output tile
    int ipp = 0;                    // K blocks per slice
    size_t pool_bytes = 0;          // unpooled conv output in the workspace when a 2x2 pool follows
    size_t partial_bytes = 0;       // float32 partial sums in the workspace
    int small_c = 0;                // 3-channel stems: 1 = 8 taps x 8 channels per K block, 2 = pixel pairs
    int s_packed = 0;               // filter taps per row in the packed weights (S, or S + 1 in pair mode)
    int patch = 0;                  // 1: task on the patch kernel (conv_patch.cu)
    int narrow = 0;                 // patch kernel on a regrouped 16-channel input (stems with few channels)
    size_t pre_bytes = 0;           // regrouped input in the workspace
    PatchTiling pt = {};
    DwTiling dw = {};
    StemTiling stem = {};
    int small = 0;                  // 1: task of few pixels on conv_small.cu: 8 / small_kw groups of 16 * small_mt pixels x 8 * small_nt
    int small_mt = 0, small_nt = 0, small_kw = 0;   // filters per block, small_kw warps to a group
    int bias_align = 4;             // alignment of the packed bias that the kernel's widest read of it needs
    double est_us = 0.0;            // the planner's cost-model estimate of the task's time
};

namespace cprune {

// CUDA-core direct convolution, any dense shape (fallback family and small-C stems)
cprune_status launch_conv_direct(const cprune_plan *plan, const void *x, const void *w, const float *b,
                                 const void *res, void *y, cudaStream_t st);
// depthwise 3x3 and 5x5
cprune_status launch_depthwise(cprune_plan *plan, const void *x, const void *w, const float *b,
                               const void *res, void *y, cudaStream_t st);
// channel groups (of 8 channels) one depthwise CTA handles, for c8 groups in the tensor
int depthwise_groups(int c8);
cprune_status plan_depthwise(cprune_plan *plan);    // fills plan->dw
// a depthwise task and the 1x1 task that reads its result as one kernel
bool plan_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, DwProjTiling *out);
// (its tensor maps, of the input and of the 1x1 filters: once for all passes of a model, whose buffers stay where they are)
cprune_status encode_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, const DwProjTiling &t, const void *x, const void *w2, CUtensorMap *tm);
cprune_status launch_depthwise_project(const cprune_plan *dw, const cprune_plan *proj, const DwProjTiling &t, const CUtensorMap *tm, const void *w, const float *b,
                                       const float *b2, const void *res, void *y, cudaStream_t st);
// tcgen05 implicit GEMM
cprune_status plan_conv_tensor(cprune_plan *plan);  // fills tile fields of plan->info; UNSUPPORTED if not eligible
cprune_status launch_conv_tensor(cprune_plan *plan, const void *x, const void *w, const float *b, const void *res,
                                 void *y, void *partial, cudaStream_t st, bool input_regrouped = false);
// tasks of few pixels (part of the tensor family; warp-level MMAs)
bool plan_conv_small(cprune_plan *plan, bool other_is_direct);     // takes the planned task over where it is faster
cprune_status launch_conv_small(const cprune_plan *plan, const void *x, const void *w, const float *b, const void *res, void *y,
                                cudaStream_t st);
// stride-1 R x S > 1 tasks with the input patch resident in shared memory (part of the tensor family)
cprune_status plan_conv_patch(cprune_plan *plan);   // UNSUPPORTED if the task is not eligible or would waste the tile
cprune_status launch_conv_patch(cprune_plan *plan, const void *x, const void *w, const float *b, const void *res,
                                void *y, void *scratch, cudaStream_t st, bool input_regrouped = false);
// regrouped 16-channel input of a stem plan (plan->narrow) written to `scratch` from the benchmark's bf16 input or straight
// from the float32 image (cast and regrouping in one pass)
cprune_status regroup_stem_input(const cprune_plan *plan, const void *x, int x_is_f32, void *scratch, cudaStream_t st);
// cprune_task_run with one more option: the regrouped input of a stem plan is already in the workspace
cprune_status task_run_internal(cprune_plan *plan, const void *x, const void *w_packed, const float *b_packed, const void *residual,
                                void *y, void *workspace, cudaStream_t st, bool input_regrouped);
// where in a task's workspace the regrouped stem input lives
inline void *stem_scratch(const cprune_plan *plan, void *workspace) { return (char *)workspace + plan->pool_bytes; }
// a model's first task straight from the float32 image (fills plan->stem; stem.ok == 0 where it is not supported)
void plan_conv_stem(cprune_plan *plan);
cprune_status pack_conv_stem(const cprune_plan *plan, const float *w, void *w_stem, cudaStream_t st);
cprune_status launch_conv_stem(const cprune_plan *plan, const float *x, const void *w_packed, const float *b, void *y, cudaStream_t st);
// filters of a regrouped stem (plan->narrow) and their size
cprune_status pack_conv_patch(const cprune_plan *plan, const float *w, void *w_packed, cudaStream_t st);
size_t packed_weight_bytes_patch(const cprune_plan *plan);
// tiled bf16 tensor map with a 128- or 32-byte swizzle (inner box extent 64 or 16 elements); out-of-bounds
// elements read as zero
cprune_status encode_tiled_bf16_swz(CUtensorMap *map, const void *ptr, int rank, const unsigned long long *dims,
                                    const unsigned long long *strides_bytes, const unsigned *box, int swizzle_bytes, bool for_loads);
// tiled bf16 tensor map without swizzle, out-of-bounds elements read as zero
cprune_status encode_tiled_bf16(CUtensorMap *map, const void *ptr, int rank, const unsigned long long *dims,
                                const unsigned long long *strides_bytes, const unsigned *box);
// adds the float32 partial sums [splits][M][k_alloc] of a split reduction in index order, then bias, residual (bf16 [M][k_pad]
// or NULL) and activation; y bf16 [M][k_pad]
cprune_status launch_splitk_finalize(const float *partial, int splits, long long M, int k_alloc, int k_pad, const float *bias,
                                     const void *res, int act, void *y, cudaStream_t st);
// 2x2 stride-2 max-pool as a separate pass (used when a plan asks for a pool and the conv kernel
// does not fuse it): x [N][H][W][c] -> y [N][H/2][W/2][c]
cprune_status launch_maxpool(const void *x, int N, int H, int W, int c_pad, int k, int stride, int pad, void *y,
                             cudaStream_t st);

}  // namespace cprune
