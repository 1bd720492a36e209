// Shared host/device helpers of the cprune library (status word, error capture, bf16 vectors).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cprune.h"

namespace cprune {

// bits of the device status word
enum : int { STATUS_TIMEOUT = 1, STATUS_BAD_DATA = 2 };

// Device address of the per-device status word (resolved once per device).
int *device_status_word();

// Records a failing CUDA call for cprune_last_cuda_error() and returns CPRUNE_ERR_CUDA.
cprune_status cuda_fail(cudaError_t e, const char *what);

#define CPRUNE_CUDA_CHECK(expr)                                     \
    do {                                                            \
        cudaError_t e__ = (expr);                                   \
        if (e__ != cudaSuccess) return ::cprune::cuda_fail(e__, #expr); \
    } while (0)

#define CPRUNE_LAUNCH_CHECK(name)                                   \
    do {                                                            \
        cudaError_t e__ = cudaGetLastError();                       \
        if (e__ != cudaSuccess) return ::cprune::cuda_fail(e__, name); \
    } while (0)

// Programmatic dependent launch.  A kernel of a model's launch chain lets its successor start as early as possible
// (pdl_trigger) and waits for its predecessor's results (pdl_wait) only after its own set-up, so that launch
// latency and set-up overlap the predecessor's tail.  Both are no-ops in a kernel launched the ordinary way.
// A kernel that uses tensor memory lets its successor start only once it has its columns: a block of a later kernel that got them first
// would keep them while it waits for this kernel, which would wait for them, and an allocation has no limit.  (The warp that allocates triggers.)
// A chain begins with a kernel that waits BEFORE it lets its successor start (cast, regrouping, stem): everything that was enqueued
// before the chain is then complete when the second kernel starts.  Kernels may therefore read packed parameters ahead of their wait,
// even those that a kernel just before the chain packed, and no kernel of a pass starts while the pass before it still reads the
// same activations (whose lines could stay in an L1).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// True while the calling thread enqueues a chain whose kernels may overlap their predecessors' tails.
bool chain_launch_enabled();
void set_chain_launch(bool on);

// Launches a kernel that calls pdl_wait() before it touches what its predecessors write; inside a chain the launch carries the
// programmatic-serialization attribute.  pair: clusters of two blocks.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained_as(bool pair, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (chain_launch_enabled()) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (pair) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = 2;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    return launch_chained_as(false, kernel, grid, block, smem, st, static_cast<Args &&>(args)...);
}

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }
inline long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

__device__ __forceinline__ float apply_act(float v, int act) {
    if (act == CPRUNE_ACT_RELU) return fmaxf(v, 0.f);
    if (act == CPRUNE_ACT_RELU6) return fminf(fmaxf(v, 0.f), 6.f);
    return v;
}

// 8 bf16 values carried in one 16-byte vector.  The members are plain words so that a copy of the struct is ONE 16-byte
// load or store (with __nv_bfloat162 members, whose assignment is user-defined, it is four 4-byte ones).
struct alignas(16) bf16x8 {
    uint32_t w[4];
};

__device__ __forceinline__ bf16x8 ldg8(const bf16x8 *p) {
    uint4 u = __ldg(reinterpret_cast<const uint4 *>(p));
    bf16x8 r;
    r.w[0] = u.x; r.w[1] = u.y; r.w[2] = u.z; r.w[3] = u.w;
    return r;
}

__device__ __forceinline__ void unpack8(const bf16x8 &a, float *f) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // a bf16 is the upper half of the float32 with the same value
        f[2 * i] = __uint_as_float(a.w[i] << 16);
        f[2 * i + 1] = __uint_as_float(a.w[i] & 0xffff0000u);
    }
}

__device__ __forceinline__ bf16x8 pack8(const float *f) {
    bf16x8 r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        r.w[i] = *reinterpret_cast<const uint32_t *>(&t);
    }
    return r;
}

// D += A x B for one warp: A 16 rows x 16, B 16 x 8, bf16 factors, float32 sums.
__device__ __forceinline__ void mma_16816(float *d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

}  // namespace cprune
