// L1-norm filter selection and slicing (paper Sec. 3.5, last paragraph; Sec. 2.1 / Fig. 2).
//
// Two kernels on the caller's stream:
//   l1_norm_kernel       one CTA per filter: n_k = sum rint(|w| * 2^40) as int64 (order independent)
//   select_slice_kernel  every CTA works out the ascending list of kept filters for itself, in shared memory, and copies its
//                        share of w[kept], b[kept] and w_next[:, kept] (or w_next[kept] for a depthwise consumer)
// What bounds them is latency: the copies are a few megabytes.  One kernel each for ranking, compaction and every slice cost
// six launches that wait for one another: 512 filters of 512 x 3 x 3 with their consumer took 40.4 us per call; with every
// CTA repeating the selection (a few thousand cycles, all at the same time) the call takes 23.8 us.  More than SELECT_MAX
// filters (whose norms do not fit a CTA's shared memory) take the separate kernels:
//   rank_kernel      rank_k = #{j : n_j > n_k or (n_j == n_k and j < k)};  keep_k = rank_k < keep
//   compact_kernel   ascending list of the kept indices (single CTA, chunked block scan)
//   gather kernels
#include <mutex>
#include <string>

#include "common.cuh"

namespace cprune {

__device__ int g_status_word;

static thread_local std::string t_last_error;

cprune_status cuda_fail(cudaError_t e, const char *what) {
    t_last_error = std::string(what) + ": " + cudaGetErrorString(e);
    (void)cudaGetLastError();
    return CPRUNE_ERR_CUDA;
}

int *device_status_word() {
    static std::mutex mu;
    static int *ptrs[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!ptrs[dev]) {
        int *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, g_status_word) != cudaSuccess) return nullptr;
        ptrs[dev] = p;
    }
    return ptrs[dev];
}

constexpr int NORM_THREADS = 256;

// accumulate != 0: the norm is added to what norms[] holds (integer adds: any order gives the same bits)
__global__ void __launch_bounds__(NORM_THREADS) l1_norm_kernel(const float *__restrict__ w, size_t inner,
                                                                long long *__restrict__ norms, int *status, int accumulate) {
    pdl_trigger();
    const float *row = w + (size_t)blockIdx.x * inner;
    long long acc = 0;
    bool bad = false;
    auto add = [&](float v) {
        const float a = fabsf(v);
        bad |= !(a < 1024.f);  // also catches NaN and Inf
        acc += __double2ll_rn((double)a * 1099511627776.0);
    };
    if (((reinterpret_cast<uintptr_t>(row) | (inner * sizeof(float))) & 15) == 0) {
        const float4 *row4 = reinterpret_cast<const float4 *>(row);
        const int n4 = (int)(inner >> 2);
        for (int i0 = threadIdx.x; i0 < n4; i0 += 4 * NORM_THREADS) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = i0 + u * NORM_THREADS < n4 ? __ldg(row4 + i0 + u * NORM_THREADS) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) { add(v[u].x); add(v[u].y); add(v[u].z); add(v[u].w); }
        }
    } else {
        for (size_t i = threadIdx.x; i < inner; i += NORM_THREADS) add(row[i]);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ long long part[NORM_THREADS / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    if (bad) atomicOr(status, STATUS_BAD_DATA);
    __syncthreads();
    if (threadIdx.x == 0) {
        long long s = 0;
        for (int i = 0; i < NORM_THREADS / 32; ++i) s += part[i];
        norms[blockIdx.x] = accumulate ? norms[blockIdx.x] + s : s;
    }
}

constexpr int RANK_THREADS = 256;

__global__ void __launch_bounds__(RANK_THREADS) rank_kernel(const long long *__restrict__ norms, int K, int keep_k,
                                                             int *__restrict__ keep) {
    __shared__ long long tile[RANK_THREADS];
    int k = blockIdx.x * RANK_THREADS + threadIdx.x;
    long long mine = k < K ? norms[k] : 0;
    int rank = 0;
    for (int base = 0; base < K; base += RANK_THREADS) {
        int j = base + threadIdx.x;
        tile[threadIdx.x] = j < K ? norms[j] : 0;
        __syncthreads();
        int lim = min(RANK_THREADS, K - base);
        for (int t = 0; t < lim; ++t) {
            long long other = tile[t];
            int jj = base + t;
            rank += (other > mine) || (other == mine && jj < k);
        }
        __syncthreads();
    }
    if (k < K) keep[k] = rank < keep_k ? 1 : 0;
}

constexpr int COMPACT_THREADS = 1024;

__global__ void __launch_bounds__(COMPACT_THREADS) compact_kernel(const int *__restrict__ keep, int K,
                                                                  int *__restrict__ kept_idx) {
    __shared__ int warp_sum[COMPACT_THREADS / 32];
    __shared__ int running;
    if (threadIdx.x == 0) running = 0;
    __syncthreads();
    for (int base = 0; base < K; base += COMPACT_THREADS) {
        int k = base + threadIdx.x;
        int f = k < K ? keep[k] : 0;
        int incl = f;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if ((threadIdx.x & 31) >= o) incl += t;
        }
        if ((threadIdx.x & 31) == 31) warp_sum[threadIdx.x >> 5] = incl;
        __syncthreads();
        int before = running;
        for (int wi = 0; wi < (int)(threadIdx.x >> 5); ++wi) before += warp_sum[wi];
        if (f) kept_idx[before + incl - 1] = k;
        __syncthreads();
        if (threadIdx.x == COMPACT_THREADS - 1) running = before + incl;
        __syncthreads();
    }
}

// out[j][i] = in[idx[j]][i]
__global__ void gather_rows_kernel(const float *__restrict__ in, size_t inner, const int *__restrict__ idx,
                                   int n_idx, float *__restrict__ out) {
    size_t total = (size_t)n_idx * inner;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        size_t j = e / inner, i = e - j * inner;
        out[e] = in[(size_t)idx[j] * inner + i];
    }
}

// out[o][j][i] = in[o][idx[j]][i]
__global__ void gather_cols_kernel(const float *__restrict__ in, int outer, int cols, size_t inner,
                                   const int *__restrict__ idx, int n_idx, float *__restrict__ out) {
    size_t total = (size_t)outer * n_idx * inner;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        size_t i = e % inner;
        size_t t = e / inner;
        size_t j = t % n_idx, o = t / n_idx;
        out[e] = in[((size_t)o * cols + idx[j]) * inner + i];
    }
}

constexpr int SLICE_THREADS = 256;
constexpr int SELECT_MAX = 8192;          // norms and list in shared memory: 12 bytes per filter

struct SliceParams {
    const long long *norms;
    int K, keep_k;
    int *kept_idx;
    const float *w;          // null: only the list is wanted
    float *w_out;
    size_t inner;            // floats per filter of w
    const float *b;
    float *b_out;
    const float *wn;         // consumer, or null: wn_outer x (K of which keep_k are kept) x wn_inner
    float *wn_out;
    int wn_outer, wn_inner;
    int row_ctas;            // CTAs that copy filters of w; the others copy the consumer
};

// The ascending list of the keep_k largest norms (ties: lower index) of the K in `key`, by the CTA: a radix selection finds
// the smallest kept norm eight bits at a time, a scan over the filters then places every kept one.
__device__ __forceinline__ void select_list(const long long *key, int K, int keep_k, int *list) {
    __shared__ int hist[256];
    __shared__ unsigned long long top;
    __shared__ int digit_s, need_s;
    __shared__ int warp_sum[SLICE_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long all = 0;
    for (int k = tid; k < K; k += SLICE_THREADS) all |= (unsigned long long)key[k];
    if (tid == 0) top = 0;
    __syncthreads();
    {
        unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)all), hi = __reduce_or_sync(0xffffffffu, (unsigned)(all >> 32));
        if (lane == 0) atomicOr(&top, ((unsigned long long)hi << 32) | lo);
    }
    __syncthreads();
    // norms are never negative, unless weights that break the precondition (infinite, NaN) made them so: these rank last
    const unsigned long long flip = top & (1ull << 63);
    unsigned long long prefix = 0;
    int need = keep_k;                     // how many of the norms that share the prefix are kept
    int shift = top ? (63 - __clzll((long long)top)) / 8 * 8 : 0;
    for (; shift >= 0; shift -= 8) {
        hist[tid] = 0;
        __syncthreads();
        for (int k = tid; k < K; k += SLICE_THREADS) {
            const unsigned long long v = (unsigned long long)key[k] ^ flip;
            if (((v ^ prefix) >> shift) < 256) atomicAdd(&hist[(int)((v >> shift) & 255)], 1);
        }
        __syncthreads();
        if (warp == 0) {
            // lane l holds the eight digits 255 - 8 l downwards; the digit at which the count from above reaches `need`
            int c[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) { c[j] = hist[255 - (lane * 8 + j)]; sum += c[j]; }
            int before = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o) before += t;
            }
            before -= sum;
            if (before < need && need <= before + sum) {
                int j = 0;
                while (before + c[j] < need) { before += c[j]; ++j; }
                digit_s = 255 - (lane * 8 + j);
                need_s = need - before;
            }
        }
        __syncthreads();
        prefix |= (unsigned long long)digit_s << shift;
        need = need_s;
    }
    // `prefix` is the smallest kept norm, `need` how many filters that have exactly it are kept: those with the lowest indices
    const int per = (K + SLICE_THREADS - 1) / SLICE_THREADS;
    const int k0 = min(tid * per, K), k1 = min(k0 + per, K);
    int mine = 0;                          // larger norms (upper half) and equal norms (lower half) among this thread's filters
    for (int k = k0; k < k1; ++k) {
        const unsigned long long v = (unsigned long long)key[k] ^ flip;
        mine += (v > prefix ? 1 << 16 : 0) + (v == prefix ? 1 : 0);
    }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int at = incl - mine;
    for (int q = 0; q < warp; ++q) at += warp_sum[q];
    int larger = at >> 16, equal = at & 0xffff;
    for (int k = k0; k < k1; ++k) {
        const unsigned long long v = (unsigned long long)key[k] ^ flip;
        if (v > prefix) {
            list[larger + min(equal, need)] = k;
            ++larger;
        } else if (v == prefix) {
            if (equal < need) list[larger + equal] = k;
            ++equal;
        }
    }
    __syncthreads();
}

// out[j][i] = in[list[j]][i], elements e0 .. e1 of the output
template <int INNER>
__device__ __forceinline__ void slice_columns(const float *__restrict__ in, float *__restrict__ out, const int *list, int inner_rt, int e0, int e1) {
    const int inner = INNER ? INNER : inner_rt;
    for (int e = e0 + (int)threadIdx.x; e < e1; e += 4 * SLICE_THREADS) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = e + u * SLICE_THREADS;
            if (q < e1) {
                const int j = q / inner;
                v[u] = __ldg(in + (size_t)list[j] * inner + (q - j * inner));
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (e + u * SLICE_THREADS < e1) out[e + u * SLICE_THREADS] = v[u];
    }
}

__global__ void __launch_bounds__(SLICE_THREADS) select_slice_kernel(const SliceParams p) {
    extern __shared__ __align__(16) unsigned char slice_smem[];
    long long *key = reinterpret_cast<long long *>(slice_smem);
    int *list = reinterpret_cast<int *>(key + p.K);
    pdl_wait();
    for (int k = threadIdx.x; k < p.K; k += SLICE_THREADS) key[k] = p.norms[k];
    __syncthreads();
    select_list(key, p.K, p.keep_k, list);
    if (blockIdx.x == 0)
        for (int j = threadIdx.x; j < p.keep_k; j += SLICE_THREADS) {
            p.kept_idx[j] = list[j];
            if (p.b) p.b_out[j] = __ldg(p.b + list[j]);
        }
    if (!p.w) return;
    if ((int)blockIdx.x < p.row_ctas) {
        const bool vec = (((uintptr_t)p.w | (uintptr_t)p.w_out | (p.inner * 4)) & 15) == 0;
        if (vec && p.inner >= 256) {
            const int n4 = (int)(p.inner >> 2);
            for (int j = blockIdx.x; j < p.keep_k; j += p.row_ctas) {
                const float4 *src = reinterpret_cast<const float4 *>(p.w) + (size_t)list[j] * n4;
                float4 *dst = reinterpret_cast<float4 *>(p.w_out) + (size_t)j * n4;
                for (int i0 = threadIdx.x; i0 < n4; i0 += 4 * SLICE_THREADS) {
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i0 + u * SLICE_THREADS < n4) v[u] = __ldg(src + i0 + u * SLICE_THREADS);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i0 + u * SLICE_THREADS < n4) dst[i0 + u * SLICE_THREADS] = v[u];
                }
            }
        } else {
            // short or unaligned rows: all kept filters as one run of elements
            const int total = p.keep_k * (int)p.inner, per = (total + p.row_ctas - 1) / p.row_ctas;
            const int e0 = min((int)blockIdx.x * per, total);
            slice_columns<0>(p.w, p.w_out, list, (int)p.inner, e0, min(e0 + per, total));
        }
    } else if (p.wn) {
        // the consumer: several CTAs per outer index when there are few of those
        const int cta = blockIdx.x - p.row_ctas, ctas = gridDim.x - p.row_ctas;
        const int row = p.keep_k * p.wn_inner;
        const int parts = max(1, ctas / p.wn_outer), per = (row + parts - 1) / parts;
        for (int u = cta; u < p.wn_outer * parts; u += ctas) {
            const int o = u / parts, e0 = min((u - o * parts) * per, row), e1 = min(e0 + per, row);
            const float *in = p.wn + (size_t)o * p.K * p.wn_inner;
            float *out = p.wn_out + (size_t)o * row;
            if (p.wn_inner == 9) slice_columns<9>(in, out, list, 9, e0, e1);
            else if (p.wn_inner == 1) slice_columns<1>(in, out, list, 1, e0, e1);
            else slice_columns<0>(in, out, list, p.wn_inner, e0, e1);
        }
    }
}

// Scratch of the allocation-free entry point: norms (int64) followed by keep flags (int32) for up
// to CPRUNE_SELECT_STATIC_MAX_FILTERS filters.  In host code this name is only a handle for
// cudaGetSymbolAddress, never a pointer that a kernel may be given.
constexpr size_t STATIC_NORM_BYTES = (size_t)CPRUNE_SELECT_STATIC_MAX_FILTERS * sizeof(long long);
constexpr size_t STATIC_KEEP_BYTES = (size_t)CPRUNE_SELECT_STATIC_MAX_FILTERS * sizeof(int);
static __device__ __align__(256) unsigned char g_select_scratch[STATIC_NORM_BYTES + STATIC_KEEP_BYTES];

// Device address of g_select_scratch on the current device, looked up once per device.
static cprune_status select_scratch_address(unsigned char **out) {
    static std::mutex mu;
    static unsigned char *ptrs[64] = {nullptr};
    int dev = 0;
    CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(mu);
    if (!ptrs[dev]) {
        unsigned char *p = nullptr;
        CPRUNE_CUDA_CHECK(cudaGetSymbolAddress((void **)&p, g_select_scratch));
        ptrs[dev] = p;
    }
    *out = ptrs[dev];
    return CPRUNE_OK;
}

static int grid_for(size_t total, int threads) {
    size_t g = (total + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 148 * 16) g = 148 * 16;
    return (int)g;
}

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

static cprune_status launch_select_slice(SliceParams p, cudaStream_t st) {
    // about four CTAs per SM, shared between the two copies in proportion to what they move (at least 4 KB per CTA)
    const double rows = p.w ? (double)p.keep_k * p.inner : 0.0;
    const double cols = p.wn ? (double)p.wn_outer * p.keep_k * p.wn_inner : 0.0;
    const int most = 148 * 4;
    double ctas = (rows + cols) / 1024.0;
    if (ctas > most) ctas = most;
    int rc = (int)(ctas * rows / (rows + cols + 1.0) + 0.5), cc = (int)(ctas * cols / (rows + cols + 1.0) + 0.5);
    if (rc < 1) rc = 1;
    if (cc < 1) cc = p.wn ? 1 : 0;
    p.row_ctas = rc;
    const size_t smem = (size_t)p.K * (sizeof(long long) + sizeof(int));
    static std::mutex attr_mu;
    static bool attr_set[64] = {false};    // the shared-memory limit of a kernel is a per-device attribute
    {
        int dev = 0;
        CPRUNE_CUDA_CHECK(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return CPRUNE_ERR_UNSUPPORTED;
        std::lock_guard<std::mutex> lock(attr_mu);
        if (!attr_set[dev]) {
            CPRUNE_CUDA_CHECK(cudaFuncSetAttribute(select_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SELECT_MAX * 12));
            attr_set[dev] = true;
        }
    }
    // may start while the norms are being computed (it waits for them)
    const bool chained = chain_launch_enabled();
    set_chain_launch(true);
    const cudaError_t e = launch_chained(select_slice_kernel, dim3((unsigned)(rc + cc)), dim3(SLICE_THREADS), smem, st, p);
    set_chain_launch(chained);
    if (e != cudaSuccess) return cuda_fail(e, "select_slice_kernel");
    return CPRUNE_OK;
}

cprune_status select_launch(const float *w, const float *b, int K, int C, int R, int S, int keep_k,
                            const float *w_next, int K2, int R2, int S2, int next_is_depthwise, int32_t *kept_idx,
                            float *w_out, float *b_out, float *w_next_out, long long *norms, int *keep,
                            int *status, cudaStream_t st) {
    size_t inner = (size_t)C * R * S;
    l1_norm_kernel<<<K, NORM_THREADS, 0, st>>>(w, inner, norms, status, 0);
    CPRUNE_LAUNCH_CHECK("l1_norm_kernel");
    if (K <= SELECT_MAX && (size_t)keep_k * R2 * S2 < ((size_t)1 << 30)) {
        SliceParams p = {norms, K, keep_k, kept_idx, w, w_out, inner, b, b_out, w_next, w_next_out,
                         next_is_depthwise ? 1 : K2, R2 * S2, 0};
        return launch_select_slice(p, st);
    }
    rank_kernel<<<(K + RANK_THREADS - 1) / RANK_THREADS, RANK_THREADS, 0, st>>>(norms, K, keep_k, keep);
    CPRUNE_LAUNCH_CHECK("rank_kernel");
    compact_kernel<<<1, COMPACT_THREADS, 0, st>>>(keep, K, kept_idx);
    CPRUNE_LAUNCH_CHECK("compact_kernel");
    gather_rows_kernel<<<grid_for((size_t)keep_k * inner, 256), 256, 0, st>>>(w, inner, kept_idx, keep_k, w_out);
    CPRUNE_LAUNCH_CHECK("gather_rows_kernel");
    if (b) {
        gather_rows_kernel<<<grid_for(keep_k, 256), 256, 0, st>>>(b, 1, kept_idx, keep_k, b_out);
        CPRUNE_LAUNCH_CHECK("gather_rows_kernel");
    }
    if (w_next) {
        size_t in2 = (size_t)R2 * S2;
        if (next_is_depthwise) {
            gather_rows_kernel<<<grid_for((size_t)keep_k * in2, 256), 256, 0, st>>>(w_next, in2, kept_idx, keep_k,
                                                                                    w_next_out);
        } else {
            gather_cols_kernel<<<grid_for((size_t)K2 * keep_k * in2, 256), 256, 0, st>>>(w_next, K2, K, in2, kept_idx,
                                                                                         keep_k, w_next_out);
        }
        CPRUNE_LAUNCH_CHECK("gather consumer");
    }
    return CPRUNE_OK;
}

}  // namespace cprune

using namespace cprune;

extern "C" {

const char *cprune_status_string(cprune_status s) {
    switch (s) {
        case CPRUNE_OK: return "ok";
        case CPRUNE_ERR_INVALID_ARG: return "invalid argument";
        case CPRUNE_ERR_UNSUPPORTED: return "unsupported";
        case CPRUNE_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case CPRUNE_ERR_CUDA: return "CUDA error";
        case CPRUNE_ERR_TIMEOUT: return "device-side wait timed out";
        case CPRUNE_ERR_INTERNAL: return "internal error";
        case CPRUNE_ERR_BAD_DATA: return "non-finite or out-of-range weight";
    }
    return "unknown status";
}

const char *cprune_last_cuda_error(void) { return t_last_error.c_str(); }

int cprune_padded_channels(int C) { return C <= 0 ? 0 : (C <= 128 ? (C + 7) / 8 * 8 : (C + 15) / 16 * 16); }

size_t cprune_select_workspace_bytes(int K) {
    if (K <= 0) return 0;
    return align_up((size_t)K * sizeof(long long), 256) + align_up((size_t)K * sizeof(int), 256);
}

cprune_status cprune_select_filters(const float *w, const float *b, int K, int C, int R, int S, int keep_k,
                                    const float *w_next, int K2, int R2, int S2, int next_is_depthwise,
                                    int32_t *kept_idx, float *w_out, float *b_out, float *w_next_out,
                                    void *workspace, size_t workspace_bytes, void *stream) {
    if (!w || !kept_idx || !w_out || K <= 0 || C <= 0 || R <= 0 || S <= 0) return CPRUNE_ERR_INVALID_ARG;
    if (keep_k < 1 || keep_k > K) return CPRUNE_ERR_INVALID_ARG;
    if (b && !b_out) return CPRUNE_ERR_INVALID_ARG;
    if (w_next && (!w_next_out || R2 <= 0 || S2 <= 0 || (!next_is_depthwise && K2 <= 0))) return CPRUNE_ERR_INVALID_ARG;
    if ((size_t)C * R * S > 8192) return CPRUNE_ERR_UNSUPPORTED;
    if (!workspace || ((uintptr_t)workspace & 15)) return CPRUNE_ERR_INVALID_ARG;
    if (workspace_bytes < cprune_select_workspace_bytes(K)) return CPRUNE_ERR_WORKSPACE_TOO_SMALL;
    int *status = device_status_word();
    if (!status) return cuda_fail(cudaGetLastError(), "status word");
    long long *norms = (long long *)workspace;
    int *keep = (int *)((char *)workspace + align_up((size_t)K * sizeof(long long), 256));
    return select_launch(w, b, K, C, R, S, keep_k, w_next, K2, R2, S2, next_is_depthwise, kept_idx, w_out, b_out,
                         w_next_out, norms, keep, status, (cudaStream_t)stream);
}

cprune_status cprune_select_filters_static(const float *w, const float *b, int K, int C, int R, int S, int keep_k,
                                           const float *w_next, int K2, int R2, int S2, int next_is_depthwise,
                                           int32_t *kept_idx, float *w_out, float *b_out, float *w_next_out,
                                           void *stream) {
    if (!w || !kept_idx || !w_out || K <= 0 || C <= 0 || R <= 0 || S <= 0) return CPRUNE_ERR_INVALID_ARG;
    if (keep_k < 1 || keep_k > K) return CPRUNE_ERR_INVALID_ARG;
    if (b && !b_out) return CPRUNE_ERR_INVALID_ARG;
    if (w_next && (!w_next_out || R2 <= 0 || S2 <= 0 || (!next_is_depthwise && K2 <= 0))) return CPRUNE_ERR_INVALID_ARG;
    if ((size_t)C * R * S > 8192) return CPRUNE_ERR_UNSUPPORTED;
    if (K > CPRUNE_SELECT_STATIC_MAX_FILTERS) return CPRUNE_ERR_WORKSPACE_TOO_SMALL;   // beyond the fixed buffer
    unsigned char *scratch = nullptr;
    cprune_status st = select_scratch_address(&scratch);
    if (st != CPRUNE_OK) return st;
    int *status = device_status_word();
    if (!status) return cuda_fail(cudaGetLastError(), "status word");
    // every norm and keep flag below K is written before it is read, so stale contents are harmless
    long long *norms = (long long *)scratch;
    int *keep = (int *)(scratch + STATIC_NORM_BYTES);
    return select_launch(w, b, K, C, R, S, keep_k, w_next, K2, R2, S2, next_is_depthwise, kept_idx, w_out, b_out,
                         w_next_out, norms, keep, status, (cudaStream_t)stream);
}

cprune_status cprune_select_shared(const float *const *w_list, const size_t *inner, int n_members, int K, int keep_k,
                                   int32_t *kept_idx, void *workspace, size_t workspace_bytes, void *stream) {
    if (!w_list || !inner || n_members < 1 || K <= 0 || !kept_idx) return CPRUNE_ERR_INVALID_ARG;
    if (keep_k < 1 || keep_k > K) return CPRUNE_ERR_INVALID_ARG;
    for (int m = 0; m < n_members; ++m) {
        if (!w_list[m] || inner[m] == 0) return CPRUNE_ERR_INVALID_ARG;
        if (inner[m] > 8192) return CPRUNE_ERR_UNSUPPORTED;
    }
    if ((size_t)n_members > (size_t)1 << 9) return CPRUNE_ERR_UNSUPPORTED;   // keeps the int64 sums far from overflow
    if (!workspace || ((uintptr_t)workspace & 15)) return CPRUNE_ERR_INVALID_ARG;
    if (workspace_bytes < cprune_select_workspace_bytes(K)) return CPRUNE_ERR_WORKSPACE_TOO_SMALL;
    int *status = device_status_word();
    if (!status) return cuda_fail(cudaGetLastError(), "status word");
    cudaStream_t st = (cudaStream_t)stream;
    long long *norms = (long long *)workspace;
    int *keep = (int *)((char *)workspace + align_up((size_t)K * sizeof(long long), 256));
    for (int m = 0; m < n_members; ++m) {
        l1_norm_kernel<<<K, NORM_THREADS, 0, st>>>(w_list[m], inner[m], norms, status, m > 0);
        CPRUNE_LAUNCH_CHECK("l1_norm_kernel");
    }
    if (K <= SELECT_MAX) {
        SliceParams p = {norms, K, keep_k, kept_idx, nullptr, nullptr, 0, nullptr, nullptr, nullptr, nullptr, 0, 0, 0};
        return launch_select_slice(p, st);
    }
    rank_kernel<<<(K + RANK_THREADS - 1) / RANK_THREADS, RANK_THREADS, 0, st>>>(norms, K, keep_k, keep);
    CPRUNE_LAUNCH_CHECK("rank_kernel");
    compact_kernel<<<1, COMPACT_THREADS, 0, st>>>(keep, K, kept_idx);
    CPRUNE_LAUNCH_CHECK("compact_kernel");
    return CPRUNE_OK;
}

cprune_status cprune_gather_rows(const float *in, int rows, size_t inner, const int32_t *idx, int n_idx, float *out,
                                 void *stream) {
    if (!in || !idx || !out || rows <= 0 || inner == 0 || n_idx <= 0 || n_idx > rows) return CPRUNE_ERR_INVALID_ARG;
    gather_rows_kernel<<<grid_for((size_t)n_idx * inner, 256), 256, 0, (cudaStream_t)stream>>>(in, inner, idx, n_idx, out);
    CPRUNE_LAUNCH_CHECK("gather_rows_kernel");
    return CPRUNE_OK;
}

cprune_status cprune_gather_columns(const float *in, int outer, int cols, size_t inner, const int32_t *idx, int n_idx,
                                    float *out, void *stream) {
    if (!in || !idx || !out || outer <= 0 || cols <= 0 || inner == 0 || n_idx <= 0 || n_idx > cols)
        return CPRUNE_ERR_INVALID_ARG;
    gather_cols_kernel<<<grid_for((size_t)outer * n_idx * inner, 256), 256, 0, (cudaStream_t)stream>>>(
        in, outer, cols, inner, idx, n_idx, out);
    CPRUNE_LAUNCH_CHECK("gather_cols_kernel");
    return CPRUNE_OK;
}

cprune_status cprune_poll_device_status(void *stream) {
    int *status = device_status_word();
    if (!status) return cuda_fail(cudaGetLastError(), "status word");
    int h = 0;
    cudaStream_t st = (cudaStream_t)stream;
    CPRUNE_CUDA_CHECK(cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st));
    CPRUNE_CUDA_CHECK(cudaStreamSynchronize(st));
    if (h) {
        CPRUNE_CUDA_CHECK(cudaMemsetAsync(status, 0, sizeof(int), st));
        CPRUNE_CUDA_CHECK(cudaStreamSynchronize(st));
    }
    if (h & STATUS_TIMEOUT) return CPRUNE_ERR_TIMEOUT;
    if (h & STATUS_BAD_DATA) return CPRUNE_ERR_BAD_DATA;
    return CPRUNE_OK;
}

}  // extern "C"
