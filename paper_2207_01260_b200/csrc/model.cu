// Whole-model runner: the aggregate of a network's tasks enqueued back to back on one stream
// (paper Sec. 3.1: the model is the aggregate of its tasks' programs and is timed as a whole),
// optionally replayed as a CUDA graph so that one replay costs one host call.
#include <map>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "plan.h"

struct ModelTensor {
    int n = 0, h = 0, w = 0, c = 0, c_pad = 0;
    size_t offset = 0, bytes = 0;
    bool defined = false;
};

// A depthwise task that runs as one kernel with the next task
struct ModelPair {
    DwProjTiling t = {};                 // t.ok: it does
    CUtensorMap tm[2];
};

struct cprune_model {
    int N, H, W, C;
    mutable std::mutex mu;               // pairs, graphs and launches change when a tensor's address is handed out, perhaps by another thread
    bool ran = false;                    // a pass has been enqueued
    std::vector<cprune_task_desc> tasks;
    std::vector<ModelPair> pairs;        // per task
    std::map<int, ModelTensor> tensors;
    char *arena = nullptr;
    size_t arena_bytes = 0;
    char *workspace = nullptr;
    size_t workspace_bytes = 0;
    int classes = 0;
    int launches = 0;
    // captured launch sequences: slot 2 serves cprune_model_run, slots 0 and 1 the two device-side
    // input buffers of cprune_model_run_host
    struct GraphSlot {
        cudaGraphExec_t exec = nullptr;
        const float *x = nullptr;
        float *logits = nullptr;
        cudaStream_t stream = nullptr;
    } graphs[3];
    cudaStream_t capture_stream = nullptr;   // private stream the launch sequence is recorded on
    // host-buffer path: double-buffered device copies of the input and of the logits
    float *host_x[2] = {nullptr, nullptr};
    float *host_logits[2] = {nullptr, nullptr};
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t copied[2] = {nullptr, nullptr}, done[2] = {nullptr, nullptr};
    unsigned long long host_calls = 0;
};

namespace cprune {

static size_t align256(size_t v) { return (v + 255) / 256 * 256; }

static void *tensor_ptr(const cprune_model *m, int id) {
    auto it = m->tensors.find(id);
    return it == m->tensors.end() ? nullptr : (void *)(m->arena + it->second.offset);
}

static cprune_status enqueue_chain(cprune_model *m, const float *x, float *logits, cudaStream_t st);

// The kernels of one pass are launched as a chain: each may start while its predecessor drains (see common.cuh).
static cprune_status enqueue(cprune_model *m, const float *x, float *logits, cudaStream_t st) {
    set_chain_launch(true);
    cprune_status s = enqueue_chain(m, x, logits, st);
    set_chain_launch(false);
    return s;
}

// Pairs of a depthwise task and the 1x1 task that reads its result, run as one kernel where the caller allows it
// (CPRUNE_CONV_WITH_NEXT) and nothing else reads the tensor between them, which is then not stored.  Filters and biases that the
// kernel cannot read where they are (off 16 and 4 bytes) leave the tasks separate, and a pass refuses them as the tasks do.
static void find_pairs(cprune_model *m) {
    m->pairs.assign(m->tasks.size(), ModelPair());
    for (size_t t = 0; t + 1 < m->tasks.size(); ++t) {
        const cprune_task_desc &d = m->tasks[t], &e = m->tasks[t + 1];
        if (d.op != CPRUNE_OP_CONV || e.op != CPRUNE_OP_CONV || d.p0 != CPRUNE_CONV_WITH_NEXT || e.in != d.out || e.res == d.out) continue;
        bool read = false;
        for (size_t u = t + 2; u < m->tasks.size(); ++u) read = read || m->tasks[u].in == d.out || m->tasks[u].res == d.out;
        const bool aligned = !(((uintptr_t)d.w | (uintptr_t)e.w) & 15) && !(((uintptr_t)d.b | (uintptr_t)e.b) & 3);
        if (!read && aligned) plan_depthwise_project(d.plan, e.plan, &m->pairs[t].t);
    }
}

// The depthwise task whose result the passes do not store, or -1.
static int unstored(const cprune_model *m, int id) {
    for (size_t t = 0; t < m->pairs.size(); ++t)
        if (m->pairs[t].t.ok && m->tasks[t].out == id) return (int)t;
    return -1;
}

static cprune_status store_tensor(const cprune_model *m, int t, cudaStream_t st) {
    const cprune_task_desc &d = m->tasks[t];
    return task_run_internal(d.plan, tensor_ptr(m, d.in), d.w, d.b, nullptr, tensor_ptr(m, d.out), m->workspace, st, false);
}

// How the model's first task gets at the float32 image when it is the only reader of the input: straight (the stem kernel
// casts on the way in), through the regrouped copy of the patch kernel (cast and regrouping in one pass), or, otherwise,
// from the bf16 NHWC copy that every model can make.  The stem kernel's bulk copies need an image on a 16-byte boundary.
enum { INPUT_CAST = 0, INPUT_REGROUP = 1, INPUT_DIRECT = 2 };
static int input_path(const cprune_model *m, bool aligned = true) {
    if (m->tasks.empty()) return INPUT_CAST;
    const cprune_task_desc &d0 = m->tasks[0];
    if (d0.op != CPRUNE_OP_CONV || d0.in != 0 || d0.res == 0 || !d0.plan) return INPUT_CAST;
    for (size_t t = 1; t < m->tasks.size(); ++t)
        if (m->tasks[t].in == 0 || m->tasks[t].res == 0) return INPUT_CAST;
    if (d0.plan->stem.ok && aligned) return INPUT_DIRECT;
    return d0.plan->patch && d0.plan->narrow ? INPUT_REGROUP : INPUT_CAST;
}

// Kernels that one run of a conv task enqueues.
static int conv_launches(const cprune_plan *plan) {
    const bool tensor = plan->info.kernel == CPRUNE_KERNEL_TENSOR;
    return 1 + (plan->opts.pool && !(tensor && plan->fused_pool) ? 1 : 0) + (plan->splits > 1 ? 1 : 0) + (plan->patch && plan->narrow ? 1 : 0);
}

// The model's first task from the float32 image (path: INPUT_DIRECT or INPUT_REGROUP).
static cprune_status run_first_task(const cprune_model *m, int path, const float *x, void *y, cudaStream_t st) {
    const cprune_task_desc &d = m->tasks[0];
    if (path == INPUT_DIRECT) return launch_conv_stem(d.plan, x, d.w, d.b, y, st);
    const cprune_status s = regroup_stem_input(d.plan, x, 1, stem_scratch(d.plan, m->workspace), st);
    return s != CPRUNE_OK ? s : task_run_internal(d.plan, tensor_ptr(m, 0), d.w, d.b, nullptr, y, m->workspace, st, true);
}

static cprune_status run_pair(const cprune_model *m, size_t t, cudaStream_t st) {
    const cprune_task_desc &d = m->tasks[t], &e = m->tasks[t + 1];
    return launch_depthwise_project(d.plan, e.plan, m->pairs[t].t, m->pairs[t].tm, d.w, d.b, e.b, e.res >= 0 ? tensor_ptr(m, e.res) : nullptr,
                                    tensor_ptr(m, e.out), st);
}

static cprune_status enqueue_chain(cprune_model *m, const float *x, float *logits, cudaStream_t st) {
    const int path = input_path(m, ((uintptr_t)x & 15) == 0);
    cprune_status s = CPRUNE_OK;
    if (path == INPUT_CAST) s = cprune_cast_input(x, (size_t)m->N * m->H * m->W, m->C, tensor_ptr(m, 0), st);
    if (s != CPRUNE_OK) return s;
    for (size_t t = 0; t < m->tasks.size(); ++t) {
        const cprune_task_desc &d = m->tasks[t];
        const ModelTensor &in = m->tensors[d.in];
        void *pin = tensor_ptr(m, d.in);
        const bool last = t + 1 == m->tasks.size();
        void *pout = last ? (void *)logits : tensor_ptr(m, d.out);
        switch (d.op) {
            case CPRUNE_OP_CONV:
                if (m->pairs[t].t.ok) {
                    s = run_pair(m, t, st);
                    ++t;
                } else if (t == 0 && path != INPUT_CAST) s = run_first_task(m, path, x, pout, st);
                else s = task_run_internal(d.plan, pin, d.w, d.b, d.res >= 0 ? tensor_ptr(m, d.res) : nullptr, pout, m->workspace, st, false);
                break;
            case CPRUNE_OP_BLOCK:
                s = cprune_block_run(d.block, pin, d.w, d.b, pout, m->workspace, st);
                break;
            case CPRUNE_OP_MAXPOOL:
                s = cprune_maxpool(pin, in.n, in.h, in.w, in.c, d.p0, d.p1, d.p2, pout, st);
                break;
            case CPRUNE_OP_GAP:
                s = cprune_global_avgpool(pin, in.n, in.h, in.w, in.c, pout, st);
                break;
            case CPRUNE_OP_FC:
                s = cprune_fc(pin, in.n, d.p0, d.w, d.b, d.p1, d.p2, last ? 1 : 0, pout, st);
                break;
            default:
                s = CPRUNE_ERR_INTERNAL;
        }
        if (s != CPRUNE_OK) return s;
    }
    return CPRUNE_OK;
}

}  // namespace cprune

using namespace cprune;

extern "C" {

cprune_status cprune_model_create(int N, int H, int W, int C, const cprune_task_desc *tasks, int n_tasks,
                                  cprune_model **out) {
    if (!out) return CPRUNE_ERR_INVALID_ARG;
    *out = nullptr;
    if (N <= 0 || H <= 0 || W <= 0 || C <= 0 || !tasks || n_tasks <= 0) return CPRUNE_ERR_INVALID_ARG;
    if (tasks[n_tasks - 1].op != CPRUNE_OP_FC) return CPRUNE_ERR_INVALID_ARG;
    cprune_model *m = new cprune_model();
    m->N = N; m->H = H; m->W = W; m->C = C;
    m->tasks.assign(tasks, tasks + n_tasks);
    ModelTensor t0;
    t0.n = N; t0.h = H; t0.w = W; t0.c = C; t0.c_pad = cprune_padded_channels(C); t0.defined = true;
    m->tensors[0] = t0;
    m->launches = 1;
    cprune_status st = CPRUNE_OK;
    for (int t = 0; t < n_tasks && st == CPRUNE_OK; ++t) {
        const cprune_task_desc &d = m->tasks[t];
        auto it = m->tensors.find(d.in);
        if (it == m->tensors.end() || d.out <= 0) { st = CPRUNE_ERR_INVALID_ARG; break; }
        const ModelTensor in = it->second;
        ModelTensor o;
        o.n = in.n; o.defined = true;
        switch (d.op) {
            case CPRUNE_OP_CONV: {
                if (!d.plan || !d.w || !d.b) { st = CPRUNE_ERR_INVALID_ARG; break; }
                const cprune_plan_info &i = d.plan->info;
                if (i.N != in.n || i.H != in.h || i.W != in.w || i.C != in.c) { st = CPRUNE_ERR_INVALID_ARG; break; }
                if ((d.plan->opts.residual != 0) != (d.res >= 0)) { st = CPRUNE_ERR_INVALID_ARG; break; }
                if (d.res >= 0) {
                    auto r = m->tensors.find(d.res);
                    if (r == m->tensors.end() || r->second.h != i.P || r->second.w != i.Q || r->second.c != i.K) {
                        st = CPRUNE_ERR_INVALID_ARG;
                        break;
                    }
                }
                o.h = i.out_h; o.w = i.out_w; o.c = i.K;
                if (i.workspace_bytes > m->workspace_bytes) m->workspace_bytes = i.workspace_bytes;
                m->launches += conv_launches(d.plan);
                break;
            }
            case CPRUNE_OP_BLOCK: {
                if (!d.block || !d.w || !d.b) { st = CPRUNE_ERR_INVALID_ARG; break; }
                cprune_block_info bi;
                if (cprune_block_query(d.block, &bi) != CPRUNE_OK || bi.N != in.n || bi.H != in.h || bi.W != in.w || bi.C_in != in.c) {
                    st = CPRUNE_ERR_INVALID_ARG;
                    break;
                }
                o.h = bi.H; o.w = bi.W; o.c = bi.C_out;
                if (bi.workspace_bytes > m->workspace_bytes) m->workspace_bytes = bi.workspace_bytes;
                m->launches += bi.splits > 1 ? 2 : 1;
                break;
            }
            case CPRUNE_OP_MAXPOOL:
                if (d.p0 <= 0 || d.p1 <= 0 || d.p2 < 0 || in.h + 2 * d.p2 < d.p0 || in.w + 2 * d.p2 < d.p0) {
                    st = CPRUNE_ERR_INVALID_ARG;
                    break;
                }
                o.h = (in.h + 2 * d.p2 - d.p0) / d.p1 + 1; o.w = (in.w + 2 * d.p2 - d.p0) / d.p1 + 1; o.c = in.c;
                m->launches += 1;
                break;
            case CPRUNE_OP_GAP:
                o.h = 1; o.w = 1; o.c = in.c;
                m->launches += 1;
                break;
            case CPRUNE_OP_FC:
                if (!d.w || !d.b || in.h * in.w != 1 || in.c != d.p0 || d.p1 <= 0) { st = CPRUNE_ERR_INVALID_ARG; break; }
                o.h = 1; o.w = 1; o.c = d.p1;
                m->launches += 1;
                if (t == n_tasks - 1) m->classes = d.p1;
                break;
            default:
                st = CPRUNE_ERR_INVALID_ARG;
        }
        if (st != CPRUNE_OK) break;
        o.c_pad = cprune_padded_channels(o.c);
        if (m->tensors.count(d.out)) { st = CPRUNE_ERR_INVALID_ARG; break; }   // single assignment
        m->tensors[d.out] = o;
    }
    if (st != CPRUNE_OK) { delete m; return st; }
    const int path = input_path(m);
    if (path != INPUT_CAST) m->launches -= 1;               // no separate cast of the image
    if (path == INPUT_DIRECT) m->launches += 1 - conv_launches(m->tasks[0].plan);
    find_pairs(m);
    for (size_t t = 0; t < m->pairs.size(); ++t)
        if (m->pairs[t].t.ok) m->launches -= conv_launches(m->tasks[t + 1].plan);
    size_t off = 0;
    for (auto &kv : m->tensors) {
        kv.second.bytes = (size_t)kv.second.n * kv.second.h * kv.second.w * kv.second.c_pad * 2;
        kv.second.offset = off;
        off += align256(kv.second.bytes);
    }
    m->arena_bytes = off;
    cudaError_t e = cudaMalloc((void **)&m->arena, m->arena_bytes);
    if (e == cudaSuccess && m->workspace_bytes) e = cudaMalloc((void **)&m->workspace, m->workspace_bytes);
    if (e != cudaSuccess) {
        if (m->arena) cudaFree(m->arena);
        delete m;
        return cuda_fail(e, "cudaMalloc(model activations)");
    }
    for (size_t t = 0; t < m->pairs.size() && st == CPRUNE_OK; ++t) {
        const cprune_task_desc &d = m->tasks[t];
        if (m->pairs[t].t.ok) st = encode_depthwise_project(d.plan, m->tasks[t + 1].plan, m->pairs[t].t, tensor_ptr(m, d.in), m->tasks[t + 1].w, m->pairs[t].tm);
    }
    if (st != CPRUNE_OK) { cprune_model_destroy(m); return st; }
    *out = m;
    return CPRUNE_OK;
}

static cprune_status run_graph(cprune_model *m, int slot, const float *x, float *logits, cudaStream_t st) {
    cprune_model::GraphSlot &g = m->graphs[slot];
    if (g.exec && g.x == x && g.logits == logits && g.stream == st) {
        CPRUNE_CUDA_CHECK(cudaGraphLaunch(g.exec, st));
        return CPRUNE_OK;
    }
    if (g.exec) { cudaGraphExecDestroy(g.exec); g.exec = nullptr; }
    // first call for this (x, logits, stream): run eagerly (this also encodes tensor maps and sets
    // kernel attributes outside of any capture), then record the same sequence for later replays
    cprune_status s = enqueue(m, x, logits, st);
    if (s != CPRUNE_OK) return s;
    // the caller's stream may be the legacy default stream, which cannot be captured: record on a
    // private stream and replay the graph on the caller's
    if (!m->capture_stream) CPRUNE_CUDA_CHECK(cudaStreamCreateWithFlags(&m->capture_stream, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    CPRUNE_CUDA_CHECK(cudaStreamBeginCapture(m->capture_stream, cudaStreamCaptureModeThreadLocal));
    s = enqueue(m, x, logits, m->capture_stream);
    cudaError_t e = cudaStreamEndCapture(m->capture_stream, &graph);
    if (s != CPRUNE_OK) { if (graph) cudaGraphDestroy(graph); return s; }
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&g.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) { g.exec = nullptr; return cuda_fail(e, "cudaGraphInstantiate"); }
    g.x = x; g.logits = logits; g.stream = st;
    return CPRUNE_OK;
}

cprune_status cprune_model_run(cprune_model *m, const float *x, float *logits, int use_graph, void *stream) {
    if (!m || !x || !logits) return CPRUNE_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    std::lock_guard<std::mutex> lock(m->mu);
    m->ran = true;
    if (!use_graph) return enqueue(m, x, logits, st);
    return run_graph(m, 2, x, logits, st);
}

cprune_status cprune_model_run_host(cprune_model *m, const float *x_host, float *logits_host, void *stream) {
    if (!m || !x_host || !logits_host) return CPRUNE_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(m->mu);
    m->ran = true;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t x_bytes = (size_t)m->N * m->H * m->W * m->C * sizeof(float);
    const size_t l_bytes = (size_t)m->N * m->classes * sizeof(float);
    if (!m->copy_stream) {   // first call: set up the two device-side buffer pairs (allocates)
        CPRUNE_CUDA_CHECK(cudaStreamCreateWithFlags(&m->copy_stream, cudaStreamNonBlocking));
        for (int i = 0; i < 2; ++i) {
            CPRUNE_CUDA_CHECK(cudaMalloc((void **)&m->host_x[i], x_bytes));
            CPRUNE_CUDA_CHECK(cudaMalloc((void **)&m->host_logits[i], l_bytes));
            CPRUNE_CUDA_CHECK(cudaEventCreateWithFlags(&m->copied[i], cudaEventDisableTiming));
            CPRUNE_CUDA_CHECK(cudaEventCreateWithFlags(&m->done[i], cudaEventDisableTiming));
        }
    }
    const int slot = (int)(m->host_calls & 1);
    // the copy of this call's input may overlap the previous call's kernels; it only has to wait
    // until the call before that one has finished with the same device buffer
    if (m->host_calls >= 2) CPRUNE_CUDA_CHECK(cudaStreamWaitEvent(m->copy_stream, m->done[slot], 0));
    CPRUNE_CUDA_CHECK(cudaMemcpyAsync(m->host_x[slot], x_host, x_bytes, cudaMemcpyHostToDevice, m->copy_stream));
    CPRUNE_CUDA_CHECK(cudaEventRecord(m->copied[slot], m->copy_stream));
    CPRUNE_CUDA_CHECK(cudaStreamWaitEvent(st, m->copied[slot], 0));
    cprune_status s = run_graph(m, slot, m->host_x[slot], m->host_logits[slot], st);
    if (s != CPRUNE_OK) return s;
    CPRUNE_CUDA_CHECK(cudaMemcpyAsync(logits_host, m->host_logits[slot], l_bytes, cudaMemcpyDeviceToHost, st));
    CPRUNE_CUDA_CHECK(cudaEventRecord(m->done[slot], st));
    ++m->host_calls;
    return CPRUNE_OK;
}

cprune_status cprune_model_tensor(const cprune_model *m, int id, const void **ptr, int *n, int *h, int *w, int *c_pad) {
    if (!m) return CPRUNE_ERR_INVALID_ARG;
    auto it = m->tensors.find(id);
    if (it == m->tensors.end()) return CPRUNE_ERR_INVALID_ARG;
    if (ptr) {
        std::lock_guard<std::mutex> lock(m->mu);
        if (const int t = unstored(m, id); t >= 0) {
            // from now on the passes store it; what the last one left out is made up for
            cprune_model *own = const_cast<cprune_model *>(m);
            if (own->ran) {
                if (!own->capture_stream) CPRUNE_CUDA_CHECK(cudaStreamCreateWithFlags(&own->capture_stream, cudaStreamNonBlocking));
                CPRUNE_CUDA_CHECK(cudaDeviceSynchronize());
                const cprune_status s = store_tensor(m, t, own->capture_stream);
                if (s != CPRUNE_OK) return s;
                CPRUNE_CUDA_CHECK(cudaStreamSynchronize(own->capture_stream));
            }
            own->pairs[t].t.ok = 0;
            own->launches += conv_launches(m->tasks[t + 1].plan);
            for (auto &g : own->graphs)
                if (g.exec) { cudaGraphExecDestroy(g.exec); g.exec = nullptr; }
        }
        *ptr = m->arena + it->second.offset;
    }
    if (n) *n = it->second.n;
    if (h) *h = it->second.h;
    if (w) *w = it->second.w;
    if (c_pad) *c_pad = it->second.c_pad;
    return CPRUNE_OK;
}

cprune_status cprune_model_copy_tensor(const cprune_model *m, int id, void *dst, void *stream) {
    if (!m || !dst) return CPRUNE_ERR_INVALID_ARG;
    auto it = m->tensors.find(id);
    if (it == m->tensors.end()) return CPRUNE_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(m->mu);
    if (const int t = unstored(m, id); t >= 0) {
        const cprune_status s = store_tensor(m, t, (cudaStream_t)stream);      // (its input is stored)
        if (s != CPRUNE_OK) return s;
    }
    CPRUNE_CUDA_CHECK(cudaMemcpyAsync(dst, m->arena + it->second.offset, it->second.bytes, cudaMemcpyDeviceToDevice,
                                      (cudaStream_t)stream));
    return CPRUNE_OK;
}

int cprune_model_launches(const cprune_model *m) {
    if (!m) return 0;
    std::lock_guard<std::mutex> lock(m->mu);
    return m->launches;
}

int cprune_model_reads_image(const cprune_model *m) { return m && input_path(m) == INPUT_DIRECT ? 1 : 0; }

cprune_status cprune_model_task_table(const cprune_model *m, cprune_task_entry *entries, int max_entries, int *n_entries) {
    if (!m || !n_entries || max_entries < 0 || (max_entries > 0 && !entries)) return CPRUNE_ERR_INVALID_ARG;
    std::vector<cprune_task_entry> table;
    for (size_t t = 0; t < m->tasks.size(); ++t) {
        const cprune_task_desc &d = m->tasks[t];
        if (d.op != CPRUNE_OP_CONV) continue;
        bool found = false;
        for (auto &e : table)
            if (e.plan == d.plan) { ++e.count; found = true; break; }
        if (!found) table.push_back(cprune_task_entry{d.plan, 1, (int)t});
    }
    *n_entries = (int)table.size();
    for (int j = 0; j < (int)table.size() && j < max_entries; ++j) entries[j] = table[j];
    return CPRUNE_OK;
}

cprune_status cprune_model_time_tasks(cprune_model *m, int reps, double *ms, void *stream) {
    if (!m || !ms || reps < 1) return CPRUNE_ERR_INVALID_ARG;
    int n = 0;
    cprune_status s = cprune_model_task_table(m, nullptr, 0, &n);
    if (s != CPRUNE_OK) return s;
    std::vector<cprune_task_entry> table(n);
    s = cprune_model_task_table(m, table.data(), n, &n);
    if (s != CPRUNE_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    std::lock_guard<std::mutex> lock(m->mu);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    CPRUNE_CUDA_CHECK(cudaEventCreate(&e0));
    CPRUNE_CUDA_CHECK(cudaEventCreate(&e1));
    // the first task as the model runs it: from a float32 image (zeros), for which the place of the bf16 copy has room up to four channels
    const ModelTensor &t0 = m->tensors[0];
    const size_t image_bytes = (size_t)m->N * m->H * m->W * m->C * sizeof(float);
    const int path = image_bytes <= t0.bytes ? input_path(m) : (int)INPUT_CAST;
    float *image = (float *)tensor_ptr(m, 0);
    if (path != INPUT_CAST && cudaMemsetAsync(image, 0, image_bytes, st) != cudaSuccess) s = cuda_fail(cudaGetLastError(), "cudaMemsetAsync");
    // mean milliseconds of `run` over reps back-to-back runs, 0 after an error
    auto time = [&](auto run) -> double {
        for (int r = 0; r <= reps && s == CPRUNE_OK; ++r) {
            if (r == 1 && cudaEventRecord(e0, st) != cudaSuccess) s = CPRUNE_ERR_CUDA;   // run 0 is the untimed one
            if (s == CPRUNE_OK) s = run();
        }
        float t = 0.f;
        if (s == CPRUNE_OK && (cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
                               cudaEventElapsedTime(&t, e0, e1) != cudaSuccess)) s = cuda_fail(cudaGetLastError(), "task timing");
        return s == CPRUNE_OK ? (double)t / reps : 0.0;
    };
    auto time_task = [&](int t) {
        const cprune_task_desc &d = m->tasks[t];
        void *pin = tensor_ptr(m, d.in), *pout = tensor_ptr(m, d.out);
        const void *res = d.res >= 0 ? tensor_ptr(m, d.res) : nullptr;
        return time([&] { return t == 0 && path != INPUT_CAST ? run_first_task(m, path, image, pout, st) : task_run_internal(d.plan, pin, d.w, d.b, res, pout, m->workspace, st, false); });
    };
    // a pair's kernel, shared out in proportion to the two tasks' own times (the depthwise task first: it stores what the other one reads)
    std::map<std::pair<const cprune_plan *, const cprune_plan *>, std::pair<double, double>> pair_times;
    auto time_pair = [&](int t) {
        auto &p = pair_times[{m->tasks[t].plan, m->tasks[t + 1].plan}];
        if (p.first == 0.0 && s == CPRUNE_OK) {
            const double a = time_task(t), b = time_task(t + 1), both = time([&] { return run_pair(m, t, st); });
            if (s == CPRUNE_OK) p = {both * (a / (a + b)), both * (b / (a + b))};
        }
        return p;
    };
    for (int j = 0; j < n && s == CPRUNE_OK; ++j) {
        double sum = 0.0, alone = -1.0;
        for (int t = 0; t < (int)m->tasks.size() && s == CPRUNE_OK; ++t) {
            if (m->tasks[t].op != CPRUNE_OP_CONV || m->tasks[t].plan != table[j].plan) continue;
            if (m->pairs[t].t.ok) sum += time_pair(t).first;
            else if (t > 0 && m->pairs[t - 1].t.ok) sum += time_pair(t - 1).second;
            else {
                if (alone < 0.0) alone = time_task(t);
                sum += alone;
            }
        }
        ms[j] = sum / table[j].count;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return s;
}

cprune_status cprune_model_destroy(cprune_model *m) {
    if (!m) return CPRUNE_ERR_INVALID_ARG;
    for (auto &g : m->graphs)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    if (m->capture_stream) cudaStreamDestroy(m->capture_stream);
    if (m->copy_stream) cudaStreamDestroy(m->copy_stream);
    for (int i = 0; i < 2; ++i) {
        if (m->host_x[i]) cudaFree(m->host_x[i]);
        if (m->host_logits[i]) cudaFree(m->host_logits[i]);
        if (m->copied[i]) cudaEventDestroy(m->copied[i]);
        if (m->done[i]) cudaEventDestroy(m->done[i]);
    }
    if (m->arena) cudaFree(m->arena);
    if (m->workspace) cudaFree(m->workspace);
    delete m;
    return CPRUNE_OK;
}

}  // extern "C"
