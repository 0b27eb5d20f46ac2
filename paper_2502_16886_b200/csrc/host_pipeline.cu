// The pass of Algorithm 1 for a run of layers whose caches live in HOST memory, pipelined over three streams.  With the cache
// on the host the copies dominate (two 16 MB arrays in and nearly two out per layer of 8K positions, 1.2 ms of PCIe against
// 0.1 ms of kernels), and PCIe carries both directions at once (55 GB/s alone, 50 each way together), so the pipeline aims at
// one direction's time: a layer's K travels first and is scored, and its kept rows leave, while its V arrives.  Nothing
// waits on the host but the row count: a kernel writes it into pinned memory behind the copy of K.  (The status word read into
// pageable memory held the next layer's copies back: four layers of 8K positions 4.7 ms.  Rows written to host memory by the
// copy kernel itself: 43 GB/s beside a copy in the other direction.)
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "refree_internal.cuh"

namespace refree {
namespace {

struct Slot {
    char *q, *k, *v, *ko, *vo;
    int32_t *lengths, *status;
    int64_t *offsets;
};

// What a layer in flight tells the host.
struct HostMeta { long long rows; int32_t status; };

__global__ void host_meta_kernel(const int64_t *rows, const int32_t *status, volatile HostMeta *out)
{
    out->rows = *rows;
    out->status = *status;
}

// The context that the calling thread's work goes to.  The handle alone does not tell: after cudaDeviceReset the same handle
// stands for another context, in which the old streams and events are gone; the number is never used again.
struct Context {
    CUcontext handle = nullptr;
    unsigned long long id = 0;                       // 0: not known
};
Context current_context()
{
    typedef CUresult (*GetCurrent)(CUcontext *);
    typedef CUresult (*GetId)(CUcontext, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        auto look_up = [](const char *name) {
            void *fn = nullptr;
            cudaDriverEntryPointQueryResult res;
            return cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &res) == cudaSuccess && res == cudaDriverEntryPointSuccess ? fn : nullptr;
        };
        get_current = reinterpret_cast<GetCurrent>(look_up("cuCtxGetCurrent"));
        get_id = reinterpret_cast<GetId>(look_up("cuCtxGetId"));
    });
    Context c;
    if (!get_current || !get_id) return c;
    auto known = [&] { return get_current(&c.handle) == CUDA_SUCCESS && c.handle && get_id(c.handle, &c.id) == CUDA_SUCCESS; };
    // a thread that has not called the runtime yet (or not since a reset) has no context until the device is set
    int dev = 0;
    if (known() || (cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess && known())) return c;
    return {};
}

// Streams, events and the pinned words of one call.  Making them takes half a millisecond, so they are kept for the next call
// in the same context: a call takes a set for itself and gives it back idle; a handful are kept, whatever the number of threads.
struct HostPipe {
    Context ctx;
    cudaStream_t in = nullptr, comp = nullptr, out = nullptr;
    struct { cudaEvent_t k_in, v_in, k_done, v_done, out_done; } ev[2] = {};
    HostMeta *meta = nullptr;                        // two, pinned

    bool make()
    {
        for (cudaStream_t *st : {&in, &comp, &out})
            if (cudaStreamCreateWithFlags(st, cudaStreamNonBlocking) != cudaSuccess) return false;
        for (auto &e : ev)
            for (cudaEvent_t *x : {&e.k_in, &e.v_in, &e.k_done, &e.v_done, &e.out_done})
                if (cudaEventCreateWithFlags(x, cudaEventDisableTiming) != cudaSuccess) return false;
        return cudaHostAlloc(reinterpret_cast<void **>(&meta), 2 * sizeof(HostMeta), cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess;
    }
    void destroy()
    {
        for (auto &e : ev)
            for (cudaEvent_t x : {e.k_in, e.v_in, e.k_done, e.v_done, e.out_done})
                if (x) cudaEventDestroy(x);
        for (cudaStream_t st : {in, comp, out})
            if (st) cudaStreamDestroy(st);
        if (meta) cudaFreeHost(meta);
    }
};
constexpr int kKeptPipes = 4;
std::mutex g_pipes_mutex;
HostPipe g_pipes[kKeptPipes];                        // idle sets, of any context
int g_num_pipes = 0;

bool take_pipe(HostPipe &hp)
{
    const Context ctx = current_context();
    if (ctx.id) {
        std::lock_guard<std::mutex> hold(g_pipes_mutex);
        for (int i = 0; i < g_num_pipes;) {
            const Context &c = g_pipes[i].ctx;
            const bool same = c.id == ctx.id;
            if (same) hp = g_pipes[i];
            // a set of a context that is gone (its handle stands for another now) is forgotten: its streams went with it
            if (same || c.handle == ctx.handle) g_pipes[i] = g_pipes[--g_num_pipes]; else ++i;
            if (same) return true;
        }
    }
    hp.ctx = ctx;
    if (hp.make()) return true;
    hp.destroy();
    return false;
}

void give_pipe(HostPipe &hp, bool sound)
{
    if (sound && hp.ctx.id) {
        std::lock_guard<std::mutex> hold(g_pipes_mutex);
        if (g_num_pipes < kKeptPipes) {
            g_pipes[g_num_pipes++] = hp;
            return;
        }
    }
    hp.destroy();
}

inline size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct PipeSizes {
    size_t q, kv, out, lengths, offsets, status, seq, ws;
    size_t total() const { return 2 * (q + 2 * kv + 2 * out + lengths + offsets + status) + 2 * seq + ws; }
};

refree_status pipe_sizes(const refree_params *p, int64_t total_tokens, int64_t kv_elems, int64_t capacity_rows,
                         PipeSizes &z)
{
    if (!p || kv_elems < 0 || capacity_rows < 0 || total_tokens < 0) return REFREE_ERR_INVALID_ARG;
    size_t ws = 0;
    const refree_status st = refree_workspace_size(p, total_tokens, &ws);
    if (st != REFREE_OK) return st;
    const size_t esz = p->dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const size_t U = (size_t)p->num_seqs * p->num_kv_heads;
    z.q = up256((size_t)p->num_seqs * p->num_q_heads * p->window * p->head_dim * esz);
    z.kv = up256((size_t)kv_elems * esz);
    z.out = up256((size_t)capacity_rows * p->head_dim * esz);
    z.lengths = up256(U * sizeof(int32_t));
    z.offsets = up256((U + 1) * sizeof(int64_t));
    z.status = up256(sizeof(int32_t));
    z.seq = up256((size_t)p->num_seqs * sizeof(int32_t));
    z.ws = up256(ws);
    return REFREE_OK;
}

}  // namespace
}  // namespace refree

using namespace refree;

extern "C" {

refree_status refree_host_pipeline_arena_size(const refree_params *p, int64_t total_tokens, int64_t kv_elems,
                                              int64_t capacity_rows, size_t *bytes)
{
    if (!bytes) return REFREE_ERR_INVALID_ARG;
    PipeSizes z;
    const refree_status st = pipe_sizes(p, total_tokens, kv_elems, capacity_rows, z);
    if (st != REFREE_OK) return st;
    *bytes = z.total();
    return REFREE_OK;
}

refree_status refree_compress_layers_host(const refree_params *p, int32_t num_layers,
                                          const void *const *q_win, const void *const *k, const void *const *v,
                                          int64_t kv_elems, const int32_t *seq_start, const int32_t *seq_len,
                                          int64_t total_tokens, void *const *k_out, void *const *v_out,
                                          int64_t capacity_rows, int32_t *const *lengths, int64_t *const *offsets,
                                          void *arena, size_t arena_bytes)
{
    PipeSizes z;
    refree_status st = pipe_sizes(p, total_tokens, kv_elems, capacity_rows, z);
    if (st != REFREE_OK) return st;
    if (num_layers < 0 || !q_win || !k || !v || !seq_start || !seq_len || !k_out || !v_out || !lengths || !offsets)
        return REFREE_ERR_INVALID_ARG;
    for (int l = 0; l < num_layers; ++l)
        if (!q_win[l] || !k[l] || !v[l] || !k_out[l] || !v_out[l] || !lengths[l] || !offsets[l]) return REFREE_ERR_INVALID_ARG;
    if (!arena || arena_bytes < z.total() || (reinterpret_cast<uintptr_t>(arena) & 255)) return REFREE_ERR_WORKSPACE;
    if (num_layers == 0) return REFREE_OK;

    const size_t esz = p->dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const size_t U = (size_t)p->num_seqs * p->num_kv_heads;
    const size_t q_bytes = (size_t)p->num_seqs * p->num_q_heads * p->window * p->head_dim * esz;
    const size_t kv_bytes = (size_t)kv_elems * esz;
    const size_t row_bytes = (size_t)p->head_dim * esz;

    char *a = static_cast<char *>(arena);
    auto take = [&](size_t bytes) { char *r = a; a += bytes; return r; };
    int32_t *d_start = reinterpret_cast<int32_t *>(take(z.seq));
    int32_t *d_len = reinterpret_cast<int32_t *>(take(z.seq));
    char *d_ws = take(z.ws);
    Slot slot[2];
    for (int i = 0; i < 2; ++i) {
        slot[i].q = take(z.q); slot[i].k = take(z.kv); slot[i].v = take(z.kv);
        slot[i].ko = take(z.out); slot[i].vo = take(z.out);
        slot[i].lengths = reinterpret_cast<int32_t *>(take(z.lengths));
        slot[i].offsets = reinterpret_cast<int64_t *>(take(z.offsets));
        slot[i].status = reinterpret_cast<int32_t *>(take(z.status));
    }
    st = check_kv_layout(p, slot[0].k, slot[0].v, true);
    if (st != REFREE_OK) return st;
    const Workspace lay = workspace_layout(*p, total_tokens);
    const bool ranges = p->rank_mode == REFREE_RANK_POSITION || p->force_full;
    HostPipe hp;
    if (!take_pipe(hp)) return REFREE_ERR_CUDA;

    refree_status result = REFREE_OK;
    bool sound = true;                               // no CUDA call has failed
    auto cu = [&](cudaError_t e) {
        if (e == cudaSuccess) return true;
        sound = false;
        if (result == REFREE_OK) result = REFREE_ERR_CUDA;
        return false;
    };

    // layer l: its copies in, its kernels
    auto begin = [&](int l) {
        const Slot &sl = slot[l & 1];
        auto &ev = hp.ev[l & 1];
        // inputs of the slot are free once layer l - 2 has been compressed
        if (l >= 2) cu(cudaStreamWaitEvent(hp.in, ev.v_done, 0));
        cu(cudaMemcpyAsync(sl.q, q_win[l], q_bytes, cudaMemcpyHostToDevice, hp.in));
        cu(cudaMemcpyAsync(sl.k, k[l], kv_bytes, cudaMemcpyHostToDevice, hp.in));
        cu(cudaEventRecord(ev.k_in, hp.in));
        cu(cudaMemcpyAsync(sl.v, v[l], kv_bytes, cudaMemcpyHostToDevice, hp.in));
        cu(cudaEventRecord(ev.v_in, hp.in));
        // outputs of the slot are free once the rows of layer l - 2 have left
        cu(cudaStreamWaitEvent(hp.comp, ev.k_in, 0));
        if (l >= 2) cu(cudaStreamWaitEvent(hp.comp, ev.out_done, 0));
        cu(cudaMemsetAsync(sl.status, 0, sizeof(int32_t), hp.comp));
        if (result != REFREE_OK) return;
        CompactJob job = {};
        if (!cu(enqueue_selection(*p, sl.q, sl.k, sl.v, d_start, d_len, total_tokens, sl.ko, nullptr, capacity_rows, sl.lengths,
                                  sl.offsets, nullptr, nullptr, d_ws, lay, sl.status, hp.comp, job))) return;
        if (!cu(launch_compact(*p, job, d_start, d_len, ranges, capacity_rows, sl.status, hp.comp))) return;
        host_meta_kernel<<<1, 1, 0, hp.comp>>>(sl.offsets + U, sl.status, hp.meta + (l & 1));
        count_launches(1);
        if (!cu(cudaGetLastError())) return;
        cu(cudaEventRecord(ev.k_done, hp.comp));
        cu(cudaStreamWaitEvent(hp.comp, ev.v_in, 0));
        job.k_out[0] = nullptr;
        job.v_out[0] = sl.vo;
        job.offsets_out[0] = nullptr;                // (on their way to the host since k_done: read, not formed again)
        if (!cu(launch_compact(*p, job, d_start, d_len, ranges, capacity_rows, sl.status, hp.comp))) return;
        cu(cudaEventRecord(ev.v_done, hp.comp));
    };
    // kept rows of layer j come back once their number is known on the host
    auto finish = [&](int j) {
        const Slot &sl = slot[j & 1];
        auto &ev = hp.ev[j & 1];
        if (!cu(cudaEventSynchronize(ev.k_done))) return;
        const HostMeta m = hp.meta[j & 1];
        cu(cudaStreamWaitEvent(hp.out, ev.k_done, 0));
        cu(cudaMemcpyAsync(lengths[j], sl.lengths, U * sizeof(int32_t), cudaMemcpyDeviceToHost, hp.out));
        cu(cudaMemcpyAsync(offsets[j], sl.offsets, (U + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, hp.out));
        if (m.status & REFREE_DEV_TIMEOUT) { result = REFREE_ERR_TIMEOUT; return; }
        if (m.status & REFREE_DEV_CAPACITY) { result = REFREE_ERR_CAPACITY; return; }
        if (m.status & REFREE_DEV_NONFINITE) { result = REFREE_ERR_NONFINITE; return; }
        cu(cudaMemcpyAsync(k_out[j], sl.ko, (size_t)m.rows * row_bytes, cudaMemcpyDeviceToHost, hp.out));
        cu(cudaStreamWaitEvent(hp.out, ev.v_done, 0));
        cu(cudaMemcpyAsync(v_out[j], sl.vo, (size_t)m.rows * row_bytes, cudaMemcpyDeviceToHost, hp.out));
        cu(cudaEventRecord(ev.out_done, hp.out));
    };

    cu(cudaMemcpyAsync(d_start, seq_start, p->num_seqs * sizeof(int32_t), cudaMemcpyHostToDevice, hp.in));
    cu(cudaMemcpyAsync(d_len, seq_len, p->num_seqs * sizeof(int32_t), cudaMemcpyHostToDevice, hp.in));
    for (int l = 0; l <= num_layers && result == REFREE_OK; ++l) {
        if (l < num_layers) begin(l);
        if (l >= 1 && result == REFREE_OK) finish(l - 1);
    }

    // leave nothing in flight, whatever happened
    cu(cudaStreamSynchronize(hp.in));
    cu(cudaStreamSynchronize(hp.comp));
    cu(cudaStreamSynchronize(hp.out));
    give_pipe(hp, sound);
    return result;
}

}  // extern "C"
