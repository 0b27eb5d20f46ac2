// Stand-ins for the launchers that the host pipeline calls: each logs what its kernels read and write (fake_runtime.cpp).
#include <cstdio>

#include "refree_internal.cuh"

void say(const char *fmt, ...);
long num(const void *h);
const char *dead(const void *h);

extern "C" refree_status refree_workspace_size(const refree_params *, int64_t, size_t *bytes) { *bytes = 4096; return REFREE_OK; }

namespace refree {
void count_launches(int) {}
Workspace workspace_layout(const refree_params &, int64_t) { Workspace w = {}; w.total = 4096; return w; }
refree_status check_kv_layout(const refree_params *, const void *, const void *, bool) { return REFREE_OK; }

cudaError_t enqueue_selection(const refree_params &p, const void *q_win, const void *k, const void *v, const int32_t *seq_start,
                              const int32_t *seq_len, int64_t, void *k_out, void *v_out, int64_t, int32_t *lengths, int64_t *offsets,
                              int32_t *, float *, char *ws, const Workspace &, int32_t *status, Stream cs, CompactJob &job)
{
    const bool ranges = p.rank_mode == REFREE_RANK_POSITION || p.force_full;
    const size_t U = (size_t)p.num_seqs * p.num_kv_heads;
    say("op %ld select r %ld 1 r %ld 1 r %ld 4 r %ld 4 w %ld %zu w %ld 1 w %ld 4%s", num(cs), num(q_win), num(k), num(seq_start), num(seq_len),
        num(lengths), 4 * U, num(ws), num(status), dead(cs));
    if (!ranges) say("op %ld offsets w %ld %zu w %ld 1", num(cs), num(offsets), 8 * (U + 1), num(ws + 1024));
    job = compact_job(k, v, lengths, offsets, ranges ? nullptr : reinterpret_cast<int32_t *>(ws + 1024), ranges ? offsets : nullptr, k_out, v_out);
    return cudaSuccess;
}

cudaError_t launch_compact(const refree_params &p, const CompactJob &job, const int32_t *seq_start, const int32_t *seq_len, bool, int64_t,
                           int32_t *status, Stream st)
{
    const size_t U = (size_t)p.num_seqs * p.num_kv_heads;
    char moved[160] = "";
    int at = 0;
    if (job.k_out[0]) at += snprintf(moved + at, sizeof moved - at, " r %ld 1 w %ld 1", num(job.k[0]), num(job.k_out[0]));
    if (job.v_out[0]) at += snprintf(moved + at, sizeof moved - at, " r %ld 1 w %ld 1", num(job.v[0]), num(job.v_out[0]));
    if (job.kept[0]) at += snprintf(moved + at, sizeof moved - at, " r %ld 1", num(job.kept[0]));
    say("op %ld rows r %ld %zu r %ld 4 r %ld 4 %c %ld %zu w %ld 4%s%s", num(st), num(job.lengths[0]), 4 * U, num(seq_start), num(seq_len),
        job.offsets_out[0] ? 'w' : 'r', num(job.offsets_out[0] ? job.offsets_out[0] : job.offsets[0]), 8 * (U + 1), num(status), moved, dead(st));
    return cudaSuccess;
}
}  // namespace refree
