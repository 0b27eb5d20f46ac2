// C-ABI entry points: argument checks, workspace layout, launch sequences.
#include <string.h>

#include <algorithm>
#include <cmath>
#include <atomic>
#include <mutex>

#include "refree_internal.cuh"

namespace refree {

static std::atomic<long long> g_launches{0};
void count_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

int sm_count()
{
    static std::mutex m;
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    std::lock_guard<std::mutex> lock(m);
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
        cached[dev] = n;
    }
    return cached[dev];
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Window rows scored at once: the whole window when a scoring path takes it, else a chunk that one does
// (512 query rows on the tensor-core path, 1024 on the generic one).
static int chunk_window(const refree_params &p)
{
    const int G = p.num_q_heads / p.num_kv_heads;
    if ((int64_t)G * p.window <= kMaxRows) return p.window;
    const int cap = (p.dtype == REFREE_DTYPE_BF16 && p.head_dim == 128) ? 512 : kMaxRows;
    return std::max(1, cap / G);
}

Workspace workspace_layout(const refree_params &p, int64_t total_tokens)
{
    Workspace w;
    const int64_t U = (int64_t)p.num_seqs * p.num_kv_heads;
    const int64_t G = p.num_q_heads / p.num_kv_heads;
    const int wc = chunk_window(p);
    const int64_t rows = G * wc;
    const int64_t tiles = total_tokens / kTile + p.num_seqs;
    size_t off = 0;
    // partials: per (64 positions, head, row) for the generic path, per (range + unit, column half, padded row) for the tensor-core path
    const int64_t rows_pad = (rows + kTile - 1) / kTile * kTile;
    const int64_t part_items = std::max<int64_t>((total_tokens / 64 + p.num_seqs) * p.num_kv_heads * rows, 2 * (256 + U) * rows_pad);
    size_t part_bytes = (size_t)part_items * sizeof(float2);
    if (score_w1_supported(p)) part_bytes = std::max(part_bytes, score_w1_scratch_bytes(p, total_tokens));
    w.part_off = off;   w.part_bytes = align256(part_bytes);                                               off += w.part_bytes;
    w.lse_off = off;    w.lse_bytes = align256((size_t)(U * rows_pad) * sizeof(float));                    off += w.lse_bytes;
    w.grp_off = off;    w.grp_bytes = align256((size_t)(tiles * p.num_kv_heads * 4) * sizeof(GroupPartial));  off += w.grp_bytes;
    w.cut_off = off;    w.cut_bytes = align256((size_t)U * sizeof(Cut));                                   off += w.cut_bytes;
    w.scores_off = off; w.scores_bytes = align256((size_t)(p.num_kv_heads * total_tokens) * sizeof(float)); off += w.scores_bytes;
    w.kept_off = off;   w.kept_bytes = align256((size_t)(p.num_kv_heads * total_tokens) * sizeof(int32_t)); off += w.kept_bytes;
    w.chk_off = off;    w.chk_bytes = 0;
    if (wc < p.window) {
        const size_t esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
        w.chk_bytes = align256((size_t)p.num_seqs * p.num_q_heads * wc * p.head_dim * esz) +
                      align256((size_t)(p.num_kv_heads * total_tokens) * sizeof(float)) +
                      align256((size_t)p.num_seqs * sizeof(int32_t));
    }
    off += w.chk_bytes;
    w.total = off;
    return w;
}

static refree_status check_params(const refree_params *p, int64_t total_tokens)
{
    if (!p) return REFREE_ERR_INVALID_ARG;
    if (p->num_seqs < 1 || p->num_q_heads < 1 || p->num_kv_heads < 1) return REFREE_ERR_INVALID_ARG;
    if (p->num_q_heads % p->num_kv_heads != 0) return REFREE_ERR_INVALID_ARG;
    if (p->window < 1 || p->sink < 0) return REFREE_ERR_INVALID_ARG;
    if (!(p->threshold >= 0.0f && p->threshold < 1.0f)) return REFREE_ERR_INVALID_ARG;
    if (p->rank_mode != REFREE_RANK_POSITION && p->rank_mode != REFREE_RANK_SCORE) return REFREE_ERR_INVALID_ARG;
    if (p->scope != REFREE_SCOPE_HEAD && p->scope != REFREE_SCOPE_LAYER) return REFREE_ERR_INVALID_ARG;
    if (p->dtype != REFREE_DTYPE_F32 && p->dtype != REFREE_DTYPE_BF16) return REFREE_ERR_INVALID_ARG;
    if (total_tokens < 0 || total_tokens > 0x7fffffffLL - kTile) return REFREE_ERR_INVALID_ARG;
    if (p->head_dim != 64 && p->head_dim != 128) return REFREE_ERR_UNSUPPORTED;
    if (p->num_seqs > kMaxSeqs) return REFREE_ERR_UNSUPPORTED;
    if ((int64_t)p->num_seqs * p->num_kv_heads > 65535) return REFREE_ERR_UNSUPPORTED;
    if ((int64_t)(p->num_q_heads / p->num_kv_heads) * p->window > kMaxRows &&
        ((int64_t)(p->num_q_heads / p->num_kv_heads) * p->window > kMaxRowsChunked ||
         p->num_q_heads / p->num_kv_heads > kMaxGroupChunked))
        return REFREE_ERR_UNSUPPORTED;
    return REFREE_OK;
}

refree_status check_kv_layout(const refree_params *p, const void *k, const void *v, bool need_v)
{
    const int esz = p->dtype == REFREE_DTYPE_F32 ? 4 : 2;
    if (p->kv_tokens < 0) return REFREE_ERR_INVALID_ARG;
    if (p->k_stride_tok < p->head_dim || p->k_stride_seq < 0 || p->k_stride_head < 0) return REFREE_ERR_INVALID_ARG;
    // 16-byte vector access to every row
    if ((reinterpret_cast<uintptr_t>(k) & 15) || (p->k_stride_tok * esz) % 16 || (p->k_stride_head * esz) % 16 ||
        (p->k_stride_seq * esz) % 16)
        return REFREE_ERR_UNSUPPORTED;
    if (need_v) {
        if (p->v_stride_tok < p->head_dim || p->v_stride_seq < 0 || p->v_stride_head < 0) return REFREE_ERR_INVALID_ARG;
        if ((reinterpret_cast<uintptr_t>(v) & 15) || (p->v_stride_tok * esz) % 16 || (p->v_stride_head * esz) % 16 ||
            (p->v_stride_seq * esz) % 16)
            return REFREE_ERR_UNSUPPORTED;
    }
    return REFREE_OK;
}

static refree_status from_cuda(cudaError_t e) { return e == cudaSuccess ? REFREE_OK : REFREE_ERR_CUDA; }

static bool use_tc(const refree_params &p, const void *q_win)
{
    return score_tc_supported(p) && !(reinterpret_cast<uintptr_t>(q_win) & 15);
}

namespace {
// Lengths of the sequences as a chunk of window rows sees them: cut after the chunk's last row.
__global__ void chunk_lens_kernel(const int32_t *seq_len, int32_t *len_c, int num_seqs, int rows_after)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < num_seqs) len_c[s] = max(0, max(seq_len[s], 0) - rows_after);
}

// scores += chunk scores * (chunk rows that see the position), i.e. the chunk's column sums over G; the last
// chunk divides by the rows of the whole window that see the position (Eq. 2).
__global__ void chunk_accumulate_kernel(refree_params p, const int32_t *seq_len, const int32_t *len_c, const float *sc,
                                        float *scores, int64_t total_tokens, int wc, int last)
{
    __shared__ int s_pack, s_pack_c;
    const int Hkv = p.num_kv_heads, s = blockIdx.y / Hkv, g = blockIdx.y % Hkv;
    if (threadIdx.x == 0) {
        int a = 0, b = 0;
        for (int t = 0; t < s; ++t) { a += max(seq_len[t], 0); b += len_c[t]; }
        s_pack = a;
        s_pack_c = b;
    }
    __syncthreads();
    const int n = max(seq_len[s], 0), nc = len_c[s];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float acc = scores[(int64_t)g * total_tokens + s_pack + i];
        if (i < nc) {
            const int cnt_c = max(1, min(min(wc, nc), nc - i));
            acc += sc[(int64_t)g * total_tokens + s_pack_c + i] * (float)cnt_c;
        }
        if (last) acc /= (float)max(1, min(min(p.window, n), n - i));
        scores[(int64_t)g * total_tokens + s_pack + i] = acc;
    }
}
}  // namespace

static cudaError_t run_score(const refree_params &p, const void *q_win, const void *k,
                             const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                             float *scores, char *ws, const Workspace &lay, int32_t *dev_status,
                             Stream st, GroupPartial *groups = nullptr, int32_t *sel_lengths = nullptr)
{
    const int wc = chunk_window(p);
    if (wc < p.window) {
        // Window too long for one pass: chunks of window rows from the last backwards, each scored as a window of
        // its own over the sequences cut at its last row (K is read again per chunk), then weighted back to column
        // sums and added up.  The chunks' scores are exact column sums up to one rounding each.
        const size_t esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
        const size_t row_bytes = (size_t)p.head_dim * esz;
        char *qc = ws + lay.chk_off;
        float *sc = reinterpret_cast<float *>(qc + align256((size_t)p.num_seqs * p.num_q_heads * wc * row_bytes));
        int32_t *len_c = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(sc) +
                                                    align256((size_t)(p.num_kv_heads * total_tokens) * sizeof(float)));
        cudaError_t e = cudaMemsetAsync(scores, 0, (size_t)(p.num_kv_heads * total_tokens) * sizeof(float), st);
        if (e != cudaSuccess) return e;
        const int gx = (int)std::min<int64_t>(1024, (total_tokens + 255) / 256);
        for (int t1 = p.window; t1 > 0; t1 -= wc) {
            const int t0 = std::max(0, t1 - wc), wcur = t1 - t0;
            refree_params pc = p;
            pc.window = wcur;
            e = cudaMemcpy2DAsync(qc, (size_t)wcur * row_bytes, (const char *)q_win + (size_t)t0 * row_bytes,
                                  (size_t)p.window * row_bytes, (size_t)wcur * row_bytes,
                                  (size_t)p.num_seqs * p.num_q_heads, cudaMemcpyDeviceToDevice, st);
            if (e != cudaSuccess) return e;
            chunk_lens_kernel<<<(p.num_seqs + 255) / 256, 256, 0, st>>>(seq_len, len_c, p.num_seqs, p.window - t1);
            count_launches(1);
            e = run_score(pc, qc, k, seq_start, len_c, total_tokens, sc, ws, lay, dev_status, st, nullptr);
            if (e != cudaSuccess) return e;
            chunk_accumulate_kernel<<<dim3(gx, p.num_seqs * p.num_kv_heads), 256, 0, st>>>(p, seq_len, len_c, sc, scores,
                                                                                         total_tokens, wcur, t0 == 0);
            count_launches(1);
        }
        return cudaGetLastError();
    }
    if (use_tc(p, q_win))
        return launch_score_tc(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st, groups, sel_lengths);
    if (score_w1_supported(p))
    {
        W1Group g = {};
        g.layers = 1;
        g.q_win[0] = q_win;
        g.k[0] = k;
        g.scratch = ws + lay.part_off;
        g.scores = scores;
        g.groups = groups;
        g.cuts = sel_lengths ? reinterpret_cast<Cut *>(ws + lay.cut_off) : nullptr;
        g.sel_lengths[0] = sel_lengths;
        return launch_score_w1(p, g, seq_start, seq_len, total_tokens, dev_status, st);
    }
    return launch_score_generic(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st, groups, sel_lengths);
}

// Whether the scoring of a layer leaves the budgets too (position ranking per head): it does so from per-32-position sums of
// squares instead of every score.
static bool rule_with_scores(const refree_params &p, const void *q_win, int64_t total_tokens)
{
    return p.rank_mode == REFREE_RANK_POSITION && p.scope == REFREE_SCOPE_HEAD && !p.force_full && total_tokens > 0 &&
           total_tokens <= kGroupSelectMaxTokens && chunk_window(p) == p.window &&
           (use_tc(p, q_win) || score_w1_supported(p) || score_generic_rule(p, total_tokens));
}

}  // namespace refree

using namespace refree;

extern "C" {

void refree_default_params(refree_params *p)
{
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->window = 1;
    p->sink = 4;
    p->threshold = 0.01f;
    p->rank_mode = REFREE_RANK_POSITION;
    p->scope = REFREE_SCOPE_HEAD;
    p->keep_window = 1;
    p->force_full = 0;
    p->dtype = REFREE_DTYPE_BF16;
}

int64_t refree_kernel_launch_count(void) { return (int64_t)g_launches.load(std::memory_order_relaxed); }

const char *refree_status_string(refree_status s)
{
    switch (s) {
    case REFREE_OK: return "ok";
    case REFREE_ERR_INVALID_ARG: return "invalid argument";
    case REFREE_ERR_UNSUPPORTED: return "unsupported shape, type or alignment";
    case REFREE_ERR_WORKSPACE: return "workspace missing or too small";
    case REFREE_ERR_CAPACITY: return "output capacity too small";
    case REFREE_ERR_CUDA: return "CUDA runtime error";
    case REFREE_ERR_TIMEOUT: return "a bounded on-device wait gave up";
    case REFREE_ERR_NONFINITE: return "non-finite score";
    case REFREE_ERR_STATIC_LIMIT: return "problem exceeds the built-in scratch of the no-allocation entry point";
    }
    return "unknown status";
}

refree_status refree_workspace_size(const refree_params *p, int64_t total_tokens, size_t *bytes)
{
    if (!bytes) return REFREE_ERR_INVALID_ARG;
    const refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    *bytes = workspace_layout(*p, total_tokens).total;
    return REFREE_OK;
}

refree_status refree_score(const refree_params *p, const void *q_win, const void *k,
                           const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                           float *scores, void *workspace, size_t workspace_bytes,
                           int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    if (!q_win || !k || !seq_start || !seq_len || !scores) return REFREE_ERR_INVALID_ARG;
    st = check_kv_layout(p, k, nullptr, false);
    if (st != REFREE_OK) return st;
    const Workspace lay = workspace_layout(*p, total_tokens);
    if (!workspace || workspace_bytes < lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    if (total_tokens == 0) return REFREE_OK;
    return from_cuda(run_score(*p, q_win, k, seq_start, seq_len, total_tokens, scores, (char *)workspace, lay,
                               device_status, (cudaStream_t)stream));
}

refree_status refree_select_budget(const refree_params *p, const float *scores,
                                   const int32_t *seq_len, int64_t total_tokens,
                                   int32_t *lengths, int64_t *offsets,
                                   int32_t *kept_idx, int64_t capacity_rows,
                                   void *workspace, size_t workspace_bytes,
                                   int32_t *device_status, void *stream)
{
    const refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    if (!scores || !seq_len || !lengths || !offsets || capacity_rows < 0) return REFREE_ERR_INVALID_ARG;
    const Workspace lay = workspace_layout(*p, total_tokens);
    if (!workspace || workspace_bytes < lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    return from_cuda(launch_select(*p, scores, seq_len, total_tokens, select_out(lengths, offsets, kept_idx), capacity_rows,
                                   (char *)workspace, lay, device_status, (cudaStream_t)stream));
}

refree_status refree_compact(const refree_params *p, const void *k, const void *v,
                             const int32_t *seq_start, const int32_t *seq_len,
                             const int32_t *lengths, const int64_t *offsets,
                             const int32_t *kept_idx, void *k_out, void *v_out,
                             int64_t capacity_rows, int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, 0);
    if (st != REFREE_OK) return st;
    if (!k || !v || !seq_start || !seq_len || !lengths || !offsets || !kept_idx || !k_out || !v_out ||
        capacity_rows < 0)
        return REFREE_ERR_INVALID_ARG;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    if ((reinterpret_cast<uintptr_t>(k_out) & 15) || (reinterpret_cast<uintptr_t>(v_out) & 15))
        return REFREE_ERR_UNSUPPORTED;
    return from_cuda(launch_compact(*p, compact_job(k, v, lengths, offsets, kept_idx, nullptr, k_out, v_out), seq_start, seq_len,
                                     false, capacity_rows, device_status, (cudaStream_t)stream));
}

refree_status refree_compact_paged(const refree_params *p, const void *k, const void *v,
                                   const int32_t *seq_start, const int32_t *seq_len,
                                   const int32_t *lengths, const int64_t *offsets, const int32_t *kept_idx,
                                   const int32_t *block_table, int32_t max_blocks_per_unit, int32_t block_rows,
                                   void *k_pool, void *v_pool, int64_t num_blocks,
                                   int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, 0);
    if (st != REFREE_OK) return st;
    if (!k || !v || !seq_start || !seq_len || !lengths || !block_table || !k_pool || !v_pool ||
        max_blocks_per_unit < 1 || block_rows < 1 || num_blocks < 0)
        return REFREE_ERR_INVALID_ARG;
    const bool ranges = p->rank_mode == REFREE_RANK_POSITION || p->force_full;
    if (!ranges && (!kept_idx || !offsets)) return REFREE_ERR_INVALID_ARG;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    if ((reinterpret_cast<uintptr_t>(k_pool) & 15) || (reinterpret_cast<uintptr_t>(v_pool) & 15))
        return REFREE_ERR_UNSUPPORTED;
    return from_cuda(launch_compact_paged(*p, k, v, seq_start, seq_len, lengths, offsets, ranges ? nullptr : kept_idx,
                                          ranges, block_table, max_blocks_per_unit, block_rows, k_pool, v_pool,
                                          num_blocks, device_status, (cudaStream_t)stream));
}

refree_status refree_compact_inplace(const refree_params *p, void *k, void *v,
                                     const int32_t *seq_start, const int32_t *seq_len,
                                     const int64_t *offsets, const int32_t *kept_idx, int32_t anchor,
                                     int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, 0);
    if (st != REFREE_OK) return st;
    if (!k || !v || !seq_start || !seq_len || !offsets) return REFREE_ERR_INVALID_ARG;
    if (anchor != REFREE_ANCHOR_FRONT && anchor != REFREE_ANCHOR_BACK) return REFREE_ERR_INVALID_ARG;
    const bool ranges = p->rank_mode == REFREE_RANK_POSITION || p->force_full;
    if (!ranges && !kept_idx) return REFREE_ERR_INVALID_ARG;
    if (!ranges && anchor == REFREE_ANCHOR_BACK) return REFREE_ERR_UNSUPPORTED;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    return from_cuda(launch_compact_inplace(*p, k, v, seq_start, seq_len, offsets, ranges ? nullptr : kept_idx, ranges,
                                            anchor == REFREE_ANCHOR_BACK, device_status, (cudaStream_t)stream));
}

static refree_status check_decode(const refree_params *p, int64_t max_rows)
{
    if (!p) return REFREE_ERR_INVALID_ARG;
    if (p->num_seqs < 1 || p->num_q_heads < 1 || p->num_kv_heads < 1) return REFREE_ERR_INVALID_ARG;
    if (p->num_q_heads % p->num_kv_heads != 0) return REFREE_ERR_INVALID_ARG;
    if (p->dtype != REFREE_DTYPE_F32 && p->dtype != REFREE_DTYPE_BF16) return REFREE_ERR_INVALID_ARG;
    if (max_rows < 0 || max_rows > 0x7fffffffLL - 4096) return REFREE_ERR_INVALID_ARG;
    if (p->head_dim != 64 && p->head_dim != 128) return REFREE_ERR_UNSUPPORTED;
    if ((int64_t)p->num_seqs * p->num_kv_heads > 65535) return REFREE_ERR_UNSUPPORTED;
    if (p->num_q_heads / p->num_kv_heads > 16) return REFREE_ERR_UNSUPPORTED;
    return REFREE_OK;
}

refree_status refree_decode_workspace_size(const refree_params *p, int64_t max_rows_per_unit, size_t *bytes)
{
    const refree_status st = check_decode(p, max_rows_per_unit);
    if (st != REFREE_OK) return st;
    if (!bytes) return REFREE_ERR_INVALID_ARG;
    *bytes = decode_workspace_bytes(*p, max_rows_per_unit);
    return REFREE_OK;
}

refree_status refree_decode_attention(const refree_params *p, const void *q_new,
                                      const void *k_c, const void *v_c, const int64_t *offsets,
                                      int64_t max_rows_per_unit, float *out,
                                      void *workspace, size_t workspace_bytes,
                                      int32_t *device_status, void *stream)
{
    const refree_status st = check_decode(p, max_rows_per_unit);
    if (st != REFREE_OK) return st;
    if (!q_new || !k_c || !v_c || !offsets || !out) return REFREE_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(k_c) & 15) || (reinterpret_cast<uintptr_t>(v_c) & 15)) return REFREE_ERR_UNSUPPORTED;
    if (!workspace || workspace_bytes < decode_workspace_bytes(*p, max_rows_per_unit) ||
        (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    return from_cuda(launch_decode_attention(*p, q_new, k_c, v_c, offsets, max_rows_per_unit, out, workspace,
                                             device_status, (cudaStream_t)stream));
}

refree_status refree_decode_attention_inplace(const refree_params *p, const void *q_new,
                                              const void *k, const void *v,
                                              const int32_t *seq_start, const int32_t *seq_len,
                                              const int32_t *lengths, int32_t anchor,
                                              int64_t max_rows_per_unit, float *out,
                                              void *workspace, size_t workspace_bytes,
                                              int32_t *device_status, void *stream)
{
    refree_status st = check_decode(p, max_rows_per_unit);
    if (st != REFREE_OK) return st;
    if (!q_new || !k || !v || !seq_start || !seq_len || !lengths || !out) return REFREE_ERR_INVALID_ARG;
    if (anchor != REFREE_ANCHOR_FRONT && anchor != REFREE_ANCHOR_BACK) return REFREE_ERR_INVALID_ARG;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    // the rows of a unit must be back to back, and every unit must start on a whole row
    const int64_t d = p->head_dim;
    if (p->k_stride_tok != d || p->v_stride_tok != d || p->k_stride_seq % d || p->k_stride_head % d ||
        p->v_stride_seq % d || p->v_stride_head % d)
        return REFREE_ERR_UNSUPPORTED;
    if (!workspace || workspace_bytes < decode_workspace_bytes(*p, max_rows_per_unit) ||
        (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    return from_cuda(launch_decode_attention(*p, q_new, k, v, nullptr, max_rows_per_unit, out, workspace, device_status,
                                             (cudaStream_t)stream, seq_start, seq_len, lengths,
                                             anchor == REFREE_ANCHOR_BACK));
}

}  // extern "C"

namespace refree {
// Scoring and selection of one layer, up to the launch that `job` then needs (budgets; with score ranking the index list and
// the offsets too).
cudaError_t enqueue_selection(const refree_params &p, const void *q_win, const void *k, const void *v, const int32_t *seq_start,
                              const int32_t *seq_len, int64_t total_tokens, void *k_out, void *v_out, int64_t capacity_rows,
                              int32_t *lengths, int64_t *offsets, int32_t *kept_idx, float *scores, char *ws, const Workspace &lay,
                              int32_t *device_status, Stream cs, CompactJob &job)
{
    float *sc = scores ? scores : reinterpret_cast<float *>(ws + lay.scores_off);
    const bool ranges = p.rank_mode == REFREE_RANK_POSITION || p.force_full;
    int32_t *kept = kept_idx ? kept_idx : (ranges ? nullptr : reinterpret_cast<int32_t *>(ws + lay.kept_off));
    cudaError_t e = cudaSuccess;
    // a frozen layer needs no scores unless the caller asked for them
    GroupPartial *groups = rule_with_scores(p, q_win, total_tokens) ? reinterpret_cast<GroupPartial *>(ws + lay.grp_off) : nullptr;
    if (total_tokens > 0 && (!p.force_full || scores))
        e = run_score(p, q_win, k, seq_start, seq_len, total_tokens, sc, ws, lay, device_status, cs, groups, lengths);
    if (e != cudaSuccess) return e;
    // with two-range kept sets the copy forms the offsets and the index list itself: no launch for them (fp32 d 64, a layer of
    // 8 heads x 3000 positions with its list 81.3 -> 77.6 us, d 128, 1500 positions 40.5 -> 37.0)
    job = compact_job(k, v, lengths, offsets, ranges ? nullptr : kept, ranges ? offsets : nullptr, k_out, v_out, ranges ? kept : nullptr);
    job.after_rule = ranges && !groups;
    return launch_select(p, sc, seq_len, total_tokens, select_out(lengths, offsets, kept), capacity_rows, ws, lay, device_status, cs,
                         !ranges, groups != nullptr);
}
}  // namespace refree

extern "C" {

// The launch sequence of one layer.  `cs` takes scoring and selection; compaction goes to `cc`
// (after `scored`, recorded on `cs`, when the two differ).
static refree_status enqueue_layer(const refree_params *p, const void *q_win, const void *k, const void *v,
                                   const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                                   void *k_out, void *v_out, int64_t capacity_rows, int32_t *lengths,
                                   int64_t *offsets, int32_t *kept_idx, float *scores, char *ws,
                                   const Workspace &lay, int32_t *device_status, Stream cs,
                                   Stream cc, cudaEvent_t scored)
{
    CompactJob job = {};
    if (enqueue_selection(*p, q_win, k, v, seq_start, seq_len, total_tokens, k_out, v_out, capacity_rows, lengths, offsets, kept_idx,
                          scores, ws, lay, device_status, cs, job) != cudaSuccess)
        return REFREE_ERR_CUDA;
    if (cc.s != cs.s && (cudaEventRecord(scored, cs) != cudaSuccess || cudaStreamWaitEvent(cc, scored, 0) != cudaSuccess))
        return REFREE_ERR_CUDA;
    const bool ranges = p->rank_mode == REFREE_RANK_POSITION || p->force_full;
    return from_cuda(launch_compact(*p, job, seq_start, seq_len, ranges, capacity_rows, device_status, cc));
}

refree_status refree_compress_layer(const refree_params *p, const void *q_win,
                                    const void *k, const void *v,
                                    const int32_t *seq_start, const int32_t *seq_len,
                                    int64_t total_tokens,
                                    void *k_out, void *v_out, int64_t capacity_rows,
                                    int32_t *lengths, int64_t *offsets,
                                    int32_t *kept_idx, float *scores,
                                    void *workspace, size_t workspace_bytes,
                                    int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    if (!q_win || !k || !v || !seq_start || !seq_len || !k_out || !v_out || !lengths || !offsets ||
        capacity_rows < 0)
        return REFREE_ERR_INVALID_ARG;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    if ((reinterpret_cast<uintptr_t>(k_out) & 15) || (reinterpret_cast<uintptr_t>(v_out) & 15))
        return REFREE_ERR_UNSUPPORTED;
    const Workspace lay = workspace_layout(*p, total_tokens);
    if (!workspace || workspace_bytes < lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    cudaStream_t cs = (cudaStream_t)stream;
    return enqueue_layer(p, q_win, k, v, seq_start, seq_len, total_tokens, k_out, v_out, capacity_rows, lengths,
                         offsets, kept_idx, scores, (char *)workspace, lay, device_status, cs, cs, nullptr);
}

refree_status refree_compress_layer_inplace(const refree_params *p, const void *q_win, void *k, void *v,
                                            const int32_t *seq_start, const int32_t *seq_len,
                                            int64_t total_tokens, int32_t *lengths, int64_t *offsets,
                                            int32_t anchor, void *workspace, size_t workspace_bytes,
                                            int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    if (!q_win || !k || !v || !seq_start || !seq_len || !lengths || !offsets) return REFREE_ERR_INVALID_ARG;
    if (anchor != REFREE_ANCHOR_FRONT && anchor != REFREE_ANCHOR_BACK) return REFREE_ERR_INVALID_ARG;
    const bool ranges = p->rank_mode == REFREE_RANK_POSITION || p->force_full;
    if (!ranges && anchor == REFREE_ANCHOR_BACK) return REFREE_ERR_UNSUPPORTED;
    st = check_kv_layout(p, k, v, true);
    if (st != REFREE_OK) return st;
    const Workspace lay = workspace_layout(*p, total_tokens);
    if (!workspace || workspace_bytes < lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    char *ws = (char *)workspace;
    cudaStream_t cs = (cudaStream_t)stream;
    float *sc = reinterpret_cast<float *>(ws + lay.scores_off);
    int32_t *kept = ranges ? nullptr : reinterpret_cast<int32_t *>(ws + lay.kept_off);
    GroupPartial *groups = nullptr;
    if (rule_with_scores(*p, q_win, total_tokens))
        groups = reinterpret_cast<GroupPartial *>(ws + lay.grp_off);
    cudaError_t e = cudaSuccess;
    if (total_tokens > 0 && !p->force_full)
        e = run_score(*p, q_win, k, seq_start, seq_len, total_tokens, sc, ws, lay, device_status, cs, groups, lengths);
    if (e != cudaSuccess) return REFREE_ERR_CUDA;
    // the end-anchored kernel forms the offsets itself: no emit launch
    const bool lean = anchor == REFREE_ANCHOR_BACK;
    e = launch_select(*p, sc, seq_len, total_tokens, select_out(lengths, offsets, kept), (int64_t)p->num_kv_heads * total_tokens, ws,
                      lay, device_status, cs, !lean, groups != nullptr);
    if (e != cudaSuccess) return REFREE_ERR_CUDA;
    return from_cuda(launch_compact_inplace(*p, k, v, seq_start, seq_len, offsets, kept, ranges, lean, device_status, cs,
                                            lean ? lengths : nullptr, lean ? offsets : nullptr));
}

// ---- a run of device-resident layers, compaction of layer l under the scoring of layer l + 1 ----
namespace {
struct LayerPipe {
    bool ready = false;
    cudaStream_t hi = nullptr, lo = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr, scored[2] = {nullptr, nullptr}, compacted[2] = {nullptr, nullptr};
};
std::mutex g_pipe_mutex;
LayerPipe g_pipe[64];

// Streams and events of the current device, made on first use and kept until the process exits.
LayerPipe *layer_pipe()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_pipe_mutex);
    LayerPipe &lp = g_pipe[dev];
    if (lp.ready) return &lp;
    int least = 0, greatest = 0;
    if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) return nullptr;
    bool ok = cudaStreamCreateWithPriority(&lp.hi, cudaStreamNonBlocking, greatest) == cudaSuccess &&
              cudaStreamCreateWithPriority(&lp.lo, cudaStreamNonBlocking, least) == cudaSuccess &&
              cudaEventCreateWithFlags(&lp.fork, cudaEventDisableTiming) == cudaSuccess &&
              cudaEventCreateWithFlags(&lp.join, cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; i < 2 && ok; ++i)
        ok = cudaEventCreateWithFlags(&lp.scored[i], cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&lp.compacted[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) return nullptr;
    lp.ready = true;
    return &lp;
}

// What a group of `layers` layers of a run keeps between its launches (struct TcGroup).
struct BatchLayout {
    size_t part_off, part_bytes, grp_off, tickets_off, cut_off, scores_off, kept_off, total;
};
BatchLayout batch_layout(const refree_params &p, int64_t total_tokens, int layers)
{
    BatchLayout b;
    const int64_t heads = (int64_t)p.num_kv_heads * layers, U = p.num_seqs * heads, tiles = total_tokens / kTile + p.num_seqs;
    const int64_t rows_pad = ((int64_t)(p.num_q_heads / p.num_kv_heads) * p.window + kTile - 1) / kTile * kTile;
    size_t off = 0;
    b.part_off = off;    b.part_bytes = align256((size_t)(2 * (256 * layers + U) * rows_pad) * sizeof(float2)); off += b.part_bytes;
    b.grp_off = off;     off += align256((size_t)(tiles * heads * 4) * sizeof(GroupPartial));
    b.tickets_off = off; off += align256((size_t)(2 * U) * sizeof(uint32_t));
    b.cut_off = off;     off += align256((size_t)U * sizeof(Cut));
    b.scores_off = off;  off += align256((size_t)(heads * total_tokens) * sizeof(float));
    b.kept_off = off;    if (p.rank_mode == REFREE_RANK_SCORE) off += align256((size_t)(heads * total_tokens) * sizeof(int32_t));
    b.total = off;
    return b;
}

// The same for runs with a single query row, where a group is finished before the next begins.
struct W1BatchLayout {
    size_t scratch_off, scratch_bytes, grp_off, cut_off, scores_off, kept_off, total;
};
W1BatchLayout w1_batch_layout(const refree_params &p, int64_t total_tokens, int layers)
{
    W1BatchLayout b;
    const int64_t heads = (int64_t)p.num_kv_heads * layers, tiles = total_tokens / kTile + p.num_seqs;
    size_t off = 0;
    b.scratch_off = off; b.scratch_bytes = align256(score_w1_scratch_bytes(p, total_tokens)) * layers; off += b.scratch_bytes;
    b.grp_off = off;     off += align256((size_t)(tiles * heads * 4) * sizeof(GroupPartial));
    b.cut_off = off;     off += align256((size_t)(p.num_seqs * heads) * sizeof(Cut));
    b.scores_off = off;  off += align256((size_t)(heads * total_tokens) * sizeof(float));
    b.kept_off = off;    if (p.rank_mode == REFREE_RANK_SCORE) off += align256((size_t)(heads * total_tokens) * sizeof(int32_t));
    b.total = off;
    return b;
}
constexpr size_t kW1BatchBytes = (size_t)96 << 20;
// As many layers to a launch as the workspace holds.
int w1_batch(const refree_params &p, int64_t total_tokens, int num_layers, size_t workspace_bytes)
{
    int n = std::min(kMaxBatch, num_layers);
    while (n > 1 && w1_batch_layout(p, total_tokens, n).total > workspace_bytes) --n;
    return n;
}

// Layers of a run that one launch scores together, at most kMaxBatch.  A launch costs some 20 us beyond its tiles (setup, the
// first loads, normalisers, the stopping rule, the last CTA of the chain), paid once per group.
//   `copy` (the scoring moves an earlier group's rows): the rows of the last group, 2.7 us per layer and item (128 positions
// of a KV head) of an SM, move without scoring beside them, those of the others at about a third of that time; so the sum is
// smallest at a number of groups near sqrt(1.75 layers items / launch), where a launch counts 13 us at 129 to 256 query rows
// and 24 below, where there is less to hide rows behind.  Beyond 256 rows Q leaves little room for rows on their way and
// the fewest groups win.  Measured, us, 8 KV heads unless said (groups of 1, 2, 3, 4, 8): 256 rows, 8 layers of 32K positions
// 693, 666, 685, 706, 747; four 370, 370, 370, 383; 16 of 8K 616, 453, 430, 396, 385; four 177, 138, 137, 132; 64 rows,
// eight of 4K, 16 heads 274, 213, 208, 194, 183; 128 rows, 16 of 30K, 2 heads 550, 385, 407, 359, 321; 448 rows, 4 of the
// ragged batch of eight 645, 680, 682, 608; 512 rows, 8 of 20K 717, 710, 713, 749, 700; 4 of 16K 324, 331, 331, 310.
//   Else (score ranking, rows that are not contiguous) selection and copy are launches of their own and every group pays for
// them: 32K x 8 ranked by score 896, 714, 657, 588, 548; 20K x 8 908, 762, 701, 633, 589; the ragged batch x 4 1011, 864,
// 864, 791.
int run_batch(const refree_params &p, int64_t total_tokens, int num_layers, size_t workspace_bytes, bool copy)
{
    int n = std::min(kMaxBatch, num_layers);
    const int rows = p.num_q_heads / p.num_kv_heads * p.window;
    if (copy && rows <= 256) {
        const double items = (double)(total_tokens / kTile + p.num_seqs) * p.num_kv_heads / sm_count();
        const int groups = std::max(1, (int)std::lround(std::sqrt(1.75 * num_layers * items / (rows > 128 ? 13.0 : 24.0))));
        n = std::min(n, (num_layers + groups - 1) / groups);
    }
    while (n > 1 && ((copy && !score_tc_can_copy(p, total_tokens, n)) || 2 * batch_layout(p, total_tokens, n).total > workspace_bytes)) --n;
    return n;
}

// Whether a layer's output lies over the cache of one of the layers that could share a launch with it: a caller may write
// a layer into the memory of an earlier one, whose rows have been moved by then if the layers are moved one by one.
bool outputs_over_caches(const refree_params &p, int num_layers, const void *const *k, const void *const *v, void *const *k_out,
                         void *const *v_out, int64_t capacity_rows)
{
    const size_t esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2, out = (size_t)capacity_rows * p.head_dim * esz;
    auto extent = [&](int64_t seq, int64_t tok, int64_t head) {
        return p.kv_tokens < 1 ? 0 : (size_t)((p.num_seqs - 1) * seq + (p.kv_tokens - 1) * tok + (p.num_kv_heads - 1) * head + p.head_dim) * esz;
    };
    const size_t kb = extent(p.k_stride_seq, p.k_stride_tok, p.k_stride_head), vb = extent(p.v_stride_seq, p.v_stride_tok, p.v_stride_head);
    auto meet = [](const void *x, size_t nx, const void *y, size_t ny) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(x), b = reinterpret_cast<uintptr_t>(y);
        return a < b + ny && b < a + nx;
    };
    for (int l = 1; l < num_layers; ++l)
        for (int m = std::max(0, l - kMaxBatch + 1); m < l; ++m)
            if (meet(k_out[l], out, k[m], kb) || meet(k_out[l], out, v[m], vb) || meet(v_out[l], out, k[m], kb) || meet(v_out[l], out, v[m], vb))
                return true;
    return false;
}
}  // namespace

refree_status refree_layers_workspace_size(const refree_params *p, int64_t total_tokens, size_t *bytes)
{
    const refree_status st = refree_workspace_size(p, total_tokens, bytes);
    if (st != REFREE_OK) return st;
    *bytes *= 2;
    if (score_tc_supported(*p)) *bytes = std::max(*bytes, 2 * batch_layout(*p, total_tokens, kMaxBatch).total);
    if (score_w1_supported(*p)) *bytes = std::max(*bytes, w1_batch_layout(*p, total_tokens, w1_batch(*p, total_tokens, kMaxBatch, kW1BatchBytes)).total);
    return st;
}

refree_status refree_compress_layers(const refree_params *p, int32_t num_layers,
                                     const void *const *q_win, const void *const *k, const void *const *v,
                                     const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                                     void *const *k_out, void *const *v_out, int64_t capacity_rows,
                                     int32_t *const *lengths, int64_t *const *offsets,
                                     void *workspace, size_t workspace_bytes,
                                     int32_t *device_status, void *stream)
{
    refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    if (num_layers < 0 || !q_win || !k || !v || !seq_start || !seq_len || !k_out || !v_out || !lengths || !offsets ||
        capacity_rows < 0)
        return REFREE_ERR_INVALID_ARG;
    for (int l = 0; l < num_layers; ++l) {
        if (!q_win[l] || !k[l] || !v[l] || !k_out[l] || !v_out[l] || !lengths[l] || !offsets[l])
            return REFREE_ERR_INVALID_ARG;
        st = check_kv_layout(p, k[l], v[l], true);
        if (st != REFREE_OK) return st;
        if ((reinterpret_cast<uintptr_t>(k_out[l]) & 15) || (reinterpret_cast<uintptr_t>(v_out[l]) & 15))
            return REFREE_ERR_UNSUPPORTED;
    }
    const Workspace lay = workspace_layout(*p, total_tokens);
    if (!workspace || workspace_bytes < 2 * lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return REFREE_ERR_WORKSPACE;
    if (num_layers == 0) return REFREE_OK;
    // One layer has nothing to overlap with (fp32, 111 positions, w = 1: 57 us on two streams, 45 this way).
    if (num_layers == 1) {
        const Stream cs = (cudaStream_t)stream;
        return enqueue_layer(p, q_win[0], k[0], v[0], seq_start, seq_len, total_tokens, k_out[0], v_out[0], capacity_rows,
                             lengths[0], offsets[0], nullptr, nullptr, (char *)workspace, lay, device_status, cs, cs, nullptr);
    }
    // Tensor-core path: one stream, layers in groups, no internal streams or events.  With position ranking and the rows of
    // a unit contiguous the scoring kernel of a group moves the kept rows of an earlier group with a warp of its own, and
    // the last group is compacted by a launch of its own; else selection and copy of a group are launches between.
    bool fused = total_tokens > 0 && !p->force_full;
    for (int l = 0; l < num_layers && fused; ++l) fused = use_tc(*p, q_win[l]);
    const bool one_by_one = outputs_over_caches(*p, num_layers, k, v, k_out, v_out, capacity_rows);
    const bool by_score = p->rank_mode == REFREE_RANK_SCORE;
    const bool copy = fused && !by_score && score_tc_can_copy(*p, total_tokens);
    if (fused) {
        // Group by group: launch j takes the column pass and the stopping rule of group j - 1, the row pass of group j and
        // the rows of group j - 2; then the last group's rows.  (Beyond their own launch the scores of a group are read by
        // the selection that follows it, before launch j + 1 writes into the same half of the workspace.)
        cudaStream_t cs = (cudaStream_t)stream;
        const int n = one_by_one ? 1 : run_batch(*p, total_tokens, num_layers, workspace_bytes, copy);
        const int ngroups = (num_layers + n - 1) / n;
        auto first_of = [&](int j) { return j < ngroups ? (int)((int64_t)num_layers * j / ngroups) : num_layers; };
        const BatchLayout bl = batch_layout(*p, total_tokens, n);
        const bool rule = !by_score && p->scope == REFREE_SCOPE_HEAD && total_tokens <= kGroupSelectMaxTokens;
        auto group_of = [&](int j) {
            TcGroup t = {};
            char *ws = (char *)workspace + (size_t)(j & 1) * bl.total;
            const int l0 = first_of(j);
            t.layers = first_of(j + 1) - l0;
            t.part = reinterpret_cast<float2 *>(ws + bl.part_off);
            t.scores = reinterpret_cast<float *>(ws + bl.scores_off);
            if (rule) {                                  // it runs inside the launch that finishes the group
                t.groups = reinterpret_cast<GroupPartial *>(ws + bl.grp_off);
                t.tickets = reinterpret_cast<uint32_t *>(ws + bl.tickets_off);
                t.cuts = reinterpret_cast<Cut *>(ws + bl.cut_off);
            }
            for (int l = 0; l < t.layers; ++l) {
                t.q_win[l] = q_win[l0 + l];
                t.k[l] = k[l0 + l];
                t.sel_lengths[l] = lengths[l0 + l];
            }
            return t;
        };
        // The first launch of the run is chained to what is ahead of it on the stream, which may still be writing Q and K: it
        // waits before it reads anything.  The launches behind it read Q and K before their wait.
        for (int j = 0; j <= ngroups; ++j) {
            TcGroup beg, fin;
            TcCopyJob job = {};
            if (j < ngroups) beg = group_of(j);
            if (j >= 1) fin = group_of(j - 1);
            if (copy && j >= 2) {
                const int l0 = first_of(j - 2);
                job.layers = first_of(j - 1) - l0;
                for (int l = 0; l < job.layers; ++l) {
                    job.k[l] = (const unsigned char *)k[l0 + l];
                    job.v[l] = (const unsigned char *)v[l0 + l];
                    job.k_out[l] = (unsigned char *)k_out[l0 + l];
                    job.v_out[l] = (unsigned char *)v_out[l0 + l];
                    job.lengths[l] = lengths[l0 + l];
                    job.offsets_out[l] = offsets[l0 + l];
                }
                job.capacity_rows = capacity_rows;
            }
            if (launch_score_tc_pipe(*p, j < ngroups ? &beg : nullptr, j >= 1 ? &fin : nullptr, seq_start, seq_len,
                                     total_tokens, device_status, cs, job.layers ? &job : nullptr, j == 0) != cudaSuccess)
                return REFREE_ERR_CUDA;
            if (j == 0) continue;
            const int l0 = first_of(j - 1);
            char *ws = (char *)workspace + (size_t)((j - 1) & 1) * bl.total;
            if (!rule) {
                Workspace sl = lay;                              // (the selection wants room for its records and counts)
                sl.cut_off = bl.cut_off;
                sl.part_off = bl.part_off;
                sl.part_bytes = bl.part_bytes;
                SelectOut so = {};
                so.layers = fin.layers;
                for (int l = 0; l < fin.layers; ++l) {
                    so.lengths[l] = lengths[l0 + l];
                    so.offsets[l] = offsets[l0 + l];
                    so.kept[l] = by_score ? reinterpret_cast<int32_t *>(ws + bl.kept_off) + (int64_t)l * p->num_kv_heads * total_tokens
                                          : nullptr;
                }
                if (launch_select(*p, fin.scores, seq_len, total_tokens, so, capacity_rows, ws, sl, device_status, cs, by_score) !=
                    cudaSuccess)
                    return REFREE_ERR_CUDA;
            }
            if (copy && j < ngroups) continue;                   // a later launch moves the rows
            CompactJob cj = {};
            cj.layers = fin.layers;
            for (int l = 0; l < fin.layers; ++l) {
                cj.k[l] = (const char *)k[l0 + l];
                cj.v[l] = (const char *)v[l0 + l];
                cj.lengths[l] = lengths[l0 + l];
                cj.offsets[l] = offsets[l0 + l];
                cj.kept[l] = by_score ? reinterpret_cast<const int32_t *>(ws + bl.kept_off) + (int64_t)l * p->num_kv_heads * total_tokens
                                      : nullptr;
                cj.offsets_out[l] = by_score ? nullptr : offsets[l0 + l];
                cj.k_out[l] = (char *)k_out[l0 + l];
                cj.v_out[l] = (char *)v_out[l0 + l];
            }
            if (launch_compact(*p, cj, seq_start, seq_len, !by_score, capacity_rows, device_status, cs) != cudaSuccess)
                return REFREE_ERR_CUDA;
        }
        return REFREE_OK;
    }
    // Single query row: scoring is a chain of short kernels, so the layers of a group go through each of them together, and
    // then through one copy.  (In place of one layer after the other with the copies on a second stream; a run, us: eight
    // layers of 32K positions 548 -> 512, 16 of 8K 543 -> 272, eight of 333 198 -> 18, with score ranking at 32K 653 -> 459.)
    // Queries that start on 16 bytes take another kernel than those that do not: a run with both goes layer by layer, so that
    // each layer takes the one that it takes alone.
    int on16 = 0;
    for (int l = 0; l < num_layers; ++l) on16 += !(reinterpret_cast<uintptr_t>(q_win[l]) & 15);
    const int w1_n = total_tokens > 0 && !p->force_full && score_w1_supported(*p) && (on16 == 0 || on16 == num_layers)
                         ? one_by_one ? 1 : w1_batch(*p, total_tokens, num_layers, workspace_bytes) : 0;
    if (w1_n > 0 && w1_batch_layout(*p, total_tokens, w1_n).total <= workspace_bytes) {
        cudaStream_t cs = (cudaStream_t)stream;
        char *ws = (char *)workspace;
        const W1BatchLayout bl = w1_batch_layout(*p, total_tokens, w1_n);
        const bool rule = !by_score && p->scope == REFREE_SCOPE_HEAD && total_tokens <= kGroupSelectMaxTokens;
        const int64_t layer_scores = (int64_t)p->num_kv_heads * total_tokens;
        const int ngroups = (num_layers + w1_n - 1) / w1_n;
        for (int j = 0; j < ngroups; ++j) {
            const int l0 = (int)((int64_t)num_layers * j / ngroups), n = (int)((int64_t)num_layers * (j + 1) / ngroups) - l0;
            W1Group g = {};
            SelectOut so = {};
            CompactJob cj = {};
            g.layers = so.layers = cj.layers = n;
            g.scratch = ws + bl.scratch_off;
            g.scores = reinterpret_cast<float *>(ws + bl.scores_off);
            g.groups = rule ? reinterpret_cast<GroupPartial *>(ws + bl.grp_off) : nullptr;
            g.cuts = rule ? reinterpret_cast<Cut *>(ws + bl.cut_off) : nullptr;
            for (int l = 0; l < n; ++l) {
                g.q_win[l] = q_win[l0 + l];
                g.k[l] = k[l0 + l];
                g.sel_lengths[l] = so.lengths[l] = lengths[l0 + l];
                so.offsets[l] = offsets[l0 + l];
                so.kept[l] = by_score ? reinterpret_cast<int32_t *>(ws + bl.kept_off) + l * layer_scores : nullptr;
                cj.k[l] = (const char *)k[l0 + l];
                cj.v[l] = (const char *)v[l0 + l];
                cj.lengths[l] = lengths[l0 + l];
                cj.offsets[l] = offsets[l0 + l];
                cj.kept[l] = so.kept[l];
                cj.offsets_out[l] = by_score ? nullptr : offsets[l0 + l];
                cj.k_out[l] = (char *)k_out[l0 + l];
                cj.v_out[l] = (char *)v_out[l0 + l];
            }
            if (launch_score_w1(*p, g, seq_start, seq_len, total_tokens, device_status, cs) != cudaSuccess) return REFREE_ERR_CUDA;
            if (!rule) {
                Workspace sl = lay;
                sl.cut_off = bl.cut_off;
                sl.part_off = bl.scratch_off;               // (the logits have been read: room for the counts of the index list)
                sl.part_bytes = bl.scratch_bytes;
                if (launch_select(*p, g.scores, seq_len, total_tokens, so, capacity_rows, ws, sl, device_status, cs, by_score) !=
                    cudaSuccess)
                    return REFREE_ERR_CUDA;
            }
            if (launch_compact(*p, cj, seq_start, seq_len, !by_score, capacity_rows, device_status, cs) != cudaSuccess)
                return REFREE_ERR_CUDA;
        }
        return REFREE_OK;
    }
    LayerPipe *lp = layer_pipe();
    if (!lp) return REFREE_ERR_CUDA;
    cudaStream_t cs = (cudaStream_t)stream;
    bool ok = cudaEventRecord(lp->fork, cs) == cudaSuccess && cudaStreamWaitEvent(lp->hi, lp->fork, 0) == cudaSuccess &&
              cudaStreamWaitEvent(lp->lo, lp->fork, 0) == cudaSuccess;
    refree_status result = ok ? REFREE_OK : REFREE_ERR_CUDA;
    for (int l = 0; l < num_layers && result == REFREE_OK; ++l) {
        const int slot = l & 1;
        // the half of the workspace is free once the compaction of layer l - 2 has read its budgets
        if (l >= 2 && cudaStreamWaitEvent(lp->hi, lp->compacted[slot], 0) != cudaSuccess) { result = REFREE_ERR_CUDA; break; }
        result = enqueue_layer(p, q_win[l], k[l], v[l], seq_start, seq_len, total_tokens, k_out[l], v_out[l],
                               capacity_rows, lengths[l], offsets[l], nullptr, nullptr,
                               (char *)workspace + (size_t)slot * lay.total, lay, device_status, lp->hi, lp->lo,
                               lp->scored[slot]);
        if (result != REFREE_OK) break;
        if (cudaEventRecord(lp->compacted[slot], lp->lo) != cudaSuccess) { result = REFREE_ERR_CUDA; break; }
    }
    // the caller's stream continues after everything that was enqueued, whatever happened
    if (ok) {
        if (cudaEventRecord(lp->join, lp->hi) != cudaSuccess || cudaStreamWaitEvent(cs, lp->join, 0) != cudaSuccess ||
            cudaEventRecord(lp->join, lp->lo) != cudaSuccess || cudaStreamWaitEvent(cs, lp->join, 0) != cudaSuccess)
            if (result == REFREE_OK) result = REFREE_ERR_CUDA;
    }
    return result;
}

refree_status refree_host_arena_size(const refree_params *p, int64_t total_tokens,
                                     int64_t kv_elems, int64_t capacity_rows, size_t *bytes)
{
    if (!bytes || kv_elems < 0 || capacity_rows < 0) return REFREE_ERR_INVALID_ARG;
    const refree_status st = check_params(p, total_tokens);
    if (st != REFREE_OK) return st;
    const size_t esz = p->dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const size_t U = (size_t)p->num_seqs * p->num_kv_heads;
    size_t tot = 0;
    tot += align256((size_t)p->num_seqs * p->num_q_heads * p->window * p->head_dim * esz);  // q_win
    tot += 2 * align256((size_t)kv_elems * esz);                                            // k, v
    tot += 2 * align256((size_t)p->num_seqs * sizeof(int32_t));                             // seq_start, seq_len
    tot += 2 * align256((size_t)capacity_rows * p->head_dim * esz);                         // k_out, v_out
    tot += align256(U * sizeof(int32_t)) + align256((U + 1) * sizeof(int64_t));             // lengths, offsets
    tot += align256((size_t)capacity_rows * sizeof(int32_t));                               // kept_idx
    tot += align256((size_t)p->num_kv_heads * total_tokens * sizeof(float));                // scores
    tot += align256(sizeof(int32_t));                                                       // device status
    tot += workspace_layout(*p, total_tokens).total;
    *bytes = tot;
    return REFREE_OK;
}

refree_status refree_compress_layer_host(const refree_params *p, const void *q_win,
                                         const void *k, const void *v, int64_t kv_elems,
                                         const int32_t *seq_start, const int32_t *seq_len,
                                         int64_t total_tokens,
                                         void *k_out, void *v_out, int64_t capacity_rows,
                                         int32_t *lengths, int64_t *offsets,
                                         int32_t *kept_idx, float *scores,
                                         void *arena, size_t arena_bytes, void *stream)
{
    size_t need = 0;
    refree_status st = refree_host_arena_size(p, total_tokens, kv_elems, capacity_rows, &need);
    if (st != REFREE_OK) return st;
    if (!q_win || !k || !v || !seq_start || !seq_len || !k_out || !v_out || !lengths || !offsets)
        return REFREE_ERR_INVALID_ARG;
    if (!arena || arena_bytes < need || (reinterpret_cast<uintptr_t>(arena) & 255)) return REFREE_ERR_WORKSPACE;
    cudaStream_t cs = (cudaStream_t)stream;
    const size_t esz = p->dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const size_t U = (size_t)p->num_seqs * p->num_kv_heads;
    char *a = (char *)arena;
    auto take = [&](size_t bytes) { char *r = a; a += align256(bytes); return r; };
    const size_t q_bytes = (size_t)p->num_seqs * p->num_q_heads * p->window * p->head_dim * esz;
    const size_t kv_bytes = (size_t)kv_elems * esz;
    const size_t row_bytes = (size_t)p->head_dim * esz;
    char *d_q = take(q_bytes), *d_k = take(kv_bytes), *d_v = take(kv_bytes);
    int32_t *d_start = (int32_t *)take(p->num_seqs * sizeof(int32_t));
    int32_t *d_len = (int32_t *)take(p->num_seqs * sizeof(int32_t));
    char *d_ko = take(capacity_rows * row_bytes), *d_vo = take(capacity_rows * row_bytes);
    int32_t *d_lengths = (int32_t *)take(U * sizeof(int32_t));
    int64_t *d_offsets = (int64_t *)take((U + 1) * sizeof(int64_t));
    int32_t *d_kept = (int32_t *)take((size_t)capacity_rows * sizeof(int32_t));
    float *d_scores = (float *)take((size_t)p->num_kv_heads * total_tokens * sizeof(float));
    int32_t *d_status = (int32_t *)take(sizeof(int32_t));
    char *d_ws = a;
    const size_t ws_bytes = workspace_layout(*p, total_tokens).total;

    cudaError_t e;
    if ((e = cudaMemcpyAsync(d_q, q_win, q_bytes, cudaMemcpyHostToDevice, cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if ((e = cudaMemcpyAsync(d_k, k, kv_bytes, cudaMemcpyHostToDevice, cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if ((e = cudaMemcpyAsync(d_v, v, kv_bytes, cudaMemcpyHostToDevice, cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if ((e = cudaMemcpyAsync(d_start, seq_start, p->num_seqs * sizeof(int32_t), cudaMemcpyHostToDevice, cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if ((e = cudaMemcpyAsync(d_len, seq_len, p->num_seqs * sizeof(int32_t), cudaMemcpyHostToDevice, cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if ((e = cudaMemsetAsync(d_status, 0, sizeof(int32_t), cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    st = refree_compress_layer(p, d_q, d_k, d_v, d_start, d_len, total_tokens, d_ko, d_vo, capacity_rows,
                               d_lengths, d_offsets, kept_idx ? d_kept : nullptr, scores ? d_scores : nullptr,
                               d_ws, ws_bytes, d_status, stream);
    if (st != REFREE_OK) return st;
    int32_t h_status = 0;
    cudaMemcpyAsync(lengths, d_lengths, U * sizeof(int32_t), cudaMemcpyDeviceToHost, cs);
    cudaMemcpyAsync(offsets, d_offsets, (U + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, cs);
    cudaMemcpyAsync(&h_status, d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, cs);
    if ((e = cudaStreamSynchronize(cs)) != cudaSuccess) return REFREE_ERR_CUDA;
    if (h_status & REFREE_DEV_TIMEOUT) return REFREE_ERR_TIMEOUT;
    if (h_status & REFREE_DEV_CAPACITY) return REFREE_ERR_CAPACITY;
    if (h_status & REFREE_DEV_NONFINITE) return REFREE_ERR_NONFINITE;
    const int64_t rows = offsets[U];
    cudaMemcpyAsync(k_out, d_ko, (size_t)rows * row_bytes, cudaMemcpyDeviceToHost, cs);
    cudaMemcpyAsync(v_out, d_vo, (size_t)rows * row_bytes, cudaMemcpyDeviceToHost, cs);
    if (kept_idx) cudaMemcpyAsync(kept_idx, d_kept, (size_t)rows * sizeof(int32_t), cudaMemcpyDeviceToHost, cs);
    if (scores)
        cudaMemcpyAsync(scores, d_scores, (size_t)p->num_kv_heads * total_tokens * sizeof(float), cudaMemcpyDeviceToHost, cs);
    return from_cuda(cudaStreamSynchronize(cs));
}

}  // extern "C"
