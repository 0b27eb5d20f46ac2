// Internal declarations shared by the kernels of the compression-pass library.
#pragma once

#include <mutex>
#include <utility>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "refreekv.h"

namespace refree {

constexpr int kMaxSeqs = 1024;   // sequences per call (prefix tables live in shared memory)
constexpr int kTile = 128;       // positions per scoring tile
constexpr int kMaxRows = 1024;   // G * window handled by the generic scoring path
// Longer windows (Section 4.4 studies windows of up to a tenth of the sequence) are scored in chunks of query rows
// that the scoring paths take, each chunk a window of its own over a sequence cut at its last row.
constexpr int kMaxRowsChunked = 32768;
constexpr int kMaxGroupChunked = 256;   // query heads per KV head when the window is chunked

// Bounded spin: polls before a wait gives up and reports REFREE_DEV_TIMEOUT.
constexpr uint32_t kSpinLimit = 1u << 22;
// The stopping rule fed by per-32-position records sums each group at a scale set by the group's own largest
// score and shifts the sums to the unit's scale, so it drops up to one unit of the fixed point per element and per
// group: about n * 2^(L - 54) of C_n with L = log2(groups), against n * 2^-60 for the rule that reads every score.
// That is 2^-29 at 32K positions and still 2^-25 at 128K, far inside the near-tie band; longer sequences take the
// rule that reads every score.
constexpr int64_t kGroupSelectMaxTokens = 131072;

// Layout of the caller-provided workspace.  All offsets are multiples of 256.
struct Workspace {
    size_t part_off, part_bytes;       // per (tile, head, row) softmax partials (float2: max, sum)
    size_t lse_off, lse_bytes;         // generic path: per (unit, row) log2-sum-exp of the row's logits
    size_t grp_off, grp_bytes;         // per 32 positions: exact partial sum of squared scores (GroupPartial)
    size_t cut_off, cut_bytes;         // per unit selection result (struct Cut)
    size_t scores_off, scores_bytes;   // scratch scores when the caller passes none
    size_t kept_off, kept_bytes;       // scratch kept_idx when the caller passes none
    size_t chk_off, chk_bytes;         // chunked windows: one chunk's query rows, its scores, its sequence lengths
    size_t total;
};

// Result of the stopping rule for one unit, enough to enumerate its kept set.
//   position ranking: kept = [0, min(b, lead)) U [n - (b - lead), n)
//   score ranking:    kept = the first min(b, lead + w_eff) protected positions in
//                     order (leading then window), plus unprotected positions whose
//                     key is above `tau`, plus the first `ties` (by position) whose
//                     key equals `tau`.
struct Cut {
    int32_t b;          // budget (kept count)
    int32_t ties;       // score ranking: number of positions with key == tau to keep
    uint64_t tau;       // score ranking: key threshold (score bits << 32, or the fixed-point layer key)
    int32_t prot_kept;  // score ranking: protected positions kept
    int32_t sbias;      // fixed-point exponent bias of the unit's squares (see select.cu)
};

// Sum of squared scores of 32 consecutive positions of one unit, written by the
// scoring kernel so that the stopping rule need not re-read every score.
//   max_bits  bit pattern of the largest score of the group (0 when all are zero)
//   sum       sum over the group of floor(a^2 * 2^(308 - 2E)), E = exponent field of
//             max_bits (at least 1): exact integer squares, at most 2^61 in total
// Records of unit (s, g) are contiguous: index (tiles[s] * Hkv + g * tiles_of(s)) * 4 + i / 32.
struct GroupPartial {
    uint32_t max_bits;
    uint32_t pad;
    unsigned long long sum;
};
constexpr int kGroupShift = 8;   // the squared mantissa (below 2^48) of the group's largest score lands below 2^56

Workspace workspace_layout(const refree_params &p, int64_t total_tokens);

// Bookkeeping for refree_kernel_launch_count(): every launcher adds the kernels it enqueued.
void count_launches(int n);

// Multiprocessors of the current device (looked up once per device; launch geometry is sized by it).
int sm_count();

inline __host__ __device__ int ceil_div(int a, int b) { return (a + b - 1) / b; }

// |a| as an integer: non-negative floats order like their bit patterns
__device__ inline uint32_t mag_bits(float a) { return __float_as_uint(a) & 0x7fffffffu; }

// floor(a^2 * 2^S) from the bits of |a|, where 2 * exponent_field + sbias is the left
// shift of the exact 48-bit squared mantissa (S = sbias + 300); non-finite values count as zero
__device__ inline unsigned long long sq_fixed(uint32_t bits, int sbias)
{
    const uint32_t e = bits >> 23;
    if (e == 255u) return 0ull;
    const uint32_t m = (bits & 0x7fffffu) | (e ? 0x800000u : 0u);
    const unsigned long long mm = (unsigned long long)m * m;     // exact, below 2^48
    const int sh = 2 * (int)(e ? e : 1u) + sbias;
    if (sh >= 0) return sh < 16 ? mm << sh : ~0ull >> 2;
    return -sh < 48 ? mm >> -sh : 0ull;
}

template <typename T> __device__ inline float to_float(T v);
template <> __device__ inline float to_float<float>(float v) { return v; }
template <> __device__ inline float to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename Tv> __device__ inline Tv warp_incl_scan(Tv x)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Tv y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// ---- dependent launches ------------------------------------------------------
// Every kernel of a call may be launched while the kernel before it on the stream drains (programmatic dependent
// launch), which takes the launch latency out of a chain of short kernels.  Rules that keep this safe:
//   - nothing is written to global memory before dependency_wait(), and at least one thread of the grid waits on every path,
//     so that the end of a kernel means the end of all before it;
//   - the first kernel of a call triggers its dependents after its wait, later ones may do so at once: the inputs of the call
//     (sequence tables, queries, keys, values) were complete before the first one and may be read before any wait;
//   - a result of an earlier kernel of the call may be read before the wait only behind a kernel that triggers after its own:
//     what was ahead of that one is complete then.  (The index list reads scores this way, behind the two kernels of score
//     ranking, the merge of the decode step the lengths, behind its attention kernel; the triggers that must stay behind their
//     waits say so.)
// A stream, and whether the next launch on it may be chained this way.  Also where a second stream works beside it (a run
// of layers on two streams, us, chained and not: fp32 d 64, eight layers of 3000 positions, 32 rows, 208 and 287; bf16 d 64,
// four of 32K 325 and 370; windows in chunks, six layers of 2000 positions, 1200 rows, 766 and 841).
struct Stream {
    cudaStream_t s;
    bool chain;
    int carveout = -1;       // share of an SM's shared memory that the next launch asks for, percent
    Stream(cudaStream_t st, bool chained = true) : s(st), chain(chained) {}
    operator cudaStream_t() const { return s; }
};

__device__ inline void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ inline void trigger_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_dependent_cluster(void (*kernel)(P...), int cluster, dim3 grid, dim3 block, size_t smem, Stream st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[3];
    int n = 0;
    if (st.carveout >= 0) {
        attr[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[n++].val.sharedMemCarveout = st.carveout;
    }
    if (st.chain) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, Stream st, A... args)
{
    return launch_dependent_cluster(kernel, 1, grid, block, smem, st, args...);
}

// Dynamic shared memory above the default limit is allowed once per kernel and device (always with the same size).
template <typename Kern>
inline cudaError_t allow_smem(Kern kern, size_t smem)
{
    static std::mutex m;                           // one per kernel type; kernels of one type are told apart by address
    static std::vector<std::pair<int, Kern>> done;
    if (smem <= 48 * 1024) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> hold(m);
    for (const auto &d : done)
        if (d.first == dev && d.second == kern) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) done.emplace_back(dev, kern);
    return e;
}

// ---- launchers (defined in the .cu files) ----------------------------------
cudaError_t launch_score_generic(const refree_params &p, const void *q_win, const void *k,
                                 const int32_t *seq_start, const int32_t *seq_len,
                                 int64_t total_tokens, float *scores, char *ws, const Workspace &lay,
                                 int32_t *dev_status, Stream st, GroupPartial *groups = nullptr, int32_t *sel_lengths = nullptr);
// Whether launch_score_generic evaluates the stopping rule too, given `groups` and `sel_lengths` (short calls).
bool score_generic_rule(const refree_params &p, int64_t total_tokens);

// Layers of a run that one launch scores together, at most (see refree_compress_layers).
constexpr int kMaxBatch = 8;

// Rows of other layers (position ranking: a prefix and a suffix per unit) that the tensor-core scoring
// kernel moves with a warp of its own while it scores, HBM being nearly idle then.  The budgets are read
// on the device; the kernel forms their running sum itself.
struct TcCopyJob {
    int layers;                                  // 0: nothing to move
    const unsigned char *k[kMaxBatch], *v[kMaxBatch];    // source caches (same strides and sequences as the scored layers)
    unsigned char *k_out[kMaxBatch], *v_out[kMaxBatch];  // dense outputs [capacity_rows, d]
    const int32_t *lengths[kMaxBatch];           // [num_seqs * num_kv_heads] budgets
    int64_t *offsets_out[kMaxBatch];             // [units + 1] running sum of the budgets
    int64_t capacity_rows;
    int nslots, piece_rows;         // pieces in flight and their rows; set by the launcher
};

// Returns false when the shape is outside what the tensor-core path handles.
bool score_tc_supported(const refree_params &p);
// True when launch_score_tc can also carry a TcCopyJob for these parameters (rows of a unit contiguous in
// K and V, few enough units, shared memory left for the pieces in flight).
bool score_tc_can_copy(const refree_params &p, int64_t total_tokens, int layers = 1);
// Both passes of one layer.  With `groups` and `sel_lengths` (position ranking per head) the stopping rule is evaluated
// too: budgets to sel_lengths, Cut records to the workspace.  The same for launch_score_w1.
cudaError_t launch_score_tc(const refree_params &p, const void *q_win, const void *k,
                            const int32_t *seq_start, const int32_t *seq_len,
                            int64_t total_tokens, float *scores, char *ws, const Workspace &lay,
                            int32_t *dev_status, Stream st, GroupPartial *groups = nullptr,
                            int32_t *sel_lengths = nullptr);

// A group of consecutive layers of a run that the same launches score.  What a launch keeps of a layer follows what it
// keeps of the layer before.
struct TcGroup {
    int layers;
    const void *q_win[kMaxBatch], *k[kMaxBatch];
    float2 *part;           // layers x [256 + units of a layer, column half, padded rows]: partials between the two passes
    float *scores;          // [layers x Hkv, total_tokens]
    GroupPartial *groups;   // nullable: records for the stopping rule (position ranking per head)
    // nullable: the launch that finishes the group evaluates the rule too
    uint32_t *tickets;      // [2 units]
    Cut *cuts;              // [units]
    int32_t *sel_lengths[kMaxBatch];
};
// One launch of a run: the column pass of `finish`, then the row pass of `begin` (either may be null), and the
// rows of `copy` (nullable) moved beside them.  `first`: the launch is ordered behind all that is ahead of it on the
// stream; later launches of the run start while the one before drains.  A launch clears the tickets of its `begin` group.
cudaError_t launch_score_tc_pipe(const refree_params &p, const TcGroup *begin, const TcGroup *finish,
                                 const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                                 int32_t *dev_status, Stream st, const TcCopyJob *copy, bool first);

// Single query row per head (the paper's default reduced attention): a stream over K on the fp32 pipes.
bool score_w1_supported(const refree_params &p);
size_t score_w1_scratch_bytes(const refree_params &p, int64_t total_tokens);
struct W1Group {
    int layers;
    const void *q_win[kMaxBatch], *k[kMaxBatch];
    char *scratch;          // layers x score_w1_scratch_bytes, each rounded up to 256
    float *scores;          // [layers x Hkv, total_tokens]
    GroupPartial *groups;   // nullable; a layer's tiles x Hkv x 4 after another
    Cut *cuts;              // nullable: with `groups` the stopping rule is evaluated too
    int32_t *sel_lengths[kMaxBatch];
};
cudaError_t launch_score_w1(const refree_params &p, const W1Group &g, const int32_t *seq_start, const int32_t *seq_len,
                            int64_t total_tokens, int32_t *dev_status, Stream st);

// The layers of a run that one launch of the selection or of the copy takes together, one layer in the other calls.
struct SelectOut {
    int layers;
    int32_t *lengths[kMaxBatch];
    int64_t *offsets[kMaxBatch];
    int32_t *kept[kMaxBatch];       // nullable: index lists
};
struct CompactJob {
    int layers;
    const char *k[kMaxBatch], *v[kMaxBatch];
    const int32_t *lengths[kMaxBatch];
    const int64_t *offsets[kMaxBatch];      // read unless offsets_out forms them
    const int32_t *kept[kMaxBatch];         // nullable with position ranges
    int64_t *offsets_out[kMaxBatch];        // nullable: the kernel forms the running sum of the budgets itself
    int32_t *kept_out[kMaxBatch];           // nullable, position ranges: the kernel writes the index list
    char *k_out[kMaxBatch], *v_out[kMaxBatch];      // either null: those rows are not moved
    bool after_rule;                        // behind a launch that chose the budgets from the scores (position ranking)
};

// The stopping rule of every unit from the records that the scoring left (position ranking per head).
cudaError_t launch_unit_rules(const refree_params &p, const float *scores, const int32_t *seq_len, int64_t total_tokens,
                              const GroupPartial *groups, int64_t layer_groups, const SelectOut &out, Cut *cuts, Stream st);

// Scores of layer l at scores + l Hkv total_tokens, Cut records at ws + lay.cut_off, units after units.
cudaError_t launch_select(const refree_params &p, const float *scores, const int32_t *seq_len,
                          int64_t total_tokens, const SelectOut &out, int64_t capacity_rows, char *ws, const Workspace &lay,
                          int32_t *dev_status, Stream st, bool emit = true, bool have_budgets = false);
inline SelectOut select_out(int32_t *lengths, int64_t *offsets, int32_t *kept)
{
    SelectOut o = {};
    o.layers = 1;
    o.lengths[0] = lengths; o.offsets[0] = offsets; o.kept[0] = kept;
    return o;
}

cudaError_t launch_compact(const refree_params &p, const CompactJob &job, const int32_t *seq_start, const int32_t *seq_len,
                           bool position_ranges, int64_t capacity_rows, int32_t *dev_status, Stream st);
inline CompactJob compact_job(const void *k, const void *v, const int32_t *lengths, const int64_t *offsets, const int32_t *kept,
                              int64_t *offsets_out, void *k_out, void *v_out, int32_t *kept_out = nullptr)
{
    CompactJob j = {};
    j.layers = 1;
    j.k[0] = (const char *)k; j.v[0] = (const char *)v;
    j.lengths[0] = lengths; j.offsets[0] = offsets; j.kept[0] = kept; j.offsets_out[0] = offsets_out;
    j.kept_out[0] = kept_out;
    j.k_out[0] = (char *)k_out; j.v_out[0] = (char *)v_out;
    return j;
}

// Strides and alignment of a layer's caches.
refree_status check_kv_layout(const refree_params *p, const void *k, const void *v, bool need_v);
// Scoring and selection of one layer; launch_compact with `job` is what is left of it.
cudaError_t enqueue_selection(const refree_params &p, const void *q_win, const void *k, const void *v, const int32_t *seq_start,
                              const int32_t *seq_len, int64_t total_tokens, void *k_out, void *v_out, int64_t capacity_rows,
                              int32_t *lengths, int64_t *offsets, int32_t *kept_idx, float *scores, char *ws, const Workspace &lay,
                              int32_t *device_status, Stream cs, CompactJob &job);

// With `lengths` and `offsets_out` (end-anchored form only) the kernel takes the budgets from `lengths` and
// writes their running sum itself, so the selection need not emit offsets first.
cudaError_t launch_compact_inplace(const refree_params &p, void *k, void *v, const int32_t *seq_start,
                                   const int32_t *seq_len, const int64_t *offsets, const int32_t *kept_idx,
                                   bool position_ranges, bool anchor_back, int32_t *dev_status, Stream st,
                                   const int32_t *lengths = nullptr, int64_t *offsets_out = nullptr);

cudaError_t launch_compact_paged(const refree_params &p, const void *k, const void *v, const int32_t *seq_start,
                                 const int32_t *seq_len, const int32_t *lengths, const int64_t *offsets,
                                 const int32_t *kept_idx, bool position_ranges, const int32_t *block_table,
                                 int max_blocks_per_unit, int block_rows, void *k_pool, void *v_pool,
                                 int64_t num_blocks, int32_t *dev_status, Stream st);

size_t decode_workspace_bytes(const refree_params &p, int64_t max_rows);
cudaError_t launch_decode_attention(const refree_params &p, const void *q_new, const void *k_c, const void *v_c,
                                    const int64_t *offsets, int64_t max_rows, float *out, void *workspace,
                                    int32_t *dev_status, Stream st, const int32_t *seq_start = nullptr,
                                    const int32_t *seq_len = nullptr, const int32_t *lengths = nullptr,
                                    bool anchor_back = false);

}  // namespace refree
