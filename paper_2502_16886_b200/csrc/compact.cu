// Step S7: gather the kept K and V rows of every unit into the dense ragged
// output (Algorithm 1, "Compress" steps).  Pure data movement: 16-byte vector
// loads and stores, several rows in flight per thread.  Rows are copied bit for
// bit.  With position ranking the kept set is two contiguous ranges, so the
// source row follows from (b, m, n) and no index list is read.
#include <mutex>
#include <cooperative_groups.h>

#include <algorithm>

#include "refree_internal.cuh"

namespace refree {
namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 4;

__device__ inline int4 ld_stream(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ inline void st_stream(int4 *p, const int4 &v)
{
    asm volatile("st.global.cs.v4.s32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

__global__ void __launch_bounds__(kThreads)
compact_kernel(refree_params p, const __grid_constant__ CompactJob job, const int32_t *seq_start, const int32_t *seq_len,
               int position_ranges, int64_t capacity_rows, int32_t *dev_status)
{
    __shared__ long long s_part[kThreads / 32];
    const int Hkv = p.num_kv_heads;
    const int u = blockIdx.y, s = u / Hkv, g = u % Hkv, layer = blockIdx.z;
    const char *const k = job.k[layer], *const v = job.v[layer];
    const int32_t *const lengths = job.lengths[layer], *const kept_idx = job.kept[layer];
    int64_t *const offsets_out = job.offsets_out[layer];
    dependency_wait();
    trigger_dependents();
    const int esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const int row_bytes = p.head_dim * esz;
    const int vec_per_row = row_bytes >> 4;
    const int vshift = 31 - __clz(vec_per_row);
    const int n = max(seq_len[s], 0);
    const int b = lengths[u];
    int64_t off;
    if (offsets_out) {
        // fused pass: the running sum of the budgets is formed here instead of in a launch of its own
        long long part = 0;
        for (int t = threadIdx.x; t < u; t += kThreads) part += lengths[t];
        for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
        __syncthreads();
        off = 0;
        for (int wv = 0; wv < kThreads / 32; ++wv) off += s_part[wv];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            offsets_out[u] = off;
            if (u == (int)gridDim.y - 1) offsets_out[u + 1] = off + b;
        }
    } else {
        off = job.offsets[layer][u];
    }
    if (b < 0 || b > n || off < 0 || off + b > capacity_rows) {
        if (threadIdx.x == 0 && blockIdx.x == 0 && dev_status) atomicOr(dev_status, REFREE_DEV_CAPACITY);
        return;
    }
    const int head = min(b, min(p.sink, n));
    const int64_t tok0 = seq_start[s];
    if (int32_t *const list = job.kept_out[layer])
        for (int t = blockIdx.x * kThreads + threadIdx.x; t < b; t += gridDim.x * kThreads) list[off + t] = t < head ? t : n - b + t;
    const char *kb = k + ((int64_t)s * p.k_stride_seq + tok0 * p.k_stride_tok + (int64_t)g * p.k_stride_head) * esz;
    const char *vb = v + ((int64_t)s * p.v_stride_seq + tok0 * p.v_stride_tok + (int64_t)g * p.v_stride_head) * esz;
    const int64_t k_tok = p.k_stride_tok * esz, v_tok = p.v_stride_tok * esz;
    const bool move_k = job.k_out[layer] != nullptr, move_v = job.v_out[layer] != nullptr;
    char *ko = job.k_out[layer] + off * row_bytes, *vo = job.v_out[layer] + off * row_bytes;
    const int32_t *idx = kept_idx ? kept_idx + off : nullptr;
    const int64_t nvec = (int64_t)b << vshift;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t e0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; e0 < nvec; e0 += stride * kUnroll) {
        int4 kv[kUnroll], vv[kUnroll];
        bool good[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            const int64_t e = e0 + r * stride;
            good[r] = false;
            if (e < nvec) {
                const int t = (int)(e >> vshift), c = (int)(e & (vec_per_row - 1));
                const int src = position_ranges ? (t < head ? t : n - b + t) : idx[t];
                // an index list is the caller's: a row outside the sequence is reported, never read
                good[r] = src >= 0 && src < n;
                if (good[r]) {
                    if (move_k) kv[r] = *reinterpret_cast<const int4 *>(kb + (int64_t)src * k_tok + c * 16);
                    if (move_v) vv[r] = ld_stream(reinterpret_cast<const int4 *>(vb + (int64_t)src * v_tok + c * 16));
                } else if (dev_status) {
                    atomicOr(dev_status, REFREE_DEV_CAPACITY);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            const int64_t e = e0 + r * stride;
            if (e < nvec && good[r]) {
                if (move_k) st_stream(reinterpret_cast<int4 *>(ko + e * 16), kv[r]);
                if (move_v) st_stream(reinterpret_cast<int4 *>(vo + e * 16), vv[r]);
            }
        }
    }
}


// In-place form of the same step.  Every kept row moves towards the front of its own unit
// (destination index t <= source index), so rows can be overwritten as soon as whoever
// needs their old contents has read them.  The kept rows of all units, in order, are cut
// into rounds of as many 16-byte pieces as the grid holds in registers; in a round every
// thread loads its pieces, the grid synchronises, and every thread stores them.  A round
// reads only rows at or beyond its own destinations, which lie beyond every destination of
// the rounds before it, so one grid barrier per round is all the ordering needed.
constexpr int kUnrollInplace = 4;
constexpr int kInplaceTable = 1024;   // running sums held in shared memory (8 KB)

__global__ void __launch_bounds__(kThreads, 4)
compact_inplace_kernel(refree_params p, char *k, char *v, const int32_t *seq_start, const int32_t *seq_len,
                       const int64_t *offsets, const int32_t *kept_idx, int position_ranges, int32_t *dev_status)
{
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const int Hkv = p.num_kv_heads, U = p.num_seqs * Hkv;
    const int esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const int vec_per_row = (p.head_dim * esz) >> 4;
    const int vshift = 31 - __clz(vec_per_row);
    // the running sums are searched once per piece: keep them in shared memory when they fit
    __shared__ int64_t s_off[kInplaceTable];
    const int64_t *tab = offsets;
    if (U + 1 <= kInplaceTable) {
        for (int i = threadIdx.x; i <= U; i += kThreads) s_off[i] = __ldg(offsets + i);
        __syncthreads();
        tab = s_off;
    }
    const int64_t total_vec = max((long long)tab[U], 0ll) << vshift;
    const int64_t lanes = (int64_t)gridDim.x * kThreads;
    const int64_t per_round = lanes * kUnrollInplace;
    const int64_t k_tok = p.k_stride_tok * esz, v_tok = p.v_stride_tok * esz;
    bool bad = false;
    for (int64_t base = 0; base < total_vec; base += per_round) {     // the same trip count in every thread
        int4 kv[kUnrollInplace], vv[kUnrollInplace];
        char *kd[kUnrollInplace], *vd[kUnrollInplace];
#pragma unroll
        for (int r = 0; r < kUnrollInplace; ++r) {
            kd[r] = vd[r] = nullptr;
            const int64_t e = base + r * lanes + (int64_t)blockIdx.x * kThreads + threadIdx.x;
            if (e >= total_vec) continue;
            const int64_t row = e >> vshift;
            const int c = (int)(e & (vec_per_row - 1));
            int lo = 0, hi = U;                                       // unit whose rows contain `row`
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (tab[mid] <= row) lo = mid; else hi = mid;
            }
            const int u = lo, s = u / Hkv, g = u % Hkv;
            const int64_t off = tab[u];
            const int n = max(__ldg(seq_len + s), 0);
            const int64_t b64 = tab[u + 1] - off;
            const int t = (int)(row - off);
            if (off < 0 || b64 < 0 || b64 > n) { bad = true; continue; }
            const int b = (int)b64;
            const int head = min(b, min(p.sink, n));
            const int src = position_ranges ? (t < head ? t : n - b + t) : __ldg(kept_idx + row);
            if (src < t || src >= n) { bad = true; continue; }
            if (src == t) continue;                                   // already in place
            const int64_t tok0 = __ldg(seq_start + s);
            char *kb = k + ((int64_t)s * p.k_stride_seq + tok0 * p.k_stride_tok + (int64_t)g * p.k_stride_head) * esz + c * 16;
            char *vb = v + ((int64_t)s * p.v_stride_seq + tok0 * p.v_stride_tok + (int64_t)g * p.v_stride_head) * esz + c * 16;
            kv[r] = __ldcg(reinterpret_cast<const int4 *>(kb + (int64_t)src * k_tok));
            vv[r] = __ldcg(reinterpret_cast<const int4 *>(vb + (int64_t)src * v_tok));
            kd[r] = kb + (int64_t)t * k_tok;
            vd[r] = vb + (int64_t)t * v_tok;
        }
        grid.sync();
#pragma unroll
        for (int r = 0; r < kUnrollInplace; ++r) {
            if (kd[r]) {
                *reinterpret_cast<int4 *>(kd[r]) = kv[r];
                *reinterpret_cast<int4 *>(vd[r]) = vv[r];
            }
        }
    }
    if (bad && dev_status) atomicOr(dev_status, REFREE_DEV_CAPACITY);
}

// In place, anchored at the END of every unit's region (position ranking only): the kept set is
// the `head` leading rows plus the suffix [n - (b - head), n), so it is enough to lift the leading
// rows to just below the suffix; the compacted cache of the unit is then rows [n - b, n) of its
// own region.  At most `sink` rows move per unit.  The move is upwards and may overlap itself
// (n - b < head), so the rows go in blocks of 256 pieces from the top down, each block loaded by
// all threads before any of it is stored; a block's destinations lie above everything that the
// blocks after it still have to read.
__global__ void __launch_bounds__(kThreads)
compact_inplace_back_kernel(refree_params p, char *k, char *v, const int32_t *seq_start, const int32_t *seq_len,
                            const int64_t *offsets, const int32_t *lengths, int64_t *offsets_out, int32_t *dev_status)
{
    __shared__ long long s_part[kThreads / 32];
    const int Hkv = p.num_kv_heads;
    const int u = blockIdx.x, s = u / Hkv, g = u % Hkv;
    const int esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const int vec_per_row = (p.head_dim * esz) >> 4;
    const int vshift = 31 - __clz(vec_per_row);
    // Behind the selection of the same call everything but the budgets was complete before that began: tables and leading rows
    // are read while it drains (a thread has one piece of K and of V where they are few).
    if (!lengths) dependency_wait();
    const int n = max(seq_len[s], 0), lead = min(p.sink, n);
    const int64_t tok0 = seq_start[s];
    char *kb = k + ((int64_t)s * p.k_stride_seq + tok0 * p.k_stride_tok + (int64_t)g * p.k_stride_head) * esz;
    char *vb = v + ((int64_t)s * p.v_stride_seq + tok0 * p.v_stride_tok + (int64_t)g * p.v_stride_head) * esz;
    const int64_t k_tok = p.k_stride_tok * esz, v_tok = p.v_stride_tok * esz;
    const bool few = lead << vshift <= kThreads, mine = few && (int)threadIdx.x < lead << vshift;
    int4 kv = {}, vv = {};
    auto load = [&](int e) {
        const int row = e >> vshift, c = e & (vec_per_row - 1);
        kv = __ldcg(reinterpret_cast<const int4 *>(kb + (int64_t)row * k_tok + c * 16));
        vv = __ldcg(reinterpret_cast<const int4 *>(vb + (int64_t)row * v_tok + c * 16));
    };
    if (mine) load(threadIdx.x);
    if (lengths) dependency_wait();
    // (after the wait: blocks of the next call that came earlier would sit on SMs that the selection still needs; fp32 d 64, six
    // sequences of 80 to 641 positions x 8 heads 30.5 us, 27.3 this way)
    trigger_dependents();
    int64_t off, b64;
    if (lengths) {
        // fused pass: budgets come straight from the selection, and the running sum is formed here
        b64 = lengths[u];
        long long part = 0;
        for (int t = threadIdx.x; t < u; t += kThreads) part += lengths[t];
        for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
        __syncthreads();                             // (and the leading rows have been read)
        off = 0;
        for (int wv = 0; wv < kThreads / 32; ++wv) off += s_part[wv];
        if (threadIdx.x == 0) {
            offsets_out[u] = off;
            if (u == (int)gridDim.x - 1) offsets_out[u + 1] = off + b64;
        }
    } else {
        off = offsets[u];
        b64 = offsets[u + 1] - off;
        __syncthreads();
    }
    if (off < 0 || b64 < 0 || b64 > n) {
        if (threadIdx.x == 0 && dev_status) atomicOr(dev_status, REFREE_DEV_CAPACITY);
        return;
    }
    const int b = (int)b64, head = min(b, lead), shift = n - b;
    if (shift == 0 || head == 0) return;
    const int total_vec = head << vshift;
    auto store = [&](int e) {
        const int row = e >> vshift, c = e & (vec_per_row - 1);
        *reinterpret_cast<int4 *>(kb + (int64_t)(row + shift) * k_tok + c * 16) = kv;
        *reinterpret_cast<int4 *>(vb + (int64_t)(row + shift) * v_tok + c * 16) = vv;
    };
    if (few) {
        if ((int)threadIdx.x < total_vec) store(threadIdx.x);
        return;
    }
    for (int c0 = (total_vec - 1) / kThreads * kThreads; c0 >= 0; c0 -= kThreads) {
        const int e = c0 + threadIdx.x;
        if (e < total_vec) load(e);
        __syncthreads();
        if (e < total_vec) store(e);
    }
}

// Paged form of the same step: row t of unit u goes to row t % block_rows of the block
// block_table[u][t / block_rows] of a pool of fixed-size blocks (the layout of a paged
// serving cache).  Same gather as compact_kernel; only the destination address differs.
__global__ void __launch_bounds__(kThreads)
compact_paged_kernel(refree_params p, const char *k, const char *v, const int32_t *seq_start,
                     const int32_t *seq_len, const int32_t *lengths, const int64_t *offsets,
                     const int32_t *kept_idx, int position_ranges, const int32_t *block_table,
                     int max_blocks_per_unit, int block_rows, char *k_pool, char *v_pool, int64_t num_blocks,
                     int32_t *dev_status)
{
    const int Hkv = p.num_kv_heads;
    const int u = blockIdx.y, s = u / Hkv, g = u % Hkv;
    dependency_wait();
    trigger_dependents();
    const int esz = p.dtype == REFREE_DTYPE_F32 ? 4 : 2;
    const int row_bytes = p.head_dim * esz;
    const int vec_per_row = row_bytes >> 4;
    const int vshift = 31 - __clz(vec_per_row);
    const int n = max(seq_len[s], 0);
    const int b = lengths[u];
    if (b < 0 || b > n || (int64_t)b > (int64_t)max_blocks_per_unit * block_rows || (kept_idx && offsets[u] < 0)) {
        if (threadIdx.x == 0 && blockIdx.x == 0 && dev_status) atomicOr(dev_status, REFREE_DEV_CAPACITY);
        return;
    }
    const int head = min(b, min(p.sink, n));
    const int64_t tok0 = seq_start[s];
    const char *kb = k + ((int64_t)s * p.k_stride_seq + tok0 * p.k_stride_tok + (int64_t)g * p.k_stride_head) * esz;
    const char *vb = v + ((int64_t)s * p.v_stride_seq + tok0 * p.v_stride_tok + (int64_t)g * p.v_stride_head) * esz;
    const int64_t k_tok = p.k_stride_tok * esz, v_tok = p.v_stride_tok * esz;
    const int32_t *idx = kept_idx ? kept_idx + offsets[u] : nullptr;
    const int32_t *table = block_table + (int64_t)u * max_blocks_per_unit;
    const int64_t nvec = (int64_t)b << vshift;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    bool bad = false;
    for (int64_t e0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; e0 < nvec; e0 += stride * kUnroll) {
        int4 kv[kUnroll], vv[kUnroll];
        int64_t dst[kUnroll];
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            const int64_t e = e0 + r * stride;
            dst[r] = -1;
            if (e < nvec) {
                const int t = (int)(e >> vshift), c = (int)(e & (vec_per_row - 1));
                const int src = position_ranges ? (t < head ? t : n - b + t) : idx[t];
                const int blk = __ldg(table + t / block_rows);
                if (blk < 0 || blk >= num_blocks || src < 0 || src >= n) { bad = true; continue; }
                kv[r] = *reinterpret_cast<const int4 *>(kb + (int64_t)src * k_tok + c * 16);
                vv[r] = ld_stream(reinterpret_cast<const int4 *>(vb + (int64_t)src * v_tok + c * 16));
                dst[r] = ((int64_t)blk * block_rows + t % block_rows) * row_bytes + c * 16;
            }
        }
#pragma unroll
        for (int r = 0; r < kUnroll; ++r) {
            if (dst[r] >= 0) {
                st_stream(reinterpret_cast<int4 *>(k_pool + dst[r]), kv[r]);
                st_stream(reinterpret_cast<int4 *>(v_pool + dst[r]), vv[r]);
            }
        }
    }
    if (bad && dev_status) atomicOr(dev_status, REFREE_DEV_CAPACITY);
}

}  // namespace

// Whether a copy is launched behind the selection while that drains.  Its blocks then land on whichever SMs are free at
// that moment, and those of one long unit end up side by side: 2 us of launch latency saved, but 129 us against 105 for a
// copy of 250 MB out of a ragged batch (eight sequences of 92 to 19791 positions, 16 heads).  So only where the cache is
// small enough for the latency to count.
static int64_t cache_bytes(const refree_params &p, int layers)      // K and V; 0: the caller does not say
{
    const int64_t rows = layers * p.kv_tokens * p.num_kv_heads * (p.k_stride_seq != 0 ? p.num_seqs : 1);
    return rows * p.head_dim * (p.dtype == REFREE_DTYPE_F32 ? 8 : 4);
}
static Stream copy_stream(const refree_params &p, Stream st, int layers = 1)
{
    return Stream(st.s, st.chain && cache_bytes(p, layers) <= (int64_t)64 << 20);
}

cudaError_t launch_compact(const refree_params &p, const CompactJob &job, const int32_t *seq_start, const int32_t *seq_len,
                           bool position_ranges, int64_t capacity_rows, int32_t *dev_status, Stream st)
{
    const int U = p.num_seqs * p.num_kv_heads;
    const int ranges = position_ranges ? 1 : 0;
    // Two waves of blocks; four times as many for a large copy of several layers, or of three sequences and more, so that a
    // long unit among short ones is not left to one or two blocks (us: seven layers of twelve sequences of 83 to 15815
    // positions, 8 heads, 928 and 527; one layer of thirteen of 77 to 26835, 16 heads, 565 and 444 with its scoring; four
    // of eleven, ranked by score, 1089 and 1015; small copies would pay for the blocks, 18 and 25, and so would units of one
    // length, two of 16000 positions ranked by score 244 and 255).
    Stream cs = copy_stream(p, st, job.layers);
    const int per_sm = !cs.chain && (job.layers > 1 || p.num_seqs > 2) ? 32 : 8;
    int gx = max(1, (sm_count() * per_sm) / (U * job.layers));
    // Position ranges: no more blocks than the longest unit there can be has rows for, two pieces to a thread, four behind a launch
    // of the stopping rule; a block without rows waits, reads tables and budgets and holds the next launch up like the others.  And
    // a copy of up to 32 MB behind such a launch, which fills an SM's shared memory, asks for the same split of it: an SM changes
    // its split only when it is empty, so blocks that wait there for the rule to end kept the next call's scoring away.  (A layer
    // with its list, us, without either, with the first, with both: bf16 d 64, 600 positions x 2 heads 24.5, 17.5, 17.5, 2000 x 4
    // 34.7, 35.4, 31.2; fp32 d 128, 1500 x 2 31.0, 22.7, 22.4; of 46 MB, 2800 x 16, 59.9, 60.3, 61.7; 112 such calls on average 8.7 %
    // less.  Behind launches with little shared memory the split costs: a single query row, 20000 x 8 51.4 and 57.5; two pieces and
    // four there: 700 x 4 of it 9.9 and 10.6.  Ranked by score, where few rows are kept, fewer blocks gain nothing: bf16 d 64,
    // 1500 x 2 42.1 and 45.2.)
    if (position_ranges && p.kv_tokens > 0) {
        const int64_t pieces = std::min<int64_t>(p.kv_tokens, INT32_MAX) * p.head_dim * (p.dtype == REFREE_DTYPE_F32 ? 4 : 2) / 16;
        const int64_t per_block = (int64_t)kThreads * (job.after_rule ? 4 : 2);
        gx = (int)std::min<int64_t>(gx, (pieces + per_block - 1) / per_block);
    }
    if (job.after_rule && cs.chain && cache_bytes(p, job.layers) <= (int64_t)32 << 20) cs.carveout = 100;
    const cudaError_t e = launch_dependent(compact_kernel, dim3(gx, U, job.layers), dim3(kThreads), 0,
                                           cs, p, job, seq_start, seq_len, ranges, capacity_rows, dev_status);
    count_launches(1);
    return e;
}

cudaError_t launch_compact_inplace(const refree_params &p, void *k, void *v, const int32_t *seq_start,
                                   const int32_t *seq_len, const int64_t *offsets, const int32_t *kept_idx,
                                   bool position_ranges, bool anchor_back, int32_t *dev_status, Stream st,
                                   const int32_t *lengths, int64_t *offsets_out)
{
    if (anchor_back) {
        const cudaError_t e = launch_dependent(compact_inplace_back_kernel, dim3(p.num_seqs * p.num_kv_heads), dim3(kThreads), 0, st, p,
                                               (char *)k, (char *)v, seq_start, seq_len, offsets, lengths, offsets_out, dev_status);
        count_launches(1);
        return e;
    }
    static std::mutex grid_mutex;                 // the per-device grid size is looked up once, under a lock
    static int grid_blocks[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::unique_lock<std::mutex> hold(grid_mutex);
    if (grid_blocks[dev] == 0) {
        // every block of the grid must be resident at once: the rounds end in a grid-wide barrier
        int sms = 0, per_sm = 0, coop = 0;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
        if (!coop) return cudaErrorNotSupported;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, compact_inplace_kernel, kThreads, 0)) != cudaSuccess)
            return e;
        if (per_sm < 1) return cudaErrorLaunchOutOfResources;
        grid_blocks[dev] = sms * std::min(per_sm, 4);
    }
    const int grid = grid_blocks[dev];
    hold.unlock();
    refree_params pv = p;
    char *kc = (char *)k, *vc = (char *)v;
    int ranges = position_ranges ? 1 : 0;
    void *args[9] = {&pv, &kc, &vc, &seq_start, &seq_len, &offsets, &kept_idx, &ranges, &dev_status};
    e = cudaLaunchCooperativeKernel((const void *)compact_inplace_kernel, dim3(grid), dim3(kThreads), args, 0, st);
    if (e != cudaSuccess) return e;
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_compact_paged(const refree_params &p, const void *k, const void *v, const int32_t *seq_start,
                                 const int32_t *seq_len, const int32_t *lengths, const int64_t *offsets,
                                 const int32_t *kept_idx, bool position_ranges, const int32_t *block_table,
                                 int max_blocks_per_unit, int block_rows, void *k_pool, void *v_pool,
                                 int64_t num_blocks, int32_t *dev_status, Stream st)
{
    const int U = p.num_seqs * p.num_kv_heads;
    const int gx = max(1, (sm_count() * 8) / U);
    const cudaError_t e = launch_dependent(compact_paged_kernel, dim3(gx, U), dim3(kThreads), 0, copy_stream(p, st), p, (const char *)k, (const char *)v,
                                           seq_start, seq_len, lengths, offsets, kept_idx, position_ranges ? 1 : 0, block_table,
                                           max_blocks_per_unit, block_rows, (char *)k_pool, (char *)v_pool, num_blocks, dev_status);
    count_launches(1);
    return e;
}

}  // namespace refree
