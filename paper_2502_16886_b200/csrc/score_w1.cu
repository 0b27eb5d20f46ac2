// Scoring for the paper's default reduced attention, w = 1 (Section 3.2 "Reducing
// Overhead", k = 1; Algorithm 1 uses Q[..., -1, :]): one query per head, so the
// logits are G numbers per position and the step is a pure stream over K.
//
//   logits  y[h][i] = (q_h . k_i / sqrt(d)) * log2(e) for the G heads of the KV head.
//           bf16: a warp owns a span of positions of one unit; 16 rows x d of K go from
//           global memory straight into the A fragments of mma.m16n8k16 (16 bytes per lane,
//           the four lanes of a row 64 contiguous bytes per instruction), the queries
//           sit in the B fragments, loaded the same way so the element order inside a
//           k-step cancels.  The tensor-core instruction is used as a dot-product unit
//           (it replaces ~50 fp32 instructions per row); the kernel is bound by the K stream.
//           fp32 (or unaligned queries): lane groups per row on the fp32 pipes, shuffle-reduced.
//           y goes to the workspace (4 G bytes per position against 256 for the K row),
//           with one (max, sum 2^(y - max)) record per head and span
//   scores  L_h = log2 sum_i 2^(y_h[i]) from the span records, then
//           a'[i] = (1/G) sum_h 2^(y_h[i] - L_h)   (Eq. 2 with one row: cnt = 1)
//
// Short calls take one kernel instead (w1_unit_kernel): a cluster of blocks per unit keeps the logits in shared memory and
// goes from K to the budget in one launch.
//
// K is read once (intensity G flop/B, far below the ridge).
#include <cooperative_groups.h>

#include <algorithm>

#include "refree_internal.cuh"
#include "select_groups.cuh"

namespace refree {
namespace {

namespace cg = cooperative_groups;

constexpr int kThreadsW1 = 256;
constexpr int kChunk = 256;          // positions per block iteration
constexpr int kMaxG = 16;
constexpr int kMinSpan = 32;         // positions per (max, sum) record of the mma path: a multiple of 16
constexpr int kMaxSpan = 512;
constexpr float kLog2eW1 = 1.4426950408889634f;

struct W1Tables {
    int32_t pack[kMaxSeqs + 1];
    int32_t chunks[kMaxSeqs + 1];    // 256-position chunks before sequence s
    int32_t spans[kMaxSeqs + 1];     // spans (the unit of the (max, sum) records) before sequence s
    int32_t tiles[kMaxSeqs + 1];     // 128-position tiles before sequence s (index of the GroupPartial records)
    int32_t len[kMaxSeqs];
};

// By the first warp, 32 sequences at a time (a thread walking them would wait for each length in turn).
__device__ inline void build_w1_tables(W1Tables &t, const int32_t *seq_len, int B, int span)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int a = 0, b = 0, c = 0, e = 0;
        for (int s0 = 0; s0 < B; s0 += 32) {
            const int s = s0 + lane, n = s < B ? max(seq_len[s], 0) : 0;
            const int nb = ceil_div(n, kChunk), nc = ceil_div(n, kTile), ne = ceil_div(n, span);
            const int ai = warp_incl_scan(n), bi = warp_incl_scan(nb), ci = warp_incl_scan(nc), ei = warp_incl_scan(ne);
            if (s < B) {
                t.pack[s] = a + ai - n; t.chunks[s] = b + bi - nb; t.tiles[s] = c + ci - nc; t.spans[s] = e + ei - ne;
                t.len[s] = n;
            }
            a += __shfl_sync(0xffffffffu, ai, 31); b += __shfl_sync(0xffffffffu, bi, 31);
            c += __shfl_sync(0xffffffffu, ci, 31); e += __shfl_sync(0xffffffffu, ei, 31);
        }
        if (lane == 0) { t.pack[B] = a; t.chunks[B] = b; t.tiles[B] = c; t.spans[B] = e; }
    }
    __syncthreads();
}

struct W1Item { int s, g, chunk, n, pos0; };

// items ordered (sequence, head, piece); `before` counts the pieces (chunks or spans) ahead of a sequence
__device__ inline W1Item decode_w1(const W1Tables &t, const int32_t *before, int piece_len, int B, int Hkv, int item)
{
    int lo = 0, hi = B;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((int64_t)before[mid] * Hkv <= item) lo = mid; else hi = mid;
    }
    W1Item it;
    it.s = lo;
    const int cs = before[lo + 1] - before[lo];
    const int rem = item - before[lo] * Hkv;
    it.g = rem / cs;
    it.chunk = rem % cs;
    it.n = t.len[lo];
    it.pos0 = it.chunk * piece_len;
    return it;
}

__device__ inline float ex2(float x)
{
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// (max, sum) records combine as m = max, z = z1 2^(m1 - m) + z2 2^(m2 - m)
__device__ inline void merge_stats(float &m, float &z, float mo, float zo)
{
    const float mn = fmaxf(m, mo);
    z = mn == -INFINITY ? 0.f : z * ex2(m - mn) + zo * ex2(mo - mn);
    m = mn;
}

template <typename T> struct Row16;                       // 16 bytes of a K row as floats
template <> struct Row16<__nv_bfloat16> {
    static constexpr int kElems = 8;
    __device__ static void load(const void *p, float (&f)[8])
    {
        const uint4 r = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            f[2 * i] = __uint_as_float(w[i] << 16);
            f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
};
template <> struct Row16<float> {
    static constexpr int kElems = 4;
    __device__ static void load(const void *p, float (&f)[8])
    {
        const float4 r = *reinterpret_cast<const float4 *>(p);
        f[0] = r.x; f[1] = r.y; f[2] = r.z; f[3] = r.w;
    }
};

// The layers of a group, one to a grid row; what a layer keeps follows that of the layer before.
struct W1Args {
    refree_params p;
    int layers;
    const void *q_win[kMaxBatch], *k[kMaxBatch];
    int64_t layer_logits, layer_stats, layer_groups;        // elements per layer (scores: Hkv total_tokens)
    const int32_t *seq_start, *seq_len;
    float *logits;          // [Hq][total_tokens]
    float2 *stats;          // [spans_total * Hkv][G]: (max, sum) per span and head
    int span;               // positions per record
    GroupPartial *groups;   // nullable
    float *scores;
    int64_t total_tokens;
    int32_t *dev_status;
    // w1_unit_kernel: budgets and records (nullable)
    int32_t *sel_lengths[kMaxBatch];
    Cut *sel_cuts;
};

// A K row is covered by LPR = row_bytes / 16 lanes, 16 bytes each, so a warp reads
// 32 / LPR whole rows per load instruction (fully coalesced).  Each lane keeps its
// slice of the G queries in registers; the partial dot products meet by shuffles.
template <typename T, int D, int GMAX>
__global__ void __launch_bounds__(kThreadsW1)
w1_logits_kernel(const __grid_constant__ W1Args a)
{
    constexpr int E = Row16<T>::kElems;              // elements per lane and row
    constexpr int LPR = D / E;                       // lanes per row: 8, 16 or 32
    constexpr int RPW = 32 / LPR;                    // rows per warp and load
    constexpr int kWarpsW1 = kThreadsW1 / 32;
    constexpr int kRowsPerWarp = kChunk / kWarpsW1;  // 32 positions of the chunk per warp
    __shared__ W1Tables tb;
    __shared__ float2 red[kWarpsW1 * RPW][GMAX];
    const refree_params &p = a.p;
    const int layer = blockIdx.y;
    const T *const q_win = static_cast<const T *>(a.q_win[layer]), *const k = static_cast<const T *>(a.k[layer]);
    float *const logits = a.logits + layer * a.layer_logits;
    float2 *const stats = a.stats + layer * a.layer_stats;
    const int B = p.num_seqs, Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / LPR, part = lane % LPR;   // row of the load this lane helps with, its 16-byte slice
    const float scale = kLog2eW1 * rsqrtf((float)D);
    dependency_wait();
    trigger_dependents();
    build_w1_tables(tb, a.seq_len, B, kChunk);      // one record per block chunk: span == kChunk
    const int items = tb.chunks[B] * Hkv;
    int cur_u = -1;
    float qreg[GMAX][E];
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const W1Item it = decode_w1(tb, tb.chunks, kChunk, B, Hkv, item);
        const int u = it.s * Hkv + it.g;
        if (u != cur_u) {                            // this lane's slice of the unit's G queries, pre-scaled
#pragma unroll
            for (int h = 0; h < GMAX; ++h)
#pragma unroll
                for (int e = 0; e < E; ++e)
                    qreg[h][e] = h < G ? to_float(q_win[((int64_t)it.s * p.num_q_heads + it.g * G + h) * D + part * E + e]) * scale
                                       : 0.f;
            cur_u = u;
        }
        const char *base = reinterpret_cast<const char *>(
            k + (int64_t)it.s * p.k_stride_seq + (int64_t)a.seq_start[it.s] * p.k_stride_tok + (int64_t)it.g * p.k_stride_head);
        const int64_t tok_bytes = p.k_stride_tok * (int64_t)sizeof(T);
        // after the butterfly every lane of a row group holds all G logits of the row: lane l of the
        // group takes heads l, l + LPR, ... (one store and one running (max, sum) update per head)
        constexpr int HPL = (GMAX + LPR - 1) / LPR;
        float m[HPL], z[HPL];
#pragma unroll
        for (int j = 0; j < HPL; ++j) { m[j] = -INFINITY; z[j] = 0.f; }
        float *unit_logits = logits + (int64_t)(it.g * G) * a.total_tokens + tb.pack[it.s];
        const int wpos0 = it.pos0 + warp * kRowsPerWarp;
#pragma unroll 4
        for (int r = 0; r < kRowsPerWarp; r += RPW) {
            const int i = wpos0 + r + sub;
            const bool valid = i < it.n;
            float kf[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) kf[e] = 0.f;
            if (valid) Row16<T>::load(base + (int64_t)i * tok_bytes + part * 16, kf);
            float y[GMAX];
#pragma unroll
            for (int h = 0; h < GMAX; ++h) {
                float acc = 0.f;
#pragma unroll
                for (int e = 0; e < E; ++e) acc = fmaf(kf[e], qreg[h][e], acc);
                y[h] = acc;
            }
#pragma unroll
            for (int o = LPR / 2; o; o >>= 1)
#pragma unroll
                for (int h = 0; h < GMAX; ++h)
                    if (h < G) y[h] += __shfl_xor_sync(0xffffffffu, y[h], o);
#pragma unroll
            for (int j = 0; j < HPL; ++j) {
                float mine = 0.f;
#pragma unroll
                for (int h = j * LPR; h < GMAX && h < (j + 1) * LPR; ++h) mine = (part == h - j * LPR) ? y[h] : mine;
                const int head = part + j * LPR;
                if (head < G && valid) {
                    unit_logits[(int64_t)head * a.total_tokens + i] = mine;
                    merge_stats(m[j], z[j], mine, 1.f);
                }
            }
        }
        // block (max, sum) per head: the RPW row groups of every warp, in a fixed order
#pragma unroll
        for (int j = 0; j < HPL; ++j)
            if (part + j * LPR < GMAX) red[warp * RPW + sub][part + j * LPR] = make_float2(m[j], z[j]);
        __syncthreads();
        if (threadIdx.x < G) {
            float mm = -INFINITY, zz = 0.f;
            for (int wv = 0; wv < kWarpsW1 * RPW; ++wv) merge_stats(mm, zz, red[wv][threadIdx.x].x, red[wv][threadIdx.x].y);
            stats[((int64_t)(tb.chunks[it.s] * Hkv) + (int64_t)it.g * (tb.chunks[it.s + 1] - tb.chunks[it.s]) +
                     it.chunk) * G + threadIdx.x] = make_float2(mm, zz);
        }
        __syncthreads();
    }
}

__device__ inline void mma_bf16_16x8x16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ inline uint4 ld_row16(const char *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// bf16 logits on mma.m16n8k16.  Lane (r, c) = (lane / 4, lane % 4) of a warp loads, for rows r and
// r + 8 of a 16-row block, the 16-byte pieces at byte 64 j + 16 c of the row (the four lanes of a
// row read two whole 32-byte sectors per instruction); the four 32-bit words of a piece feed two
// k-steps as (a0, a2) resp. (a1, a3).  The B operand
// is the query of head r (and r + 8 for the second column tile) cut the same way, so every product
// pairs the same element of k_i and q_h whatever slot of the k-step it occupies.  The accumulator
// of lane (r, c) holds heads 2c, 2c + 1 for rows r and r + 8.  NT column tiles cover G <= 8 NT heads.
// Bound by the stream over K.  The warps of one wave of blocks walk the spans of all layers of the group, and a warp asks for
// the next 16 rows (of its next span too) before it works on those it has: a block per layer and piece of the grid, with the
// rows of a step loaded and used in turn, kept HBM at 4.8 TB/s (eight layers of 32K positions x 8 heads, 107 us).
// AHEAD: the loads ahead.  Not with two column tiles of 128-element rows, whose registers they overflow (124 bytes of spills
// inside the stream; two layers of 16000 and 15000 positions x 2 heads, groups of 16, 85.6 us with, 81.8 without).
template <int D, int NT, bool AHEAD>
__global__ void __launch_bounds__(kThreadsW1, 2)
w1_logits_mma_kernel(const __grid_constant__ W1Args a)
{
    constexpr int CH = D / 32;                       // 16-byte pieces per lane and row
    constexpr int kWarpsW1 = kThreadsW1 / 32;
    __shared__ W1Tables tb;
    const refree_params &p = a.p;
    const int B = p.num_seqs, Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 2, c = lane & 3;
    const float scale = kLog2eW1 * rsqrtf((float)D);
    dependency_wait();
    trigger_dependents();
    build_w1_tables(tb, a.seq_len, B, a.span);
    const int per_layer = tb.spans[B] * Hkv;
    const int64_t items = (int64_t)per_layer * a.layers, step = (int64_t)gridDim.x * kWarpsW1;
    const int64_t tok_bytes = p.k_stride_tok * (int64_t)sizeof(__nv_bfloat16);
    // a span of a layer: what it reads
    struct Span { W1Item it; int layer, end; const char *base; };
    auto span_of = [&](int64_t item) {
        Span sp;
        sp.layer = a.layers > 1 ? (int)(item / per_layer) : 0;
        sp.it = decode_w1(tb, tb.spans, a.span, B, Hkv, (int)(item - (int64_t)sp.layer * per_layer));
        sp.end = min(sp.it.n, sp.it.pos0 + a.span);
        sp.base = static_cast<const char *>(a.k[sp.layer]) +
                  ((int64_t)sp.it.s * p.k_stride_seq + (int64_t)a.seq_start[sp.it.s] * p.k_stride_tok + (int64_t)sp.it.g * p.k_stride_head) * 2;
        return sp;
    };
    uint4 ka[CH], kb[CH];
    auto load = [&](const Span &sp, int row0) {      // rows row0 + r and row0 + 8 + r; missing ones are zero
        const int i0 = row0 + r, i1 = i0 + 8;
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const int off = j * 64 + c * 16;
            ka[j] = i0 < sp.end ? ld_row16(sp.base + (int64_t)i0 * tok_bytes + off) : make_uint4(0u, 0u, 0u, 0u);
            kb[j] = i1 < sp.end ? ld_row16(sp.base + (int64_t)i1 * tok_bytes + off) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    int64_t item = (int64_t)blockIdx.x * kWarpsW1 + warp;
    if (item >= items) return;
    Span sp = span_of(item);
    if (AHEAD) load(sp, sp.it.pos0);
    int cur_u = -1;
    uint4 qf[NT][CH];
    for (;;) {
        const W1Item it = sp.it;
        const int layer = sp.layer, end = sp.end;
        float *const logits = a.logits + layer * a.layer_logits;
        float2 *const stats = a.stats + layer * a.layer_stats;
        const int u = (layer * B + it.s) * Hkv + it.g;
        if (u != cur_u) {
            const char *const q_win = static_cast<const char *>(a.q_win[layer]);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const int head = t * 8 + r;
                const char *qrow = q_win + ((int64_t)it.s * p.num_q_heads + it.g * G + min(head, G - 1)) * D * 2;
#pragma unroll
                for (int j = 0; j < CH; ++j) {
                    qf[t][j] = *reinterpret_cast<const uint4 *>(qrow + j * 64 + c * 16);
                    if (head >= G) qf[t][j] = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            cur_u = u;
        }
        float *unit_logits = logits + (int64_t)(it.g * G) * a.total_tokens + tb.pack[it.s];
        item += step;
        const bool more = item < items;
        if (AHEAD && more) sp = span_of(item);       // the next span: its first rows are asked for under this one's last
        float m[NT][2], z[NT][2];
#pragma unroll
        for (int t = 0; t < NT; ++t) { m[t][0] = m[t][1] = -INFINITY; z[t][0] = z[t][1] = 0.f; }
        const char *const base = static_cast<const char *>(a.k[layer]) +
                                 ((int64_t)it.s * p.k_stride_seq + (int64_t)a.seq_start[it.s] * p.k_stride_tok + (int64_t)it.g * p.k_stride_head) * 2;
        const Span cur = {it, layer, end, base};
#pragma unroll(AHEAD ? 1 : 2)
        for (int row0 = it.pos0; row0 < end; row0 += 16) {
            const int i0 = row0 + r, i1 = i0 + 8;
            const bool v0 = i0 < end, v1 = i1 < end;
            uint4 xa[CH], xb[CH];
            if (!AHEAD) load(cur, row0);
#pragma unroll
            for (int j = 0; j < CH; ++j) { xa[j] = ka[j]; xb[j] = kb[j]; }
            if (AHEAD) {
                if (row0 + 16 < end) load(cur, row0 + 16);
                else if (more) load(sp, sp.it.pos0);
            }
            float acc[NT][4];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll
                for (int j = 0; j < CH; ++j) {
                    mma_bf16_16x8x16(acc[t], xa[j].x, xb[j].x, xa[j].y, xb[j].y, qf[t][j].x, qf[t][j].y);
                    mma_bf16_16x8x16(acc[t], xa[j].z, xb[j].z, xa[j].w, xb[j].w, qf[t][j].z, qf[t][j].w);
                }
            }
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int head = t * 8 + 2 * c + e;
                    if (head < G) {
                        const float y0 = acc[t][e] * scale, y1 = acc[t][2 + e] * scale;
                        float *dst = unit_logits + (int64_t)head * a.total_tokens;
                        if (v0) dst[i0] = y0;
                        if (v1) dst[i1] = y1;
                        const float ym = fmaxf(v0 ? y0 : -INFINITY, v1 ? y1 : -INFINITY);
                        if (ym > -INFINITY) {
                            const float mn = fmaxf(m[t][e], ym);
                            z[t][e] = z[t][e] * ex2(m[t][e] - mn) + (v0 ? ex2(y0 - mn) : 0.f) + (v1 ? ex2(y1 - mn) : 0.f);
                            m[t][e] = mn;
                        }
                    }
                }
        }
        // one record per head and span: the eight row lanes of a column pair combine in a fixed order
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    const float mo = __shfl_xor_sync(0xffffffffu, m[t][e], o);
                    const float zo = __shfl_xor_sync(0xffffffffu, z[t][e], o);
                    merge_stats(m[t][e], z[t][e], mo, zo);
                }
                const int head = t * 8 + 2 * c + e;
                if (r == 0 && head < G)
                    stats[((int64_t)tb.spans[it.s] * Hkv + (int64_t)it.g * (tb.spans[it.s + 1] - tb.spans[it.s]) +
                             it.chunk) * G + head] = make_float2(m[t][e], z[t][e]);
            }
        if (!more) break;
        if (!AHEAD) sp = span_of(item);
    }
}

// A unit from K to its budget in one cluster of blocks, the logits in shared memory (bf16, same products as
// w1_logits_mma_kernel).  Bound by latency: the two kernels above are some twenty dependent round trips to memory, half
// of them between the kernels; here the blocks meet twice, in distributed shared memory.
constexpr int kThreadsUnit = 256;
constexpr int kMaxClusterW1 = 8;
constexpr int64_t kUnitTokens = 8192;        // see launch_score_w1

template <int D, int NT>
__global__ void __launch_bounds__(kThreadsUnit)
w1_unit_kernel(const __grid_constant__ W1Args a, int stride)
{
    constexpr int CH = D / 32;                       // 16-byte pieces per lane and row
    constexpr int kWarpsUnit = kThreadsUnit / 32;
    extern __shared__ float ylog[];                  // [G][stride], this block's positions
    __shared__ float2 red[kWarpsUnit][8 * NT];
    __shared__ float lse[8 * NT];
    __shared__ BlockRuleShared<kThreadsUnit> rule;
    __shared__ uint32_t wmax[kWarpsUnit], cmax[kMaxClusterW1];
    __shared__ float2 cstat[8 * NT];
    cg::cluster_group cl = cg::this_cluster();
    const int nblk = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const refree_params &p = a.p;
    const int layer = blockIdx.y;
    const __nv_bfloat16 *const q_win = static_cast<const __nv_bfloat16 *>(a.q_win[layer]), *const k = static_cast<const __nv_bfloat16 *>(a.k[layer]);
    GroupPartial *const groups = a.groups ? a.groups + layer * a.layer_groups : nullptr;
    float *const scores = a.scores + (int64_t)layer * p.num_kv_heads * a.total_tokens;
    const int Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int u = blockIdx.x / nblk, s = u / Hkv, g = u - s * Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 2, c = lane & 3;
    const float scale = kLog2eW1 * rsqrtf((float)D);
    dependency_wait();
    trigger_dependents();
    int pack = 0, tiles = 0;                         // positions and tiles of the sequences before this one
    for (int s0 = 0; s0 < s; s0 += 32) {
        const int nn = s0 + lane < s ? max(a.seq_len[s0 + lane], 0) : 0;
        pack += __reduce_add_sync(0xffffffffu, nn);
        tiles += __reduce_add_sync(0xffffffffu, ceil_div(nn, kTile));
    }
    const int n = max(a.seq_len[s], 0);
    if (n == 0) {                                    // keeps nothing (the whole cluster leaves)
        if (rank == 0 && threadIdx.x == 0 && a.sel_cuts) {
            Cut cut;
            cut.b = 0; cut.ties = 0; cut.tau = 0; cut.prot_kept = 0; cut.sbias = 0;
            a.sel_lengths[layer][u] = 0;
            a.sel_cuts[layer * p.num_seqs * Hkv + u] = cut;
        }
        return;
    }
    const int per = ceil_div(n, 32 * nblk) * 32;     // positions [first, end) are this block's
    const int first = rank * per, end = min(n, first + per);
    uint4 qf[NT][CH];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const int head = t * 8 + r;
        const char *qrow = reinterpret_cast<const char *>(q_win + ((int64_t)s * p.num_q_heads + g * G + min(head, G - 1)) * D);
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            qf[t][j] = *reinterpret_cast<const uint4 *>(qrow + j * 64 + c * 16);
            if (head >= G) qf[t][j] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    const char *base = reinterpret_cast<const char *>(
        k + (int64_t)s * p.k_stride_seq + (int64_t)a.seq_start[s] * p.k_stride_tok + (int64_t)g * p.k_stride_head);
    const int64_t tok_bytes = p.k_stride_tok * (int64_t)sizeof(__nv_bfloat16);
    float m[NT][2], z[NT][2];
#pragma unroll
    for (int t = 0; t < NT; ++t) { m[t][0] = m[t][1] = -INFINITY; z[t][0] = z[t][1] = 0.f; }
#pragma unroll 2
    for (int row0 = first + warp * 16; row0 < end; row0 += kWarpsUnit * 16) {
        const int i0 = row0 + r, i1 = i0 + 8;
        const bool v0 = i0 < end, v1 = i1 < end;
        uint4 ka[CH], kb[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            const int off = j * 64 + c * 16;
            ka[j] = v0 ? ld_row16(base + (int64_t)i0 * tok_bytes + off) : make_uint4(0u, 0u, 0u, 0u);
            kb[j] = v1 ? ld_row16(base + (int64_t)i1 * tok_bytes + off) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < CH; ++j) {
                mma_bf16_16x8x16(acc, ka[j].x, kb[j].x, ka[j].y, kb[j].y, qf[t][j].x, qf[t][j].y);
                mma_bf16_16x8x16(acc, ka[j].z, kb[j].z, ka[j].w, kb[j].w, qf[t][j].z, qf[t][j].w);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int head = t * 8 + 2 * c + e;
                if (head < G) {
                    const float y0 = acc[e] * scale, y1 = acc[2 + e] * scale;
                    if (v0) ylog[head * stride + i0 - first] = y0;
                    if (v1) ylog[head * stride + i1 - first] = y1;
                    const float ym = fmaxf(v0 ? y0 : -INFINITY, v1 ? y1 : -INFINITY);
                    if (ym > -INFINITY) {
                        const float mn = fmaxf(m[t][e], ym);
                        z[t][e] = z[t][e] * ex2(m[t][e] - mn) + (v0 ? ex2(y0 - mn) : 0.f) + (v1 ? ex2(y1 - mn) : 0.f);
                        m[t][e] = mn;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                const float mo = __shfl_xor_sync(0xffffffffu, m[t][e], o);
                const float zo = __shfl_xor_sync(0xffffffffu, z[t][e], o);
                merge_stats(m[t][e], z[t][e], mo, zo);
            }
            if (r == 0) red[warp][t * 8 + 2 * c + e] = make_float2(m[t][e], z[t][e]);
        }
    __syncthreads();
    for (int h = warp; h < G; h += kWarpsUnit) {     // the block's (max, sum) per head
        float mm = -INFINITY, zz = 0.f;
        if (lane < kWarpsUnit) { const float2 x = red[lane][h]; mm = x.x; zz = x.y; }
#pragma unroll
        for (int o = 1; o < kWarpsUnit; o <<= 1) {
            const float mo = __shfl_xor_sync(0xffffffffu, mm, o);
            const float zo = __shfl_xor_sync(0xffffffffu, zz, o);
            merge_stats(mm, zz, mo, zo);
        }
        if (lane == 0) cstat[h] = make_float2(mm, zz);
    }
    cl.sync();
    for (int h = warp; h < G; h += kWarpsUnit) {     // L_h = log2 sum_i 2^(y_h[i]), the same bits in every block
        float mm = -INFINITY, zz = 0.f;
        if (lane < nblk) { const float2 x = *cl.map_shared_rank(&cstat[h], lane); mm = x.x; zz = x.y; }
#pragma unroll
        for (int o = 1; o < kMaxClusterW1; o <<= 1) {
            const float mo = __shfl_xor_sync(0xffffffffu, mm, o);
            const float zo = __shfl_xor_sync(0xffffffffu, zz, o);
            merge_stats(mm, zz, mo, zo);
        }
        if (lane == 0) lse[h] = mm + log2f(zz);
    }
    __syncthreads();
    float *sc_out = scores + (int64_t)g * a.total_tokens + pack;
    GroupPartial *grp = groups ? groups + ((int64_t)tiles * Hkv + (int64_t)g * ceil_div(n, kTile)) * 4 : nullptr;
    uint32_t run_max = 0;
    for (int i0 = first + warp * 32; i0 < end; i0 += kThreadsUnit) {
        const int i = i0 + lane;
        const bool valid = i < n;
        float sc = 0.f;
        if (valid) {
            float tot = 0.f;
            for (int h = 0; h < G; ++h) tot += ex2(ylog[h * stride + i - first] - lse[h]);
            sc = tot / (float)G;
            if (!isfinite(sc) && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_NONFINITE);
            sc_out[i] = sc;
        }
        if (grp) {                                   // exact sum of squares of these 32 positions
            const uint32_t bits = (valid && isfinite(sc)) ? mag_bits(sc) : 0u;
            const uint32_t mx = __reduce_max_sync(0xffffffffu, bits);
            unsigned long long sq = sq_fixed(bits, kGroupShift - 2 * max(1, (int)(mx >> 23)));
#pragma unroll
            for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0) { GroupPartial gp; gp.max_bits = mx; gp.pad = 0u; gp.sum = sq; grp[i0 >> 5] = gp; }
            run_max = max(run_max, mx);
        }
    }
    if (lane == 0) wmax[warp] = run_max;
    __syncthreads();
    if (threadIdx.x == 0) {                          // the block's largest score goes to the first block
        uint32_t mx = 0;
        for (int wv = 0; wv < kWarpsUnit; ++wv) mx = max(mx, wmax[wv]);
        *cl.map_shared_rank(&cmax[rank], 0) = mx;
    }
    __threadfence();
    cl.sync();                                       // scores and records of the cluster are visible to the first block
    if (rank != 0 || !a.sel_cuts) return;
    uint32_t unit_max = 0;
    for (int b = 0; b < nblk; ++b) unit_max = max(unit_max, cmax[b]);
    const UnitRule ur(p, sc_out, n, grp, unit_max);
    block_unit_rule<kThreadsUnit>(ur, rule, a.sel_lengths[layer] + u, a.sel_cuts + layer * p.num_seqs * Hkv + u);
}

// kAhead chunks of a block have their logits in flight together.
template <int GMAX, int kAhead>
__global__ void __launch_bounds__(kThreadsW1, GMAX > 8 ? 2 : GMAX <= 4 && kAhead == 1 ? 5 : 4)
w1_scores_kernel(const __grid_constant__ W1Args a)
{
    constexpr int kWarpsW1 = kThreadsW1 / 32;
    __shared__ W1Tables tb;
    __shared__ float2 red[kWarpsW1][GMAX];
    __shared__ float lse[GMAX];
    const refree_params &p = a.p;
    const int layer = blockIdx.y;
    float *const logits = a.logits + layer * a.layer_logits;
    float2 *const stats = a.stats + layer * a.layer_stats;
    GroupPartial *const groups = a.groups ? a.groups + layer * a.layer_groups : nullptr;
    float *const scores = a.scores + (int64_t)layer * p.num_kv_heads * a.total_tokens;
    const int B = p.num_seqs, Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    trigger_dependents();
    build_w1_tables(tb, a.seq_len, B, a.span);
    dependency_wait();
    const int items = tb.chunks[B] * Hkv;
    // a block takes consecutive chunks, so it stays inside one unit as long as it can
    const int per = ceil_div(items, (int)gridDim.x);
    const int first = blockIdx.x * per, last = min(items, first + per);
    int cur_u = -1;
    for (int item = first; item < last;) {
        const W1Item it = decode_w1(tb, tb.chunks, kChunk, B, Hkv, item);
        const int u = it.s * Hkv + it.g;
        if (u != cur_u) {
            // L_h = log2 sum_i 2^(y_h[i]) from the unit's span records, combined in a fixed order
            const int cs = tb.spans[it.s + 1] - tb.spans[it.s];
            const float2 *st = stats + ((int64_t)tb.spans[it.s] * Hkv + (int64_t)it.g * cs) * G;
            float m[GMAX], z[GMAX];
#pragma unroll
            for (int h = 0; h < GMAX; ++h) { m[h] = -INFINITY; z[h] = 0.f; }
            for (int c = threadIdx.x; c < cs; c += kThreadsW1)
#pragma unroll
                for (int h = 0; h < GMAX; ++h)
                    if (h < G) { const float2 pr = st[(int64_t)c * G + h]; merge_stats(m[h], z[h], pr.x, pr.y); }
#pragma unroll
            for (int h = 0; h < GMAX; ++h)
                if (h < G) {
#pragma unroll
                    for (int o = 16; o; o >>= 1) {
                        const float mo = __shfl_xor_sync(0xffffffffu, m[h], o);
                        const float zo = __shfl_xor_sync(0xffffffffu, z[h], o);
                        merge_stats(m[h], z[h], mo, zo);
                    }
                    if (lane == 0) red[warp][h] = make_float2(m[h], z[h]);
                }
            __syncthreads();
            if (threadIdx.x < G) {
                float mm = -INFINITY, zz = 0.f;
                for (int wv = 0; wv < kWarpsW1; ++wv) merge_stats(mm, zz, red[wv][threadIdx.x].x, red[wv][threadIdx.x].y);
                lse[threadIdx.x] = mm + log2f(zz);
            }
            cur_u = u;
            __syncthreads();
        }
        // the run of this block's chunks inside the unit, kAhead of them at a time: their logits are in flight together
        const int run = min(last - item, ceil_div(it.n, kChunk) - it.chunk);
        const float *const y = logits + (int64_t)(it.g * G) * a.total_tokens + tb.pack[it.s];
        float *const dst = scores + (int64_t)it.g * a.total_tokens + tb.pack[it.s];
        GroupPartial *const grp = groups ? groups + ((int64_t)tb.tiles[it.s] * Hkv + (int64_t)it.g * ceil_div(it.n, kTile)) * 4 : nullptr;
        for (int j0 = 0; j0 < run; j0 += kAhead) {
            float yl[kAhead][GMAX];
            if constexpr (kAhead > 1) {
#pragma unroll
                for (int j = 0; j < kAhead; ++j) {
                    const int i = it.pos0 + (j0 + j) * kChunk + threadIdx.x;
#pragma unroll
                    for (int h = 0; h < GMAX; ++h)
                        if (h < G) yl[j][h] = j0 + j < run && i < it.n ? y[(int64_t)h * a.total_tokens + i] : 0.f;
                }
            }
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
                if (j0 + j >= run) continue;
                const int pos0 = it.pos0 + (j0 + j) * kChunk, i = pos0 + threadIdx.x;
                const bool valid = i < it.n;
                float sc = 0.f;
                if (valid) {
                    float tot = 0.f;
                    if constexpr (kAhead > 1) {
#pragma unroll
                        for (int h = 0; h < GMAX; ++h)
                            if (h < G) tot += ex2(yl[j][h] - lse[h]);
                    } else {
                        for (int h = 0; h < G; ++h) tot += ex2(y[(int64_t)h * a.total_tokens + i] - lse[h]);
                    }
                    sc = tot / (float)G;
                    if (!isfinite(sc) && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_NONFINITE);
                    dst[i] = sc;
                }
                if (grp) {                            // exact sum of squares of this warp's 32 positions
                    const uint32_t bits = (valid && isfinite(sc)) ? mag_bits(sc) : 0u;
                    const uint32_t mx = __reduce_max_sync(0xffffffffu, bits);
                    unsigned long long sq = sq_fixed(bits, kGroupShift - 2 * max(1, (int)(mx >> 23)));
                    for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                    const int q = (pos0 >> 5) + warp;
                    if (lane == 0 && q * 32 < ceil_div(it.n, kTile) * kTile) {
                        GroupPartial gp; gp.max_bits = mx; gp.pad = 0u; gp.sum = sq;
                        grp[q] = gp;
                    }
                }
            }
        }
        item += run;
    }
}


template <int GMAX>
cudaError_t run_w1_scores(W1Args &a, int layers, int64_t chunk_items, Stream st)
{
    // One wave of blocks over all layers: a block reads the unit's records (some 300 per head) before its first chunk.  (A grid
    // of four blocks an SM for every layer: 55 us for eight layers of 32K positions, 12 this way; of four blocks of 16 heads, two of
    // which an SM holds: four layers of 32K positions x 2 heads 176 us with the rest of the run, 136 this way.)
    constexpr int kPerSm = GMAX > 8 ? 2 : 4;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(chunk_items, sm_count() * kPerSm / layers));
    // Where a block has one chunk, and with 16 heads' logits to a chunk, one is enough, in a short body (fp32 d 64, 3000 positions
    // x 2 heads, a layer 21.2 us with four, 20.7 with one; scoring of 9000 x 2, groups of 16, 23.2 and 21.1).
    auto *kern = GMAX > 8 || chunk_items <= grid ? w1_scores_kernel<GMAX, 1> : w1_scores_kernel<GMAX, GMAX <= 4 ? 4 : GMAX <= 8 ? 2 : 1>;
    const cudaError_t e = launch_dependent(kern, dim3(grid, layers), dim3(kThreadsW1), 0, st, a);
    count_launches(1);
    return e;
}

cudaError_t run_w1_scores_g(W1Args &a, int layers, int64_t chunk_items, Stream st, int G)
{
    if (G <= 4) return run_w1_scores<4>(a, layers, chunk_items, st);
    if (G <= 8) return run_w1_scores<8>(a, layers, chunk_items, st);
    return run_w1_scores<16>(a, layers, chunk_items, st);
}

template <typename T, int D>
cudaError_t run_w1_lanes(W1Args &a, int layers, int grid, Stream st, int G)
{
    auto *kern = G <= 4 ? w1_logits_kernel<T, D, 4> : G <= 8 ? w1_logits_kernel<T, D, 8> : w1_logits_kernel<T, D, 16>;
    const cudaError_t e = launch_dependent(kern, dim3(grid, layers), dim3(kThreadsW1), 0, st, a);
    count_launches(1);
    return e;
}

template <int D>
cudaError_t run_w1_mma(W1Args &a, int grid, Stream st, int G)
{
    auto *kern = G <= 8 ? w1_logits_mma_kernel<D, 1, true> : w1_logits_mma_kernel<D, 2, D == 64>;
    const cudaError_t e = launch_dependent(kern, dim3(grid), dim3(kThreadsW1), 0, st, a);
    count_launches(1);
    return e;
}

template <int D>
cudaError_t run_w1_unit(const W1Args &a, int layers, int units, int cluster, int stride, Stream st, int G)
{
    auto *kern = G <= 8 ? w1_unit_kernel<D, 1> : w1_unit_kernel<D, 2>;
    const cudaError_t e = launch_dependent_cluster(kern, cluster, dim3(units * cluster, layers), dim3(kThreadsUnit),
                                                   (size_t)G * stride * sizeof(float), st, a, stride);
    count_launches(1);
    return e;
}

}  // namespace

bool score_w1_supported(const refree_params &p)
{
    return p.window == 1 && p.num_q_heads / p.num_kv_heads <= kMaxG && (p.head_dim == 64 || p.head_dim == 128);
}

size_t score_w1_scratch_bytes(const refree_params &p, int64_t total_tokens)
{
    const int64_t spans = total_tokens / kMinSpan + p.num_seqs;          // the shortest span bounds the record count
    return (size_t)p.num_q_heads * total_tokens * sizeof(float) + 256 +
           (size_t)spans * p.num_q_heads * sizeof(float2);
}

cudaError_t launch_score_w1(const refree_params &p, const W1Group &g, const int32_t *seq_start, const int32_t *seq_len,
                            int64_t total_tokens, int32_t *dev_status, Stream st)
{
    const int layers = g.layers;
    W1Args a = {};
    a.p = p;
    a.layers = layers;
    bool aligned = true;
    for (int l = 0; l < layers; ++l) {
        a.q_win[l] = g.q_win[l];
        a.k[l] = g.k[l];
        a.sel_lengths[l] = g.sel_lengths[l];
        aligned = aligned && !(reinterpret_cast<uintptr_t>(g.q_win[l]) & 15);
    }
    a.seq_start = seq_start;
    a.seq_len = seq_len;
    const size_t logits_bytes = ((size_t)p.num_q_heads * total_tokens * sizeof(float) + 255) & ~(size_t)255;
    const size_t per_layer = (score_w1_scratch_bytes(p, total_tokens) + 255) & ~(size_t)255;
    a.logits = reinterpret_cast<float *>(g.scratch);
    a.stats = reinterpret_cast<float2 *>(g.scratch + logits_bytes);
    a.layer_logits = (int64_t)(per_layer / sizeof(float));
    a.layer_stats = (int64_t)(per_layer / sizeof(float2));
    a.layer_groups = (total_tokens / kTile + p.num_seqs) * p.num_kv_heads * 4;
    a.groups = g.groups;
    a.scores = g.scores;
    a.total_tokens = total_tokens;
    a.dev_status = dev_status;
    const bool sel = g.groups && g.cuts;
    a.sel_cuts = sel ? g.cuts : nullptr;
    const int G = p.num_q_heads / p.num_kv_heads;
    const bool f32 = p.dtype == REFREE_DTYPE_F32;
    const int64_t chunk_items = (total_tokens / kChunk + p.num_seqs) * p.num_kv_heads;
    cudaError_t e;
    const bool mma = !f32 && aligned;
    // A cluster per unit while the whole call is short (no unit is longer than the call) and its logits fit the default
    // limit of shared memory.  A layer compacted in place, 8 KV heads, with the two kernels below and this way: sequences of
    // 1000, 333 and 517 positions 21.0 and 15.4 us, one of 200 19.4 and 13.7, of 4096 21.1 and 16.8, of 8192 22.1 and 21.5,
    // eight of 1000 24.1 and 23.0.  Beyond the line (four layers, us): of 9000 104.0 and 103.9, of 12000 110 and 121, of 16000
    // 112 and 137.
    const int64_t cluster = std::min<int64_t>(kMaxClusterW1, (total_tokens + 127) / 128);
    if (mma && total_tokens <= kUnitTokens) {
        const int stride = (int)((total_tokens + 32 * cluster - 1) / (32 * cluster) * 32 + 8);   // (+ 8 spreads the heads over the banks)
        if ((size_t)G * stride * sizeof(float) <= 40 * 1024) {
            const int U = p.num_seqs * p.num_kv_heads;
            return p.head_dim == 64 ? run_w1_unit<64>(a, layers, U, (int)cluster, stride, st, G)
                                    : run_w1_unit<128>(a, layers, U, (int)cluster, stride, st, G);
        }
    }
    if (mma) {
        // one span per warp when the pass fits a single wave of 2 blocks per SM; capped so that
        // short sequences still spread over the machine
        const int64_t warps = (int64_t)sm_count() * 2 * (kThreadsW1 / 32);
        const int64_t rows = total_tokens * p.num_kv_heads;
        int64_t span = (rows + warps - 1) / warps;
        span = std::min<int64_t>(kMaxSpan, std::max<int64_t>(kMinSpan, (span + 15) / 16 * 16));
        a.span = (int)span;
        const int64_t span_items = (total_tokens / span + p.num_seqs) * p.num_kv_heads * layers;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((span_items + 7) / 8, sm_count() * 2));
        e = p.head_dim == 64 ? run_w1_mma<64>(a, grid, st, G) : run_w1_mma<128>(a, grid, st, G);
    } else {
        a.span = kChunk;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(chunk_items, sm_count() * 8));
        if (p.head_dim == 64)
            e = f32 ? run_w1_lanes<float, 64>(a, layers, grid, st, G) : run_w1_lanes<__nv_bfloat16, 64>(a, layers, grid, st, G);
        else
            e = f32 ? run_w1_lanes<float, 128>(a, layers, grid, st, G) : run_w1_lanes<__nv_bfloat16, 128>(a, layers, grid, st, G);
    }
    if (e != cudaSuccess) return e;
    e = run_w1_scores_g(a, layers, chunk_items, st, G);
    if (e != cudaSuccess || !sel) return e;
    SelectOut out = {};
    out.layers = layers;
    for (int l = 0; l < layers; ++l) out.lengths[l] = g.sel_lengths[l];
    return launch_unit_rules(p, g.scores, seq_len, total_tokens, g.groups, a.layer_groups, out, g.cuts, st);
}

}  // namespace refree
