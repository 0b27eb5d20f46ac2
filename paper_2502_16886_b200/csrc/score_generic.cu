// Generic scoring path (steps S1-S3) on the plain fp32 pipes: any supported dtype, head_dim 64 or 128, any window and
// query-group size.  It serves the fp32 cache and the shapes the tensor-core path does not take.  Three kernels (short calls take
// one, score_unit_generic):
//   stats   per (64 positions, KV head, window row): max and sum of 2^(y - max) over the visible positions,
//           y = (q.k / sqrt(d)) * log2(e)
//   combine per (unit, row): L = log2 sum_i 2^(y_i) over the whole row
//   colsum  per (64 positions, KV head): a'[i] = (1/G) sum_rows 2^(y - L) / cnt(i)   (Eq. 2)
//
// stats and colsum are bound by fp32 multiply-adds: a block of 256 threads forms the logits of 64 rows x 64 positions, a
// thread 4 x 4 of them from 16-byte pieces of the rows in shared memory (8 loads for 64 multiply-adds; rows padded by 16
// bytes, so the eight lanes of a load phase touch all banks once).  Units of up to 16 or 32 query rows take chunks of that
// many rows, 1 x 4 or 2 x 4 logits a thread.  The grids are (position tiles x KV heads, row chunks) for stats and
// position tiles x KV heads for colsum: 64 positions and not 128, because the small caches that come this way have too
// few tiles to fill the machine.  The second and third kernel are dependent launches: their blocks find their place in
// the batch and load K and Q while the kernel before drains.  Measured, us for the three kernels, against a warp per row
// with one multiply-add per shared-memory load and 128-position tiles: fp32 d 64, 512 positions x 2 heads, 64 rows
// 64 -> 18; 3000 x 8, 256 rows 268 -> 64; fp32 d 128, 2999 x 8, 256 rows 495 -> 115; bf16 d 64, 4000 x 2, 256 rows
// 217 -> 41.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "refree_internal.cuh"
#include "select_groups.cuh"

namespace refree {
namespace {

constexpr int kThreads = 256;
constexpr int kPT = 64;                 // positions of a tile
constexpr float kLog2e = 1.4426950408889634f;

struct Item { int s, g, tile_global, pos0, n, pack; };

// Sequence and tile of item `item` (= global tile * Hkv + head), found by a warp, 32 sequences at a time; s = -1 past
// the last.  The block shares the result.
__device__ inline void find_item(Item *out, const int32_t *seq_len, int B, int Hkv, int item)
{
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, want = item / Hkv;
        int tiles0 = 0, pack0 = 0;
        if (lane == 0) out->s = -1;
        __syncwarp();
        for (int s0 = 0; s0 < B; s0 += 32) {
            const int n = s0 + lane < B ? max(seq_len[s0 + lane], 0) : 0, nt = ceil_div(n, kPT);
            const int ti = warp_incl_scan(nt), pi = warp_incl_scan(n);
            if (nt > 0 && want >= tiles0 + ti - nt && want < tiles0 + ti) {
                out->s = s0 + lane;
                out->g = item % Hkv;
                out->tile_global = want;
                out->pos0 = (want - (tiles0 + ti - nt)) * kPT;
                out->n = n;
                out->pack = pack0 + pi - n;
            }
            tiles0 += __shfl_sync(0xffffffffu, ti, 31);
            pack0 += __shfl_sync(0xffffffffu, pi, 31);
            if (want < tiles0) break;
        }
    }
    __syncthreads();
}

// ROWS rows of D elements to shared memory as fp32, rows D + 4 floats apart; missing rows are zero.
// vec: every row starts on 16 bytes.
template <typename T, int D, int ROWS>
__device__ inline void load_rows(float *dst, const T *src, int64_t stride, int have, bool vec)
{
    constexpr int kE = 16 / sizeof(T), kV = D / kE;                   // elements per 16 bytes, 16-byte pieces per row
    for (int e = threadIdx.x; e < ROWS * kV; e += kThreads) {
        const int r = e / kV, c = (e % kV) * kE;
        float f[kE];
        if (r < have) {
            const T *p = src + (int64_t)r * stride + c;
            if (vec) {
                const uint4 x = *reinterpret_cast<const uint4 *>(p);
                const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                if (sizeof(T) == 4) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[i] = __uint_as_float(w[i]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        f[(2 * i) % kE] = __uint_as_float(w[i] << 16);
                        f[(2 * i + 1) % kE] = __uint_as_float(w[i] & 0xffff0000u);
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < kE; ++i) f[i] = to_float(p[i]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kE; ++i) f[i] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kE; i += 4)
            *reinterpret_cast<float4 *>(dst + r * (D + 4) + c + i) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
    }
}

// Query rows [r0, r0 + 16 RA) of unit (s, g); row r = head-in-group * window + window row.  They are back to back.
template <typename T, int D, int RA>
__device__ inline void load_q(float *dst, const refree_params &p, const T *q_win, int s, int g, int r0, bool vec)
{
    const int G = p.num_q_heads / p.num_kv_heads;
    load_rows<T, D, 16 * RA>(dst, q_win + (((int64_t)s * p.num_q_heads + (int64_t)g * G) * p.window + r0) * D, D, min(16 * RA, G * p.window - r0), vec);
}

// acc[a][b] = q row (ty + 16 a) . k row (tx + 16 b)
template <int D, int RA>
__device__ inline void dot_tile(const float *qs, const float *ks, float (&acc)[RA][4])
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
        float4 q[RA], k[4];
#pragma unroll
        for (int a = 0; a < RA; ++a) q[a] = *reinterpret_cast<const float4 *>(qs + (ty + 16 * a) * (D + 4) + c);
#pragma unroll
        for (int b = 0; b < 4; ++b) k[b] = *reinterpret_cast<const float4 *>(ks + (tx + 16 * b) * (D + 4) + c);
#pragma unroll
        for (int a = 0; a < RA; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                acc[a][b] = fmaf(q[a].x, k[b].x, acc[a][b]);
                acc[a][b] = fmaf(q[a].y, k[b].y, acc[a][b]);
                acc[a][b] = fmaf(q[a].z, k[b].z, acc[a][b]);
                acc[a][b] = fmaf(q[a].w, k[b].w, acc[a][b]);
            }
    }
}

template <typename T, int D>
__device__ inline const T *k_tile(const refree_params &p, const T *k, const int32_t *seq_start, const Item &it)
{
    return k + (int64_t)it.s * p.k_stride_seq + ((int64_t)seq_start[it.s] + it.pos0) * p.k_stride_tok + (int64_t)it.g * p.k_stride_head;
}

// (max, sum 2^(y - max)) over the 64 positions of a tile for a row of the chunk, in every lane of the row; y comes as the
// products of four positions and is scaled and masked on the way.
__device__ inline float2 tile_stats(float (&y)[4], int pos0, int n, int qpos, float scale)
{
    const int tx = threadIdx.x & 15;
    float m = -INFINITY, z = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int pos = pos0 + tx + 16 * b;
        y[b] = pos <= qpos && pos < n ? y[b] * scale : -INFINITY;
        m = fmaxf(m, y[b]);
    }
#pragma unroll
    for (int o = 8; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (m > -INFINITY) {
#pragma unroll
        for (int b = 0; b < 4; ++b) z += exp2f(y[b] - m);
    }
#pragma unroll
    for (int o = 8; o; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    return make_float2(m, z);
}

template <typename T, int D, int RA>
__global__ void __launch_bounds__(kThreads)
score_stats_generic(refree_params p, const T *q_win, const T *k, const int32_t *seq_start, const int32_t *seq_len, float2 *part, int q_vec)
{
    extern __shared__ __align__(16) float gsm[];
    __shared__ Item it;
    float *ks = gsm, *qs = gsm + kPT * (D + 4);
    const int Hkv = p.num_kv_heads, R = (p.num_q_heads / Hkv) * p.window, r0 = blockIdx.y * 16 * RA;
    dependency_wait();
    trigger_dependents();
    find_item(&it, seq_len, p.num_seqs, Hkv, blockIdx.x);
    if (it.s < 0) return;
    load_rows<T, D, kPT>(ks, k_tile<T, D>(p, k, seq_start, it), p.k_stride_tok, min(kPT, it.n - it.pos0), true);
    load_q<T, D, RA>(qs, p, q_win, it.s, it.g, r0, q_vec);
    __syncthreads();
    float acc[RA][4];
    dot_tile<D, RA>(qs, ks, acc);
    const float scale = kLog2e / sqrtf((float)D);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < RA; ++a) {
        const int r = r0 + ty + 16 * a, qpos = it.n - p.window + r % p.window;     // below zero: the row is not there
        const float2 st = tile_stats(acc[a], it.pos0, it.n, qpos, scale);
        if (tx == 0 && r < R) part[((int64_t)it.tile_global * Hkv + it.g) * R + r] = st;
    }
}

// (reference, sum) of a row over the tiles warp, warp + 8, ... of a unit's nt, `of(t)` being the row's record of tile t.
template <typename Of>
__device__ inline float2 combine_share(int nt, Of of)
{
    constexpr int kWarps = kThreads / 32;
    float M = -INFINITY, Z = 0.f;
    for (int t0 = threadIdx.x >> 5; t0 < nt; t0 += 8 * kWarps) {
        float2 x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = t0 + q * kWarps < nt ? of(t0 + q * kWarps) : make_float2(-INFINITY, 0.f);
        float m = M;
#pragma unroll
        for (int q = 0; q < 8; ++q) m = fmaxf(m, x[q].x);
        if (m == -INFINITY) continue;
        float z = Z * exp2f(M - m);
#pragma unroll
        for (int q = 0; q < 8; ++q) z += x[q].y * exp2f(x[q].x - m);
        Z = z;
        M = m;
    }
    return make_float2(M, Z);
}
// log2 of the row's sum from the shares of the warps
__device__ inline float combine_warps(const float2 (&red)[kThreads / 32][32], int lane)
{
    constexpr int kWarps = kThreads / 32;
    float m = -INFINITY, z = 0.f;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) m = fmaxf(m, red[q][lane].x);
#pragma unroll
    for (int q = 0; q < kWarps; ++q) z += m > -INFINITY ? red[q][lane].y * exp2f(red[q][lane].x - m) : 0.f;
    return m + log2f(z);
}

// One block per (unit, 32 rows): lane = row, the warps share the tiles.
__global__ void __launch_bounds__(kThreads)
score_combine_generic(refree_params p, const int32_t *seq_len, const float2 *part, float *lse)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ float2 red[kWarps][32];
    __shared__ int s_tiles;
    const int Hkv = p.num_kv_heads, R = (p.num_q_heads / Hkv) * p.window;
    const int u = blockIdx.y, s = u / Hkv, g = u - s * Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = blockIdx.x * 32 + lane;
    trigger_dependents();
    if (warp == 0) {                              // tiles before the sequence
        int t = 0;
        for (int i = lane; i < s; i += 32) t += ceil_div(max(seq_len[i], 0), kPT);
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s_tiles = t;
    }
    __syncthreads();
    const int nt = ceil_div(max(seq_len[s], 0), kPT);
    dependency_wait();
    float2 share = make_float2(-INFINITY, 0.f);
    if (r < R) {
        const float2 *src = part + ((int64_t)s_tiles * Hkv + g) * R + r;
        share = combine_share(nt, [&](int t) { return src[(int64_t)t * Hkv * R]; });
    }
    red[warp][lane] = share;
    __syncthreads();
    if (warp == 0 && r < R) lse[(int64_t)u * R + r] = combine_warps(red, lane);
}

// sum[b] += 2^(y - L) over the rows of a chunk that see position tx + 16 b of the tile; L[r] for r < R.
template <int RA>
__device__ inline void tile_colsum(const float (&acc)[RA][4], const refree_params &p, const float *L, int r0, int R, int n, int pos0,
                                   float scale, float (&sum)[4])
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < RA; ++a) {
        const int r = r0 + ty + 16 * a, qpos = n - p.window + r % p.window;
        const float l = r < R && qpos >= 0 ? L[r] : 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (r < R && pos0 + tx + 16 * b <= qpos) sum[b] += exp2f(fmaf(acc[a][b], scale, -l));
    }
}
// The tile's scores (Eq. 2), a thread of the first kPT each; the row groups' shares meet in `red`.
__device__ inline float tile_score(const refree_params &p, const float (&sum)[4], float (&red)[16][kPT], int pos, int n)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int b = 0; b < 4; ++b) red[ty][tx + 16 * b] = sum[b];
    __syncthreads();
    if (threadIdx.x >= kPT || pos >= n) return 0.f;
    float tot = 0.f;
#pragma unroll
    for (int q = 0; q < 16; ++q) tot += red[q][threadIdx.x];
    const int cnt = min(min(p.window, n), n - pos);
    return tot / (float)cnt / (float)(p.num_q_heads / p.num_kv_heads);
}

template <typename T, int D, int RA>
__global__ void __launch_bounds__(kThreads)
score_colsum_generic(refree_params p, const T *q_win, const T *k, const int32_t *seq_start, const int32_t *seq_len, const float *lse,
                     int64_t total_tokens, float *scores, int32_t *dev_status, int q_vec)
{
    extern __shared__ __align__(16) float gsm[];
    __shared__ Item it;
    __shared__ float red[16][kPT];
    float *ks = gsm, *qs = gsm + kPT * (D + 4);
    const int Hkv = p.num_kv_heads, R = p.num_q_heads / Hkv * p.window;
    trigger_dependents();
    find_item(&it, seq_len, p.num_seqs, Hkv, blockIdx.x);
    if (it.s < 0) { dependency_wait(); return; }
    load_rows<T, D, kPT>(ks, k_tile<T, D>(p, k, seq_start, it), p.k_stride_tok, min(kPT, it.n - it.pos0), true);
    const float scale = kLog2e / sqrtf((float)D);
    const float *L = lse + ((int64_t)it.s * Hkv + it.g) * R;
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
    for (int r0 = 0; r0 < R; r0 += 16 * RA) {
        __syncthreads();                          // the rows before have been read
        load_q<T, D, RA>(qs, p, q_win, it.s, it.g, r0, q_vec);
        __syncthreads();
        float acc[RA][4];
        dot_tile<D, RA>(qs, ks, acc);
        if (r0 == 0) dependency_wait();
        tile_colsum<RA>(acc, p, L, r0, R, it.n, it.pos0, scale, sum);
    }
    const int pos = it.pos0 + (int)threadIdx.x;
    const float sc = tile_score(p, sum, red, pos, it.n);
    if (threadIdx.x < kPT && pos < it.n) {
        if (!isfinite(sc) && dev_status) atomicOr(dev_status, REFREE_DEV_NONFINITE);
        scores[(int64_t)it.g * total_tokens + it.pack + pos] = sc;
    }
}

// A short unit in one cluster of blocks, a tile to a block, from K to its scores, and to its budget where the rule can follow
// (position ranking per head).  Bound by latency: the three kernels above and the rule are each a microsecond of work between
// two trips to memory; here the blocks meet in distributed shared memory, and a thread keeps its 4 x 4 products of query and
// key from one pass to the next.  Same sums in the same order as the three kernels.
// One chunk of rows and one tile to a block: the products are bound by the multiply-adds of the SMs that take part (a tile of
// 64 rows x 64 positions x 64 columns 1.1 us), so longer units and more rows are faster spread over the whole GPU twice (a
// layer, us, three kernels and this way: fp32 d 64, 2 heads of 512 positions, 64 rows 20 and 16; 8 heads of 200, 64 rows
// 22 and 20; two tiles to a block, bf16 d 64, 16 heads of 700, 64 rows 28.7 and 31.0; two tiles of four chunks, fp32 d 64,
// 8 heads of 600, 256 rows 40.9 and 53.4).
struct UnitArgs {
    refree_params p;
    const void *q_win, *k;
    const int32_t *seq_start, *seq_len;
    int64_t total_tokens;
    float *scores;
    GroupPartial *groups;    // nullable: records of the stopping rule; then the budget is chosen too
    int32_t *sel_lengths;
    Cut *sel_cuts;
    int32_t *dev_status;
    int q_vec;
};
constexpr int kMaxClusterUnit = 8;
constexpr int kUnitRows = 64;

template <typename T, int D, int RA>
__global__ void __launch_bounds__(kThreads)
score_unit_generic(const __grid_constant__ UnitArgs a)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) float gsm[];
    __shared__ float red[16][kPT];
    __shared__ float2 share[kThreads / 32][32];
    __shared__ float2 rec[kUnitRows];                // (reference, sum) of the rows over this block's tile
    __shared__ float lse[kUnitRows];
    __shared__ BlockRuleShared<kThreads> rule;
    __shared__ uint32_t wmax[2], cmax[kMaxClusterUnit];
    cg::cluster_group cl = cg::this_cluster();
    const int nblk = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const refree_params &p = a.p;
    const T *const q_win = static_cast<const T *>(a.q_win), *const k = static_cast<const T *>(a.k);
    const int Hkv = p.num_kv_heads, R = p.num_q_heads / Hkv * p.window;
    const int u = blockIdx.x / nblk, s = u / Hkv, g = u - s * Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float *const ks = gsm, *const qs = ks + kPT * (D + 4);
    dependency_wait();
    trigger_dependents();
    int pack = 0, tiles128 = 0;                      // positions and 128-position tiles of the sequences before this one
    for (int s0 = 0; s0 < s; s0 += 32) {
        const int nn = s0 + lane < s ? max(a.seq_len[s0 + lane], 0) : 0;
        pack += __reduce_add_sync(0xffffffffu, nn);
        tiles128 += __reduce_add_sync(0xffffffffu, ceil_div(nn, kTile));
    }
    Item it;
    it.s = s; it.g = g; it.pack = pack; it.pos0 = rank * kPT;
    it.n = max(a.seq_len[s], 0);
    const int n = it.n, nt = ceil_div(n, kPT);
    if (n == 0) {                                    // keeps nothing (the whole cluster leaves)
        if (rank == 0 && threadIdx.x == 0 && a.groups) {
            Cut cut;
            cut.b = 0; cut.ties = 0; cut.tau = 0; cut.prot_kept = 0; cut.sbias = 0;
            a.sel_lengths[u] = 0;
            a.sel_cuts[u] = cut;
        }
        return;
    }
    const float scale = kLog2e / sqrtf((float)D);
    float acc[RA][4];
    if (rank < nt) {
        load_rows<T, D, kPT>(ks, k_tile<T, D>(p, k, a.seq_start, it), p.k_stride_tok, min(kPT, n - it.pos0), true);
        load_q<T, D, RA>(qs, p, q_win, s, g, 0, a.q_vec);
        __syncthreads();
        dot_tile<D, RA>(qs, ks, acc);
#pragma unroll
        for (int x = 0; x < RA; ++x) {
            const int r = ty + 16 * x, qpos = n - p.window + r % p.window;
            float y[4] = {acc[x][0], acc[x][1], acc[x][2], acc[x][3]};
            const float2 st = tile_stats(y, it.pos0, n, qpos, scale);
            if (tx == 0 && r < R) rec[r] = st;
        }
    }
    cl.sync();
    // 32 rows to a block: L of a row from all tiles of the unit, told to every block
    for (int r0 = rank * 32; r0 < R; r0 += nblk * 32) {
        const int r = r0 + lane;
        share[warp][lane] = r < R ? combine_share(nt, [&](int t) { return cl.map_shared_rank(rec, t)[r]; }) : make_float2(-INFINITY, 0.f);
        __syncthreads();
        const float l = combine_warps(share, lane);
        if (r < R && warp < nblk) cl.map_shared_rank(lse, warp)[r] = l;      // (eight warps, at most eight blocks)
        __syncthreads();
    }
    cl.sync();
    float *const sc_out = a.scores + (int64_t)g * a.total_tokens + pack;
    GroupPartial *const grp = a.groups ? a.groups + ((int64_t)tiles128 * Hkv + (int64_t)g * ceil_div(n, kTile)) * 4 : nullptr;
    uint32_t run_max = 0;
    if (rank < nt) {
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
        tile_colsum<RA>(acc, p, lse, 0, R, n, it.pos0, scale, sum);
        const int pos = it.pos0 + (int)threadIdx.x;
        const float sc = tile_score(p, sum, red, pos, n);
        if (threadIdx.x < kPT) {
            if (pos < n) {
                if (!isfinite(sc) && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_NONFINITE);
                sc_out[pos] = sc;
            }
            if (grp && it.pos0 + 32 * warp < n) {    // exact sum of squares of these 32 positions
                const uint32_t bits = (pos < n && isfinite(sc)) ? mag_bits(sc) : 0u;
                run_max = __reduce_max_sync(0xffffffffu, bits);
                unsigned long long sq = sq_fixed(bits, kGroupShift - 2 * max(1, (int)(run_max >> 23)));
#pragma unroll
                for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (lane == 0) { GroupPartial gp; gp.max_bits = run_max; gp.pad = 0u; gp.sum = sq; grp[(it.pos0 >> 5) + warp] = gp; }
            }
        }
    }
    if (!grp) return;                                // (nothing remote is read after the barrier before)
    if (warp < 2 && lane == 0) wmax[warp] = run_max;
    __syncthreads();
    if (threadIdx.x == 0) *cl.map_shared_rank(&cmax[rank], 0) = max(wmax[0], wmax[1]);
    __threadfence();
    cl.sync();                                       // scores and records of the cluster are visible to the first block
    if (rank != 0) return;
    uint32_t unit_max = 0;
    for (int b = 0; b < nblk; ++b) unit_max = max(unit_max, cmax[b]);
    const UnitRule ur(p, sc_out, n, grp, unit_max);
    block_unit_rule<kThreads>(ur, rule, a.sel_lengths + u, a.sel_cuts + u);
}

// Whether a call takes the cluster per unit: no unit is longer than the call, and the blocks (most of them idle where the call
// is many short sequences) fit the SMs at once.  (bf16 rows of 128 come here only with queries that do not start on 16 bytes:
// no variants for those.)
bool one_launch(const refree_params &p, int64_t total_tokens)
{
    const int64_t blocks = (total_tokens + kPT - 1) / kPT * p.num_seqs * p.num_kv_heads;
    return blocks <= 2 * sm_count() && (p.dtype == REFREE_DTYPE_F32 || p.head_dim == 64) && total_tokens > 0 && total_tokens <= kMaxClusterUnit * kPT &&
           p.num_q_heads / p.num_kv_heads * (int64_t)p.window <= kUnitRows;
}

template <typename T, int D, int RA>
cudaError_t run_unit(const UnitArgs &a, Stream st)
{
    auto *kern = score_unit_generic<T, D, RA>;
    constexpr size_t smem = (size_t)(kPT + 16 * RA) * (D + 4) * sizeof(float);
    cudaError_t e = allow_smem(kern, std::max<size_t>(smem, 64 * 1024));      // (some of the kernel's is static)
    if (e != cudaSuccess) return e;
    const int cluster = (int)((a.total_tokens + kPT - 1) / kPT);
    e = launch_dependent_cluster(kern, cluster, dim3(a.p.num_seqs * a.p.num_kv_heads * cluster), dim3(kThreads), smem, st, a);
    count_launches(1);
    return e;
}
template <typename T, int D>
cudaError_t run_unit_rows(const UnitArgs &a, Stream st)
{
    const int R = a.p.num_q_heads / a.p.num_kv_heads * a.p.window;
    return R <= 16 ? run_unit<T, D, 1>(a, st) : R <= 32 ? run_unit<T, D, 2>(a, st) : run_unit<T, D, 4>(a, st);
}

template <typename T, int D, int RA>
cudaError_t run_rows(const refree_params &p, const void *q_win, const void *k, const int32_t *seq_start,
                const int32_t *seq_len, int64_t total_tokens, float *scores, char *ws,
                const Workspace &lay, int32_t *dev_status, Stream st)
{
    constexpr int kSmem = (kPT + 16 * RA) * (D + 4) * (int)sizeof(float);
    {
        static std::mutex m;                      // the shared-memory limit is raised once per device
        static bool set[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> hold(m);
        if (!set[dev]) {
            cudaError_t e = cudaFuncSetAttribute(score_stats_generic<T, D, RA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(score_colsum_generic<T, D, RA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
            if (e != cudaSuccess) return e;
            set[dev] = true;
        }
    }
    const int G = p.num_q_heads / p.num_kv_heads, R = G * p.window;
    const unsigned items = (unsigned)((total_tokens / kPT + p.num_seqs) * p.num_kv_heads);
    float2 *part = reinterpret_cast<float2 *>(ws + lay.part_off);
    float *lse = reinterpret_cast<float *>(ws + lay.lse_off);
    const int q_vec = (reinterpret_cast<uintptr_t>(q_win) & 15) == 0;
    cudaError_t e = launch_dependent(score_stats_generic<T, D, RA>, dim3(items, (R + 16 * RA - 1) / (16 * RA)), dim3(kThreads), kSmem, st, p,
                                     (const T *)q_win, (const T *)k, seq_start, seq_len, part, q_vec);
    if (e == cudaSuccess)
        e = launch_dependent(score_combine_generic, dim3((R + 31) / 32, p.num_seqs * p.num_kv_heads), dim3(kThreads), 0, st, p, seq_len,
                             (const float2 *)part, lse);
    // The blocks of a chained launch land on the SMs that are free at that moment, several to one while others come free later.
    // That costs more than the launch where they take long and are too few to fill the machine: 36 blocks of 800 rows 111 to
    // 168 us against 78 (a run of eight layers of 1078 positions 1195 -> 903), 79 of 400 rows (four layers of 5000 positions)
    // 319 -> 257; with 8 blocks there is room for each (500 positions 182, not chained 210).
    const unsigned sms = (unsigned)sm_count();
    const bool spread = R > 256 && items >= sms / 8 && items < 2 * sms;
    if (e == cudaSuccess)
        e = launch_dependent(score_colsum_generic<T, D, RA>, dim3(items), dim3(kThreads), kSmem, Stream(st.s, st.chain && !spread), p, (const T *)q_win, (const T *)k,
                             seq_start, seq_len, (const float *)lse, total_tokens, scores, dev_status, q_vec);
    if (e != cudaSuccess) return e;
    count_launches(3);
    return cudaGetLastError();
}

template <typename T, int D>
cudaError_t run(const refree_params &p, const void *q_win, const void *k, const int32_t *seq_start,
                const int32_t *seq_len, int64_t total_tokens, float *scores, char *ws,
                const Workspace &lay, int32_t *dev_status, Stream st)
{
    const int R = p.num_q_heads / p.num_kv_heads * p.window;
    if (R <= 16) return run_rows<T, D, 1>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st);
    if (R <= 32) return run_rows<T, D, 2>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st);
    return run_rows<T, D, 4>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st);
}

}  // namespace

bool score_generic_rule(const refree_params &p, int64_t total_tokens) { return one_launch(p, total_tokens); }

cudaError_t launch_score_generic(const refree_params &p, const void *q_win, const void *k,
                                 const int32_t *seq_start, const int32_t *seq_len,
                                 int64_t total_tokens, float *scores, char *ws, const Workspace &lay,
                                 int32_t *dev_status, Stream st, GroupPartial *groups, int32_t *sel_lengths)
{
    const bool f32 = p.dtype == REFREE_DTYPE_F32;
    if (one_launch(p, total_tokens)) {
        UnitArgs a = {};
        a.p = p;
        a.q_win = q_win; a.k = k;
        a.seq_start = seq_start; a.seq_len = seq_len;
        a.total_tokens = total_tokens;
        a.scores = scores;
        a.groups = sel_lengths ? groups : nullptr;
        a.sel_lengths = sel_lengths;
        a.sel_cuts = reinterpret_cast<Cut *>(ws + lay.cut_off);
        a.dev_status = dev_status;
        a.q_vec = (reinterpret_cast<uintptr_t>(q_win) & 15) == 0;
        if (p.head_dim == 64) return f32 ? run_unit_rows<float, 64>(a, st) : run_unit_rows<__nv_bfloat16, 64>(a, st);
        return run_unit_rows<float, 128>(a, st);
    }
    if (p.head_dim == 64)
        return f32 ? run<float, 64>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st)
                   : run<__nv_bfloat16, 64>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st);
    return f32 ? run<float, 128>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st)
               : run<__nv_bfloat16, 128>(p, q_win, k, seq_start, seq_len, total_tokens, scores, ws, lay, dev_status, st);
}

}  // namespace refree
