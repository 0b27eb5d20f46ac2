// Decode-step attention over the compacted ragged cache: the consumer of the pass
// (Algorithm 1 returns K_c, V_c "for generation"; Section 3.3 batches sequences of
// different budgets).  One new query per (sequence, query head):
//     out[s, h, :] = softmax(q[s, h] . K_c[u]^T / sqrt(d)) V_c[u],   u = s Hkv + g(h),
// over rows [offsets[u], offsets[u + 1]) of the dense ragged cache.
//
// The step streams K_c and V_c once (G query heads share every row): HBM-bound.
//
//   bf16   block = (unit, span of rows), four warps take 16-row blocks round-robin.  A block
//          of 16 rows is contiguous in the compacted cache: one lane of the warp copies it with
//          cp.async.bulk into the warp's private shared-memory ring (three blocks in flight,
//          mbarrier-signalled).  mma.m16n8k16 serves as the dot-product unit:
//            S^T[head, row] = Q K^T   A = the G (<= 16) queries, B = 8 rows of K; each
//                                     lane reads 16-byte pieces of "its" row and the
//                                     queries are cut the same way, so the order of the
//                                     elements inside a k-step cancels;
//            O[head, col]  += P V     A = the probabilities straight from the S^T
//                                     accumulators (split into two bf16 terms, so the
//                                     product carries 16 mantissa bits), B = V: a lane
//                                     reads 16-byte pieces of four rows and interleaves
//                                     row pairs with byte permutes.  The eight columns of
//                                     an output tile are spread over the row (column
//                                     (t / 8) 64 + 8 n + t % 8 for tile t, slot n); the
//                                     order is undone when the result is stored.
//          Running (max, sum) per head (online softmax), warps merged through shared memory.
//   fp32   (or unaligned bf16 pointers) lanes own columns, dot products by warp shuffles.
//
// How the rows are cut into blocks (decode_shape has the rule and what both sides measured):
//   fixed     the same span of rows for every block, sized for the longest unit, so that its blocks fill the SMs once;
//             a second small kernel merges the records of units that took several blocks;
//   cluster   short units: a cluster per unit, merged through distributed shared memory, so the step is one launch;
//   planned   very ragged lengths: a unit's block count follows its length (make_plan), then the same second kernel.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "refree_internal.cuh"

namespace refree {
namespace {

// Warps of a block (NW): eight and one block an SM, so that a unit has few records to merge (32K rows of 8 units: 28.9 us
// and 31.1 with four); four and two blocks an SM in a cluster, where a short unit spreads over more SMs (six sequences of
// 96 to 1500 rows, 24 units: 9.9 us, 14.3 with eight).
constexpr float kLog2eDec = 1.4426950408889634f;
constexpr int kDecStages = 3;       // 16-row blocks of K and V in flight per warp
constexpr int kPlanUnits = 128;     // most units that a plan is made for
constexpr int kMinRows = 64;        // fewest rows worth a block: a 16-row block for each of four warps

constexpr int kClusterRows = 320;   // most rows of a block of a cluster
constexpr int kMaxClusterDec = 8;   // blocks of a cluster

enum DecMode { kFixed, kCluster, kPlanned };

struct DecArgs {
    refree_params p;
    const void *q, *kc, *vc;
    const int64_t *offsets;
    // strided ragged cache (what refree_compact_inplace leaves): rows of unit (s, g) sit in the unit's own
    // region of the original K / V arrays; `lengths` non-null selects this form and `offsets` is unused
    const int32_t *seq_start, *seq_len, *lengths;
    int anchor_back;
    float *out;      // [B, Hq, d]
    float *part;     // fixed, planned: [record, G, d + 2]: un-normalised output (block order), max, sum
    int mode;        // DecMode
    int blocks;      // blocks per unit (fixed, cluster) or of the grid (planned)
    int span;        // fixed: rows per block
    int cap;         // most rows of a unit
    int native;      // 1: partials hold the mma tile order, 0: plain column order
    int32_t *dev_status;
};

// First row (in rows of head_dim elements from the array's start) and row count of unit u in K and in V.
__device__ inline int64_t unit_len(const DecArgs &a, int u)
{
    if (!a.lengths) return a.offsets[u + 1] - a.offsets[u];
    const int n = max(a.seq_len[u / a.p.num_kv_heads], 0);
    return max(0, min(a.lengths[u], n));
}
// The loads go out together, and the strides are divided by the constant head dimension: this is the head of every call's
// chain of waits (a 64-bit division is a routine of some hundred instructions; both, 1.9 us before the first row was asked for).
template <int D>
__device__ inline void unit_rows(const DecArgs &a, int u, int64_t &lo_k, int64_t &lo_v, int64_t &len64)
{
    if (!a.lengths) {
        const int64_t lo = a.offsets[u], hi = a.offsets[u + 1];
        lo_k = lo_v = lo;
        len64 = hi - lo;
        return;
    }
    const int Hkv = a.p.num_kv_heads, s = u / Hkv, g = u - s * Hkv;
    const int n0 = a.seq_len[s], b = a.lengths[u], start = a.seq_start[s];
    const int n = max(n0, 0);
    len64 = max(0, min(b, n));
    const int64_t first = (int64_t)start + (a.anchor_back ? n - len64 : 0);
    lo_k = (int64_t)((uint64_t)((int64_t)s * a.p.k_stride_seq + (int64_t)g * a.p.k_stride_head) / D) + first;
    lo_v = (int64_t)((uint64_t)((int64_t)s * a.p.v_stride_seq + (int64_t)g * a.p.v_stride_head) / D) + first;
}
__device__ inline int clamp_len(const DecArgs &a, int64_t len64) { return (int)max((int64_t)0, min(len64, (int64_t)a.cap)); }

// Which rows a block takes: rows [x span, (x + 1) span) of unit u, the x-th of its nblocks pieces; its record if several.
struct Piece {
    int u, x, span, nblocks, rec;
    int len;                // rows of the unit
    int64_t lo_k, lo_v;     // its first row in K and in V
};

// Cut of all units into at most a.blocks pieces of nearly the same number of rows, by one warp: a unit of n rows gets
// ceil(n / share) pieces, with the share of blocks - U / 4, - U / 2 or - U pieces, whichever first suffices (the last
// always does: a unit wastes less than one piece).  want < 0: the piece of record -want - 1 (u < 0 when there is none), else the pieces of unit `want`.  The counts
// come from one float factor, a little small so that rounding cannot add a piece; every warp computes the same.
__device__ inline Piece make_plan(const DecArgs &a, int want)
{
    const int U = a.p.num_seqs * a.p.num_kv_heads, lane = threadIdx.x & 31;
    int len[kPlanUnits / 32];
    float total = 0.f;
#pragma unroll
    for (int i = 0; i < kPlanUnits / 32; ++i) {
        len[i] = -1;
        if (32 * i < U) {
            if (32 * i + lane < U) len[i] = clamp_len(a, unit_len(a, 32 * i + lane));
            total += (float)max(len[i], 0);
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    float rate = 0.f;                                    // pieces per row
#pragma unroll 1
    for (int c = 1; c <= 4; c *= 2) {
        rate = fminf((float)(a.blocks - U * c / 4) / total * 0.99998f, 1.f / (float)kMinRows);
        int n = 0;
#pragma unroll
        for (int i = 0; i < kPlanUnits / 32; ++i)
            if (32 * i < U) n += len[i] >= 0 ? max(1, (int)ceilf((float)len[i] * rate)) : 0;
        if (__reduce_add_sync(0xffffffffu, n) <= a.blocks) break;
    }
    Piece pc = {-1, 0, 16, 0, 0, 0, 0, 0};
    int before = 0;
#pragma unroll
    for (int i = 0; i < kPlanUnits / 32; ++i) {
        if (32 * i >= U || pc.u >= 0) continue;
        const int n = len[i] >= 0 ? max(1, (int)ceilf((float)len[i] * rate)) : 0;
        const int incl = before + warp_incl_scan(n);
        const unsigned hit = __ballot_sync(0xffffffffu, want >= 0 ? 32 * i + lane == want : (n > 0 && -want - 1 < incl));
        if (hit) {
            const int l = __ffs(hit) - 1;
            const int un = __shfl_sync(0xffffffffu, n, l), ul = __shfl_sync(0xffffffffu, len[i], l);
            const int first = __shfl_sync(0xffffffffu, incl, l) - un;
            pc.u = 32 * i + l;
            pc.span = max(16, (ceil_div(ul, un) + 15) / 16 * 16);
            pc.nblocks = ceil_div(ul, pc.span);
            pc.x = want >= 0 ? 0 : -want - 1 - first;
            pc.rec = first + pc.x;
        }
        before = __shfl_sync(0xffffffffu, incl, 31);
    }
    return pc;
}

// Piece x of unit u where the unit alone decides.
__device__ inline Piece unit_piece(const DecArgs &a, int u, int x, int len)
{
    const int span = a.mode == kFixed ? a.span : max(kMinRows, (ceil_div(len, a.blocks) + 15) / 16 * 16);
    return {u, x, span, ceil_div(len, span), u * a.blocks + x, 0, 0, 0};
}

__device__ inline float dec_ex2(float x)
{
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ inline void dec_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ inline uint4 dec_ld16(const char *p, bool valid)
{
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (valid)
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// ---- per-warp staging ring: bulk copies (TMA engine, no tensor map) signalled on an mbarrier ----
__device__ inline uint32_t dec_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ inline void dec_bar_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(dec_smem(bar)) : "memory");
}
__device__ inline void dec_bar_expect(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(dec_smem(bar)), "r"(bytes) : "memory");
}
// contiguous global -> shared copy; addresses 16-byte aligned, size a multiple of 16
__device__ inline void dec_bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dec_smem(dst)), "l"(src), "r"(bytes), "r"(dec_smem(bar)) : "memory");
}
// bounded wait for the phase with the given parity; false when it gave up
__device__ inline bool dec_bar_wait(uint64_t *bar, uint32_t parity)
{
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(dec_smem(bar)), "r"(parity) : "memory");
        if (ok) return true;
        if (it > 64) __nanosleep(it > 4096 ? 256 : 32);
    }
    return false;
}

// p = hi + lo with hi, lo bf16: packs two probabilities per register for the A operand
__device__ inline void split_pack(float p0, float p1, uint32_t &hi, uint32_t &lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(p0, p1);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(p0 - hf.x, p1 - hf.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// column of the output that slot `idx` of the block order holds
__device__ __host__ inline int native_col(int idx, int native)
{
    if (!native) return idx;
    const int t = idx >> 3, n = idx & 7;
    return (t >> 3) * 64 + n * 8 + (t & 7);
}

// Merge the warps' (max, sum, O) through shared memory in warp order and store the block's
// result: the final output when the unit has one block, a record otherwise.  sm: [NW][GP][D + 2] floats, then the
// block's own record [GP][D + 2] (cluster), then the factors [GP][NW + 1].
// Two ways to the same bits: every thread works out what the warps count for its element, or that is done once per head and
// shared, with a barrier more.  The first is faster while a thread has one element, the second beyond (bf16 d 64, groups of one,
// 300 rows 4.23 and 4.33 us; fp32 d 64, groups of sixteen, five sequences of 1651 to 84 18.9 and 17.4).  fp32 rows of 64 in
// groups of up to four have the first alone: beside the second their loop over the rows got slower (16 heads, eight sequences of
// 2435 to 95 rows 40.0 and 41.7).
enum Merge { kPerElement, kPerHead, kBySize };
template <int D, int NW, Merge FORM>
__device__ inline void merge_and_store(const DecArgs &a, float *sm, int GP, int G, const Piece &pc)
{
    float *const fac = sm + (NW + 1) * GP * (D + 2);
    __syncthreads();
    const int Hkv = a.p.num_kv_heads, s = pc.u / Hkv, g = pc.u - s * Hkv;
    float *recs = a.mode == kCluster ? sm + NW * GP * (D + 2) : a.part + (int64_t)pc.rec * G * (D + 2);
    if (FORM == kPerElement || (FORM == kBySize && G * (D + 2) <= 32 * NW)) {
        for (int e = threadIdx.x; e < G * (D + 2); e += 32 * NW) {
            const int h = e / (D + 2), idx = e % (D + 2);
            float M = -INFINITY, L = 0.f, val = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) M = fmaxf(M, sm[(w * GP + h) * (D + 2) + D]);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float *rec = sm + (w * GP + h) * (D + 2);
                const float f = rec[D] == -INFINITY ? 0.f : dec_ex2(rec[D] - M);
                val += rec[idx < D ? idx : 0] * f;
                L += rec[D + 1] * f;
            }
            if (pc.nblocks > 1)
                recs[e] = idx < D ? val : (idx == D ? M : L);
            else if (idx < D)
                a.out[((int64_t)s * a.p.num_q_heads + g * G + h) * D + native_col(idx, a.native)] = L > 0.f ? val / L : 0.f;
        }
        return;
    }
    if (threadIdx.x < G) {
        const int h = threadIdx.x;
        float m[NW], l[NW], M = -INFINITY, L = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            m[w] = sm[(w * GP + h) * (D + 2) + D];
            l[w] = sm[(w * GP + h) * (D + 2) + D + 1];
            M = fmaxf(M, m[w]);
        }
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float f = m[w] == -INFINITY ? 0.f : dec_ex2(m[w] - M);
            fac[h * (NW + 1) + w] = f;
            L += l[w] * f;
        }
        fac[h * (NW + 1) + NW] = L;
        if (pc.nblocks > 1) { recs[h * (D + 2) + D] = M; recs[h * (D + 2) + D + 1] = L; }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < G * (D / 2); e += 32 * NW) {
        const int h = e / (D / 2), idx = 2 * (e % (D / 2));
        float2 val = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float2 x = *reinterpret_cast<const float2 *>(sm + (w * GP + h) * (D + 2) + idx);
            const float f = fac[h * (NW + 1) + w];
            val.x += x.x * f;
            val.y += x.y * f;
        }
        if (pc.nblocks == 1) {
            const float L = fac[h * (NW + 1) + NW];
            float *out = a.out + ((int64_t)s * a.p.num_q_heads + g * G + h) * D;
            out[native_col(idx, a.native)] = L > 0.f ? val.x / L : 0.f;
            out[native_col(idx + 1, a.native)] = L > 0.f ? val.y / L : 0.f;
        } else {
            *reinterpret_cast<float2 *>(recs + h * (D + 2) + idx) = val;
        }
    }
}

// Cluster: the blocks of a unit merge their records, every block a share of the output.  All blocks of the cluster come
// here, those without rows too.
template <int D, int NW>
__device__ inline void merge_cluster(const DecArgs &a, float *sm, int GP, int G, const Piece &pc)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (pc.nblocks > 1) {
        const int Hkv = a.p.num_kv_heads, s = pc.u / Hkv, g = pc.u % Hkv;
        float *recs = sm + NW * GP * (D + 2);
        for (int e = blockIdx.x * 32 * NW + threadIdx.x; e < G * D; e += gridDim.x * 32 * NW) {
            const int h = e / D, idx = e % D;
            float mm[kMaxClusterDec], ll[kMaxClusterDec], vv[kMaxClusterDec], M = -INFINITY;
#pragma unroll
            for (int b = 0; b < kMaxClusterDec; ++b) {
                const float *rec = cl.map_shared_rank(recs, b < pc.nblocks ? b : 0) + h * (D + 2);
                mm[b] = b < pc.nblocks ? rec[D] : -INFINITY;
                ll[b] = rec[D + 1];
                vv[b] = rec[idx];
                M = fmaxf(M, mm[b]);
            }
            float L = 0.f, val = 0.f;
#pragma unroll
            for (int b = 0; b < kMaxClusterDec; ++b) {
                const float f = mm[b] == -INFINITY ? 0.f : dec_ex2(mm[b] - M);
                val += vv[b] * f;
                L += ll[b] * f;
            }
            a.out[((int64_t)s * a.p.num_q_heads + g * G + h) * D + native_col(idx, a.native)] = L > 0.f ? val / L : 0.f;
        }
    }
    cl.sync();                                       // nobody leaves while its record may still be read
}

// bf16 path.  UPPER: the group has more than eight query heads (rows 8..15 of the A operand).
template <int D, bool UPPER, int NW>
__device__ inline void decode_mma(const DecArgs &a, const Piece &pc, float *dec_sm)
{
    constexpr int CH = D / 32;          // 16-byte pieces per lane of a K (or Q) row
    constexpr int HF = D / 64;          // 128-byte halves of a V row
    constexpr int NT = D / 8;           // output tiles of eight columns
    constexpr int GP = UPPER ? 16 : 8;
    const refree_params &p = a.p;
    const int Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int u = pc.u, s = u / Hkv, g = u % Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 2, c = lane & 3;
    const int64_t lo = pc.lo_k, lo_v = pc.lo_v;
    const int begin = pc.x * pc.span, end = min(pc.len, begin + pc.span);
    const float scale = kLog2eDec * rsqrtf((float)D);

    // queries of heads r (and r + 8), cut into the 16-byte pieces at byte 64 j + 16 c
    uint4 qa[CH], qb[CH];
    {
        const char *qrow = reinterpret_cast<const char *>(a.q) +
                           ((int64_t)s * p.num_q_heads + g * G) * D * (int64_t)sizeof(__nv_bfloat16);
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            qa[j] = dec_ld16(qrow + (int64_t)r * D * 2 + j * 64 + c * 16, r < G);
            qb[j] = UPPER ? dec_ld16(qrow + (int64_t)(r + 8) * D * 2 + j * 64 + c * 16, r + 8 < G) : make_uint4(0u, 0u, 0u, 0u);
        }
    }
    const char *kbase = reinterpret_cast<const char *>(a.kc) + lo * D * 2;
    const char *vbase = reinterpret_cast<const char *>(a.vc) + lo_v * D * 2;

    float o[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t) o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};

    // K: B operand of the two S^T products (rows row0 + r and row0 + 8 + r);
    // V: rows 2c, 2c + 1, 8 + 2c, 9 + 2c of the block, piece r of each 128-byte half.
    // A 16-row block of K (and of V) is contiguous in the compacted cache, so one lane brings it in
    // with a bulk copy into the warp's own ring: kDecStages blocks per warp are in flight at the
    // price of two instructions each (registers could hold one, and per-lane cp.async costs more
    // to issue than the products of the block).  The ring is private to the warp: its lanes wait on
    // the warp's barriers and lane 0 refills a slot after all lanes have read it.
    constexpr int kBlockBytes = 16 * D * 2;          // one 16-row block of K (or V)
    unsigned char *ring = reinterpret_cast<unsigned char *>(dec_sm) + (size_t)warp * kDecStages * 2 * kBlockBytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(dec_sm) +
                                                  (size_t)NW * kDecStages * 2 * kBlockBytes) + warp * kDecStages;
    if (lane == 0) {
#pragma unroll
        for (int st = 0; st < kDecStages; ++st) dec_bar_init(bars + st);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    auto issue = [&](int row0, int slot) {           // lane 0 only
        if (row0 < end) {
            const uint32_t bytes = (uint32_t)min(16, end - row0) * D * 2;
            dec_bar_expect(bars + slot, 2 * bytes);
            dec_bulk_copy(ring + (size_t)slot * 2 * kBlockBytes, kbase + (int64_t)row0 * D * 2, bytes, bars + slot);
            dec_bulk_copy(ring + (size_t)slot * 2 * kBlockBytes + kBlockBytes, vbase + (int64_t)row0 * D * 2, bytes, bars + slot);
        }
    };
    const int first = begin + warp * 16, stride = NW * 16;
    if (lane == 0)
#pragma unroll
        for (int st = 0; st < kDecStages; ++st) issue(first + st * stride, st);
    int slot = 0;
    uint32_t parity = 0;
    bool timed_out = false;
    for (int row0 = first; row0 < end; row0 += stride) {
        const int vr[4] = {row0 + 2 * c, row0 + 2 * c + 1, row0 + 8 + 2 * c, row0 + 9 + 2 * c};
        if (!dec_bar_wait(bars + slot, parity)) { timed_out = true; break; }
        const unsigned char *kblk = ring + (size_t)slot * 2 * kBlockBytes, *vblk = kblk + kBlockBytes;
        uint4 k1[CH], k2[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            k1[j] = *reinterpret_cast<const uint4 *>(kblk + r * D * 2 + j * 64 + c * 16);
            k2[j] = *reinterpret_cast<const uint4 *>(kblk + (8 + r) * D * 2 + j * 64 + c * 16);
        }
        float s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < CH; ++j) {
            dec_mma(s1, qa[j].x, qb[j].x, qa[j].y, qb[j].y, k1[j].x, k1[j].y);
            dec_mma(s1, qa[j].z, qb[j].z, qa[j].w, qb[j].w, k1[j].z, k1[j].w);
            dec_mma(s2, qa[j].x, qb[j].x, qa[j].y, qb[j].y, k2[j].x, k2[j].y);
            dec_mma(s2, qa[j].z, qb[j].z, qa[j].w, qb[j].w, k2[j].z, k2[j].w);
        }
        // lane (r, c): y[hh][0..3] = logits of head r + 8 hh for rows vr[0..3]
        float y[2][4];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            y[hh][0] = vr[0] < end ? s1[2 * hh] * scale : -INFINITY;
            y[hh][1] = vr[1] < end ? s1[2 * hh + 1] * scale : -INFINITY;
            y[hh][2] = vr[2] < end ? s2[2 * hh] * scale : -INFINITY;
            y[hh][3] = vr[3] < end ? s2[2 * hh + 1] * scale : -INFINITY;
        }
        float f[2], pr[2][4];
        bool grew = false;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float bm = fmaxf(fmaxf(y[hh][0], y[hh][1]), fmaxf(y[hh][2], y[hh][3]));
            bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
            bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));      // row0 is valid, so bm is finite
            const float mn = fmaxf(m[hh], bm);
            f[hh] = dec_ex2(m[hh] - mn);                              // 0 on the first block
            grew |= mn != m[hh];
            m[hh] = mn;
            float sum = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) { pr[hh][i] = dec_ex2(y[hh][i] - mn); sum += pr[hh][i]; }
            l[hh] = l[hh] * f[hh] + sum;
        }
        if (__any_sync(0xffffffffu, grew)) {
#pragma unroll
            for (int t = 0; t < NT; ++t) { o[t][0] *= f[0]; o[t][1] *= f[0]; o[t][2] *= f[1]; o[t][3] *= f[1]; }
        }
        uint32_t ah[4], al[4];                        // a0, a1, a2, a3 of the P operand, high and low terms
        split_pack(pr[0][0], pr[0][1], ah[0], al[0]);
        split_pack(pr[1][0], pr[1][1], ah[1], al[1]);
        split_pack(pr[0][2], pr[0][3], ah[2], al[2]);
        split_pack(pr[1][2], pr[1][3], ah[3], al[3]);
        if (!UPPER) ah[1] = ah[3] = al[1] = al[3] = 0u;
        // rows past the end of a short last block hold what the slot held before: their probabilities
        // are zero, and zero times a stale NaN must not reach the sums
        uint4 v[4][HF];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int hf = 0; hf < HF; ++hf)
                v[i][hf] = vr[i] < end ? *reinterpret_cast<const uint4 *>(vblk + (vr[i] - row0) * D * 2 + hf * 128 + r * 16)
                                       : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int hf = 0; hf < HF; ++hf) {
            const uint32_t w0[4] = {v[0][hf].x, v[0][hf].y, v[0][hf].z, v[0][hf].w};
            const uint32_t w1[4] = {v[1][hf].x, v[1][hf].y, v[1][hf].z, v[1][hf].w};
            const uint32_t w2[4] = {v[2][hf].x, v[2][hf].y, v[2][hf].z, v[2][hf].w};
            const uint32_t w3[4] = {v[3][hf].x, v[3][hf].y, v[3][hf].z, v[3][hf].w};
#pragma unroll
            for (int wi = 0; wi < 4; ++wi)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t sel = e ? 0x7632u : 0x5410u;
                    const uint32_t b0 = __byte_perm(w0[wi], w1[wi], sel), b1 = __byte_perm(w2[wi], w3[wi], sel);
                    const int t = hf * 8 + 2 * wi + e;
                    dec_mma(o[t], ah[0], ah[1], ah[2], ah[3], b0, b1);
                    dec_mma(o[t], al[0], al[1], al[2], al[3], b0, b1);
                }
        }
        __syncwarp();                                // every lane has read the slot
        if (lane == 0) issue(row0 + kDecStages * stride, slot);
        if (++slot == kDecStages) { slot = 0; parity ^= 1u; }
    }
    if (__any_sync(0xffffffffu, timed_out)) {
        if (lane == 0 && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_TIMEOUT);
        for (int st = 0; st < kDecStages; ++st) dec_bar_wait(bars + st, 0) || dec_bar_wait(bars + st, 1);   // let copies in flight land
    }
    __syncthreads();                                 // the ring's memory now takes the warps' records
    // the four column lanes of a head hold partial sums of l
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 1);
        l[hh] += __shfl_xor_sync(0xffffffffu, l[hh], 2);
    }
    float *mine = dec_sm + (size_t)warp * GP * (D + 2);
#pragma unroll
    for (int hh = 0; hh < (UPPER ? 2 : 1); ++hh) {
        float *rec = mine + (r + 8 * hh) * (D + 2);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            rec[t * 8 + 2 * c] = o[t][2 * hh];
            rec[t * 8 + 2 * c + 1] = o[t][2 * hh + 1];
        }
        if (c == 0) { rec[D] = m[hh]; rec[D + 1] = l[hh]; }
    }
    merge_and_store<D, NW, (D == 64 ? kBySize : kPerHead)>(a, dec_sm, GP, G, pc);
}

// fp32 caches and unaligned bf16 pointers: a warp takes rows round-robin, every lane owns
// E = D / 32 columns; the G dot products of a row meet by shuffles.
template <typename T, int D, int GMAX, int NW>
__device__ inline void decode_lanes(const DecArgs &a, const Piece &pc, float *dec_sm)
{
    constexpr int E = D / 32;
    const refree_params &p = a.p;
    const int Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int u = pc.u, s = u / Hkv, g = u % Hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t lo = pc.lo_k, lo_v = pc.lo_v;
    const int begin = pc.x * pc.span, end = min(pc.len, begin + pc.span);
    const float scale = kLog2eDec * rsqrtf((float)D);
    const T *q = static_cast<const T *>(a.q) + ((int64_t)s * p.num_q_heads + g * G) * D;
    const T *kc = static_cast<const T *>(a.kc) + lo * D, *vc = static_cast<const T *>(a.vc) + lo_v * D;
    float qr[GMAX][E], o[GMAX][E], m[GMAX], l[GMAX];
#pragma unroll
    for (int h = 0; h < GMAX; ++h) {
        m[h] = -INFINITY; l[h] = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            qr[h][e] = h < G ? to_float(q[(int64_t)h * D + lane * E + e]) * scale : 0.f;
            o[h][e] = 0.f;
        }
    }
    // RB rows at a time: their loads are in flight together, and their dot products and exponentials do not wait for one
    // another (a row at a time was a chain of some 300 cycles)
    constexpr int RB = GMAX <= 8 ? 4 : 2;
    for (int row0 = begin + warp; row0 < end; row0 += NW * RB) {
        float kf[RB][E], vf[RB][E];
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const bool in = row0 + i * NW < end;
            const int row = in ? row0 + i * NW : end - 1;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                kf[i][e] = to_float(kc[(int64_t)row * D + lane * E + e]);
                const float x = to_float(vc[(int64_t)row * D + lane * E + e]);
                vf[i][e] = in ? x : 0.f;             // (zero times an infinity must not reach the sums)
            }
        }
#pragma unroll
        for (int h = 0; h < GMAX; ++h)
            if (h < G) {
                float y[RB];
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    y[i] = 0.f;
#pragma unroll
                    for (int e = 0; e < E; ++e) y[i] = fmaf(kf[i][e], qr[h][e], y[i]);
                }
#pragma unroll
                for (int ofs = 16; ofs; ofs >>= 1)
#pragma unroll
                    for (int i = 0; i < RB; ++i) y[i] += __shfl_xor_sync(0xffffffffu, y[i], ofs);
                float mn = m[h];
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    if (row0 + i * NW >= end) y[i] = -INFINITY;
                    mn = fmaxf(mn, y[i]);
                }
                const float f = dec_ex2(m[h] - mn);
                float pv[RB];
                l[h] *= f;
#pragma unroll
                for (int e = 0; e < E; ++e) o[h][e] *= f;
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    pv[i] = dec_ex2(y[i] - mn);
                    l[h] += pv[i];
#pragma unroll
                    for (int e = 0; e < E; ++e) o[h][e] = fmaf(pv[i], vf[i][e], o[h][e]);
                }
                m[h] = mn;
            }
    }
    float *mine = dec_sm + (size_t)warp * GMAX * (D + 2);
#pragma unroll
    for (int h = 0; h < GMAX; ++h) {
        float *rec = mine + h * (D + 2);
#pragma unroll
        for (int e = 0; e < E; ++e) rec[lane * E + e] = o[h][e];
        if (lane == 0) { rec[D] = m[h]; rec[D + 1] = l[h]; }
    }
    merge_and_store<D, NW, (D == 64 && GMAX == 4 ? kPerElement : kPerHead)>(a, dec_sm, GMAX, G, pc);
}

// Every thread of the grid waits for what is ahead on the stream before it reads anything.  CLUSTER: a unit's blocks are a
// cluster.
template <int D, int GP, int NW, bool CLUSTER, typename Body>
__device__ inline void decode_block(const DecArgs &a, float *dec_sm, Body body)
{
    dependency_wait();
    trigger_dependents();                            // behind the wait: the merge reads the lengths before its own
    Piece pc;
    int64_t lo_k = 0, lo_v = 0, len64 = 0;
    if (a.mode == kPlanned) {
        pc = make_plan(a, -(int)blockIdx.x - 1);
        if (pc.u >= 0) unit_rows<D>(a, pc.u, lo_k, lo_v, len64);
    } else {
        unit_rows<D>(a, blockIdx.y, lo_k, lo_v, len64);
        pc = unit_piece(a, blockIdx.y, blockIdx.x, clamp_len(a, len64));
    }
    pc.len = clamp_len(a, len64);
    pc.lo_k = lo_k;
    pc.lo_v = lo_v;
    const int Hkv = a.p.num_kv_heads, G = a.p.num_q_heads / Hkv;
    if (pc.u >= 0 && pc.x == 0) {
        if (threadIdx.x == 0 && len64 > a.cap && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_CAPACITY);
        if (pc.nblocks == 0)                // empty segment: the output row is zero
            for (int e = threadIdx.x; e < G * D; e += 32 * NW)
                a.out[((int64_t)(pc.u / Hkv) * a.p.num_q_heads + (pc.u % Hkv) * G) * D + e] = 0.f;
    }
    if (pc.u >= 0 && pc.x < pc.nblocks) body(pc);
    if (CLUSTER) merge_cluster<D, NW>(a, dec_sm, GP, G, pc);
}

template <int D, bool UPPER, int NW>                 // four warps: the blocks of a cluster, eight: those of a cut
__global__ void __launch_bounds__(32 * NW, 8 / NW)
decode_mma_kernel(DecArgs a)
{
    extern __shared__ float dec_sm[];
    decode_block<D, UPPER ? 16 : 8, NW, NW == 4>(a, dec_sm, [&](const Piece &pc) { decode_mma<D, UPPER, NW>(a, pc, dec_sm); });
}

template <typename T, int D, int GMAX, int NW>
__global__ void __launch_bounds__(32 * NW)
decode_lanes_kernel(DecArgs a)
{
    extern __shared__ float dec_sm[];
    decode_block<D, GMAX, NW, false>(a, dec_sm, [&](const Piece &pc) { decode_lanes<T, D, GMAX, NW>(a, pc, dec_sm); });
}

// One block per (unit, head) merges the unit's records and normalises.  kCombineThreads / D groups of threads, one
// thread per column, take every such record; sixteen of them are loaded at once (their (max, sum) words are the same for
// every thread of a group, so the merge weights are simply recomputed by each), so the merge is one round trip to memory
// for up to 32 (d = 128) records, plus one exchange between the groups.  Lengths are read before the wait for the
// attention kernel: its blocks triggered this launch after their own wait, so they were complete.
constexpr int kCombineThreads = 256;
template <int D>
__global__ void __launch_bounds__(kCombineThreads)
decode_combine_kernel(DecArgs a)
{
    constexpr int kGroups = kCombineThreads / D;
    __shared__ float2 ml[kGroups];
    __shared__ float part[kGroups][D];
    const refree_params &p = a.p;
    const int Hkv = p.num_kv_heads, G = p.num_q_heads / Hkv;
    const int u = blockIdx.x / G, h = blockIdx.x % G, s = u / Hkv, g = u % Hkv;
    const int grp = threadIdx.x / D, col = threadIdx.x % D;
    trigger_dependents();
    const Piece pc = a.mode == kPlanned ? make_plan(a, u) : unit_piece(a, u, 0, clamp_len(a, unit_len(a, u)));
    dependency_wait();
    const int nblocks = pc.nblocks;
    if (nblocks <= 1) return;                       // written by the attention kernel itself
    const float *rec0 = a.part + ((int64_t)pc.rec * G + h) * (D + 2);
    const int64_t stride = (int64_t)G * (D + 2);
    float M = -INFINITY, L = 0.f, val = 0.f;
    for (int b0 = grp; b0 < nblocks; b0 += 16 * kGroups) {
        float mm[16], ll[16], vv[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const bool in = b0 + q * kGroups < nblocks;
            const float *rec = rec0 + (int64_t)(in ? b0 + q * kGroups : b0) * stride;
            mm[q] = in ? __ldcg(rec + D) : -INFINITY;
            ll[q] = in ? __ldcg(rec + D + 1) : 0.f;
            vv[q] = in ? __ldcg(rec + col) : 0.f;
        }
        float mn = M;
#pragma unroll
        for (int q = 0; q < 16; ++q) mn = fmaxf(mn, mm[q]);
        const float f0 = M == -INFINITY ? 0.f : dec_ex2(M - mn);
        val *= f0;
        L *= f0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const float f = mm[q] == -INFINITY ? 0.f : dec_ex2(mm[q] - mn);
            val += vv[q] * f;
            L += ll[q] * f;
        }
        M = mn;
    }
    part[grp][col] = val;
    if (col == 0) ml[grp] = make_float2(M, L);
    __syncthreads();
    if (grp == 0) {
        float mt = M, lt = 0.f, vt = 0.f;
#pragma unroll
        for (int q = 1; q < kGroups; ++q) mt = fmaxf(mt, ml[q].x);
#pragma unroll
        for (int q = 0; q < kGroups; ++q) {
            const float f = ml[q].x == -INFINITY ? 0.f : dec_ex2(ml[q].x - mt);
            vt += part[q][col] * f;
            lt += ml[q].y * f;
        }
        a.out[((int64_t)s * p.num_q_heads + g * G + h) * D + native_col(col, a.native)] = lt > 0.f ? vt / lt : 0.f;
    }
}

template <typename Kern>
cudaError_t run_kernel(Kern kern, const DecArgs &a, dim3 grid, int warps, size_t smem, Stream st)
{
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_dependent_cluster(kern, a.mode == kCluster ? a.blocks : 1, grid, dim3(32 * warps), smem, st, a);
}

// Shared memory: the warps' records, then the block's own, then the merge's factors (the staging ring of the mma form uses the
// space before).
constexpr size_t record_smem(int D, int NW, int gp) { return (size_t)(NW + 1) * gp * (D + 2 + 1) * sizeof(float); }

template <typename T, int D, int NW>
cudaError_t run_lanes(const DecArgs &a, dim3 grid, int G, Stream st)
{
    const int gp = G <= 4 ? 4 : (G <= 8 ? 8 : 16);
    const size_t smem = record_smem(D, NW, gp);
    if (gp == 4) return run_kernel(decode_lanes_kernel<T, D, 4, NW>, a, grid, NW, smem, st);
    if (gp == 8) return run_kernel(decode_lanes_kernel<T, D, 8, NW>, a, grid, NW, smem, st);
    return run_kernel(decode_lanes_kernel<T, D, 16, NW>, a, grid, NW, smem, st);
}

template <int D, int NW>
cudaError_t run_mma(const DecArgs &a, dim3 grid, int G, Stream st)
{
    const size_t ring = (size_t)NW * kDecStages * 2 * 16 * D * 2 + (size_t)NW * kDecStages * sizeof(uint64_t);
    const size_t smem = std::max(ring, record_smem(D, NW, G <= 8 ? 8 : 16));
    if (G <= 8) return run_kernel(decode_mma_kernel<D, false, NW>, a, grid, NW, smem, st);
    return run_kernel(decode_mma_kernel<D, true, NW>, a, grid, NW, smem, st);
}

template <int D>
cudaError_t run_attention(const DecArgs &a, dim3 grid, int G, bool f32, Stream st)
{
    if (a.mode == kCluster) return run_mma<D, 4>(a, grid, G, st);      // (only the mma form goes by clusters)
    if (a.native) return run_mma<D, 8>(a, grid, G, st);
    return f32 ? run_lanes<float, D, 8>(a, grid, G, st) : run_lanes<__nv_bfloat16, D, 8>(a, grid, G, st);
}

// How a cache of at most max_rows rows per unit is cut: the mode, and the blocks per unit or of the grid.  Times are of one
// call, 128-element rows, groups of four.
int decode_shape(const refree_params &p, int64_t max_rows, bool mma, int &blocks)
{
    const int64_t U = (int64_t)p.num_seqs * p.num_kv_heads, sms = sm_count();
    // a cluster of at least four blocks, while a block has at most kClusterRows rows: one launch in place of two, and one
    // place in the stream's chain.  24 units of 1000 / 2000 / 5000 rows: 8.6 / 11.2 / 19.2 us, fixed 10.3 / 12.0 / 19.1;
    // 8 units of 2500 / 4096: 10.1 / 12.8, fixed 10.8 / 10.9.  Clusters of two lose: 104 units of 500 rows 11.9, fixed 9.9.
    // (fp32 rows take the issue slots of many warps and keep the fixed cut, which has more of them.)
    const int64_t n = std::min<int64_t>({(max_rows + kMinRows - 1) / kMinRows, (int64_t)kMaxClusterDec, 2 * sms / U});
    if (mma && n >= 4 && (max_rows + n - 1) / n <= kClusterRows) {
        blocks = (int)n;
        return kCluster;
    }
    // about one block per SM (one wave: prologue and merge are paid once), at least a 16-row block per warp
    const int64_t fixed = std::max<int64_t>(1, std::min<int64_t>(sms / U, (max_rows + 127) / 128));
    // Lengths are on the device; what the host has is their sum, if the caller says how many tokens the cache holds.  By the
    // fixed cut the longest unit's blocks set the time; by the plan the rows spread over the SMs, less what its rounding
    // wastes, and a call takes some 2 us longer: its head, and more records of the longest unit to merge.  That is counted in rows
    // of a block: 250 (bf16), 400 with groups of seven and more of 128 elements, whose records are large, 600 with fewer than
    // eight units, whose records are many; 50 of fp32, whose rows take five times as long, but 300 where the fixed cut leaves a
    // unit whole and needs no second launch.  Us a call, fixed and planned: 8 heads, sequences of 20000, 10000 and 5000 rows 42.2
    // and 30.4; of 9000 and 5000 19.5 and 19.3; 13 of 100 to 9000 86.6 and 53.2; 4 heads, eight of 2531 to 16214 48.4 and 32.2,
    // three of 6000 to 3000 14.8 and 15.4; 2 heads, 30000 and 3000 18.0 and 20.1; 2 heads of groups of 16, 6000 to 100 13.0 and
    // 13.9, 12000 to 80 in one 15.3 and 19.7; fp32, 8 heads, 900, 2600 and 300 36.4 and 23.6; 16 heads, six of 1200 to 200 31.7
    // and 38.4, of 5000 and 1000 173 and 65.  (Of 716 batches of 2 to 20 sequences the rule takes the slower form by more than
    // 5 % in 44, in five of them the plan.)
    const int64_t rows = p.kv_tokens * p.num_kv_heads * (p.k_stride_seq != 0 ? p.num_seqs : 1);     // kv_tokens is per sequence, or of all
    const int64_t more = mma ? (U < 8 ? 600 : p.head_dim == 128 && p.num_q_heads / p.num_kv_heads >= 7 ? 400 : 250) : fixed == 1 ? 300 : 50;
    if (p.num_seqs > 1 && p.kv_tokens > 0 && U <= kPlanUnits && U < sms &&
        rows / (sms - (2 * U <= sms ? U / 2 : U)) + more < (max_rows + fixed - 1) / fixed) {
        blocks = (int)sms;
        return kPlanned;
    }
    blocks = (int)fixed;
    return kFixed;
}

}  // namespace

size_t decode_workspace_bytes(const refree_params &p, int64_t max_rows)
{
    // (whatever the mode of a call: the larger of the fixed and the planned form's records)
    const int64_t U = (int64_t)p.num_seqs * p.num_kv_heads;
    return (size_t)std::max<int64_t>(U, sm_count()) * (p.num_q_heads / p.num_kv_heads) * (p.head_dim + 2) * sizeof(float) + 256;
}

cudaError_t launch_decode_attention(const refree_params &p, const void *q_new, const void *k_c, const void *v_c,
                                    const int64_t *offsets, int64_t max_rows, float *out, void *workspace,
                                    int32_t *dev_status, Stream st, const int32_t *seq_start,
                                    const int32_t *seq_len, const int32_t *lengths, bool anchor_back)
{
    DecArgs a;
    a.p = p;
    a.q = q_new; a.kc = k_c; a.vc = v_c;
    a.offsets = offsets;
    a.seq_start = seq_start; a.seq_len = seq_len; a.lengths = lengths;
    a.anchor_back = anchor_back ? 1 : 0;
    a.out = out;
    a.part = static_cast<float *>(workspace);
    a.dev_status = dev_status;
    const bool f32 = p.dtype == REFREE_DTYPE_F32;
    const bool aligned = !((reinterpret_cast<uintptr_t>(q_new) | reinterpret_cast<uintptr_t>(k_c) |
                            reinterpret_cast<uintptr_t>(v_c)) & 15);
    a.native = !f32 && aligned ? 1 : 0;
    a.mode = decode_shape(p, max_rows, a.native != 0, a.blocks);
    a.span = (int)std::max<int64_t>(16, ((max_rows + a.blocks - 1) / a.blocks + 15) / 16 * 16);
    a.cap = (int)std::min<int64_t>(a.mode == kFixed ? (int64_t)a.span * a.blocks : (max_rows + 15) / 16 * 16, INT_MAX / 2);
    const int U = p.num_seqs * p.num_kv_heads, G = p.num_q_heads / p.num_kv_heads;
    const dim3 grid = a.mode == kPlanned ? dim3(a.blocks) : dim3(a.blocks, U);
    cudaError_t e = p.head_dim == 64 ? run_attention<64>(a, grid, G, f32, st) : run_attention<128>(a, grid, G, f32, st);
    count_launches(1);
    if (e != cudaSuccess || a.mode == kCluster || a.blocks == 1) return e;
    e = p.head_dim == 64 ? launch_dependent(decode_combine_kernel<64>, dim3(U * G), dim3(kCombineThreads), 0, st, a)
                         : launch_dependent(decode_combine_kernel<128>, dim3(U * G), dim3(kCombineThreads), 0, st, a);
    count_launches(1);
    return e;
}

}  // namespace refree
