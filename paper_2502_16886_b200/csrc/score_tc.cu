// Tensor-core scoring path (steps S1-S3) for bf16 caches with head_dim 128.
//
// The window logits S = Q K^T are the one dense contraction of the pass; they run
// on tcgen05.mma with the accumulator in tensor memory, operands staged in shared
// memory by TMA (128-byte swizzle, no multicast).  A row's softmax normaliser needs
// all of the row, and the column sums need every row's normaliser, so the logits are
// formed twice (storing them would cost more HBM traffic than K itself):
//
//   pass 1  D[row, position] = Q_blk K_tile^T (M = 128 rows, N = 128 positions): Z[row] = sum over the positions of a
//           run of tiles of 2^(y - c[row]), per half of a tile's columns; the pairs (c, Z) go to the workspace
//   pass 2  on entering a unit, L[row] = log2 sum_i 2^(y_i) is merged from those pairs; then D[position, row] =
//           K_tile Q^T (M = 128 positions, N = up to 256 rows) and
//           a'[i] = sum over the rows that see i of 2^(y - L[row])  (Eq. 2)
//
// Both passes use the same shared-memory images of Q and K (K-major, so either can be the A or the B operand); only
// the roles swap, which puts each pass's reduction inside a lane.
//
// Order of the sums.  A budget follows from fp32 scores, and about one unit in 10^4 lies so near a tie that the last bits
// of a score decide it (two units of 19200: criterion within 4e-9 of the threshold).  So every sum here has one order,
// whatever else is in the launch: a row's terms inside a run in the order of the tiles, the runs cut at the ranges of a
// single layer (see Split), records merged in their order, a position's terms by halves of a product's columns.  A layer
// gets the same bits from every entry point, in every group of layers, with every workspace.
//
// Why this form.  The epilogue (a multiply-add, an exponential and an addition per logit and pass) takes longer than the
// products; the two groups of eight epilogue warps take products in turn and run out of step, so that one sums while the
// other waits for its next accumulator.  An accumulator is handed back as soon as its last values sit in registers.  In
// pass 1 a group has two accumulators of 128 columns: pairs of tiles as one N = 256 product per group are held until the
// second tile's logits are read, and the product that follows comes late (us a pass: four layers of the ragged batch of
// eight, 448 rows, 757 and 725 as here; eight of 20K positions, 512 rows, 783 and 769; 16 of 8K, 256 rows, 443 and 437).
// All sixteen warps sharing every product is faster where runs are short (16 layers of 8K 396, of 2K 154 and here 180;
// eight of 32K 671 and here 681; the ragged batch 738), but takes a row's or position's terms in another order, and
// layers that share a launch then round differently from the same layers one by one.
//
// Persistent CTAs (one per SM) take contiguous ranges of (unit, tile) items; warp 16 issues TMA, warp 17 issues MMA,
// warps 0-15 are the epilogue, warp 18 moves rows of another layer, warp 19 adds the warps' shares of a column sum,
// stores the scores and the records of the stopping rule.  Every wait is bounded: on a timeout the CTA records
// REFREE_DEV_TIMEOUT, stops issuing work, and falls through to the common exit where tensor memory is released.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "refree_internal.cuh"
#include "select_groups.cuh"

namespace refree {
namespace {

constexpr int kEpiWarps = 16;
constexpr int kThreadsTc = (kEpiWarps + 4) * 32;     // + TMA warp, MMA warp, copy warp, finishing warp
constexpr int kMaxCopySlots = 10;
constexpr int kMaxCopyUnits = 1024;                 // units whose running budget sum fits the CTA's table
constexpr int kD = 128;
constexpr int kHalfBytes = kTile * 128;          // one 64-column half of a 128-row tile: 16 KB
constexpr int kTileBytes = 2 * kHalfBytes;       // 32 KB
constexpr int kMaxRowsTc = 512;
constexpr int kMaxCtas = 256;
constexpr float kLog2e = 1.4426950408889634f;
// 2^100: the sum of a tile's half above this is taken again with a fresh reference.  A row has fewer than 2^25 such sums, so
// neither a run's nor the row's total can leave the range of fp32.
constexpr float kZLimit = 1.2676506e30f;

// ------------------------------------------------------------------ PTX ------
__device__ inline uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ inline void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ inline void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ inline void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ inline bool mbar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false (and raises the CTA's abort flag) when it gives up.
__device__ inline bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        if (mbar_try(bar, parity)) return true;
        if (it > 64) {
            if (*abort_flag) return false;
            __nanosleep(it > 4096 ? 256 : 32);
        }
    }
    *abort_flag = 1;
    return false;
}
// The same for a whole warp, which goes on or gives up as one.
__device__ inline bool mbar_wait_warp(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}
__device__ inline void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ inline void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1) : "memory");
}
// K tiles carry an L2 eviction priority: the row pass reads a tile first (keep it: the column pass comes back for
// it), the column pass reads it last (let it go first).
__device__ inline void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2, uint64_t pol)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "l"(pol) : "memory");
}
__device__ inline void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2, int c3, uint64_t pol)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(pol) : "memory");
}

__device__ inline void tmem_alloc(uint32_t *dst_smem, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// One lane of a converged warp, the same one every time.
__device__ inline bool elect_one()
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
    return ok != 0;
}
// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate; issued by one thread.
// The two shared-memory descriptors are passed as their low words (start address
// and leading offset, see desc_lo) plus the common high word: one thread issues
// every MMA of the CTA, so the issue path is kept to a few instructions.
__device__ inline void umma_bf16(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                 uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
                 "setp.ne.b32 p, %5, 0;\n\t"
                 "mov.b64 da, {%1, %3};\n\t"
                 "mov.b64 db, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// The mbarrier receives one arrival once every MMA issued so far by this thread has completed.
__device__ inline void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Tensor-memory loads are split into issue and wait so that the next chunk can be
// in flight while the current one is consumed.  The wait names the destination
// registers as in/out operands: the compiler must not read them before it.
#define RF_OUT16(r, o) "=r"(r[o+0]), "=r"(r[o+1]), "=r"(r[o+2]), "=r"(r[o+3]), "=r"(r[o+4]), "=r"(r[o+5]), "=r"(r[o+6]), "=r"(r[o+7]), \
                       "=r"(r[o+8]), "=r"(r[o+9]), "=r"(r[o+10]), "=r"(r[o+11]), "=r"(r[o+12]), "=r"(r[o+13]), "=r"(r[o+14]), "=r"(r[o+15])
#define RF_IO16(r, o) "+r"(r[o+0]), "+r"(r[o+1]), "+r"(r[o+2]), "+r"(r[o+3]), "+r"(r[o+4]), "+r"(r[o+5]), "+r"(r[o+6]), "+r"(r[o+7]), \
                      "+r"(r[o+8]), "+r"(r[o+9]), "+r"(r[o+10]), "+r"(r[o+11]), "+r"(r[o+12]), "+r"(r[o+13]), "+r"(r[o+14]), "+r"(r[o+15])
__device__ inline void tmem_ld_issue(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : RF_OUT16(r, 0) : "r"(taddr) : "memory");
}
__device__ inline void tmem_ld_issue(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : RF_OUT16(r, 0), RF_OUT16(r, 16) : "r"(taddr) : "memory");
}
__device__ inline void tmem_ld_wait(uint32_t (&r)[16]) { asm volatile("tcgen05.wait::ld.sync.aligned;" : RF_IO16(r, 0) :: "memory"); }
__device__ inline void tmem_ld_wait(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" : RF_IO16(r, 0), RF_IO16(r, 16) :: "memory");
}
__device__ inline float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 B
// apart, groups of 8 rows 1024 B apart (the layout TMA writes with SWIZZLE_128B).
// Low word: start address / 16 in bits 0-13, leading byte offset (unused with
// swizzle) in bits 16-29.  A byte offset o (multiple of 16) inside the operand
// adds o / 16 to the low word.  High word: stride byte offset / 16 in bits 0-13,
// descriptor version 1 in bits 14-15, swizzle mode 2 (128 B) in bits 29-31.
__device__ inline uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128.
__host__ __device__ inline uint32_t make_idesc(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// ---------------------------------------------------------------- shapes -----
struct TcShape {
    int R;        // query rows per unit: G * window
    int Rpad;     // rows of the shared-memory Q image (multiple of 128)
    int rblocks;  // 128-row blocks: pass-1 products per tile (A operands)
    int cblocks;  // pass-2 products per tile: 1 up to 256 rows, else 2
    int ncol;     // pass-2 columns (rows of Q) per product: a multiple of 32, cblocks * ncol >= R
    int stages;   // K tile ring depth
    int slots;    // pass 2: tiles whose column sums may wait for the finishing warp (a power of two)
    int rank4;    // K tensor map has a sequence axis
};

// What the consumers of an item (one tile of one unit) need to know about it.  The TMA thread walks the
// items and leaves one record per item in a ring in shared memory, written before the item's K tile is
// requested; the MMA thread and the epilogue warps read it after the barriers that order them behind
// that request, instead of each walking the item list in registers.
struct ItemInfo {
    int32_t u;        // unit = (layer of the group * sequences + sequence) * KV heads + KV head
    int32_t g;        // row of the score array: layer * KV heads + KV head
    int32_t n;        // length of the sequence
    int32_t tile;     // tile index inside the sequence
    int32_t ntiles;   // tiles of the sequence
    int32_t pack;     // positions before the sequence in the packed score array
    int32_t ib;       // pass 2: index of the unit's first item; pass 1: index of the run's record
    int32_t flags;    // kNewUnit .. below
};
// kNewUnit: first item of its unit in this pass of the CTA (Q is loaded again); kRunLast: the last of a run (pass 1: the
// tiles of one unit in one range, see Ranges); kPassLast: nothing more is loaded in this pass.
constexpr int32_t kNewUnit = 1, kRunLast = 2, kPassLast = 4;
constexpr int kInfoRing = 16;   // the TMA thread runs at most ring stages + accumulators in flight ahead of the epilogue
// Pass 2: tiles whose column sums wait for the finishing warp.  That warp is slower per tile than the sixteen
// epilogue warps together while rows are being copied beside them, and catches up under the row pass that follows:
// the ring is deep enough to let it fall behind instead of holding the epilogue back.
constexpr int kStageSlots = 8;
constexpr int kRuleList = 16;   // units whose stopping rule a CTA evaluates when it has left its passes
struct StageSlot {
    ItemInfo info;                            // the staged tile's record, copied beside its sums
    float sum[4][kTile];                      // partial column sums (share = product * 2 + half of its columns)
};

// Per-sequence tables of the CTA behind the tail, sized by the number of sequences:
// pack[B + 1], tiles[B + 1] (running sums of lengths and of tiles), len[B], start[B], ne[B + 1] (non-empty
// sequences before each).
struct SeqView {
    const int32_t *pack, *tiles, *len, *start, *ne;
};

struct ItemTc {
    int s, g, n, tok0, pack;
    int tile, ntiles;      // tile index inside the sequence, tiles of the sequence
};

// Item of one layer: ordered (sequence, KV head, tile), so consecutive items mostly share a unit.
__device__ inline ItemTc decode_item_tc(const SeqView &sv, int B, int Hkv, int item)
{
    int lo = 0, hi = B;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((int64_t)sv.tiles[mid] * Hkv <= item) lo = mid; else hi = mid;
    }
    ItemTc it;
    it.s = lo;
    it.ntiles = sv.tiles[lo + 1] - sv.tiles[lo];
    const int rem = item - sv.tiles[lo] * Hkv;
    it.g = rem / it.ntiles;
    it.tile = rem % it.ntiles;
    it.n = sv.len[lo];
    it.tok0 = sv.start[lo];
    it.pack = sv.pack[lo];
    return it;
}

// Ranges: the split of one layer's items over `ctas` CTAs.  A change of unit inside a range costs about as much as a few
// tiles (the accumulators drain, the new unit's normalisers are merged from the partials, Q is reloaded), so what the
// ranges get equal shares of is  items + pen * (changes of unit): item i of the o-th non-empty unit sits at
// v = i + pen * o, and range c takes the items with v in [c V / ctas, (c + 1) V / ctas).  `pen` stays below the
// share of a range, so none is empty.
// A launch over one layer gives every CTA one range.  The layers of a group are cut into the same ranges, and a CTA takes
// several that follow one another: the sums of pass 1 begin and end with the ranges, so that a layer's scores are the same
// bits whatever other layers share its launch.
constexpr int kUnitChangeTiles = 3;
struct Split {
    int items, ctas, pen, Hkv;      // of one layer
    int64_t V;
};

// a / b for non-negative operands; 32-bit where both fit (a 64-bit division is a routine of some hundred instructions)
__device__ inline int64_t div_nonneg(int64_t a, int64_t b)
{
    return ((uint64_t)(a | b) >> 32) == 0 ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
}

__device__ inline Split make_split(const SeqView &sv, int B, int Hkv, int grid)
{
    Split sp;
    sp.Hkv = Hkv;
    sp.items = sv.tiles[B] * Hkv;
    sp.ctas = max(1, min(grid, sp.items));
    sp.pen = max(0, min(kUnitChangeTiles, sp.items / sp.ctas - 1));
    sp.V = (int64_t)sp.items + (int64_t)sp.pen * max(0, sv.ne[B] * Hkv - 1);
    return sp;
}

// first item of range c (c == ctas: one past the last item)
__device__ inline int range_begin(const Split &sp, const SeqView &sv, int B, int c)
{
    const int64_t t = div_nonneg((int64_t)c * sp.V + sp.ctas - 1, sp.ctas);      // smallest v of the range's share
    if (t >= sp.V) return sp.items;
    const int Hkv = sp.Hkv;
    auto key = [&](int q) { return (int64_t)sv.tiles[q] * Hkv + (int64_t)sp.pen * sv.ne[q] * Hkv; };   // v of a sequence's first item
    int lo = 0, hi = B;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (key(mid) <= t) lo = mid; else hi = mid;
    }
    const int nt = sv.tiles[lo + 1] - sv.tiles[lo];
    const int64_t rel = t - key(lo);
    const int g = (int)min((int64_t)(Hkv - 1), div_nonneg(rel, nt + sp.pen));
    const int64_t r = rel - (int64_t)g * (nt + sp.pen);
    // a v that falls between two units belongs to the first item of the second
    return sv.tiles[lo] * Hkv + g * nt + (int)min(r, (int64_t)nt);
}

// Range that holds item x of unit u (of one layer).
__device__ inline int range_of_item(const Split &sp, const SeqView &sv, int x, int u)
{
    const int ord = sv.ne[u / sp.Hkv] * sp.Hkv + u % sp.Hkv;
    const int64_t v = (int64_t)x + (int64_t)sp.pen * ord;
    return (int)min((int64_t)(sp.ctas - 1), div_nonneg(v * sp.ctas, sp.V));
}

// Items of a group are numbered layer after layer.  First item of range q, counted over the layers of the group.
__device__ inline int group_range_begin(const Split &sp, const SeqView &sv, int B, int q)
{
    const int l = q / sp.ctas;
    return l * sp.items + range_begin(sp, sv, B, q - l * sp.ctas);
}
// The ranges and items of this CTA in a pass over a group: items [first, first + count), ranges from `q` on; the first of those
// ends before item `first_end`.
struct Share { int q, first, count, first_end; };
// What a CTA does, found by one warp behind the sequence tables and shared: the lanes look up the range boundaries side by
// side, and the unit that pass 2 begins with (its last item's) and the ranges that hold its records.  Every warp by itself, one
// boundary after the other, took 2.2 us at the head of every launch.  (With the first launch of a call chained to what is
// ahead of it, us: four layers one by one of 4K positions, 128 rows 162 -> 144, of 2K, 256 rows 159 -> 144; 16 layers of 8K as
// a run 388 -> 378.)
struct Plan {
    Split sp;
    Share a, b;                               // pass 1, pass 2
    int b_layer, b_unit, b_ib, b_ntiles, b_tile, b_clo, b_chi;
};
__device__ inline void make_plan(Plan &plan, const SeqView &sv, int B, int Hkv, int split_ctas, int layers_a, int layers_b)
{
    const int lane = threadIdx.x & 31;
    const Split sp = make_split(sv, B, Hkv, split_ctas);
    // lanes 0 to 2: first, next and last boundary of pass 1; 3 to 5: of pass 2
    const int layers = lane < 3 ? layers_a : layers_b, Q = layers * sp.ctas, ctas = min((int)gridDim.x, Q);
    const bool on = lane < 6 && (int)blockIdx.x < ctas && sp.items > 0;
    int q = 0, x = 0;
    if (on) {
        const int which = lane < 3 ? lane : lane - 3;
        q = (int)div_nonneg((int64_t)(blockIdx.x + (which == 2 ? 1 : 0)) * Q, ctas) + (which == 1 ? 1 : 0);
        x = group_range_begin(sp, sv, B, q);
    }
    Share sh[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        sh[i].q = __shfl_sync(0xffffffffu, q, 3 * i);
        sh[i].first = __shfl_sync(0xffffffffu, x, 3 * i);
        sh[i].first_end = __shfl_sync(0xffffffffu, x, 3 * i + 1);
        sh[i].count = __shfl_sync(0xffffffffu, x, 3 * i + 2) - sh[i].first;
    }
    int layer = 0, u = 0, ib = 0, nt = 1, tile = 0, c = 0;
    if (sh[1].count > 0) {
        const int last = sh[1].first + sh[1].count - 1;
        layer = last / sp.items;
        const ItemTc it = decode_item_tc(sv, B, Hkv, last - layer * sp.items);
        u = it.s * Hkv + it.g;
        ib = sv.tiles[it.s] * Hkv + it.g * it.ntiles;
        nt = it.ntiles;
        tile = it.tile;
        c = range_of_item(sp, sv, lane == 0 ? ib : ib + nt - 1, u);
    }
    const int chi = __shfl_sync(0xffffffffu, c, 1);
    if (lane == 0) {
        plan.sp = sp;
        plan.a = sh[0]; plan.b = sh[1];
        plan.b_layer = layer; plan.b_unit = u; plan.b_ib = ib; plan.b_ntiles = nt; plan.b_tile = tile; plan.b_clo = c; plan.b_chi = chi;
    }
}
struct TcSmemTail {
    uint64_t k_full[4], k_empty[4], q_full, q_empty, epi_bar;
    uint64_t p1_full[4], p1_empty[4];         // pass 1: accumulator (group * 2 + slot), 128 tensor-memory columns each
    uint64_t p2_full[2], p2_empty[2];         // pass 2: accumulators of 256 columns, one per group of eight warps
    uint64_t chunk_ready[kStageSlots];        // pass 2: every share of a tile has been staged
    uint64_t stage_free[kStageSlots];         // pass 2: the finishing warp has read the slot
    uint64_t c_full[kMaxCopySlots];           // row copy: a piece has landed in its slot
    uint32_t tmem_base;
    int abort_flag;
    Plan plan;
    int rule_n;                               // units waiting in rule_unit / rule_max
    int rule_unit[kRuleList];
    uint32_t rule_max[kRuleList];             // bit pattern of the unit's largest score
    BlockRuleShared<kThreadsTc> rule;
    alignas(16) ItemInfo info[kInfoRing];
    alignas(16) float lse[kMaxRowsTc];        // pass 2: log2-sum-exp of the unit's rows
};

// Pass 1 leaves one record per (range, unit, half of a tile's columns); record of range c and unit u of layer l.
__device__ inline int record_index(int l, int c, int u, int U) { return l * (kMaxCtas + U) + c + u; }

struct TcArgs {
    refree_params p;
    TcShape sh;
    const int32_t *seq_start, *seq_len;
    int split_ctas;      // ranges of a layer, at most
    // Pass 1 writes the partials of group `a`, pass 2 reads those of group `b` and writes its scores.
    int layers_a, layers_b;
    float2 *part_a;      // [layers (kMaxCtas + units)][2][Rpad]: one (c, Z) per (range, unit, half of the columns) and row
    const float2 *part_b;
    GroupPartial *groups; // nullable: per 32 positions, exact sum of squared scores for the stopping rule
    float *scores;
    int64_t total_tokens;
    int32_t *dev_status;
    // Stopping rule inside the launch (position ranking per head): the CTA whose finishing warp completes a unit's
    // last tile (a ticket per unit) evaluates the rule from the unit's records when it has left its passes.  All nullable.
    int32_t *sel_lengths[kMaxBatch];   // budgets out, per layer of the group
    Cut *sel_cuts;             // [units]
    uint32_t *tickets;         // [2 units] tiles finished per unit, then the unit's largest score; zero when the launch begins
    uint32_t *tickets_next;    // [2 units] those of the launch that follows, cleared by this one
    int dependent;             // launched with programmatic stream serialization: 1, behind another launch of the call; 2, its first
    TcCopyJob cj;          // rows of earlier layers to move while these are scored (nslots == 0: none)
};
struct TcMaps {
    CUtensorMap q[kMaxBatch], k[kMaxBatch];
};

// budget of unit u of the group that pass 2 works on
__device__ inline int32_t *unit_length(const TcArgs &a, int u)
{
    const int U = a.p.num_seqs * a.p.num_kv_heads, l = u / U;
    return a.sel_lengths[l] + (u - l * U);
}

// Barrier among the epilogue warps, built on an mbarrier so that it is bounded like
// every other wait of the kernel (one arrival per warp).
__device__ inline bool epi_sync(TcSmemTail &tl, uint32_t &phase)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&tl.epi_bar);
    const bool ok = mbar_wait(&tl.epi_bar, phase, &tl.abort_flag);
    phase ^= 1;
    return ok;
}

// Loop state that survives from one pass to the other when both run in one launch.  `icount` numbers the
// items a role has gone through in this launch (both passes): its low bits index the info ring.  `p2` counts the products
// of pass 2.
struct RingState { int stage = 0; uint32_t kphase = 0, qphase = 0, icount = 0; };
struct MmaState : RingState { uint32_t p2 = 0; bool first = true; };
struct EpiState { uint32_t ephase = 0, icount = 0; };

// --------------------------------------------------------- producer / MMA -----
// Loads one pass's tiles, run by run (a run: the CTA's tiles of one unit, in pass 1 those of one range).
// The column pass walks a CTA's items backwards: the row pass before it (at the end of the launch before) left its last K tiles in L2, and those are asked for first.
template <bool PASS1>
__device__ inline void producer_loop(const TcArgs &a, const TcMaps &maps,
                                     unsigned char *smem_q, unsigned char *smem_k, TcSmemTail &tl, const SeqView &sv,
                                     const Split &sp, const Share &share, RingState &rs)
{
    const TcShape &sh = a.sh;
    const int B = a.p.num_seqs, Hkv = a.p.num_kv_heads, G = a.p.num_q_heads / Hkv, U = B * Hkv;
    const int item0 = share.first, item1 = share.first + share.count;
    uint64_t pol;
    if (PASS1) asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    bool ok = true;
    int q = share.q, range_end = share.first_end, last_u = -1;      // pass 1: the range of item x, and the item it ends at
    for (int x = PASS1 ? item0 : item1 - 1; ok && x >= item0 && x < item1;) {
        const int layer = x / sp.items;
        const ItemTc it = decode_item_tc(sv, B, Hkv, x - layer * sp.items);
        if (PASS1 && x >= range_end) range_end = group_range_begin(sp, sv, B, ++q + 1);      // (no range is empty)
        const int g = it.g, u = layer * U + it.s * Hkv + g;
        const CUtensorMap *const mapq = &maps.q[layer], *const mapk = &maps.k[layer];
        const int run = PASS1 ? min(it.ntiles - it.tile, range_end - x) : min(it.tile + 1, x - item0 + 1);
        const bool last_run = PASS1 ? x + run >= item1 : x - run < item0;
        const int ib = PASS1 ? record_index(layer, q - layer * sp.ctas, it.s * Hkv + g, U)
                             : layer * sp.items + sv.tiles[it.s] * Hkv + g * it.ntiles;
        const bool new_unit = u != last_u;
        last_u = u;
        auto load = [&](unsigned char *dst, int half, int tile) {
            if (sh.rank4)
                tma_load_4d(dst, mapk, &tl.k_full[rs.stage], half * 64, it.tok0 + tile * kTile, g, it.s, pol);
            else
                tma_load_3d(dst, mapk, &tl.k_full[rs.stage], half * 64, it.tok0 + tile * kTile, g, pol);
        };
        for (int j = 0; j < run && ok; ++j) {
            const int tile = PASS1 ? it.tile + j : it.tile - j;
            const bool last = j + 1 == run;
            // the ring entry was last used sixteen items ago, which every consumer has long left behind
            ItemInfo &inf = tl.info[rs.icount++ & (kInfoRing - 1)];
            const int flags = (j == 0 && new_unit ? kNewUnit : 0) | (last ? kRunLast : 0) | (last && last_run ? kPassLast : 0);
            // The K tile first: the MMA thread learns of a unit change from the record, which it reads once
            // the tile has landed, and only then gives the Q image back.
            ok = mbar_wait_warp(&tl.k_empty[rs.stage], rs.kphase ^ 1, &tl.abort_flag);
            if (!ok) break;
            if (elect_one()) {
                inf.u = u; inf.g = layer * Hkv + g; inf.n = it.n; inf.tile = tile; inf.ntiles = it.ntiles; inf.pack = it.pack;
                inf.ib = ib;
                inf.flags = flags;
                mbar_expect_tx(&tl.k_full[rs.stage], (uint32_t)kTileBytes);      // (release) orders the record before the tile
                unsigned char *dst = smem_k + (size_t)rs.stage * kTileBytes;
                load(dst, 0, tile);
                load(dst + kHalfBytes, 1, tile);
            }
            __syncwarp();
            if (new_unit && j == 0) {
                ok = mbar_wait_warp(&tl.q_empty, rs.qphase ^ 1, &tl.abort_flag);
                if (!ok) break;
                if (elect_one()) {
                    mbar_expect_tx(&tl.q_full, (uint32_t)sh.Rpad * 256u);
                    const int row0 = (it.s * a.p.num_q_heads + g * G) * a.p.window;
                    for (int h = 0; h < 2; ++h)
                        for (int b = 0; b < sh.rblocks; ++b)
                            tma_load_2d(smem_q + (size_t)h * sh.Rpad * 128 + (size_t)b * kHalfBytes, mapq, &tl.q_full,
                                        h * 64, row0 + b * kTile);
                }
                __syncwarp();
                rs.qphase ^= 1;
            }
            if (++rs.stage == sh.stages) { rs.stage = 0; rs.kphase ^= 1; }
        }
        x += PASS1 ? run : -run;
    }
    // Before leaving, let every copy this thread started land (bounded): the ring's
    // full barriers complete only when their bytes have arrived.
    if (!ok) {
        for (int s2 = 0; s2 < sh.stages; ++s2)
            for (uint32_t itw = 0; itw < 4096; ++itw) {
                if (mbar_try(&tl.k_full[s2], 0) || mbar_try(&tl.k_full[s2], 1)) break;
                __nanosleep(64);
            }
    }
}

// A unit begins: its Q must have landed (and the one before is given back with the products issued so far).
__device__ inline bool mma_new_unit(TcSmemTail &tl, MmaState &ms)
{
    if (!ms.first && elect_one()) umma_commit(&tl.q_empty);
    ms.first = false;
    if (!mbar_wait_warp(&tl.q_full, ms.qphase, &tl.abort_flag)) return false;
    ms.qphase ^= 1;
    tc_fence_after();
    return true;
}

// Pass 1: D[row, position] = Q_blk K_tile^T.  Row block rb goes to accumulator pair rb & 1 (the group of epilogue warps
// that takes it), which alternates between its two accumulators of 128 columns: the product of a pair's next block runs
// while the epilogue reads the current one.
__device__ inline void mma_loop_pass1(const TcArgs &a, unsigned char *smem_q, unsigned char *smem_k, TcSmemTail &tl,
                                      uint32_t tmem_base, MmaState &ms)
{
    const TcShape &sh = a.sh;
    const uint32_t q_lo = desc_lo(smem_u32(smem_q)), k_lo = desc_lo(smem_u32(smem_k));
    const uint32_t q_half = (uint32_t)(sh.Rpad * 128) >> 4;      // distance between the two 64-column halves of Q
    const uint32_t idesc = make_idesc(kTile);
    uint32_t cnt0 = 0, cnt1 = 0;                                 // products per pair
    for (;;) {
        if (!mbar_wait_warp(&tl.k_full[ms.stage], ms.kphase, &tl.abort_flag)) return;
        tc_fence_after();
        const int flags = tl.info[ms.icount++ & (kInfoRing - 1)].flags;
        if ((flags & kNewUnit) && !mma_new_unit(tl, ms)) return;
        const uint32_t kt = k_lo + (uint32_t)ms.stage * (kTileBytes >> 4);
        for (int rb = 0; rb < sh.rblocks; ++rb) {
            const uint32_t pair = (uint32_t)(rb & 1), cnt = pair ? cnt1 : cnt0, acc = 2u * pair + (cnt & 1u);
            // a pair covers the columns of an accumulator of pass 2: the last product left there must have been handed back
            const uint32_t before = (ms.p2 + 1u - pair) >> 1;
            if (cnt == 0 && before > 0 && !mbar_wait_warp(&tl.p2_empty[pair], (before - 1u) & 1u, &tl.abort_flag)) return;
            if (!mbar_wait_warp(&tl.p1_empty[acc], ((cnt >> 1) & 1u) ^ 1u, &tl.abort_flag)) return;
            tc_fence_after();
            const uint32_t qa = q_lo + (uint32_t)rb * (kHalfBytes >> 4);
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint32_t h = kk >> 2, ko = (kk & 3) * 2;      // 32 bytes per K step of 16
                    umma_bf16(tmem_base + acc * 128u, qa + h * q_half + ko, kt + h * (kHalfBytes >> 4) + ko, kDescHi, idesc, kk > 0);
                }
                umma_commit(&tl.p1_full[acc]);
                if (rb + 1 == sh.rblocks) umma_commit(&tl.k_empty[ms.stage]);
            }
            __syncwarp();
            if (pair) ++cnt1; else ++cnt0;
        }
        if (++ms.stage == sh.stages) { ms.stage = 0; ms.kphase ^= 1; }
        if (flags & kPassLast) break;
    }
}

// Pass 2: D[position, row] = K_tile Q^T, `ncol` rows of Q per product.  `more`: pass 1 follows in this launch; Q is then
// given back with the last product, so that the next Q travels while the epilogue still works on this one's.
__device__ inline void mma_loop_pass2(const TcArgs &a, unsigned char *smem_q, unsigned char *smem_k, TcSmemTail &tl,
                                      uint32_t tmem_base, MmaState &ms, bool more)
{
    const TcShape &sh = a.sh;
    const uint32_t q_lo = desc_lo(smem_u32(smem_q)), k_lo = desc_lo(smem_u32(smem_k));
    const uint32_t q_half = (uint32_t)(sh.Rpad * 128) >> 4;
    const uint32_t idesc = make_idesc(sh.ncol);
    for (;;) {
        if (!mbar_wait_warp(&tl.k_full[ms.stage], ms.kphase, &tl.abort_flag)) return;
        tc_fence_after();
        const int flags = tl.info[ms.icount++ & (kInfoRing - 1)].flags;
        if ((flags & kNewUnit) && !mma_new_unit(tl, ms)) return;
        const uint32_t ka = k_lo + (uint32_t)ms.stage * (kTileBytes >> 4);
        for (int cb = 0; cb < sh.cblocks; ++cb) {
            const uint32_t buf = ms.p2 & 1u;
            if (!mbar_wait_warp(&tl.p2_empty[buf], ((ms.p2 >> 1) & 1u) ^ 1u, &tl.abort_flag)) return;
            tc_fence_after();
            const uint32_t qb = q_lo + (uint32_t)cb * (uint32_t)(sh.ncol * 128 >> 4);
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint32_t h = kk >> 2, ko = (kk & 3) * 2;
                    umma_bf16(tmem_base + buf * 256u, ka + h * (kHalfBytes >> 4) + ko, qb + h * q_half + ko, kDescHi, idesc, kk > 0);
                }
                umma_commit(&tl.p2_full[buf]);
                if (cb + 1 == sh.cblocks) umma_commit(&tl.k_empty[ms.stage]);
            }
            __syncwarp();
            ++ms.p2;
        }
        if (++ms.stage == sh.stages) { ms.stage = 0; ms.kphase ^= 1; }
        if (flags & kPassLast) break;
    }
    if (more) {
        if (elect_one()) umma_commit(&tl.q_empty);
        ms.first = true;
    }
}

// ------------------------------------------------------------- epilogues -----
// Give an accumulator back: every load of this warp from it has landed.
__device__ inline void release_acc(uint64_t *bar, int lane)
{
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

// Pass 1: lane = query row, 64 logits of the row in registers.
template <bool MASKED>
__device__ inline float row_sum_regs(const uint32_t (&ra)[32], const uint32_t (&rb)[32], float scale, float cref, int limit)
{
    float z0 = 0.f, z1 = 0.f;
    const float nc = -cref;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const uint32_t (&cur)[32] = c ? rb : ra;
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            float e0 = ex2(fmaf(__uint_as_float(cur[i]), scale, nc));
            float e1 = ex2(fmaf(__uint_as_float(cur[i + 1]), scale, nc));
            if (MASKED) {
                e0 = (c * 32 + i < limit) ? e0 : 0.f;
                e1 = (c * 32 + i + 1 < limit) ? e1 : 0.f;
            }
            z0 += e0;
            z1 += e1;
        }
    }
    return z0 + z1;
}
__device__ inline float row_max_regs(const uint32_t (&ra)[32], const uint32_t (&rb)[32], float scale, int limit)
{
    float m = -INFINITY;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const uint32_t (&cur)[32] = c ? rb : ra;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (c * 32 + i < limit) m = fmaxf(m, __uint_as_float(cur[i]) * scale);
    }
    return m;
}

// Two groups of eight warps take the row blocks in turn (block rb goes to group rb & 1); inside a group a warp is
// (lane quarter) x (half of each tile's columns), and adds its half of tile after tile of a run in their order.
__device__ inline void epilogue_pass1(const TcArgs &a, TcSmemTail &tl, uint32_t tmem_base, EpiState &es)
{
    const TcShape &sh = a.sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group = (warp >> 2) & 1, half = warp >> 3, lane_base = (warp & 3) * 32;
    if (group >= sh.rblocks) return;             // a single row block: all of it is the first group's
    const float scale = kLog2e * rsqrtf((float)kD);
    const int w = a.p.window;
    uint32_t cnt = 0;                            // products this group has taken
    // running reference and sum of this lane's rows (row blocks group and group + 2) over its half of the columns
    float cref[2] = {-INFINITY, -INFINITY}, zsum[2] = {0.f, 0.f};
    int rmod[2];
    bool rows_here[2];                           // a warp without rows of the unit hands its products back unread
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int row0 = (group + 2 * j) * kTile + lane_base;
        rmod[j] = (row0 + lane) % w;             // offset of the row's query inside the window
        rows_here[j] = row0 < sh.R;
    }
    for (;;) {
        const ItemInfo *inf = &tl.info[es.icount++ & (kInfoRing - 1)];
        int flags = 0, tile_start = 0, n = 0, rec = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int rb = group + 2 * j;
            if (rb >= sh.rblocks) continue;
            const uint32_t acc = 2u * (uint32_t)group + (cnt & 1u);
            if (!mbar_wait(&tl.p1_full[acc], (cnt >> 1) & 1u, &tl.abort_flag)) return;
            ++cnt;
            tc_fence_after();
            if (j == 0) { flags = inf->flags; tile_start = inf->tile * kTile; n = inf->n; rec = inf->ib; }   // valid once a product of the item is
            if (!rows_here[j]) {
                release_acc(&tl.p1_empty[acc], lane);
                continue;
            }
            const uint32_t taddr = tmem_base + acc * 128u + (uint32_t)(half * 64) + ((uint32_t)lane_base << 16);
            uint32_t ra[32], rb2[32];
            tmem_ld_issue(taddr, ra);
            tmem_ld_issue(taddr + 32, rb2);
            tmem_ld_wait(ra);
            tmem_ld_wait(rb2);
            // the logits are in registers: the accumulator goes back to the MMA warp before any arithmetic
            release_acc(&tl.p1_empty[acc], lane);
            const bool full = tile_start + kTile <= n - w + 1;      // tile wholly before the window
            // visible positions of the tile, [0, limit), up to this row's own position, inside this warp's columns.  (Lanes past the
            // unit's rows go along with the others: what they add up is never stored.)
            int limit = full ? kTile : n - w + rmod[j] - tile_start + 1;
            limit = max(0, min(64, limit - half * 64));
            const bool uniform = __all_sync(0xffffffffu, limit == 64);
            bool need_max = (cref[j] == -INFINITY) && limit > 0;
            float zt = 0.f;
            for (int attempt = 0; attempt < 2; ++attempt) {
                if (__any_sync(0xffffffffu, need_max)) {
                    const float m = row_max_regs(ra, rb2, scale, limit);
                    if (need_max && m > cref[j]) {
                        zsum[j] = (cref[j] == -INFINITY) ? 0.f : zsum[j] * ex2(cref[j] - m);
                        cref[j] = m;
                    }
                }
                zt = uniform ? row_sum_regs<false>(ra, rb2, scale, cref[j], limit)
                             : row_sum_regs<true>(ra, rb2, scale, cref[j], limit);
                need_max = !(zt <= kZLimit) && limit > 0;       // overflow against a stale reference
                if (attempt == 1 || !__any_sync(0xffffffffu, need_max)) break;
            }
            if (limit > 0) zsum[j] += zt;
        }
        if (flags & kRunLast) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int row = (group + 2 * j) * kTile + lane_base + lane;
                if (group + 2 * j < sh.rblocks && row < sh.R)
                    a.part_a[((int64_t)rec * 2 + half) * sh.Rpad + row] = make_float2(cref[j], zsum[j]);
                cref[j] = -INFINITY;
                zsum[j] = 0.f;
            }
        }
        if (flags & kPassLast) break;
    }
}

// Pass 2: lane = position; 16 rows' terms 2^(y - L[row]).
// r0 = the first row; pos_gap = i - (n - w): row r sees position i iff (r mod w) >= pos_gap.
template <bool MASKED>
__device__ inline void col_sum16(const uint32_t (&cur)[16], float scale, const float *lse, int r0, int R, int w,
                                 int pos_gap, float &s0, float &s1)
{
    int rloc = MASKED ? r0 % w : 0;
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float4 L = *reinterpret_cast<const float4 *>(lse + r0 + i);
        float e[4];
        e[0] = ex2(fmaf(__uint_as_float(cur[i]), scale, -L.x));
        e[1] = ex2(fmaf(__uint_as_float(cur[i + 1]), scale, -L.y));
        e[2] = ex2(fmaf(__uint_as_float(cur[i + 2]), scale, -L.z));
        e[3] = ex2(fmaf(__uint_as_float(cur[i + 3]), scale, -L.w));
        if (MASKED) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (rloc < pos_gap || r0 + i + j >= R) e[j] = 0.f;     // hidden by causality, or padding
                if (++rloc == w) rloc = 0;
            }
        }
        s0 += e[0] + e[2];
        s1 += e[1] + e[3];
    }
}

// One product's share of a warp: `nch` chunks of 16 columns (rows of Q) come from tensor memory one chunk at a
// time, the next in flight while 2^(y - L[row]) is summed over the current one; the accumulator is handed back
// as soon as the last load has landed.
template <bool MASKED>
__device__ inline float col_product(int nch, uint32_t taddr, uint64_t *empty_bar, int lane, float scale, const float *lse,
                                    int r0, int R, int w, int pos_gap)
{
    uint32_t b0[16], b1[16];
    float s0 = 0.f, s1 = 0.f;
    if (nch == 0) {                                                 // none of the unit's rows
        release_acc(empty_bar, lane);
        return 0.f;
    }
    tmem_ld_issue(taddr, b0);
    tmem_ld_wait(b0);
    for (int c = 0; c < nch; c += 2) {
        if (c + 1 < nch) tmem_ld_issue(taddr + 16 * (c + 1), b1); else release_acc(empty_bar, lane);
        col_sum16<MASKED>(b0, scale, lse, r0 + 16 * c, R, w, pos_gap, s0, s1);
        if (c + 1 < nch) {
            tmem_ld_wait(b1);
            if (c + 2 < nch) tmem_ld_issue(taddr + 16 * (c + 2), b0); else release_acc(empty_bar, lane);
            col_sum16<MASKED>(b1, scale, lse, r0 + 16 * (c + 1), R, w, pos_gap, s0, s1);
            if (c + 2 < nch) tmem_ld_wait(b0);
        }
    }
    return s0 + s1;
}

// L[row] = log2 sum over the row of 2^y for the rows of unit u of a layer, merged from the (reference, sum) pairs that
// pass 1 left per (range, unit, column half), in ascending record order (the same in every CTA that needs the unit).
// Called by all epilogue threads; [c_lo, c_hi] = the ranges that hold the unit's items.
__device__ inline bool merge_unit_lse(const TcArgs &a, TcSmemTail &tl, int layer, int u, int c_lo, int c_hi, uint32_t &ephase)
{
    const TcShape &sh = a.sh;
    const int tid = threadIdx.x;
    // two threads per row when there are enough threads: even and odd records, then one exchange
    const int per_row = 2 * sh.R <= kEpiWarps * 32 ? 2 : 1;
    const int r = tid / per_row, sub = tid % per_row;
    float M = -INFINITY, Z = 0.f;
    if (r < sh.R) {
        const float2 *rec = a.part_b + (int64_t)record_index(layer, c_lo, u, a.p.num_seqs * a.p.num_kv_heads) * 2 * sh.Rpad + r;
        const int nrec = 2 * (c_hi - c_lo + 1);             // records: (range, column half)
        constexpr int kBatch = 20;                          // independent loads in flight per thread: mostly all there are
        for (int s0 = sub; s0 < nrec; s0 += kBatch * per_row) {
            float2 pr[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                pr[q] = s0 + q * per_row < nrec ? __ldcg(rec + (int64_t)(s0 + q * per_row) * sh.Rpad) : make_float2(0.f, 0.f);
            // Z 2^M + y 2^x, record after record, at the larger of the two references.  What a step scales by depends on
            // the references alone, so the exponentials do not wait for the sums.
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const bool up = pr[q].y > 0.f && pr[q].x > M;
                const float f = ex2(up ? M - pr[q].x : pr[q].x - M);
                if (pr[q].y > 0.f) Z = fmaf(up ? Z : pr[q].y, f, up ? pr[q].y : Z);
                if (up) M = pr[q].x;
            }
        }
    }
    if (per_row == 2) {
        const float M2 = __shfl_xor_sync(0xffffffffu, M, 1), Z2 = __shfl_xor_sync(0xffffffffu, Z, 1);
        // (even records) then (odd records), in that order on both lanes
        const float Ma = sub ? M2 : M, Za = sub ? Z2 : Z, Mb = sub ? M : M2, Zb = sub ? Z : Z2;
        if (Zb > 0.f) {
            if (Za > 0.f) {
                if (Mb > Ma) { Z = Za * ex2(Ma - Mb) + Zb; M = Mb; }
                else { Z = Za + Zb * ex2(Mb - Ma); M = Ma; }
            } else { Z = Zb; M = Mb; }
        } else { Z = Za; M = Ma; }
    }
    // a row that sees nothing adds 2^(-inf) = 0
    if (r < sh.R && sub == 0) tl.lse[r] = Z > 0.f ? M + log2f(Z) : INFINITY;
    // columns past the unit's rows (padding of the last product) never count
    for (int rr = sh.R + tid; rr < sh.cblocks * sh.ncol; rr += kEpiWarps * 32) tl.lse[rr] = INFINITY;
    return epi_sync(tl, ephase);
}

// Pass 2, the sixteen epilogue warps.  Two groups of eight warps take the products in turn (product j goes to
// group j & 1 and to accumulator j & 1), so the groups run out of step: while one waits for its next accumulator,
// stages a tile or refills its pipeline, the other keeps the exponential units busy.  Inside a group a warp is
// (lane quarter) x (half of the product's columns); it leaves its share of the tile's column sums in a staging
// slot, and the finishing warp adds the shares.
__device__ inline void epilogue_pass2(const TcArgs &a, TcSmemTail &tl, StageSlot *stage, const SeqView &sv, uint32_t tmem_base,
                                      int item0, int nitems, const Split &sp, EpiState &es)
{
    const TcShape &sh = a.sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group = (warp >> 2) & 1, half = warp >> 3, lane_base = (warp & 3) * 32;
    const float scale = kLog2e * rsqrtf((float)kD);
    const int w = a.p.window, Hkv = a.p.num_kv_heads;
    const int pos_in_tile = lane_base + lane;
    const int c_width = sh.ncol >> 1, c_begin = half * c_width;     // this warp's columns of a product
    const uint32_t taddr = tmem_base + (uint32_t)group * 256u + (uint32_t)c_begin + ((uint32_t)lane_base << 16);
    const int slot_shift = 31 - __clz(sh.slots);
    uint32_t gcnt = 0;                                             // products this group has taken
    int next_change = 0;                                           // item (relative) at which the next unit begins
    for (int item = 0; item < nitems; ++item) {
        const ItemInfo *inf = &tl.info[es.icount++ & (kInfoRing - 1)];
        if (item == next_change) {   // `item` counts the pass's items in the order they come: from the CTA's last one backwards
            // A unit begins: all sixteen warps meet (the two groups share L), whichever group takes the item's
            // products.  The unit is looked up in the sequence tables, not in the item's record, which a warp
            // that takes none of the item's products has no barrier to wait for.  The normalisers do not wait
            // for the tile either: the partials come from the row pass, not from anything this pass loads.
            const Plan &pl = tl.plan;
            int layer = pl.b_layer, u = pl.b_unit, tile = pl.b_tile, c_lo = pl.b_clo, c_hi = pl.b_chi;
            if (item > 0) {
                const int x = item0 + (nitems - 1 - item);
                layer = x / sp.items;
                const ItemTc it = decode_item_tc(sv, a.p.num_seqs, Hkv, x - layer * sp.items);
                const int ib = sv.tiles[it.s] * Hkv + it.g * it.ntiles;
                u = it.s * Hkv + it.g;
                tile = it.tile;
                c_lo = range_of_item(sp, sv, ib, u);
                c_hi = range_of_item(sp, sv, ib + it.ntiles - 1, u);
                if (!epi_sync(tl, es.ephase)) return;              // nobody still reads the previous unit's L
            }
            if (!merge_unit_lse(a, tl, layer, u, c_lo, c_hi, es.ephase)) return;
            next_change = item + tile + 1;                         // the unit's earlier tiles follow
        }
        for (int cb = 0; cb < sh.cblocks; ++cb) {
            const uint32_t j = (uint32_t)item * (uint32_t)sh.cblocks + (uint32_t)cb;      // product index in this pass
            if ((int)(j & 1u) != group) continue;
            if (!mbar_wait(&tl.p2_full[group], gcnt & 1u, &tl.abort_flag)) return;
            ++gcnt;
            tc_fence_after();
            // the item's record is valid once one of its products is
            const int tile_start = inf->tile * kTile, n = inf->n;
            const int pos_gap = tile_start + pos_in_tile - (n - w);
            // chunks with rows of the unit among this warp's columns (the last product is padded: 400 rows, whose products of 224
            // went through the masked sums tile after tile, four layers of 8000 positions x 8 heads 196 us, 166 this way)
            const int r0 = cb * sh.ncol + c_begin, nch = (max(0, min(c_width, sh.R - r0)) + 15) >> 4;
            // tile wholly before the window and wholly inside the sequence: every row sees every position
            const bool full = tile_start + kTile <= n - w + 1 && r0 + 16 * nch <= max(sh.R, r0);
            const float part = full ? col_product<false>(nch, taddr, &tl.p2_empty[group], lane, scale, tl.lse, r0, sh.R, w, pos_gap)
                                    : col_product<true>(nch, taddr, &tl.p2_empty[group], lane, scale, tl.lse, r0, sh.R, w, pos_gap);
            // the slot's previous tile has been read by the finishing warp
            const uint32_t slot = (uint32_t)item & (uint32_t)(sh.slots - 1);
            if (!mbar_wait(&tl.stage_free[slot], (((uint32_t)item >> slot_shift) & 1u) ^ 1u, &tl.abort_flag)) return;
            stage[slot].sum[cb * 2 + half][pos_in_tile] = part;
            // the tile's record travels with its sums (the ring it came from may be reused before the tile is finished)
            if (cb == 0 && half == 0 && lane_base == 0 && lane < 8)
                reinterpret_cast<uint32_t *>(&stage[slot].info)[lane] = reinterpret_cast<const uint32_t *>(inf)[lane];
            __syncwarp();
            if (lane == 0) mbar_arrive(&tl.chunk_ready[slot]);
        }
    }
}

// Pass 2, the finishing warp: a'[i] = (sum of the warps' shares, in a fixed order) / (G * rows that see i)  (Eq. 2), the score
// store, and per 32 positions the record the stopping rule reads.
__device__ inline void finisher_pass2(const TcArgs &a, TcSmemTail &tl, StageSlot *stage, const SeqView &sv, int nitems)
{
    const int lane = threadIdx.x & 31;
    const int w = a.p.window;
    const float g = (float)(a.p.num_q_heads / a.p.num_kv_heads);
    const int slot_shift = 31 - __clz(a.sh.slots);
    // This CTA's tiles of a unit are counted once, when its run of them ends: the warp that brings the unit's count
    // to its number of tiles sees every other tile's scores and records (fenced before their counts were added).
    // The rule is some ten dependent loads, scans and shuffles, 28 us for one warp beside sixteen that keep the exponential
    // unit busy.  So the unit goes on the CTA's list, for all its threads when they have left the passes; but the warp
    // evaluates it itself where it has time for that, beyond 256 query rows (two products a tile, and a long row pass behind)
    // and with a unit for every fourth CTA at most.  Measured, us a pass, by the list and by the warp: ragged batch of eight
    // x 4 layers, 448 rows (32 units a launch) 722 and 710, 20K x 8, 512 rows (16) 762 and 758, two layers of 17.5K, 512 rows
    // (32) 239 and 229; 32K x 8, 256 rows (16) 674 and 674, 32K x 8, 64 rows (8) 219 and 241, 2K x 16, 256 rows (64) 180 and 188.
    int run_u = -1, run_ntiles = 0, run_ib = 0, run_tiles = 0;
    uint32_t run_max = 0;                       // largest score of the run (bit pattern)
    const int Hkv = a.p.num_kv_heads, U1 = a.p.num_seqs * Hkv, U = U1 * a.layers_b;
    const bool two_products = a.sh.cblocks > 1;
    const int listed = two_products && 4 * U <= (int)gridDim.x ? 0 : kRuleList;
    auto close_run = [&]() {
        if (run_u < 0 || run_tiles == 0) return;
        if (lane == 0) atomicMax(&a.tickets[U + run_u], run_max);      // the unit's largest score, beside its count
        __threadfence();
        __syncwarp();
        uint32_t old = 0;
        if (lane == 0) old = atomicAdd(&a.tickets[run_u], (uint32_t)run_tiles);
        old = __shfl_sync(0xffffffffu, old, 0);
        if ((int)old + run_tiles == run_ntiles) {
            __threadfence();
            uint32_t umax = 0;
            if (lane == 0) umax = atomicMax(&a.tickets[U + run_u], 0u);
            umax = __shfl_sync(0xffffffffu, umax, 0);
            const int k = tl.rule_n;                                       // only this warp appends
            if (k < listed) {
                __syncwarp();
                if (lane == 0) { tl.rule_unit[k] = run_u; tl.rule_max[k] = umax; tl.rule_n = k + 1; }
                __syncwarp();
            } else {
                const int l = run_u / U1, u = run_u - l * U1, s = u / Hkv, g = u - s * Hkv;
                const Cut cut = select_unit_from_groups_warp(a.p, a.scores + (int64_t)(l * Hkv + g) * a.total_tokens + sv.pack[s],
                                                             sv.len[s], a.groups + (int64_t)run_ib * 4, umax);
                if (lane == 0) {
                    *unit_length(a, run_u) = cut.b;
                    if (a.sel_cuts) a.sel_cuts[run_u] = cut;
                }
            }
        }
        run_tiles = 0;
    };
    for (int t = 0; t < nitems; ++t) {
        const uint32_t slot = (uint32_t)t & (uint32_t)(a.sh.slots - 1);
        if (!mbar_wait(&tl.chunk_ready[slot], ((uint32_t)t >> slot_shift) & 1u, &tl.abort_flag)) return;
        const ItemInfo *inf = &stage[slot].info;
        const int n = inf->n, tile = inf->tile;
        const int inf_u = inf->u, inf_ntiles = inf->ntiles, inf_ib = inf->ib;     // the record may be reused after the slot is freed
        float *dst = a.scores + (int64_t)inf->g * a.total_tokens + inf->pack;
        GroupPartial *grp = a.groups ? a.groups + ((int64_t)inf->ib + tile) * 4 : nullptr;
        uint32_t tile_max = 0;
        // A lane takes four consecutive positions: the shares come as 16-byte loads, the scores leave as one 16-byte store
        // where their row starts on 16 bytes, and the 32 positions of a record are eight neighbouring lanes.  (Few
        // instructions that go through the memory pipe: the sixteen epilogue warps keep it busy, and this warp paces the pass.)
        const int p0 = 4 * lane, i0 = tile * kTile + p0;
        float tot[4];
        {
            const float4 x = *reinterpret_cast<const float4 *>(&stage[slot].sum[0][p0]);
            const float4 y = *reinterpret_cast<const float4 *>(&stage[slot].sum[1][p0]);
            tot[0] = x.x + y.x; tot[1] = x.y + y.y; tot[2] = x.z + y.z; tot[3] = x.w + y.w;
        }
        if (two_products) {
            const float4 x = *reinterpret_cast<const float4 *>(&stage[slot].sum[2][p0]);
            const float4 y = *reinterpret_cast<const float4 *>(&stage[slot].sum[3][p0]);
            tot[0] += x.x; tot[1] += x.y; tot[2] += x.z; tot[3] += x.w;
            tot[0] += y.x; tot[1] += y.y; tot[2] += y.z; tot[3] += y.w;
        }
        float sc[4];
        uint32_t bits[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i0 + k;
            const int cnt_i = max(1, min(min(w, n), n - i));
            sc[k] = i < n ? tot[k] / ((float)cnt_i * g) : 0.f;
            bits[k] = (i < n && isfinite(sc[k])) ? mag_bits(sc[k]) : 0u;
            if (i < n && !isfinite(sc[k]) && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_NONFINITE);
        }
        if (i0 + 3 < n && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
            *reinterpret_cast<float4 *>(dst + i0) = make_float4(sc[0], sc[1], sc[2], sc[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i0 + k < n) dst[i0 + k] = sc[k];
        }
        if (grp) {
            // 32 positions = lanes 8q .. 8q + 7: largest score, and the exact squares summed at a scale set by it
            uint32_t mx = max(max(bits[0], bits[1]), max(bits[2], bits[3]));
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const int shift = kGroupShift - 2 * max(1, (int)(mx >> 23));
            unsigned long long sq = sq_fixed(bits[0], shift) + sq_fixed(bits[1], shift) + sq_fixed(bits[2], shift) +
                                    sq_fixed(bits[3], shift);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if ((lane & 7) == 0) { GroupPartial gp; gp.max_bits = mx; gp.pad = 0u; gp.sum = sq; grp[lane >> 3] = gp; }
            tile_max = __reduce_max_sync(0xffffffffu, mx);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&tl.stage_free[slot]);
        if (a.tickets) {
            if (inf_u != run_u) {
                close_run();
                run_u = inf_u; run_ntiles = inf_ntiles; run_ib = inf_ib; run_tiles = 0;
                run_max = 0;
            }
            ++run_tiles;
            run_max = max(run_max, tile_max);
        }
    }
    if (a.tickets) close_run();
}

// ------------------------------------------------------------- row copy -----
// Compaction of another layer by one warp of the scoring CTA (position ranking: the kept rows of a unit
// are rows [0, head) and [n - (b - head), n) of its cache, contiguous in memory when a unit's rows are).
// Destination rows are cut into pieces of 32 (or 8) rows; piece k belongs to CTA k mod grid, and inside the CTA
// to one lane of the warp, which owns a slot of shared memory.  A piece travels global -> shared -> global
// with the bulk-copy engine (no tensor map, no multicast): the load is signalled on the slot's mbarrier,
// the store is a bulk group.  Nothing here touches the registers or pipes of the scoring warps.
__device__ inline void copy_loop(const TcArgs &a, TcSmemTail &tl, const SeqView &sv, unsigned char *smem_c, int32_t *coff)
{
    const TcCopyJob &cj = a.cj;
    const int lane = threadIdx.x & 31;
    const int Hkv = a.p.num_kv_heads, U = a.p.num_seqs * Hkv, units = cj.layers * U;
    // running sum of the budgets over all layers (clamped to [0, n]); a budget out of range is reported
    int carry = 0;
    bool bad = false;
    for (int base = 0; base < units; base += 32) {
        const int x_u = base + lane;
        int b = 0;
        if (x_u < units) {
            const int l = x_u / U, u = x_u - l * U;
            b = cj.lengths[l][u];
            const int n = sv.len[u / Hkv];
            if (b < 0 || b > n) { bad = true; b = max(0, min(b, n)); }
        }
        const int x = warp_incl_scan(b);
        if (x_u < units) coff[x_u] = carry + x - b;
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) coff[units] = carry;
    __syncwarp();
    const int rows = carry;
    if (blockIdx.x == 0)
        for (int l = 0; l < cj.layers; ++l) {
            for (int u = lane; u <= U; u += 32) cj.offsets_out[l][u] = coff[l * U + u] - coff[l * U];
            bad |= (int64_t)(coff[(l + 1) * U] - coff[l * U]) > cj.capacity_rows;
        }
    bad = __any_sync(0xffffffffu, bad);
    if (blockIdx.x == 0 && lane == 0 && bad && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_CAPACITY);
    const int nslots = cj.nslots;
    if (lane >= nslots || rows <= 0) return;

    // Lane j owns slot j and every nslots-th piece of this CTA, and runs its own load -> wait -> store -> wait
    // chain; the lanes drift apart, which spreads the requests in time.
    const int64_t k_tok = a.p.k_stride_tok * 2, v_tok = a.p.v_stride_tok * 2;      // bytes (bf16)
    const int piece_rows = cj.piece_rows;
    const int64_t pieces_per_array = ((int64_t)rows + piece_rows - 1) / piece_rows, pieces = 2 * pieces_per_array;
    int64_t next = blockIdx.x + (int64_t)lane * gridDim.x;      // next piece of this lane
    const int64_t step = (int64_t)nslots * gridDim.x;
    int r_cur = 0, r_end = 0, u_cur = 0, arr = 0;      // rows [r_cur, r_end) of the current piece still to cut
    unsigned char *slot = smem_c + (size_t)lane * piece_rows * (kD * 2);
    uint64_t *bar = &tl.c_full[lane];
    // the moved rows are used once: they should not push the scored layer's K tiles out of L2
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    uint32_t loads = 0;
    bool ok = true;
    while (ok) {
        // the next run of rows that is contiguous in source and destination
        bool has = true;
        if (r_cur >= r_end) {
            if (next >= pieces) {
                has = false;
            } else {
                arr = next >= pieces_per_array ? 1 : 0;
                const int64_t pk = next - (arr ? pieces_per_array : 0);
                next += step;
                r_cur = (int)(pk * piece_rows);
                r_end = (int)min((int64_t)r_cur + piece_rows, (int64_t)rows);
                int lo = 0, hi = units;                         // largest u with coff[u] <= r_cur
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (coff[mid] <= r_cur) lo = mid; else hi = mid;
                }
                u_cur = lo;
            }
        }
        if (!has) break;
        unsigned char *dst = nullptr;
        uint32_t bytes = 0;
        if (has) {
            while (coff[u_cur + 1] <= r_cur) ++u_cur;           // skip units that keep nothing (r_cur < rows = coff[units])
            const int b = coff[u_cur + 1] - coff[u_cur], t = r_cur - coff[u_cur];
            const int layer = u_cur / U, u = u_cur - layer * U, sq = u / Hkv, g = u - sq * Hkv;
            const int n = sv.len[sq], head = min(b, min(a.p.sink, n));
            int src_row, run;
            if (t < head) { src_row = t; run = head - t; }
            else { src_row = n - b + t; run = b - t; }
            run = min(run, r_end - r_cur);
            const int64_t row = r_cur - coff[layer * U], room = cj.capacity_rows - row;     // in the layer's output
            if (room <= 0) { r_cur += run; continue; }
            run = (int)min((int64_t)run, room);
            const int64_t tok = (int64_t)sv.start[sq] + src_row;
            const unsigned char *src =
                arr == 0 ? cj.k[layer] + ((int64_t)sq * a.p.k_stride_seq + (int64_t)g * a.p.k_stride_head) * 2 + tok * k_tok
                         : cj.v[layer] + ((int64_t)sq * a.p.v_stride_seq + (int64_t)g * a.p.v_stride_head) * 2 + tok * v_tok;
            dst = (arr ? cj.v_out[layer] : cj.k_out[layer]) + row * (kD * 2);
            bytes = (uint32_t)run * (kD * 2);
            r_cur += run;
            mbar_expect_tx(bar, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                         ::"r"(smem_u32(slot)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol) : "memory");
            ok = mbar_wait(bar, loads & 1u, &tl.abort_flag);
            ++loads;
            if (ok) {
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;"
                             ::"l"(dst), "r"(smem_u32(slot)), "r"(bytes), "l"(pol) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            }
        }
        ok = ok && !tl.abort_flag;
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------- kernels ----
// The stopping rule of the units on the CTA's list, by all threads of the CTA.
__device__ inline void evaluate_rules(const TcArgs &a, TcSmemTail &tl, const SeqView &sv)
{
    const int Hkv = a.p.num_kv_heads, U1 = a.p.num_seqs * Hkv, items = sv.tiles[a.p.num_seqs] * Hkv;
    for (int k = 0; k < tl.rule_n; ++k) {
        const int u = tl.rule_unit[k], l = u / U1, s = (u - l * U1) / Hkv, g = (u - l * U1) - s * Hkv;
        const int nt = sv.tiles[s + 1] - sv.tiles[s];
        const UnitRule ur(a.p, a.scores + (int64_t)(l * Hkv + g) * a.total_tokens + sv.pack[s], sv.len[s],
                          a.groups + ((int64_t)l * items + (int64_t)sv.tiles[s] * Hkv + (int64_t)g * nt) * 4, tl.rule_max[k]);
        block_unit_rule<kThreadsTc>(ur, tl.rule, unit_length(a, u), a.sel_cuts ? a.sel_cuts + u : nullptr);
    }
}

// MODE 1: pass 1 alone; 2: pass 2 alone; 3: pass 2 of one group of layers (`_b`), then pass 1 of the next (`_a`) - the
// steady state of a run of layers.  The partials that pass 2 reads were completed by the launch before.
template <int MODE>
__global__ void __launch_bounds__(kThreadsTc, 1)
score_tc_kernel(const __grid_constant__ TcMaps maps_a, const __grid_constant__ TcMaps maps_b, const __grid_constant__ TcArgs a)
{
    constexpr bool P1 = MODE != 2, P2 = MODE != 1;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const TcShape &sh = a.sh;
    unsigned char *smem_q = smem;
    unsigned char *smem_k = smem + (size_t)sh.Rpad * 256;
    unsigned char *smem_c = smem_k + (size_t)sh.stages * kTileBytes;        // pieces of the row copy
    StageSlot *stage = reinterpret_cast<StageSlot *>(smem_c + (size_t)a.cj.nslots * a.cj.piece_rows * (kD * 2));
    TcSmemTail &tl = *reinterpret_cast<TcSmemTail *>(stage + sh.slots);
    int32_t *tab = reinterpret_cast<int32_t *>(&tl + 1);
    const int B = a.p.num_seqs;
    int32_t *t_pack = tab, *t_tiles = tab + (B + 1), *t_len = tab + 2 * (B + 1), *t_start = tab + 2 * (B + 1) + B;
    int32_t *t_ne = tab + 4 * B + 2;
    int32_t *coff = tab + 5 * B + 3;             // row copy: running sum of the budgets, units + 1 entries
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == kEpiWarps * 32) {
        for (int l = 0; P1 && l < a.layers_a; ++l) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&maps_a.q[l]) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&maps_a.k[l]) : "memory");
        }
        for (int l = 0; P2 && l < a.layers_b; ++l) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&maps_b.q[l]) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&maps_b.k[l]) : "memory");
        }
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < 4; ++s) { mbar_init(&tl.k_full[s], 1); mbar_init(&tl.k_empty[s], 1); }
        mbar_init(&tl.q_full, 1);
        mbar_init(&tl.q_empty, 1);
        // a group of eight warps hands an accumulator back
        for (int b = 0; b < 4; ++b) { mbar_init(&tl.p1_full[b], 1); mbar_init(&tl.p1_empty[b], kEpiWarps / 2); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tl.p2_full[b], 1); mbar_init(&tl.p2_empty[b], kEpiWarps / 2); }
        for (int b = 0; b < kStageSlots; ++b) {
            mbar_init(&tl.chunk_ready[b], sh.cblocks * (kEpiWarps / 2));
            mbar_init(&tl.stage_free[b], 1);
        }
        mbar_init(&tl.epi_bar, kEpiWarps);
        for (int b = 0; b < kMaxCopySlots; ++b) mbar_init(&tl.c_full[b], 1);
        tl.abort_flag = 0;
        tl.rule_n = 0;
        fence_barrier_init();
    }
    SeqView sv;
    sv.pack = t_pack; sv.tiles = t_tiles; sv.len = t_len; sv.start = t_start; sv.ne = t_ne;
    // the first launch of a call reads nothing before what is ahead of it on the stream has completed
    if (a.dependent == 2) asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int t = threadIdx.x; t < B; t += kThreadsTc) t_start[t] = a.seq_start[t];
    if (warp == 1) {                             // running sums over the sequences, 32 at a time
        int32_t pa = 0, ti = 0, ne = 0;
        for (int s0 = 0; s0 < B; s0 += 32) {
            const int s = s0 + lane;
            const int n = s < B ? max(a.seq_len[s], 0) : 0, nt = ceil_div(n, kTile);
            const int pi = warp_incl_scan(n), tinc = warp_incl_scan(nt);
            const unsigned nonempty = __ballot_sync(0xffffffffu, n > 0);
            if (s < B) {
                t_len[s] = n;
                t_pack[s] = pa + pi - n;
                t_tiles[s] = ti + tinc - nt;
                t_ne[s] = ne + __popc(nonempty & ((1u << lane) - 1u));
            }
            pa += __shfl_sync(0xffffffffu, pi, 31);
            ti += __shfl_sync(0xffffffffu, tinc, 31);
            ne += __popc(nonempty);
        }
        if (lane == 0) { t_pack[B] = pa; t_tiles[B] = ti; t_ne[B] = ne; }
        __syncwarp();
        // a layer's items in min(SMs, items) ranges, so that no range is empty
        make_plan(tl.plan, sv, B, a.p.num_kv_heads, a.split_ctas, P1 ? a.layers_a : 0, P2 ? a.layers_b : 0);
    }
    if (warp == kEpiWarps + 1) tmem_alloc(&tl.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tl.tmem_base;
    const Split sp = tl.plan.sp;
    const Share sh_a = tl.plan.a, sh_b = tl.plan.b;       // pass 1, pass 2
    const int na = sh_a.count, b0 = sh_b.first, nb = sh_b.count;

    // A run of layers: the launch that follows may put a CTA on an SM as soon as this one's has left it (programmatic
    // dependent launch; 8K positions: 41 us a layer against 45 without).  What such an early CTA does before griddepcontrol.wait must not need this launch's results:
    // its setup, and the loads of Q and K and the products on them, which are the caller's inputs.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool inputs_only = warp == kEpiWarps || warp == kEpiWarps + 1;
    if (a.dependent == 1 && !inputs_only) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && !inputs_only) {
        const int t0 = threadIdx.x < kEpiWarps * 32 ? threadIdx.x : threadIdx.x - 64;
        if (P1 && a.tickets_next)
            for (int t = t0; t < 2 * B * a.p.num_kv_heads * a.layers_a; t += kThreadsTc - 64) a.tickets_next[t] = 0u;
        if (P2 && a.tickets)                      // an empty sequence has no tile to finish: it keeps nothing
            for (int t = t0; t < B * a.p.num_kv_heads * a.layers_b; t += kThreadsTc - 64)
                if (t_len[t / a.p.num_kv_heads % B] == 0) {
                    Cut cut;
                    cut.b = 0; cut.ties = 0; cut.tau = 0; cut.prot_kept = 0; cut.sbias = 0;
                    *unit_length(a, t) = 0;
                    if (a.sel_cuts) a.sel_cuts[t] = cut;
                }
    }

    if (warp < kEpiWarps) {
        EpiState es;
        if (P2) epilogue_pass2(a, tl, stage, sv, tmem_base, b0, nb, sp, es);
        if (P1 && na > 0 && !tl.abort_flag) epilogue_pass1(a, tl, tmem_base, es);
    } else if (warp == kEpiWarps) {
        RingState rs;
        if (P2) producer_loop<false>(a, maps_b, smem_q, smem_k, tl, sv, sp, sh_b, rs);
        if (P1) producer_loop<true>(a, maps_a, smem_q, smem_k, tl, sv, sp, sh_a, rs);
    } else if (warp == kEpiWarps + 1) {
        // All lanes of this warp and of the TMA warp walk their loops and one elected lane issues.  With a single lane in them the
        // operands of every instruction went through the registers of a diverged warp, and products came at half the tensor
        // cores' rate (N = 128: 116 cycles, 72 this way; us a run: 16 layers of 8K positions 428 -> 387, 32K x 8 688 -> 663,
        // the ragged batch of eight x 4 697 -> 657, 20K x 8, 512 rows, 756 -> 731).
        MmaState ms;
        if (P2 && nb > 0) mma_loop_pass2(a, smem_q, smem_k, tl, tmem_base, ms, P1);
        __syncwarp();
        if (P1 && na > 0 && !tl.abort_flag) mma_loop_pass1(a, smem_q, smem_k, tl, tmem_base, ms);
    } else if (warp == kEpiWarps + 2) {
        if (a.cj.nslots > 0) copy_loop(a, tl, sv, smem_c, coff);
    } else {
        if (P2) finisher_pass2(a, tl, stage, sv, nb);
    }
    __syncwarp();
    // Common exit.  In the normal case the epilogue has consumed every accumulator,
    // which implies every MMA and every copy has completed.
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0 && tl.abort_flag && a.dev_status) atomicOr(a.dev_status, REFREE_DEV_TIMEOUT);
    if (warp == kEpiWarps + 1) tmem_dealloc(tmem_base, 512);
    if (P2 && a.tickets && !tl.abort_flag) evaluate_rules(a, tl, sv);
}

// ------------------------------------------------------------------ host -----
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

bool shape_for(const refree_params &p, TcShape &sh)
{
    if (p.dtype != REFREE_DTYPE_BF16 || p.head_dim != kD) return false;
    const int G = p.num_q_heads / p.num_kv_heads;
    const int64_t R = (int64_t)G * p.window;
    // One window row has a path of its own (score_w1.cu); few rows are padded to 32, at any length: a layer takes the same
    // form alone and in a run.  (2 to 31 rows, us, here and with the generic kernels: a layer of 200 positions 33 and 37, 2000
    // 37 and 30, 8192 x 8 heads 58 and 74, 32768 x 8 121 and 246; a run of four of 1000 x 8 54 and 141.)
    if (R > kMaxRowsTc || (R < 32 && p.window == 1)) return false;
    sh.R = (int)R;
    sh.rblocks = (sh.R + kTile - 1) / kTile;
    sh.Rpad = sh.rblocks * kTile;
    sh.cblocks = sh.R > 256 ? 2 : 1;
    sh.ncol = ((sh.R + sh.cblocks - 1) / sh.cblocks + 31) / 32 * 32;   // rows past R are masked
    sh.stages = sh.Rpad <= 256 ? 4 : 2;
    sh.slots = kStageSlots;
    sh.rank4 = p.k_stride_seq != 0;
    return true;
}

size_t smem_bytes(const TcShape &sh, int num_seqs, int copy_slots = 0, int piece_rows = 0, int copy_units = 0)
{
    return 1024 + (size_t)sh.Rpad * 256 + (size_t)sh.stages * kTileBytes + (size_t)copy_slots * piece_rows * (kD * 2) +
           (size_t)sh.slots * sizeof(StageSlot) + sizeof(TcSmemTail) + (size_t)(5 * num_seqs + 3) * sizeof(int32_t) +
           (copy_slots ? (size_t)(copy_units + 1) * sizeof(int32_t) : 0);
}

constexpr size_t kSmemLimit = 232448;

// As many staging slots as fit beside the sequence tables (two at least).
bool fit_slots(const refree_params &p, TcShape &sh)
{
    for (sh.slots = kStageSlots; sh.slots >= 2; sh.slots >>= 1)
        if (smem_bytes(sh, p.num_seqs) <= kSmemLimit) return true;
    return false;
}

// Per-device facts, looked up once per device under a lock.
struct DevInfo { bool ready = false; int sms = 0; };
std::mutex g_dev_mutex;
DevInfo g_dev[64];

cudaError_t device_info(DevInfo &out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    DevInfo &d = g_dev[dev];
    if (!d.ready) {
        int n = 0;
        e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(score_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(score_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(score_tc_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
        if (e != cudaSuccess) return e;
        d.sms = std::min(n, kMaxCtas);
        d.ready = true;
    }
    out = d;
    return cudaSuccess;
}

// Ring depth and pieces in flight when the launch also copies rows.  Up to 256 query rows the K ring gives up two of its
// four stages and the finishing warp half of its slots, and pieces of 32 rows take what is left (nine of them).
// Measured at 32K positions, 8 units, us a layer: 2 stages and 9 pieces 88, 2 and 5 95, 3 and 5 95, 3 and 4 100: bytes in
// flight for the copy count for more than a deeper ring.  Beyond 256 rows Q takes 128 KB; the finishing warp keeps two
// slots and nine pieces of 8 rows fit: 18 KB in flight per SM, which is enough because such a layer is scored for twice
// as long (20K positions, 8 units of 512 rows, us a layer: rows moved beside the next layer's scoring by a kernel of its
// own, which found no room on the SMs, 117; four pieces of 16 rows 101; nine of 8 100).  False when fewer than three fit.
bool copy_shape(const refree_params &p, TcShape &sh, int layers, int &nslots, int &piece_rows)
{
    const int U = p.num_seqs * p.num_kv_heads * layers;
    sh.stages = 2;
    for (piece_rows = 32, sh.slots = 4; piece_rows >= 8; piece_rows /= 4, sh.slots /= 2)
        for (nslots = kMaxCopySlots; nslots >= 3; --nslots)
            if (smem_bytes(sh, p.num_seqs, nslots, piece_rows, U) <= kSmemLimit) return true;
    return false;
}

}  // namespace

bool score_tc_can_copy(const refree_params &p, int64_t total_tokens, int layers)
{
    TcShape sh;
    int nslots = 0, piece_rows = 0;
    if (!shape_for(p, sh)) return false;
    if (p.k_stride_tok != kD || p.v_stride_tok != kD) return false;          // a unit's rows back to back
    if ((int64_t)p.num_seqs * p.num_kv_heads * layers > kMaxCopyUnits) return false;
    if ((int64_t)p.num_kv_heads * total_tokens * layers > 0x7fffffffLL) return false;  // row counts held in 32 bits
    if (p.rank_mode != REFREE_RANK_POSITION && !p.force_full) return false;
    return copy_shape(p, sh, layers, nslots, piece_rows);
}

bool score_tc_supported(const refree_params &p)
{
    TcShape sh;
    if (!shape_for(p, sh)) return false;
    if (p.kv_tokens <= 0 || p.kv_tokens > 0x7fffffffLL) return false;
    if (!fit_slots(p, sh)) return false;
    return encode_fn() != nullptr;
}

namespace {

cudaError_t encode_maps(const refree_params &p, const TcShape &sh, const void *q_win, const void *k, CUtensorMap &mapq,
                        CUtensorMap &mapk)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)kD, (cuuint64_t)p.num_seqs * p.num_q_heads * p.window};
        const cuuint64_t strides[1] = {(cuuint64_t)kD * 2};
        const cuuint32_t box[2] = {64, kTile}, estr[2] = {1, 1};
        if (enc(&mapq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(q_win), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)p.kv_tokens, (cuuint64_t)p.num_kv_heads, (cuuint64_t)p.num_seqs};
        const cuuint64_t strides[3] = {(cuuint64_t)p.k_stride_tok * 2, (cuuint64_t)p.k_stride_head * 2,
                                       (cuuint64_t)p.k_stride_seq * 2};
        const cuuint32_t box[4] = {64, kTile, 1, 1}, estr[4] = {1, 1, 1, 1};
        if (enc(&mapk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, sh.rank4 ? 4 : 3, const_cast<void *>(k), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

}  // namespace

// One launch of a run of layers: pass 2 of `finish` (nullable), then pass 1 of `begin` (nullable), and the rows
// of `copy` (nullable) beside them.  The partials that pass 2 reads were completed by an earlier launch on the
// stream, so no CTA waits for another: the launch is not a cooperative one.
cudaError_t launch_score_tc_pipe(const refree_params &p, const TcGroup *begin, const TcGroup *finish,
                                 const int32_t *seq_start, const int32_t *seq_len, int64_t total_tokens,
                                 int32_t *dev_status, Stream st, const TcCopyJob *copy, bool first)
{
    if (!begin && !finish) return cudaErrorInvalidValue;
    TcShape sh;
    if (!shape_for(p, sh)) return cudaErrorInvalidValue;
    int copy_slots = 0, piece_rows = 0;
    if (copy ? !copy_shape(p, sh, copy->layers, copy_slots, piece_rows) : !fit_slots(p, sh)) return cudaErrorInvalidValue;
    TcMaps maps[2];                                     // of `begin`, of `finish`
    cudaError_t e = cudaSuccess;
    for (int which = 0; which < 2; ++which) {
        const TcGroup *g = which ? finish : begin;
        for (int l = 0; g && l < g->layers; ++l)
            if ((e = encode_maps(p, sh, g->q_win[l], g->k[l], maps[which].q[l], maps[which].k[l])) != cudaSuccess) return e;
    }
    DevInfo di;
    e = device_info(di);
    if (e != cudaSuccess) return e;
    const int layers = std::max(begin ? begin->layers : 0, finish ? finish->layers : 0);
    const int64_t max_items = (total_tokens / kTile + p.num_seqs) * p.num_kv_heads * layers;
    // with rows to move, every SM takes part whatever the number of scoring items
    const int ctas = copy ? di.sms : (int)std::max<int64_t>(1, std::min<int64_t>(di.sms, max_items));
    TcArgs a = {};
    a.p = p;
    a.sh = sh;
    a.seq_start = seq_start;
    a.seq_len = seq_len;
    a.total_tokens = total_tokens;
    a.dev_status = dev_status;
    a.split_ctas = di.sms;
    if (begin) {
        a.layers_a = begin->layers;
        a.part_a = begin->part;
        a.tickets_next = begin->tickets;
    }
    if (finish) {
        a.layers_b = finish->layers;
        a.part_b = finish->part;
        a.scores = finish->scores;
        a.groups = finish->groups;
        if (finish->tickets) {                          // the rule runs inside the launch
            a.tickets = finish->tickets;
            a.sel_cuts = finish->cuts;
            for (int l = 0; l < finish->layers; ++l) a.sel_lengths[l] = finish->sel_lengths[l];
        }
    }
    if (copy) a.cj = *copy;
    a.cj.nslots = copy ? copy_slots : 0;
    a.cj.piece_rows = piece_rows;
    const size_t smem = smem_bytes(sh, p.num_seqs, a.cj.nslots, piece_rows, p.num_seqs * p.num_kv_heads * a.cj.layers);
    if (smem > kSmemLimit) return cudaErrorInvalidValue;
    // A launch may start while the one before drains (unless the stream is not to be chained): its CTAs set themselves up and
    // then wait (griddepcontrol.wait) until that launch has completed and its results are visible.  The first one of a call
    // waits before it reads anything, since what is ahead of it may still be writing Q and K.
    a.dependent = !st.chain ? 0 : first ? 2 : 1;
    auto *kern = begin && finish ? score_tc_kernel<3> : begin ? score_tc_kernel<1> : score_tc_kernel<2>;
    e = launch_dependent(kern, dim3(ctas), dim3(kThreadsTc), smem, st, maps[0], maps[1], a);
    if (e != cudaSuccess) return e;
    count_launches(1);
    return cudaGetLastError();
}

// Both passes of one layer: a run of one, two launches of which the second starts while the first drains.  (One
// cooperative launch for both, which waited on flags between the passes, was slower: score, selection and copy of a
// layer of 8 units of 256 rows, us, 8K positions 72.1 -> 68.1, 32K 154.0 -> 152.1.)
cudaError_t launch_score_tc(const refree_params &p, const void *q_win, const void *k,
                            const int32_t *seq_start, const int32_t *seq_len,
                            int64_t total_tokens, float *scores, char *ws, const Workspace &lay,
                            int32_t *dev_status, Stream st, GroupPartial *groups, int32_t *sel_lengths)
{
    TcGroup g = {};
    g.layers = 1;
    g.q_win[0] = q_win;
    g.k[0] = k;
    g.part = reinterpret_cast<float2 *>(ws + lay.part_off);
    g.scores = scores;
    g.groups = groups;                                  // (no tickets: the rule is a launch of its own)
    cudaError_t e = launch_score_tc_pipe(p, &g, nullptr, seq_start, seq_len, total_tokens, dev_status, st, nullptr, true);
    if (e != cudaSuccess) return e;
    e = launch_score_tc_pipe(p, nullptr, &g, seq_start, seq_len, total_tokens, dev_status, st, nullptr, false);
    if (e != cudaSuccess || !groups || !sel_lengths) return e;
    return launch_unit_rules(p, scores, seq_len, total_tokens, groups, 0, select_out(sel_lengths, nullptr, nullptr),
                             reinterpret_cast<Cut *>(ws + lay.cut_off), st);
}

}  // namespace refree
