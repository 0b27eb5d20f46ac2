// Position ranking, one budget per (sequence, KV head), from the per-32-position records (GroupPartial) that a
// scoring kernel leaves: the arithmetic of the stopping rule, evaluated by a block per unit (a launch of its own, the
// cluster kernel of a single query row, a scoring CTA that has left its passes) or by a warp (a scoring CTA that
// completed more units than its list holds).
// Integer sums throughout, so the two agree bit for bit whatever the order of their additions.
#pragma once

#include <limits.h>

#include "refree_internal.cuh"

namespace refree {

// Smallest fixed-point C with 1 - sqrt(C / Cn) < T, i.e. Cn - C < Cn * T * (2 - T); ~0 when there is none.
__device__ inline unsigned long long crossing_level(unsigned long long Cn, double T)
{
    const double lim = (double)Cn * (T * (2.0 - T));
    const double c = ceil(lim);
    if (!(c >= 1.0)) return ~0ull;                 // T = 0: never met
    const unsigned long long dmax = (unsigned long long)c - 1ull;     // largest dropped mass that still meets the rule
    return dmax >= Cn ? 0ull : Cn - dmax;
}

// Common scale of a unit's groups: the largest score's squared mantissa below 2^(56 - L), L = log2 of the group count.
__device__ inline int groups_sbias(uint32_t max_bits, int ng, int &emax, int &L)
{
    emax = max(1, (int)(max_bits >> 23));
    L = 0;
    while ((1 << L) < ng) ++L;
    return kGroupShift - 2 * emax - L;
}

// The rule of one unit, in pieces that a warp or a block puts together.  `sc` = the unit's scores, `gp` = its records,
// `mx` = bit pattern of its largest score.  Reads go around L1 (the data may have been written by other SMs a moment
// ago).  Everything is integer sums, so the result does not depend on who adds what.
struct UnitRule {
    const float *sc;
    const uint4 *raw;
    double threshold;
    int n, lead, floor_b, ng, emax, L, sbias;
    uint32_t mx;

    __device__ inline UnitRule(const refree_params &p, const float *scores, int len, const GroupPartial *gp, uint32_t max_bits)
        : sc(scores), raw(reinterpret_cast<const uint4 *>(gp)), threshold((double)p.threshold), n(len), lead(min(p.sink, len)),
          floor_b(p.keep_window ? min(len, min(p.sink, len) + min(p.window, len)) : min(len, 1)), ng(ceil_div(len, 32)), mx(max_bits)
    {
        sbias = groups_sbias(mx, ng, emax, L);
    }
    __device__ inline Cut keep_all() const
    {
        Cut cut;
        cut.b = n; cut.ties = 0; cut.tau = 0; cut.prot_kept = 0; cut.sbias = 0;
        return cut;
    }
    __device__ inline Cut cut_at(int jstar) const
    {
        Cut cut = keep_all();
        cut.sbias = sbias;
        cut.b = max(jstar == INT_MAX ? n : jstar, floor_b);
        return cut;
    }
    __device__ inline unsigned long long square(int i) const { return sq_fixed(mag_bits(__ldcg(sc + i)), sbias); }
    // groups in ranked order: rank r = group ng - 1 - r
    __device__ inline uint4 record(int r) const { return __ldcg(raw + (ng - 1 - r)); }
    // sum of a group at the unit's scale
    __device__ inline unsigned long long whole(const uint4 &rec) const
    {
        const unsigned long long sum = ((unsigned long long)rec.w << 32) | rec.z;
        const int shift = 2 * (emax - max(1, (int)(rec.x >> 23))) + L;
        return shift < 64 ? sum >> shift : 0ull;
    }
    // the same without the leading positions (ranked first, apart)
    __device__ inline unsigned long long rest_of(const uint4 &rec, int r) const
    {
        const int k = ng - 1 - r;
        unsigned long long v = whole(rec);
        if (32 * k < lead) {
            unsigned long long in = 0;
            for (int i = 32 * k; i < min(lead, 32 * k + 32); ++i) in += square(i);
            v = v > in ? v - in : 0ull;
        }
        return v;
    }
    // mass of the leading positions, by a warp
    __device__ inline unsigned long long sink_mass() const
    {
        unsigned long long sink = 0;
        for (int i = threadIdx.x & 31; i < lead; i += 32) sink += square(i);
        for (int o = 16; o; o >>= 1) sink += __shfl_xor_sync(0xffffffffu, sink, o);
        return sink;
    }
    // rank count of a crossing among the leading positions, by a warp, 32 at a time; INT_MAX: none
    __device__ inline int cross_lead(unsigned long long c_min) const
    {
        const int lane = threadIdx.x & 31;
        unsigned long long c = 0;
        for (int i0 = 0; i0 < lead; i0 += 32) {
            const int i = i0 + lane;
            const unsigned long long xi = warp_incl_scan(i < lead ? square(i) : 0ull);
            const unsigned m = __ballot_sync(0xffffffffu, i < lead && c + xi >= c_min);
            if (m) return i0 + __ffs(m);
            c += __shfl_sync(0xffffffffu, xi, 31);
        }
        return INT_MAX;
    }
    // rank count of the crossing inside the group of rank r, `base` being the sum before it, by a warp
    __device__ inline int cross_group(int r, unsigned long long base, unsigned long long c_min) const
    {
        const int lane = threadIdx.x & 31, k = ng - 1 - r;
        const int hi = min(n, 32 * k + 32) - 1, lo = max(lead, 32 * k);
        const int pos = hi - lane;
        const unsigned long long x = warp_incl_scan(pos >= lo ? square(pos) : 0ull);
        const unsigned mp = __ballot_sync(0xffffffffu, pos >= lo && base + x >= c_min);
        // rank count of position pos: the leading ones, then n-1 down to pos
        return lead + (n - (mp ? hi - (__ffs(mp) - 1) : lo));
    }
    // rank count of the crossing inside ranks [q0, q1) of the groups, `run` being the sum before them, by a warp
    __device__ inline int cross_run(int q0, int q1, unsigned long long run, unsigned long long c_min) const
    {
        const int lane = threadIdx.x & 31;
        for (int rb = q0; rb < q1; rb += 32) {
            const int r = rb + lane;
            const unsigned long long v = r < q1 ? rest_of(record(r), r) : 0ull;
            const unsigned long long vi = warp_incl_scan(v);
            const unsigned m = __ballot_sync(0xffffffffu, r < q1 && run + vi >= c_min);
            if (m) {
                const int src = __ffs(m) - 1;
                return cross_group(rb + src, run + __shfl_sync(0xffffffffu, vi - v, src), c_min);
            }
            run += __shfl_sync(0xffffffffu, vi, 31);
        }
        return INT_MAX;
    }
};

// The whole rule for one unit by a block of NT threads (all call it): two round trips to L2, one block scan.  Budget and
// record go to *length and *cut_out (nullable).  The block synchronises before it returns.
template <int NT> struct BlockRuleShared {
    unsigned long long sum[NT / 32];
    int first;                                             // first thread in whose run of groups the sum crosses
};
template <int NT>
__device__ inline void block_unit_rule(const UnitRule &ur, BlockRuleShared<NT> &sh, int32_t *length, Cut *cut_out)
{
    typedef unsigned long long u64;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto store = [&](const Cut &cut) {
        *length = cut.b;
        if (cut_out) *cut_out = cut;
    };
    if (ur.n <= 0 || ur.mx == 0u) {                        // (the same in every thread)
        if (tid == 0) store(ur.keep_all());
        __syncthreads();
        return;
    }
    // groups in ranked order: thread t owns a contiguous run of ranks
    const int per = ceil_div(ur.ng, NT);
    const int r0 = min(ur.ng, tid * per), r1 = min(ur.ng, r0 + per);
    constexpr int kRun = 4;                                // a short run's records are loaded together and kept
    u64 local = 0, sink, kept[kRun] = {};
    uint4 rec[kRun];
    const bool short_run = per <= kRun;
    if (short_run)
#pragma unroll
        for (int q = 0; q < kRun; ++q) rec[q] = r0 + q < r1 ? ur.record(r0 + q) : make_uint4(0u, 0u, 0u, 0u);
    const u64 lead_inc = warp_incl_scan(ur.lead <= 32 && lane < ur.lead ? ur.square(lane) : 0ull);     // (usually four positions)
    if (ur.lead <= 32) {
        sink = __shfl_sync(0xffffffffu, lead_inc, 31);     // all of them in the last-ranked group
        auto rest = [&](const uint4 &x, int r) {
            const u64 v = ur.whole(x);
            return r < ur.ng - 1 ? v : (v > sink ? v - sink : 0ull);
        };
        if (short_run) {
#pragma unroll
            for (int q = 0; q < kRun; ++q) {
                if (r0 + q < r1) kept[q] = rest(rec[q], r0 + q);
                local += kept[q];
            }
        } else {
            for (int r = r0; r < r1; ++r) local += rest(ur.record(r), r);
        }
    } else {
        if (short_run) {
#pragma unroll
            for (int q = 0; q < kRun; ++q) {
                if (r0 + q < r1) kept[q] = ur.rest_of(rec[q], r0 + q);
                local += kept[q];
            }
        } else {
            for (int r = r0; r < r1; ++r) local += ur.rest_of(ur.record(r), r);
        }
        sink = ur.sink_mass();                             // every warp for itself
    }
    const u64 inc = warp_incl_scan(local);
    if (tid == 0) sh.first = INT_MAX;
    if (lane == 31) sh.sum[warp] = inc;
    __syncthreads();
    u64 before = 0, total = 0;
#pragma unroll
    for (int x = 0; x < NT / 32; ++x) { const u64 v = sh.sum[x]; before += x < warp ? v : 0ull; total += v; }
    const u64 c_min = crossing_level(sink + total, ur.threshold);
    int jstar = INT_MAX;
    if (ur.lead <= 32) {
        const unsigned m = __ballot_sync(0xffffffffu, lane < ur.lead && lead_inc >= c_min);
        if (m) jstar = __ffs(m);
    } else {
        jstar = ur.cross_lead(c_min);
    }
    const u64 run_end = sink + before + inc;
    if (jstar == INT_MAX && c_min != ~0ull) {
        const unsigned m = __ballot_sync(0xffffffffu, r0 < r1 && run_end >= c_min);
        if (m && lane == 0) atomicMin(&sh.first, warp * 32 + __ffs(m) - 1);
    }
    __syncthreads();
    const int owner = sh.first;
    if (owner != INT_MAX && (owner >> 5) == warp) {
        u64 base = run_end - local;                        // the sum before the thread's run
        if (short_run) {                                   // the owner knows in which of its groups the sum crosses
            int r = r0;
#pragma unroll
            for (int q = 0; q + 1 < kRun; ++q)
                if (r == r0 + q && r + 1 < r1 && base + kept[q] < c_min) { base += kept[q]; ++r; }
            base = __shfl_sync(0xffffffffu, base, owner & 31);
            r = __shfl_sync(0xffffffffu, r, owner & 31);
            jstar = ur.cross_group(r, base, c_min);
        } else {
            base = __shfl_sync(0xffffffffu, base, owner & 31);
            jstar = ur.cross_run(min(ur.ng, owner * per), min(ur.ng, owner * per + per), base, c_min);
        }
    }
    if (warp == (owner == INT_MAX ? 0 : owner >> 5) && lane == 0) store(ur.cut_at(jstar));
    __syncthreads();                                       // the shared words may be used again
}

// The whole rule for one unit by one warp (all 32 lanes call it).
__device__ inline Cut select_unit_from_groups_warp(const refree_params &p, const float *sc, int n, const GroupPartial *gp, uint32_t mx)
{
    const int lane = threadIdx.x & 31;
    const UnitRule ur(p, sc, n, gp, mx);
    if (n <= 0 || mx == 0u) return ur.keep_all();
    const unsigned long long sink = ur.sink_mass();
    // lane t owns a contiguous run of ranks and sums it, eight records in flight at a time
    const int per = ceil_div(ur.ng, 32);
    const int r0 = min(ur.ng, lane * per), r1 = min(ur.ng, r0 + per);
    unsigned long long local = 0;
    for (int r = r0; r < r1; r += 8) {
        uint4 rec[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) rec[q] = r + q < r1 ? ur.record(r + q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int q = 0; q < 8; ++q) if (r + q < r1) local += ur.rest_of(rec[q], r + q);
    }
    const unsigned long long inc = warp_incl_scan(local);
    const unsigned long long c_min = crossing_level(sink + __shfl_sync(0xffffffffu, inc, 31), ur.threshold);
    int jstar = ur.cross_lead(c_min);
    if (jstar == INT_MAX && c_min != ~0ull) {
        // the lane in whose run the cumulative sum reaches c_min
        const unsigned mrun = __ballot_sync(0xffffffffu, r0 < r1 && sink + inc >= c_min);
        if (mrun) {
            const int owner = __ffs(mrun) - 1;
            const unsigned long long run = sink + __shfl_sync(0xffffffffu, inc - local, owner);
            jstar = ur.cross_run(min(ur.ng, owner * per), min(ur.ng, owner * per + per), run, c_min);
        }
    }
    return ur.cut_at(jstar);
}

}  // namespace refree
